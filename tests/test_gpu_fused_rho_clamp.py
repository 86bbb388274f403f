"""qst_get_rho without a loss forms no likelihood: parameters whose likelihood clamps leave no warning behind for the next
step (fused and general contexts alike)."""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _povm():
    """{|0><0|, |1><1|, |+><+|, |-><-|} / 2."""
    kets = [np.array([1, 0]), np.array([0, 1]), np.array([1, 1]) / np.sqrt(2), np.array([1, -1]) / np.sqrt(2)]
    m = np.stack([np.outer(k, k) / 2 for k in kets])
    return np.ascontiguousarray(np.stack([m, np.zeros_like(m)], -1).reshape(-1))


@pytest.mark.parametrize("N,fused", [(1, 7), (4, 7), (6, 7), (7, 7), (4, -1), (7, -1)])
def test_no_warning_left_behind(N, fused):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, H = 4 ** N, 2 * N
    pure = np.zeros(synth.theta_size(N), np.float32)
    pure[2 * H * n] = 2.0  # t = (2, 0, ..., 0): outcomes with a |1><1| factor have q = 0
    good = synth.init_theta(N, 6).astype(np.float32)
    f = torch.full((n,), 1.0 / n, device="cuda")
    rho = torch.empty(1 << N, 1 << N, dtype=torch.complex64, device="cuda")
    o = qst.qst_default_options()
    o.fused_max_qubits = fused
    ctx = qst.qst_init(N, povm=_povm(), opt=o)
    try:
        qst.qst_set_params(ctx, pure)
        assert qst.qst_get_rho(ctx, f, rho, want_loss=True)[1] == qst.QST_W_CLAMP
        assert qst.qst_get_rho(ctx, f, rho)[1] == qst.QST_OK
        got = rho.cpu().numpy()
        assert got[0, 0] == 1.0 and np.count_nonzero(got) == 1
        qst.qst_set_params(ctx, good)
        assert qst.qst_step(ctx, f)[1] == qst.QST_OK
    finally:
        qst.qst_destroy(ctx)
