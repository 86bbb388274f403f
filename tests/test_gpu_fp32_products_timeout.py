"""A tensor-core product whose operand copies never come (injected; the waits end at their limit) leaves its result
unwritten, whether a tile is one CTA's (N = 11) or shared by a cluster (N = 7 to 10): rho formed after it is still that
of the parameters before, bit for bit."""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mapping", [qst.QST_MAP_CHOL_H, qst.QST_MAP_CHOL_DELTA])
@pytest.mark.parametrize("N", [7, 8, 9, 10, 11])
def test_result_unwritten(N, mapping):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    o = qst.qst_default_options()
    o.mapping = mapping
    o.fused_max_qubits = -1
    f = torch.full((4 ** N,), 1.0 / 4 ** N, device="cuda")
    theta = [torch.from_numpy(synth.init_theta(N, s).astype(np.float32)).cuda() for s in (1, 2)]
    rho = [torch.zeros(1 << N, 1 << N, dtype=torch.complex64, device="cuda") for _ in range(3)]
    ctx = qst.qst_init(N, opt=o)
    try:
        qst.qst_set_params(ctx, theta[0])
        qst.qst_get_rho(ctx, f, rho[0], want_loss=True)
        qst.qst_set_params(ctx, theta[1])
        qst.qst_inject_wait_timeout(qst.QST_INJECT_TC_LOADS, 1)
        try:
            with pytest.raises(qst.QstError) as e:
                qst.qst_get_rho(ctx, f, rho[1], want_loss=True)
            assert e.value.status == qst.QST_E_TIMEOUT
        finally:
            qst.qst_inject_wait_timeout(qst.QST_INJECT_TC_LOADS, 0)
        qst.qst_sync(ctx)
        assert torch.equal(rho[1], rho[0])
        qst.qst_get_rho(ctx, f, rho[2], want_loss=True)  # works again, with the new parameters
        assert not torch.equal(rho[2], rho[0]) and bool(torch.isfinite(rho[2].abs()).all())
    finally:
        qst.qst_destroy(ctx)
