"""qst_get_rho and qst_reconstruct of small FP32 contexts, which run as one launch: rho and its loss against the
oracle at every size of that path, into device and host memory and without rho, and rho unchanged by the call.
Tolerance: FP32 products of d terms and N 4 x 4 maps, 1e-5 of the largest entry and of the loss."""
import numpy as np
import pytest

import oracle as O
from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

M = O.tetrahedral_povm()


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    if not os.path.exists(qst.LIB_PATH):
        from paper_2207_05341_gb300 import build
        build.build()
    qst.load()


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
def test_rho_and_loss(N):
    d = 1 << N
    f64 = synth.frequencies(synth.multinomial_counts(
        O.born_probabilities(synth.ginibre_mixed(N, max(1, d // 2), 60 + N), M).real, 10**5, 70 + N)).astype(np.float32)
    theta = synth.init_theta(N, 80 + N).astype(np.float32)
    o = qst.qst_default_options()
    o.fused_max_qubits = 7
    ctx = qst.qst_init(N, opt=o)
    try:
        qst.qst_set_params(ctx, theta)
        f = torch.from_numpy(f64).cuda()
        rho = torch.empty(d, d, dtype=torch.complex64, device="cuda")
        loss, st = qst.qst_get_rho(ctx, f, rho, want_loss=True)
        host = np.empty((d, d), np.complex64)
        loss_h, _ = qst.qst_get_rho(ctx, f, host, want_loss=True)
        loss_n, _ = qst.qst_reconstruct(ctx, f, 0)
        want_l, _, _ = O.loss_and_grad(theta.astype(np.float64), f64.astype(np.float64), M, N)
    finally:
        qst.qst_destroy(ctx)
    got = rho.cpu().numpy()
    assert st == qst.QST_OK and loss == loss_h == loss_n
    want = _rho(theta.astype(np.float64), f64.astype(np.float64), N)
    assert np.array_equal(got, host)
    assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max()
    assert abs(loss - want_l) <= 1e-5 * abs(want_l)


def _rho(theta, f, N):
    n, H, d = 4 ** N, 2 * N, 1 << N
    W1, W2T = theta[:H * n].reshape(H, n), theta[H * n:2 * H * n].reshape(H, n)
    b2, b1 = theta[2 * H * n:2 * H * n + n], theta[2 * H * n + n:]
    pre = W1 @ f + b1
    R = (np.where(pre > 0, pre, 0.01 * pre) @ W2T + b2).reshape(d, d)
    low = np.tril(R, -1) + 1j * np.triu(R, 1).T
    T = low + low.conj().T + np.diag(np.diag(R))
    X = T @ T
    return X / np.trace(X).real
