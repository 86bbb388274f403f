"""FP64 contexts spread their products (16 x 16 tiles, K split over a cluster) and POVM passes (small tiles)
over the GPU: loss, gradient and rho against the oracle at every size up to N = 8 and at N = 10's tiling
through N = 9, for Chol_H (full and lower products) and Chol_Delta, at the FP64 bar of 1e-10."""
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


@pytest.mark.parametrize("N", [3, 4, 5, 6, 7, 8, 9])
def test_loss_gradient_and_probabilities(N):
    rho = synth.ginibre_mixed(N, 3, 30 + N)
    f = synth.frequencies(synth.multinomial_counts(O.born_probabilities(rho, M).real, 10**5, 40 + N))
    theta = synth.init_theta(N, 50 + N)
    o = qst.qst_default_options()
    o.precision = qst.QST_FP64
    ctx = qst.qst_init(N, opt=o)
    try:
        th, fd = torch.from_numpy(theta).cuda(), torch.from_numpy(f).cuda()
        g = torch.empty_like(th)
        loss, _ = qst.qst_loss_grad(ctx, th, fd, g)
        p = torch.empty(4 ** N, dtype=torch.float64, device="cuda")
        qst.qst_probs(ctx, torch.from_numpy(rho).cuda(), p)
        want_l, want_g, _ = O.loss_and_grad(theta, f, M, N)
        want_p = O.born_probabilities(rho, M).real
        assert abs(loss - want_l) <= 1e-10 * abs(want_l)
        assert np.linalg.norm(g.cpu().numpy() - want_g) <= 1e-10 * np.linalg.norm(want_g)
        assert np.abs(p.cpu().numpy() - want_p).max() <= 1e-10 * want_p.max()
    finally:
        qst.qst_destroy(ctx)
