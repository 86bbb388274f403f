"""The CNN's output layer reads and writes parameters 16 bytes at a time where they lie on 16-byte boundaries and one by
one elsewhere (qst_loss_grad takes theta and dtheta at any real's address): the same sums either way, so loss and
gradient have to be equal to the last bit."""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,prec,offsets", [(3, qst.QST_FP32, (1, 1)), (4, qst.QST_FP64, (1, 1)),
                                            (5, qst.QST_FP64, (1, 0)), (6, qst.QST_FP32, (0, 3)),
                                            (7, qst.QST_FP32, (2, 0)), (9, qst.QST_FP32, (1, 2))])
def test_loss_grad_of_parameters_off_16_bytes(N, prec, offsets):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dt = torch.float64 if prec == qst.QST_FP64 else torch.float32
    theta = torch.from_numpy(synth.init_theta_cnn(N, 40 + N)).to("cuda", dt)
    f = torch.from_numpy(np.random.default_rng(N).dirichlet(np.ones(4**N))).to("cuda", dt)
    o = qst.qst_default_options()
    o.precision, o.network = prec, qst.QST_NET_CNN
    ctx = qst.qst_init(N, opt=o)
    try:
        g = torch.zeros_like(theta)
        L, _ = qst.qst_loss_grad(ctx, theta, f, g)
        th = torch.zeros(theta.numel() + 4, dtype=dt, device="cuda")[offsets[0]:offsets[0] + theta.numel()]
        th.copy_(theta)
        buf = torch.full((theta.numel() + 4,), 7.0, dtype=dt, device="cuda")
        g2 = buf[offsets[1]:offsets[1] + theta.numel()]
        L2, _ = qst.qst_loss_grad(ctx, th, f, g2)
    finally:
        qst.qst_destroy(ctx)
    assert L2 == L
    assert torch.equal(g2, g)
    assert bool((buf[:offsets[1]] == 7).all()) and bool((buf[offsets[1] + theta.numel():] == 7).all())
