"""A call that refuses its f leaves nothing running on the context's stream: the hidden layer is enqueued beside the check
and reads the caller's f and parameters."""
import pytest

from paper_2207_05341_gb300 import qst

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,prec,net", [(11, qst.QST_FP32, qst.QST_NET_FNN), (10, qst.QST_FP64, qst.QST_NET_FNN),
                                        (10, qst.QST_FP32, qst.QST_NET_CNN)])
def test_stream_is_idle_after_a_refusal(N, prec, net):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dt = torch.float64 if prec == qst.QST_FP64 else torch.float32
    o = qst.qst_default_options()
    o.precision, o.network = prec, net
    s = torch.cuda.Stream()
    f = torch.full((4 ** N,), 1.0 / 4 ** N, device="cuda", dtype=dt)
    f[1] = float("nan")
    theta = torch.zeros(qst.qst_theta_size_net(N, net), device="cuda", dtype=dt)
    dtheta = torch.empty_like(theta)
    torch.cuda.synchronize()
    ctx = qst.qst_init(N, opt=o, stream=s.cuda_stream)
    try:
        qst.qst_set_params(ctx, theta)
        for call in (lambda: qst.qst_loss_grad(ctx, theta, f, dtheta), lambda: qst.qst_step(ctx, f),
                     lambda: qst.qst_get_rho(ctx, f, None, want_loss=True)):
            for _ in range(5):
                with pytest.raises(qst.QstError) as e:
                    call()
                idle = s.query()
                assert e.value.status == qst.QST_E_INPUT and idle
    finally:
        qst.qst_destroy(ctx)
