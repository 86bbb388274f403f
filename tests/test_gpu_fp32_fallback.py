"""Which products an FP32 context runs: with an injected failure of the tensor-core products' copies a context that has
their operand planes reports QST_E_TIMEOUT, one whose budget has no room for them runs on the CUDA cores, untouched."""
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mapping", [qst.QST_MAP_CHOL_H, qst.QST_MAP_CHOL_DELTA])
@pytest.mark.parametrize("N", [7, 9])
def test_path_by_budget(N, mapping):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 4 ** N
    f = torch.full((n,), 1.0 / n, device="cuda")
    theta = torch.from_numpy(synth.init_theta(N, 4)).float().cuda()
    g = torch.empty_like(theta)
    # parameters, Rprop state, scratch; the planes take 30 n bytes more
    for limit, planes in ((0, True), (2 * 4 * theta.numel() + 60 * n + (1 << 20), False)):
        o = qst.qst_default_options()
        o.mapping, o.device_memory_limit, o.fused_max_qubits = mapping, limit, -1
        ctx = qst.qst_init(N, opt=o)
        qst.qst_inject_wait_timeout(qst.QST_INJECT_TC_LOADS, 1)
        try:
            if planes:
                with pytest.raises(qst.QstError) as e:
                    qst.qst_loss_grad(ctx, theta, f, g)
                assert e.value.status == qst.QST_E_TIMEOUT
            else:
                assert qst.qst_loss_grad(ctx, theta, f, g)[1] == qst.QST_OK
        finally:
            qst.qst_inject_wait_timeout(qst.QST_INJECT_TC_LOADS, 0)
            qst.qst_destroy(ctx)
