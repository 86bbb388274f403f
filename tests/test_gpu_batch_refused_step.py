"""A refused qst_batch_step leaves nothing in flight: with iterations still running and the first tomography's f bad, the
checks of the others have ended when the call returns, so that the next steps with the earlier inputs (which reduce
through the same partial sums, on the batch's stream) give the bits of a run without the refused call."""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NS = (7, 9, 8, 9, 4)


def _run(refused):
    rng = np.random.default_rng(5)
    fs = [torch.from_numpy(rng.dirichlet(np.ones(4**N)).astype(np.float32)).cuda() for N in NS]
    other = [f.clone() for f in fs]
    other[0][3] = float("nan")
    thetas = [torch.from_numpy(synth.init_theta(N, 40 + b).astype(np.float32)).cuda() for b, N in enumerate(NS)]
    torch.cuda.synchronize()
    b = qst.qst_batch_init(list(NS))
    try:
        for i, th in enumerate(thetas):
            qst.qst_batch_set_params(b, i, th)
        losses = []
        for _ in range(4):
            for _ in range(2):
                qst.qst_batch_step(b, fs)
            if refused:
                with pytest.raises(qst.QstError) as e:
                    qst.qst_batch_step(b, other)
                assert e.value.status == qst.QST_E_INPUT
            losses.append(qst.qst_batch_step(b, fs, want_losses=True))
        qst.qst_batch_sync(b)
        for i, th in enumerate(thetas):
            qst.qst_get_params(qst.qst_batch_context(b, i), th)
        torch.cuda.synchronize()
        return losses, [th.cpu() for th in thetas]
    finally:
        qst.qst_batch_destroy(b)


def test_steps_around_a_refused_step():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    want, got = _run(False), _run(True)
    assert got[0] == want[0]
    for a, c in zip(got[1], want[1]):
        assert torch.equal(a, c)
