"""qst_batch_reconstruct without losses: the states are ordered before whatever follows on the batch's stream (its
synchronisation and the next iteration, which uses the same buffers), and a refused call has waited for them."""
import ctypes

import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NS = (10, 9, 4, 8, 10)


def _inputs():
    rng = np.random.default_rng(3)
    return ([torch.from_numpy(rng.dirichlet(np.ones(4**N)).astype(np.float32)).cuda() for N in NS],
            [torch.from_numpy(synth.init_theta(N, 50 + b).astype(np.float32)).cuda() for b, N in enumerate(NS)],
            [torch.zeros((1 << N, 1 << N), dtype=torch.complex64, device="cuda") for N in NS])


def _run(want_losses):
    fs, thetas, rhos = _inputs()
    torch.cuda.synchronize()
    b = qst.qst_batch_init(list(NS))
    try:
        for i, th in enumerate(thetas):
            qst.qst_batch_set_params(b, i, th)
        states = []
        for _ in range(3):
            qst.qst_batch_reconstruct(b, fs, 2, rhos, want_losses=want_losses)
            qst.qst_batch_sync(b)
            states.append([r.cpu() for r in rhos])
            qst.qst_batch_reconstruct(b, fs, 1, rhos, want_losses=want_losses)  # and straight on with the iterations
        last = qst.qst_batch_reconstruct(b, fs, 2, None, want_losses=True)
        return states, last
    finally:
        qst.qst_batch_destroy(b)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qst.load()


def test_states_and_the_iterations_after_them():
    (want, want_last), (got, got_last) = _run(True), _run(False)
    assert got_last == want_last
    for w, g in zip(want, got):
        assert all(torch.equal(x, y) for x, y in zip(w, g))


def test_a_refused_call_has_waited():
    fs, thetas, rhos = _inputs()
    b = qst.qst_batch_init(list(NS))
    try:
        for i, th in enumerate(thetas):
            qst.qst_batch_set_params(b, i, th)
        qst.qst_batch_reconstruct(b, fs, 0, rhos)  # each f's hidden layer is kept
        want = [r.cpu() for r in rhos]
        fs[-1] = fs[-1].clone()
        fs[-1][7] = -1.0
        for r in rhos:
            r.zero_()
        torch.cuda.synchronize()
        fp = (ctypes.c_void_p * len(NS))(*[f.data_ptr() for f in fs])
        rp = (ctypes.c_void_p * len(NS))(*[r.data_ptr() for r in rhos])
        assert qst.load().qst_batch_reconstruct(b, fp, 0, rp, None) == qst.QST_E_INPUT
        got = [r.clone() for r in rhos]
        torch.cuda.synchronize()
        assert all(torch.equal(g.cpu(), w) for g, w in zip(got[:-1], want[:-1]))
        assert not bool(got[-1].abs().any())
    finally:
        qst.qst_batch_destroy(b)
