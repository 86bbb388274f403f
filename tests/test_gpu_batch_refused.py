"""qst_batch_reconstruct enqueues every tomography before it waits for the first: where one is refused, those before it
have been waited for, with the loss and the state that they have on their own, and the refusal is returned."""
import ctypes

import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,bad", [((4, 9, 3), 2), ((9, 8, 4), 1), ((3, 7), 0)])
def test_losses_before_a_refused_tomography(Ns, bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = qst.load()
    rng = np.random.default_rng(sum(Ns))
    fs = [torch.from_numpy(rng.dirichlet(np.ones(4**N)).astype(np.float32)).cuda() for N in Ns]
    thetas = [synth.init_theta(N, 30 + N).astype(np.float32) for N in Ns]
    want = []
    for N, f, th in zip(Ns, fs, thetas):
        c = qst.qst_init(N)
        try:
            qst.qst_set_params(c, th)
            rho = torch.empty((1 << N, 1 << N), dtype=torch.complex64, device="cuda")
            want.append((qst.qst_get_rho(c, f, rho, want_loss=True)[0], rho))
        finally:
            qst.qst_destroy(c)
    fs[bad] = fs[bad].clone()
    fs[bad][1] = float("nan")
    rhos = [torch.zeros((1 << N, 1 << N), dtype=torch.complex64, device="cuda") for N in Ns]
    losses = (ctypes.c_double * len(Ns))(*([-7.0] * len(Ns)))
    b = qst.qst_batch_init(list(Ns))
    try:
        for i, th in enumerate(thetas):
            qst.qst_batch_set_params(b, i, th)
        fp = (ctypes.c_void_p * len(Ns))(*[f.data_ptr() for f in fs])
        rp = (ctypes.c_void_p * len(Ns))(*[r.data_ptr() for r in rhos])
        torch.cuda.synchronize()
        assert lib.qst_batch_reconstruct(b, fp, 0, rp, losses) == qst.QST_E_INPUT
        done = [(losses[i], rhos[i].clone()) for i in range(bad)]
    finally:
        qst.qst_batch_destroy(b)
    for i, (loss, rho) in enumerate(done):
        assert loss == want[i][0] and torch.equal(rho, want[i][1])
    assert all(losses[i] == -7.0 for i in range(bad, len(Ns)))
