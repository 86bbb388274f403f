"""FP32 matrix products on the tensor cores (three-term BF16 operands) against 64 bits.

With W1 = W2 = 0 and b1 = 0 the network gives t = b2 exactly, so T is known exactly and rho = X / Tr X
shows the product alone.  Per entry, |X_ij - exact| <= c S_ij with S = |T| |T| (componentwise):
the dropped term pairs cost at most 3 * 2^-26, the two full-size steps of a 32-element block at most
4 * 2^-23 (truncation, two per step), the sum of the 2d / 32 blocks (2d / 32) 2^-24, the two scalings and
the division by the trace 4 * 2^-24 with the trace's own relative error on top (a sum of positive terms:
the same bound).  The bar is twice c, for the trace, on every entry.
"""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    if not os.path.exists(qst.LIB_PATH):
        from paper_2207_05341_gb300 import build
        build.build()
    qst.load()


def _theta(N, t):
    n, H = 4 ** N, 2 * N
    return np.concatenate([np.zeros(2 * H * n, np.float32), t.astype(np.float32), np.zeros(H, np.float32)])


def _T(t, N, lower):
    R = t.astype(np.float32).astype(np.float64).reshape(1 << N, 1 << N)
    low = np.tril(R, -1) + 1j * np.triu(R, 1).T
    return low + np.diag(np.diag(R)) + (0 if lower else low.conj().T)


def _rho(N, t, mapping, limit=0):
    o = qst.qst_default_options()
    o.mapping = mapping
    o.fused_max_qubits = -1
    o.device_memory_limit = limit
    ctx = qst.qst_init(N, opt=o)
    try:
        f = torch.full((4 ** N,), 1.0 / 4 ** N, device="cuda")
        rho = torch.empty(1 << N, 1 << N, dtype=torch.complex64, device="cuda")
        qst.qst_set_params(ctx, _theta(N, t))
        qst.qst_get_rho(ctx, f, rho)
        g = torch.empty(qst.qst_theta_size(N), device="cuda")
        loss, _ = qst.qst_loss_grad(ctx, torch.from_numpy(_theta(N, t)).cuda(), f, g)
        n, H = 4 ** N, 2 * N
        return rho.cpu().numpy().astype(np.complex128), g[2 * H * n:2 * H * n + n].cpu().numpy().astype(np.float64)
    finally:
        qst.qst_destroy(ctx)


def _values(N, spread, seed):
    r = np.random.default_rng(seed)
    t = r.standard_normal(4 ** N)
    if spread == "wide":  # entries over twelve orders of magnitude
        t *= 10.0 ** r.uniform(-12, 0, 4 ** N)
    elif spread == "tiny":
        t *= 2.0 ** -60
    elif spread == "huge":
        t *= 2.0 ** 40
    return t.astype(np.float32)


@pytest.mark.parametrize("mapping", [qst.QST_MAP_CHOL_H, qst.QST_MAP_CHOL_DELTA])
@pytest.mark.parametrize("N,spread", [(7, "plain"), (7, "wide"), (7, "tiny"), (7, "huge"), (8, "plain"),
                                      (9, "wide"), (10, "plain"), (11, "plain")])
def test_rho_entry_by_entry(N, spread, mapping):
    d = 1 << N
    t = _values(N, spread, 10 * N + len(spread))
    T = _T(t, N, mapping == qst.QST_MAP_CHOL_DELTA)
    A = T.conj().T
    X, S = A @ T, np.abs(A) @ np.abs(T)
    rho, _ = _rho(N, t, mapping)
    tr = np.trace(X).real
    c = 3 * 2.0 ** -26 + 4 * 2.0 ** -23 + (2 * d / 32) * 2.0 ** -24 + 4 * 2.0 ** -24
    assert np.all(np.abs(rho * tr - X) <= 2 * c * S)


@pytest.mark.parametrize("mapping", [qst.QST_MAP_CHOL_H, qst.QST_MAP_CHOL_DELTA])
def test_a_budget_without_room_for_the_planes_keeps_the_cuda_core_products(mapping):
    """The operand planes are optional: a budget that held a context before still does, with the same
    results to FP32 rounding (the gradient through a product whose terms cancel: 100 times the bar above)."""
    N = 7
    d, nn = 1 << N, 4 ** N
    t = _values(N, "plain", 5)
    P = qst.qst_theta_size(N)
    tight = 2 * 4 * P + 60 * nn + (1 << 20)  # parameters, Rprop state, scratch; the planes take 30 nn more
    a, ga = _rho(N, t, mapping)
    b, gb = _rho(N, t, mapping, tight)
    c = 3 * 2.0 ** -26 + 4 * 2.0 ** -23 + (2 * d / 32) * 2.0 ** -24 + 4 * 2.0 ** -24
    T = np.abs(_T(t, N, mapping == qst.QST_MAP_CHOL_DELTA))
    S = T.T @ T
    assert np.all(np.abs(a - b) * np.trace(S) <= 4 * c * S)
    assert np.linalg.norm(ga - gb) <= 100 * c * np.linalg.norm(gb)


def test_an_injected_timeout_is_reported_and_the_context_recovers():
    N = 7
    t = _values(N, "plain", 6)
    f = torch.full((4 ** N,), 1.0 / 4 ** N, device="cuda")
    o = qst.qst_default_options()
    o.fused_max_qubits = -1
    ctx = qst.qst_init(N, opt=o)
    try:
        qst.qst_set_params(ctx, _theta(N, t))
        want = [qst.qst_step(ctx, f)[0] for _ in range(2)]
        qst.qst_set_params(ctx, _theta(N, t))
        qst.qst_inject_wait_timeout(qst.QST_INJECT_TC_LOADS, 1)
        try:
            with pytest.raises(qst.QstError) as e:
                qst.qst_step(ctx, f)
            assert e.value.status == qst.QST_E_TIMEOUT
        finally:
            qst.qst_inject_wait_timeout(qst.QST_INJECT_TC_LOADS, 0)
        qst.qst_set_params(ctx, _theta(N, t))
        assert [qst.qst_step(ctx, f)[0] for _ in range(2)] == want
    finally:
        qst.qst_destroy(ctx)
