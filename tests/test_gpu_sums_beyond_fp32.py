"""The sums over the 4^N axis carry FP32's terms beyond FP32's range, as FP64 sums do: hidden gradients dh = sum_i W2_i dt_i
whose partial sums (not their terms) exceed the largest FP32 number.  Where the whole sum does too the gradient is
infinite with the right sign, and an Rprop step moves the parameter; where the sum cancels it is finite and right.

W1 and b1 are 0, so that h = 0 and t = b2 whatever W2 is (and LeakyReLU's slope is 0.01); rows 0 and 1 of W2 are A and
-A, A about 1e37 with the signs of dL/dt, taken from a call with W2 = 0.  Tolerance of the finite case: FP32 partial sums of at most 64 terms a thread."""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BIG = np.float32(1e37)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qst.load()


class Net:
    """Offsets of the parameters used here."""

    def __init__(self, N, net):
        n = 4 ** N
        H = 4 * N if net == qst.QST_NET_CNN else 2 * N
        self.size, self.n = qst.qst_theta_size_net(N, net), n
        if net == qst.QST_NET_CNN:  # W2^T, b2, W1, b1, convolution
            self.w2, self.b2, self.b1 = 0, H * n, H * n + n + H * 640
        else:  # W1, W2^T, b2, b1
            self.w2, self.b2, self.b1 = H * n, 2 * H * n, 2 * H * n + n


def _grad(ctx, theta, f):
    g = torch.empty(theta.size, device="cuda")
    qst.qst_loss_grad(ctx, torch.from_numpy(theta).cuda(), f, g)
    return g.cpu().numpy()


def _theta(ctx, p, f, cancel):
    """(theta, A): parameters whose dh_0 = -dh_1 = sum A dt."""
    b2 = np.random.default_rng(p.n).standard_normal(p.n).astype(np.float32)
    theta = np.zeros(p.size, np.float32)
    theta[p.b2:p.b2 + p.n] = b2
    dt = _grad(ctx, theta, f)[p.b2:p.b2 + p.n]
    theta[p.b2:p.b2 + p.n] *= np.float32(2.0 * np.abs(dt).mean())  # dL/dt goes as 1 / t: 0.5 on average then
    dt = _grad(ctx, theta, f)[p.b2:p.b2 + p.n]
    A = BIG * np.sign(dt)
    if cancel:
        a = np.abs(dt.astype(np.float64))
        A[p.n // 2:] *= np.float32(-a[:p.n // 2].sum() / a[p.n // 2:].sum())
    theta[p.w2:p.w2 + p.n] = A
    theta[p.w2 + p.n:p.w2 + 2 * p.n] = -A
    return theta, A.astype(np.float64)


CASES = [(4, qst.QST_NET_FNN), (6, qst.QST_NET_FNN), (7, qst.QST_NET_FNN), (8, qst.QST_NET_FNN), (4, qst.QST_NET_CNN),
         (7, qst.QST_NET_CNN)]


def _context(N, net):
    o = qst.qst_default_options()
    o.network, o.lr = net, 1e-3
    f = np.random.default_rng(N).dirichlet(np.full(4 ** N, 5.0)).astype(np.float32)
    return qst.qst_init(N, opt=o), torch.from_numpy(f).cuda()


@pytest.mark.parametrize("N,net", CASES)
def test_gradient(N, net):
    p = Net(N, net)
    ctx, f = _context(N, net)
    try:
        theta, _ = _theta(ctx, p, f, False)
        g = _grad(ctx, theta, f)
        assert np.isfinite(g[p.b2:p.b2 + p.n]).all()
        assert g[p.b1] == np.inf and g[p.b1 + 1] == -np.inf
        theta, A = _theta(ctx, p, f, True)
        g = _grad(ctx, theta, f).astype(np.float64)
        terms = 0.01 * A * g[p.b2:p.b2 + p.n]
        for j, sign in ((0, 1.0), (1, -1.0)):
            assert abs(g[p.b1 + j] - sign * terms.sum()) <= 64 * 2.0 ** -24 * np.abs(terms).sum()
    finally:
        qst.qst_destroy(ctx)


@pytest.mark.parametrize("N,net", CASES)
def test_step(N, net):
    p = Net(N, net)
    ctx, f = _context(N, net)
    try:
        theta, _ = _theta(ctx, p, f, False)
        qst.qst_set_params(ctx, theta)
        qst.qst_step(ctx, f)
        after = np.empty_like(theta)
        qst.qst_get_params(ctx, after)
        assert after[p.b1] == np.float32(-1e-3) and after[p.b1 + 1] == np.float32(1e-3)
    finally:
        qst.qst_destroy(ctx)


@pytest.mark.parametrize("N,net", CASES)
def test_infinite_terms(N, net):
    """Terms that overflow themselves: the sums are infinite, not NaN, and the step moves."""
    p = Net(N, net)
    ctx, f = _context(N, net)
    try:
        theta, A = _theta(ctx, p, f, False)
        A = (A / BIG * 3e38).astype(np.float32)
        theta[p.b2:p.b2 + p.n] *= np.float32(2.0 ** -4)  # |dL/dt| 8 on average
        theta[p.w2:p.w2 + p.n], theta[p.w2 + p.n:p.w2 + 2 * p.n] = A, -A
        g = _grad(ctx, theta, f)
        assert g[p.b1] == np.inf and g[p.b1 + 1] == -np.inf
        qst.qst_set_params(ctx, theta)
        qst.qst_step(ctx, f)
        after = np.empty_like(theta)
        qst.qst_get_params(ctx, after)
        assert after[p.b1] == np.float32(-1e-3) and after[p.b1 + 1] == np.float32(1e-3)
    finally:
        qst.qst_destroy(ctx)
