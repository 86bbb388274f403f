"""What users of this framework have it do, as cases that can be timed.

Each case is one pass through the public binding (``paper_2207_05341_gb300.qst``) with what a
program has in hand beforehand: frequencies of a simulated experiment on the GPU, initial network
parameters, a context on the program's own stream.  Kinds:

  train      ``qst_reconstruct``: a few iterations of the reconstruction loop (CUDA graph replay), then
             the density matrix, its loss and the parameters, as a loop does between two looks at the
             state.  The steps start small (a run resumed near its end): Rprop moves a parameter by its
             sign alone, so that an entry whose gradient is rounding noise about zero goes either way in
             any precision, and with the first steps of a new run those entries would say more about the
             rounding than the results do.  The work is the same.
  loss_grad  ``qst_loss_grad``: loss and full gradient for parameters the program holds itself
             (the autograd bridge, any optimiser of torch)
  probs      ``qst_probs``: Born probabilities of a density matrix under the product POVM
  batch      ``qst_batch_reconstruct``: many tomographies of mixed sizes, one graph launch an iteration
  counts     ``qst_sample_counts``: a simulated experiment's counts and frequencies
  fidelity   ``qst_state_fidelity``: fidelity of the current estimate with the target state

The expected values of ``exact`` are plain torch in 64 bits.
"""
import math

import torch

from paper_2207_05341_gb300 import qst

PRECISIONS = {"fp64": qst.QST_FP64, "fp32": qst.QST_FP32, "mixed": qst.QST_MIXED, "mixed_bf16": qst.QST_MIXED_BF16}
MAPS = {"chol_h": qst.QST_MAP_CHOL_H, "abs_p": qst.QST_MAP_ABS_P, "chol_delta": qst.QST_MAP_CHOL_DELTA}
NETS = {"fnn": qst.QST_NET_FNN, "cnn": qst.QST_NET_CNN}


def listed():
    return [
        # a two-minute tutorial size: one iteration is a few small kernels, so its latency is the cost
        {"name": "train_n4", "kind": "train", "N": 4, "precision": "fp32", "map": "chol_h", "net": "fnn",
         "iters": 1, "lr": 1e-6, "P": 2.0, "rank": 2, "shots": 100000},
        # the POVM map alone at the largest size of the paper (11 qubits)
        {"name": "probs_n11", "kind": "probs", "N": 11, "precision": "fp32", "rank": 4},
        # the reference precision, for checks and small studies
        {"name": "loss_grad_n7_fp64", "kind": "loss_grad", "N": 7, "precision": "fp64", "map": "chol_h",
         "net": "fnn", "P": 2.0, "rank": 8, "shots": 1000000},
        # training from torch at a mid size, in the default precision
        {"name": "loss_grad_n9", "kind": "loss_grad", "N": 9, "precision": "fp32", "map": "chol_h", "net": "fnn",
         "P": 2.0, "rank": 16, "shots": 1000000},
        # training from torch at the largest size of the paper, products on tensor cores
        {"name": "loss_grad_n11_mixed", "kind": "loss_grad", "N": 11, "precision": "mixed", "map": "chol_h",
         "net": "fnn", "P": 2.0, "rank": 1, "shots": 10000000},
        # the headline workload: 11 qubits, 10^7 shots, both precisions
        {"name": "train_n11_mixed", "kind": "train", "N": 11, "precision": "mixed", "map": "chol_h", "net": "fnn",
         "iters": 4, "lr": 1e-6, "P": 2.0, "rank": 1, "shots": 10000000},
        {"name": "train_n11_fp32", "kind": "train", "N": 11, "precision": "fp32", "map": "chol_h", "net": "fnn",
         "iters": 4, "lr": 1e-6, "P": 2.0, "rank": 1, "shots": 10000000},
        # the P-order absolute projection: an eigendecomposition in every iteration
        {"name": "train_n9_abs_p", "kind": "train", "N": 9, "precision": "fp32", "map": "abs_p", "net": "fnn",
         "iters": 2, "lr": 1e-6, "P": 1.5, "rank": 8, "shots": 1000000},
        # the convolutional mapping network
        {"name": "train_n10_cnn_mixed", "kind": "train", "N": 10, "precision": "mixed", "map": "chol_h",
         "net": "cnn", "iters": 4, "lr": 1e-6, "P": 2.0, "rank": 4, "shots": 10000000},
        # a study over many states: sizes 3 to 9 mixed, as the sweeps over states and ranks run them
        {"name": "batch_48", "kind": "batch", "B": 48, "Nmin": 3, "Nmax": 9, "precision": "fp32", "iters": 8,
         "lr": 1e-6, "sizes": 1, "shots": 100000},
        # a simulated experiment of the headline workload
        {"name": "counts_n11", "kind": "counts", "N": 11, "shots": 10000000, "rank": 1},
        # the estimate judged against its target, between iterations
        {"name": "fidelity_n10", "kind": "fidelity", "N": 10, "precision": "fp32", "w": 0.9, "shots": 10000000},
    ]


def draw(rng):
    """One more case of the same ranges; sizes are numbers of qubits, so the work is spread over its logarithm."""
    kind = rng.choice(["train", "train", "train", "loss_grad", "loss_grad", "probs", "batch", "counts", "fidelity"])
    shots = int(10 ** rng.uniform(4, 7))
    if kind == "probs":
        precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        N = rng.randint(1, 12 if precision == "fp32" else 10)
        return {"kind": kind, "N": N, "precision": precision, "rank": rng.randint(1, min(1 << N, 32))}
    if kind == "batch":
        lo = rng.randint(3, 6)
        return {"kind": kind, "B": int(round(2 ** rng.uniform(2, 5.9))), "Nmin": lo, "Nmax": rng.randint(lo, 9),
                "precision": rng.choice(["fp32", "mixed"]), "iters": rng.randint(1, 8), "lr": 1e-6,
                "sizes": rng.randrange(1 << 20), "shots": shots}
    if kind == "counts":
        return {"kind": kind, "N": rng.randint(3, 11), "shots": shots, "rank": rng.randint(1, 8)}
    if kind == "fidelity":
        return {"kind": kind, "N": rng.randint(3, 10), "precision": "fp32", "w": round(rng.uniform(0.5, 1.0), 3),
                "shots": shots}
    c = {"kind": kind, "net": "fnn", "map": "chol_h", "P": 2.0, "shots": shots}
    # a gradient through the eigendecomposition has the conditioning of its smallest gaps: trained, not compared
    form = rng.choice(["fp32", "fp32", "mixed", "mixed", "mixed_bf16", "cnn", "delta", "fp64"] +
                      (["abs_p", "abs_p"] if kind == "train" else []))
    c["precision"] = form if form in PRECISIONS else "fp32"
    if form in ("mixed", "mixed_bf16"):
        c["N"] = rng.randint(7, 11)
    elif form == "cnn":
        c["net"], c["N"] = "cnn", rng.randint(3, 10)
        if c["N"] >= 7 and rng.random() < 0.5:
            c["precision"] = "mixed"
    elif form == "abs_p":
        c["map"], c["P"], c["N"] = "abs_p", round(rng.uniform(1.0, 3.0), 2), rng.randint(3, 9)
    elif form == "delta":
        c["map"], c["N"] = "chol_delta", rng.randint(3, 10)
    elif form == "fp64":
        c["N"] = rng.randint(2, 8)
    else:
        c["N"] = rng.randint(2, 11)
    if kind == "train":
        c["iters"], c["lr"] = rng.randint(1, 4), 1e-6
    c["rank"] = rng.randint(1, min(1 << c["N"], 32))
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1))
    return g


def _complex_normal(shape, g):
    return torch.complex(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64),
                         torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))


def _target(N, rank, g):
    """A rank-r random state after a depolarising channel of strength 0.1, complex128."""
    d = 1 << N
    a = _complex_normal((d, rank), g)
    rho = a @ a.conj().T
    rho = 0.5 * (rho + rho.conj().T)
    rho = 0.9 * rho / rho.diagonal().real.sum()
    return rho + (0.1 / d) * torch.eye(d, device="cuda", dtype=rho.dtype)


def _povm():
    s = torch.tensor([[1, 1, 1], [-1, -1, 1], [-1, 1, -1], [1, -1, -1]], dtype=torch.float64) / math.sqrt(3.0)
    m = torch.zeros(4, 2, 2, dtype=torch.complex128)
    for a in range(4):
        x, y, z = s[a].tolist()
        m[a] = torch.tensor([[1 + z, complex(x, -y)], [complex(x, y), 1 - z]], dtype=torch.complex128) / 4
    return m.cuda()


def _born(X, N):
    """q_k = Tr[(M_k1 x ... x M_kN) X], one qubit after the other from the most significant."""
    M = _povm()
    t = X.reshape(1, 1 << N, 1 << N)
    for q in range(N):
        h = 1 << (N - q - 1)
        t = t.reshape(4 ** q, 2, h, 2, h)
        t = torch.einsum("aji,kixjy->kaxy", M, t).reshape(4 ** (q + 1), h, h)
    return t.reshape(-1).real


def _frequencies(N, rank, shots, g):
    """Counts of a simulated experiment over its total (Poisson counts about shots * P), float64."""
    P = _born(_target(N, rank, g), N).clamp_min(0.0)
    counts = torch.poisson((P * float(shots)).float(), generator=g).double()
    counts[0] += 1.0  # never empty
    return counts / counts.sum()


def _theta(N, net, g, dtype):
    """Uniform in +-1/sqrt(fan_in), in the library's layout."""
    n = 4 ** N

    def u(size, fan):
        return (torch.rand(size, generator=g, device="cuda", dtype=torch.float32) * 2 - 1) / math.sqrt(fan)
    if net == "cnn":
        H = 4 * N
        parts = [u(H * n, H), u(n, H), u(H * 640, 640), u(H, 640), u(90, 9), u(10, 9)]
    else:
        H = 2 * N
        parts = [u(H * n, n), u(H * n, H), u(n, H), u(H, n)]
    return torch.cat(parts).to(dtype)


def _real(precision):
    return torch.float64 if precision == "fp64" else torch.float32


def _inputs(case, seed):
    """The frequencies and initial parameters of a single tomography, in its precision."""
    g = _gen(seed)
    f = _frequencies(case["N"], case.get("rank", 1), case["shots"], g).to(_real(case["precision"]))
    return f, _theta(case["N"], case.get("net", "fnn"), g, _real(case["precision"]))


def _sizes(case):
    import random
    r = random.Random(case["sizes"])
    return [r.randint(case["Nmin"], case["Nmax"]) for _ in range(case["B"])]


def _batch_inputs(case, seed):
    got = []
    for b, N in enumerate(_sizes(case)):
        g = _gen(seed * 64 + b)
        rank = 1 + b % min(8, 1 << N)
        got.append((_frequencies(N, rank, case["shots"] * N, g).float(), _theta(N, "fnn", g, torch.float32)))
    return got


def _options(case):
    o = qst.qst_default_options()
    o.precision = PRECISIONS[case["precision"]]
    o.mapping = MAPS[case.get("map", "chol_h")]
    o.network = NETS[case.get("net", "fnn")]
    o.P = case.get("P", 2.0)
    o.lr = case.get("lr", o.lr)
    return o


class State:
    """What a program holds: buffers, a stream and a context that goes with it."""

    def __init__(self, case):
        self.case, self.ctx, self.batch = case, 0, 0

    def __del__(self):
        try:
            qst.qst_destroy(self.ctx)
            qst.qst_batch_destroy(self.batch)
        except Exception:  # at the interpreter's end
            pass


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "batch":
        sizes, got = _sizes(case), _batch_inputs(case, seed)
        s.stream = torch.cuda.Stream()
        s.f = [f for f, _ in got]
        s.rho = [torch.empty(1 << N, 1 << N, dtype=torch.complex64, device="cuda") for N in sizes]
        torch.cuda.synchronize()
        s.batch = qst.qst_batch_init(sizes, opt=_options(case), stream=s.stream.cuda_stream)
        for b, (_, theta) in enumerate(got):
            qst.qst_batch_set_params(s.batch, b, theta)
        torch.cuda.synchronize()
        return s
    N, d = case["N"], 1 << case["N"]
    if kind == "probs":
        cdt = torch.complex128 if case["precision"] == "fp64" else torch.complex64
        s.rho = _target(N, case["rank"], _gen(seed)).to(cdt).contiguous()
        s.p = torch.empty(4 ** N, dtype=_real(case["precision"]), device="cuda")
        s.ctx = qst.qst_init(N, opt=_options(case))
    elif kind == "counts":
        s.P = _born(_target(N, case["rank"], _gen(seed)), N).clamp_min(0.0).contiguous()
        s.seed = int(seed)
        s.counts = torch.empty(4 ** N, dtype=torch.int64, device="cuda")
        s.f = torch.empty(4 ** N, dtype=torch.float32, device="cuda")
        s.ctx = qst.qst_init(N)
    elif kind == "loss_grad":
        s.f, s.theta = _inputs(case, seed)
        s.dtheta = torch.empty_like(s.theta)
        s.ctx = qst.qst_init(N, opt=_options(case))
    elif kind == "fidelity":
        s.f, s.theta = _inputs(case, seed)
        s.psi = _complex_normal((d,), _gen(seed + 7)).to(torch.complex64)
        s.ctx = qst.qst_init(N, opt=_options(case))
        qst.qst_set_params(s.ctx, s.theta)
    else:
        s.f, s.theta = _inputs(case, seed)
        s.rho = torch.empty(d, d, dtype=torch.complex128 if case["precision"] == "fp64" else torch.complex64,
                            device="cuda")
        s.stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        s.ctx = qst.qst_init(N, opt=_options(case), stream=s.stream.cuda_stream)
        qst.qst_graph_enable(s.ctx, True)
        qst.qst_set_params(s.ctx, s.theta)
    torch.cuda.synchronize()
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "probs":
        qst.qst_probs(s.ctx, s.rho, s.p)
        return s.p
    if kind == "counts":
        qst.qst_sample_counts(s.ctx, s.P, s.case["shots"], s.seed, s.counts, s.f)
        return {"counts": s.counts, "f": s.f}
    if kind == "loss_grad":
        loss, _ = qst.qst_loss_grad(s.ctx, s.theta, s.f, s.dtheta)
        return {"loss": loss, "dtheta": s.dtheta}
    if kind == "fidelity":
        return qst.qst_state_fidelity(s.ctx, s.f, s.psi, s.case["w"])
    if kind == "batch":
        losses = qst.qst_batch_reconstruct(s.batch, s.f, s.case["iters"], s.rho)
        return {"losses": torch.tensor(losses, dtype=torch.float32), "rho": s.rho}
    loss, _ = qst.qst_reconstruct(s.ctx, s.f, s.case["iters"], s.rho)
    qst.qst_get_params(s.ctx, s.theta)
    return {"loss": loss, "rho": s.rho, "theta": s.theta}


# ---------------------------------------------------------------- work
def _tomography(N, r, net, mapping, train):
    """(bytes, flops) of one loss and gradient; train: of one iteration with Rprop."""
    n, d = 4 ** N, 2 ** N
    P = 4 * N * n + n + 4 * N * 640 if net == "cnn" else 4 * N * n + n + 2 * N
    # gradient: parameters read, gradient written.  Rprop: parameters and step words read and written.
    moved = r * ((4 if train else 2) * P + n)
    # chol_h: X = T T (Hermitian) and G T; chol_delta: triangular factors; abs_p: an eigendecomposition
    # (4/3 + 2 complex products to reduce and rotate), X and the four products around its derivative
    matrix = {"chol_h": 12, "chol_delta": 4, "abs_p": 8 * 3.4 + 4 + 32}[mapping] * d ** 3
    return moved, matrix + 8 * P + 6 * N * n


def work(case):
    kind, N = case["kind"], case.get("N", 0)
    n, d = 4 ** N, 2 ** N
    r = 8 if case.get("precision") == "fp64" else 4
    if kind == "probs":  # the lower triangle read, p written
        return {"bytes": 2.0 * n * r, "flops": 3.0 * N * n}
    if kind == "counts":  # P read, counts and frequencies written
        return {"bytes": 20.0 * n, "flops": 2.0 * n}
    if kind == "fidelity":  # the output layer read for T; T reduced to its eigenvalues
        return {"bytes": 4.0 * n * (2 * N + 1), "flops": 8 * (4 / 3) * d ** 3 + 4.0 * N * n}
    if kind == "loss_grad":
        b, f = _tomography(N, r, case["net"], case["map"], False)
        return {"bytes": float(b), "flops": float(f)}
    one = [(N, case.get("net", "fnn"), case.get("map", "chol_h"))] if kind == "train" else \
        [(N, "fnn", "chol_h") for N in _sizes(case)]
    total = {"bytes": 0.0, "flops": 0.0}
    for N, net, mapping in one:
        b, f = _tomography(N, r, net, mapping, True)
        n, d = 4 ** N, 2 ** N
        H = 4 * N if net == "cnn" else 2 * N
        # after the iterations: the output layer read for the final state, rho written, the parameters copied out
        out = 2 * r * (4 * N * n + n) if kind == "train" else 0
        total["bytes"] += case["iters"] * b + r * (H + 1) * n + 2 * r * n + out
        total["flops"] += case["iters"] * f + 4 * d ** 3 + 2 * H * n + 3 * N * n
    return total


# ---------------------------------------------------------------- expected values in 64 bits
def _output_matrix(t, d, lower):
    R = t.reshape(d, d)
    low = torch.tril(R, -1)
    im = torch.triu(R, 1).T
    diag = torch.diag(R.diagonal())
    if lower:
        return torch.complex(low + diag, im.contiguous())
    return torch.complex(low + low.T + diag, im - im.T)


def _network(theta, f, N, net):
    n = 4 ** N
    if net == "cnn":
        H, d = 4 * N, 2 ** N
        w2, b2, w1, b1, cw, cb = torch.split(theta, [H * n, n, H * 640, H, 90, 10])
        img = torch.nn.functional.conv2d(f.reshape(1, 1, d, d), cw.reshape(10, 1, 3, 3), cb, padding=1)
        feat = torch.nn.functional.max_pool2d(torch.relu(img), max(1, d // 8)).reshape(-1)
        h = torch.nn.functional.leaky_relu(w1.reshape(H, 640) @ feat + b1, 0.01)
        return h @ w2.reshape(H, n) + b2
    H = 2 * N
    w1, w2, b2, b1 = torch.split(theta, [H * n, H * n, n, H])
    h = torch.nn.functional.leaky_relu(w1.reshape(H, n) @ f + b1, 0.01)
    return h @ w2.reshape(H, n) + b2


def _state(t, N, mapping, P):
    """X of the state map, unnormalised."""
    T = _output_matrix(t, 1 << N, mapping == "chol_delta")
    if mapping == "chol_delta":
        return T.conj().T @ T
    if mapping == "abs_p":
        lam, Q = torch.linalg.eigh(T)
        return (Q * lam.abs().pow(P)) @ Q.conj().T
    return T @ T


def _loss(theta, f, N, net, mapping, P):
    X = _state(_network(theta, f, N, net), N, mapping, P)
    p = _born(X, N) / X.diagonal().real.sum()
    seen = f > 0
    return -(f[seen] * torch.log(p[seen])).sum(), X


def _loss_grad(theta, f, N, net, mapping, P):
    theta = theta.detach().requires_grad_(True)
    loss, _ = _loss(theta, f, N, net, mapping, P)
    (g,) = torch.autograd.grad(loss, theta)
    return loss.detach(), g


def _train(theta, f, N, net, mapping, P, iters, lr):
    step, before = torch.full_like(theta, lr), torch.zeros_like(theta)
    for _ in range(iters):
        g = _loss_grad(theta, f, N, net, mapping, P)[1]
        same = g * before
        step = torch.where(same > 0, (step * 1.2).clamp(max=50.0), torch.where(same < 0, (step * 0.5).clamp(min=1e-6), step))
        before = torch.where(same < 0, torch.zeros_like(g), g)
        theta = theta - torch.sign(before) * step
    with torch.no_grad():
        loss, X = _loss(theta, f, N, net, mapping, P)
    return loss, X / X.diagonal().real.sum(), theta


def exact(case, seed):
    kind = case["kind"]
    if kind == "counts":
        return None
    if kind == "batch":
        losses, rhos = [], []
        for N, (f, theta) in zip(_sizes(case), _batch_inputs(case, seed)):
            loss, rho, _ = _train(theta.double(), f.double(), N, "fnn", "chol_h", 2.0, case["iters"], case["lr"])
            losses.append(loss)
            rhos.append(rho)
        return {"losses": torch.stack(losses), "rho": rhos}
    N = case["N"]
    if kind == "probs":
        cdt = torch.complex128 if case["precision"] == "fp64" else torch.complex64
        rho = _target(N, case["rank"], _gen(seed)).to(cdt).to(torch.complex128)
        low = torch.tril(rho, -1)
        return _born(low + low.conj().T + torch.diag(rho.diagonal()), N)
    f, theta = (x.double() for x in _inputs(case, seed))
    if kind == "fidelity":
        T = _output_matrix(_network(theta, f, N, "fnn"), 1 << N, False)
        lam, Q = torch.linalg.eigh(T)
        root = (Q * lam.abs()) @ Q.conj().T / lam.square().sum().sqrt()
        psi = _complex_normal((1 << N,), _gen(seed + 7)).to(torch.complex64).to(torch.complex128)
        psi = psi / psi.abs().square().sum().sqrt()
        w, d = case["w"], 1 << N
        lo, hi = math.sqrt((1 - w) / d), math.sqrt(w + (1 - w) / d)
        other = lo * root + (hi - lo) * torch.outer(root @ psi, psi.conj())
        return float(torch.linalg.svdvals(other).sum() ** 2)
    if kind == "loss_grad":
        loss, g = _loss_grad(theta, f, N, case["net"], case["map"], case["P"])
        return {"loss": float(loss), "dtheta": g}
    loss, rho, theta = _train(theta, f, N, case["net"], case["map"], case["P"], case["iters"], case["lr"])
    return {"loss": float(loss), "rho": rho, "theta": theta}
