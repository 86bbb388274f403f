"""Draws through the guide table against the oracle's integer sampler, count by count: distributions that put one,
few or all outcomes into a bucket, shots around the sizes where the table starts and changes its number of
buckets, total weights that are powers of two and one off, P and counts off 16-byte alignment, weights of every
binary exponent, and counts past the table of quotients."""
import numpy as np
import pytest

import oracle as O
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


def _distribution(kind, n, r):
    p = np.zeros(n)
    if kind == "one":
        p[n // 3] = 1.0
    elif kind == "uniform":
        p[:] = 1.0 / n
    elif kind == "first":
        p[0], p[1:] = 0.9, 0.1 / (n - 1)
    elif kind == "last":
        p[-1], p[:-1] = 0.9, 0.1 / (n - 1)
    elif kind == "exponents":
        p = 2.0 ** -r.integers(1, 60, n).astype(float) * r.random(n)
        p[::7] = -p[::7]
        p[1::7] = 0.0
    elif kind == "half":
        p[n // 2:] = r.random(n - n // 2)
        p /= p.sum()
    elif kind == "above":
        p[:] = 2.0 ** -52
        p[0] += 0.5
    return p


@pytest.mark.parametrize("kind", ["one", "uniform", "first", "last", "exponents", "half", "above"])
@pytest.mark.parametrize("N,shots,offset", [(1, 5000, 0), (3, 4095, 0), (3, 4096, 1), (5, 100000, 1), (6, 16384, 0),
                                            (7, 300001, 0), (5, 1 << 19, 0), (6, (1 << 19) - 1, 0), (6, 1 << 19, 1),
                                            (7, 600001, 0), (9, 1 << 20, 1)])
def test_counts_equal_the_oracle(kind, N, shots, offset):
    n = 4 ** N
    P = _distribution(kind, n, np.random.default_rng(N + shots))
    ctx = qst.qst_init(N)
    try:
        pd = torch.zeros(n + offset, dtype=torch.float64, device="cuda")[offset:]
        pd.copy_(torch.from_numpy(P))
        counts = torch.empty(n + offset, dtype=torch.int64, device="cuda")[offset:]
        f = torch.empty(n, device="cuda")
        qst.qst_sample_counts(ctx, pd, shots, 17, counts, f)
        want = O.multinomial_counts_integer(P, shots, 17)
        assert np.array_equal(counts.cpu().numpy(), want)
        assert np.array_equal(f.cpu().numpy(), (want / shots).astype(np.float32))
    finally:
        qst.qst_destroy(ctx)


@pytest.mark.parametrize("N,total", [(6, 0.9995 * 4**6), (6, 0.9999 * 4**6), (6, 2048.0), (6, 2047.0), (7, 4000.0),
                                     (9, 4095.5)])
def test_total_weights_up_to_64_bits(N, total):
    """P need not sum to 1: total weights of 63 and 64 bits (sums from 2^10 to below 2^12)."""
    n, shots = 4 ** N, 1 << 19
    P = np.full(n, total / n)
    if N == 9:
        P *= np.random.default_rng(N).random(n) * 2.0
        P *= total / P.sum()
    assert P.max() <= 1.0
    ctx = qst.qst_init(N)
    try:
        counts = torch.empty(n, dtype=torch.int64, device="cuda")
        qst.qst_sample_counts(ctx, torch.from_numpy(P).cuda(), shots, 23, counts)
        assert np.array_equal(counts.cpu().numpy(), O.multinomial_counts_integer(P, shots, 23))
    finally:
        qst.qst_destroy(ctx)
