"""The ordering of the Jacobi sweeps without eigenvectors (host only): every round m = 1 .. d - 1 once per sweep, the
subspace bases in the reduced form that the kernels' coset numbering takes (pivot bits distinct, ascending, clear in the
other vectors), passes of the sizes that the kernels have, and A_P's order where the partition is the same."""
import os

import numpy as np
import pytest

from paper_2207_05341_gb300 import qst

PASSES = {9: 41, 10: 73, 11: 145}  # other N: the order of QST_MAP_ABS_P


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not os.path.exists(qst.LIB_PATH):
        from paper_2207_05341_gb300 import build
        build.build()
    qst.load()


@pytest.mark.parametrize("N", list(range(1, 13)))
def test_every_round_once(N):
    d, sched = 1 << N, qst.qst_jacobi_values_schedule(N)
    if N in PASSES:
        assert len(sched) == PASSES[N]
    else:
        assert sched == qst.qst_jacobi_schedule(N)
    assert len(sched) % 2 == 1
    seen = np.zeros(d, dtype=int)
    for basis in sched:
        assert len(basis) in ((1, 2) if N <= 5 else (2, 3, 4) if N == 9 else (3, 4))
        tops = [v.bit_length() - 1 for v in basis]
        assert tops == sorted(set(tops))
        span = [0]
        for i, v in enumerate(basis):
            assert 0 < v < d and all(not (v >> t) & 1 for k, t in enumerate(tops) if k != i)
            span += [x ^ v for x in span]
        for m in span[1:]:
            seen[m] += 1
    assert seen[0] == 0 and np.all(seen[1:] == 1)


def test_arguments():
    for N in (0, 13):
        with pytest.raises(qst.QstError):
            qst.qst_jacobi_values_schedule(N)
