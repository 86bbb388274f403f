"""State fidelity at the sizes whose sweeps without eigenvectors use their own partition of the rounds (9 <= N <= 11):
FP64 against the oracle to the 1e-9 of the other FP64 sizes.  16 sweeps: a round that the partition missed would leave
its entries off the diagonal, however many sweeps run."""
import numpy as np
import pytest

import oracle as O
from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [9, 10])
def test_values_partition_fp64(N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    psi = synth.haar_pure(N, 500 + N)
    P = O.born_probabilities(synth.depolarized(psi, 0.1), O.tetrahedral_povm()).real
    f = synth.frequencies(synth.multinomial_counts(P, 10**5, 510 + N))
    theta = synth.init_theta(N, 520 + N)
    o = qst.qst_default_options()
    o.precision = qst.QST_FP64
    ctx = qst.qst_init(N, opt=o)
    try:
        qst.qst_set_params(ctx, theta)
        got = qst.qst_state_fidelity(ctx, torch.from_numpy(f).cuda(), torch.from_numpy(psi).cuda(), 0.9, sweeps=16)
    finally:
        qst.qst_destroy(ctx)
    want = O.fidelity(O.state_from_theta(theta, f, N, mapping="chol_h", P=2.0, network="fnn", decision=np.float64),
                      O.noisy_target(psi, 0.9))
    assert abs(got - want) < 1e-9, (got, want)
