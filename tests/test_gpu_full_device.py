"""A device with little memory left: the operand planes of the FP32 products, which a context can do without, leave room
for the scratch that calls allocate on first use, so that a context that fits has all its calls."""
import numpy as np
import pytest

from paper_2207_05341_gb300 import qst, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 11
MB = 1 << 20


def _calls(ctx, f, psi, P, counts):
    qst.qst_set_params(ctx, synth.init_theta(N, 3).astype(np.float32))
    qst.qst_sample_counts(ctx, P, 1 << 20, 5, counts)
    qst.qst_classical_fidelity(ctx, f, P, samples=1000, seed=1)
    return qst.qst_classical_fidelity(ctx, f, P), qst.qst_state_fidelity(ctx, f, psi, 0.9)


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_first_use_scratch_after_init_on_a_nearly_full_device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, d = 4 ** N, 1 << N
    f = torch.full((n,), 1.0 / n, device="cuda")
    P = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    counts = torch.empty(n, dtype=torch.int64, device="cuda")
    psi = torch.zeros(d, dtype=torch.complex64, device="cuda")
    psi[0] = 1.0
    f0 = _free()
    ctx = qst.qst_init(N)
    f1 = _free()
    want = _calls(ctx, f, psi, P, counts)  # every kernel is loaded now
    f2 = _free()
    qst.qst_destroy(ctx)
    planes, first_use = 30 * n, f1 - f2
    assert planes > 100 * MB and first_use > 100 * MB
    spare = (f0 - f1) - planes + first_use + 64 * MB  # all but the planes, and some
    fill = torch.empty(_free() - spare, dtype=torch.uint8, device="cuda")
    try:
        ctx = qst.qst_init(N)
        try:
            got = _calls(ctx, f, psi, P, counts)
        finally:
            qst.qst_destroy(ctx)
    finally:
        del fill
        torch.cuda.empty_cache()
    # the same results, to the rounding of the products on the CUDA cores
    assert np.allclose(got, want, rtol=1e-4)
