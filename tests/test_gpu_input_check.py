"""The check of the frequencies on the GPU accepts and refuses what the rule says (finite, >= 0, sum within
1e-4 of 1), at sizes below, at and above one block's share, aligned and not, and for bad entries anywhere."""
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


def _accepts(f):
    v = f.astype(np.float64)
    return bool(np.all(np.isfinite(v)) and np.all(v >= 0) and abs(v.sum() - 1.0) <= 1e-4)


@pytest.mark.parametrize("prec,dt", [(qst.QST_FP32, np.float32), (qst.QST_FP64, np.float64)])
@pytest.mark.parametrize("N,offset", [(1, 0), (2, 1), (5, 0), (5, 3), (8, 0), (8, 1)])
def test_what_is_accepted_and_what_is_refused(N, offset, prec, dt):
    n = 4 ** N
    r = np.random.default_rng(N)
    good = r.random(n)
    good /= good.sum()
    cases = [good, good * 1.00009, good * 1.00011, good * 0.99989]
    for at, v in ((0, np.nan), (n - 1, np.inf), (n // 2, -np.inf), (n - 1, -1e-30), (0, -0.0)):
        c = good.copy()
        c[at] = v
        cases.append(c if v != 0 else c / c.sum())
    o = qst.qst_default_options()
    o.precision = prec
    ctx = qst.qst_init(N, opt=o)
    try:
        theta = torch.from_numpy(np.full(qst.qst_theta_size(N), 0.1, dt)).cuda()
        qst.qst_set_params(ctx, theta)
        buf = torch.zeros(n + offset, dtype=torch.float64 if prec == qst.QST_FP64 else torch.float32, device="cuda")
        f = buf[offset:]
        g = torch.empty_like(theta)
        for c in cases:
            c = c.astype(dt)
            f.copy_(torch.from_numpy(c))
            if _accepts(c):
                if offset == 0:  # an accepted f has to be aligned for the kernels' vector loads
                    qst.qst_loss_grad(ctx, theta, f, g)
                continue
            for call in (lambda: qst.qst_loss_grad(ctx, theta, f, g), lambda: qst.qst_step(ctx, f),
                         lambda: qst.qst_step(ctx, c)):
                with pytest.raises(qst.QstError) as e:
                    call()
                assert e.value.status == qst.QST_E_INPUT
        assert qst.qst_iterations(ctx) == 0
    finally:
        qst.qst_destroy(ctx)


@pytest.mark.parametrize("N", [4, 8])
def test_a_refused_input_between_two_steps_changes_nothing(N):
    n = 4 ** N
    r = np.random.default_rng(7)
    f = torch.from_numpy((lambda v: v / v.sum())(r.random(n)).astype(np.float32)).cuda()
    bad = (2 * f).contiguous()
    theta = torch.from_numpy((0.1 * r.standard_normal(qst.qst_theta_size(N))).astype(np.float32)).cuda()
    got = []
    for refuse in (False, True):
        ctx = qst.qst_init(N)
        try:
            qst.qst_set_params(ctx, theta)
            losses = []
            for k in range(4):
                losses.append(qst.qst_step(ctx, f)[0])
                if refuse and k == 1:
                    with pytest.raises(qst.QstError):
                        qst.qst_step(ctx, bad)
            got.append(losses)
        finally:
            qst.qst_destroy(ctx)
    assert got[0] == got[1]
