"""The float prior and gradient step on sums of two floats, against the same
formulas in extended precision (numpy longdouble): values over many orders of
magnitude, cancellations, exact zeros, denormals, infinities, odd grids.

Tolerance: the inputs and outputs are float and the working precision is 2^-45
or better relative to a result that has not cancelled by more than 2^16, so
each output is the correctly rounded one, or its neighbour on a near tie: half
a unit in the last place plus 1 %.  The prior's value is an FP64 sum: 1e-13.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


def _ulps(got, want):
    """|got - want| in units of the last place of the float nearest to want."""
    want = np.asarray(want, np.longdouble)
    u = np.spacing(np.maximum(np.abs(want.astype(np.float32)), np.finfo(np.float32).tiny)).astype(np.longdouble)
    return np.abs(np.asarray(got, np.longdouble) - want) / u


def _prior(x, shape, beta):
    x = x.reshape(shape).astype(np.longdouble)
    g, v = np.zeros_like(x), np.longdouble(0)
    for a in range(3):
        d = np.diff(x, axis=a)
        v += (d * d).sum()
        lo, hi = [slice(None)] * 3, [slice(None)] * 3
        lo[a], hi[a] = slice(0, -1), slice(1, None)
        g[tuple(hi)] += d
        g[tuple(lo)] -= d
    return (np.longdouble(beta) * g).reshape(-1), 0.5 * np.longdouble(beta) * v


IMAGES = {
    "smooth": lambda r, n: 100 + np.cumsum(r.uniform(-1e-3, 1e-3, n)),
    "rough": lambda r, n: 10.0 ** r.uniform(-6, 6, n),
    "wide": lambda r, n: 10.0 ** r.uniform(-30, 14, n) * (r.random(n) < 0.7),
    "flat": lambda r, n: np.full(n, 0.1),
    "tiny": lambda r, n: 10.0 ** r.uniform(-41, -28, n),
}


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 300), (5, 7, 3), (33, 29, 31)])
@pytest.mark.parametrize("image", list(IMAGES))
@pytest.mark.parametrize("beta", [7e-7, 0.3, 1e-30])
def test_prior(mc, shape, image, beta):
    import torch
    n = int(np.prod(shape))
    x = IMAGES[image](np.random.default_rng(n), n).astype(np.float32)
    want_g, want_v = _prior(x, shape, beta)
    xd = torch.as_tensor(x).cuda()
    g = torch.empty(n, dtype=torch.float32, device="cuda")
    v = torch.empty(1, dtype=torch.float64, device="cuda")
    for gg, vv in ((g, v), (g, None), (None, v)):
        mc.mc_prior_quadratic(shape, beta, xd, gg, vv)
    assert _ulps(g.cpu().numpy(), want_g).max() <= 0.505
    assert abs(v.item() - float(want_v)) <= 1e-13 * float(want_v)


@pytest.mark.parametrize("alpha", [1.0, 0.5, 0.125, 2.0 ** -19, 1.7, 30.0])
@pytest.mark.parametrize("prior", [False, True])
def test_pgd_step(mc, alpha, prior):
    import torch
    rng = np.random.default_rng(7)
    n = 40_000
    s = 10.0 ** rng.uniform(-4, 3, n)
    s[::17] = 0.0
    s[5::1001] = 10.0 ** rng.uniform(-60, 60, len(s[5::1001]))
    x = (10.0 ** rng.uniform(-8, 6, n)).astype(np.float32)
    x[::13] = 0.0
    x[7::101] = (10.0 ** rng.uniform(-44, -20, len(x[7::101]))).astype(np.float32)
    bp = (s * rng.uniform(0, 2, n)).astype(np.float32)
    bp[3::11] = s[3::11].astype(np.float32)  # steps of almost nothing
    gp = (s * rng.uniform(-1, 1, n) * (rng.random(n) < 0.9)).astype(np.float32) if prior else None
    xd = torch.as_tensor(x).cuda()
    mc.mc_pgd_step(alpha, torch.as_tensor(s).cuda(), torch.as_tensor(bp).cuda(), xd,
                   torch.as_tensor(gp).cuda() if prior else None)
    sl, xl = s.astype(np.longdouble), x.astype(np.longdouble)
    with np.errstate(divide="ignore", invalid="ignore"):
        grad = sl - bp.astype(np.longdouble) + (gp.astype(np.longdouble) if prior else 0)
        want = np.where(sl > 0, np.maximum(xl - np.longdouble(alpha) * (xl / sl) * grad, 0), 0)
    got = xd.cpu().numpy()
    # a result that has cancelled below x 2^-16 comes from the FP64 formula,
    # whose error is that of its terms
    slack = np.where(want < xl * 2.0 ** -16, 1e-15 * np.longdouble(alpha + 1) * xl * (1 + np.abs(grad) / np.where(sl > 0, sl, 1)), 0)
    with np.errstate(all="ignore"):  # equal infinities, and sums too large for a float, have no distance
        ok = (got == want.astype(np.float32)) | (_ulps(got, want) <= 0.505)
        ok |= np.abs(got.astype(np.longdouble) - want) <= slack + 1e-45
        ok |= np.isnan(want)  # infinity times zero: see test_not_finite
    bad = np.flatnonzero(~ok)
    assert len(bad) == 0, [(s[i], x[i], bp[i], gp[i] if prior else 0, got[i], want[i]) for i in bad[:5]]


def test_not_finite(mc):
    """Infinities and NaN take the FP64 formulas' way."""
    import torch
    inf, nan = np.inf, np.nan
    s = np.array([1.0, 1.0, 1.0, 1.0, inf, nan, -1.0, 1.0])
    x = np.array([1.0, inf, nan, 1.0, 1.0, 1.0, 1.0, 0.0], np.float32)
    bp = np.array([inf, 1.0, 1.0, nan, 1.0, 1.0, 1.0, 5.0], np.float32)
    xd = torch.as_tensor(x).cuda()
    mc.mc_pgd_step(1.0, torch.as_tensor(s).cuda(), torch.as_tensor(bp).cuda(), xd)
    with np.errstate(all="ignore"):
        xn = x.astype(np.float64) - (x / s) * (s - bp)
        want = np.where((s > 0) & (xn > 0), xn, 0).astype(np.float32)
    assert np.array_equal(xd.cpu().numpy(), want)
    img = np.ones((3, 4, 5), np.float32)
    img[1, 2, 3], img[0, 0, 0] = np.inf, np.nan
    g = torch.empty(60, dtype=torch.float32, device="cuda")
    v = torch.empty(1, dtype=torch.float64, device="cuda")
    mc.mc_prior_quadratic((3, 4, 5), 0.5, torch.as_tensor(img).cuda().reshape(-1), g, v)
    with np.errstate(all="ignore"):
        want_g, want_v = _prior(img, (3, 4, 5), 0.5)
    got = g.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want_g.astype(np.float32)))
    assert np.array_equal(got[~np.isnan(got)], want_g.astype(np.float32)[~np.isnan(got)])
    assert np.isnan(v.item())
