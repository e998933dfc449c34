"""The float prior's gradient and the gradient step are no further from the
exact results than the FP64 formulas rounded to float once, element by element:
where the sums of two floats leave the rounding open, the kernel takes the FP64
formula itself.  Large images with differences that nearly cancel, where 45
bits before the last rounding would show.

The FP64 formulas are restated in numpy, rounded where the kernels round: the
step's last product and sum are one fused operation (formed in extended
precision here, which holds the product of two doubles on the machines these
tests run on).
"""
import numpy as np
import pytest

from tests.test_gpu_two_float import _prior

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


def _no_further(got, formula, want):
    err = np.abs(got.astype(np.longdouble) - want)
    bad = np.flatnonzero(~((got == formula) | (err <= np.abs(formula.astype(np.longdouble) - want))))
    assert len(bad) == 0, (len(bad), got[bad[:4]], formula[bad[:4]], want[bad[:4]])


def _gradient_f64(x, shape, beta):
    nz, ny, nx = shape
    x = x.reshape(nz, ny, nx).astype(np.float64)
    g = np.zeros_like(x)
    g[:, :, 1:] += x[:, :, 1:] - x[:, :, :-1]
    g[:, :, :-1] += x[:, :, :-1] - x[:, :, 1:]
    g[:, 1:] += x[:, 1:] - x[:, :-1]
    g[:, :-1] += x[:, :-1] - x[:, 1:]
    g[1:] += x[1:] - x[:-1]
    g[:-1] += x[:-1] - x[1:]
    return (beta * g).reshape(-1).astype(np.float32)


def _ramps(shape, bend, rng):
    """Steep in all directions, slightly bent: neighbours' differences cancel."""
    z, y, x = np.meshgrid(*(np.arange(k, dtype=np.float64) for k in shape), indexing="ij")
    img = 300 + 2.7 * x + 1.3 * y + 0.9 * z + bend * (0.5 * x * x - 0.3 * y * y + 0.1 * z * z)
    return (img * (1 + bend * 1e-3 * rng.uniform(-1, 1, shape))).reshape(-1).astype(np.float32)


@pytest.mark.parametrize("bend", [1e-1, 1e-2, 1e-3])
@pytest.mark.parametrize("value", [False, True])
def test_prior_gradient(mc, bend, value):
    import torch
    shape, beta = (96, 101, 103), 7.3e-3
    x = _ramps(shape, bend, np.random.default_rng(5))
    g = torch.empty(len(x), dtype=torch.float32, device="cuda")
    v = torch.empty(1, dtype=torch.float64, device="cuda") if value else None
    mc.mc_prior_quadratic(shape, beta, torch.as_tensor(x).cuda(), g, v)
    _no_further(g.cpu().numpy(), _gradient_f64(x, shape, beta), _prior(x, shape, beta)[0])


@pytest.mark.parametrize("alpha", [1.0, 0.5, 2.0 ** -7, 1.9])
@pytest.mark.parametrize("left", [1.0, 1e-3, 1e-4])
def test_step(mc, alpha, left):
    """`left` of the voxel's value is what the step leaves of it."""
    import torch
    rng = np.random.default_rng(6)
    n = 1_000_003
    s = 10.0 ** rng.uniform(-4, 3, n)
    x = (10.0 ** rng.uniform(-3, 5, n)).astype(np.float32)
    gp = (s * rng.uniform(-0.5, 0.5, n)).astype(np.float32)
    # (1 - alpha) + alpha (bp - gp) / s is about left
    bp = (s * (1 - (1 - left * rng.uniform(0.5, 2, n)) / alpha) + gp).astype(np.float32)
    xd = torch.as_tensor(x).cuda()
    mc.mc_pgd_step(alpha, torch.as_tensor(s).cuda(), torch.as_tensor(bp).cuda(), xd, torch.as_tensor(gp).cuda())
    grad = s - bp.astype(np.float64) + gp.astype(np.float64)
    L = np.longdouble
    t = alpha * (x.astype(np.float64) / s)
    formula = np.maximum((x.astype(L) - t.astype(L) * grad.astype(L)).astype(np.float64), 0).astype(np.float32)
    want = np.maximum(x.astype(L) - L(alpha) * (x.astype(L) / s.astype(L)) * (s.astype(L) - bp.astype(L) + gp.astype(L)), 0)
    _no_further(xd.cpu().numpy(), formula, want)
