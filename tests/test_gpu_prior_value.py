"""The float prior's value is an FP64 sum: against extended precision, one
pair of voxels at a time and over whole images, alone and together with the
gradient, whose accuracy is checked in each of the calls.

Tolerance of a pair: roundings of the difference (counted twice in its
square), of the square and of the product with beta / 2: 4 * 2^-53.  Of an image
of n voxels, all terms positive: a thread's chain of n / 256 * 3 sums at most,
ten more in its block, ten over the blocks: (4 + 3 n / 256 + 20) 2^-53.  The
gradient: correctly rounded, or the neighbour on a near tie: 0.505 units in the
last place, as in test_gpu_two_float.py.
"""
import numpy as np
import pytest

from tests.test_gpu_two_float import IMAGES, _prior, _ulps

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


@pytest.mark.parametrize("with_gradient", [False, True])
def test_pairs(mc, with_gradient):
    import torch
    rng = np.random.default_rng(3)
    k, beta = 400, 0.3
    x = (10.0 ** rng.uniform(-4, 4, (k, 2))).astype(np.float32)
    x[::7, 1] = 0.0
    x[3::50] = (10.0 ** rng.uniform(-44, -36, x[3::50].shape)).astype(np.float32)
    xd = torch.as_tensor(x).cuda()
    v = torch.empty(k, dtype=torch.float64, device="cuda")
    g = torch.empty(2, dtype=torch.float32, device="cuda")
    for i in range(k):
        mc.mc_prior_quadratic((1, 1, 2), beta, xd[i], g if with_gradient else None, v[i:i + 1])
    d = x[:, 0].astype(np.longdouble) - x[:, 1]
    want = np.longdouble(beta) / 2 * d * d
    err = np.abs(v.cpu().numpy() - want)
    assert np.all(err <= 4 * U * want + 1e-300), (err / want).max()


@pytest.mark.parametrize("shape", [(1, 1, 300), (5, 7, 3), (33, 29, 31), (64, 64, 65)])
@pytest.mark.parametrize("image", list(IMAGES))
@pytest.mark.parametrize("beta", [7e-7, 0.3])
def test_each_call(mc, shape, image, beta):
    """Gradient and value together, and each alone, into fresh outputs."""
    import torch
    n = int(np.prod(shape))
    x = IMAGES[image](np.random.default_rng(n + 1), n).astype(np.float32)
    want_g, want_v = _prior(x, shape, beta)
    xd = torch.as_tensor(x).cuda()
    for with_g, with_v in ((True, True), (True, False), (False, True)):
        g = torch.full((n,), float("nan"), dtype=torch.float32, device="cuda")
        v = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
        mc.mc_prior_quadratic(shape, beta, xd, g if with_g else None, v if with_v else None)
        if with_g:
            assert _ulps(g.cpu().numpy(), want_g).max() <= 0.505
        if with_v:
            assert abs(v.item() - want_v) <= (24 + 3 * n / 256) * U * want_v
