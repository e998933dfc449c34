"""The log-likelihoods of an ML-EM run, summed in groups of iterations, and the
FP64 logarithm they use: against the oracle at counts of iterations around the
groups' ends, through both entry points, and per bin against numpy.

Tolerance: the projections are FP32 (relative 1e-6, see test_gpu_parity.py);
with images that make them exact, a log-likelihood is a sum of FP64 terms of
one unit in the last place each (1e-14 of the sum of their sizes).
"""
import numpy as np
import pytest

import oracle
from paper_2105_13324_gb300 import phantoms as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


@pytest.mark.parametrize("iters", [1, 2, 7, 33])
@pytest.mark.parametrize("m,n,row_len", [(3000, 700, (1, 6)), (5000, 400, (40, 60))])
def test_loglik_sequence(mc, iters, m, n, row_len):
    import torch
    rows, cols = P.random_events(m, n, row_len, 3, 5)
    s = mc.mc_system_from_events(m, n, rows, cols, 0, 4 * n)
    a = oracle.system_matrix(oracle.system_counts(rows, cols, m, n), oracle.histories_per_voxel(n, 0, 4 * n))
    y = P.poisson_counts(a @ np.linspace(1, 3, n), 1e5, 4)
    x0 = oracle.mlem_init(a, y)
    want, lls = oracle.mlem(a, y, x0, iters, with_loglik=True)
    yd = torch.as_tensor(y).cuda()
    seqs = []
    for f in (mc.mlem_iterate, mc.mlem_iterate_noalloc):
        x = torch.as_tensor(x0.astype(np.float32)).cuda()
        ll = f(s, yd, x, iters, loglik=True)
        assert np.linalg.norm(x.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
        np.testing.assert_allclose(ll, np.asarray(lls)[:iters], rtol=1e-6)
        seqs.append(ll)
    assert np.array_equal(*seqs)


def test_log_per_bin(mc):
    """One entry per row, so that q = x exactly: y ln q - q over q from the
    smallest normal floats to the largest, and around 1."""
    import torch
    rng = np.random.default_rng(0)
    q = np.concatenate([(10.0 ** rng.uniform(-37, 38, 4000)), 10.0 ** rng.uniform(-3, 3, 4000),
                        1 + rng.uniform(-0.01, 0.01, 2000),
                        [1.0, 2.0, 0.5, 1.1754944e-38, 3e38, 0.99999994, 1.0000001, 0.70710677, 0.7071068, 1.4142135,
                         1.4142137, 1e-40]]).astype(np.float32)
    n = len(q)
    s = mc.mc_system_from_events(n, n, np.arange(n), np.arange(n), 0, n)
    y = np.ones(n, np.float32)
    v = torch.zeros(1, dtype=torch.float64, device="cuda")
    for lo in range(0, n, 500):  # sums small enough that one wrong log shows
        yy = np.zeros(n, np.float32)
        yy[lo:lo + 500] = y[lo:lo + 500]
        xx = np.where(yy > 0, q, 0).astype(np.float32)
        mc.mc_loglik(s, torch.as_tensor(xx).cuda(), torch.as_tensor(yy).cuda(), v)
        qq = xx[lo:lo + 500].astype(np.float64)
        terms = np.log(qq) - qq
        assert abs(v.item() - terms.sum()) <= 1e-14 * np.abs(np.concatenate([np.log(qq), qq])).sum()
