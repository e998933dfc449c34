"""The streaming layout's tiles for rows of 16 to 32 entries on average (the
automatic choice there), against the oracle: ragged rows, empty rows, rows of
more than 32 and of hundreds of entries among them, a last tile of one row.

Tolerance: FP32 sums of at most 700 positive terms in 32 strided parts,
relative 1e-6 element by element as for the other layouts.
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


@pytest.mark.parametrize("m,n,row_len,used,long", [(257, 400, (16, 16), 1.0, 0), (5000, 900, (1, 40), 1.0, 700),
                                                   (4001, 700, (31, 33), 0.7, 0), (1, 40, (31, 31), 1.0, 0)])
def test_tiles_match_oracle(mc, m, n, row_len, used, long):
    import torch
    rows, cols = P.random_events(m, n, row_len, 4, 9, rows_used=used)
    if long:
        rows = np.r_[rows, np.full(long, 3, np.int32)].astype(np.int32)
        cols = np.r_[cols, np.arange(long, dtype=np.int32)].astype(np.int32)
    s = mc.mc_system_from_events(m, n, rows, cols, 0, 3 * n + 1)
    assert mc.mc_system_set_spmv_layout(s, 0, 0) == (0, 0)
    a = oracle.system_matrix(oracle.system_counts(rows, cols, m, n), oracle.histories_per_voxel(n, 0, 3 * n + 1))
    rng = np.random.default_rng(3)
    x, r = rng.uniform(0.5, 2, n).astype(np.float32), rng.uniform(0.5, 2, m).astype(np.float32)
    q = mc.mc_project(s, torch.as_tensor(x).cuda(), torch.empty(m, device="cuda")).cpu().numpy()
    b = mc.mc_backproject(s, torch.as_tensor(r).cuda(), torch.empty(n, device="cuda")).cpu().numpy()
    np.testing.assert_allclose(q, a @ x.astype(np.float64), rtol=1e-6)
    np.testing.assert_allclose(b, a.T @ r.astype(np.float64), rtol=1e-6)
    y = P.poisson_counts(a @ x.astype(np.float64), 50.0 * m, 2)
    x0 = oracle.mlem_init(a, y)
    xd = torch.as_tensor(x0.astype(np.float32)).cuda()
    mc.mlem_iterate(s, torch.as_tensor(y).cuda(), xd, 5)
    want = oracle.mlem(a, y, x0, 5)
    assert np.linalg.norm(xd.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("lens", [[(1, 2)], [(18, 30)], [(1, 2), (18, 30), (1, 6)]])
def test_batches_with_and_without_tiles(mc, lens):
    """The batch kernels of batches whose systems are all warp chunks, all
    tiles, or mixed, against the oracle."""
    import torch
    sysm, ys, xs, want = [], [], [], []
    for i, rl in enumerate(lens):
        m, n = 3000 + 7 * i, 1100 + i
        rows, cols = P.random_events(m, n, rl, 2, 20 + i)
        sysm.append(mc.mc_system_from_events(m, n, rows, cols, 0, 2 * n))
        a = oracle.system_matrix(oracle.system_counts(rows, cols, m, n), oracle.histories_per_voxel(n, 0, 2 * n))
        y = P.poisson_counts(a @ np.linspace(1, 2, n), 20.0 * m, i)
        ys.append(torch.as_tensor(y).cuda())
        xs.append(torch.empty(n, dtype=torch.float32, device="cuda"))
        want.append(oracle.mlem(a, y, oracle.mlem_init(a, y), 6))
    b = mc.mc_batch_create(sysm, ys, xs)
    for run in (mc.mc_batch_mlem, mc.mc_batch_mlem_persistent):
        run(b, 6)
        for x, w in zip(xs, want):
            assert np.linalg.norm(x.cpu().numpy() - w) <= 1e-5 * np.linalg.norm(w)
