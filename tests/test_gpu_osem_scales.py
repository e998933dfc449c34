"""Ordered subsets whose systems scale the image differently: one subset holds
the rounded matrix A itself (no scale), the others counts (1 / n_v), so that each
update has to leave the image as the next subset reads it.

Tolerance: FP32 sums, relative L2 of 1e-5 as in test_gpu_osem.py.
"""
import numpy as np
import pytest
import scipy.sparse as sp

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


@pytest.mark.parametrize("n_sub,rounded", [(2, (0,)), (2, (1,)), (5, (1, 2)), (5, (0, 4)), (1, (0,))])
@pytest.mark.parametrize("row_len", [(1, 6), (20, 30), (60, 90)])
def test_mixed_subsets(mc, n_sub, rounded, row_len):
    import torch
    rpv, views, n = 40, 20, 700
    m, count = rpv * views, 3 * n + n // 2  # 3 or 4 histories a voxel
    rows, cols = P.random_events(m, n, row_len, 3, 8)
    nv = oracle.histories_per_voxel(n, 0, count)
    a = sp.csr_matrix(oracle.system_matrix(oracle.system_counts(rows, cols, m, n), nv))
    subsets = [oracle.subset_rows(m, rpv, n_sub, k) for k in range(n_sub)]
    s = mc.mc_system_from_events(m, n, rows, cols, 0, count)
    parts = [mc.mc_system_subset(s, rpv, n_sub, k) for k in range(n_sub)]
    half = a.copy()
    half.data = half.data.astype(np.float16).astype(np.float64)
    pick = np.zeros(m, bool)
    for k in rounded:
        parts[k].set_value_type("f16_a")
        pick[subsets[k]] = True
    d = sp.diags(pick.astype(np.float64))
    both = sp.csr_matrix(d @ half + (sp.identity(m) - d) @ a)
    y = P.poisson_counts(a @ np.linspace(1, 3, n), 40.0 * m, 4)
    x0 = oracle.mlem_init(a, y)
    x = torch.as_tensor(x0.astype(np.float32)).cuda()
    mc.osem_iterate(parts, parts, torch.as_tensor(y).cuda(), x, 3)
    want = oracle.osem(both, both, subsets, y, x0.astype(np.float32), 3)
    assert np.linalg.norm(x.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
