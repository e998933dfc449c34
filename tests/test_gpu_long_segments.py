"""The streaming layout on long rows and columns: tiles at the mean length where
a warp takes a row instead of a thread (80), single rows around the length that
a warp sums in a thread's stead (128), and the longest that the layout takes.

Tolerance: FP32 sums of at most 2047 positive terms in 32 strided parts (64
terms each, then five levels): 70 roundings of 2^-24 each at the very most,
4.2e-6, and typically a tenth; 1e-6 as for the other layouts holds by far for the
short ones, 4.2e-6 for these.  The two ways of summing a row add in one order:
equal bits.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


def _events(lengths, n, seed):
    """Rows of the given lengths, distinct columns in each."""
    rng = np.random.default_rng(seed)
    cols = np.concatenate([np.sort(rng.permutation(n)[:k]) for k in lengths])
    return np.repeat(np.arange(len(lengths)), lengths).astype(np.int32), cols.astype(np.int32)


def _project(mc, rows, cols, m, n, x):
    import torch
    s = mc.mc_system_from_events(m, n, rows, cols, 0, 2 * n + 1)
    assert mc.mc_system_set_spmv_layout(s, 0, 0) == (0, 0)
    return s, mc.mc_project(s, torch.as_tensor(x).cuda(), torch.empty(m, device="cuda")).cpu().numpy()


@pytest.mark.parametrize("name,lengths,n", [
    ("79", [79] * 300, 2100), ("80", [80] * 300, 2100), ("81", [81] * 300, 2100),
    ("mixed", ([20] * 40 + [127, 128, 129, 0, 700, 2047]) * 6, 2100), ("few", [2047, 1, 2047], 2100),
    ("hundreds", [300, 310, 0, 290] * 60, 2100), ("one", [2047], 2047),
])
def test_against_oracle(mc, name, lengths, n):
    import torch
    m = len(lengths)
    rows, cols = _events(lengths, n, 4)
    rng = np.random.default_rng(2)
    x, r = rng.uniform(0.5, 2, n).astype(np.float32), rng.uniform(0.5, 2, m).astype(np.float32)
    s, q = _project(mc, rows, cols, m, n, x)
    a = oracle.system_matrix(oracle.system_counts(rows, cols, m, n), oracle.histories_per_voxel(n, 0, 2 * n + 1))
    np.testing.assert_allclose(q, a @ x.astype(np.float64), rtol=4.2e-6)
    # the same lengths as columns
    t = mc.mc_system_from_events(n, m, cols, rows, 0, 2 * m + 1)
    assert mc.mc_system_set_spmv_layout(t, 0, 0) == (0, 0)
    b = mc.mc_backproject(t, torch.as_tensor(x).cuda(), torch.empty(m, device="cuda")).cpu().numpy()
    at = oracle.system_matrix(oracle.system_counts(cols, rows, n, m), oracle.histories_per_voxel(m, 0, 2 * m + 1))
    np.testing.assert_allclose(b, at.T @ x.astype(np.float64), rtol=4.2e-6)
    # with the log-likelihood, which takes the same sums
    y = np.ones(m, np.float32)
    v = torch.zeros(1, dtype=torch.float64, device="cuda")
    mc.mc_loglik(s, torch.as_tensor(x).cuda(), torch.as_tensor(y).cuda(), v)
    q64 = q.astype(np.float64)
    want = (np.log(q64, where=q64 > 0, out=np.zeros(m)) - q64).sum()
    assert abs(v.item() - want) <= 1e-13 * (np.abs(np.log(q64, where=q64 > 0, out=np.zeros(m))) + q64).sum()


@pytest.mark.parametrize("length", [33, 80, 127, 128, 129, 500])
def test_same_bits_by_thread_and_by_warp(mc, length):
    """A row among short ones (its tile is taken by threads, or its own warp) and
    among long ones (warps)."""
    n = 2100
    x = np.random.default_rng(2).uniform(0.5, 2, n).astype(np.float32)
    out = []
    for other in (17, 400):
        rows, cols = _events([length] + [other] * 500, n, 4)
        out.append(_project(mc, rows, cols, 501, n, x)[1][0])
    assert out[0] == out[1]
