"""Matrix assembly by sorted segments, against the oracle's sums: columns and
rows at the edges of the warp sort's lengths (1 .. 1024 elements, and one
beyond, which the radix path takes), repeated events, keys too wide for 32
bits, and the two-pass transpose of entries beyond the L2.  Integer work:
exact equality.
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


def _check(mc, rows, cols, m, n, weights):
    first, count = 3, 2 * n + 5
    if weights is None:
        s = mc.mc_system_from_events(m, n, rows, cols, first, count)
        want = oracle.system_counts(rows, cols, m, n)
    else:
        s = mc.mc_system_from_weighted_events(m, n, rows, cols, weights, first, count)
        want = oracle.system_weights(rows, cols, weights, m, n)
    want.sort_indices()
    cp, ri, cnt, _ = s.export_csc()
    csc, csr = s.export_values()
    assert np.array_equal(cp, want.indptr) and np.array_equal(ri, want.indices)
    assert np.array_equal(csc, want.data.astype(np.float64))
    t = want.tocsr()
    t.sort_indices()
    rp, ci, rcnt = s.export_csr()
    assert np.array_equal(rp, t.indptr) and np.array_equal(ci, t.indices)
    assert np.array_equal(csr, t.data.astype(np.float64))
    n_ev = oracle.system_counts(rows, cols, m, n)
    n_ev.sort_indices()
    assert np.array_equal(cnt, n_ev.data) and s.info()["max_count"] == n_ev.data.max()
    t = n_ev.tocsr()
    t.sort_indices()
    assert np.array_equal(rcnt, t.data)
    # the projector values written with the entries, and the column sums
    import torch
    b = torch.empty(n, dtype=torch.float32, device="cuda")
    mc.mc_backproject(s, torch.ones(m, dtype=torch.float32, device="cuda"), b)
    sens = torch.empty(n, dtype=torch.float64, device="cuda")
    mc.mc_sensitivity(s, sens)
    nv = oracle.histories_per_voxel(n, first, count)
    ref = np.asarray(want.astype(np.float64).sum(0)).ravel() / np.maximum(nv, 1)
    np.testing.assert_allclose(sens.cpu().numpy(), ref, rtol=1e-13)
    np.testing.assert_allclose(b.cpu().numpy(), ref, rtol=1e-5)  # FP32 sums of up to ~1000 positive terms


def _weights(rng, n):
    return rng.integers(1, 1 << 46, n, dtype=np.uint64)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("length", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1023, 1024, 1025])
def test_column_and_row_lengths(mc, length, weighted):
    """One long column and one long row among short ones, some events repeated."""
    rng = np.random.default_rng(length)
    m, n = 1500, 1300
    cols = np.concatenate([np.full(length, 7), rng.integers(0, n, 30_000), rng.permutation(n)[:min(length, n)]])
    rows = np.concatenate([rng.integers(0, m, length), rng.integers(0, m, 30_000), np.full(min(length, n), 1499)])
    keep = (cols != 7) | (np.arange(len(cols)) < length)  # column 7 has exactly `length` events
    rows, cols = rows[keep].astype(np.int32), cols[keep].astype(np.int32)
    p = rng.permutation(len(rows))
    _check(mc, rows[p], cols[p], m, n, _weights(rng, len(rows)) if weighted else None)


@pytest.mark.parametrize("m,n", [(1 << 28, 300), (300, 1 << 25)])
def test_wide_keys(mc, m, n):
    """Row (column) numbers that leave no room for the event's place in 32 bits."""
    rng = np.random.default_rng(1)
    rows = rng.integers(0, m, 40_000).astype(np.int32)
    cols = rng.integers(0, n, 40_000).astype(np.int32)
    s = mc.mc_system_from_weighted_events(m, n, rows, cols, _weights(rng, len(rows)), 0, n)
    order = np.lexsort((rows, cols))
    key = cols[order].astype(np.int64) * m + rows[order]
    assert len(np.unique(key)) == s.info()["nnz"]
    cp, ri, _, _ = s.export_csc()
    assert np.array_equal(np.repeat(np.arange(n), np.diff(cp)) * m + ri, np.unique(key))
    rp, ci, _ = s.export_csr()
    got = np.repeat(np.arange(m, dtype=np.int64), np.diff(rp)) * n + ci
    assert np.array_equal(got, np.unique(rows.astype(np.int64) * n + cols))


def test_two_pass_transpose(mc):
    """More than 256 MB of entries: row blocks, some of them empty or ragged."""
    rng = np.random.default_rng(2)
    m, n, k = 150_001, 170_003, 18_000_000
    rows = rng.integers(0, m, k).astype(np.int32)
    rows[(rows > 60_000) & (rows < 61_000)] = 60_000 - (np.arange(((rows > 60_000) & (rows < 61_000)).sum()) % 997).astype(np.int32)
    cols = rng.integers(0, n, k).astype(np.int32)
    _check(mc, rows, cols, m, n, _weights(rng, k))
