"""Matrix assembly by sorted segments at lengths that are exact: one column and
one row of a given length among short ones, up to the longest that a warp sorts
(1024) and beyond, where the CSR (rows) or the whole matrix (columns) comes from
the radix sort; the two-pass transpose of unweighted entries.  Integer work:
exact equality.
"""
import numpy as np
import pytest

import oracle
from tests.test_gpu_segments import _check, _weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


def _events(rng, m, n, col_events, row_entries, others):
    """Column 7 has exactly col_events events, row m - 1 exactly row_entries
    entries; the other events stay off both."""
    c = rng.integers(0, n - 1, others)
    cols = [np.full(col_events, 7), np.where(c >= 7, c + 1, c), 8 + rng.permutation(n - 8)[:row_entries]]
    rows = [rng.integers(0, m - 1, col_events), rng.integers(0, m - 1, others), np.full(row_entries, m - 1)]
    rows, cols = np.concatenate(rows).astype(np.int32), np.concatenate(cols).astype(np.int32)
    p = rng.permutation(len(rows))
    rows, cols = rows[p], cols[p]
    counts = oracle.system_counts(rows, cols, m, n)
    assert np.bincount(cols, minlength=n).max() == col_events
    assert np.diff(counts.tocsr().indptr).max() == max(row_entries, np.bincount(rows)[:m - 1].max()) == row_entries
    return rows, cols


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("col_events,row_entries", [
    (257, 256), (512, 511), (513, 513), (767, 769), (1023, 1023), (1024, 1024),  # a warp each
    (200, 1025), (1024, 1600), (300, 5000),                                      # long row: its CSR by radix sort
    (1025, 900), (4000, 1024),                                                   # long column: all by radix sort
])
def test_exact_lengths(mc, weighted, col_events, row_entries):
    rng = np.random.default_rng(col_events * 7 + row_entries)
    m, n = 1700, 6000
    # 20 events a column on average: beyond the buckets' rule
    rows, cols = _events(rng, m, n, col_events, row_entries, 120_000)
    _check(mc, rows, cols, m, n, _weights(rng, len(rows)) if weighted else None)


@pytest.mark.parametrize("weighted", [False, True])
def test_all_rows_long(mc, weighted):
    rng = np.random.default_rng(3)
    m, n, k = 37, 9000, 200_000
    rows, cols = rng.integers(0, m, k).astype(np.int32), rng.integers(0, n, k).astype(np.int32)
    assert np.diff(oracle.system_counts(rows, cols, m, n).tocsr().indptr).min() > 1024
    _check(mc, rows, cols, m, n, _weights(rng, k) if weighted else None)


def test_two_pass_transpose_unweighted(mc):
    """More than 256 MB of 8-byte entries, some of them repeated events."""
    import torch
    m, n, k = 150_001, 170_003, 36_000_000
    g = torch.Generator(device="cuda").manual_seed(4)
    keys = torch.randint(0, m * n, (k,), dtype=torch.int64, device="cuda", generator=g)
    keys[::1000] = keys[1::1000]
    s = mc.mc_system_from_keys(m, n, keys, 0, n)
    want, counts = torch.unique(keys, return_counts=True)
    i = s.info()
    assert i["nnz"] == len(want) > (256 << 20) // 8 and i["max_count"] == counts.max().item()
    cp, ri, cnt, _ = s.export_csc()
    v = torch.as_tensor(np.repeat(np.arange(n), np.diff(cp))).cuda()
    assert torch.equal(v * m + torch.as_tensor(ri).cuda().long(), want)
    assert torch.equal(torch.as_tensor(cnt.astype(np.int64)).cuda(), counts)
    rp, ci, rcnt = s.export_csr()
    order = torch.argsort(want % m * n + want // m)
    t = want[order]
    j = torch.as_tensor(np.repeat(np.arange(m), np.diff(rp))).cuda()
    assert torch.equal(j, t % m) and torch.equal(torch.as_tensor(ci).cuda().long(), t // m)
    assert torch.equal(torch.as_tensor(rcnt.astype(np.int64)).cuda(), counts[order])
