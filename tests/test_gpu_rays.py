"""The float forced-detection kernel at its edges, against the oracle: fewer
copies than a warp, views around the warp's width, one history, grids of one
voxel, one slab and odd sizes, unscattered copies only.

Tolerance: a float weight differs from the oracle's by the rounding of some
tens of operations (~1e-5), and a copy lands in another bin, or changes its
history's later collisions, with a probability of ~1e-4 (see
test_gpu_histories.py): 1e-3 of the entries and 1e-3 of the weight.
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


def _slab():
    p = P.slab_phantom(12, 9.0, P.WATER, 60.0, extra_rows=(P.BONE,))
    return p


PHANTOMS = {
    "voxel": (lambda: P.uniform_phantom(1, 50.0), 1, 50.0),
    "slab": (_slab, 12, 9.0),
    "torso19": (lambda: P.torso_phantom(19, 13.5, seed=6), 19, 13.5),
    "vacuum": (lambda: P.vacuum_phantom(6, 20.0), 6, 20.0),
}


@pytest.mark.parametrize("name,views,first,count,primary", [
    ("torso19", 1, 0, 1, False), ("torso19", 31, 0, 1, False), ("torso19", 32, 5, 3, False),
    ("torso19", 33, 0, 257, False), ("torso19", 120, (1 << 33) + 11, 3000, False), ("torso19", 7, 0, 6001, True),
    ("voxel", 9, 0, 2000, False), ("slab", 40, 3, 4000, False), ("vacuum", 5, 0, 3000, False),
])
def test_float_rays_match_oracle(mc, name, views, first, count, primary):
    make, n, h = PHANTOMS[name]
    ph, g = make(), P.spect_geometry(views, 360.0, n, h, n, h)
    pr = oracle.Problem(ph, g, primary_only=primary, forced_detection=True)
    rows, cols, q, _ = oracle.run_fd(pr, 13, first, count)
    want = oracle.system_weights(rows, cols, q, pr.n_rows, pr.n_voxels).tocsc()
    s = mc.mc_build_system_range(ph, g, first, count, 13, primary_only=primary, forced=True)
    cp, ri, _, _ = s.export_csc()
    w, _ = s.export_values()
    got_key = np.repeat(np.arange(pr.n_voxels), np.diff(cp)) * pr.n_rows + ri
    want_key = np.repeat(np.arange(pr.n_voxels), np.diff(want.indptr)) * pr.n_rows + want.indices
    common, ig, iw = np.intersect1d(got_key, want_key, return_indices=True)
    slack = 1e-3 * len(want_key) + 1
    assert len(got_key) + len(want_key) - 2 * len(common) <= 2 * slack
    off = np.abs(w[ig] - want.data[iw]) > 1e-3 * want.data[iw]
    assert off.sum() <= slack
    if len(common):
        same = ~off
        assert abs(w[ig][same].sum() - want.data[iw][same].sum()) <= 1e-4 * want.data[iw][same].sum()
    assert abs(s.info()["n_events"] - len(rows)) <= 2 * slack
