"""The production photon-history kernel (float, analog) at its edges, against
the FP64 oracle on the same streams: launches that fill part of a warp, one
warp's takes exactly, or none of its later rounds; a grid of one voxel and odd
grids; histories whose number needs 64 bits; unscattered photons only; a
vacuum, where every photon leaves without a flight; a medium of many scatters.

Tolerance: float uniforms differ from the oracle's by at most 2^-24 and float
positions by ~1e-5 mm, so a decision flips with probability ~1e-4 per history
at most; 1e-3 of the histories (and of the detections) leaves a factor of ten.
Everything else is integer bookkeeping and has to be exact.
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


def _geometry(n, h, views=9, arc=360.0, **kw):
    return P.spect_geometry(views, arc, n, h, n, h, **kw)


PROBLEMS = {
    "water": lambda: (P.water_cylinder_phantom(), _geometry(32, 4.0)),
    "torso23": lambda: (P.torso_phantom(23, 11.1, seed=4), _geometry(23, 11.1, 7, 180.0)),
    "voxel": lambda: (P.uniform_phantom(1, 60.0), _geometry(1, 60.0, hole_diam_mm=9.0)),
    "vacuum": lambda: (P.vacuum_phantom(5, 20.0), _geometry(5, 20.0, hole_diam_mm=9.0)),
    # an opaque block: many collisions per history, long rejection runs
    "bone": lambda: (P.uniform_phantom(9, 30.0, (6.0, 0.5148, 8.0)), _geometry(9, 30.0, hole_diam_mm=9.0, window_frac=1.2)),
}


@pytest.mark.parametrize("name,first,count,primary", [
    ("water", 0, 1, False), ("water", 7, 31, False), ("water", 0, 33, False), ("water", 3, 129, False),
    ("water", 12345, 152 * 8 * 4 * 32 + 17, False), ("water", 0, 1_500_007, True),
    ("torso23", 0, 700_001, False), ("torso23", (1 << 32) - 1000, 50_003, False),
    ("torso23", (5 << 32) + 77, 50_003, True), ("voxel", 0, 100_003, False), ("vacuum", 2, 100_003, False),
    ("bone", 0, 60_001, False),
])
def test_float_histories_match_oracle(mc, name, first, count, primary):
    ph, g = PROBLEMS[name]()
    pr = oracle.Problem(ph, g, primary_only=primary)
    rows, cols, fates = oracle.run(pr, 11, first, count)
    s = mc.mc_build_system_range(ph, g, first, count, 11, primary_only=primary)
    i = s.info()
    assert sum(i["fates"]) == count
    slack = 1e-3 * count + 1 if name != "vacuum" else 0
    assert np.all(np.abs(np.array(i["fates"], np.int64) - fates.astype(np.int64)) <= slack)
    cp, ri, cnt, nv = s.export_csc()
    assert np.array_equal(nv, oracle.histories_per_voxel(pr.n_voxels, first, count))
    got_v = np.repeat(np.arange(pr.n_voxels), np.diff(cp))
    key_g = np.repeat(got_v * pr.n_rows + ri, cnt)
    key_o = cols * pr.n_rows + rows
    assert np.all(np.diff(key_g) >= 0) and len(key_g) == i["n_events"]
    # detections only one side has (as multisets)
    assert len(key_g) + len(key_o) - 2 * _common(key_g, key_o) <= 2e-3 * len(key_o) + 2


def _common(a, b):
    """Size of the multiset intersection."""
    ka, ca = np.unique(a, return_counts=True)
    kb, cb = np.unique(b, return_counts=True)
    _, ia, ib = np.intersect1d(ka, kb, return_indices=True)
    return int(np.minimum(ca[ia], cb[ib]).sum())
