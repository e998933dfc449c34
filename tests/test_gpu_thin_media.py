"""Media so thin that their attenuation is a denormal float: a photon still draws
its first flight before it leaves, as in the FP64 oracle, and the detections
are the same ones.

Tolerance: a float acceptance or detector bin differs from the oracle's with a
probability of ~1e-5: 1e-3 of the detections and one.  (A photon that left
without the draw would be offered other random words: about all would differ.)
"""
import numpy as np
import pytest

import oracle
from paper_2105_13324_gb300 import phantoms as P
from tests.test_gpu_histories import _common

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


@pytest.mark.parametrize("density", [1e-38, 3e-37, 1e-35])
@pytest.mark.parametrize("primary", [False, True])
def test_detections_of_thin_media(mc, density, primary):
    row = (density,) + tuple(P.WATER[1:])
    ph, g = P.uniform_phantom(5, 20.0, row), P.spect_geometry(9, 360.0, 5, 20.0, 5, 20.0, hole_diam_mm=9.0)
    ph.material[:] = 1
    ph.rho[0] = 0.0  # nothing else attenuates
    pr = oracle.Problem(ph, g, primary_only=primary)
    count = 100_003
    rows, cols, fates = oracle.run(pr, 11, 2, count)
    s = mc.mc_build_system_range(ph, g, 2, count, 11, primary_only=primary)
    assert np.array_equal(s.info()["fates"], fates) and len(rows) > 100
    cp, ri, cnt, _ = s.export_csc()
    got = np.repeat(np.repeat(np.arange(pr.n_voxels), np.diff(cp)) * pr.n_rows + ri, cnt)
    want = cols.astype(np.int64) * pr.n_rows + rows
    assert len(got) + len(want) - 2 * _common(got, want) <= 2e-3 * len(want) + 2
