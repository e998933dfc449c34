"""A plan made on one stream and built on another: everything the plan holds,
the forced-detection map included, is complete when mc_plan_create returns.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("forced", [True, False])
def test_creation_leaves_nothing_queued(mc, forced):
    """A grid whose map takes ~0.1 ms to pack: the stream is idle on return."""
    import torch
    n = 256
    ph, g = P.uniform_phantom(n, 1.0), P.spect_geometry(2, 360.0, 8, 32.0, 8, 32.0)
    s = torch.cuda.Stream()
    for _ in range(3):
        plan = mc.mc_plan_create(ph, g, stream=s, forced=forced)
        idle = s.query()
        s.synchronize()
        plan.free()
        assert idle


def test_build_on_another_stream(mc):
    import torch
    ph, g = P.torso_phantom(24, 10.0, seed=2), P.spect_geometry(9, 360.0, 24, 10.0, 24, 10.0)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    one = mc.mc_build_system(ph, g, 20_000, 3, forced=True)
    for _ in range(3):
        plan = mc.mc_plan_create(ph, g, stream=a, forced=True)
        two = mc.mc_plan_build(plan, 0, 20_000, 3, stream=b)
        for x, y in zip(one.export_csc() + one.export_values(), two.export_csc() + two.export_values()):
            assert np.array_equal(x, y)
        plan.free()
