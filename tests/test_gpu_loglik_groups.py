"""The log-likelihoods of ML-EM are summed in groups of iterations, as many as
fit the partial sums' room: iteration counts around the ends of the first and
second group, of the static room of mlem_iterate_noalloc (2^18 sums) and of the
64 MB of mlem_iterate.  Each value is the same sum whatever the group: equal to
that of a run one iteration at a time, bit for bit, and so is the image.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
M, N = 1 << 21, 1500


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


@pytest.fixture(scope="module")
def system(mc):
    import torch
    g = torch.Generator(device="cuda").manual_seed(2)
    keys = torch.randint(0, M * N, (2_500_000,), dtype=torch.int64, device="cuda", generator=g)
    s = mc.mc_system_from_keys(M, N, keys, 0, 3 * N + 1)
    y = torch.poisson(torch.full((M,), 2.0, device="cuda"), generator=g)
    return s, y, torch.rand(N, device="cuda", generator=g) + 0.5


# lanes per row, and the iterations in a group: room / (2^21 lanes / 256 blocks)
@pytest.mark.parametrize("call,lanes,group", [("noalloc", 8, 4), ("noalloc", 32, 1), ("alloc", 32, 32)])
def test_around_the_groups(mc, system, call, lanes, group):
    import torch
    s, y, x0 = system
    assert mc.mc_system_set_spmv_layout(s, lanes, 0) == (lanes, 0)
    run = mc.mlem_iterate_noalloc if call == "noalloc" else mc.mlem_iterate
    x, want, images = x0.clone(), [], {}
    for k in range(1, 2 * group + 2):
        want.append(mc.mlem_iterate(s, y, x, 1, loglik=True)[0])
        images[k] = x.clone()
    for iters in sorted({max(group - 1, 1), group, group + 1, 2 * group, 2 * group + 1}):
        x = x0.clone()
        got = run(s, y, x, iters, loglik=True)
        assert np.array_equal(got, np.array(want[:iters]))
        assert torch.equal(x, images[iters])
