"""The FP64 logarithm of the log-likelihood, one value at a time, against
numpy's extended precision.

A system of one bin with A = 1 and y = 2^127: the log-likelihood is
2^127 ln q - q, and q is below half a unit in the last place of the product,
so it is the logarithm scaled by a power of two.

Tolerance: correct rounding (half a unit in the last place) and, before it, the
reduction's own errors: the low parts and the r^4 bracket in float (2^-70 each
where ln q has units of 2^-64 and more, 2^-26 r^4 with |r| < 2^-11) and the
FP64 roundings of terms below 2^-22 (2^-75): 0.04 of a unit together.  0.55.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


def _values():
    rng = np.random.default_rng(11)
    near = 1 + np.concatenate([rng.uniform(-2e-3, 2e-3, 1500), np.arange(-20, 21) * 2.0 ** -23, 2.0 ** -np.arange(2, 24)])
    mid = np.exp(rng.uniform(-1.5, 1.5, 3000))
    far = 10.0 ** rng.uniform(-37.5, 12, 1500)
    # the table's intervals: 2^13 floats from 0x3F34EAAB on, their first and last
    edge = (0x3F34EAAB + (np.arange(0, 1024, 7)[:, None] << 13) + np.array([-1, 0, 1])).astype(np.uint32).ravel()
    q = np.concatenate([near, mid, far, [1.0, 2.0, 0.5, 1.1754944e-38]]).astype(np.float32)
    return np.concatenate([q, edge.view(np.float32), 2 * edge.view(np.float32)])


def test_log_within_055_ulp(mc):
    import torch
    q = _values()
    s = mc.mc_system_from_events(1, 1, np.zeros(1, np.int32), np.zeros(1, np.int32), 0, 1)
    qd = torch.as_tensor(q).cuda()
    y = torch.full((1,), 2.0 ** 127, device="cuda")
    out = torch.empty(len(q), dtype=torch.float64, device="cuda")
    for i in range(len(q)):
        mc.mc_loglik(s, qd[i:i + 1], y, out[i:i + 1])
    got = out.cpu().numpy() * 2.0 ** -127
    want = np.log(q.astype(np.longdouble))
    ulp = np.spacing(np.abs(want.astype(np.float64))).astype(np.longdouble)
    one = q == 1
    # at q = 1 the value is -q alone
    assert np.all(got[one] == -2.0 ** -127)
    err = np.abs(got.astype(np.longdouble) - want)[~one] / ulp[~one]
    worst = int(np.argmax(err))
    assert err[worst] <= 0.55, (q[~one][worst], float(err[worst]))
