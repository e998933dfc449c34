"""Where mlem_iterate keeps the partial sums of its log-likelihoods: the
system's own block, which other calls use, stays what it was, and nothing more
is held after the call.
"""
import ctypes
import threading

import numpy as np
import pytest

from paper_2105_13324_gb300 import phantoms as P

pytestmark = pytest.mark.gpu

USED_MEM_CURRENT = 7  # cudaMemPoolAttrUsedMemCurrent


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2105_13324_gb300 import build as B
    from paper_2105_13324_gb300 import mcspect
    mcspect.load(B.build())
    return mcspect


def _pool_bytes():
    """Bytes in use of the device's default memory pool."""
    import torch
    torch.cuda.synchronize()
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    pool, v = ctypes.c_void_p(), ctypes.c_uint64()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolGetAttribute(pool, USED_MEM_CURRENT, ctypes.byref(v)) == 0
    return v.value


def _system(mc, m=60_000, n=3000, stream=None):
    import torch
    rows, cols = P.random_events(m, n, (1, 6), 3, 5)
    s = mc.mc_system_from_events(m, n, rows, cols, 0, 4 * n, stream=stream)
    rng = np.random.default_rng(1)
    y, x = rng.poisson(4.0, m).astype(np.float32), rng.uniform(0.5, 1.5, n).astype(np.float32)
    return s, torch.as_tensor(y).cuda(), torch.as_tensor(x).cuda()


def test_nothing_is_kept(mc):
    s, y, x = _system(mc)
    mc.mlem_iterate(s, y, x, 1, loglik=True)
    mc.mlem_iterate(s, y, x, 60)  # the same buffers of 60 iterations' values, so that only partials can grow
    ll = mc.mlem_iterate(s, y, x, 1, loglik=True)
    before = _pool_bytes()
    for _ in range(3):
        ll = mc.mlem_iterate(s, y, x, 60, loglik=True)
    assert np.all(np.isfinite(ll))
    assert _pool_bytes() - before <= 4096  # 60 values of 8 bytes, in the pool's granularity


def test_with_a_likelihood_queued_before(mc):
    """A system made on one stream, mc_loglik queued and mlem_iterate called on
    another, while a thread makes other systems on the first."""
    import torch
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    s, y, x0 = _system(mc, stream=a)
    ref, ry, rx = _system(mc)
    want_v = torch.zeros(1, dtype=torch.float64, device="cuda")
    mc.mc_loglik(ref, rx, ry, want_v)
    want = mc.mlem_iterate(ref, ry, rx, 40, loglik=True)
    torch.cuda.synchronize()
    stop = threading.Event()

    def others():
        while not stop.is_set():
            t, _, _ = _system(mc, 9000, 500, stream=a)
            t.free()

    th = threading.Thread(target=others)
    th.start()
    try:
        for _ in range(5):
            x, v = x0.clone(), torch.zeros(1, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            with torch.cuda.stream(b):
                torch.cuda._sleep(2_000_000)
                mc.mc_loglik(s, x, y, v, stream=b)
                got = mc.mlem_iterate(s, y, x, 40, loglik=True, stream=b)
            assert np.array_equal(got, want)
            assert v.item() == want_v.item() and torch.equal(x, rx)
    finally:
        stop.set()
        th.join()


def test_layout_change_behind_a_queued_likelihood(mc):
    """A layout with more forward blocks than the system's partial sums cover,
    set on the stream that still has a likelihood to do."""
    import torch
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for change in (lambda s: mc.mc_system_set_spmv_layout(s, 32, 32, stream=b), lambda s: mc.mc_system_autotune(s, stream=b)):
        s, y, x = _system(mc, stream=a)
        ref, _, _ = _system(mc)
        v = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(3)]
        mc.mc_loglik(ref, x, y, v[0])
        torch.cuda.synchronize()
        with torch.cuda.stream(b):
            torch.cuda._sleep(5_000_000)
            mc.mc_loglik(s, x, y, v[1], stream=b)
            change(s)
            others = [_system(mc, 9000, 500, stream=a)[0] for _ in range(3)]
            mc.mc_loglik(s, x, y, v[2], stream=b)
        torch.cuda.synchronize()
        for t in others:
            t.free()
        assert v[1].item() == v[0].item()
        # another layout adds the rows' FP32 sums in another order: 1e-6 of the terms
        assert abs(v[2].item() - v[0].item()) <= 1e-6 * y.sum().item() * 10
