"""The forced-detection kernel's traversal step, compiled for the host from the
library's own source, ends within nx + ny + nz steps whatever the map holds:
the true distance map, one of zeros, one of the largest values, and rays with
NaN or infinite faces.  On the true map the rays' attenuation integrals are
those of a voxel walk in float64.

Tolerance of that: FP32 sums of at most 3 * 19 terms, relative 1e-4.
"""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

pytest.importorskip("scipy.ndimage")

from tests.distance_map_ref import distance_map_by_filters  # noqa: E402

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_13324_gb300", "csrc",
                   "forced.cuh")
PRELUDE = r"""
#include <cfenv>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
static inline float __uint_as_float(uint32_t u) { float f; std::memcpy(&f, &u, 4); return f; }
static inline int __float_as_int(float f) { int i; std::memcpy(&i, &f, 4); return i; }
static inline uint32_t __ldg(const uint16_t *p) { return *p; }
static inline float __fadd_rd(float a, float b) {
  volatile float x = a, y = b;
  std::fesetround(FE_DOWNWARD);
  volatile float s = x + y;
  std::fesetround(FE_TONEAREST);
  return s;
}
template <typename T> struct TArgs { const uint16_t *cubes; int nx, ny, nz; };
"""
DRIVER = r"""
extern "C" int walk(const uint16_t *cubes, int nx, int ny, int nz, const float *f, const int *i, int limit, float *sum) {
  TArgs<float> a{cubes, nx, ny, nz};
  float2 s_mu[256];
  for (int m = 0; m < 256; ++m) { s_mu[m].x = 0.25f * (float)m; s_mu[m].y = 0.0f; }
  Ray r;
  r.tx = f[0]; r.ty = f[1]; r.tz = f[2]; r.dtx = f[3]; r.dty = f[4]; r.dtz = f[5];
  r.kpx = f[6]; r.kpy = f[7]; r.kpz = f[8]; r.t_grid = f[9];
  r.sig = 1.0f; r.ie3 = 0.0f; r.pref = 1.0f; r.t = 0.0f; r.sum = 0.0f;
  r.ix = i[0]; r.iy = i[1]; r.iz = i[2]; r.sx = i[3]; r.sy = i[4]; r.sz = i[5];
  r.key = 0;
  int n = 0;
  while (n < limit) {
    ++n;
    if (ray_step(a, s_mu, r)) { *sum = r.sum; return n; }
  }
  return -1;
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    text = open(SRC).read()
    ray = re.search(r"^struct Ray \{.*?^\};\n", text, re.S | re.M).group(0)
    step = re.search(r"^__device__ __forceinline__ float faces_crossed.*?^__device__ __forceinline__ bool ray_step.*?^\}\n",
                     text, re.S | re.M).group(0)
    d = tmp_path_factory.mktemp("ray_step")
    src, lib = d / "step.cpp", d / "step.so"
    src.write_text(PRELUDE + ray + step + DRIVER)
    subprocess.run(["g++", "-O1", "-frounding-math", "-ffp-contract=off", "-fPIC", "-shared", "-o", str(lib), str(src)],
                   check=True)
    fn = ctypes.CDLL(str(lib)).walk

    def run(mat, dmap, f, i, limit):
        nz, ny, nx = mat.shape
        cubes = np.ascontiguousarray(mat.astype(np.uint16) | (dmap.astype(np.uint16) << 8))
        fa, ia = np.array(f, np.float32), np.array(i, np.int32)
        s = ctypes.c_float(0.0)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        n = fn(p(cubes), nx, ny, nz, p(fa), p(ia), limit, ctypes.byref(s))
        return n, s.value
    return run


def _ray(shape, h, p, d):
    """The traversal's start, as the kernel prepares it, in float64."""
    n = np.array(shape[::-1])
    half = 0.5 * n * h
    ix = np.clip(np.floor((p + half) / h).astype(int), 0, n - 1)
    s = np.where(d > 0, 1, -1)
    with np.errstate(divide="ignore"):
        t = np.where(d != 0, ((ix + (s > 0)) * h - half - p) / d, np.inf)
        dt = np.where(d != 0, h / np.abs(d), 0.0)
    last = np.where(s > 0, n - 1 - ix, ix)
    t_grid = np.where(d != 0, t + last * dt, np.inf).min()
    return list(t) + list(dt) + list(np.abs(d) / h) + [t_grid], list(ix) + list(s)


def _rays(shape, h, count, seed):
    rng = np.random.default_rng(seed)
    for k in range(count):
        d = rng.normal(size=3)
        if k % 5 == 0:
            d[k // 5 % 3] = 0.0
        d /= np.linalg.norm(d)
        p = (rng.random(3) - 0.5) * np.array(shape[::-1]) * h
        yield p, d


def _volume(seed):
    mat = np.ones((13, 19, 17), np.uint8)
    mat[:, 5:11, 4:9] = 2
    mat[6, 15, :] = 3
    return mat


def _voxel_walk(mat, h, p, d):
    n = np.array(mat.shape[::-1])
    half = 0.5 * n * h
    cuts = [0.0]
    for a in range(3):
        if d[a]:
            t = (np.arange(n[a] + 1) * h - half[a] - p[a]) / d[a]
            cuts += list(t[t > 0])
    end = min(max(((np.array([0, n[a]]) * h - half[a] - p[a]) / d[a])) for a in range(3) if d[a])
    cuts = np.unique([c for c in cuts if c <= end] + [end])
    mid = 0.5 * (cuts[1:] + cuts[:-1])
    q = p[None, :] + mid[:, None] * d[None, :]
    i = np.clip(np.floor((q + half) / h).astype(int), 0, n - 1)
    return float((0.25 * mat[i[:, 2], i[:, 1], i[:, 0]] * np.diff(cuts)).sum())


def test_integrals_on_the_true_map(walk):
    mat, h = _volume(0), 4.0
    dmap = distance_map_by_filters(mat)
    for p, d in _rays(mat.shape, h, 400, 1):
        n, s = walk(mat, dmap, *_ray(mat.shape, h, p, d), sum(mat.shape))
        assert n > 0
        want = _voxel_walk(mat, h, p, d)
        assert abs(s - want) <= 1e-4 * want + 1e-4


@pytest.mark.parametrize("value", [0, 1, 255])
def test_ends_on_any_map(walk, value):
    mat, h = _volume(0), 4.0
    dmap = np.full(mat.shape, value, np.uint8)
    for p, d in _rays(mat.shape, h, 200, 2):
        n, _ = walk(mat, dmap, *_ray(mat.shape, h, p, d), sum(mat.shape))
        assert n > 0, (p, d)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_ends_on_any_ray(walk, bad):
    mat, h = _volume(0), 4.0
    dmap = distance_map_by_filters(mat)
    for k, (p, d) in enumerate(_rays(mat.shape, h, 300, 3)):
        f, i = _ray(mat.shape, h, p, d)
        rng = np.random.default_rng(k)
        f[rng.integers(0, 10)] = bad
        if k % 2:
            f[0] = f[1] = f[2] = bad
        if k % 3 == 0:
            f[9] = bad
        n, _ = walk(mat, dmap, f, i, sum(mat.shape))
        assert n > 0, (f, i)
