// forced.cuh -- float forced detection (paper Sec. 4, "forced detection"):
// the weighted copy of every queued interaction towards every view.  Included
// by transport_f32.cu; transport.cuh has the double path and the contract's
// formulas in their literal order.
#pragma once

#include "transport.cuh"

namespace mcs {

// A copy is first drawn and tested -- direction in the view's acceptance cone,
// scattered energy in the window, detector bin -- and, if it can count,
// becomes a ray: its traversal of the grid to the boundary still to be done.
// Rays take very different numbers of steps (18 on average on the 128^3
// torso) and a third of the copies never become one, so each warp keeps a
// stack of prepared rays in shared memory: 32 copies are drawn at a time, and
// a lane whose ray has ended takes the next one as soon as kRayIdle lanes of
// the warp are without.
//
// Bound by latency and issue together: each step is one dependent load of the
// grid (material and distance in one 16-bit word), of which the L1 -- what the
// stacks leave of it -- holds few lines.  The launch takes what an SM holds:
// seven blocks at 68 registers (six run alike, eight are 5 % slower, five 7 %).
// 2^21 histories of the 128^3 torso towards 120 views (3.9e8 copies, 2.6e8
// events): 24 ms, 33 with a lane per copy to its end; the same events.  Rays of
// unequal length are handed out when 8 lanes are idle: 4 to 16 within 2 %.
constexpr int kRayThreads = 128;
constexpr int kRayPool = 64;   // rays waiting per warp: 31 before a round of 32 at most
constexpr int kRayQuads = 5;   // 16-byte words per ray
constexpr int kRayEnded = 64;  // ended rays per warp: 31 and 32 more at most
constexpr int kRayIdle = 8;    // lanes without a ray before the warp hands out new ones
constexpr int kRayChunk = 256; // copies a warp takes at a time in a large launch

// tx..: ray parameter of the next face per axis; dtx..: its step per voxel;
// kpx..: voxels per unit length; sx..: the index's step (any value on an axis
// the ray does not move along: it crosses no face there); t_grid: the grid's
// exit; pref: the weight but for the transmission; t, sum: how far along, and
// the attenuation integral up to there.  On the stack the signs of dtx.. hold
// sx.. .
struct Ray {
  float tx, ty, tz, dtx, dty, dtz, kpx, kpy, kpz, t_grid, sig, ie3, pref, t, sum;
  int ix, iy, iz, sx, sy, sz;
  unsigned long long key;
};

__device__ __forceinline__ void ray_put(uint4 (*pool)[kRayPool], int s, const Ray &r) {
  const auto w = [](float x) { return __float_as_uint(x); };
  const auto sg = [&](float x, int d) { return w(x) | ((uint32_t)d & 0x80000000u); };
  pool[0][s] = make_uint4(w(r.tx), w(r.ty), w(r.tz), w(r.t_grid));
  pool[1][s] = make_uint4(sg(r.dtx, r.sx), sg(r.dty, r.sy), sg(r.dtz, r.sz), w(r.pref));
  pool[2][s] = make_uint4(w(r.kpx), w(r.kpy), w(r.kpz), w(r.sig));
  pool[3][s] = make_uint4((uint32_t)r.ix, (uint32_t)r.iy, (uint32_t)r.iz, w(r.ie3));
  pool[4][s] = make_uint4(w(r.t), (uint32_t)r.key, (uint32_t)(r.key >> 32), w(r.sum));
}
__device__ __forceinline__ void ray_get(uint4 (*pool)[kRayPool], int s, Ray &r) {
  const auto f = [](uint32_t x) { return __uint_as_float(x); };
  const auto sg = [](uint32_t x) { return 1 | ((int)x >> 31); };
  const uint4 a = pool[0][s], b = pool[1][s], c = pool[2][s], d = pool[3][s], e = pool[4][s];
  r.tx = f(a.x); r.ty = f(a.y); r.tz = f(a.z); r.t_grid = f(a.w);
  r.dtx = fabsf(f(b.x)); r.dty = fabsf(f(b.y)); r.dtz = fabsf(f(b.z)); r.pref = f(b.w);
  r.sx = sg(b.x); r.sy = sg(b.y); r.sz = sg(b.z);
  r.kpx = f(c.x); r.kpy = f(c.y); r.kpz = f(c.z); r.sig = f(c.w);
  r.ix = (int)d.x; r.iy = (int)d.y; r.iz = (int)d.z; r.ie3 = f(d.w);
  r.t = f(e.x); r.key = (unsigned long long)e.z << 32 | e.y; r.sum = f(e.w);
}

// The copy of record q towards view k, up to the traversal: its direction is
// uniform in the collimator's acceptance cone about the view's normal, drawn
// from the copy's own Philox block (counter (k, 1 + n, h_lo, h_hi)); the
// weight is the survival at the interaction times the angular probability
// of that direction times the collimator's open fraction (times the
// transmission); the copy is binned like an analog detection.  False: it
// cannot count.
__device__ __forceinline__ bool make_ray(const TArgs<float> &a, const FdRec<float> &q, int k, const float *sig_tab,
                                         Ray &r) {
  uint32_t w0 = (uint32_t)k, w1 = 1u + q.n, w2 = (uint32_t)q.h, w3 = (uint32_t)(q.h >> 32);
  philox_rounds(w0, w1, w2, w3, a.rk);
  const float u0 = uniform<float>(w0), u1 = uniform<float>(w1), u2 = uniform<float>(w2), u3 = uniform<float>(w3);
  const float ck = a.view_cs[2 * k], sk = a.view_cs[2 * k + 1];
  // 1 - cos is a few 1e-3 at most: sin^2 = (1 - cos)(1 + cos) keeps float's
  // relative precision where 1 - cos^2 would cancel
  const float om = u0 * a.one_m_cos_max;
  const float ct = 1.0f - om;
  const float st = sqrt0<float>(om * (2.0f - om));
  float cph, sph;
  cos_sin_2pi<float>(u1, cph, sph);
  const float dx = ct * ck - st * cph * sk, dy = ct * sk + st * cph * ck, dz = st * sph;
  if (!(a.ratio * st < ct)) return false;
  const float x = a.ratio * st / ct;
  const float pass = (float)(2.0 / kPi) * (acos(x) - x * sqrt0<float>(1.0f - x * x));
  float ang, e1;
  if (q.n == 0) {
    ang = a.omega_4pi;
    e1 = q.e;
  } else {
    const float mu_s = q.d[0] * dx + q.d[1] * dy + q.d[2] * dz;
    e1 = __fdividef(q.e, 1.0f + q.e * (float)(1.0 / kMec2) * (1.0f - mu_s));
    if (e1 < a.e_low) return false;
    Energy<float> en;
    en.set(q.e, a, sig_tab);
    ang = a.omega * kn_pdf_sr<float>(q.e, mu_s, en);
  }
  r.pref = q.keep * ang * pass;
  // detector bin
  const float px = q.p[0], py = q.p[1], pz = q.p[2];
  {
    const float t = (a.plane - (px * ck + py * sk)) / ct;
    const float qx = px + t * dx, qy = py + t * dy, qz = pz + t * dz;
    float au = -qx * sk + qy * ck;
    float bv = qz;
    const float rr = sqrt0<float>(-2.0f * ln_normal(u2));
    float cb, sb;
    cos_sin_2pi<float>(u3, cb, sb);
    au += a.sigma * (rr * cb);
    bv += a.sigma * (rr * sb);
    const float fu = floor(au / a.bin + a.half_bu);
    const float fv = floor(bv / a.bin + a.half_bv);
    if (!(fu >= 0.0f && fu < (float)a.bins_u && fv >= 0.0f && fv < (float)a.bins_v)) return false;
    const uint64_t row = ((uint64_t)k * a.bins_v + (uint64_t)fv) * a.bins_u + (uint64_t)fu;
    uint32_t v;
    div_magic(a.first_v + (uint32_t)(q.h - a.first), a.n_vox, a.magic_n, v);
    r.key = (unsigned long long)v * a.n_rows + row;
  }
  // the traversal's start
  Energy<float> en;
  en.set(e1, a, sig_tab);
  r.sig = en.sig;
  r.ie3 = en.ie3;
  r.ix = voxel_index<float>(px, a.hx, a.h, a.inv_h, a.hx_h, a.nx);
  r.iy = voxel_index<float>(py, a.hy, a.h, a.inv_h, a.hy_h, a.ny);
  r.iz = voxel_index<float>(pz, a.hz, a.h, a.inv_h, a.hz_h, a.nz);
  r.sx = dx > 0.0f ? 1 : (dx < 0.0f ? -1 : 0);
  r.sy = dy > 0.0f ? 1 : (dy < 0.0f ? -1 : 0);
  r.sz = dz > 0.0f ? 1 : (dz < 0.0f ? -1 : 0);
  const float rx = r.sx ? 1.0f / dx : 0.0f, ry = r.sy ? 1.0f / dy : 0.0f, rz = r.sz ? 1.0f / dz : 0.0f;
  // the first face on an axis lies at (i + (s > 0)) h - half, t = (face - p) / d;
  // each later face of that axis is h / |d| further along the ray
  const float ox = -a.hx - px, oy = -a.hy - py, oz = -a.hz - pz;
  r.tx = r.sx ? fmaf((float)(r.ix + (r.sx > 0)), a.h, ox) * rx : INFINITY;
  r.ty = r.sy ? fmaf((float)(r.iy + (r.sy > 0)), a.h, oy) * ry : INFINITY;
  r.tz = r.sz ? fmaf((float)(r.iz + (r.sz > 0)), a.h, oz) * rz : INFINITY;
  r.dtx = a.h * fabsf(rx); r.dty = a.h * fabsf(ry); r.dtz = a.h * fabsf(rz);
  r.kpx = fabsf(dx) * a.inv_h; r.kpy = fabsf(dy) * a.inv_h; r.kpz = fabsf(dz) * a.inv_h;
  // the ray leaves the grid at the last face of the first axis to run out
  r.t_grid = fminf(fminf(r.sx ? fmaf((float)(r.sx > 0 ? a.nx - 1 - r.ix : r.ix), r.dtx, r.tx) : INFINITY,
                         r.sy ? fmaf((float)(r.sy > 0 ? a.ny - 1 - r.iy : r.iy), r.dty, r.ty) : INFINITY),
                   r.sz ? fmaf((float)(r.sz > 0 ? a.nz - 1 - r.iz : r.iz), r.dtz, r.tz) : INFINITY);
  r.t = r.sum = 0.0f;
  return true;
}

// Faces crossed on one axis up to tc: all D on an axis that leaves the cube (its
// D-th face c is at tc), floor((tc - t) per) + 1 on the others, 0 where the next
// face t lies beyond tc, as a float (at most D <= kSkipCap).  The floor is by a
// round-down add of 1.5 2^23; a negative or NaN argument (no face) ends at 0.
__device__ __forceinline__ float faces_crossed(float c, float tc, float t, float per, float D) {
  const float n = __fadd_rd((tc - t) * per, 12582912.0f) - 12582911.0f;
  return c == tc ? D : fminf(fmaxf(n, 0.0f), D);
}
// a small non-negative integer held in a float, as an int
__device__ __forceinline__ int small_int(float k) { return __float_as_int(k + 8388608.0f) - 0x4B000000; }

// One step across a cube of constant mu.  The distance map gives, for the
// current voxel, the half-width D - 1 of the cube around it that holds one
// material; the ray leaves that cube at the (D - 1)-th face beyond the voxel's
// own next face on one axis, so mu times the length up to there is the exact
// integral over the cube (D = 1 is one ordinary voxel step).  Returns whether
// the ray has left the grid.  Every step that does not crosses at least one face
// outward on one axis -- a distance of 0 counts as 1, and a ray without a
// next face before the exit (or with a NaN there) ends -- so a ray ends after
// nx + ny + nz steps at most, whatever the map and the ray hold.
__device__ __forceinline__ bool ray_step(const TArgs<float> &a, const float2 *s_mu, Ray &r) {
  const uint32_t cell = __ldg(a.cubes + (uint32_t)((r.iz * a.ny + r.iy) * a.nx + r.ix));
  const float D = fmaxf(__uint_as_float(0x4B000000u | cell >> 8) - 8388608.0f, 1.0f);
  const float2 c = s_mu[cell & 255u];
  const float e = D - 1.0f;
  const float cx = fmaf(e, r.dtx, r.tx), cy = fmaf(e, r.dty, r.ty), cz = fmaf(e, r.dtz, r.tz);
  const float tc = fminf(fminf(fminf(cx, cy), cz), r.t_grid);
  r.sum = fmaf(fmaf(c.x, r.sig, c.y * r.ie3), fmaxf(tc - r.t, 0.0f), r.sum);
  r.t = fmaxf(r.t, tc);
  const float kx = faces_crossed(cx, tc, r.tx, r.kpx, D), ky = faces_crossed(cy, tc, r.ty, r.kpy, D),
              kz = faces_crossed(cz, tc, r.tz, r.kpz, D);
  r.ix += r.sx * small_int(kx);
  r.iy += r.sy * small_int(ky);
  r.iz += r.sz * small_int(kz);
  r.tx = fmaf(kx, r.dtx, r.tx);
  r.ty = fmaf(ky, r.dty, r.ty);
  r.tz = fmaf(kz, r.dtz, r.tz);
  return !(tc < r.t_grid) || (unsigned)r.ix >= (unsigned)a.nx || (unsigned)r.iy >= (unsigned)a.ny ||
         (unsigned)r.iz >= (unsigned)a.nz;
}

// Append a warp's events.  The fixed-point weight rint(w 2^48) is taken from
// the float itself: the product with 2^48 is exact.
__device__ __forceinline__ void append_events(const TArgs<float> &a, unsigned long long key, float w, int lane) {
  const long long q = __float2ll_rn(w * (float)kFdScale);
  const unsigned m = __ballot_sync(0xffffffffu, q > 0);
  if (m == 0u) return;
  unsigned long long base = 0;
  const int leader = __ffs(m) - 1;
  if (lane == leader) base = atomicAdd(a.cursor, (unsigned long long)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader) + __popc(m & ((1u << lane) - 1u));
  if (q > 0 && base < a.capacity) {
    a.events[base] = key;
    a.weights[base] = (unsigned long long)q;
  }
}

__global__ void __launch_bounds__(kRayThreads, 6) ray_kernel(const __grid_constant__ TArgs<float> a) {
  __shared__ float2 s_mu[256];
  __shared__ float s_sig[kSigTab];
  __shared__ uint4 s_pool[kRayThreads / 32][kRayQuads][kRayPool];
  __shared__ unsigned long long s_key[kRayThreads / 32][kRayEnded];
  __shared__ float s_w[kRayThreads / 32][kRayEnded];
  for (int m = threadIdx.x; m < a.n_mat; m += kRayThreads) s_mu[m] = make_float2(a.coef[3 * m], a.coef[3 * m + 1]);
  for (int i = threadIdx.x; i < kSigTab; i += kRayThreads) s_sig[i] = a.sig_tab[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  uint4 (*pool)[kRayPool] = s_pool[threadIdx.x >> 5];
  unsigned long long *end_key = s_key[threadIdx.x >> 5];
  float *end_w = s_w[threadIdx.x >> 5];
  int n_end = 0;  // ended rays waiting to be appended
  const unsigned long long n_q = *a.esc_cursor < a.esc_capacity ? *a.esc_cursor : a.esc_capacity;
  const unsigned long long total = n_q * (unsigned long long)a.n_views;
  const FdRec<float> *q = static_cast<const FdRec<float> *>(a.esc);
  // copies are taken in chunks, strided over the warps: views fastest, so
  // that a warp's rays start in one or two voxels
  const unsigned long long n_warps = (unsigned long long)gridDim.x * (kRayThreads / 32);
  unsigned long long chunk = (total / (n_warps * 4ull)) & ~31ull;
  chunk = chunk < 32ull ? 32ull : chunk > kRayChunk ? kRayChunk : chunk;
  unsigned long long next = ((unsigned long long)blockIdx.x * (kRayThreads / 32) + (threadIdx.x >> 5)) * chunk;
  unsigned long long rec = 0;         // the chunk's present record and view
  uint32_t view = 0, left = 0;        // copies left in the chunk
  int n_ray = 0;
  bool on = false;
  Ray r = {};
  for (;;) {
    unsigned idle = __ballot_sync(0xffffffffu, !on);
    int n_idle = __popc(idle);
    // 1. draw copies until the stack can fill the idle lanes; the unfinished
    // rays wait on the stack meanwhile (their registers are needed)
    if (n_ray < n_idle && (left > 0u || next < total)) {
      if (on) ray_put(pool, n_ray + __popc(~idle & lt), r);
      n_ray += 32 - n_idle;
      n_idle = 32;
      idle = 0xffffffffu;
      on = false;
      while (n_ray < n_idle) {
        if (left == 0u) {
          if (next >= total) break;
          left = (uint32_t)(total - next < chunk ? total - next : chunk);
          rec = next / (unsigned long long)a.n_views;
          view = (uint32_t)(next - rec * (unsigned long long)a.n_views);
          next += n_warps * chunk;
        }
        Ray c = {};
        uint32_t k;
        const uint32_t dr = div_magic(view + lane, (uint32_t)a.n_views, a.magic_views, k);
        bool ok = false;
        if ((uint32_t)lane < left) ok = make_ray(a, q[rec + dr], (int)k, s_sig, c);
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (ok) ray_put(pool, n_ray + __popc(m & lt), c);
        n_ray += __popc(m);
        left -= left < 32u ? left : 32u;
        rec += div_magic(view + 32u, (uint32_t)a.n_views, a.magic_views, view);
      }
      r = Ray{};
    }
    __syncwarp();
    if (n_ray == 0 && n_idle == 32) break;
    // 2. hand out rays
    {
      const int p = __popc(idle & lt);
      if (!on && p < n_ray) {
        ray_get(pool, n_ray - 1 - p, r);
        on = true;
      }
      n_ray -= n_ray < n_idle ? n_ray : n_idle;
    }
    __syncwarp();
    // 3. steps, until enough lanes have ended (all, when nothing is left to
    // hand out)
    const int go_on = n_ray > 0 || left > 0u || next < total ? 33 - kRayIdle : 1;
    bool flying = on;
    do {
      if (flying) flying = !ray_step(a, s_mu, r);
      if (flying) flying = !ray_step(a, s_mu, r);
    } while (__popc(__ballot_sync(0xffffffffu, flying)) >= go_on);
    // 4. the rays that have ended wait for the next full warp of events
    const unsigned m = __ballot_sync(0xffffffffu, on && !flying);
    if (on && !flying) {
      const int e = n_end + __popc(m & lt);
      end_key[e] = r.key;
      end_w[e] = r.pref * __expf(-r.sum);
    }
    n_end += __popc(m);
    on = flying;
    __syncwarp();
    if (n_end >= 32) {
      n_end -= 32;
      append_events(a, end_key[n_end + lane], end_w[n_end + lane], lane);
    }
  }
  append_events(a, lane < n_end ? end_key[lane] : 0ull, lane < n_end ? end_w[lane] : 0.0f, lane);
}

int launch_rays(const TransportSetup &ts, TArgs<float> &a, cudaStream_t s) {
  if (!ts.cubes_dev) {
    set_error("float forced detection needs the plan's distance map");
    return MC_EINVAL;
  }
  int per_sm = 0;
  MCS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ray_kernel, kRayThreads, 0));
  if (per_sm < 1) per_sm = 1;
  count_launch(); ray_kernel<<<device_sm_count() * per_sm, kRayThreads, 0, s>>>(a);
  MCS_LAUNCHED();
  return MC_OK;
}

}  // namespace mcs
