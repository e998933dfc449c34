// histories.cuh -- the production photon-history kernel: analog transport in
// float (paper Sec. 2).  Included by transport_f32.cu; the samplers, the
// detection kernel and the launch arguments are transport.cuh's.
#pragma once

#include "transport.cuh"

namespace mcs {

// ---------------------------------------------------------------------------
// analog production transport: warp-private photon stacks
// ---------------------------------------------------------------------------
// The same histories as transport_kernel<float> (same draws, same arithmetic,
// same decisions), scheduled so that every step runs with a full warp.  Each
// warp owns a pool of kPool photon states in shared memory holding two
// stacks: photons ready to fly (from slot 0 up) and photons at a real
// collision (from the last slot down).  Flying photons live in the lanes'
// registers.  Per round the warp does one of
//   emission   32 consecutive new histories: emission and first flight, all
//              lanes together; survivors go to the stacks;
//   collision  32 photons of the collision stack: absorption or a Compton
//              scatter; survivors go to the flight stack;
//   flight     lanes without a photon take one from the flight stack, then
//              every lane flies up to twice; photons that collide go to the
//              collision stack.
// A collision round runs when 32 photons wait (or nothing else is left), an
// emission round when the flight stack cannot fill the lanes, so lanes idle
// only within a round and in the warp's last rounds.  Nothing but the event
// queue leaves the warp: no block barrier, no waiting lanes.
//
// Random words: a history draws 5 words at emission, 2 per flight, and at a
// collision 1 + 2 per rejection trial + 1, so the stream position is odd
// before every flight and collision: 1 or 3 words into a Philox block.  A
// state keeps the block's words still to come (c1..c3, or c3 alone), and a
// flight round generates the next block once for both flights.
//
// Bound by instruction issue (75 % of the issue slots).  10^9 histories of the
// 128^3 torso: 33.0 ms, 31 warp instructions per history at 27 of 32 lanes; one
// history per lane, lanes waiting for 8 to 12 others at the same step, took
// 81.4 ms, 71 instructions at 13 lanes, with the same matrix and fates.
//
// A warp holds at most 94 photons, so kPool slots suffice: an emission round
// starts with at most 31 photons at a collision, fewer photons ready to fly
// than idle lanes, and the other lanes flying -- 31 + 31 + 32 new ones with
// all lanes counted -- and no other round adds any.
constexpr int kPool = 96;           // photon states per warp
constexpr int kPoolQuads = 4;       // 16-byte words per state
constexpr int kHistThreads = 128;
constexpr int kHistWarps = kHistThreads / 32;

// A photon in flight or at a collision.  meta: bit 0 scattered before,
// bit 1 three words into the block (else one), bits 2-9 the material at the
// pending collision, bits 10-29 flights so far (at most kStepCap < 2^20), bit
// 30 in the middle of a scatter's rejection trials (c1 counts them).
// blk: the next Philox block of the history's stream.
constexpr uint32_t kTrying = 1u << 30;
struct Photon {
  float px, py, pz, dx, dy, dz, e, sig, ie3;
  uint32_t i, meta, blk, c1, c2, c3;
};

// The pool is stored as kPoolQuads planes of 16-byte words: lanes with
// consecutive slots read and write consecutive 16-byte words, four
// conflict-free instructions a state.
__device__ __forceinline__ void pool_put(uint4 (*pool)[kPool], int s, const Photon &p) {
  const auto w = [](float x) { return __float_as_uint(x); };
  pool[0][s] = make_uint4(w(p.px), w(p.py), w(p.pz), w(p.e));
  pool[1][s] = make_uint4(w(p.dx), w(p.dy), w(p.dz), w(p.sig));
  pool[2][s] = make_uint4(w(p.ie3), p.i, p.meta, p.blk);
  pool[3][s] = make_uint4(p.c1, p.c2, p.c3, 0u);
}
__device__ __forceinline__ void pool_get(uint4 (*pool)[kPool], int s, Photon &p) {
  const auto f = [](uint32_t x) { return __uint_as_float(x); };
  const uint4 a = pool[0][s], b = pool[1][s], c = pool[2][s], d = pool[3][s];
  p.px = f(a.x); p.py = f(a.y); p.pz = f(a.z); p.e = f(a.w);
  p.dx = f(b.x); p.dy = f(b.y); p.dz = f(b.z); p.sig = f(b.w);
  p.ie3 = f(c.x); p.i = c.y; p.meta = c.z; p.blk = c.w;
  p.c1 = d.x; p.c2 = d.y; p.c3 = d.z;
}

// One Woodcock flight with words (s, r) of a lane with `fly` set, without
// branches: p moves to the collision point if that is inside the grid (else
// the photon leaves from p), and on a real collision the material goes into
// meta.  The caller has checked the cap on flights.
struct Flight { bool inside, real; };
__device__ __forceinline__ Flight fly_once(const TArgs<float> &a, const float2 *s_mu, Photon &p, bool fly, uint32_t sw,
                                           uint32_t rw) {
  const float s = flight<float>(uniform<float>(sw), a);
  const float qx = p.px + s * p.dx, qy = p.py + s * p.dy, qz = p.pz + s * p.dz;
  const int ix = __float2int_rd(fmaf(qx, a.inv_h, a.hx_h));
  const int iy = __float2int_rd(fmaf(qy, a.inv_h, a.hy_h));
  const int iz = __float2int_rd(fmaf(qz, a.inv_h, a.hz_h));
  Flight f;
  f.inside = fly && (unsigned)ix < (unsigned)a.nx && (unsigned)iy < (unsigned)a.ny && (unsigned)iz < (unsigned)a.nz;
  int m = 0;
  if (f.inside) {
    m = __ldg(a.mat + (uint32_t)((iz * a.ny + iy) * a.nx + ix));
    p.px = qx; p.py = qy; p.pz = qz;
  }
  const float2 c = s_mu[m];
  const float mu = fmaf(c.x, p.sig, c.y * p.ie3);
  f.real = f.inside && uniform<float>(rw) * a.mu_maj < mu;
  if (fly) p.meta += 1u << 10;
  if (f.real) p.meta = (p.meta & ~0x3FCu) | ((uint32_t)m << 2);
  return f;
}

// Queue an escape that a view may accept (all lanes of the warp call this).
__device__ __forceinline__ void warp_queue_escape(const TArgs<float> &a, bool want, const Photon &p, uint32_t n_draws,
                                                  int lane) {
  const unsigned m = __ballot_sync(0xffffffffu, want);
  if (m == 0u) return;
  unsigned long long base = 0;
  const int leader = __ffs(m) - 1;
  if (lane == leader) base = atomicAdd(a.esc_cursor, (unsigned long long)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  const unsigned long long q = base + __popc(m & ((1u << lane) - 1u));
  if (want && q < a.esc_capacity) {
    EscapeRec<float> e;
    e.h = a.first + p.i;
    e.n_draws = n_draws;
    e.pad = 0;
    e.p[0] = p.px; e.p[1] = p.py; e.p[2] = p.pz;
    e.d[0] = p.dx; e.d[1] = p.dy; e.d[2] = p.dz;
    static_cast<EscapeRec<float> *>(a.esc)[q] = e;
  }
}

__global__ void __launch_bounds__(kHistThreads) history_kernel(const __grid_constant__ TArgs<float> a) {
  __shared__ float2 s_mu[256];
  __shared__ float s_sig[kSigTab];
  __shared__ unsigned long long s_fates[4];
  __shared__ float s_en0[2];
  __shared__ uint4 s_pool[kHistWarps][kPoolQuads][kPool];
  for (int m = threadIdx.x; m < a.n_mat; m += kHistThreads) s_mu[m] = make_float2(a.coef[3 * m], a.coef[3 * m + 1]);
  for (int i = threadIdx.x; i < kSigTab; i += kHistThreads) s_sig[i] = a.sig_tab[i];
  if (threadIdx.x < 4) s_fates[threadIdx.x] = 0ull;
  __syncthreads();
  if (threadIdx.x == 0) {
    Energy<float> e0;
    e0.set(a.e0, a, s_sig);
    s_en0[0] = e0.sig; s_en0[1] = e0.ie3;
  }
  __syncthreads();

  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  uint4 (*pool)[kPool] = s_pool[threadIdx.x >> 5];
  int n_fly = 0, n_col = 0;  // stack heights
  uint32_t base = 0, end = 0;  // histories taken from the launch and not yet emitted
  bool more = true;
  bool on = false;  // this lane holds a flying photon
  Photon p = {};
  uint32_t f_abs = 0, f_low = 0, f_esc = 0;
  for (;;) {
    const unsigned dead = __ballot_sync(0xffffffffu, !on);
    const int n_dead = __popc(dead);
    if (more && n_col < 32 && n_fly < n_dead && base >= end) {
      uint32_t b = 0;
      if (lane == 0) {
        const unsigned long long t = atomicAdd(a.work, (unsigned long long)a.grab);
        b = t < a.count ? (uint32_t)t : 0xffffffffu;
      }
      base = __shfl_sync(0xffffffffu, b, 0);
      if (base == 0xffffffffu) {
        more = false;
        base = end = 0u;
      } else {
        const uint32_t left = (uint32_t)a.count - base;
        end = base + (left < a.grab ? left : a.grab);
      }
    }
    // 1. a collision round: 32 photons wait, or nothing else is left to do
    const bool can_emit = base < end;
    const bool idle = n_dead == 32 && n_fly == 0 && !can_emit && !more;
    if (n_col >= 32 || (idle && n_col > 0)) {
      const int k = n_col < 32 ? n_col : 32;
      const bool have = lane < k;
      Photon c = {};
      if (have) pool_get(pool, kPool - n_col + lane, c);
      n_col -= k;
      __syncwarp();
      const uint64_t h = a.first + c.i;
      const int m = (int)((c.meta >> 2) & 255u);
      const float2 cm = s_mu[m];
      const float mu_pe = cm.y * c.ie3;
      const float mu = fmaf(cm.x, c.sig, mu_pe);
      bool three = (c.meta & 2u) != 0u;  // three words into the block
      // photo-absorption, else a Klein-Nishina scatter
      const bool again = (c.meta & kTrying) != 0u;  // back from an earlier round's trials
      const float u_abs = uniform<float>(three ? c.c3 : c.c1);
      bool trying = have;
      if (have && !again && u_abs * mu < mu_pe) {
        f_abs += 1;
        trying = false;
      }
      // rejection trials on pairs of words: first the rest of the block
      // (c2, c3) where it is there, then two whole blocks, two trials each;
      // the few lanes not done by then go back to the stack and take their
      // further trials in a later round
      float mu_c = 0.0f, eps = 0.0f;
      bool ok = false;
      uint32_t w0 = 0, w1 = 0, w2 = 0, w3 = 0;
      int used = 4;  // words of (w0..w3) drawn
      uint32_t trials = again ? c.c1 : 0u;
      if (trying && !again && !three) {
        ok = compton_trial<float>(c.e, c.c2, c.c3, mu_c, eps);
        trials = 1;
      }
#pragma unroll 1
      for (int b = 0; b < 2; ++b) {
        if (trying && !ok) {
          w0 = c.blk; w1 = 0u; w2 = (uint32_t)h; w3 = (uint32_t)(h >> 32);
          philox_rounds(w0, w1, w2, w3, a.rk);
          c.blk += 1;
          ok = compton_trial<float>(c.e, w0, w1, mu_c, eps);
          used = 2;
          trials += 1;
          if (!ok && trials < kTrialCap) {
            ok = compton_trial<float>(c.e, w2, w3, mu_c, eps);
            used = 4;
            trials += 1;
          }
          if (!ok && trials >= kTrialCap) {
            atomicAdd(&s_fates[MC_FATE_CAP], 1ull);
            trying = false;
          }
        }
      }
      const bool scat = trying && ok;
      if (scat && used == 4) {  // the azimuth's word opens a new block
        w0 = c.blk; w1 = 0u; w2 = (uint32_t)h; w3 = (uint32_t)(h >> 32);
        philox_rounds(w0, w1, w2, w3, a.rk);
        c.blk += 1;
      }
      bool fly = false;
      if (scat) {
        float cp, sp;
        cos_sin_2pi<float>(uniform<float>(used == 4 ? w0 : w2), cp, sp);
        rotate<float>(c.dx, c.dy, c.dz, mu_c, cp, sp);
        const float e_new = eps * c.e;
        if (e_new < a.e_low) {
          f_low += 1;
        } else {
          Energy<float> en;
          en.set(e_new, a, s_sig);
          c.e = e_new; c.sig = en.sig; c.ie3 = en.ie3;
          c.c1 = w1; c.c2 = w2; c.c3 = w3;
          c.meta = (c.meta & ~(kTrying | 2u)) | (used == 4 ? 0u : 2u) | 1u;
          fly = true;
        }
      }
      const bool back = trying && !ok;
      const unsigned mf = __ballot_sync(0xffffffffu, fly), mb = __ballot_sync(0xffffffffu, back);
      if (fly) pool_put(pool, n_fly + __popc(mf & lt), c);
      n_fly += __popc(mf);
      n_col += __popc(mb);
      if (back) {
        c.meta |= kTrying;
        c.c1 = trials;
        pool_put(pool, kPool - n_col + __popc(mb & lt), c);
      }
      __syncwarp();
      continue;
    }
    // 2. an emission round: 32 new histories and their first flight
    if (can_emit && n_fly < n_dead) {
      Photon c = {};
      c.i = base + lane;
      const bool have = c.i < end;
      base += 32;
      uint32_t b0 = 1u, b1 = 0u, b2, b3;
      {
        const uint64_t h = a.first + c.i;
        uint32_t a0 = 0u, a1 = 0u, a2 = (uint32_t)h, a3 = (uint32_t)(h >> 32);
        b2 = a2; b3 = a3;
        philox_rounds(a0, a1, a2, a3, a.rk);
        philox_rounds(b0, b1, b2, b3, a.rk);
        uint32_t v, vi, vj, vk, r;
        div_magic(a.first_v + c.i, a.n_vox, a.magic_n, v);
        vk = div_magic(v, (uint32_t)(a.nx * a.ny), a.magic_xy, r);
        vj = div_magic(r, (uint32_t)a.nx, a.magic_x, vi);
        c.px = ((float)vi + uniform<float>(a0)) * a.h - a.hx;
        c.py = ((float)vj + uniform<float>(a1)) * a.h - a.hy;
        c.pz = ((float)vk + uniform<float>(a2)) * a.h - a.hz;
        float ct = 2.0f * uniform<float>(a3) - 1.0f;
        if (a.forced_dir) ct = ct * a.band;
        float cph, sph;
        cos_sin_2pi<float>(uniform<float>(b0), cph, sph);
        const float sth = sqrt0<float>(1.0f - ct * ct);
        c.dx = sth * cph;
        c.dy = sth * sph;
        c.dz = ct;
        c.e = a.e0; c.sig = s_en0[0]; c.ie3 = s_en0[1];
        c.meta = 2u;  // after the first flight: three words into block 1
        c.blk = 2u;
        c.c3 = b3;
      }
      const bool moves = a.mu_maj > 0.0f;  // nothing attenuates: leaves at once
      const Flight f = fly_once(a, s_mu, c, have && moves, b1, b2);
      const bool esc = have && !f.inside, virt = f.inside && !f.real;
      f_esc += esc ? 1u : 0u;
      warp_queue_escape(a, esc && fabsf(c.dz) < a.w_max, c, moves ? 6u : 5u, lane);
      const unsigned mf = __ballot_sync(0xffffffffu, virt);
      const unsigned mc = __ballot_sync(0xffffffffu, f.real);
      n_col += __popc(mc);
      if (f.inside) pool_put(pool, virt ? n_fly + __popc(mf & lt) : kPool - n_col + __popc(mc & lt), c);
      n_fly += __popc(mf);
      __syncwarp();
      continue;
    }
    if (idle) break;
    // 3. a flight round
    {
      const int r = __popc(dead & lt);
      if (!on && r < n_fly) {
        pool_get(pool, n_fly - 1 - r, p);
        on = true;
      }
      n_fly -= n_fly < n_dead ? n_fly : n_dead;
      __syncwarp();
      const uint64_t h = a.first + p.i;
      uint32_t n0 = p.blk, n1 = 0u, n2 = (uint32_t)h, n3 = (uint32_t)(h >> 32);
      philox_rounds(n0, n1, n2, n3, a.rk);
      const bool three = (p.meta & 2u) != 0u;
      const bool cap1 = on && p.meta >= kStepCap << 10;
      const Flight f1 = fly_once(a, s_mu, p, on && !cap1, three ? p.c3 : p.c1, three ? n0 : p.c2);
      const bool go = f1.inside && !f1.real;
      const bool cap2 = go && p.meta >= kStepCap << 10;
      const Flight f2 = fly_once(a, s_mu, p, go && !cap2, three ? n1 : p.c3, three ? n2 : n0);
      if (cap1 || cap2) atomicAdd(&s_fates[MC_FATE_CAP], 1ull);
      const bool real = f1.real || f2.real;
      const bool esc = on && !cap1 && !cap2 && (go ? !f2.inside : !f1.inside);
      f_esc += esc ? 1u : 0u;
      // words drawn so far: the position before the round (one or three
      // words into block blk - 1), two per flight, one for the escape
      warp_queue_escape(a, esc && fabsf(p.dz) < a.w_max && !(a.primary_only && (p.meta & 1u)), p,
                        4u * p.blk - (three ? 0u : 2u) + (go ? 2u : 0u), lane);
      if (f1.real && !three) {
        p.meta |= 2u;  // the block's last word is left; the next block is not drawn from yet
      } else {
        if (f1.real) p.meta &= ~2u;
        p.c1 = n1; p.c2 = n2; p.c3 = n3;
        p.blk += 1;
      }
      const unsigned mc = __ballot_sync(0xffffffffu, real);
      n_col += __popc(mc);
      if (real) pool_put(pool, kPool - n_col + __popc(mc & lt), p);
      on = f2.inside && !f2.real;
      __syncwarp();
    }
  }
  // fates: warp sums, then one shared atomic per warp and fate
  const uint32_t f[3] = {f_abs, f_low, f_esc};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    unsigned long long c = f[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0 && c) atomicAdd(&s_fates[k], c);
  }
  __syncthreads();
  if (threadIdx.x < 4 && s_fates[threadIdx.x]) atomicAdd(&a.fates[threadIdx.x], s_fates[threadIdx.x]);
}

// The analog float path: history_kernel, then detection.
static int launch_histories(const TransportSetup &ts, cudaStream_t s) {
  if (ts.count == 0) return MC_OK;
  TArgs<float> a;
  make_targs<float>(ts, a);
  int per_sm = 0;
  MCS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, history_kernel, kHistThreads, 0));
  if (per_sm < 1) per_sm = 1;
  const int64_t full = (int64_t)device_sm_count() * per_sm;
  const int64_t need = (int64_t)((ts.count + kHistThreads - 1) / kHistThreads);
  const int grid = (int)(need < full ? need : full);
  // about eight takes per warp in a small launch, 256 histories a take in a large one
  const uint64_t per_warp = ts.count / ((uint64_t)grid * kHistWarps * 8u);
  a.grab = per_warp >= 256u ? 256u : per_warp < 32u ? 32u : (uint32_t)per_warp & ~31u;
  count_launch(); history_kernel<<<grid, kHistThreads, 0, s>>>(a);
  MCS_LAUNCHED();
  if (ts.ev_mid) MCS_CUDA(cudaEventRecord(ts.ev_mid, s));
  count_launch(); detect_kernel<float, false><<<device_sm_count() * 8, 256, 0, s>>>(a);
  MCS_LAUNCHED();
  return MC_OK;
}

}  // namespace mcs
