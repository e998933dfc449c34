// assemble.cu -- tally assembly: detection events (v, j) -> the count matrix
// C_jv of Eq. (IMC) (Sec. 5.1: T_ij estimated by Monte Carlo; Sec. 2: tallies
// are counts of histories).
//
// Events arrive as 64-bit keys v*M + j in arbitrary order (the transport
// kernel appends them with atomics), weighted ones with a fixed-point weight.
// Three ways lead to the same CSC and CSR: buckets (a thread per column and per
// row) for unweighted events in short columns and rows, sorted segments (a warp
// per column and per row of up to 1024 elements) for weighted events and longer
// ones, and a stable LSD radix sort by (v, j) with a run-length pass for columns
// beyond that, which also makes the CSR where rows are.  Everything is integer
// work, so the matrix is bit-identical from run to run.  No floating-point
// atomics.
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include <vector>

#include "internal.cuh"

namespace mcs {

// ---------------------------------------------------------------------------
// exclusive scan (u32), reduce-then-scan over tiles of 2048 elements
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *s_warp, uint32_t &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    uint32_t w = lane < nw ? s_warp[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) s_warp[lane] = w;  // inclusive per warp
  }
  __syncthreads();
  total = s_warp[(blockDim.x >> 5) - 1];
  const uint32_t before = warp > 0 ? s_warp[warp - 1] : 0u;
  return before + x - v;
}

__global__ void scan_reduce_kernel(const uint32_t *in, uint32_t *sums, int64_t n) {
  __shared__ uint32_t s_warp[32];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  uint32_t acc = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
    if (i < n) acc += in[i];
  }
  uint32_t total;
  block_exclusive_scan(acc, s_warp, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void scan_apply_kernel(const uint32_t *in, uint32_t *out, const uint32_t *offsets, int64_t n) {
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_items[kScanTile];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  // coalesced load into shared memory, then each thread scans 8 consecutive items
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
    s_items[k * kScanThreads + threadIdx.x] = i < n ? in[i] : 0u;
  }
  __syncthreads();
  uint32_t local[kScanItems];
  uint32_t acc = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    local[k] = acc;
    acc += s_items[threadIdx.x * kScanItems + k];
  }
  uint32_t total;
  const uint32_t pre = block_exclusive_scan(acc, s_warp, total) + (offsets ? offsets[blockIdx.x] : 0u);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) s_items[threadIdx.x * kScanItems + k] = pre + local[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
    if (i < n) out[i] = s_items[k * kScanThreads + threadIdx.x];
  }
}

int exclusive_scan_u32(const uint32_t *in, uint32_t *out, int64_t n, cudaStream_t s) {
  if (n <= 0) return MC_OK;
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  if (tiles == 1) {
    count_launch(); scan_apply_kernel<<<1, kScanThreads, 0, s>>>(in, out, nullptr, n);
    MCS_LAUNCHED();
    return MC_OK;
  }
  DevBuf sums, offs;
  MCS_TRY(sums.alloc(tiles * sizeof(uint32_t), s));
  MCS_TRY(offs.alloc(tiles * sizeof(uint32_t), s));
  count_launch(); scan_reduce_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(in, sums.as<uint32_t>(), n);
  MCS_LAUNCHED();
  MCS_TRY(exclusive_scan_u32(sums.as<uint32_t>(), offs.as<uint32_t>(), tiles, s));
  count_launch(); scan_apply_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(in, out, offs.as<uint32_t>(), n);
  MCS_LAUNCHED();
  return MC_OK;
}

// ---------------------------------------------------------------------------
// LSD radix sort of u64 keys (optional u32 payload), 8-bit digits
// ---------------------------------------------------------------------------
// Per pass: a histogram of the digit per tile of kSortTile keys, an exclusive
// scan of the digit-major counts (global start of each (digit, tile)), and a
// stable scatter.  The scatter first orders the tile by digit in shared
// memory, then writes the tile out in that order, so that each digit's run
// goes to consecutive addresses.  Within the tile, warp w holds the
// contiguous positions [w * 32 * kSortRounds, (w + 1) * 32 * kSortRounds):
// each warp ranks its keys among its own keys of the same digit (running
// per-warp digit counters), and a key's place in the ordered tile is the
// digit's start in the tile, plus the keys of that digit in earlier warps,
// plus its rank -- the tile order, so the sort is stable.
constexpr int kSortThreads = 256;
constexpr int kSortRounds = 12;
constexpr int kSortTile = kSortThreads * kSortRounds;  // 3072 keys

__global__ void radix_hist_kernel(const uint64_t *keys, int64_t n, int shift, uint32_t *counts, int64_t n_tiles) {
  __shared__ uint32_t s_hist[256];
  s_hist[threadIdx.x] = 0u;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kSortTile;
#pragma unroll 4
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t i = base + (int64_t)r * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&s_hist[(keys[i] >> shift) & 255u], 1u);
  }
  __syncthreads();
  counts[(int64_t)threadIdx.x * n_tiles + blockIdx.x] = s_hist[threadIdx.x];
}

// exclusive scan of one value per thread over a 256-thread block
__device__ __forceinline__ uint32_t block_exclusive_scan_256(uint32_t v, uint32_t *s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  uint32_t before = 0;
  for (int w = 0; w < warp; ++w) before += s_warp[w];
  return before + x - v;
}

// Stable scatter: the key at tile position p goes to
//   offset[digit][tile] + (number of earlier keys of this tile with the same digit).
template <bool VALS>
__global__ void __launch_bounds__(kSortThreads) radix_scatter_kernel(const uint64_t *kin, const uint32_t *vin,
                                                                     uint64_t *kout, uint32_t *vout, int64_t n,
                                                                     int shift, const uint32_t *counts,
                                                                     const uint32_t *offsets, int64_t n_tiles) {
  constexpr int kWarps = kSortThreads / 32;
  constexpr int kWarpKeys = 32 * kSortRounds;
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  __shared__ uint64_t s_keys[kSortTile];
  __shared__ uint32_t s_vals[VALS ? kSortTile : 1];
  __shared__ uint32_t s_shift[256], s_start[256], s_warp[kWarps];
  __shared__ uint32_t s_wc[kWarps][256];  // per warp and digit: keys so far, then the warp's start in the tile
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t tile_off = (int64_t)threadIdx.x * n_tiles + blockIdx.x;
  const uint32_t start = block_exclusive_scan_256(counts[tile_off], s_warp);
  s_start[threadIdx.x] = start;
  // output position of ordered-tile position p with this digit: p + shift
  // (the digit's global start minus its start in the tile, modulo 2^32)
  s_shift[threadIdx.x] = offsets[tile_off] - start;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) s_wc[w][threadIdx.x] = 0u;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kSortTile;
  const int64_t left = n - base;
  const int cnt = left < kSortTile ? (int)left : kSortTile;
  const uint32_t lt_mask = (1u << lane) - 1u;
  uint32_t *wc = s_wc[warp];
  uint64_t key[kSortRounds];
  uint32_t val[kSortRounds];
  uint32_t slot[kSortRounds];  // digit | (rank among the warp's keys of that digit) << 8
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int p = warp * kWarpKeys + r * 32 + lane;
    key[r] = p < cnt ? kin[base + p] : 0ull;
    if (VALS) val[r] = p < cnt ? vin[base + p] : 0u;
  }
  // 1. rank each key among the warp's keys of its digit, in tile order
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const bool valid = warp * kWarpKeys + r * 32 + lane < cnt;
    const uint32_t digit = valid ? (uint32_t)((key[r] >> shift) & 255u) : 256u;
    // lanes holding the same digit: one vote per digit bit (and one on
    // validity), intersected -- measured faster in this kernel than
    // match.any (the same masks)
    uint32_t peers = __ballot_sync(0xffffffffu, valid);
    if (!valid) peers = ~peers;
#pragma unroll
    for (int bit = 0; bit < 8; ++bit) {
      const uint32_t bb = __ballot_sync(0xffffffffu, (digit >> bit) & 1u);
      peers &= ((digit >> bit) & 1u) ? bb : ~bb;
    }
    const int leader = __ffs(peers) - 1;
    uint32_t before = 0u;
    if (valid && lane == leader) before = wc[digit];
    before = __shfl_sync(0xffffffffu, before, leader);
    if (valid && lane == leader) wc[digit] = before + __popc(peers);
    __syncwarp();
    slot[r] = valid ? digit | ((before + __popc(peers & lt_mask)) << 8) : kNone;
  }
  __syncthreads();
  // 2. per digit: each warp's start in the ordered tile
  {
    uint32_t run = s_start[threadIdx.x];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = s_wc[w][threadIdx.x];
      s_wc[w][threadIdx.x] = run;
      run += c;
    }
  }
  __syncthreads();
  // 3. order the tile by digit in shared memory
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    if (slot[r] != kNone) {
      const uint32_t pos = wc[slot[r] & 255u] + (slot[r] >> 8);
      s_keys[pos] = key[r];
      if (VALS) s_vals[pos] = val[r];
    }
  }
  __syncthreads();
  // 4. write the tile out in digit order: each digit's keys are consecutive
  for (int p = threadIdx.x; p < cnt; p += kSortThreads) {
    const uint64_t k = s_keys[p];
    const uint32_t pos = (uint32_t)p + s_shift[(uint32_t)((k >> shift) & 255u)];
    kout[pos] = k;
    if (VALS) vout[pos] = s_vals[p];
  }
}

int radix_sort_u64(uint64_t *keys, uint64_t *keys_alt, uint32_t *vals, uint32_t *vals_alt, int64_t n, int bits,
                   bool *result_in_alt, cudaStream_t s, int first_bit) {
  *result_in_alt = false;
  if (n <= 1 || bits <= 0) return MC_OK;
  if (n >= (int64_t)0xFFFFFFFFll) {
    set_error("radix sort: %lld keys exceed the 32-bit offset range", (long long)n);
    return MC_EINVAL;
  }
  const int64_t n_tiles = (n + kSortTile - 1) / kSortTile;
  DevBuf counts, offsets;
  MCS_TRY(counts.alloc(256 * n_tiles * sizeof(uint32_t), s));
  MCS_TRY(offsets.alloc(256 * n_tiles * sizeof(uint32_t), s));
  uint64_t *kin = keys, *kout = keys_alt;
  uint32_t *vin = vals, *vout = vals_alt;
  bool in_alt = false;
  for (int shift = first_bit; shift < bits; shift += 8) {
    count_launch(); radix_hist_kernel<<<(unsigned)n_tiles, kSortThreads, 0, s>>>(kin, n, shift, counts.as<uint32_t>(), n_tiles);
    MCS_LAUNCHED();
    MCS_TRY(exclusive_scan_u32(counts.as<uint32_t>(), offsets.as<uint32_t>(), 256 * n_tiles, s));
    count_launch();
    if (vin)
      radix_scatter_kernel<true><<<(unsigned)n_tiles, kSortThreads, 0, s>>>(kin, vin, kout, vout, n, shift,
                                                                           counts.as<uint32_t>(),
                                                                           offsets.as<uint32_t>(), n_tiles);
    else
      radix_scatter_kernel<false><<<(unsigned)n_tiles, kSortThreads, 0, s>>>(kin, nullptr, kout, nullptr, n, shift,
                                                                            counts.as<uint32_t>(),
                                                                            offsets.as<uint32_t>(), n_tiles);
    MCS_LAUNCHED();
    uint64_t *tk = kin; kin = kout; kout = tk;
    uint32_t *tv = vin; vin = vout; vout = tv;
    in_alt = !in_alt;
  }
  *result_in_alt = in_alt;
  return MC_OK;
}

// ---------------------------------------------------------------------------
// run-length encoding of sorted keys
// ---------------------------------------------------------------------------
__global__ void head_flags_kernel(const uint64_t *keys, int64_t n, uint32_t *flags) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    flags[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

__global__ void compact_heads_kernel(const uint64_t *keys, const uint32_t *flags, const uint32_t *idx, int64_t n,
                                     uint64_t *ukeys, uint32_t *upos) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (flags[i]) {
      ukeys[idx[i]] = keys[i];
      upos[idx[i]] = (uint32_t)i;
    }
  }
}

__global__ void run_lengths_kernel(const uint32_t *upos, int64_t nu, int64_t n, uint32_t *cnt) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += (int64_t)gridDim.x * blockDim.x)
    cnt[u] = (u + 1 < nu ? upos[u + 1] : (uint32_t)n) - upos[u];
}

// (v*M + j) -> row j, column v; histogram of the column (or row) index.
__global__ void split_keys_kernel(const uint64_t *ukeys, int64_t nu, uint64_t m, uint32_t *major_out,
                                  uint32_t *minor_out, uint32_t *major_hist) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = ukeys[u];
    const uint32_t major = (uint32_t)(k / m), minor = (uint32_t)(k % m);
    if (major_out) major_out[u] = major;
    minor_out[u] = minor;
    atomicAdd(&major_hist[major], 1u);
  }
}

// Pointer array of a sorted sequence of major indices: ptr[c] = the first
// position whose major index is >= c, ptr[n_major] = nu.  Position u writes
// the entries c in (major of u - 1, major of u] (the last position also
// (major, n_major]), so every entry is written once and no histogram or scan
// is needed.
__device__ __forceinline__ void fill_ptr(uint32_t *ptr, int64_t u, int64_t nu, int64_t major, int64_t prev,
                                         int64_t n_major) {
  for (int64_t c = prev + 1; c <= major; ++c) ptr[c] = (uint32_t)u;
  if (u == nu - 1)
    for (int64_t c = major + 1; c <= n_major; ++c) ptr[c] = (uint32_t)nu;
}

// Sorted unique keys v*M + j -> CSC row indices j, col_ptr, and the
// transposed keys (j << b) | v for the CSR.  The loop runs the same number of
// times on every thread of a block (the shuffle needs whole warps).
__global__ void csc_split_kernel(const uint64_t *ukeys, int64_t nu, uint64_t m, int b, uint32_t *row_idx,
                                 uint32_t *col_ptr, int64_t n_cols, uint64_t *tkeys) {
  const int lane = threadIdx.x & 31;
  for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x; u0 < nu; u0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = u0 + threadIdx.x;
    const bool valid = u < nu;
    const uint64_t k = valid ? ukeys[u] : 0ull;
    const uint64_t v = k / m, j = k - v * m;
    uint64_t vp = __shfl_up_sync(0xffffffffu, v, 1);
    if (lane == 0) vp = (valid && u > 0) ? ukeys[u - 1] / m : 0ull;
    if (valid) {
      row_idx[u] = (uint32_t)j;
      tkeys[u] = (j << b) | v;
      fill_ptr(col_ptr, u, nu, (int64_t)v, u == 0 ? -1 : (int64_t)vp, n_cols);
    }
  }
}

// Sorted keys (j << b) | v -> CSR column indices v and row_ptr.
__global__ void csr_split_kernel(const uint64_t *tkeys, int64_t nu, int b, uint32_t *col_idx, uint32_t *row_ptr,
                                 int64_t n_rows) {
  const uint64_t mask = (1ull << b) - 1ull;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = tkeys[u];
    col_idx[u] = (uint32_t)(k & mask);
    fill_ptr(row_ptr, u, nu, (int64_t)(k >> b), u == 0 ? -1 : (int64_t)(tkeys[u - 1] >> b), n_rows);
  }
}

// n_v = #{h in [first, first+count) : h mod N = v}
__global__ void histories_per_voxel_kernel(uint64_t first, uint64_t count, uint64_t n_vox, uint32_t *n_v,
                                           float *inv_n) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_vox; v += (uint64_t)gridDim.x * blockDim.x) {
    // number of h in [0, x) with h = v (mod N)
    auto below = [&](uint64_t x) -> uint64_t { return x > v ? (x - v - 1) / n_vox + 1 : 0; };
    const uint64_t c = below(first + count) - below(first);
    n_v[v] = (uint32_t)c;
    inv_n[v] = c ? (float)(1.0 / (double)c) : 0.0f;
  }
}

// S_v = sum_j C_jv over CSC column v, and the largest count.
__global__ void column_sums_kernel(const uint32_t *col_ptr, const uint32_t *cnt, int64_t n_cols, double *colsum,
                                   float *inv_colsum, unsigned int *max_count) {
  uint32_t mymax = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_cols; v += (int64_t)gridDim.x * blockDim.x) {
    uint64_t acc = 0;
    for (uint32_t k = col_ptr[v]; k < col_ptr[v + 1]; ++k) {
      acc += cnt[k];
      mymax = cnt[k] > mymax ? cnt[k] : mymax;
    }
    colsum[v] = (double)acc;
    inv_colsum[v] = acc ? (float)(1.0 / (double)acc) : 0.0f;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, mymax, o);
    mymax = y > mymax ? y : mymax;
  }
  if ((threadIdx.x & 31) == 0 && mymax) atomicMax(max_count, mymax);
}

// Weighted tallies (forced detection): the weight sum of each run of equal
// keys, wsum[u] = sum of w[perm[e]] over the run's sorted positions e, as an
// exact 64-bit integer sum (the weights are fixed point).
__global__ void iota_kernel(uint32_t *out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (uint32_t)i;
}

// A CSC entry's weight sum and count side by side, so that the CSR can
// gather both with one 16-byte load.
struct alignas(16) WEntry {
  uint64_t w;
  uint32_t cnt, pad;
};

__global__ void run_weights_kernel(const uint32_t *upos, const uint32_t *ucnt, int64_t nu, const uint32_t *perm,
                                   const uint64_t *w, uint64_t *wsum, WEntry *ent) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += (int64_t)gridDim.x * blockDim.x) {
    uint64_t acc = 0;
    const uint32_t c = ucnt[u], b = upos[u], e = b + c;
    for (uint32_t k = b; k < e; ++k) acc += w[perm[k]];
    wsum[u] = acc;
    WEntry x;
    x.w = acc; x.cnt = c; x.pad = 0u;
    ent[u] = x;
  }
}

// out_cnt[i] = ent[perm[i]].cnt, out_w[i] = ent[perm[i]].w
__global__ void gather_entries_kernel(const uint32_t *perm, int64_t n, const WEntry *ent, uint32_t *out_cnt,
                                      uint64_t *out_w) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const WEntry x = ent[perm[i]];
    out_cnt[i] = x.cnt;
    out_w[i] = x.w;
  }
}

// S_v = sum over column v of the fixed-point weights, in column order
__global__ void column_weight_sums_kernel(const uint32_t *col_ptr, const uint64_t *wq, int64_t n_cols, double *colsum,
                                          float *inv_colsum) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_cols; v += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (uint32_t k = col_ptr[v]; k < col_ptr[v + 1]; ++k) acc += (double)wq[k] * (1.0 / kFdScale);
    colsum[v] = acc;
    inv_colsum[v] = acc > 0.0 ? (float)(1.0 / acc) : 0.0f;
  }
}

static int grid_for(int64_t n, int threads = 256) {
  int64_t g = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)device_sm_count() * 32;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

static int bits_for(uint64_t range) {
  int b = 0;
  while (b < 64 && (range >> b) != 0) ++b;
  return b;
}

// Quotient of a key by a fixed divisor: the estimate by floor((2^64 - 1) / m)
// is the true quotient or one less.
struct Div64 { uint64_t m, magic; };
static Div64 make_div(uint64_t m) { return Div64{m, ~0ull / m}; }
__device__ __forceinline__ uint64_t div_key(uint64_t k, const Div64 &d) {
  const uint64_t q = __umul64hi(k, d.magic);
  return k - q * d.m >= d.m ? q + 1 : q;
}

// ---------------------------------------------------------------------------
// assembly by buckets (unweighted events, short columns and rows)
// ---------------------------------------------------------------------------
// Events are counted per column and each event's row is placed in its
// column's bucket (in any order); every bucket is then sorted by row, one
// thread per bucket, with equal rows merged into a count.  The CSR is made
// the same way from the CSC entries.  Sorting makes the result unique: the
// same sorted, merged CSC and CSR as the radix path, in a few passes over
// the events instead of one per digit.  Taken only when no column holds more
// than kBucketLen events and no row more than kBucketLen entries.
constexpr int kBucketLen = 64;

__global__ void bucket_count_kernel(const uint64_t *keys, int64_t n, Div64 m, uint32_t *cnt) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&cnt[div_key(keys[i], m)], 1u);
}

// event i -> its row, at start[column] + (its place among the column's
// events, in arrival order at the atomic)
__global__ void bucket_fill_kernel(const uint64_t *keys, int64_t n, Div64 m, const uint32_t *start,
                                   uint32_t *cursor, uint32_t *minor) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = keys[i];
    const uint64_t v = div_key(k, m);
    minor[start[v] + atomicAdd(&cursor[v], 1u)] = (uint32_t)(k - v * m.m);
  }
}

// Compare-exchange of (a[i], w[i]) and (a[k], w[k]) by a.
__device__ __forceinline__ void cmp_swap(uint32_t &ai, uint32_t &wi, uint32_t &ak, uint32_t &wk) {
  if (ak < ai) {
    const uint32_t t = ai, u = wi;
    ai = ak; wi = wk;
    ak = t; wk = u;
  }
}

// Sort bucket c = [start[c], start[c + 1]) of `minor` ascending, with its
// payload (cnt_in, or 1 per element when cnt_in is NULL), merge equal
// values (payloads summed) and write the u merged values and payloads to
// the bucket's first u places of minor and cnt_out; uniq[c] = u.  Buckets of
// up to 8 elements are sorted in registers (Batcher's odd-even merge
// network, unused places holding the largest value); longer ones, up to
// kBucketLen, by insertion in a local array.  A longer bucket sets
// *overflow and is left as it is.
__global__ void bucket_sort_merge_kernel(const uint32_t *start, int64_t n_major, uint32_t *minor,
                                         const uint32_t *cnt_in, uint32_t *cnt_out, uint32_t *uniq,
                                         unsigned int *overflow) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_major;
       c += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t b = start[c];
    const int len = (int)(start[c + 1] - b);
    if (len > kBucketLen) {
      atomicOr(overflow, 1u);
      continue;
    }
    if (len <= 8) {
      uint32_t r[8], q[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        r[k] = k < len ? minor[b + k] : 0xffffffffu;
        q[k] = k < len ? (cnt_in ? cnt_in[b + k] : 1u) : 0u;
      }
      // odd-even merge sort of 8: sorted pairs, fours, then eight
#pragma unroll
      for (int k = 0; k < 8; k += 2) cmp_swap(r[k], q[k], r[k + 1], q[k + 1]);
#pragma unroll
      for (int k = 0; k < 8; k += 4) {
        cmp_swap(r[k], q[k], r[k + 2], q[k + 2]);
        cmp_swap(r[k + 1], q[k + 1], r[k + 3], q[k + 3]);
        cmp_swap(r[k + 1], q[k + 1], r[k + 2], q[k + 2]);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) cmp_swap(r[k], q[k], r[k + 4], q[k + 4]);
      cmp_swap(r[2], q[2], r[4], q[4]);
      cmp_swap(r[3], q[3], r[5], q[5]);
      cmp_swap(r[1], q[1], r[2], q[2]);
      cmp_swap(r[3], q[3], r[4], q[4]);
      cmp_swap(r[5], q[5], r[6], q[6]);
      // merge equal values and write, all from registers (the loads are done)
      int u = 0;
      uint32_t last = 0u, acc = 0u;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (k < len) {
          if (u > 0 && r[k] == last) {
            acc += q[k];
          } else {
            if (u > 0) {
              minor[b + u - 1] = last;
              cnt_out[b + u - 1] = acc;
            }
            last = r[k];
            acc = q[k];
            ++u;
          }
        }
      }
      if (u > 0) {
        minor[b + u - 1] = last;
        cnt_out[b + u - 1] = acc;
      }
      uniq[c] = (uint32_t)u;
      continue;
    }
    uint32_t a[kBucketLen], w[kBucketLen];
    {
      for (int k = 0; k < len; ++k) {  // insertion sort while loading
        const uint32_t x = minor[b + k], y = cnt_in ? cnt_in[b + k] : 1u;
        int t = k;
        for (; t > 0 && a[t - 1] > x; --t) {
          a[t] = a[t - 1];
          w[t] = w[t - 1];
        }
        a[t] = x;
        w[t] = y;
      }
    }
    int u = 0;
    for (int k = 0; k < len; ++k) {
      if (u > 0 && a[k] == a[u - 1]) {
        w[u - 1] += w[k];
      } else {
        a[u] = a[k];
        w[u] = w[k];
        ++u;
      }
    }
    for (int k = 0; k < u; ++k) {
      minor[b + k] = a[k];
      cnt_out[b + k] = w[k];
    }
    uniq[c] = (uint32_t)u;
  }
}

// CSC: bucket c's merged entries to [col_ptr[c], col_ptr[c + 1]), and the
// number of entries of each row
__global__ void bucket_compact_kernel(const uint32_t *start, const uint32_t *col_ptr, int64_t n_cols,
                                      const uint32_t *minor, const uint32_t *cnt, uint32_t *row_idx,
                                      uint32_t *csc_cnt, uint32_t *row_hist) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_cols;
       c += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t b = start[c], o = col_ptr[c], u = col_ptr[c + 1] - o;
    for (uint32_t k = 0; k < u; ++k) {
      const uint32_t j = minor[b + k];
      row_idx[o + k] = j;
      csc_cnt[o + k] = cnt[b + k];
      atomicAdd(&row_hist[j], 1u);
    }
  }
}

// CSR buckets: every CSC entry (j, v) to row j's bucket (any order)
__global__ void transpose_fill_kernel(const uint32_t *col_ptr, int64_t n_cols, const uint32_t *row_idx,
                                      const uint32_t *csc_cnt, const uint32_t *row_ptr, uint32_t *cursor,
                                      uint32_t *col_idx, uint32_t *csr_cnt) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_cols;
       c += (int64_t)gridDim.x * blockDim.x) {
    for (uint32_t k = col_ptr[c]; k < col_ptr[c + 1]; ++k) {
      const uint32_t j = row_idx[k];
      const uint32_t pos = row_ptr[j] + atomicAdd(&cursor[j], 1u);
      col_idx[pos] = (uint32_t)c;
      csr_cnt[pos] = csc_cnt[k];
    }
  }
}

// The CSC and CSR of n > 0 unweighted events by buckets.  Sets *done, or
// leaves the system's matrix unfinished (and the keys untouched) when a
// column or a row is too long for a bucket.
static int assemble_buckets(mc_system *sys, const uint64_t *keys, int64_t n, cudaStream_t s, bool *done) {
  *done = false;
  const int64_t M = sys->n_rows, N = sys->n_cols;
  const Div64 dm = make_div((uint64_t)M);
  DevBuf ccnt, start, flag;
  MCS_TRY(ccnt.alloc((size_t)(N + 1) * sizeof(uint32_t), s));
  MCS_TRY(start.alloc((size_t)(N + 1) * sizeof(uint32_t), s));
  MCS_TRY(flag.alloc(sizeof(unsigned int), s));
  MCS_CUDA(cudaMemsetAsync(ccnt.p, 0, (size_t)(N + 1) * sizeof(uint32_t), s));
  MCS_CUDA(cudaMemsetAsync(flag.p, 0, sizeof(unsigned int), s));
  count_launch(); bucket_count_kernel<<<grid_for(n), 256, 0, s>>>(keys, n, dm, ccnt.as<uint32_t>());
  MCS_LAUNCHED();
  MCS_TRY(exclusive_scan_u32(ccnt.as<uint32_t>(), start.as<uint32_t>(), N + 1, s));
  // events into column buckets, sorted and merged
  DevBuf minor, ecnt;
  MCS_TRY(minor.alloc((size_t)n * sizeof(uint32_t), s));
  MCS_TRY(ecnt.alloc((size_t)n * sizeof(uint32_t), s));
  MCS_CUDA(cudaMemsetAsync(ccnt.p, 0, (size_t)(N + 1) * sizeof(uint32_t), s));  // now the bucket cursors
  count_launch();
  bucket_fill_kernel<<<grid_for(n), 256, 0, s>>>(keys, n, dm, start.as<uint32_t>(), ccnt.as<uint32_t>(),
                                                 minor.as<uint32_t>());
  MCS_LAUNCHED();
  // ccnt becomes the merged entries per column (ccnt[N] stays 0 for the scan)
  count_launch();
  bucket_sort_merge_kernel<<<grid_for(N), 256, 0, s>>>(start.as<uint32_t>(), N, minor.as<uint32_t>(), nullptr,
                                                       ecnt.as<uint32_t>(), ccnt.as<uint32_t>(),
                                                       flag.as<unsigned int>());
  MCS_LAUNCHED();
  MCS_TRY(sys->col_ptr.alloc((size_t)(N + 1) * sizeof(uint32_t), s));
  MCS_TRY(exclusive_scan_u32(ccnt.as<uint32_t>(), sys->col_ptr.as<uint32_t>(), N + 1, s));
  uint32_t nnz = 0, too_long = 0;
  MCS_CUDA(cudaMemcpyAsync(&nnz, sys->col_ptr.as<uint32_t>() + N, sizeof(nnz), cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaMemcpyAsync(&too_long, flag.p, sizeof(too_long), cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaStreamSynchronize(s));
  if (too_long) return MC_OK;  // a column of more than kBucketLen events
  const size_t nnz_b = (size_t)(nnz > 0 ? nnz : 1);
  MCS_TRY(sys->row_idx.alloc(nnz_b * sizeof(uint32_t), s));
  MCS_TRY(sys->csc_cnt.alloc(nnz_b * sizeof(uint32_t), s));
  DevBuf rhist;
  MCS_TRY(rhist.alloc((size_t)(M + 1) * sizeof(uint32_t), s));
  MCS_CUDA(cudaMemsetAsync(rhist.p, 0, (size_t)(M + 1) * sizeof(uint32_t), s));
  count_launch();
  bucket_compact_kernel<<<grid_for(N), 256, 0, s>>>(start.as<uint32_t>(), sys->col_ptr.as<uint32_t>(), N,
                                                    minor.as<uint32_t>(), ecnt.as<uint32_t>(),
                                                    sys->row_idx.as<uint32_t>(), sys->csc_cnt.as<uint32_t>(),
                                                    rhist.as<uint32_t>());
  MCS_LAUNCHED();
  minor.release();
  ecnt.release();
  start.release();
  ccnt.release();
  // CSR: the CSC entries into row buckets, each sorted by column
  MCS_TRY(sys->row_ptr.alloc((size_t)(M + 1) * sizeof(uint32_t), s));
  MCS_TRY(exclusive_scan_u32(rhist.as<uint32_t>(), sys->row_ptr.as<uint32_t>(), M + 1, s));
  MCS_TRY(sys->col_idx.alloc(nnz_b * sizeof(uint32_t), s));
  MCS_TRY(sys->csr_cnt.alloc(nnz_b * sizeof(uint32_t), s));
  MCS_CUDA(cudaMemsetAsync(rhist.p, 0, (size_t)(M + 1) * sizeof(uint32_t), s));  // the row cursors
  count_launch();
  transpose_fill_kernel<<<grid_for(N), 256, 0, s>>>(sys->col_ptr.as<uint32_t>(), N, sys->row_idx.as<uint32_t>(),
                                                    sys->csc_cnt.as<uint32_t>(), sys->row_ptr.as<uint32_t>(),
                                                    rhist.as<uint32_t>(), sys->col_idx.as<uint32_t>(),
                                                    sys->csr_cnt.as<uint32_t>());
  MCS_LAUNCHED();
  // rows hold distinct columns: the sort leaves every entry (rhist takes the
  // per-row counts, unused)
  count_launch();
  bucket_sort_merge_kernel<<<grid_for(M), 256, 0, s>>>(sys->row_ptr.as<uint32_t>(), M, sys->col_idx.as<uint32_t>(),
                                                       sys->csr_cnt.as<uint32_t>(), sys->csr_cnt.as<uint32_t>(),
                                                       rhist.as<uint32_t>(), flag.as<unsigned int>());
  MCS_LAUNCHED();
  MCS_CUDA(cudaMemcpyAsync(&too_long, flag.p, sizeof(too_long), cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaStreamSynchronize(s));
  if (too_long) return MC_OK;  // a row of more than kBucketLen entries
  sys->nnz = nnz;
  *done = true;
  return MC_OK;
}

// The CSR of the nu > 0 entries whose keys (j << b) | v, b = bits of N - 1, stand
// in CSC order: sorted with the counts `cnt` (or, weighted, the CSC position of
// each entry, whose weight and count `went` holds) as payload, then columns and
// row_ptr (allocated by the caller) in sorted order.  tkeys and cnt are used up.
static int csr_by_radix(mc_system *sys, DevBuf &tkeys, DevBuf &cnt, DevBuf &went, int64_t nu, cudaStream_t s) {
  const int64_t M = sys->n_rows;
  const int b = bits_for((uint64_t)sys->n_cols - 1);
  DevBuf tkeys_alt, tcnt_alt, tperm;
  MCS_TRY(sys->col_idx.alloc((size_t)nu * sizeof(uint32_t), s));
  MCS_TRY(sys->csr_cnt.alloc((size_t)nu * sizeof(uint32_t), s));
  MCS_TRY(tkeys_alt.alloc((size_t)nu * sizeof(uint64_t), s));
  MCS_TRY(tcnt_alt.alloc((size_t)nu * sizeof(uint32_t), s));
  if (sys->weighted) {
    MCS_TRY(tperm.alloc((size_t)nu * sizeof(uint32_t), s));
    count_launch(); iota_kernel<<<grid_for(nu), 256, 0, s>>>(tperm.as<uint32_t>(), nu);
    MCS_LAUNCHED();
  }
  uint32_t *payload = sys->weighted ? tperm.as<uint32_t>() : cnt.as<uint32_t>();
  bool talt = false;
  // the entries are in (v, j) order: a stable sort on the j bits of
  // (j << b) | v alone gives (j, v) order
  MCS_TRY(radix_sort_u64(tkeys.as<uint64_t>(), tkeys_alt.as<uint64_t>(), payload, tcnt_alt.as<uint32_t>(), nu,
                         b + bits_for((uint64_t)M - 1), &talt, s, b));
  const uint64_t *tk = talt ? tkeys_alt.as<uint64_t>() : tkeys.as<uint64_t>();
  const uint32_t *tc = talt ? tcnt_alt.as<uint32_t>() : payload;
  count_launch();
  csr_split_kernel<<<grid_for(nu), 256, 0, s>>>(tk, nu, b, sys->col_idx.as<uint32_t>(), sys->row_ptr.as<uint32_t>(), M);
  MCS_LAUNCHED();
  if (sys->weighted) {
    MCS_TRY(sys->csr_wq.alloc((size_t)nu * sizeof(uint64_t), s));
    count_launch();
    gather_entries_kernel<<<grid_for(nu), 256, 0, s>>>(tc, nu, went.as<WEntry>(), sys->csr_cnt.as<uint32_t>(),
                                                       sys->csr_wq.as<uint64_t>());
    MCS_LAUNCHED();
  } else {
    MCS_CUDA(cudaMemcpyAsync(sys->csr_cnt.p, tc, (size_t)nu * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
  }
  return MC_OK;
}

// ---------------------------------------------------------------------------
// assembly by sorted segments (weighted events, and columns or rows too long
// for the buckets above)
// ---------------------------------------------------------------------------
// The events are placed in their columns' segments as above; a warp then
// sorts each column by row in its registers, counts the distinct rows, and,
// once the column pointers are known, sorts again and writes the merged
// entries, their projector values and the column sums.  The CSR is made the
// same way: entries placed in their rows' segments, a warp per row (by radix
// sort where a row has more than kSegLen entries).  Sorting twice (~2 warp
// instructions per event) is cheaper than writing the sorted events out and
// reading them back.  Integer work on whole segments, so the matrix does not
// depend on the order of arrival.
//
// Bound by the placement passes (a scattered store per entry, and a returning
// atomic per run of events of one column) and by memory otherwise: about 110
// bytes a weighted event in all against ~310 for the radix sort's nine passes
// and its gather.  2.6e8 weighted events of a forced-detection build: 38.3 ->
// 18.3 ms; 7.3e7 counted events in columns of ~35 (which the buckets tried
// first, in vain): 14.4 -> 6.7 ms, with its first projections.
constexpr int kSegLen = 1024;  // longest segment: 32 elements per lane
// Segments of up to 256 elements and longer ones are two launches of each
// kernel: with 8 keys a lane instead of 32 an SM holds twice the warps.
constexpr int kShortK = 8;
constexpr int kRowBlocks = 1024;  // row blocks of the two-pass transpose, at most

__device__ __forceinline__ uint32_t key_min(uint32_t a, uint32_t b) { return min(a, b); }
__device__ __forceinline__ uint32_t key_max(uint32_t a, uint32_t b) { return max(a, b); }
__device__ __forceinline__ uint64_t key_min(uint64_t a, uint64_t b) { return a < b ? a : b; }
__device__ __forceinline__ uint64_t key_max(uint64_t a, uint64_t b) { return a < b ? b : a; }

// Ascending bitonic sort of 32 K keys over a warp, element lane K + k in
// r[k].  Each merge starts with a comparison against the mirrored position,
// so that every comparison puts the smaller key first.  Blocked order keeps
// all but 15 of the stages inside the lanes.
template <int K, typename Key> __device__ __forceinline__ void warp_sort(Key (&r)[K], int lane) {
#pragma unroll
  for (int size = 2; size <= K; size <<= 1) {
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int j = i ^ (size - 1);
      if (j > i) { const Key a = key_min(r[i], r[j]), b = key_max(r[i], r[j]); r[i] = a; r[j] = b; }
    }
#pragma unroll
    for (int d = size / 4; d > 0; d >>= 1)
#pragma unroll
      for (int i = 0; i < K; ++i)
        if (!(i & d)) { const Key a = key_min(r[i], r[i + d]), b = key_max(r[i], r[i + d]); r[i] = a; r[i + d] = b; }
  }
#pragma unroll
  for (int lanes = 2; lanes <= 32; lanes <<= 1) {
    Key o[K];
#pragma unroll
    for (int k = 0; k < K; ++k) o[k] = __shfl_xor_sync(0xffffffffu, r[K - 1 - k], lanes - 1);
    const bool low0 = !(lane & (lanes >> 1));
#pragma unroll
    for (int k = 0; k < K; ++k) r[k] = low0 ? key_min(r[k], o[k]) : key_max(r[k], o[k]);
#pragma unroll
    for (int d = lanes / 4; d > 0; d >>= 1) {
      const bool low = !(lane & d);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const Key x = __shfl_xor_sync(0xffffffffu, r[k], d);
        r[k] = low ? key_min(r[k], x) : key_max(r[k], x);
      }
    }
#pragma unroll
    for (int d = K / 2; d > 0; d >>= 1)
#pragma unroll
      for (int i = 0; i < K; ++i)
        if (!(i & d)) { const Key a = key_min(r[i], r[i + d]), b = key_max(r[i], r[i + d]); r[i] = a; r[i + d] = b; }
  }
}

// Sort the len <= 32 K keys key(0..len-1), unused places last; with `out`
// (shared memory, 32 K keys) the sorted keys are left there.  Returns the
// number of distinct keys >> lb where out is NULL.
template <int K, typename Key, typename F>
__device__ __forceinline__ uint32_t sort_segment(uint32_t len, int lb, int lane, Key *out, const F &key) {
  Key r[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t e = 32u * k + lane;
    r[k] = e < len ? key(e) : ~(Key)0;
  }
  warp_sort<K, Key>(r, lane);
  if (out) {
#pragma unroll
    for (int k = 0; k < K; ++k) out[lane * K + k] = r[k];
    __syncwarp();
    return 0u;
  }
  Key prev = __shfl_up_sync(0xffffffffu, r[K - 1], 1);
  uint32_t n = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t e = (uint32_t)(lane * K + k);
    n += e < len && (e == 0u || (prev >> lb) != (r[k] >> lb)) ? 1u : 0u;
    prev = r[k];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  return n;
}

// ... with K the smallest power of two that holds len (MAXK at most)
template <int MAXK, typename Key, typename F>
__device__ __forceinline__ uint32_t sort_segment_any(uint32_t len, int lb, int lane, Key *out, const F &key) {
  if (len <= 32) return sort_segment<1, Key>(len, lb, lane, out, key);
  if (len <= 64) return sort_segment<2, Key>(len, lb, lane, out, key);
  if (len <= 128) return sort_segment<4, Key>(len, lb, lane, out, key);
  if (MAXK <= 8 || len <= 256) return sort_segment<8, Key>(len, lb, lane, out, key);
  if (len <= 512) return sort_segment<(MAXK > 8 ? 16 : 8), Key>(len, lb, lane, out, key);
  return sort_segment<MAXK, Key>(len, lb, lane, out, key);
}

__global__ void max_value_kernel(const uint32_t *v, int64_t n, unsigned int *out) {
  uint32_t mx = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    mx = max(mx, v[i]);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(out, mx);
}

// Events per column; neighbouring events of one column (forced detection
// appends a record's copies together) take one atomic.
__global__ void segment_count_kernel(const uint64_t *keys, int64_t n, Div64 m, uint32_t *cnt) {
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane; i0 < n; i0 += (int64_t)gridDim.x * blockDim.x) {
    const bool valid = i0 + lane < n;
    const uint32_t v = valid ? (uint32_t)div_key(keys[i0 + lane], m) : 0xffffffffu;
    const uint32_t vp = __shfl_up_sync(0xffffffffu, v, 1);
    const bool head = lane == 0 || v != vp;
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    if (head && valid) {
      const unsigned later = lane < 31 ? heads >> (lane + 1) : 0u;
      atomicAdd(&cnt[v], later ? (uint32_t)__ffs(later) : 32u - lane);
    }
  }
}

// Events into their columns' segments: cursor[v] starts at the segment's
// first place.  Four rounds of a warp are in flight at once (the atomics
// return a place each).
template <bool W>
__global__ void __launch_bounds__(256) segment_fill_kernel(const uint64_t *keys, const uint64_t *weights, int64_t n,
                                                         Div64 m, uint32_t *cursor, uint32_t *rows, uint64_t *w) {
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i0 = warp * (32 * U); i0 < n; i0 += n_warps * (32 * U)) {
    uint32_t row[U], place[U];
    uint64_t wt[U];
    int leader[U];
    bool valid[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + 32 * u + lane;
      valid[u] = i < n;
      const uint64_t k = valid[u] ? keys[i] : 0ull;
      if (W) wt[u] = valid[u] ? weights[i] : 0ull;
      const uint64_t q = div_key(k, m);
      row[u] = (uint32_t)(k - q * m.m);
      const uint32_t v = valid[u] ? (uint32_t)q : 0xffffffffu;
      const uint32_t vp = __shfl_up_sync(0xffffffffu, v, 1);
      const bool head = lane == 0 || v != vp;
      const unsigned heads = __ballot_sync(0xffffffffu, head);
      leader[u] = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
      place[u] = 0u;
      if (head && valid[u]) {
        const unsigned later = lane < 31 ? heads >> (lane + 1) : 0u;
        place[u] = atomicAdd(&cursor[v], later ? (uint32_t)__ffs(later) : 32u - lane);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t p = __shfl_sync(0xffffffffu, place[u], leader[u]) + (uint32_t)(lane - leader[u]);
      if (valid[u]) {
        rows[p] = row[u];
        if (W) w[p] = wt[u];
      }
    }
  }
}

constexpr int kSegThreads = 256;

// distinct rows of each column
template <int MAXK>
__global__ void __launch_bounds__(kSegThreads) segment_unique_kernel(const uint32_t *start, int64_t n_seg,
                                                                  uint32_t shortest, const uint32_t *rows,
                                                                  uint32_t *uniq) {
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = ((int64_t)gridDim.x * kSegThreads) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * kSegThreads + threadIdx.x) >> 5; c < n_seg; c += n_warps) {
    const uint32_t b = start[c], len = start[c + 1] - b;
    if (len < shortest || len > 32u * MAXK) continue;  // another launch's
    uint32_t u = len;
    if (len > 1u)
      u = sort_segment_any<MAXK, uint32_t>(len, 0, lane, nullptr, [&](uint32_t e) { return rows[b + e]; });
    if (lane == 0) uniq[c] = u;
  }
}

// One CSR entry on its way to its row's segment.
template <bool W> struct SegEntry;
template <> struct alignas(8) SegEntry<false> { uint32_t col, cnt; };
template <> struct alignas(16) SegEntry<true> { uint32_t col, cnt; uint64_t w; };

// The merged CSC entries of each column in row order, with their values, the
// column sums and the number of entries per row.  Weighted: keys hold the
// event's place in the segment below the row (lb bits).
template <typename Key, int MAXK, bool W>
__global__ void __launch_bounds__(kSegThreads) segment_merge_kernel(const uint32_t *start, const uint32_t *col_ptr,
                                                                 int64_t n_seg, uint32_t shortest, const uint32_t *rows,
                                                                 const uint64_t *w, int lb, uint32_t *row_idx,
                                                                 uint32_t *cnt, uint64_t *wq, float *val,
                                                                 double *colsum, float *inv_colsum,
                                                                 unsigned int *max_count, uint32_t *row_hist) {
  extern __shared__ __align__(16) unsigned char seg_smem[];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  Key *s_key = reinterpret_cast<Key *>(seg_smem) + (threadIdx.x >> 5) * (32 * MAXK);
  const int64_t n_warps = ((int64_t)gridDim.x * kSegThreads) >> 5;
  const uint32_t mask_lb = (1u << lb) - 1u;
  uint32_t mx = 0;
  for (int64_t c = ((int64_t)blockIdx.x * kSegThreads + threadIdx.x) >> 5; c < n_seg; c += n_warps) {
    const uint32_t b = start[c], len = start[c + 1] - b;
    if (len < shortest || len > 32u * MAXK) continue;
    uint32_t out = col_ptr[c];
    uint64_t w_lo = 0, w_hi = 0;  // the column's weights, summed exactly
    if (len > 0u) {
      sort_segment_any<MAXK, Key>(len, lb, lane, s_key, [&](uint32_t e) {
        return W ? (Key)(((Key)rows[b + e] << lb) | (Key)e) : (Key)rows[b + e];
      });
      for (uint32_t e0 = 0; e0 < len; e0 += 32) {
        const uint32_t e = e0 + lane;
        const Key k = e < len ? s_key[e] : (Key)0;
        const uint32_t row = (uint32_t)(k >> lb);
        const bool head = e < len && (e == 0u || (uint32_t)(s_key[e - 1] >> lb) != row);
        const unsigned heads = __ballot_sync(0xffffffffu, head);
        if (head) {
          uint32_t n = 1;
          uint64_t acc = W ? w[b + ((uint32_t)k & mask_lb)] : 0ull;
          for (uint32_t t = e + 1; t < len && (uint32_t)(s_key[t] >> lb) == row; ++t) {
            n += 1;
            if (W) acc += w[b + ((uint32_t)s_key[t] & mask_lb)];
          }
          const uint32_t o = out + __popc(heads & lt);
          row_idx[o] = row;
          cnt[o] = n;
          if (W) {
            wq[o] = acc;
            val[o] = __ull2float_rn(acc) * (float)(1.0 / kFdScale);
            w_lo += (uint32_t)acc;
            w_hi += acc >> 32;
          } else {
            val[o] = (float)n;
          }
          atomicAdd(&row_hist[row], 1u);
          mx = max(mx, n);
        }
        out += __popc(heads);
      }
      __syncwarp();
    }
    double sum = (double)len;
    if (W) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        w_lo += __shfl_xor_sync(0xffffffffu, w_lo, o);
        w_hi += __shfl_xor_sync(0xffffffffu, w_hi, o);
      }
      sum = ((double)w_hi * 4294967296.0 + (double)w_lo) * (1.0 / kFdScale);
    }
    if (lane == 0) {
      colsum[c] = sum;
      inv_colsum[c] = sum > 0.0 ? (float)(1.0 / sum) : 0.0f;
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0 && mx) atomicMax(max_count, mx);
}

// CSC entries into their rows' segments (cursor[j] starts at row_ptr[j])
template <bool W>
__global__ void __launch_bounds__(kSegThreads) segment_transpose_kernel(const uint32_t *col_ptr, int64_t n_cols,
                                                                     const uint32_t *row_idx, const uint32_t *cnt,
                                                                     const uint64_t *wq, uint32_t *cursor,
                                                                     SegEntry<W> *out) {
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = ((int64_t)gridDim.x * kSegThreads) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * kSegThreads + threadIdx.x) >> 5; c < n_cols; c += n_warps) {
    const uint32_t e = col_ptr[c + 1];
#pragma unroll 4
    for (uint32_t k = col_ptr[c] + lane; k < e; k += 32) {
      SegEntry<W> x;
      x.col = (uint32_t)c;
      x.cnt = cnt[k];
      if constexpr (W) x.w = wq[k];
      out[atomicAdd(&cursor[row_idx[k]], 1u)] = x;
    }
  }
}

// CSC entries as keys (j << b) | v in CSC order, weighted with their weight and
// count side by side, for csr_by_radix.
template <bool W>
__global__ void __launch_bounds__(kSegThreads) segment_keys_kernel(const uint32_t *col_ptr, int64_t n_cols,
                                                                const uint32_t *row_idx, const uint32_t *cnt,
                                                                const uint64_t *wq, int b, uint64_t *tkeys,
                                                                WEntry *ent) {
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = ((int64_t)gridDim.x * kSegThreads) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * kSegThreads + threadIdx.x) >> 5; c < n_cols; c += n_warps) {
    const uint32_t e = col_ptr[c + 1];
    for (uint32_t k = col_ptr[c] + lane; k < e; k += 32) {
      tkeys[k] = ((uint64_t)row_idx[k] << b) | (uint64_t)c;
      if constexpr (W) {
        WEntry x;
        x.w = wq[k]; x.cnt = cnt[k]; x.pad = 0u;
        ent[k] = x;
      }
    }
  }
}

// The same in two passes, for matrices beyond the L2.  Pass 1 sorts tiles of
// CSC entries by block of 2^shift rows in shared memory and appends each run
// to its row block's part of the CSR range; in pass 2 one thread block takes a
// row block and places its entries in their rows' segments, with cursors in
// shared memory.  2.5e8 entries of 16 bytes (a forced-detection matrix): 3.4 +
// 5.7 ms against 11.9 ms for the direct transpose, whose returning global
// atomics run at 50 G/s at best and whose sectors are written back half full.
// Pass 2 is bound by its 16-byte stores to random sectors (44 G/s).  An entry
// on its way holds its row within the block and its count (at most kSegLen:
// 11 bits) in one word.
constexpr int kPartThreads = 512;
constexpr int kPartCntBits = 11;
constexpr int kBlockRows = 4096;  // rows of a row block at most
template <bool W> constexpr int part_items() { return W ? 8 : 16; }  // entries per thread
template <bool W> struct PartSmem {
  SegEntry<W> item[kPartThreads * part_items<W>()];
  uint16_t block[kPartThreads * part_items<W>()];
  uint32_t cnt[kRowBlocks], base[kRowBlocks], warp[32];
};

// largest i in [lo, hi) with v[i] <= x (v[lo] <= x)
__device__ __forceinline__ int64_t find_le(const uint32_t *v, int64_t lo, int64_t hi, uint32_t x) {
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (v[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

// column of the first entry of each tile, and of the last entry
__global__ void tile_columns_kernel(const uint32_t *col_ptr, int64_t n_cols, uint32_t nnz, uint32_t tile,
                                    int64_t n_tiles, uint32_t *first) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= n_tiles; t += (int64_t)gridDim.x * blockDim.x)
    first[t] = (uint32_t)find_le(col_ptr, 0, n_cols + 1, t < n_tiles ? (uint32_t)t * tile : nnz - 1u);
}

template <bool W>
__global__ void __launch_bounds__(kPartThreads) partition_rows_kernel(const uint32_t *col_ptr, const uint32_t *tile_col,
                                                                   uint32_t nnz, const uint32_t *row_idx,
                                                                   const uint32_t *cnt, const uint64_t *wq, int shift,
                                                                   uint32_t *cursor, SegEntry<W> *out) {
  constexpr int I = part_items<W>(), T = kPartThreads * I;
  extern __shared__ __align__(16) unsigned char seg_smem[];
  PartSmem<W> &sm = *reinterpret_cast<PartSmem<W> *>(seg_smem);
  const uint32_t p0 = blockIdx.x * (uint32_t)T;
  const uint32_t n = min((uint32_t)T, nnz - p0);
  for (int b = threadIdx.x; b < kRowBlocks; b += kPartThreads) sm.cnt[b] = 0u;
  __syncthreads();
  const int64_t c0 = tile_col[blockIdx.x], c1 = tile_col[blockIdx.x + 1];
  SegEntry<W> x[I];
  uint32_t place[I];  // block | (place among the tile's entries of the block) << 10
#pragma unroll
  for (int k = 0; k < I; ++k) {
    const uint32_t e = threadIdx.x + k * kPartThreads;
    place[k] = 0u;
    if (e < n) {
      const uint32_t row = row_idx[p0 + e], b = row >> shift;
      x[k].cnt = ((row - (b << shift)) << kPartCntBits) | cnt[p0 + e];
      if constexpr (W) x[k].w = wq[p0 + e];
      x[k].col = (uint32_t)find_le(col_ptr, c0, c1 + 1, p0 + e);
      place[k] = b | (atomicAdd(&sm.cnt[b], 1u) << 10);
    }
  }
  __syncthreads();
  // each row block's start in the tile, and its run's place in the output
  const uint32_t n0 = sm.cnt[2 * threadIdx.x], n1 = sm.cnt[2 * threadIdx.x + 1];
  uint32_t total;
  const uint32_t at = block_exclusive_scan(n0 + n1, sm.warp, total);
  sm.cnt[2 * threadIdx.x] = at;
  sm.cnt[2 * threadIdx.x + 1] = at + n0;
  if (n0) sm.base[2 * threadIdx.x] = atomicAdd(&cursor[2 * threadIdx.x], n0) - at;
  if (n1) sm.base[2 * threadIdx.x + 1] = atomicAdd(&cursor[2 * threadIdx.x + 1], n1) - (at + n0);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < I; ++k) {
    if (threadIdx.x + k * kPartThreads < n) {
      const uint32_t b = place[k] & 1023u, p = sm.cnt[b] + (place[k] >> 10);
      sm.item[p] = x[k];
      sm.block[p] = (uint16_t)b;
    }
  }
  __syncthreads();
  for (uint32_t p = threadIdx.x; p < n; p += kPartThreads) out[sm.base[sm.block[p]] + p] = sm.item[p];
}

// first CSR position of each row block
__global__ void row_block_starts_kernel(const uint32_t *row_ptr, int64_t n_rows, int shift, uint32_t *starts) {
  const int64_t r = (int64_t)threadIdx.x << shift;
  starts[threadIdx.x] = row_ptr[r < n_rows ? r : n_rows];
}

// Pass 2: row block b = rows [b << shift, (b + 1) << shift), its entries those
// of its CSR range.  Two blocks of 512 threads per SM: the rows being filled
// are then ~300 x 2048, whose half-written lines (80 MB) stay in the L2 (chosen
// on a matrix of 2.5e8 entries).
constexpr int kPlaceThreads = 512;
template <bool W>
__global__ void __launch_bounds__(kPlaceThreads, 2) place_rows_kernel(const SegEntry<W> *in, const uint32_t *row_ptr,
                                                                   int shift, int64_t n_rows, SegEntry<W> *out) {
  __shared__ uint32_t s_cur[kBlockRows];
  extern __shared__ __align__(16) unsigned char seg_smem[];  // unused: keeps a third block off the SM
  const int64_t r0 = (int64_t)blockIdx.x << shift;
  const int n = (int)min((int64_t)1 << shift, n_rows - r0);
  const uint32_t p0 = row_ptr[r0], p1 = row_ptr[r0 + n];
  for (int r = threadIdx.x; r < n; r += kPlaceThreads) s_cur[r] = row_ptr[r0 + r];
  __syncthreads();
  constexpr int I = 8;
  for (uint32_t p = p0 + threadIdx.x; p < p1; p += I * kPlaceThreads) {
    SegEntry<W> x[I];
#pragma unroll
    for (int k = 0; k < I; ++k)
      if (p + k * kPlaceThreads < p1) x[k] = in[p + k * kPlaceThreads];
#pragma unroll
    for (int k = 0; k < I; ++k)
      if (p + k * kPlaceThreads < p1) {
        const uint32_t pos = atomicAdd(&s_cur[x[k].cnt >> kPartCntBits], 1u);
        x[k].cnt &= (1u << kPartCntBits) - 1u;
        out[pos] = x[k];
      }
  }
}

// the CSR entries of each row in column order, with their values
template <typename Key, int MAXK, bool W>
__global__ void __launch_bounds__(kSegThreads) segment_rows_kernel(const uint32_t *row_ptr, int64_t n_rows,
                                                                uint32_t shortest, const SegEntry<W> *ent, int lb, uint32_t *col_idx,
                                                                uint32_t *cnt, uint64_t *wq, float *val) {
  extern __shared__ __align__(16) unsigned char seg_smem[];
  const int lane = threadIdx.x & 31;
  Key *s_key = reinterpret_cast<Key *>(seg_smem) + (threadIdx.x >> 5) * (32 * MAXK);
  const int64_t n_warps = ((int64_t)gridDim.x * kSegThreads) >> 5;
  const uint32_t mask_lb = (1u << lb) - 1u;
  for (int64_t j = ((int64_t)blockIdx.x * kSegThreads + threadIdx.x) >> 5; j < n_rows; j += n_warps) {
    const uint32_t b = row_ptr[j], len = row_ptr[j + 1] - b;
    if (len == 0u || len < shortest || len > 32u * MAXK) continue;
    sort_segment_any<MAXK, Key>(len, lb, lane, s_key,
                                [&](uint32_t e) { return (Key)(((Key)ent[b + e].col << lb) | (Key)e); });
    for (uint32_t e = lane; e < len; e += 32) {
      const Key k = s_key[e];
      const SegEntry<W> x = ent[b + ((uint32_t)k & mask_lb)];
      col_idx[b + e] = x.col;
      cnt[b + e] = x.cnt;
      if constexpr (W) {
        wq[b + e] = x.w;
        val[b + e] = __ull2float_rn(x.w) * (float)(1.0 / kFdScale);
      } else {
        val[b + e] = (float)x.cnt;
      }
    }
    __syncwarp();
  }
}

static int max_of(const DevBuf &v, int64_t n, DevBuf &scratch, uint32_t *out, cudaStream_t s) {
  MCS_CUDA(cudaMemsetAsync(scratch.p, 0, sizeof(unsigned int), s));
  count_launch(); max_value_kernel<<<grid_for(n), 256, 0, s>>>(v.as<uint32_t>(), n, scratch.as<unsigned int>());
  MCS_LAUNCHED();
  MCS_CUDA(cudaMemcpyAsync(out, scratch.p, sizeof(*out), cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaStreamSynchronize(s));
  return MC_OK;
}

template <typename Kernel, typename... A>
static int launch_segments(Kernel *k, size_t key_bytes, int maxk, int64_t n_seg, cudaStream_t s, A... args) {
  const size_t smem = (kSegThreads / 32) * 32 * (size_t)maxk * key_bytes;
  if (smem > 48 * 1024) MCS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  count_launch();
  k<<<grid_for(n_seg * 32), kSegThreads, smem, s>>>(args...);
  MCS_LAUNCHED();
  return MC_OK;
}

// The CSC and CSR of n > 0 events (with the projector values and the column
// sums) by sorted segments.  Sets *done, or leaves the matrix unfinished (and
// the events untouched) when a column holds more than kSegLen events, which a
// mean above that shows without counting.  The events' buffers are released
// once they are not needed.
template <bool W>
static int assemble_segments(mc_system *sys, DevBuf &key_buf, DevBuf *weight_buf, int64_t n, cudaStream_t s,
                             bool *done) {
  *done = false;
  const uint64_t *keys = key_buf.as<uint64_t>(), *weights = W ? weight_buf->as<uint64_t>() : nullptr;
  const int64_t M = sys->n_rows, N = sys->n_cols;
  if (n > kSegLen * N) return MC_OK;
  const Div64 dm = make_div((uint64_t)M);
  DevBuf cnt, start, flag, tmp;
  MCS_TRY(cnt.alloc((size_t)(N + 1) * 4, s));
  MCS_TRY(start.alloc((size_t)(N + 1) * 4, s));
  MCS_TRY(flag.alloc(sizeof(unsigned int), s));
  MCS_CUDA(cudaMemsetAsync(cnt.p, 0, (size_t)(N + 1) * 4, s));
  count_launch(); segment_count_kernel<<<grid_for(n), 256, 0, s>>>(keys, n, dm, cnt.as<uint32_t>());
  MCS_LAUNCHED();
  MCS_TRY(exclusive_scan_u32(cnt.as<uint32_t>(), start.as<uint32_t>(), N + 1, s));
  uint32_t longest = 0;
  MCS_TRY(max_of(cnt, N, flag, &longest, s));
  if (longest > (uint32_t)kSegLen) return MC_OK;
  MCS_TRY(tmp.alloc((size_t)n * (W ? 12 : 4), s));  // weights, then rows
  uint64_t *const w = W ? tmp.as<uint64_t>() : nullptr;
  uint32_t *const rows = reinterpret_cast<uint32_t *>(tmp.as<uint64_t>() + (W ? n : 0));
  MCS_CUDA(cudaMemcpyAsync(cnt.p, start.p, (size_t)(N + 1) * 4, cudaMemcpyDeviceToDevice, s));  // now the cursors
  count_launch();
  segment_fill_kernel<W><<<grid_for((n + 3) / 4), 256, 0, s>>>(keys, weights, n, dm, cnt.as<uint32_t>(),
                                                               rows, w);
  MCS_LAUNCHED();
  // distinct rows per column, column pointers
  MCS_CUDA(cudaMemsetAsync(cnt.as<uint32_t>() + N, 0, 4, s));
  MCS_TRY(launch_segments(segment_unique_kernel<kShortK>, 0, 1, N, s, start.as<uint32_t>(), N, 0u, rows,
                          cnt.as<uint32_t>()));
  if (longest > 32 * kShortK)
    MCS_TRY(launch_segments(segment_unique_kernel<32>, 0, 1, N, s, start.as<uint32_t>(), N, 32u * kShortK + 1u,
                            rows, cnt.as<uint32_t>()));
  MCS_TRY(sys->col_ptr.alloc((size_t)(N + 1) * 4, s));
  MCS_TRY(exclusive_scan_u32(cnt.as<uint32_t>(), sys->col_ptr.as<uint32_t>(), N + 1, s));
  uint32_t nnz = 0;
  MCS_CUDA(cudaMemcpyAsync(&nnz, sys->col_ptr.as<uint32_t>() + N, sizeof(nnz), cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaStreamSynchronize(s));
  // CSC entries
  DevBuf rhist;
  MCS_TRY(sys->row_idx.alloc((size_t)nnz * 4, s));
  MCS_TRY(sys->csc_cnt.alloc((size_t)nnz * 4, s));
  MCS_TRY(sys->csc_val.alloc((size_t)nnz * 4, s));
  if (W) MCS_TRY(sys->csc_wq.alloc((size_t)nnz * 8, s));
  MCS_TRY(sys->colsum.alloc((size_t)N * sizeof(double), s));
  MCS_TRY(sys->inv_colsum.alloc((size_t)N * sizeof(float), s));
  // two-pass transpose from 256 MB of entries on (below, the direct one's
  // scattered stores stay in the L2), in up to kRowBlocks blocks of rows
  int shift = 0;
  if ((uint64_t)nnz * sizeof(SegEntry<W>) > (256ull << 20) && M > kRowBlocks && M <= (int64_t)kRowBlocks * kBlockRows)
    while (((M - 1) >> shift) + 1 > kRowBlocks) ++shift;
  MCS_TRY(rhist.alloc((size_t)(M + 1) * 4, s));
  MCS_CUDA(cudaMemsetAsync(rhist.p, 0, (size_t)(M + 1) * 4, s));
  MCS_CUDA(cudaMemsetAsync(flag.p, 0, sizeof(unsigned int), s));
  {
    const int lb = W ? bits_for(longest - 1) : 0;
    const bool wide = W && bits_for((uint64_t)M - 1) + lb > 32;
    auto go = [&](auto *k, size_t kb, int maxk) {
      return launch_segments(k, kb, maxk, N, s, (const uint32_t *)start.as<uint32_t>(),
                             (const uint32_t *)sys->col_ptr.as<uint32_t>(), N,
                             maxk == kShortK ? 0u : 32u * kShortK + 1u, (const uint32_t *)rows,
                             (const uint64_t *)w, lb, sys->row_idx.as<uint32_t>(),
                             sys->csc_cnt.as<uint32_t>(), sys->csc_wq.as<uint64_t>(), sys->csc_val.as<float>(),
                             sys->colsum.as<double>(), sys->inv_colsum.as<float>(), flag.as<unsigned int>(),
                             rhist.as<uint32_t>());
    };
    MCS_TRY(wide ? go(segment_merge_kernel<uint64_t, kShortK, W>, 8, kShortK) : go(segment_merge_kernel<uint32_t, kShortK, W>, 4, kShortK));
    if (longest > 32 * kShortK)
      MCS_TRY(wide ? go(segment_merge_kernel<uint64_t, 32, W>, 8, 32) : go(segment_merge_kernel<uint32_t, 32, W>, 4, 32));
  }
  tmp.release();
  uint32_t max_count = 0;
  MCS_CUDA(cudaMemcpyAsync(&max_count, flag.p, sizeof(max_count), cudaMemcpyDeviceToHost, s));
  // CSR
  const uint32_t *col_ptr = sys->col_ptr.as<uint32_t>(), *row_idx = sys->row_idx.as<uint32_t>();
  const uint32_t *csc_cnt = sys->csc_cnt.as<uint32_t>();
  const uint64_t *csc_wq = sys->csc_wq.as<uint64_t>();
  MCS_TRY(sys->row_ptr.alloc((size_t)(M + 1) * 4, s));
  MCS_TRY(exclusive_scan_u32(rhist.as<uint32_t>(), sys->row_ptr.as<uint32_t>(), M + 1, s));
  MCS_TRY(max_of(rhist, M, flag, &longest, s));  // waits, max_count included
  sys->nnz = nnz;
  sys->max_count = max_count;
  if (longest > (uint32_t)kSegLen) {
    // rows too long for a warp: the CSC stands, the CSR by radix sort (the
    // projector values then come from the counts or weights)
    key_buf.release();
    if (W) weight_buf->release();
    sys->csc_val.release();
    DevBuf tkeys, ucnt, went;
    MCS_TRY(tkeys.alloc((size_t)nnz * sizeof(uint64_t), s));
    if (W) {
      MCS_TRY(went.alloc((size_t)nnz * sizeof(WEntry), s));
    } else {
      MCS_TRY(ucnt.alloc((size_t)nnz * 4, s));
      MCS_CUDA(cudaMemcpyAsync(ucnt.p, csc_cnt, (size_t)nnz * 4, cudaMemcpyDeviceToDevice, s));
    }
    MCS_TRY(launch_segments(segment_keys_kernel<W>, 0, 1, N, s, col_ptr, N, row_idx, csc_cnt, csc_wq,
                            bits_for((uint64_t)N - 1), tkeys.as<uint64_t>(), went.as<WEntry>()));
    MCS_TRY(csr_by_radix(sys, tkeys, ucnt, went, nnz, s));
    *done = true;
    return MC_OK;
  }
  const uint32_t *row_ptr = sys->row_ptr.as<uint32_t>();
  // the matrix will be finished here: the events are not needed again, and
  // their buffers hold the entries on their way where they are large enough
  // (mapping gigabytes of fresh memory costs about 0.7 ms each)
  const size_t ent_bytes = (size_t)nnz * sizeof(SegEntry<W>);
  DevBuf ent, part;
  const auto entry_space = [&](DevBuf &b, DevBuf *old) {
    if (old && old->bytes >= ent_bytes) { b = std::move(*old); return MC_OK; }
    return b.alloc(ent_bytes, s);
  };
  if (shift > 0) {
    constexpr int tile = kPartThreads * part_items<W>();
    const int64_t n_tiles = div_up(nnz, tile);
    DevBuf starts, tile_col;
    MCS_TRY(starts.alloc((size_t)kRowBlocks * 4, s));
    MCS_TRY(tile_col.alloc((size_t)(n_tiles + 1) * 4, s));
    MCS_TRY(entry_space(part, &key_buf));
    MCS_TRY(entry_space(ent, weight_buf));
    count_launch();
    row_block_starts_kernel<<<1, kRowBlocks, 0, s>>>(row_ptr, M, shift, starts.as<uint32_t>());
    count_launch();
    tile_columns_kernel<<<grid_for(n_tiles + 1), 256, 0, s>>>(col_ptr, N, nnz, tile, n_tiles, tile_col.as<uint32_t>());
    MCS_LAUNCHED();
    MCS_CUDA(cudaFuncSetAttribute(partition_rows_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(PartSmem<W>)));
    count_launch();
    partition_rows_kernel<W><<<(unsigned)n_tiles, kPartThreads, sizeof(PartSmem<W>), s>>>(
        col_ptr, tile_col.as<uint32_t>(), nnz, row_idx, csc_cnt, csc_wq, shift, starts.as<uint32_t>(),
        part.as<SegEntry<W>>());
    MCS_LAUNCHED();
    constexpr int pad = 80 << 10;
    MCS_CUDA(cudaFuncSetAttribute(place_rows_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, pad));
    count_launch();
    place_rows_kernel<W><<<(unsigned)(((M - 1) >> shift) + 1), kPlaceThreads, pad, s>>>(part.as<SegEntry<W>>(), row_ptr,
                                                                                      shift, M, ent.as<SegEntry<W>>());
    MCS_LAUNCHED();
    part.release();
  } else {
    MCS_TRY(entry_space(ent, &key_buf));
    MCS_CUDA(cudaMemcpyAsync(rhist.p, row_ptr, (size_t)(M + 1) * 4, cudaMemcpyDeviceToDevice, s));
    MCS_TRY(launch_segments(segment_transpose_kernel<W>, 0, 1, N, s, col_ptr, N, row_idx, csc_cnt, csc_wq,
                            rhist.as<uint32_t>(), ent.as<SegEntry<W>>()));
  }
  key_buf.release();
  if (W) weight_buf->release();
  MCS_TRY(sys->col_idx.alloc((size_t)nnz * 4, s));
  MCS_TRY(sys->csr_cnt.alloc((size_t)nnz * 4, s));
  MCS_TRY(sys->csr_val.alloc((size_t)nnz * 4, s));
  if (W) MCS_TRY(sys->csr_wq.alloc((size_t)nnz * 8, s));
  {
    const int lb = bits_for(longest - 1);
    const bool wide = bits_for((uint64_t)N - 1) + lb > 32;
    auto go = [&](auto *k, size_t kb, int maxk) {
      return launch_segments(k, kb, maxk, M, s, (const uint32_t *)sys->row_ptr.as<uint32_t>(), M,
                             maxk == kShortK ? 0u : 32u * kShortK + 1u, (const SegEntry<W> *)ent.as<SegEntry<W>>(), lb, sys->col_idx.as<uint32_t>(),
                             sys->csr_cnt.as<uint32_t>(), sys->csr_wq.as<uint64_t>(), sys->csr_val.as<float>());
    };
    MCS_TRY(wide ? go(segment_rows_kernel<uint64_t, kShortK, W>, 8, kShortK) : go(segment_rows_kernel<uint32_t, kShortK, W>, 4, kShortK));
    if (longest > 32 * kShortK)
      MCS_TRY(wide ? go(segment_rows_kernel<uint64_t, 32, W>, 8, 32) : go(segment_rows_kernel<uint32_t, 32, W>, 4, 32));
  }
  sys->values_ready = true;
  *done = true;
  return MC_OK;
}

// Steps 1-4 of the assembly by a radix sort of the event keys (any events,
// weighted or not).
static int assemble_radix(mc_system *sys, DevBuf &keys, int64_t n, cudaStream_t s, const uint64_t *weights) {
  const uint64_t M = (uint64_t)sys->n_rows, N = (uint64_t)sys->n_cols;
  // 1. sort events by (v, j); weighted: with the event index as payload
  DevBuf alt, perm, perm_alt, went;
  MCS_TRY(alt.alloc((size_t)(n > 0 ? n : 1) * sizeof(uint64_t), s));
  if (weights) {
    MCS_TRY(perm.alloc((size_t)(n > 0 ? n : 1) * sizeof(uint32_t), s));
    MCS_TRY(perm_alt.alloc((size_t)(n > 0 ? n : 1) * sizeof(uint32_t), s));
    if (n > 0) {
      count_launch(); iota_kernel<<<grid_for(n), 256, 0, s>>>(perm.as<uint32_t>(), n);
      MCS_LAUNCHED();
    }
  }
  bool in_alt = false;
  MCS_TRY(radix_sort_u64(keys.as<uint64_t>(), alt.as<uint64_t>(), weights ? perm.as<uint32_t>() : nullptr,
                         weights ? perm_alt.as<uint32_t>() : nullptr, n, bits_for(M * N - 1), &in_alt, s));
  const uint64_t *sorted = in_alt ? alt.as<uint64_t>() : keys.as<uint64_t>();
  const uint32_t *sorted_perm = weights ? (in_alt ? perm_alt.as<uint32_t>() : perm.as<uint32_t>()) : nullptr;

  // 2. run-length encode; weighted: the CSC weight sums, and each entry's
  // weight and count side by side for the CSR gather
  int64_t nu = 0;
  DevBuf ukeys, ucnt;
  if (n > 0) {
    DevBuf flags, idx, upos;
    MCS_TRY(flags.alloc(n * sizeof(uint32_t), s));
    MCS_TRY(idx.alloc(n * sizeof(uint32_t), s));
    count_launch(); head_flags_kernel<<<grid_for(n), 256, 0, s>>>(sorted, n, flags.as<uint32_t>());
    MCS_LAUNCHED();
    MCS_TRY(exclusive_scan_u32(flags.as<uint32_t>(), idx.as<uint32_t>(), n, s));
    uint32_t last_idx = 0, last_flag = 0;
    MCS_CUDA(cudaMemcpyAsync(&last_idx, idx.as<uint32_t>() + (n - 1), 4, cudaMemcpyDeviceToHost, s));
    MCS_CUDA(cudaMemcpyAsync(&last_flag, flags.as<uint32_t>() + (n - 1), 4, cudaMemcpyDeviceToHost, s));
    MCS_CUDA(cudaStreamSynchronize(s));
    nu = (int64_t)last_idx + last_flag;
    MCS_TRY(ukeys.alloc(nu * sizeof(uint64_t), s));
    MCS_TRY(upos.alloc(nu * sizeof(uint32_t), s));
    MCS_TRY(ucnt.alloc(nu * sizeof(uint32_t), s));
    count_launch(); compact_heads_kernel<<<grid_for(n), 256, 0, s>>>(sorted, flags.as<uint32_t>(), idx.as<uint32_t>(), n,
                                                     ukeys.as<uint64_t>(), upos.as<uint32_t>());
    MCS_LAUNCHED();
    count_launch(); run_lengths_kernel<<<grid_for(nu), 256, 0, s>>>(upos.as<uint32_t>(), nu, n, ucnt.as<uint32_t>());
    MCS_LAUNCHED();
    if (weights) {
      MCS_TRY(sys->csc_wq.alloc(nu * sizeof(uint64_t), s));
      MCS_TRY(went.alloc(nu * sizeof(WEntry), s));
      count_launch();
      run_weights_kernel<<<grid_for(nu), 256, 0, s>>>(upos.as<uint32_t>(), ucnt.as<uint32_t>(), nu, sorted_perm,
                                                      weights, sys->csc_wq.as<uint64_t>(), went.as<WEntry>());
      MCS_LAUNCHED();
    }
  }
  alt.release();
  perm.release();
  perm_alt.release();
  keys.release();
  sys->nnz = nu;

  // 3. CSC: rows, counts and col_ptr in sorted order; the transposed keys
  const size_t nnz_b = (size_t)(nu > 0 ? nu : 1);
  const int b = bits_for(N - 1);
  DevBuf tkeys;
  {
    MCS_TRY(sys->col_ptr.alloc((N + 1) * sizeof(uint32_t), s));
    MCS_TRY(sys->row_idx.alloc(nnz_b * sizeof(uint32_t), s));
    MCS_TRY(sys->csc_cnt.alloc(nnz_b * sizeof(uint32_t), s));
    if (weights && nu == 0) MCS_TRY(sys->csc_wq.alloc(sizeof(uint64_t), s));
    if (nu > 0) {
      MCS_TRY(tkeys.alloc(nu * sizeof(uint64_t), s));
      count_launch();
      csc_split_kernel<<<grid_for(nu), 256, 0, s>>>(ukeys.as<uint64_t>(), nu, M, b, sys->row_idx.as<uint32_t>(),
                                                    sys->col_ptr.as<uint32_t>(), (int64_t)N, tkeys.as<uint64_t>());
      MCS_LAUNCHED();
      MCS_CUDA(cudaMemcpyAsync(sys->csc_cnt.p, ucnt.p, nu * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    } else {
      MCS_CUDA(cudaMemsetAsync(sys->col_ptr.p, 0, (N + 1) * sizeof(uint32_t), s));
    }
  }
  ukeys.release();

  // 4. CSR
  MCS_TRY(sys->row_ptr.alloc((M + 1) * sizeof(uint32_t), s));
  if (nu > 0) {
    MCS_TRY(csr_by_radix(sys, tkeys, ucnt, went, nu, s));
  } else {
    MCS_TRY(sys->col_idx.alloc(sizeof(uint32_t), s));
    MCS_TRY(sys->csr_cnt.alloc(sizeof(uint32_t), s));
    MCS_CUDA(cudaMemsetAsync(sys->row_ptr.p, 0, (M + 1) * sizeof(uint32_t), s));
    if (weights) MCS_TRY(sys->csr_wq.alloc(sizeof(uint64_t), s));
  }
  return MC_OK;
}

int assemble_system(mc_system *sys, DevBuf &keys, int64_t n, cudaStream_t s, DevBuf *weights) {
  const uint64_t N = (uint64_t)sys->n_cols;
  if (n >= 0xFFFFFFFFll) {  // places are 32-bit on every path below
    set_error("%lld events exceed the 2^32 limit of one build; split the history range", (long long)n);
    return MC_EINVAL;
  }
  // n_v and 1/n_v
  MCS_TRY(sys->n_v.alloc(N * sizeof(uint32_t), s));
  MCS_TRY(sys->inv_n.alloc(N * sizeof(float), s));
  count_launch(); histories_per_voxel_kernel<<<grid_for((int64_t)N), 256, 0, s>>>(sys->first, sys->count, N, sys->n_v.as<uint32_t>(),
                                                                   sys->inv_n.as<float>());
  MCS_LAUNCHED();
  sys->weighted = weights != nullptr;

  // 1-4. the CSC and CSR: by buckets (a thread per column and row) where
  // columns and rows are short, by sorted segments (a warp each) where they are
  // longer or weighted, else by a radix sort.  Columns of 16 events and more
  // on average hardly ever keep below the buckets' 64 everywhere.
  bool bucketed = false, segmented = false;
  if (!weights && n > 0 && n < 16 * (int64_t)N && n < ((int64_t)1 << 31))
    MCS_TRY(assemble_buckets(sys, keys.as<uint64_t>(), n, s, &bucketed));
  if (!bucketed && n > 0) {
    MCS_TRY(weights ? assemble_segments<true>(sys, keys, weights, n, s, &segmented)
                    : assemble_segments<false>(sys, keys, nullptr, n, s, &segmented));
  }
  if (bucketed) keys.release();
  else if (!segmented) MCS_TRY(assemble_radix(sys, keys, n, s, weights ? weights->as<uint64_t>() : nullptr));

  // 5. column sums S_v and the largest count
  if (!segmented) {
    MCS_TRY(sys->colsum.alloc(N * sizeof(double), s));
    MCS_TRY(sys->inv_colsum.alloc(N * sizeof(float), s));
    DevBuf mx;
    MCS_TRY(mx.alloc(sizeof(unsigned int), s));
    MCS_CUDA(cudaMemsetAsync(mx.p, 0, sizeof(unsigned int), s));
    count_launch(); column_sums_kernel<<<grid_for((int64_t)N), 256, 0, s>>>(sys->col_ptr.as<uint32_t>(), sys->csc_cnt.as<uint32_t>(),
                                                            (int64_t)N, sys->colsum.as<double>(),
                                                            sys->inv_colsum.as<float>(), mx.as<unsigned int>());
    MCS_LAUNCHED();
    if (weights) {
      // S_v from the weights (the kernel above gave the largest event count)
      count_launch();
      column_weight_sums_kernel<<<grid_for((int64_t)N), 256, 0, s>>>(sys->col_ptr.as<uint32_t>(),
                                                                     sys->csc_wq.as<uint64_t>(), (int64_t)N,
                                                                     sys->colsum.as<double>(),
                                                                     sys->inv_colsum.as<float>());
      MCS_LAUNCHED();
    }
    unsigned int mxh = 0;
    MCS_CUDA(cudaMemcpyAsync(&mxh, mx.p, sizeof(mxh), cudaMemcpyDeviceToHost, s));
    MCS_CUDA(cudaStreamSynchronize(s));
    sys->max_count = mxh;
  }
  return MC_OK;
}

// ---------------------------------------------------------------------------
// projector values: the counts in the storage type of sys->value_type
// ---------------------------------------------------------------------------
template <typename V> __device__ __forceinline__ V from_count(uint32_t c);
template <> __device__ __forceinline__ float from_count<float>(uint32_t c) { return (float)c; }
template <> __device__ __forceinline__ __half from_count<__half>(uint32_t c) { return __uint2half_rn(c); }
template <> __device__ __forceinline__ __nv_bfloat16 from_count<__nv_bfloat16>(uint32_t c) {
  return __uint2bfloat16_rn(c);
}

template <typename V> __global__ void convert_counts_kernel(const uint32_t *cnt, int64_t n, V *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = from_count<V>(cnt[i]);
}

// weighted systems: the fixed-point weight sums as float, rounded once from
// the integer and scaled by 2^-48 exactly (the same value as a conversion
// through double for sums below 2^53, without the slow FP64 unit)
__global__ void convert_weights_kernel(const uint64_t *wq, int64_t n, float *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = __ull2float_rn(wq[i]) * (float)(1.0 / kFdScale);
}

// rounded-A values: val = round(C_jv / n_v) per entry of the CSR (column
// index per entry) ...
template <typename V> __device__ __forceinline__ V from_double(double a);
template <> __device__ __forceinline__ __half from_double<__half>(double a) { return __double2half(a); }
template <> __device__ __forceinline__ __nv_bfloat16 from_double<__nv_bfloat16>(double a) {
  return __double2bfloat16(a);
}
template <typename V>
__global__ void a_values_csr_kernel(const uint32_t *cnt, const uint32_t *col, const uint32_t *n_v, int64_t n, V *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = from_double<V>((double)cnt[i] / (double)n_v[col[i]]);
}
// ... and per column of the CSC, with the column sums of the stored values
// (the rounded matrix's sensitivity s~_v, summed in double in row order)
template <typename V>
__global__ void a_values_csc_kernel(const uint32_t *col_ptr, const uint32_t *cnt, const uint32_t *n_v, int64_t n_cols,
                                    V *out, float *ones, double *sens, float *inv_sens) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_cols; v += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    const double nv = (double)n_v[v];
    for (uint32_t k = col_ptr[v]; k < col_ptr[v + 1]; ++k) {
      const V a = from_double<V>((double)cnt[k] / nv);
      out[k] = a;
      acc += (double)(float)a;
    }
    ones[v] = 1.0f;
    sens[v] = acc;
    inv_sens[v] = acc > 0.0 ? (float)(1.0 / acc) : 0.0f;
  }
}

// counts rounded to V: the column sums of the stored (rounded) counts
template <typename V>
__global__ void rounded_count_sums_kernel(const uint32_t *col_ptr, const uint32_t *cnt, int64_t n_cols, double *sums,
                                          float *inv_sums) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_cols; v += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (uint32_t k = col_ptr[v]; k < col_ptr[v + 1]; ++k) acc += (double)(float)from_count<V>(cnt[k]);
    sums[v] = acc;
    inv_sums[v] = acc > 0.0 ? (float)(1.0 / acc) : 0.0f;
  }
}

template <typename V> static int make_rounded_sums(mc_system *sys, cudaStream_t s) {
  const int64_t N = sys->n_cols;
  const size_t nb = (size_t)(N > 0 ? N : 1);
  MCS_TRY(sys->a_sens.alloc(nb * sizeof(double), s));
  MCS_TRY(sys->a_inv_sens.alloc(nb * sizeof(float), s));
  if (N > 0) {
    count_launch();
    rounded_count_sums_kernel<V><<<grid_for(N), 256, 0, s>>>(sys->col_ptr.as<uint32_t>(), sys->csc_cnt.as<uint32_t>(),
                                                             N, sys->a_sens.as<double>(), sys->a_inv_sens.as<float>());
  }
  MCS_LAUNCHED();
  return MC_OK;
}

template <typename V> static int make_a_values(mc_system *sys, cudaStream_t s) {
  const int64_t nnz = sys->nnz, N = sys->n_cols;
  const size_t nb = (size_t)(N > 0 ? N : 1);
  MCS_TRY(sys->a_ones.alloc(nb * sizeof(float), s));
  MCS_TRY(sys->a_sens.alloc(nb * sizeof(double), s));
  MCS_TRY(sys->a_inv_sens.alloc(nb * sizeof(float), s));
  if (nnz > 0) {
    count_launch();
    a_values_csr_kernel<V><<<grid_for(nnz), 256, 0, s>>>(sys->csr_cnt.as<uint32_t>(), sys->col_idx.as<uint32_t>(),
                                                         sys->n_v.as<uint32_t>(), nnz, sys->csr_val.as<V>());
  }
  if (N > 0) {
    count_launch();
    a_values_csc_kernel<V><<<grid_for(N), 256, 0, s>>>(sys->col_ptr.as<uint32_t>(), sys->csc_cnt.as<uint32_t>(),
                                                       sys->n_v.as<uint32_t>(), N, sys->csc_val.as<V>(),
                                                       sys->a_ones.as<float>(), sys->a_sens.as<double>(),
                                                       sys->a_inv_sens.as<float>());
  }
  MCS_LAUNCHED();
  return MC_OK;
}

int make_values(mc_system *sys, cudaStream_t s) {
  const int64_t nnz = sys->nnz;
  // assembly by segments has written the float values with the entries
  const bool ready = sys->values_ready;
  sys->values_ready = false;
  if (ready && sys->value_type == MC_VAL_F32) return MC_OK;
  const size_t es = value_storage(sys->value_type) == 0 ? 4 : 2;
  const size_t bytes = (size_t)(nnz > 0 ? nnz : 1) * es;
  MCS_TRY(sys->csr_val.alloc(bytes, s));
  MCS_TRY(sys->csc_val.alloc(bytes, s));
  if (sys->weighted && sys->value_type != MC_VAL_F32) { set_error("weighted systems keep float values"); return MC_EINVAL; }
  if (sys->value_type == MC_VAL_F16_A) return make_a_values<__half>(sys, s);
  if (sys->value_type == MC_VAL_BF16_A) return make_a_values<__nv_bfloat16>(sys, s);
  // counts beyond the type's exact range are rounded: normalise with the
  // rounded counts' column sums
  sys->rounded_counts = (sys->value_type == MC_VAL_F16 && sys->max_count > 2048u) ||
                        (sys->value_type == MC_VAL_BF16 && sys->max_count > 256u);
  if (sys->rounded_counts) {
    if (sys->value_type == MC_VAL_F16) MCS_TRY(make_rounded_sums<__half>(sys, s));
    else MCS_TRY(make_rounded_sums<__nv_bfloat16>(sys, s));
  }
  if (nnz == 0) return MC_OK;
  const int g = grid_for(nnz);
  if (sys->weighted) {
    count_launch(); convert_weights_kernel<<<g, 256, 0, s>>>(sys->csr_wq.as<uint64_t>(), nnz, sys->csr_val.as<float>());
    count_launch(); convert_weights_kernel<<<g, 256, 0, s>>>(sys->csc_wq.as<uint64_t>(), nnz, sys->csc_val.as<float>());
  } else if (sys->value_type == MC_VAL_F32) {
    count_launch(); convert_counts_kernel<float><<<g, 256, 0, s>>>(sys->csr_cnt.as<uint32_t>(), nnz, sys->csr_val.as<float>());
    count_launch(); convert_counts_kernel<float><<<g, 256, 0, s>>>(sys->csc_cnt.as<uint32_t>(), nnz, sys->csc_val.as<float>());
  } else if (sys->value_type == MC_VAL_F16) {
    count_launch(); convert_counts_kernel<__half><<<g, 256, 0, s>>>(sys->csr_cnt.as<uint32_t>(), nnz, sys->csr_val.as<__half>());
    count_launch(); convert_counts_kernel<__half><<<g, 256, 0, s>>>(sys->csc_cnt.as<uint32_t>(), nnz, sys->csc_val.as<__half>());
  } else {
    count_launch(); convert_counts_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(sys->csr_cnt.as<uint32_t>(), nnz,
                                                           sys->csr_val.as<__nv_bfloat16>());
    count_launch(); convert_counts_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(sys->csc_cnt.as<uint32_t>(), nnz,
                                                           sys->csc_val.as<__nv_bfloat16>());
  }
  MCS_LAUNCHED();
  return MC_OK;
}

}  // namespace mcs

// ---------------------------------------------------------------------------
// subset systems (ordered subsets of views, Sec. 5.3)
// ---------------------------------------------------------------------------
namespace mcs {

// row i of the subset = row map[i] of the parent: view subset + (i / rpv) * n_sub
__global__ void subset_rows_kernel(int64_t m_s, int64_t rpv, int n_sub, int subset, const uint32_t *parent_ptr,
                                   uint32_t *map, uint32_t *len) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m_s; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t view = subset + (i / rpv) * n_sub;
    const uint32_t r = (uint32_t)(view * rpv + i % rpv);
    map[i] = r;
    len[i] = parent_ptr[r + 1] - parent_ptr[r];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) len[m_s] = 0u;
}

// copy the parent's entries of each subset row; emit (col * m_s + i, count)
__global__ void subset_copy_kernel(int64_t m_s, const uint32_t *map, const uint32_t *parent_ptr,
                                   const uint32_t *parent_col, const uint32_t *parent_cnt, const uint32_t *ptr,
                                   uint32_t *col, uint32_t *cnt, uint64_t *tkeys) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m_s; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t src = parent_ptr[map[i]], dst = ptr[i], n = ptr[i + 1] - ptr[i];
    for (uint32_t k = 0; k < n; ++k) {
      const uint32_t c = parent_col[src + k];
      col[dst + k] = c;
      cnt[dst + k] = parent_cnt[src + k];
      tkeys[dst + k] = (uint64_t)c * (uint64_t)m_s + (uint64_t)i;
    }
  }
}

__global__ void sum_counts_kernel(const uint32_t *cnt, int64_t n, unsigned long long *out) {
  unsigned long long acc = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc += cnt[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, acc);
}

int subset_system(const mc_system *parent, int64_t rpv, int n_sub, int subset, mc_system *sys, cudaStream_t s) {
  const int64_t V = parent->n_rows / rpv;
  const int64_t nv_s = (V - subset + n_sub - 1) / n_sub;
  const int64_t m_s = nv_s * rpv, N = parent->n_cols;
  sys->n_rows = m_s;
  sys->n_cols = N;
  sys->first = parent->first;
  sys->count = parent->count;
  sys->parent_rows = parent->n_rows;
  sys->n_subsets = n_sub;
  sys->subset = subset;
  MCS_TRY(sys->row_map.alloc((size_t)m_s * sizeof(uint32_t), s));
  DevBuf len;
  MCS_TRY(len.alloc((size_t)(m_s + 1) * sizeof(uint32_t), s));
  MCS_TRY(sys->row_ptr.alloc((size_t)(m_s + 1) * sizeof(uint32_t), s));
  count_launch();
  subset_rows_kernel<<<grid_for(m_s), 256, 0, s>>>(m_s, rpv, n_sub, subset, parent->row_ptr.as<uint32_t>(),
                                                  sys->row_map.as<uint32_t>(), len.as<uint32_t>());
  MCS_LAUNCHED();
  MCS_TRY(exclusive_scan_u32(len.as<uint32_t>(), sys->row_ptr.as<uint32_t>(), m_s + 1, s));
  uint32_t nnz = 0;
  MCS_CUDA(cudaMemcpyAsync(&nnz, sys->row_ptr.as<uint32_t>() + m_s, 4, cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaStreamSynchronize(s));
  sys->nnz = nnz;
  const size_t nb = (size_t)(nnz > 0 ? nnz : 1);
  DevBuf tkeys, tkeys_alt, tcnt, tcnt_alt;
  MCS_TRY(sys->col_idx.alloc(nb * 4, s));
  MCS_TRY(sys->csr_cnt.alloc(nb * 4, s));
  MCS_TRY(tkeys.alloc(nb * 8, s));
  MCS_TRY(tkeys_alt.alloc(nb * 8, s));
  MCS_TRY(tcnt.alloc(nb * 4, s));
  MCS_TRY(tcnt_alt.alloc(nb * 4, s));
  count_launch();
  subset_copy_kernel<<<grid_for(m_s), 256, 0, s>>>(m_s, sys->row_map.as<uint32_t>(), parent->row_ptr.as<uint32_t>(),
                                                  parent->col_idx.as<uint32_t>(), parent->csr_cnt.as<uint32_t>(),
                                                  sys->row_ptr.as<uint32_t>(), sys->col_idx.as<uint32_t>(),
                                                  sys->csr_cnt.as<uint32_t>(), tkeys.as<uint64_t>());
  MCS_LAUNCHED();
  // CSC of the subset: sort (col * m_s + row, count)
  MCS_CUDA(cudaMemcpyAsync(tcnt.p, sys->csr_cnt.p, (size_t)nnz * 4, cudaMemcpyDeviceToDevice, s));
  bool alt = false;
  MCS_TRY(radix_sort_u64(tkeys.as<uint64_t>(), tkeys_alt.as<uint64_t>(), tcnt.as<uint32_t>(), tcnt_alt.as<uint32_t>(),
                         nnz, bits_for((uint64_t)m_s * (uint64_t)N - 1), &alt, s));
  const uint64_t *tk = alt ? tkeys_alt.as<uint64_t>() : tkeys.as<uint64_t>();
  const uint32_t *tc = alt ? tcnt_alt.as<uint32_t>() : tcnt.as<uint32_t>();
  DevBuf hist;
  MCS_TRY(hist.alloc((size_t)(N + 1) * 4, s));
  MCS_CUDA(cudaMemsetAsync(hist.p, 0, (size_t)(N + 1) * 4, s));
  MCS_TRY(sys->col_ptr.alloc((size_t)(N + 1) * 4, s));
  MCS_TRY(sys->row_idx.alloc(nb * 4, s));
  MCS_TRY(sys->csc_cnt.alloc(nb * 4, s));
  if (nnz > 0) {
    count_launch();
    split_keys_kernel<<<grid_for(nnz), 256, 0, s>>>(tk, nnz, (uint64_t)m_s, nullptr, sys->row_idx.as<uint32_t>(),
                                                    hist.as<uint32_t>());
    MCS_LAUNCHED();
    MCS_CUDA(cudaMemcpyAsync(sys->csc_cnt.p, tc, (size_t)nnz * 4, cudaMemcpyDeviceToDevice, s));
  }
  MCS_TRY(exclusive_scan_u32(hist.as<uint32_t>(), sys->col_ptr.as<uint32_t>(), N + 1, s));
  // histories per voxel are the parent's; column sums and largest count
  MCS_TRY(sys->n_v.alloc((size_t)N * 4, s));
  MCS_TRY(sys->inv_n.alloc((size_t)N * 4, s));
  MCS_CUDA(cudaMemcpyAsync(sys->n_v.p, parent->n_v.p, (size_t)N * 4, cudaMemcpyDeviceToDevice, s));
  MCS_CUDA(cudaMemcpyAsync(sys->inv_n.p, parent->inv_n.p, (size_t)N * 4, cudaMemcpyDeviceToDevice, s));
  MCS_TRY(sys->colsum.alloc((size_t)N * sizeof(double), s));
  MCS_TRY(sys->inv_colsum.alloc((size_t)N * sizeof(float), s));
  DevBuf mx;
  MCS_TRY(mx.alloc(2 * sizeof(unsigned long long), s));
  MCS_CUDA(cudaMemsetAsync(mx.p, 0, 2 * sizeof(unsigned long long), s));
  count_launch();
  column_sums_kernel<<<grid_for(N), 256, 0, s>>>(sys->col_ptr.as<uint32_t>(), sys->csc_cnt.as<uint32_t>(), N,
                                                 sys->colsum.as<double>(), sys->inv_colsum.as<float>(),
                                                 mx.as<unsigned int>());
  count_launch();
  sum_counts_kernel<<<grid_for(nnz > 0 ? nnz : 1), 256, 0, s>>>(sys->csr_cnt.as<uint32_t>(), nnz,
                                                                mx.as<unsigned long long>() + 1);
  MCS_LAUNCHED();
  unsigned long long h[2] = {0, 0};
  MCS_CUDA(cudaMemcpyAsync(h, mx.p, sizeof(h), cudaMemcpyDeviceToHost, s));
  MCS_CUDA(cudaStreamSynchronize(s));
  sys->max_count = (uint32_t)(h[0] & 0xFFFFFFFFull);
  sys->n_events = (int64_t)h[1];
  for (int f = 0; f < 4; ++f) sys->fates[f] = parent->fates[f];
  return MC_OK;
}

}  // namespace mcs
