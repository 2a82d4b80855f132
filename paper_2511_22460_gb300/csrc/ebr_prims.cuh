// Device-wide primitives of the index builder and of Algorithm 2's long
// lists: an exclusive / inclusive scan over any type with an associative
// add, a stable least-significant-digit radix sort of 64-bit or 32-bit keys
// with optional 32-bit values, and the unique of a sorted array.
//
// The scan runs in three launches (tile sums; one CTA scans the tile sums;
// each tile scans itself from its offset), so no CTA ever waits on another.
// The radix sort takes 8-bit digits from the lowest bit up, one launch per
// digit; a tile of keys is ranked by warp (__match_any_sync on the digit, in
// index order) and across warps by per-warp digit counts, so equal digits
// keep their order and the passes compose into a sort.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <utility>

#include "ebr_internal.cuh"

namespace ebr {
namespace prims {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;  // per thread: tiles of 4096
constexpr uint32_t kScanTile = kScanThreads * kScanItems;

// Block-wide exclusive scan of one value per thread (returns the thread's
// exclusive prefix, *total the block's sum).  s_warp: 32 entries of T.
template <typename T, typename Op>
__device__ __forceinline__ T block_exclusive(T v, Op op, T zero, T *s_warp, T *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y;
    // shuffle any trivially copyable T in 32-bit pieces
    static_assert(sizeof(T) % 4 == 0, "scan type size");
    uint32_t *pi = reinterpret_cast<uint32_t *>(&incl), *py = reinterpret_cast<uint32_t *>(&y);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(T) / 4); k++) py[k] = __shfl_up_sync(0xffffffffu, pi[k], o);
    if (lane >= o) incl = op(y, incl);
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    T w = lane < nw ? s_warp[lane] : zero;
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y;
      uint32_t *pi = reinterpret_cast<uint32_t *>(&wi), *py = reinterpret_cast<uint32_t *>(&y);
#pragma unroll
      for (int k = 0; k < (int)(sizeof(T) / 4); k++)
        py[k] = __shfl_up_sync(0xffffffffu, pi[k], o);
      if (lane >= o) wi = op(y, wi);
    }
    if (lane < nw) s_warp[lane] = wi;  // inclusive prefix of the warp sums
  }
  __syncthreads();
  const T before = warp > 0 ? s_warp[warp - 1] : zero;
  *total = s_warp[(blockDim.x >> 5) - 1];
  // exclusive = before + (incl - v): recompute as before + exclusive-in-warp
  T ex_in = zero;
  {
    T y;
    uint32_t *pi = reinterpret_cast<uint32_t *>(&incl), *py = reinterpret_cast<uint32_t *>(&y);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(T) / 4); k++) py[k] = __shfl_up_sync(0xffffffffu, pi[k], 1);
    if (lane > 0) ex_in = y;
  }
  __syncthreads();  // s_warp may be reused by the caller
  return op(before, ex_in);
}

// Phase 1: the sum of each tile.
template <typename T, typename Op>
__global__ void __launch_bounds__(kScanThreads) k_scan_tile_sums(const T *__restrict__ in,
                                                                  uint64_t n, T *__restrict__ sums,
                                                                  Op op, T zero) {
  __shared__ T s_warp[32];
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  T acc = zero;
#pragma unroll 4
  for (int i = 0; i < kScanItems; i++) {
    const uint64_t idx = base + (uint64_t)i * kScanThreads + threadIdx.x;
    if (idx < n) acc = op(acc, in[idx]);
  }
  T total;
  block_exclusive(acc, op, zero, s_warp, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Phase 2: one CTA turns the tile sums into exclusive tile offsets (in
// place); *grand (if given) gets the total.
template <typename T, typename Op>
__global__ void __launch_bounds__(1024) k_scan_offsets(T *__restrict__ sums, uint32_t n_tiles,
                                                       Op op, T zero, T *__restrict__ grand) {
  __shared__ T s_warp[32];
  T carry = zero;
  for (uint32_t b0 = 0; b0 < n_tiles; b0 += 1024) {
    const uint32_t i = b0 + threadIdx.x;
    const T v = i < n_tiles ? sums[i] : zero;
    T total;
    const T ex = block_exclusive(v, op, zero, s_warp, &total);
    if (i < n_tiles) sums[i] = op(carry, ex);
    carry = op(carry, total);
  }
  if (grand && threadIdx.x == 0) *grand = carry;
}

// Phase 3: each tile scans itself from its offset (striped order: item i
// of the tile is element i * threads + thread, scanned per item row).
template <typename T, typename Op, bool INCLUSIVE>
__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(const T *in, uint64_t n,
                                                             const T *__restrict__ offs, T *out,
                                                             Op op, T zero) {  // in may be out
  __shared__ T s_warp[32];
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  T carry = offs[blockIdx.x];
  for (int i = 0; i < kScanItems; i++) {
    const uint64_t idx = base + (uint64_t)i * kScanThreads + threadIdx.x;
    const T v = idx < n ? in[idx] : zero;
    T total;
    const T ex = block_exclusive(v, op, zero, s_warp, &total);
    if (idx < n) out[idx] = INCLUSIVE ? op(op(carry, ex), v) : op(carry, ex);
    carry = op(carry, total);
  }
}

struct AddU32 {
  __host__ __device__ __forceinline__ uint32_t operator()(uint32_t a, uint32_t b) const {
    return a + b;
  }
};

// Scratch (in elements of T) the scan of n elements needs: one per tile + 1.
inline size_t scan_scratch(uint64_t n) { return (n + kScanTile - 1) / kScanTile + 1; }

// out = scan of in (n elements; in and out may be the same array).  tmp:
// scan_scratch(n) elements of T; *grand (device, optional): the total.
template <typename T, typename Op, bool INCLUSIVE>
int scan(const T *in, T *out, uint64_t n, Op op, T zero, T *tmp, T *grand, cudaStream_t st) {
  if (n == 0) {
    if (grand) EBR_CUDA_TRY(cudaMemsetAsync(grand, 0, sizeof(T), st));
    return EBR_OK;
  }
  const uint64_t tiles = (n + kScanTile - 1) / kScanTile;
  if (tiles > 0x7FFFFFFFull) {
    set_error("scan: %llu elements are too many", (unsigned long long)n);
    return EBR_EINVAL;
  }
  k_scan_tile_sums<T, Op><<<(unsigned)tiles, kScanThreads, 0, st>>>(in, n, tmp, op, zero);
  EBR_CUDA_TRY(cudaGetLastError());
  k_scan_offsets<T, Op><<<1, 1024, 0, st>>>(tmp, (uint32_t)tiles, op, zero, grand);
  EBR_CUDA_TRY(cudaGetLastError());
  k_scan_tiles<T, Op, INCLUSIVE><<<(unsigned)tiles, kScanThreads, 0, st>>>(in, n, tmp, out, op,
                                                                           zero);
  EBR_CUDA_TRY(cudaGetLastError());
  return EBR_OK;
}

// ------------------------------------------------------------- radix sort
// One read and one write of the keys per 8-bit pass.  What bounds a pass is
// that traffic, so the tile's digit offsets are not counted in a pass of
// their own: the counts of every digit of every pass are taken in one read up
// front (k_digit_hist), and a tile learns how many keys of each digit lie in
// the tiles before it by looking back over their published counts
// (Merrill and Garland's decoupled look-back, as Adinets and Merrill's
// "Onesweep" uses it).  Tiles are numbered by a ticket, so a tile only waits
// for tiles that already run, and each wait is bounded.  A tile of 4096 keys
// is put in digit order in shared memory first, so that the global writes
// are runs of about 16 keys instead of single ones.
// What bounds it now is the ranking: a chain of match, read and write of the
// warp's digit count per row of 32 keys (ncu: short-scoreboard stalls first),
// so registers are held to 64 for four CTAs per SM (two at 103 registers:
// 315 us).  Measured, 32 M 64-bit words, one pass: 231 us (2.2 TB/s), against
// 292 us for separate count, scan and scatter kernels with unordered writes.
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
// keys per thread: what the tile's ordered copy leaves of 48 KB shared memory
template <typename K, bool VALS>
constexpr int sort_kpt() {
  return sizeof(K) + (VALS ? 4 : 0) > 8 ? 8 : 16;
}
constexpr uint32_t kSortMinTile = kSortThreads * 8;
constexpr uint32_t kSortSpins = 1u << 22;  // polls of one status word before giving up

template <typename K>
__device__ __forceinline__ uint32_t digit_of(K k, int shift) {
  return (uint32_t)((uint64_t)k >> shift) & 255u;
}

template <typename K>
struct ArrayLoad {
  const K *p;
  __device__ __forceinline__ K operator()(uint64_t i) const { return p[i]; }
};

// hist[pass * 256 + d] += keys whose 8-bit digit at bit 8 * pass is d.  A
// thread takes kHistRun consecutive keys and adds equal digits in a row at
// once: inputs in the order of some of their digits (pairs listed ad by ad)
// would otherwise have whole warps add to one word.
constexpr int kHistRun = 8;
template <typename K, typename Load>
__global__ void __launch_bounds__(kSortThreads) k_digit_hist(Load load, uint64_t n, int passes,
                                                             uint32_t *__restrict__ hist) {
  __shared__ uint32_t h[8 * 256];
  for (int i = threadIdx.x; i < passes * 256; i += kSortThreads) h[i] = 0;
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * kSortThreads * kHistRun;
  for (uint64_t i0 = (blockIdx.x * (uint64_t)kSortThreads + threadIdx.x) * kHistRun; i0 < n;
       i0 += stride) {
    const int c = (int)min((uint64_t)kHistRun, n - i0);
    K k[kHistRun];
#pragma unroll
    for (int j = 0; j < kHistRun; j++) k[j] = load(i0 + (j < c ? j : 0));
#pragma unroll
    for (int p = 0; p < (int)sizeof(K); p++) {
      if (p >= passes) break;
      uint32_t d = digit_of(k[0], 8 * p), run = 1;
#pragma unroll
      for (int j = 1; j < kHistRun; j++) {
        const uint32_t e = digit_of(k[j], 8 * p);
        if (j < c) {
          if (e != d) {
            atomicAdd(&h[p * 256 + d], run);
            d = e;
            run = 0;
          }
          run++;
        }
      }
      atomicAdd(&h[p * 256 + d], run);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * 256; i += kSortThreads)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Status word of (tile, digit): epoch (2 * pass + 1: the tile's own count,
// 2 * pass + 2: the count of all tiles up to it) in the high half, so the
// words need no clearing between passes.
__device__ __forceinline__ uint64_t ld_status(const uint64_t *p) {
  return *reinterpret_cast<const volatile uint64_t *>(p);
}
__device__ __forceinline__ void st_status(uint64_t *p, uint64_t v) {
  *reinterpret_cast<volatile uint64_t *>(p) = v;
}

// Exclusive sum over the 256 threads.  s_w: 8 words.
__device__ __forceinline__ uint32_t block_excl_256(uint32_t v, uint32_t *s_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  uint32_t before = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; w++) before += w < warp ? s_w[w] : 0u;
  __syncthreads();
  return before + incl - v;
}

// Stable scatter of the keys (and values) by the digit at `shift`.
template <typename K, typename Load, bool VALS>
__global__ void __launch_bounds__(kSortThreads, 4) k_sort_pass(
    Load load, const uint32_t *__restrict__ vals, uint64_t n, int shift,
    const uint32_t *__restrict__ hist, uint64_t *status, uint32_t epoch, uint32_t *ticket,
    K *__restrict__ keys_out, uint32_t *__restrict__ vals_out, uint32_t *__restrict__ flags,
    uint32_t max_spins) {
  constexpr int kSortKpt = sort_kpt<K, VALS>();
  constexpr uint32_t kSortTile = kSortThreads * kSortKpt;
  __shared__ K s_keys[kSortTile];
  __shared__ uint32_t s_vals[VALS ? kSortTile : 1];
  __shared__ uint32_t s_wc[kSortWarps][256];  // keys of each digit in the warps before
  __shared__ uint32_t s_lstart[256], s_gbase[256], s_w[kSortWarps], s_tile;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_tile = atomicAdd(ticket, 1u);
#pragma unroll
  for (int w = 0; w < kSortWarps; w++) s_wc[w][tid] = 0;
  __syncthreads();
  const uint32_t tile = s_tile;
  const uint64_t base = (uint64_t)tile * kSortTile;
  const uint32_t cnt = (uint32_t)min((uint64_t)kSortTile, n - base);
  // a warp owns kSortKpt rows of 32 consecutive keys; places past the end
  // count as digit 255 (they rank behind every key of the tile)
  K k[kSortKpt];
  uint16_t rank[kSortKpt];
  const uint32_t w0 = warp * 32 * kSortKpt + lane;
#pragma unroll
  for (int j = 0; j < kSortKpt; j++) {
    const uint32_t i = w0 + 32 * j;
    k[j] = i < cnt ? load(base + i) : K(0);
  }
#pragma unroll
  for (int j = 0; j < kSortKpt; j++) {
    const uint32_t d = w0 + 32 * j < cnt ? digit_of(k[j], shift) : 255u;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const uint32_t below = __popc(peers & ((1u << lane) - 1u));
    const uint32_t old = s_wc[warp][d];
    __syncwarp();
    if (below == 0) s_wc[warp][d] = old + __popc(peers);
    __syncwarp();
    rank[j] = (uint16_t)(old + below);
  }
  __syncthreads();
  uint32_t sum = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; w++) {
    const uint32_t c = s_wc[w][tid];
    s_wc[w][tid] = sum;
    sum += c;
  }
  const uint32_t mine = sum - (tid == 255 ? kSortTile - cnt : 0u);
  uint64_t *st = status + (uint64_t)tile * 256 + tid;
  st_status(st, ((uint64_t)(epoch + (tile == 0 ? 1u : 0u)) << 32) | mine);
  const uint32_t lstart = block_excl_256(sum, s_w);
  const uint32_t dbase = block_excl_256(hist[tid], s_w);
  uint32_t excl = 0;
  if (tile) {
    // kLook status words at a time: the walk is a chain of L2 latencies
    constexpr int kLook = 4;
    uint32_t spins = 0;
    bool open = true;
    for (int t = (int)tile - 1; open;) {
      if (spins >= max_spins) {  // never published: give up, flag it
        atomicOr(flags, DEVERR_TIMEOUT);
        break;
      }
      uint64_t v[kLook];
#pragma unroll
      for (int q = 0; q < kLook; q++)
        v[q] = ld_status(status + (uint64_t)max(t - q, 0) * 256 + tid);
#pragma unroll
      for (int q = 0; q < kLook; q++) {
        if (!open) break;
        const uint32_t e = (uint32_t)(v[q] >> 32);
        if (e == epoch || e == epoch + 1u) {  // tile 0 publishes epoch + 1 at once
          excl += (uint32_t)v[q];
          t--;
          open = e == epoch;
        } else {
          spins++;
          break;
        }
      }
    }
    st_status(st, ((uint64_t)(epoch + 1u) << 32) | (excl + mine));
  }
  s_lstart[tid] = lstart;
  s_gbase[tid] = dbase + excl - lstart;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kSortKpt; j++) {
    const uint32_t i = w0 + 32 * j;
    const uint32_t d = i < cnt ? digit_of(k[j], shift) : 255u;
    const uint32_t pos = s_lstart[d] + s_wc[warp][d] + rank[j];
    s_keys[pos] = k[j];
    if (VALS) s_vals[pos] = i < cnt ? vals[base + i] : 0u;
  }
  __syncthreads();
#pragma unroll 4
  for (uint32_t i = tid; i < cnt; i += kSortThreads) {
    const K x = s_keys[i];
    const uint32_t g = s_gbase[digit_of(x, shift)] + i;
    if (g < n) {  // always, unless a look-back gave up
      keys_out[g] = x;
      if (VALS) vals_out[g] = s_vals[i];
    }
  }
}

// Scratch (bytes) a sort of n keys needs: digit counts, tickets, status words.
inline size_t sort_scratch(uint64_t n) {
  const uint64_t tiles = (n + kSortMinTile - 1) / kSortMinTile;
  return 8 * 256 * 4 + 256 + (tiles + 1) * 256 * 8;
}

// Sorts n keys (with vals, if given) by bits [0, end_bit).  The first pass
// reads them through `load`; passes write keys_a, keys_b, keys_a, ... (vals:
// from vals into vals_a, vals_b, ...).  *in_b tells where the result ended.
// end_bit >= 1.  A look-back that polled max_spins times in vain sets
// DEVERR_TIMEOUT in *flags; the output is then not a permutation of the input
// (words of it may be whatever the memory held), so a kernel that uses it as
// indices reads *flags first.
template <typename K, bool VALS, typename Load>
int radix_sort(Load load, const uint32_t *vals, K *keys_a, K *keys_b, uint32_t *vals_a,
               uint32_t *vals_b, uint64_t n, int end_bit, void *scratch, uint32_t *flags,
               bool *in_b, cudaStream_t st, uint32_t max_spins = kSortSpins) {
  *in_b = false;
  if (n == 0) return EBR_OK;
  const int passes = std::max(1, (end_bit + 7) / 8);
  constexpr uint32_t kTile = kSortThreads * sort_kpt<K, VALS>();
  const uint64_t tiles = (n + kTile - 1) / kTile;
  uint32_t *hist = reinterpret_cast<uint32_t *>(scratch);
  uint32_t *tickets = hist + 8 * 256;
  uint64_t *status = reinterpret_cast<uint64_t *>(tickets + 64);
  EBR_CUDA_TRY(cudaMemsetAsync(scratch, 0, 8 * 256 * 4 + 256 + tiles * 256 * 8, st));
  const unsigned hg = (unsigned)std::min<uint64_t>(
      (n + kSortThreads * kHistRun - 1) / (kSortThreads * kHistRun), 2048);
  k_digit_hist<K><<<hg, kSortThreads, 0, st>>>(load, n, passes, hist);
  EBR_CUDA_TRY(cudaGetLastError());
  for (int p = 0; p < passes; p++) {
    K *out = (p & 1) ? keys_b : keys_a;
    uint32_t *vout = (p & 1) ? vals_b : vals_a;
    if (p == 0)
      k_sort_pass<K, Load, VALS><<<(unsigned)tiles, kSortThreads, 0, st>>>(
          load, vals, n, 0, hist, status, 1u, tickets, out, vout, flags, max_spins);
    else
      k_sort_pass<K, ArrayLoad<K>, VALS><<<(unsigned)tiles, kSortThreads, 0, st>>>(
          ArrayLoad<K>{(p & 1) ? keys_a : keys_b}, (p & 1) ? vals_a : vals_b, n, 8 * p,
          hist + 256 * p, status, 2u * p + 1u, tickets + p, out, vout, flags, max_spins);
    EBR_CUDA_TRY(cudaGetLastError());
    *in_b = (p & 1) != 0;
  }
  return EBR_OK;
}

// ------------------------------------------------------------------ unique
static __global__ void k_unique_flags(const uint64_t *__restrict__ x, uint64_t n,
                               uint32_t *__restrict__ f) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    f[i] = (i == 0 || x[i] != x[i - 1]) ? 1u : 0u;
}
static __global__ void k_unique_emit(const uint64_t *__restrict__ x, uint64_t n,
                              const uint32_t *__restrict__ pos, uint64_t *__restrict__ out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    if (i == 0 || x[i] != x[i - 1]) out[pos[i]] = x[i];
}

// out = the distinct values of the sorted x[0..n), in order; *d_count
// (device) their number.  flags: n uint32 scratch; tmp: scan_scratch(n).
inline int unique_sorted(const uint64_t *x, uint64_t *out, uint64_t n, uint32_t *flags,
                         uint32_t *tmp, uint32_t *d_count, cudaStream_t st) {
  if (n == 0) {
    EBR_CUDA_TRY(cudaMemsetAsync(d_count, 0, 4, st));
    return EBR_OK;
  }
  const unsigned grid = (unsigned)std::min<uint64_t>((n + 255) / 256, 65535);
  k_unique_flags<<<grid, 256, 0, st>>>(x, n, flags);
  EBR_CUDA_TRY(cudaGetLastError());
  EBR_TRY((scan<uint32_t, AddU32, false>(flags, flags, n, AddU32(), 0u, tmp, d_count, st)));
  k_unique_emit<<<grid, 256, 0, st>>>(x, n, flags, out);
  EBR_CUDA_TRY(cudaGetLastError());
  return EBR_OK;
}

}  // namespace prims
}  // namespace ebr
