// Index construction (Algorithm 1, Sec. 3.4) on the GPU.
//
// Step 1 (Block Grouping): every (k, v) pair becomes the word (h, k, l) with
// h = v >> 8 and l = v & 255, packed into as few bits as the key space and
// the inventory need; sorting the words puts each set B[k, h] in one run, and
// all runs of one window h = 256 consecutive ads side by side (repeated words
// are dropped, when there are any).
// Step 2 (Logarithmic Categorization): a run of n ads is one block of group
// g = ceil(log2 n), padded with zero bytes to 2^g slots.
// Step 3 (Storage Layout): per group, header[g] (h of each block) and
// values[g] (the low bytes) in (k, h) order, and keys[g], the row pointer
// giving each key's first block (keys[g][k] = group-g blocks with key < k).
//
// The words are sorted window-major because two of the three layouts the
// queries read follow the windows: one CTA per window finds its blocks and
// counts them (k_windows<false>), the counts are scanned, and a second walk
// (k_windows<true>) writes the window-major view; the key-major arrays then
// come from a stable sort of the blocks, half as many as the words, by
// (g, k) alone.  Measured, 2 M ads with 16 keys each (32 M pairs, 15 M
// blocks): 3.6 ms of device time for all of it with the forward table (2.7 ms
// without), against 8.0 ms without one when
// the words were sorted key-major by 7 three-kernel passes and the blocks
// again by 8 passes into the window order.
//
// The radix sort, the duplicate removal and the prefix sums are this
// library's own device primitives (ebr_prims.cuh).

#include <cstring>
#include <vector>

#include "ebr_internal.cuh"
#include "ebr_prims.cuh"

namespace ebr {
int launch_quantize(const float *x, uint64_t n, ebr_dtype dt, void *out, cudaStream_t st);
int launch_quantize_rows_fp8(const float *x, uint64_t n, uint32_t d, uint8_t *q, float *scale,
                             cudaStream_t st);

namespace {

// The (h, k, l) word of pair i (see above); kb: bits of a key.  Out-of-range
// keys and ads are flagged and read as 0.
struct PairLoad {
  const uint32_t *key, *ad;
  uint32_t n_keys, n_ads;
  int kb;
  uint32_t *flags;
  __device__ __forceinline__ uint64_t operator()(uint64_t i) const {
    uint32_t k = __ldg(key + i), a = __ldg(ad + i);
    if (k >= n_keys || a >= n_ads) {
      atomicOr(flags, (k >= n_keys ? DEVERR_BAD_BUILD_KEY : 0u) |
                          (a >= n_ads ? DEVERR_BAD_AD : 0u));
      k = k >= n_keys ? 0u : k;
      a = a >= n_ads ? 0u : a;
    }
    return ((uint64_t)(a >> 8) << (kb + 8)) | ((uint64_t)k << 8) | (a & 255u);
  }
};

// win_start[h] = first word of window h (n_win + 1 entries) of the sorted
// words, and the number of words equal to the one before them.  Nothing when
// the sort of the words gave up (*flags).
__global__ void k_window_starts(const uint64_t *__restrict__ x, uint32_t m, int wshift,
                                uint32_t n_win, uint32_t *__restrict__ win_start,
                                uint32_t *__restrict__ n_dup,
                                const uint32_t *__restrict__ flags) {
  if (*flags) return;
  uint32_t dup = 0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const uint64_t a = __ldg(x + i);
    const uint32_t h = (uint32_t)(a >> wshift);
    uint32_t from = 0;
    if (i) {
      const uint64_t p = __ldg(x + i - 1);
      dup += p == a ? 1u : 0u;
      from = (uint32_t)(p >> wshift) + 1u;
    }
    for (uint32_t w = from; w <= h; w++) win_start[w] = i;
    if (i == m - 1)
      for (uint32_t w = h + 1; w <= n_win; w++) win_start[w] = m;
  }
  dup = __reduce_add_sync(0xffffffffu, dup);
  if ((threadIdx.x & 31) == 0 && dup) atomicAdd(n_dup, dup);
}

__device__ __forceinline__ uint32_t ceil_log2(uint32_t n) {
  return n <= 1 ? 0u : 32u - __clz(n - 1);
}

constexpr int kWinThreads = 256, kWinWarps = kWinThreads / 32;
constexpr uint32_t kWinChunk = 4096;  // words walked at a time; a block has at most 256
constexpr uint32_t kWinRows = kWinChunk / kWinThreads;
constexpr uint32_t kFwdMaxWinQuads = 128;  // most forward quads of one window (176 KB to build)
// Shared memory a window of `quads` is put together in: the quads and their entries.
constexpr size_t fwd_win_smem(uint32_t quads, uint32_t quad_bytes) {
  return (size_t)quads * (quad_bytes + 1024);
}

struct WinArgs {
  const uint64_t *x;            // sorted distinct words
  const uint32_t *win_start;    // [n_win + 1]
  const uint32_t *n_dup;        // repeated words found (then nothing is walked)
  const uint32_t *flags;        // a sort before gave up (then neither)
  uint32_t n_win, n_ads;
  int kb;
  // counts (first walk)
  uint32_t *gcnt;               // [9][n_win + 1] blocks of each group and window
  uint16_t *ad_nkeys;           // [n_ads]
  uint32_t *max_keys;           // most keys of one ad
  uint32_t *run_quads;          // [8 n_win + 1] quads of each run of 32 ads; second walk: first quad
  // layout (second walk)
  const uint32_t *win_ptr[kGroups];
  uint32_t gstart[kGroups + 1];  // blocks of the groups before g
  uint32_t *wkey[kGroups];
  uint8_t *wvals[kGroups];
  uint32_t *bh;                 // [blocks] window of each block, in (g, h, k) order
  void *skey;                   // [blocks] (g, k) of each block, in that order
  uint32_t *sval;               // [blocks] its place in that order
  uint8_t *fwd;                 // forward table, or null
  const uint32_t *key_id;       // [n_keys] the keys' ids in it
  uint32_t quad_bytes, null_key;
};

// One CTA walks one window's words, kWinChunk at a time.  EMIT = false: blocks
// per group and keys per ad.  EMIT = true: the window's part of the
// window-major view, its part of the forward table (put together in shared
// memory: an ad's keys are ranked in word order, which is ascending, like the
// digits of a sort pass, and then put in the order in which the walk over the
// window's blocks meets them, so that FP32 sums over the table are the walk's)
// and the sort records of its blocks.  Bound by the
// read of the words (EMIT = false) and by the ranking and the byte stores of
// the values (true).
// K: type of a sort record, (g << kb) | k.
template <bool EMIT, typename K>
__global__ void __launch_bounds__(kWinThreads) k_windows(const __grid_constant__ WinArgs a) {
  __shared__ uint32_t s_mask[kWinChunk / 32 + 9];   // block heads of the chunk and 288 words on
  __shared__ uint32_t s_adcnt[256];
  __shared__ uint32_t s_g[kWinWarps][16];           // blocks per group: warp counts, then prefixes
  __shared__ uint32_t s_run[16];                    // blocks of each group in the chunks before
  __shared__ uint32_t s_blk[EMIT ? kWinChunk : 1];  // at a head: group << 16 | rank in its warp
  __shared__ uint16_t s_fr[EMIT ? kWinChunk : 1];   // rank of the word among its ad's in its warp
  __shared__ uint16_t s_lw[EMIT ? kWinWarps : 1][256];  // words per ad: warp counts, then prefixes
  __shared__ uint16_t s_lrun[256];                  // words per ad in the chunks before
  __shared__ uint32_t s_ubase[kGroups];
  extern __shared__ __align__(16) uint8_t s_fwd[];  // the window's quads
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (*a.flags || *a.n_dup) return;  // blocks are sets; the caller drops the repeated words first
  for (uint32_t w = blockIdx.x; w < a.n_win; w += gridDim.x) {
    const uint32_t b0 = a.win_start[w], b1 = a.win_start[w + 1];
    s_adcnt[tid] = 0;
    if (tid < 16) s_run[tid] = 0;
    const bool fwd = EMIT && a.fwd != nullptr;
    uint32_t q0 = 0, nq = 0;  // the window's first quad, and quads
    uint64_t *s_ent = nullptr;  // the quads' entries in key order: place in the walk << 32 | key id
    if (fwd) {
      s_lrun[tid] = 0;
      q0 = __ldg(a.run_quads + 8 * w);
      nq = __ldg(a.run_quads + 8 * w + 8) - q0;
      s_ent = reinterpret_cast<uint64_t *>(s_fwd + nq * a.quad_bytes);
      if (tid < kGroups) {  // the window's units in the groups before
        uint32_t u = 0;
        for (int g = 0; g < tid; g++)
          u += (a.win_ptr[g][w + 1] - a.win_ptr[g][w]) << (g >= 2 ? g - 2 : 0);
        s_ubase[tid] = u;
      }
      const uint32_t lo = (a.null_key & 0xFFFFu) * 0x10001u, hi = (a.null_key >> 16) * 0x1010101u;
      for (uint32_t i = tid; i < nq * a.quad_bytes / 4; i += kWinThreads)
        reinterpret_cast<uint32_t *>(s_fwd)[i] = (4 * i) % a.quad_bytes < 256u ? lo : hi;
    }
    uint32_t c0 = b0;
    while (c0 < b1) {
      __syncthreads();
      if (tid < 16)
        for (int q = 0; q < kWinWarps; q++) s_g[q][tid] = 0;
      if (fwd)
        for (int q = 0; q < kWinWarps; q++) s_lw[q][tid] = 0;
      // head bits of words [c0, c0 + chunk + 288); the end counts as a head
      for (uint32_t i = tid; i < kWinChunk + 288u; i += kWinThreads) {
        const uint32_t p = c0 + i;
        bool head = p == b1;
        if (p < b1) head = i == 0 || (__ldg(a.x + p) >> 8) != (__ldg(a.x + p - 1) >> 8);
        const uint32_t m = __ballot_sync(0xffffffffu, head);
        if (lane == 0) s_mask[i >> 5] = m;
      }
      __syncthreads();
      // the chunk ends at the window's end, or at its last head so that no
      // block is cut (words beyond it are walked in the next chunk)
      uint32_t end = b1 - c0;
      if (end > kWinChunk) {
        end = kWinChunk;
        while (!((s_mask[end >> 5] >> (end & 31u)) & 1u)) end--;
      }
      // a warp owns kWinRows rows of 32 consecutive words
      const uint32_t r0 = warp * 32 * kWinRows + lane;
#pragma unroll 4
      for (uint32_t r = 0; r < kWinRows; r++) {
        const uint32_t i = r0 + 32 * r;
        const bool in = i < end;
        const bool head = in && ((s_mask[i >> 5] >> lane) & 1u);
        uint32_t g = 15u;
        if (head) {  // next head: the block's length
          uint32_t wd = i >> 5;
          uint32_t m = s_mask[wd] & (0xFFFFFFFEu << lane);
          while (!m) m = s_mask[++wd];
          g = ceil_log2((wd << 5) + __ffs(m) - 1u - i);
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, g);
        const int leader = __ffs(peers) - 1;
        uint32_t old = 0;
        if (lane == leader && g < 15u) {
          old = s_g[warp][g];
          s_g[warp][g] = old + __popc(peers);
        }
        __syncwarp();
        if (EMIT) {
          old = __shfl_sync(0xffffffffu, old, leader);
          if (head) s_blk[i] = (g << 16) | (old + __popc(peers & ((1u << lane) - 1u)));
          if (fwd) {
            const uint32_t l = in ? (uint32_t)__ldg(a.x + c0 + i) & 255u : 256u + lane;
            const uint32_t same = __match_any_sync(0xffffffffu, l);
            const uint32_t below = __popc(same & ((1u << lane) - 1u));
            const uint32_t was = in ? s_lw[warp][l] : 0u;
            __syncwarp();
            if (in && below == 0) s_lw[warp][l] = (uint16_t)(was + __popc(same));
            __syncwarp();
            if (in) s_fr[i] = (uint16_t)(was + below);
          }
        } else if (in) {
          atomicAdd(&s_adcnt[(uint32_t)__ldg(a.x + c0 + i) & 255u], 1u);
        }
      }
      __syncthreads();
      if (tid < kGroups) {  // exclusive over the warps, from the chunks before
        uint32_t acc = s_run[tid];
        for (int q = 0; q < kWinWarps; q++) {
          const uint32_t c = s_g[q][tid];
          s_g[q][tid] = acc;
          acc += c;
        }
        s_run[tid] = acc;
      }
      if (fwd) {
        uint32_t acc = s_lrun[tid];
        for (int q = 0; q < kWinWarps; q++) {
          const uint32_t c = s_lw[q][tid];
          s_lw[q][tid] = (uint16_t)acc;
          acc += c;
        }
        s_lrun[tid] = (uint16_t)acc;
      }
      __syncthreads();
      if (EMIT) {
#pragma unroll 4
        for (uint32_t r = 0; r < kWinRows; r++) {
          const uint32_t i = r0 + 32 * r;
          if (i >= end) continue;
          const uint64_t word = __ldg(a.x + c0 + i);
          // this word's block starts at the last head at or before it
          uint32_t wd = i >> 5;
          uint32_t m = s_mask[wd] & (0xFFFFFFFFu >> (31 - lane));
          while (!m) m = s_mask[--wd];
          const uint32_t hp = (wd << 5) + 31u - __clz(m);
          const uint32_t e = s_blk[hp], g = e >> 16;
          const uint32_t rank =
              a.win_ptr[g][w] + s_g[hp / (32 * kWinRows)][g] + (e & 0xFFFFu);
          const uint32_t key = (uint32_t)((word >> 8) & ((1ull << a.kb) - 1ull));
          a.wvals[g][((uint64_t)rank << g) + (i - hp)] = (uint8_t)word;
          if (fwd) {
            const uint32_t l = (uint32_t)word & 255u, fr = s_lw[warp][l] + s_fr[i];
            const uint32_t qd = __ldg(a.run_quads + 8 * w + (l >> 5)) - q0 + (fr >> 2);
            // its place in the walk of the batched scan (walk_window): unit U of
            // the window's, slot s of the unit; 64 units at a time, in each
            // all first slots before all second ones
            const uint32_t in_g = s_g[hp / (32 * kWinRows)][g] + (e & 0xFFFFu), off = i - hp;
            const uint32_t U = s_ubase[g] + (g >= 2 ? (in_g << (g - 2)) + (off >> 2) : in_g);
            const uint32_t ord = ((U >> 6) << 8) | ((off & 3u) << 6) | (U & 63u);
            s_ent[qd * 128 + (l & 31u) * 4 + (fr & 3u)] =
                ((uint64_t)ord << 32) | __ldg(a.key_id + key);
          }
          if (hp == i) {
            const uint32_t q = a.gstart[g] + rank;
            a.wkey[g][rank] = key;
            a.bh[q] = w;
            reinterpret_cast<K *>(a.skey)[q] = ((K)g << a.kb) | (K)key;
            a.sval[q] = q;
          }
        }
      }
      c0 += end;
    }
    if (!EMIT) {
      __syncthreads();
      if (tid < kGroups) a.gcnt[(uint64_t)tid * (a.n_win + 1) + w] = s_run[tid];
      const uint32_t ad = w * 256u + tid, c = s_adcnt[tid];
      if (ad < a.n_ads) a.ad_nkeys[ad] = (uint16_t)c;
      const uint32_t mx = __reduce_max_sync(0xffffffffu, c);
      if (lane == 0 && mx) atomicMax(a.max_keys, mx);
      if (lane == 0) a.run_quads[8 * w + warp] = (mx + 3) / 4;
    } else if (fwd) {
      __syncthreads();
      // A warp per run, ad by ad: a lane per key (two with over 32), its row
      // the number of the ad's keys before it in the walk.
      const uint32_t qd = __ldg(a.run_quads + 8 * w + warp) - q0;
      for (uint32_t l = 0; l < 32; l++) {
        const uint32_t n = s_lrun[warp * 32 + l];
        const uint64_t *ent = s_ent + qd * 128 + l * 4;
        for (uint32_t i0 = 0; i0 < n; i0 += 32) {
          const uint32_t i = i0 + lane;
          const uint64_t x = i < n ? ent[(i >> 2) * 128 + (i & 3u)] : ~0ull;
          uint32_t r = 0;
          for (uint32_t j0 = 0; j0 < n; j0 += 32) {
            const uint32_t j = j0 + lane;
            const uint32_t o =
                j < n ? (uint32_t)(ent[(j >> 2) * 128 + (j & 3u)] >> 32) : 0xFFFFFFFFu;
            for (uint32_t t = 0; t < min(32u, n - j0); t++)
              r += __shfl_sync(0xffffffffu, o, t) < (uint32_t)(x >> 32) ? 1u : 0u;
          }
          if (i < n) {
            uint8_t *quad = s_fwd + (qd + (r >> 2)) * a.quad_bytes;
            reinterpret_cast<uint16_t *>(quad)[l * 4 + (r & 3u)] = (uint16_t)x;
            if (a.quad_bytes > 256u) quad[256 + l * 4 + (r & 3u)] = (uint8_t)(x >> 16);
          }
        }
      }
      __syncthreads();
      uint4 *dst = reinterpret_cast<uint4 *>(a.fwd + (uint64_t)q0 * a.quad_bytes);
      for (uint32_t i = tid; i < nq * a.quad_bytes / 16; i += kWinThreads)
        dst[i] = reinterpret_cast<const uint4 *>(s_fwd)[i];
    }
    __syncthreads();
  }
}

// win_ptr[g][h] (per group) from the scan over all groups' counts, and the
// totals per group (gc, 9 words).
__global__ void k_win_ptrs(const uint32_t *__restrict__ scan, uint32_t n_win,
                           uint32_t *__restrict__ win_ptr, uint32_t *__restrict__ gc) {
  const uint32_t g = blockIdx.y;
  const uint64_t row = (uint64_t)g * (n_win + 1);
  const uint32_t base = scan[row];
  for (uint32_t h = blockIdx.x * blockDim.x + threadIdx.x; h <= n_win;
       h += gridDim.x * blockDim.x) {
    const uint32_t v = scan[row + h] - base;
    win_ptr[row + h] = v;
    if (h == n_win) gc[g] = v;
  }
}

struct KeyArgs {
  const uint32_t *bh;
  const uint8_t *wvals[kGroups];
  uint32_t *header[kGroups];
  uint8_t *values[kGroups];
  uint32_t gstart[kGroups + 1];
  int kb;
  const uint32_t *flags;  // the sort of the blocks gave up (then nothing is written)
};

// p-th block in (g, k, h) order: its header and its 2^g value bytes, from its
// place q in the window-major view.
template <typename K>
__global__ void k_key_major(const K *__restrict__ skey, const uint32_t *__restrict__ sval,
                            uint32_t nb, const __grid_constant__ KeyArgs a) {
  if (*a.flags) return;
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < nb; p += gridDim.x * blockDim.x) {
    const uint32_t g = (uint32_t)(skey[p] >> a.kb), q = sval[p];
    const uint64_t rank = p - a.gstart[g], src = q - a.gstart[g];
    a.header[g][rank] = __ldg(a.bh + q);
    const uint8_t *from = a.wvals[g] + (src << g);
    uint8_t *to = a.values[g] + (rank << g);
    if (g >= 4) {
      for (uint32_t s = 0; s < (1u << g); s += 16)
        *reinterpret_cast<uint4 *>(to + s) = __ldg(reinterpret_cast<const uint4 *>(from + s));
    } else if (g == 3) {
      *reinterpret_cast<uint2 *>(to) = __ldg(reinterpret_cast<const uint2 *>(from));
    } else if (g == 2) {
      *reinterpret_cast<uint32_t *>(to) = __ldg(reinterpret_cast<const uint32_t *>(from));
    } else if (g == 1) {
      *reinterpret_cast<uint16_t *>(to) = __ldg(reinterpret_cast<const uint16_t *>(from));
    } else {
      *to = __ldg(from);
    }
  }
}

// keys[g][k] = group-g blocks with key < k: a binary search of (g, k) in the
// sorted records.
template <typename K>
__global__ void k_row_ptrs(const K *__restrict__ skey, const __grid_constant__ KeyArgs a,
                           uint32_t n_keys, uint32_t *__restrict__ keys) {
  const uint32_t g = blockIdx.y;
  for (uint64_t k = blockIdx.x * blockDim.x + threadIdx.x; k <= n_keys;
       k += gridDim.x * blockDim.x) {
    uint32_t lo = a.gstart[g], hi = a.gstart[g + 1];
    const K t = ((K)g << a.kb) + (K)k;  // k == n_keys: past the group's last key
    if (k == n_keys) lo = hi;
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if (skey[mid] < t) lo = mid + 1; else hi = mid;
    }
    keys[(uint64_t)g * ((uint64_t)n_keys + 1) + k] = lo - a.gstart[g];
  }
}

struct WinPtrs {
  const uint32_t *p[kGroups];
};

// Bytes a window's segments of the window-major view occupy once each segment
// is widened to 16-byte boundaries (the staging size of the fused scan).
// Also: the most 32-unit work chunks any window has (a unit is one 4-slot
// word in groups >= 2, one block in groups 0 and 1).
__global__ void k_win_bytes(WinPtrs wp, uint32_t n_win, unsigned int *out_max) {
  uint32_t mx = 0, mc = 0, ms = 0;
  for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < n_win; w += gridDim.x * blockDim.x) {
    uint64_t total = 0, chunks = 0, slots = 0;
    for (int g = 0; g < kGroups; g++) {
      const uint64_t lo = wp.p[g][w], hi = wp.p[g][w + 1];
      if (hi == lo) continue;
      const uint64_t k0 = (lo * 4) & ~15ull, k1 = (hi * 4 + 15) & ~15ull;
      const uint64_t v0 = (lo << g) & ~15ull, v1 = ((hi << g) + 15) & ~15ull;
      total += (k1 - k0) + (v1 - v0);
      chunks += (((hi - lo) << (g >= 2 ? g - 2 : 0)) + 31) >> 5;
      slots += (hi - lo) << g;
    }
    mx = max(mx, (uint32_t)min(total, (uint64_t)0xFFFFFFFFu));
    mc = max(mc, (uint32_t)min(chunks, (uint64_t)0xFFFFFFFFu));
    ms = max(ms, (uint32_t)min(slots, (uint64_t)0xFFFFFFFFu));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  mc = __reduce_max_sync(0xffffffffu, mc);
  ms = __reduce_max_sync(0xffffffffu, ms);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out_max, mx);
    atomicMax(out_max + 1, mc);
    atomicMax(out_max + 2, ms);
  }
}

// Key popularity from a sample of the sorted words (every step-th one).
__global__ void k_sample_keys(const uint64_t *__restrict__ x, uint32_t m, uint32_t step, int kb,
                              uint32_t *__restrict__ cnt) {
  for (uint64_t i = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) * step; i < m;
       i += (uint64_t)gridDim.x * blockDim.x * step)
    atomicAdd(&cnt[(x[i] >> 8) & ((1ull << kb) - 1ull)], 1u);
}
// Sort records that put the most frequent keys first (equal counts: by key).
constexpr int kPopBits = 24;
__global__ void k_pop_records(uint32_t *__restrict__ cnt, uint32_t n, uint32_t *__restrict__ key) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    cnt[i] = (1u << kPopBits) - 1u - min(cnt[i], (1u << kPopBits) - 1u);
    key[i] = i;
  }
}
__global__ void k_pop_ids(const uint32_t *__restrict__ key, uint32_t n, uint32_t *__restrict__ id,
                          const uint32_t *__restrict__ flags) {
  if (*flags) return;  // the sort gave up
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    id[key[i]] = i;
}

// Most quads of 1, 2, 4 and 8 aligned runs (out[0 .. 3]) and all of them (out[4]).
__global__ void k_fwd_max(const uint32_t *__restrict__ off, uint32_t n_win,
                          uint32_t *__restrict__ out) {
  uint32_t mx[4] = {0, 0, 0, 0};
  for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < n_win; w += gridDim.x * blockDim.x) {
    uint32_t o[9];
#pragma unroll
    for (int i = 0; i < 9; i++) o[i] = off[8 * (uint64_t)w + i];
#pragma unroll
    for (int g = 0; g < 4; g++)
#pragma unroll
      for (int i = 0; i < 8; i += 1 << g) mx[g] = max(mx[g], o[i + (1 << g)] - o[i]);
    if (w == n_win - 1) out[4] = o[8];
  }
#pragma unroll
  for (int g = 0; g < 4; g++) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, mx[g]);
    if ((threadIdx.x & 31) == 0) atomicMax(out + g, m);
  }
}

inline int grid_for(uint64_t n, int threads = 256, int cap = 1 << 16) {
  uint64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > (uint64_t)cap) b = cap;
  return (int)b;
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace
}  // namespace ebr

using namespace ebr;

// Bits that hold every value below n.
static int bits_for(uint64_t n) {
  int b = 0;
  while (b < 64 && (1ull << b) < n) b++;
  return b;
}

// True where a kernel can read 32-bit words at p in place (device memory of
// this device, on a word boundary; a copy takes any address).
static bool on_device(const void *p, int device) {
  if (reinterpret_cast<uintptr_t>(p) % 4) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice && at.device == device;
}

// The (g, k) sort of the blocks and the key-major arrays from it.
template <typename K>
static int build_key_major(ebr_index *ix, uint32_t nb, KeyArgs &ka, void *k0, void *k1, void *k2,
                           uint32_t *v0, uint32_t *v1, uint32_t *v2, void *scratch,
                           uint32_t *flags, uint32_t max_spins, cudaStream_t st) {
  const K *sk = (const K *)k0;
  const uint32_t *sv = v0;
  if (nb) {
    bool in_b = false;
    EBR_TRY((prims::radix_sort<K, true>(prims::ArrayLoad<K>{(const K *)k0}, v0, (K *)k1, (K *)k2,
                                        v1, v2, nb, ka.kb + 4, scratch, flags, &in_b, st,
                                        max_spins)));
    sk = (const K *)(in_b ? k2 : k1);
    sv = in_b ? v2 : v1;
    k_key_major<K><<<grid_for(nb), 256, 0, st>>>(sk, sv, nb, ka);
    EBR_CUDA_TRY(cudaGetLastError());
  }
  k_row_ptrs<K><<<dim3(grid_for((uint64_t)ix->n_keys + 1), kGroups), 256, 0, st>>>(
      sk, ka, ix->n_keys, (uint32_t *)ix->mem_keys.p);
  EBR_CUDA_TRY(cudaGetLastError());
  return EBR_OK;
}

// Device words the build reads back in one copy.
struct BuildCounts {
  uint32_t flags, n_dup, max_keys, gc[kGroups], win_max[3], fwd[5], m_unique;
};

// faults: see ebr_debug_build_index.  *forward: whether a forward table may be
// built; on return, whether one was begun.
static int build_impl(const ebr_index_desc *desc, ebr_index *ix, uint32_t faults, bool *forward,
                      cudaStream_t st) {
  const bool may_forward = *forward;
  *forward = false;
  // polls of a look-back in the sorts of the pairs, the keys by popularity, the blocks
  auto spins = [&](uint32_t fault) { return faults & fault ? 0u : prims::kSortSpins; };
  const uint64_t nnz = desc->nnz;
  const uint32_t n_keys = desc->n_keys, n_ads = desc->n_ads, n_win = (n_ads + 255) / 256;
  const int kb = bits_for(n_keys), hb = bits_for(n_win);
  ix->n_win = n_win;
  DevBuf in, pool, wpool, blocks, pop;
  int rc = EBR_OK;
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
#define BTRY(expr)                  \
  do {                              \
    rc = (expr);                    \
    if (rc != EBR_OK) goto done;    \
  } while (0)
#define BCUDA(expr)                                                                       \
  do {                                                                                    \
    cudaError_t _e = (expr);                                                              \
    if (_e != cudaSuccess) {                                                              \
      set_error("%s: %s", #expr, cudaGetErrorString(_e));                                 \
      rc = EBR_ECUDA;                                                                     \
      goto done;                                                                          \
    }                                                                                     \
  } while (0)
  {
    const uint32_t *pk = desc->post_key, *pa = desc->post_ad;
    for (auto &e : ev) BCUDA(cudaEventCreate(&e));
    // Inputs that cannot be read in place are brought over first (not part of build_ms).
    if (nnz && !(on_device(pk, ix->device) && on_device(pa, ix->device))) {
      BTRY(dev_alloc(in, nnz * 8));
      BCUDA(cudaMemcpyAsync(in.p, pk, nnz * 4, cudaMemcpyDefault, st));
      BCUDA(cudaMemcpyAsync((uint32_t *)in.p + nnz, pa, nnz * 4, cudaMemcpyDefault, st));
      pk = (const uint32_t *)in.p;
      pa = pk + nnz;
    }
    // words and the sort's scratch in one allocation, per-window arrays in another
    const size_t words_b = align_up(nnz * 8, 256);
    const size_t scr_b = align_up(
        std::max(prims::sort_scratch(nnz), (nnz + prims::scan_scratch(nnz) + 64) * 4), 256);
    const size_t gw_b = align_up((size_t)kGroups * (n_win + 1) * 4, 256);
    const size_t ws_b = align_up(((size_t)n_win + 1) * 4, 256);
    const size_t st_b = align_up(prims::scan_scratch((uint64_t)kGroups * (n_win + 1)) * 4, 256);
    const uint64_t n_runs = 8ull * n_win;
    BTRY(dev_alloc(pool, 2 * words_b + scr_b));
    BTRY(dev_alloc(wpool, 256 + ws_b + gw_b + st_b));
    BTRY(dev_alloc(ix->ad_nkeys, (size_t)n_ads * 2));
    BTRY(dev_alloc(ix->mem_winptr, (size_t)kGroups * (n_win + 1) * 4));
    BTRY(dev_alloc(ix->mem_fwd_off, (n_runs + 1) * 4));
    ix->fwd_off = (uint32_t *)ix->mem_fwd_off.p;
    uint64_t *wa = (uint64_t *)pool.p, *wb = (uint64_t *)((char *)pool.p + words_b);
    void *scratch = (char *)pool.p + 2 * words_b;
    BuildCounts *cnt = (BuildCounts *)wpool.p;
    uint32_t *win_start = (uint32_t *)((char *)wpool.p + 256);
    uint32_t *gcnt = (uint32_t *)((char *)wpool.p + 256 + ws_b);
    uint32_t *stmp = (uint32_t *)((char *)wpool.p + 256 + ws_b + gw_b);
    BuildCounts hc;
    memset(&hc, 0, sizeof(hc));
    uint32_t m = (uint32_t)nnz;
    WinArgs w;
    memset(&w, 0, sizeof(w));
    w.win_start = win_start;
    w.n_dup = &cnt->n_dup;
    w.flags = &cnt->flags;
    w.n_win = n_win;
    w.n_ads = n_ads;
    w.kb = kb;
    w.gcnt = gcnt;
    w.ad_nkeys = (uint16_t *)ix->ad_nkeys.p;
    w.max_keys = &cnt->max_keys;
    w.run_quads = ix->fwd_off;
    for (int g = 0; g < kGroups; g++) {
      ix->win_ptr[g] = (uint32_t *)ix->mem_winptr.p + (size_t)g * (n_win + 1);
      w.win_ptr[g] = ix->win_ptr[g];
    }

    BCUDA(cudaEventRecord(ev[0], st));
    BCUDA(cudaMemsetAsync(wpool.p, 0, 256 + ws_b + gw_b, st));
    BCUDA(cudaMemsetAsync(ix->fwd_off, 0, (n_runs + 1) * 4, st));
    if (nnz) {
      bool in_b = false;
      BTRY((prims::radix_sort<uint64_t, false>(PairLoad{pk, pa, n_keys, n_ads, kb, &cnt->flags},
                                               nullptr, wa, wb, nullptr, nullptr, nnz,
                                               hb + kb + 8, scratch, &cnt->flags, &in_b, st,
                                               spins(EBR_FAULT_SORT_PAIRS))));
      if (in_b) std::swap(wa, wb);  // wa: sorted
    }
    // blocks and keys per window; taken again when repeated words turn up
    for (int round = 0; round < 2; round++) {
      w.x = wa;
      if (m) {
        k_window_starts<<<grid_for(m), 256, 0, st>>>(wa, m, kb + 8, n_win, win_start,
                                                     &cnt->n_dup, &cnt->flags);
        BCUDA(cudaGetLastError());
      }
      k_windows<false, uint32_t><<<std::min<uint32_t>(n_win, 1u << 20), kWinThreads, 0, st>>>(w);
      BCUDA(cudaGetLastError());
      BTRY((prims::scan<uint32_t, prims::AddU32, false>(gcnt, gcnt, (uint64_t)kGroups * (n_win + 1),
                                                        prims::AddU32(), 0u, stmp, nullptr, st)));
      k_win_ptrs<<<dim3(grid_for((uint64_t)n_win + 1, 256, 256), kGroups), 256, 0, st>>>(
          gcnt, n_win, (uint32_t *)ix->mem_winptr.p, cnt->gc);
      BCUDA(cudaGetLastError());
      WinPtrs wp;
      for (int g = 0; g < kGroups; g++) wp.p[g] = ix->win_ptr[g];
      k_win_bytes<<<grid_for(n_win), 256, 0, st>>>(wp, n_win, cnt->win_max);
      BCUDA(cudaGetLastError());
      BTRY((prims::scan<uint32_t, prims::AddU32, false>(ix->fwd_off, ix->fwd_off, n_runs + 1,
                                                        prims::AddU32(), 0u, stmp, nullptr, st)));
      k_fwd_max<<<grid_for(n_win), 256, 0, st>>>(ix->fwd_off, n_win, cnt->fwd);
      BCUDA(cudaGetLastError());
      BCUDA(cudaMemcpyAsync(&hc, cnt, sizeof(hc), cudaMemcpyDeviceToHost, st));
      BCUDA(cudaStreamSynchronize(st));
      if (hc.flags) {
        rc = check_device_flags(hc.flags, "ebr_build_index");
        goto done;
      }
      if (!hc.n_dup) break;
      uint32_t *uflags = (uint32_t *)scratch;
      BTRY(prims::unique_sorted(wa, wb, m, uflags, uflags + m, &cnt->m_unique, st));
      std::swap(wa, wb);
      m -= hc.n_dup;
      BCUDA(cudaMemsetAsync(wpool.p, 0, 256 + ws_b + gw_b, st));
      BCUDA(cudaMemsetAsync(ix->fwd_off, 0, (n_runs + 1) * 4, st));
    }
    ix->nnz_unique = m;
    ix->max_keys_per_ad = hc.max_keys;
    ix->max_win_bytes = hc.win_max[0];
    ix->max_win_chunks = hc.win_max[1];
    ix->max_win_slots = hc.win_max[2];
    if (m == 0 || ix->max_keys_per_ad > 65535) dev_free(ix->ad_nkeys);  // counts that do not fit

    size_t hdr_off[kGroups], val_off[kGroups], hdr_total = 0, val_total = 0;
    KeyArgs ka;
    memset(&ka, 0, sizeof(ka));
    ka.kb = kb;
    ka.flags = &cnt->flags;
    for (int g = 0; g < kGroups; g++) {
      ix->n_blocks[g] = hc.gc[g];
      hdr_off[g] = hdr_total;
      val_off[g] = val_total;
      hdr_total += align_up((size_t)hc.gc[g] * 4, 256);
      val_total += align_up((size_t)hc.gc[g] << g, 256);
      ka.gstart[g + 1] = w.gstart[g + 1] = w.gstart[g] + hc.gc[g];
    }
    const uint32_t nb = w.gstart[kGroups];
    BTRY(dev_alloc(ix->mem_keys, (size_t)kGroups * ((size_t)n_keys + 1) * 4));
    BTRY(dev_alloc(ix->mem_header, hdr_total + 256));
    BTRY(dev_alloc(ix->mem_values, val_total + 256));
    BTRY(dev_alloc(ix->mem_wkey, hdr_total + 256));
    BTRY(dev_alloc(ix->mem_wvals, val_total + 256));
    for (int g = 0; g < kGroups; g++) {
      ix->keys[g] = (uint32_t *)ix->mem_keys.p + (size_t)g * ((size_t)n_keys + 1);
      ix->header[g] = (uint32_t *)((char *)ix->mem_header.p + hdr_off[g]);
      ix->values[g] = (uint8_t *)ix->mem_values.p + val_off[g];
      ix->wkey[g] = (uint32_t *)((char *)ix->mem_wkey.p + hdr_off[g]);
      ix->wvals[g] = (uint8_t *)ix->mem_wvals.p + val_off[g];
      w.wkey[g] = ix->wkey[g];
      w.wvals[g] = ix->wvals[g];
      ka.header[g] = ix->header[g];
      ka.values[g] = ix->values[g];
      ka.wvals[g] = ix->wvals[g];
    }
    // The forward table: key spaces that fit 24 bits, windows whose quads fit
    // the emitting CTA's shared memory, and padding of at most twice the
    // postings plus a quad per ad (one quad is what an ad with one key needs).
    ix->fwd_quads = hc.fwd[4];
    ix->fwd_quad_bytes = n_keys < 65536u ? 256u : 384u;
    for (int g = 0; g < 4; g++) ix->fwd_max_quads[g] = hc.fwd[g];
    *forward = may_forward && m && n_keys < (1u << 24) - 1u && hc.fwd[3] <= kFwdMaxWinQuads &&
               (uint64_t)hc.fwd[4] * 128 <= 2ull * m + 4ull * n_ads;
    if (*forward) {
      BTRY(faults & EBR_FAULT_FORWARD_MEM
               ? EBR_ENOMEM
               : dev_alloc(ix->mem_fwd, (size_t)ix->fwd_quads * ix->fwd_quad_bytes + 256));
      ix->fwd = w.fwd = (uint8_t *)ix->mem_fwd.p;
      w.quad_bytes = ix->fwd_quad_bytes;
      w.null_key = n_keys;
      // The table names a key by its popularity rank (over a sample of up to
      // 2^20 postings), so that the terms most gathers want are the first
      // ones, which the scans hold in shared memory.
      const size_t kn_b = align_up((size_t)n_keys * 4, 256);
      BTRY(dev_alloc(ix->mem_key_id, kn_b));
      ix->key_id = (uint32_t *)ix->mem_key_id.p;
      w.key_id = ix->key_id;
      BTRY(dev_alloc(pop, 6 * kn_b + prims::sort_scratch(n_keys)));
      uint32_t *pc[6];
      for (int i = 0; i < 6; i++) pc[i] = (uint32_t *)((char *)pop.p + i * kn_b);
      const uint32_t step = std::max<uint32_t>(1, m >> 20);
      bool in_b = false;
      BCUDA(cudaMemsetAsync(pc[0], 0, kn_b, st));
      k_sample_keys<<<grid_for(m / step + 1), 256, 0, st>>>(w.x, m, step, kb, pc[0]);
      BCUDA(cudaGetLastError());
      k_pop_records<<<grid_for(n_keys), 256, 0, st>>>(pc[0], n_keys, pc[1]);
      BCUDA(cudaGetLastError());
      BTRY((prims::radix_sort<uint32_t, true>(prims::ArrayLoad<uint32_t>{pc[0]}, pc[1], pc[2], pc[3],
                                              pc[4], pc[5], n_keys, kPopBits,
                                              (char *)pop.p + 6 * kn_b, &cnt->flags, &in_b, st,
                                              spins(EBR_FAULT_SORT_KEYS))));
      k_pop_ids<<<grid_for(n_keys), 256, 0, st>>>(in_b ? pc[5] : pc[4], n_keys, ix->key_id,
                                                  &cnt->flags);
      BCUDA(cudaGetLastError());
    }
    const size_t fwd_smem = w.fwd ? fwd_win_smem(hc.fwd[3], w.quad_bytes) : 0;
    // blocks: window of each, then (key, place) records three times over (the
    // sort's input and its two buffers); the sort's scratch is the words'
    const bool k32 = kb + 4 <= 32;
    const size_t rk_b = align_up((size_t)nb * (k32 ? 4 : 8), 256), rv_b = align_up((size_t)nb * 4, 256);
    const size_t bscr_b = align_up(prims::sort_scratch(nb), 256);
    BTRY(dev_alloc(blocks, 4 * rv_b + 3 * rk_b + bscr_b));
    char *bp = (char *)blocks.p;
    w.bh = (uint32_t *)bp;
    w.sval = (uint32_t *)(bp + rv_b);
    uint32_t *v1 = (uint32_t *)(bp + 2 * rv_b), *v2 = (uint32_t *)(bp + 3 * rv_b);
    w.skey = bp + 4 * rv_b;
    void *k1 = bp + 4 * rv_b + rk_b, *k2 = bp + 4 * rv_b + 2 * rk_b;
    void *bscr = bp + 4 * rv_b + 3 * rk_b;
    ka.bh = w.bh;

    BCUDA(cudaEventRecord(ev[1], st));
    BCUDA(cudaMemsetAsync(ix->mem_wvals.p, 0, val_total + 256, st));
    if (nb) {
      const uint32_t grid = std::min<uint32_t>(n_win, 1u << 20);
      auto kern = k32 ? k_windows<true, uint32_t> : k_windows<true, uint64_t>;
      BCUDA(allow_smem(kern, fwd_win_smem(kFwdMaxWinQuads, 384)));
      kern<<<grid, kWinThreads, fwd_smem, st>>>(w);
      BCUDA(cudaGetLastError());
    }
    BCUDA(cudaEventRecord(ev[2], st));
    if (k32)
      BTRY(build_key_major<uint32_t>(ix, nb, ka, w.skey, k1, k2, w.sval, v1, v2, bscr, &cnt->flags,
                                     spins(EBR_FAULT_SORT_BLOCKS), st));
    else
      BTRY(build_key_major<uint64_t>(ix, nb, ka, w.skey, k1, k2, w.sval, v1, v2, bscr, &cnt->flags,
                                     spins(EBR_FAULT_SORT_BLOCKS), st));
    BCUDA(cudaEventRecord(ev[3], st));
    BCUDA(cudaMemcpyAsync(&hc, cnt, sizeof(hc), cudaMemcpyDeviceToHost, st));
    BCUDA(cudaStreamSynchronize(st));
    if (hc.flags) {
      rc = check_device_flags(hc.flags, "ebr_build_index");
      goto done;
    }
    // Algorithm 1 is everything but the walk that writes the window-major view
    float a1 = 0.f, a2 = 0.f;
    BCUDA(cudaEventElapsedTime(&a1, ev[0], ev[1]));
    BCUDA(cudaEventElapsedTime(&ix->wm_build_ms, ev[1], ev[2]));
    BCUDA(cudaEventElapsedTime(&a2, ev[2], ev[3]));
    ix->build_ms = a1 + a2;
  }
done:
  for (DevBuf *b : {&in, &pool, &wpool, &blocks, &pop}) dev_free(*b);
  for (auto &e : ev)
    if (e) cudaEventDestroy(e);
  return rc;
#undef BTRY
#undef BCUDA
}

static int upload_embeddings(const ebr_index_desc *desc, ebr_index *ix, cudaStream_t st) {
  const uint64_t n = (uint64_t)desc->n_ads * desc->d;
  EBR_TRY(dev_alloc(ix->emb_f32, n * 4));
  EBR_CUDA_TRY(cudaMemcpyAsync(ix->emb_f32.p, desc->emb_f32, n * 4, cudaMemcpyDefault, st));
  if (desc->emb_dtype == EBR_BF16) {
    EBR_TRY(dev_alloc(ix->emb_q, n * 2));
    EBR_TRY(launch_quantize((const float *)ix->emb_f32.p, n, EBR_BF16, ix->emb_q.p, st));
  } else if (desc->emb_dtype == EBR_FP8E4M3) {
    EBR_TRY(dev_alloc(ix->emb_q, n));
    EBR_TRY(dev_alloc(ix->emb_scale, (uint64_t)desc->n_ads * 4));
    EBR_TRY(launch_quantize_rows_fp8((const float *)ix->emb_f32.p, desc->n_ads, desc->d,
                                     (uint8_t *)ix->emb_q.p, (float *)ix->emb_scale.p, st));
  }
  EBR_CUDA_TRY(cudaStreamSynchronize(st));
  return EBR_OK;
}

extern "C" void ebr_index_free(ebr_index *ix) {
  if (!ix) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(ix->device);
  dev_free(ix->mem_keys);
  dev_free(ix->mem_header);
  dev_free(ix->mem_values);
  dev_free(ix->mem_wkey);
  dev_free(ix->mem_wvals);
  dev_free(ix->mem_winptr);
  dev_free(ix->mem_fwd);
  dev_free(ix->mem_fwd_off);
  dev_free(ix->mem_key_id);
  dev_free(ix->ad_nkeys);
  dev_free(ix->emb_f32);
  dev_free(ix->emb_q);
  dev_free(ix->emb_scale);
  Workspace &w = ix->ws;
  for (DevBuf *b : {&w.wide, &w.w_dense, &w.wq, &w.lens, &w.scan, &w.work, &w.scan_tmp, &w.cand,
                    &w.ctrl, &w.io_in, &w.io_out, &w.route_stats})
    dev_free(*b);
  batch_ws_free(ix->bws);
  if (w.host_ctrl) cudaFreeHost(w.host_ctrl);
  for (auto *v : {&ix->prof_pending, &ix->prof_pool, &ix->bprof_pending})
    for (auto &ev : *v)
      for (cudaEvent_t e : ev) cudaEventDestroy(e);
  cudaSetDevice(prev);
  delete ix;
}

static int build_index(const ebr_index_desc *desc, uint32_t faults, ebr_index **out) {
  clear_error();
  if (!desc || !out) {
    set_error("ebr_build_index: null argument");
    return EBR_EINVAL;
  }
  *out = nullptr;
  const uint32_t d = desc->d;
  if (desc->n_ads == 0 || desc->n_keys == 0 || desc->n_keys == 0xFFFFFFFFu ||
      desc->nnz >= (1ULL << 31) || (desc->nnz && (!desc->post_key || !desc->post_ad)) ||
      !desc->emb_f32 || !(d == 4 || d == 8 || d == 16 || d == 32 || d == 64 || d == 128) ||
      (int)desc->emb_dtype < 0 || (int)desc->emb_dtype > 2) {
    set_error("ebr_build_index: invalid description (n_ads=%u n_keys=%u nnz=%llu d=%u dtype=%d)",
              desc->n_ads, desc->n_keys, (unsigned long long)desc->nnz, d,
              (int)desc->emb_dtype);
    return EBR_EINVAL;
  }
  int prev = 0;
  cudaGetDevice(&prev);
  EBR_CUDA_TRY(cudaSetDevice(desc->device));
  cudaStream_t st = (cudaStream_t)desc->stream;
  ebr_index *ix = nullptr;
  int rc = EBR_OK;
  // A build with a forward table that runs out of device memory, there or later, is done
  // again without one: the block-wise scan serves such an index.
  for (bool forward = true;;) {
    ix = new ebr_index();
    ix->device = desc->device;
    ix->n_ads = desc->n_ads;
    ix->n_keys = desc->n_keys;
    ix->d = d;
    ix->dtype = desc->emb_dtype;
    ix->rescore_mult = desc->rescore_mult ? desc->rescore_mult : 4;
    cudaDeviceGetAttribute(&ix->num_sms, cudaDevAttrMultiProcessorCount, desc->device);
    rc = build_impl(desc, ix, faults, &forward, st);
    if (rc == EBR_OK) rc = upload_embeddings(desc, ix, st);
    if (rc == EBR_OK) break;
    const std::string msg = ebr_last_error();
    ebr_index_free(ix);
    set_error("%s", msg.c_str());
    if (rc != EBR_ENOMEM || !forward) {
      cudaSetDevice(prev);
      return rc;
    }
    clear_error();
    forward = false;
  }
  cudaSetDevice(prev);
  *out = ix;
  return EBR_OK;
}

extern "C" int ebr_build_index(const ebr_index_desc *desc, ebr_index **out) {
  return build_index(desc, 0, out);
}

extern "C" int ebr_debug_build_index(const ebr_index_desc *desc, uint32_t faults,
                                     ebr_index **out) {
  return build_index(desc, faults, out);
}

extern "C" int ebr_index_get_info(const ebr_index *ix, ebr_index_info *out) {
  clear_error();
  if (!ix || !out) {
    set_error("ebr_index_get_info: null argument");
    return EBR_EINVAL;
  }
  memset(out, 0, sizeof(*out));
  out->n_ads = ix->n_ads;
  out->n_keys = ix->n_keys;
  out->d = ix->d;
  out->emb_dtype = ix->dtype;
  out->rescore_mult = ix->rescore_mult;
  out->nnz_unique = ix->nnz_unique;
  uint64_t bytes = 0;
  for (int g = 0; g < kGroups; g++) {
    out->n_blocks[g] = ix->n_blocks[g];
    bytes += 4ull * (ix->n_keys + 1) + 4ull * ix->n_blocks[g] + (ix->n_blocks[g] << g);
  }
  out->index_bytes = bytes;
  uint64_t per = ix->dtype == EBR_F32 ? 4 : (ix->dtype == EBR_BF16 ? 2 : 1);
  out->emb_bytes = (uint64_t)ix->n_ads * ix->d * per + (ix->dtype == EBR_FP8E4M3 ? 4ull * ix->n_ads : 0);
  out->build_ms = ix->build_ms;
  out->window_view_ms = ix->wm_build_ms;
  out->window_view_bytes = bytes - 4ull * kGroups * (ix->n_keys + 1) + 4ull * kGroups * (ix->n_win + 1);
  out->n_windows = ix->n_win;
  out->max_keys_per_ad = ix->max_keys_per_ad;
  out->max_window_slots = ix->max_win_slots;
  out->max_window_chunks = ix->max_win_chunks;
  return EBR_OK;
}

extern "C" int ebr_index_export(const ebr_index *ix, uint32_t g, uint32_t *keys, uint32_t *header,
                                uint8_t *values) {
  clear_error();
  if (!ix || g >= (uint32_t)kGroups) {
    set_error("ebr_index_export: bad index or group");
    return EBR_EINVAL;
  }
  int prev = 0;
  cudaGetDevice(&prev);
  EBR_CUDA_TRY(cudaSetDevice(ix->device));
  if (keys) EBR_CUDA_TRY(cudaMemcpy(keys, ix->keys[g], (ix->n_keys + 1ull) * 4, cudaMemcpyDeviceToHost));
  if (header && ix->n_blocks[g])
    EBR_CUDA_TRY(cudaMemcpy(header, ix->header[g], ix->n_blocks[g] * 4, cudaMemcpyDeviceToHost));
  if (values && ix->n_blocks[g])
    EBR_CUDA_TRY(cudaMemcpy(values, ix->values[g], ix->n_blocks[g] << g, cudaMemcpyDeviceToHost));
  cudaSetDevice(prev);
  return EBR_OK;
}

extern "C" int ebr_index_export_emb(const ebr_index *ix, void *codes, float *scale) {
  clear_error();
  if (!ix) {
    set_error("ebr_index_export_emb: null index");
    return EBR_EINVAL;
  }
  int prev = 0;
  cudaGetDevice(&prev);
  EBR_CUDA_TRY(cudaSetDevice(ix->device));
  uint64_t n = (uint64_t)ix->n_ads * ix->d;
  if (codes) {
    if (ix->dtype == EBR_F32)
      EBR_CUDA_TRY(cudaMemcpy(codes, ix->emb_f32.p, n * 4, cudaMemcpyDeviceToHost));
    else
      EBR_CUDA_TRY(cudaMemcpy(codes, ix->emb_q.p, n * (ix->dtype == EBR_BF16 ? 2 : 1),
                              cudaMemcpyDeviceToHost));
  }
  if (scale && ix->dtype == EBR_FP8E4M3)
    EBR_CUDA_TRY(cudaMemcpy(scale, ix->emb_scale.p, ix->n_ads * 4ull, cudaMemcpyDeviceToHost));
  cudaSetDevice(prev);
  return EBR_OK;
}
