// Batched requests: the users x ads inner products on the tensor cores
// (tcgen05.mma fed by tensor TMA, accumulators in TMEM), plus the tensor-map
// plumbing they need.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "ebr_internal.cuh"
#include "ebr_umma.cuh"

namespace ebr {

// --------------------------------------------------------------- tensor maps
static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
static std::mutex g_encode_mu;

static int get_encoder() {
  std::lock_guard<std::mutex> lk(g_encode_mu);
  if (g_encode) return EBR_OK;
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                   cudaEnableDefault, &q);
  if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) {
    set_error("cuTensorMapEncodeTiled unavailable: %s", cudaGetErrorString(e));
    return EBR_ECUDA;
  }
  g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  return EBR_OK;
}

// Row-major [rows][cols] matrix of 2-byte (BF16) or 1-byte (FP8) elements
// viewed as a 2-D tensor, boxes of 128 bytes (or 64, a whole 64-byte row) x
// box_rows rows, swizzled to match (the UMMA K-major layouts).
int make_tmap_2d(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols,
                 uint32_t elt_bytes, uint32_t box_rows) {
  EBR_TRY(get_encoder());
  const uint64_t row_bytes = cols * elt_bytes;
  const uint32_t box_bytes = row_bytes >= 128 ? 128u : 64u;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {row_bytes};
  cuuint32_t box[2] = {box_bytes / elt_bytes, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(map,
                        elt_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8,
                        2, const_cast<void *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE,
                        box_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed (%d) for %llu x %llu, box %u", (int)r,
              (unsigned long long)rows, (unsigned long long)cols, box_rows);
    return EBR_ECUDA;
  }
  return EBR_OK;
}
int make_tmap_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols,
                   uint32_t box_rows) {
  return make_tmap_2d(map, base, rows, cols, 2, box_rows);
}

// ------------------------------------------------------------ GEMM check
// out[i][b] = sum_t A[i][t] * U[b][t] for one 128-row tile per CTA: the
// tensor-core building block of the batched scan, exposed for testing (BF16,
// or FP8 E4M3 codes when F8).
template <bool F8>
__global__ void __launch_bounds__(128) k_gemm_tc(const __grid_constant__ CUtensorMap ma,
                                                 const __grid_constant__ CUtensorMap mu,
                                                 uint32_t n, uint32_t B, uint32_t d,
                                                 float *__restrict__ out,
                                                 uint32_t *__restrict__ flags) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t bar_tma, bar_mma;
  __shared__ uint32_t tmem_base, ok;
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t row_bytes = d * (F8 ? 1u : 2u);
  const uint32_t tr = row_bytes >= 128 ? 128u : 64u;  // bytes per K-tile row
  const uint32_t kb_n = row_bytes / tr, tile_elems = tr / (F8 ? 1u : 2u);
  uint8_t *sa = smem;                          // kb_n x [128 rows x tr]
  uint8_t *su = smem + (size_t)kb_n * 128 * tr;  // kb_n x [B rows x tr]
  const int warp = threadIdx.x >> 5;
  uint32_t ncols = 32;
  while (ncols < B) ncols <<= 1;
  if (warp == 0) {
    tmem_alloc(&tmem_base, ncols);
    tmem_relinquish();
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar_tma, 1);
    mbar_init(&bar_mma, 1);
    fence_mbar_init();
    ok = 1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t row0 = blockIdx.x * 128;
  if (threadIdx.x == 0) {
    mbar_arrive_expect_tx(&bar_tma, kb_n * (128u * tr + B * tr));
    for (uint32_t kb = 0; kb < kb_n; kb++) {
      tma_load_2d(sa + kb * 128u * tr, &ma, (int)(kb * tile_elems), (int)row0, &bar_tma);
      tma_load_2d(su + (size_t)kb * B * tr, &mu, (int)(kb * tile_elems), 0, &bar_tma);
    }
    if (!mbar_wait_bounded(&bar_tma, 0, kWaitTimeoutNs)) {
      ok = 0;
      atomicOr(flags, DEVERR_TIMEOUT);
    } else {
      tc_fence_after();
      const uint32_t idesc = F8 ? idesc_e4m3_f32(128, B) : idesc_bf16_f32(128, B);
      const uint32_t spt = tr / 32;
      for (uint32_t k = 0; k < kb_n * spt; k++) {
        const uint32_t kb = k / spt, kk = k % spt;
        const uint32_t aa = smem_u32(sa + kb * 128u * tr + kk * 32);
        const uint32_t ua = smem_u32(su + (size_t)kb * B * tr + kk * 32);
        const uint64_t ad = tr == 128 ? sdesc_k_sw128(aa) : sdesc_k_sw64(aa);
        const uint64_t bd = tr == 128 ? sdesc_k_sw128(ua) : sdesc_k_sw64(ua);
        if (F8)
          umma_e4m3(tmem_base, ad, bd, idesc, k > 0 ? 1u : 0u);
        else
          umma_bf16(tmem_base, ad, bd, idesc, k > 0 ? 1u : 0u);
      }
      umma_commit(&bar_mma);
      if (!mbar_wait_bounded(&bar_mma, 0, kWaitTimeoutNs)) {
        ok = 0;
        atomicOr(flags, DEVERR_TIMEOUT);
      }
    }
  }
  __syncthreads();
  tc_fence_after();
  if (ok) {
    mbar_try_wait(&bar_mma, 0);
    const uint32_t row = row0 + warp * 32 + (threadIdx.x & 31);
    for (uint32_t c = 0; c < B / 32; c++) {
      uint32_t r[32];
      tmem_ld32(tmem_base + ((uint32_t)(warp * 32) << 16) + c * 32, r);
      tmem_ld_wait();
      if (row < n)
        for (int j = 0; j < 32; j++) out[(uint64_t)row * B + c * 32 + j] = __uint_as_float(r[j]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem_base, ncols);
}

static int debug_gemm(bool f8, const void *A, uint32_t n, const void *U, uint32_t B, uint32_t d,
                      float *out, void *stream) {
  if (!A || !U || !out || n == 0 || (d != 64 && d != 128) || B < 32 || B > 256 || B % 32) {
    set_error("ebr_debug_gemm: need d in {64, 128}, B a multiple of 32 in 32..256");
    return EBR_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const uint32_t eb = f8 ? 1u : 2u;
  CUtensorMap ma, mu;
  EBR_TRY(make_tmap_2d(&ma, A, n, d, eb, 128));
  EBR_TRY(make_tmap_2d(&mu, U, B, d, eb, B));
  uint32_t *flags = nullptr;
  EBR_CUDA_TRY(cudaMallocAsync((void **)&flags, 4, st));
  EBR_CUDA_TRY(cudaMemsetAsync(flags, 0, 4, st));
  const size_t smem = 1024 + (size_t)d * eb * (128 + B);
  auto kern = f8 ? k_gemm_tc<true> : k_gemm_tc<false>;
  EBR_CUDA_TRY(allow_smem(kern, 1024 + 128 * 2 * (128 + 256)));  // (d = 128, B = 256)
  kern<<<(n + 127) / 128, 128, smem, st>>>(ma, mu, n, B, d, out, flags);
  EBR_CUDA_TRY(cudaGetLastError());
  uint32_t hf = 0;
  EBR_CUDA_TRY(cudaMemcpyAsync(&hf, flags, 4, cudaMemcpyDeviceToHost, st));
  EBR_CUDA_TRY(cudaStreamSynchronize(st));
  cudaFreeAsync(flags, st);
  return check_device_flags(hf, f8 ? "ebr_debug_gemm_e4m3" : "ebr_debug_gemm_bf16");
}

}  // namespace ebr

using namespace ebr;

extern "C" int ebr_debug_gemm_bf16(const uint16_t *A, uint32_t n, const uint16_t *U, uint32_t B,
                                   uint32_t d, float *out, void *stream) {
  clear_error();
  return debug_gemm(false, A, n, U, B, d, out, stream);
}

extern "C" int ebr_debug_gemm_e4m3(const uint8_t *A, uint32_t n, const uint8_t *U, uint32_t B,
                                   uint32_t d, float *out, void *stream) {
  clear_error();
  return debug_gemm(true, A, n, U, B, d, out, stream);
}

namespace ebr {

// A wait nobody ends: the bounded-wait path must give up and flag it.
__global__ void k_wait_timeout(uint64_t timeout_ns, uint32_t *flags) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, 0, timeout_ns))
    atomicOr(flags, DEVERR_TIMEOUT);
  __syncthreads();
}

}  // namespace ebr

extern "C" int ebr_debug_wait_timeout(uint32_t timeout_us, void *stream) {
  using namespace ebr;
  clear_error();
  if (timeout_us == 0 || timeout_us > 1000000u) {
    set_error("ebr_debug_wait_timeout: timeout_us must be 1 .. 10^6");
    return EBR_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  uint32_t *flags = nullptr;
  EBR_CUDA_TRY(cudaMallocAsync((void **)&flags, 4, st));
  EBR_CUDA_TRY(cudaMemsetAsync(flags, 0, 4, st));
  k_wait_timeout<<<1, 32, 0, st>>>((uint64_t)timeout_us * 1000ull, flags);
  EBR_CUDA_TRY(cudaGetLastError());
  uint32_t hf = 0;
  EBR_CUDA_TRY(cudaMemcpyAsync(&hf, flags, 4, cudaMemcpyDeviceToHost, st));
  EBR_CUDA_TRY(cudaStreamSynchronize(st));
  cudaFreeAsync(flags, st);
  return check_device_flags(hf, "ebr_debug_wait_timeout");
}

// =====================================================================
// Batched scan: B users against every ad, one pass over the inventory
// =====================================================================
// The users are scored in groups of 64 (blockIdx.y), each a pass of its own
// over the inventory: 64 users' expanded weights of one key are 256 bytes, so
// all of a group's warps share the lines they gather, and a group's slice of
// w^T stays in L2 (5M ads with 257 k keys: 66 MB per group, 263 MB for 256
// users, which does not).  The ad rows and the keys are read once per group;
// that is a small part of the traffic.
// Per window of 128 ads (256 without a forward table; one persistent CTA per SM,
// contiguous windows):
//   producer warp   -- tensor TMA of the window's BF16/FP8 ad rows into a
//                      stage ring; the users' vectors (and, kForwardSw, the
//                      group's slice of w^T) are loaded once;
//   MMA warp        -- tcgen05.mma with the users as the M side and the
//                      window's ads as N, in two M-tiles: the even
//                      users and the odd users (the user table is stored in
//                      that pair order), each replicated four times down the
//                      128 TMEM lanes; deep[user][ad] (Eq. 1) lands in TMEM;
//   list warps (4; 2) -- (kWalk, indexes without a forward table) lay out, per
//                      run of 32 ads, a key table T[r][i] = r-th key of ad i
//                      (the window's slice of L, transposed; short ads padded
//                      with a zero row of w^T) by a walk over the window's
//                      blocks in the window-major view of the compressed list;
//                      between windows they raise the users' running
//                      thresholds from the histograms all CTAs share (one of
//                      them does only that when there is a forward table);
//   epilogue (16)   -- thread = user pair (2u, 2u + 1) at TMEM lane u mod 32,
//                      four ads per warp at a time; a warp copies its
//                      ads' part of the forward table in by itself
//                      (cp.async, a window ahead) and turns it into T:
//                      wide[i] += w^T[T[r][i]][2u .. 2u + 1] for every row r
//                      (coalesced 8-byte loads, three or four rows in flight, paired
//                      FP32 adds, accumulators in registers), added
//                      to both users' deep scores (TMEM columns c and
//                      window + c), filtered, and each user's candidates above
//                      its running threshold go to this CTA's per-user buffer
//                      (top-m kept exactly).
// kForwardSw: a key space whose slice of w^T fits shared memory beside the rest (up to
// about 500 keys) is gathered from there.
// What bounds it: the latency of the gathers and, between them, of each
// window's chain of list, accumulators and candidates (without the gathers
// 256 users x 5M ads take 4.5 ms); the L1 pipe alone would take 3.1 ms.  The
// forward table lists an ad's keys in the order of the window-major view (rare
// keys first), so the FP32 sums are the same as the walk's; rows of four ads are
// refilled one by one to keep loads in flight within 96 registers (a spill here doubles the
// time).  Measured scans, before and after: 256 users x 5M BF16 ads (24 keys)
// 13.6 -> 8.3 ms, 128 users x 5M BF16 ads (32 keys, bitmaps) 10.6 -> 5.1 ms, 64
// users x 10M FP8 ads (32 keys of 480) 9.0 -> 4.3 ms.
namespace ebr {

constexpr int kBWin = 256;
// MODE: where an ad's keys come from (see above).
enum { kWalk = 0, kForward = 1, kForwardSw = 2 };
constexpr int kEpiWarps = 16, kEpiThreads = kEpiWarps * 32;
// kWalk: a group's lists are built anew for every group of users, which two warps
// could not do in the time of an epilogue (256 users x 5M BF16 ads of 24 keys
// 16.8 ms with two, 11.9 with four, 15.4 with one pass of two warps for all users and
// no groups).  With a forward table one of two warps raises thresholds.
constexpr int list_warps(int mode) { return mode == kWalk ? 4 : 2; }
constexpr int batch_threads(int mode) { return (kEpiWarps + list_warps(mode) + 2) * 32; }
constexpr int kMaxUsers = 256;
static_assert(kBWin % (list_warps(kWalk) * 32) == 0, "list threads split the window's ads evenly");
// List buffer: run_off[8], run_rows[8], fill[256], then the run tables.
constexpr uint32_t kListHdr = 8 + 8 + kBWin;
constexpr uint32_t kMaxBatchKeysPerAd = 64;  // longest key list the batched tables hold
// Bins of a user's score histogram: sign, 8 exponent bits and 4 of the
// mantissa (6 % wide; the bound is that much lower than the true score).
constexpr uint32_t kUserBins = 8192;
constexpr int kMapWords = kUserBins / 16 / 32;
constexpr int kUserBinShift = 51;

constexpr uint32_t kGroup = 64;   // users of one pass
constexpr int kTrimWarps = 8;     // epilogue warps that trim buffers (each needs a histogram)
// Row of user b in the batch's user table: per group of 64 the even users
// first, then the odd ones (the two M-tiles of the batched scan).
__host__ __device__ __forceinline__ uint32_t user_row(uint32_t b) {
  return (b & ~(kGroup - 1u)) + (b & 1u) * (kGroup / 2) + ((b & (kGroup - 1u)) >> 1);
}

struct CandEntry {
  unsigned long long key;  // approximate score | id
  float wide;              // the ad's wide term for this user (FP32 sum)
  uint32_t pad;
};

struct BatchArgs {
  CUtensorMap ta;  // ad rows, BF16 or FP8 [N][d], box {tile row, 128}
  CUtensorMap tu;  // users, same type [Bq][d] in pair order, box {tile row, 32}
  const uint32_t *wkey[kGroups];
  const uint8_t *wvals[kGroups];
  const uint32_t *win_ptr[kGroups];
  const uint16_t *ad_nkeys;    // [N] distinct keys of each ad
  const uint8_t *fwd;          // forward table (then w^T's rows go by its key ids), or null
  const uint32_t *fwd_off;
  uint32_t quad_bytes, max_quads;  // max_quads: of one run
  const float *wT;             // [groups][n_keys + 1][64] expanded weights, user-minor; last row 0
  uint32_t wt_rows;            // n_keys + 1
  const uint64_t *filters;     // [B][words] (rows of users without a filter are unused)
  const uint32_t *has_filter;  // [B]
  uint32_t n_ads, n_win, B, d, m, cap_u, list_cap, words;  // B: users (buffer stride)
  const uint32_t *B_dev;       // non-null: the active users (<= B) are read here at launch
  uint32_t zero_row;           // n_keys * 32: the zero row of wT, in user-pair units
  uint32_t sa, lb, tb;         // A stages, list buffers, TMEM buffers
  uint32_t tile_row, kb_n;     // bytes per K-tile row (128 or 64), K-tiles per row
  const float *ad_scale;       // FP8: [N] row scales of the ad table
  const float *user_scale;     // FP8: [Bq] row scales of the quantised users (pair order)
  // Scores counted per user over all CTAs (bins: the top bits of the ranking
  // key), for a bound on each user's kscan-th best.
  uint32_t *uhist;             // [B][kUserBins], zeroed per call
  uint32_t *umap;              // [B][kMapWords] a bit per 16 bins: counted in; zeroed per call
  const uint32_t *kscan;       // [B] candidates each user needs
  CandEntry *cand;             // [grid][B][cap_u]
  uint32_t *cand_n;            // [grid][B]
  unsigned long long *cand_thr;  // [grid][B] cut of the CTA's own trims
  Ctrl *ctrl;
};

__device__ __forceinline__ uint4 lds_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}

struct BatchSmem {
  uint64_t a_full[2], a_empty[2], t_full[2], t_empty[2], l_full[2], l_empty[2], u_full;
  uint32_t tmem_base;
  uint32_t cnt_u[kGroup], trim_u[kGroup];
  uint32_t map_u[kGroup][kMapWords];  // this CTA's part of umap
  unsigned long long thr_u[kGroup];  // running threshold: the larger of the two bounds below
  unsigned long long cut_u[kGroup];  // cut of this CTA's own trims (0: nothing was trimmed)
  uint32_t abort, stop_epi, stop_list, n_issued, n_mma;
  uint32_t finished;    // the epilogue warps are done
  uint32_t trim, meet;  // a buffer is nearly full; what a meeting of the epilogue warps is for
};

// Raises the running threshold of user g0 + b to the largest bin edge with at least
// kscan[b] counted scores at or above it (every one a distinct ad): the user's
// kscan-th best over the whole inventory is no lower, so what lies below the
// edge cannot be selected, and the proof that the merge makes is not touched.
// Counts only grow, so a snapshot gives a lower, still valid, bound.
// Only bins that umap says are in use are read: the 8192 bins are spaced by
// exponent, and where fewer ads than kscan pass a bitmap, the walk from the top
// through the empty ones around zero took 300 us at the end of every CTA
// (195 users x 85k BF16 ads, 64 of them with bitmaps: scan 1307 us; 290 with this
// and the grid of batch_grid).
__device__ __forceinline__ void raise_threshold(const BatchArgs &a, BatchSmem &sm, uint32_t g0,
                                                uint32_t b) {
  const uint32_t need = __ldg(a.kscan + g0 + b);
  const uint32_t lo = (uint32_t)(*((volatile unsigned long long *)&sm.thr_u[b]) >> kUserBinShift) >> 4;
  const uint4 *map = reinterpret_cast<const uint4 *>(a.umap + (size_t)(g0 + b) * kMapWords);
  const uint32_t *hist = a.uhist + (size_t)(g0 + b) * kUserBins;
  uint32_t cum = 0;
  for (int q = kMapWords / 4 - 1; q >= (int)(lo >> 7); q--) {
    const uint4 v = __ldcg(map + q);
#pragma unroll 1
    for (int half = 1; half >= 0; half--) {
      unsigned long long bits = half ? (unsigned long long)v.w << 32 | v.z
                                     : (unsigned long long)v.y << 32 | v.x;
      while (bits) {
        const int top = 63 - __clzll(bits);
        bits &= ~(1ull << top);
        const uint32_t g = 128u * q + 64u * half + top;
        if (g < lo) return;
        const uint4 *h = reinterpret_cast<const uint4 *>(hist) + 4 * g;
        uint32_t c[16];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const uint4 x = __ldcg(h + i);
          c[4 * i] = x.x;
          c[4 * i + 1] = x.y;
          c[4 * i + 2] = x.z;
          c[4 * i + 3] = x.w;
        }
        int bin = -1;
#pragma unroll
        for (int i = 15; i >= 0; i--) {
          cum += c[i];
          if (bin < 0 && cum >= need) bin = 16 * (int)g + i;
        }
        if (bin >= 0) {
          atomicMax(&sm.thr_u[b], (unsigned long long)bin << kUserBinShift);
          return;
        }
      }
    }
  }
}

__device__ __forceinline__ uint32_t ushift(uint32_t g) { return g >= 2 ? g - 2 : 0; }

// Walk the real slots of window w: f(ad_in_window, key).  `t`/`nt`: this
// thread's index in the walking group (whole warps).  The window's block
// range in each of the nine groups is read once (one lane per group) and the
// groups' work units are walked as one sequence, eight units per thread
// loaded before any is used, so loads stay in flight across group borders.
template <typename F>
__device__ __forceinline__ void walk_window(const BatchArgs &a, uint32_t w, int t, int nt, F f) {
  constexpr int kU = 8;
  const int lane = threadIdx.x & 31;
  uint32_t lo_l = 0, n_l = 0;
  if (lane < kGroups) {
    const uint32_t lo = __ldg(a.win_ptr[lane] + w), hi = __ldg(a.win_ptr[lane] + w + 1);
    lo_l = lo;
    n_l = (hi - lo) << ushift(lane);
  }
  uint32_t lo_g[kGroups], end_g[kGroups];  // first block, end of the group's units
  uint32_t total = 0;
#pragma unroll
  for (int g = 0; g < kGroups; g++) {
    lo_g[g] = __shfl_sync(0xffffffffu, lo_l, g);
    total += __shfl_sync(0xffffffffu, n_l, g);
    end_g[g] = total;
  }
#pragma unroll 1
  for (uint32_t u0 = t; u0 < total; u0 += kU * nt) {
    uint32_t key[kU], word[kU], gg[kU], first[kU];
#pragma unroll
    for (int e = 0; e < kU; e++) {
      const uint32_t U = u0 + e * nt;
      const bool v = U < total;
      uint32_t g = 0;
#pragma unroll
      for (int i = 0; i < kGroups - 1; i++) g += U >= end_g[i] ? 1u : 0u;
      uint32_t lo = lo_g[0], beg = 0;
#pragma unroll
      for (int i = 1; i < kGroups; i++)
        if (g == (uint32_t)i) {
          lo = lo_g[i];
          beg = end_g[i - 1];
        }
      const uint32_t us = ushift(g), u = U - beg;
      const uint32_t bk = lo + (v ? (u >> us) : 0u), wi = u & ((1u << us) - 1u);
      key[e] = v ? __ldg(a.wkey[g] + bk) : 0u;
      if (!v)
        word[e] = 0u;
      else if (g >= 2)
        word[e] = __ldg(reinterpret_cast<const uint32_t *>(a.wvals[g]) + (((uint64_t)bk << us) + wi));
      else if (g == 1)
        word[e] = __ldg(reinterpret_cast<const unsigned short *>(a.wvals[1]) + bk);
      else
        word[e] = __ldg(a.wvals[0] + bk);
      gg[e] = g;
      first[e] = (v && wi == 0) ? 1u : 0u;
    }
#pragma unroll
    for (int e = 0; e < kU; e++) {
      if (u0 + e * nt >= total) break;
      const uint32_t ns = gg[e] >= 2 ? 4u : (gg[e] == 1 ? 2u : 1u);
      for (uint32_t s = 0; s < ns; s++) {
        const uint32_t l = (word[e] >> (8 * s)) & 255u;
        if ((s == 0 && first[e]) || l != 0) f(l, key[e]);
      }
    }
  }
}

// Warp-level radix select: T with exactly `need` keys >= T among n (global).
__device__ uint64_t warp_radix_select(const CandEntry *buf, uint32_t n, uint32_t need,
                                      uint32_t *hist /* 256 words, this warp's */) {
  const int lane = threadIdx.x & 31;
  uint64_t prefix = 0;
  for (int shift = 56; shift >= 0; shift -= 8) {
    for (int i = lane; i < 256; i += 32) hist[i] = 0;
    __syncwarp();
    const uint64_t hi_mask = (shift == 56) ? 0ull : (~0ull << (shift + 8));
    for (uint32_t i = lane; i < n; i += 32) {
      const uint64_t x = buf[i].key;
      if ((x & hi_mask) == prefix) atomicAdd(&hist[(x >> shift) & 255u], 1u);
    }
    __syncwarp();
    uint32_t c[8], tot = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) {
      c[e] = hist[255 - 8 * lane - e];
      tot += c[e];
    }
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    uint32_t acc = incl - tot, dg = 0, nn = 0, whole = 0;
    bool found = false;
#pragma unroll
    for (int e = 0; e < 8; e++) {
      if (!found && acc < need && need <= acc + c[e]) {
        found = true;
        dg = 255 - 8 * lane - e;
        nn = need - acc;
        whole = (need - acc == c[e]) ? 1u : 0u;
      }
      acc += c[e];
    }
    const uint32_t bal = __ballot_sync(0xffffffffu, found);
    const int src = __ffs(bal) - 1;
    dg = __shfl_sync(0xffffffffu, dg, src);
    need = __shfl_sync(0xffffffffu, nn, src);
    whole = __shfl_sync(0xffffffffu, whole, src);
    prefix |= (uint64_t)dg << shift;
    __syncwarp();
    if (whole) break;
  }
  return prefix;
}

// Stable in-place compaction of buf[0..n) to the entries with key >= T;
// returns how many were kept.  Four entries a lane are in flight: the chain of
// reads is what it costs (with one, the end of a CTA whose 61 users had 300
// entries each took 85 us).
__device__ __noinline__ uint32_t warp_compact(CandEntry *buf, uint32_t n, uint64_t T) {
  constexpr int kU = 4;
  const int lane = threadIdx.x & 31;
  uint32_t kept = 0;
  for (uint32_t b0 = 0; b0 < n; b0 += 32 * kU) {
    CandEntry e[kU];
    uint32_t bal[kU];
#pragma unroll
    for (int u = 0; u < kU; u++) {
      const uint32_t i = b0 + 32 * u + lane;
      e[u].key = 0;
      if (i < n) e[u] = buf[i];
    }
#pragma unroll
    for (int u = 0; u < kU; u++)
      bal[u] = __ballot_sync(0xffffffffu, b0 + 32 * u + lane < n && e[u].key >= T);
    __syncwarp();  // every entry of the round is read before any is written
#pragma unroll
    for (int u = 0; u < kU; u++) {
      if ((bal[u] >> lane) & 1u) buf[kept + __popc(bal[u] & ((1u << lane) - 1u))] = e[u];
      kept += __popc(bal[u]);
    }
    __syncwarp();
  }
  return kept;
}

// Exact top-`need` of a per-user buffer, in place; returns how many were kept.
// (Trims are rare, so the keys are read again for every digit: a form that held
// them in registers made the hot loop spill.)
__device__ __forceinline__ uint32_t warp_trim(CandEntry *buf, uint32_t n, uint32_t need,
                                              uint32_t *hist, uint64_t *T_out) {
  const uint64_t T = warp_radix_select(buf, n, need, hist);
  *T_out = T;
  return warp_compact(buf, n, T);
}

struct Row4 {
  float2 x[4];
};

// Ads of a window: the block-wise lists are per 256 ads; with the forward table
// 128, so that two windows' accumulators (2 x 128 columns each) fit TMEM and
// the MMAs of one run while the other's are read.
constexpr uint32_t kFwdWin = 128;
constexpr uint32_t accum_bufs(bool fwd) { return fwd ? 2 : 1; }

// cp.async: 16 bytes global -> shared, asynchronously, and the wait for all of
// the calling thread's.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

template <bool F8, int MODE>
__global__ void __launch_bounds__(batch_threads(MODE), 1) k_batch_window(const __grid_constant__ BatchArgs a) {
  constexpr bool FWD = MODE != kWalk, SW = MODE == kForwardSw;
  constexpr int kListThreads = list_warps(MODE) * 32, kBatchThreads = batch_threads(MODE);
  constexpr int kMmaWarp = kEpiWarps + list_warps(MODE), kProdWarpB = kMmaWarp + 1;
  constexpr uint32_t kWin = FWD ? kFwdWin : kBWin;      // ads of a window
  constexpr uint32_t kWarpAds = kWin / kEpiWarps;       // of them per epilogue warp
  constexpr uint32_t kTb = accum_bufs(FWD);             // accumulator buffers
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ BatchSmem sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t kb_n = a.kb_n, tr = a.tile_row;  // K-tiles per row, bytes per tile row
  const uint32_t tile_elems = tr / (F8 ? 1u : 2u);
  const uint32_t n_mt = 2;                        // M-tiles: even users, odd users
  const uint32_t u_tile = kb_n * 128u * tr;        // one M-tile: kb_n x [128 rows x tr]
  const uint32_t a_stage = kb_n * kWin * tr;       // kb_n x [window's ad rows x tr]
  uint8_t *su = smem;                              // n_mt user tiles
  uint8_t *sa = su + (size_t)n_mt * u_tile;        // sa ad stages
  uint32_t *lists = reinterpret_cast<uint32_t *>(sa + (size_t)a.sa * a_stage);
  // key lists: kWalk a ring of window lists (32-bit row offsets in user
  // pairs), else per epilogue warp the raw quads of its ads' next window and
  // the list of its current one (row offsets, or, SW, 16-bit key ids)
  const uint32_t list_words = FWD ? 0u : kListHdr + a.list_cap;
  const uint32_t wlist_bytes = FWD ? a.max_quads * 4u * kWarpAds * (SW ? 2u : 4u) : 0u;
  const uint32_t wraw_bytes = FWD ? a.max_quads * kWarpAds * (a.quad_bytes > 256u ? 12u : 8u) : 0u;
  uint32_t *whist = lists + (FWD ? (size_t)kEpiWarps * (wlist_bytes + wraw_bytes) / 4
                                 : (size_t)a.lb * list_words);  // [kTrimWarps][256]
  float *s_wT = reinterpret_cast<float *>(whist + kTrimWarps * 256);  // SW: the slice of wT
  const float *wT = a.wT + (size_t)blockIdx.y * a.wt_rows * kGroup;

  const uint32_t w_begin = (uint32_t)(((uint64_t)a.n_win * blockIdx.x) / gridDim.x);
  const uint32_t w_end = (uint32_t)(((uint64_t)a.n_win * (blockIdx.x + 1)) / gridDim.x);
  const uint32_t my_wins = w_end - w_begin;
  const uint32_t tcols = kWin * n_mt;  // TMEM columns per window
  const uint32_t ncols = 512;
  // active users: all B, or the count a device-side loop wrote for this wave
  // (the same for every thread; none: nothing to do, nothing allocated)
  const uint32_t nB = a.B_dev ? min(*a.B_dev, a.B) : a.B;
  const uint32_t g0 = blockIdx.y * kGroup;  // the group's first user
  if (nB <= g0) return;
  const uint32_t nG = min(nB - g0, kGroup);

  for (uint32_t b = tid; b < kGroup; b += kBatchThreads) {
    sm.cnt_u[b] = 0;
    sm.trim_u[b] = 0;
    for (int i = 0; i < kMapWords; i++) sm.map_u[b][i] = 0;
    sm.thr_u[b] = 0ull;
    sm.cut_u[b] = 0ull;
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&sm.tmem_base, ncols);
    tmem_relinquish();
  }
  if (tid == 0) {
    sm.abort = 0;
    sm.stop_epi = 0;
    sm.trim = 0;
    sm.finished = 0;
    sm.n_issued = 0;
    sm.n_mma = 0;
    for (int q = 0; q < 2; q++) {
      mbar_init(&sm.a_full[q], 1);
      mbar_init(&sm.a_empty[q], 1);
      mbar_init(&sm.t_full[q], 1);
      mbar_init(&sm.t_empty[q], kEpiWarps);
      mbar_init(&sm.l_full[q], kListThreads);
      mbar_init(&sm.l_empty[q], kEpiWarps);
    }
    mbar_init(&sm.u_full, 1);
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  if (warp == kProdWarpB) {
    // ---------------------------------------------------------- producer
    if (lane == 0) {
      const uint64_t pol = l2_evict_first_policy();
      // users (per group: even users, then odd users): row r of M-tile mt
      // holds the group's user 2 (r mod 32) + mt
      constexpr uint32_t box_u = kGroup / 2;
      const uint32_t wt_bytes = SW ? a.wt_rows * kGroup * 4u : 0u;
      mbar_arrive_expect_tx(&sm.u_full, n_mt * u_tile + wt_bytes);
      if (SW) bulk_g2s(s_wT, wT, wt_bytes, &sm.u_full);
      for (uint32_t mt = 0; mt < n_mt; mt++)
        for (uint32_t r0 = 0; r0 < 128; r0 += box_u)
          for (uint32_t kb = 0; kb < kb_n; kb++)
            tma_load_2d(su + mt * u_tile + kb * 128u * tr + r0 * tr, &a.tu,
                        (int)(kb * tile_elems), (int)(g0 + mt * box_u), &sm.u_full);
      for (uint32_t j = 0; j < my_wins; j++) {
        const uint32_t s = j % a.sa;
        if (j >= a.sa && !mbar_wait_bounded(&sm.a_empty[s], ((j / a.sa) - 1) & 1u, kWaitTimeoutNs)) {
          atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
          sm.abort = 1;
          break;
        }
        if (*((volatile uint32_t *)&sm.abort)) break;
        const int row0 = (int)((w_begin + j) * kWin);
        uint8_t *dst = sa + (size_t)s * a_stage;
        mbar_arrive_expect_tx(&sm.a_full[s], a_stage);
        for (uint32_t kb = 0; kb < kb_n; kb++)
          for (uint32_t h = 0; h < kWin / 128; h++)
            tma_load_2d_hint(dst + kb * kWin * tr + h * 128u * tr, &a.ta, (int)(kb * tile_elems),
                             row0 + (int)h * 128, &sm.a_full[s], pol);
        sm.n_issued = j + 1;
      }
    }
  } else if (warp == kMmaWarp) {
    // ---------------------------------------------------------- MMA issuer
    if (lane == 0) {
      bool ok = mbar_wait_bounded(&sm.u_full, 0, kWaitTimeoutNs);
      const uint32_t idesc = F8 ? idesc_e4m3_f32(128, kWin) : idesc_bf16_f32(128, kWin);
      const uint32_t spt = tr / 32;  // 32-byte K-steps per tile row
      for (uint32_t j = 0; ok && j < my_wins; j++) {
        const uint32_t s = j % a.sa, tb = j % a.tb;
        ok = mbar_wait_bounded(&sm.a_full[s], (j / a.sa) & 1u, kWaitTimeoutNs);
        if (ok && j >= a.tb) ok = mbar_wait_bounded(&sm.t_empty[tb], ((j / a.tb) - 1) & 1u, kWaitTimeoutNs);
        if (!ok || *((volatile uint32_t *)&sm.abort)) break;
        tc_fence_after();
        const uint8_t *as = sa + (size_t)s * a_stage;
        for (uint32_t mt = 0; mt < n_mt; mt++) {
          const uint32_t dcol = tmem + tb * tcols + mt * kWin;
          for (uint32_t k = 0; k < kb_n * spt; k++) {
            const uint32_t kb = k / spt, kk = k % spt;
            const uint32_t ua = smem_u32(su + mt * u_tile + kb * 128u * tr + kk * 32);
            const uint32_t aa = smem_u32(as + kb * kWin * tr + kk * 32);
            const uint64_t ud = tr == 128 ? sdesc_k_sw128(ua) : sdesc_k_sw64(ua);
            const uint64_t ad = tr == 128 ? sdesc_k_sw128(aa) : sdesc_k_sw64(aa);
            if (F8)
              umma_e4m3(dcol, ud, ad, idesc, k > 0 ? 1u : 0u);
            else
              umma_bf16(dcol, ud, ad, idesc, k > 0 ? 1u : 0u);
          }
        }
        umma_commit(&sm.a_empty[s]);
        umma_commit(&sm.t_full[tb]);
        sm.n_mma = j + 1;
      }
      if (!ok) {
        atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
        sm.abort = 1;
      }
    }
  } else if (FWD && warp >= kEpiWarps) {
    // ---------------------------------------------------------- thresholds
    // One warp, a lane per user, as long as the epilogue runs.
    if (warp == kEpiWarps)
      while (!*((volatile uint32_t *)&sm.finished) && !*((volatile uint32_t *)&sm.abort)) {
        for (uint32_t b = lane; b < nG; b += 32) raise_threshold(a, sm, g0, b);
        __nanosleep(2000);
      }
  } else if (warp >= kEpiWarps) {
    // ---------------------------------------------------------- list builders
    // Per window: off[l] = first slot of ad l (exclusive scan of the ads' key
    // counts), then one walk of the window's blocks drops each key into its
    // ad's slot range.
    const int lt = tid - kEpiThreads;
    for (uint32_t j = 0; j < my_wins; j++) {
      const uint32_t lbuf = j % a.lb;
      if (lt == 0) {
        uint32_t stop = *((volatile uint32_t *)&sm.abort);
        if (!stop && j >= a.lb &&
            !mbar_wait_bounded(&sm.l_empty[lbuf], ((j / a.lb) - 1) & 1u, kWaitTimeoutNs)) {
          atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
          sm.abort = 1;
          stop = 1;
        }
        sm.stop_list = stop;
      }
      named_sync(2, kListThreads);
      if (sm.stop_list) break;
      if (j >= a.lb) mbar_try_wait(&sm.l_empty[lbuf], ((j / a.lb) - 1) & 1u);
      // a window has been scored since the last turn: a lane per user raises the thresholds
      if (j >= a.lb)
        for (uint32_t b = lt; b < nG; b += kListThreads) raise_threshold(a, sm, g0, b);
      uint32_t *run_off = lists + (size_t)lbuf * list_words;
      uint32_t *run_rows = run_off + 8;
      uint32_t *fill = run_off + 16;
      uint32_t *tab = run_off + kListHdr;
      const uint32_t w = w_begin + j;
      // rows of each run = most keys of its 32 ads; thread lt owns ads
      // lt, lt + kListThreads, ... (whole warps per run of 32 ads)
      constexpr int kPer = kBWin / kListThreads;
      uint32_t nk[kPer];
#pragma unroll
      for (int h = 0; h < kPer; h++) {
        const uint32_t al = lt + kListThreads * h;
        const uint32_t ad = w * kBWin + al;
        nk[h] = ad < a.n_ads ? (uint32_t)__ldg(a.ad_nkeys + ad) : 0u;
        fill[al] = 0;
        uint32_t mx = nk[h];
#pragma unroll
        for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) run_rows[al >> 5] = mx;
      }
      named_sync(2, kListThreads);
      uint32_t ro[kPer], rr[kPer];
      {
        uint32_t acc = 0;
        for (uint32_t r = 0; r < 8; r++) {
          const uint32_t rows = run_rows[r];
#pragma unroll
          for (int h = 0; h < kPer; h++)
            if (r == ((lt + kListThreads * h) >> 5)) {
              ro[h] = acc;
              rr[h] = rows;
            }
          if (lt == 0) run_off[r] = acc;
          acc += rows * 32u;
        }
      }
      // padding entries (rows nk .. rows-1) point at the zero row
#pragma unroll
      for (int h = 0; h < kPer; h++)
        for (uint32_t r = nk[h]; r < rr[h]; r++) {
          const uint32_t pos = ro[h] + r * 32u + (uint32_t)lane;
          if (pos < a.list_cap) tab[pos] = a.zero_row;
        }
      named_sync(2, kListThreads);
      walk_window(a, w, lt, kListThreads, [&](uint32_t l, uint32_t key) {
        const uint32_t rank = atomicAdd(&fill[l], 1u);
        const uint32_t pos = run_off[l >> 5] + rank * 32u + (l & 31u);
        if (rank < run_rows[l >> 5] && pos < a.list_cap) tab[pos] = key * (kGroup / 2);
      });
      mbar_arrive(&sm.l_full[lbuf]);  // release: this thread's list writes
    }
  } else {
    // ---------------------------------------------------------- epilogue
    // Thread = user pair (2u, 2u + 1): M-tile 0 holds the even users and
    // M-tile 1 the odd ones, each replicated down the 128 lanes, so lane L
    // reads both users' deep scores (columns c and 256 + c) and gathers
    // both users' weights with one 8-byte load of the user-minor w^T.
    const GroupSync gsync{1, kEpiThreads};
    const uint32_t ad_lo = warp * kWarpAds;       // this warp's ads in the window
    const uint32_t tl = tmem + ((32u * (warp % 4)) << 16);  // its TMEM lane quadrant
    const uint32_t user0 = 2 * lane, user1 = 2 * lane + 1;  // within the group
    const bool ok0 = user0 < nG, ok1 = user1 < nG;
    // FP8: deep = TMEM x (user scale) x (the ad row's scale); user rows in pair order
    const float usc0 = F8 && ok0 ? a.user_scale[g0 + lane] : 1.f;
    const float usc1 = F8 && ok1 ? a.user_scale[g0 + kGroup / 2 + lane] : 1.f;
    // which of this thread's users have a bitmap (else every ad passes)
    const bool filt0 = ok0 && a.has_filter[g0 + user0], filt1 = ok1 && a.has_filter[g0 + user1];
    const float2 *wcol = reinterpret_cast<const float2 *>(wT) + lane;
    const uint32_t s_wcol = smem_u32(s_wT) + 8u * lane;
    auto user_buf = [&](uint32_t b) {
      return a.cand + ((uint64_t)blockIdx.x * a.B + g0 + b) * a.cap_u;
    };
    // one (user, ad) score that passed the bitmap and the float test:
    // thresholded exactly, appended to the user's buffer and counted
    auto offer = [&](uint32_t user, unsigned long long thr, float score, float wide,
                     uint32_t ad) {
      const unsigned long long key = make_key(score, ad);
      if (key < thr) return;
      const uint32_t pos = atomicAdd(&sm.cnt_u[user], 1u);
      if (pos < a.cap_u) {
        CandEntry ce;
        ce.key = key;
        ce.wide = wide;
        ce.pad = 0;
        user_buf(user)[pos] = ce;
        const uint32_t bin = (uint32_t)(key >> kUserBinShift);
        atomicAdd(a.uhist + (size_t)(g0 + user) * kUserBins + bin, 1u);
        const uint32_t bit = 1u << ((bin >> 4) & 31u);
        uint32_t *word = &sm.map_u[user][bin >> 9];
        if (!(*((volatile uint32_t *)word) & bit)) {
          atomicOr(word, bit);
          atomicOr(a.umap + (g0 + user) * kMapWords + (bin >> 9), bit);
        }
      } else {
        atomicOr(&a.ctrl->flags, DEVERR_OVERFLOW);
      }
    };
    // the users marked keep the exact best m (the warps with a histogram)
    auto trim_users = [&]() {
      for (uint32_t b = warp; b < nG && warp < kTrimWarps; b += kTrimWarps) {
        if (!sm.trim_u[b]) continue;
        uint64_t T;
        const uint32_t kept = warp_trim(user_buf(b), sm.cnt_u[b], a.m, whist + warp * 256, &T);
        __syncwarp();
        if (lane == 0) {
          sm.cut_u[b] = max(sm.cut_u[b], (unsigned long long)T);
          atomicMax(&sm.thr_u[b], (unsigned long long)T);
          sm.cnt_u[b] = kept;
          sm.trim_u[b] = 0;
        }
        __syncwarp();
      }
    };
    // The warps run free of each other (each hands the list and the
    // accumulators back by itself) and meet only when a buffer is nearly full,
    // and at the end: a check asks for 512 free places, because all warps
    // together may add a window's 256 entries to a user before the next check
    // and 256 more before every warp has seen the flag.
    uint32_t j = 0;
    // FWD: this warp's ads' quads of a window, 16 bytes at a time into raw_a
    // (per quad the ads' low halves, then their high bytes); o0/o1: the run's
    // first quad and its end, read a window ahead
    const uint32_t list_a = smem_u32(lists) + warp * (wlist_bytes + wraw_bytes);
    const uint32_t raw_a = list_a + wlist_bytes;
    const uint32_t raw_q = kWarpAds * (a.quad_bytes > 256u ? 12u : 8u);
    uint32_t nq = 0, o0 = 0, o1 = 0;
    auto read_offsets = [&](uint32_t jj) {
      if (FWD && jj < my_wins) {
        const uint32_t r = (kWin / 32) * (w_begin + jj) + (ad_lo >> 5);
        o0 = __ldg(a.fwd_off + r);
        o1 = __ldg(a.fwd_off + r + 1);
      }
    };
    auto fetch_quads = [&](uint32_t jj) {  // of window jj, whose offsets are in o0, o1
      if (!FWD || jj >= my_wins) return;
      nq = o1 - o0;
      const uint8_t *src = a.fwd + (uint64_t)o0 * a.quad_bytes + (ad_lo & 31u) * 8u;
      constexpr uint32_t kLo = kWarpAds / 2, kHi = kWarpAds / 4;  // 16-byte pieces per quad
      for (uint32_t i = lane; i < nq * kLo; i += 32)
        cp_async16(raw_a + (i / kLo) * raw_q + (i % kLo) * 16u,
                   src + (uint64_t)(i / kLo) * a.quad_bytes + (i % kLo) * 16u);
      if (a.quad_bytes > 256u)
        for (uint32_t i = lane; i < nq * kHi; i += 32)
          cp_async16(raw_a + (i / kHi) * raw_q + kWarpAds * 8u + (i % kHi) * 16u,
                     src - (ad_lo & 31u) * 4u + 256u + (uint64_t)(i / kHi) * a.quad_bytes +
                         (i % kHi) * 16u);
    };
    // the list of the window whose quads have arrived: row r of this warp's
    // ads; returns the rows that hold a key
    auto make_list = [&]() -> uint32_t {
      cp_async_wait();
      __syncwarp();
      constexpr uint32_t kStep = 32 / kWarpAds;  // quads at a time
      const uint32_t ad = lane % kWarpAds;
      uint32_t last = 0;
      for (uint32_t q = lane / kWarpAds; q < nq; q += kStep) {
        const uint32_t at = raw_a + q * raw_q;
        const float2 lf = lds_f2(at + ad * 8u);
        const uint32_t lx = __float_as_uint(lf.x), ly = __float_as_uint(lf.y);
        const uint32_t hi = a.quad_bytes > 256u ? lds_u32(at + kWarpAds * 8u + ad * 4u) : 0u;
        const uint32_t k[4] = {(lx & 0xFFFFu) | ((hi & 0xFFu) << 16), (lx >> 16) | ((hi & 0xFF00u) << 8),
                               (ly & 0xFFFFu) | (hi & 0xFF0000u), (ly >> 16) | ((hi >> 24) << 16)};
#pragma unroll
        for (uint32_t r = 0; r < 4; r++) {
          const uint32_t e = (4 * q + r) * kWarpAds + ad;
          if (k[r] != a.wt_rows - 1u) last = 4 * q + r + 1;
          if (SW)
            sts_u16(list_a + 2u * e, k[r]);
          else
            sts_u32(list_a + 4u * e, k[r] * (kGroup / 2));
        }
      }
      last = __reduce_max_sync(0xffffffffu, last);  // (and the list is written)
      __syncwarp();
      return last;
    };
    // A window starts when every warp has handed back the accumulators and the
    // list that it needs: what is waited for after that comes without the other
    // epilogue warps.  (They may be in a meeting, which this warp has to join: 2.)
    // 0: abort.
    auto may_start = [&](uint32_t w) -> uint32_t {
      auto ready = [&]() {
        return (w < kTb || mbar_try_wait(&sm.t_empty[w % kTb], ((w / kTb) - 1) & 1u)) &&
               (FWD || w < a.lb || mbar_try_wait(&sm.l_empty[w % a.lb], ((w / a.lb) - 1) & 1u));
      };
      if (*((volatile uint32_t *)&sm.abort)) return 0;
      if (ready()) return 1;
      const uint64_t t0 = global_timer_ns();
      while (!*((volatile uint32_t *)&sm.trim)) {
        if (ready()) return 1;
        if (*((volatile uint32_t *)&sm.abort)) return 0;
        if (global_timer_ns() - t0 > kWaitTimeoutNs) {
          atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
          sm.abort = 1;
          return 0;
        }
      }
      return 2;
    };
    read_offsets(0);
    fetch_quads(0);
    read_offsets(1);
    if (SW) {  // the slice of wT
      if (!mbar_wait_bounded(&sm.u_full, 0, kWaitTimeoutNs)) {
        atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
        sm.abort = 1;
      }
      __syncwarp();
    }
    for (;;) {
    while (j < my_wins && !__shfl_sync(0xffffffffu, *((volatile uint32_t *)&sm.trim), 0)) {
      const uint32_t tb = j % kTb, lbuf = FWD ? 0u : j % a.lb;
      uint32_t rows, tab_a;  // rows of the list, and its first entry of this warp's ads
      constexpr uint32_t kRowEntries = FWD ? kWarpAds : 32;
      const uint32_t go = __shfl_sync(0xffffffffu, lane == 0 ? may_start(j) : 0u, 0);
      if (go == 2) break;  // a meeting comes first
      if (go == 0) {
        j = my_wins;
        break;
      }
      if (FWD) {
        rows = make_list();
        tab_a = list_a;
        fetch_quads(j + 1);
        read_offsets(j + 2);
      } else {
        bool go = true;
        if (lane == 0)
          go = !*((volatile uint32_t *)&sm.abort) &&
               mbar_wait_bounded(&sm.l_full[lbuf], (j / a.lb) & 1u, kWaitTimeoutNs);
        go = __shfl_sync(0xffffffffu, (int)go, 0) != 0;
        if (!go) {
          if (lane == 0 && !*((volatile uint32_t *)&sm.abort)) {
            atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
            sm.abort = 1;
          }
          j = my_wins;
          break;
        }
        mbar_try_wait(&sm.l_full[lbuf], (j / a.lb) & 1u);
        const uint32_t *run_off = lists + (size_t)lbuf * list_words;
        rows = run_off[8 + (ad_lo >> 5)];
        tab_a = smem_u32(run_off + kListHdr) + (run_off[ad_lo >> 5] + (ad_lo & 31u)) * 4u;
      }
      const uint32_t wbase = (w_begin + j) * kWin;
      // this warp's ads in both users' bitmaps: in one word each, read
      // before the gathers
      const uint32_t ad_w = wbase + ad_lo;
      uint32_t bits0 = ok0 ? ~0u : 0u, bits1 = ok1 ? ~0u : 0u;
      if (ad_w < a.n_ads) {
        const uint64_t *f = a.filters + (uint64_t)(g0 + user0) * a.words + (ad_w >> 6);
        if (filt0) bits0 = (uint32_t)(__ldg(f) >> (ad_w & 63u));
        if (filt1) bits1 = (uint32_t)(__ldg(f + a.words) >> (ad_w & 63u));
      }
      bool t_ok = false;  // the window's deep scores have been waited for
      for (uint32_t c = 0; c < kWarpAds; c += 4) {
        const uint32_t a0 = ad_lo + c;  // first window-local ad of these four
        // lane i holds the row scale of ad i of the four (FP8)
        const uint32_t ad_l = wbase + a0 + (lane & 3);
        const float sa_l = F8 && ad_l < a.n_ads ? __ldg(a.ad_scale + ad_l) : 1.f;
        Row4 acc;
#pragma unroll
        for (int i = 0; i < 4; i++) acc.x[i] = make_float2(0.f, 0.f);
        // row r of the run: this user pair's weights of the four ads' r-th keys
        auto load_row = [&](uint32_t r) {
          const uint32_t at = tab_a + (r * kRowEntries + c) * (SW ? 2u : 4u);
          Row4 v;
          if (SW) {
            const float2 kf = lds_f2(at);
            const uint32_t k0 = __float_as_uint(kf.x), k1 = __float_as_uint(kf.y);
            v.x[0] = lds_f2(s_wcol + (k0 & 0xFFFFu) * (kGroup * 4u));
            v.x[1] = lds_f2(s_wcol + (k0 >> 16) * (kGroup * 4u));
            v.x[2] = lds_f2(s_wcol + (k1 & 0xFFFFu) * (kGroup * 4u));
            v.x[3] = lds_f2(s_wcol + (k1 >> 16) * (kGroup * 4u));
          } else {
            const uint4 k = lds_v4(at);
            v.x[0] = __ldg(wcol + k.x);
            v.x[1] = __ldg(wcol + k.y);
            v.x[2] = __ldg(wcol + k.z);
            v.x[3] = __ldg(wcol + k.w);
          }
          return v;
        };
        auto add_row = [&](const Row4 &v) {
#pragma unroll
          for (int i = 0; i < 4; i++) acc.x[i] = add_f32x2(acc.x[i], v.x[i]);
        };
        // rows in flight, refilled in turn: four from global memory (three:
        // 8.7 ms instead of 8.3 with 256 users and 5M ads), three from shared
        // memory (four: 4.49 ms instead of 4.27 with 64 users and 10M ads)
        constexpr uint32_t kFly = SW ? 3 : 4;
        Row4 v0, v1, v2, v3;
        if (rows > 0) v0 = load_row(0);
        if (rows > 1) v1 = load_row(1);
        if (rows > 2) v2 = load_row(2);
        if (kFly > 3 && rows > 3) v3 = load_row(3);
        uint32_t r = 0;
        for (; r + kFly <= rows; r += kFly) {
          add_row(v0);
          if (r + kFly < rows) v0 = load_row(r + kFly);
          add_row(v1);
          if (r + kFly + 1 < rows) v1 = load_row(r + kFly + 1);
          add_row(v2);
          if (r + kFly + 2 < rows) v2 = load_row(r + kFly + 2);
          if (kFly > 3) {
            add_row(v3);
            if (r + kFly + 3 < rows) v3 = load_row(r + kFly + 3);
          }
        }
        if (r < rows) add_row(v0);
        if (r + 1 < rows) add_row(v1);
        if (kFly > 3 && r + 2 < rows) add_row(v2);
        if (!t_ok) {
          // the deep scores are waited for only now: the MMAs ran behind the gathers
          t_ok = mbar_wait_bounded(&sm.t_full[tb], (j / kTb) & 1u, kWaitTimeoutNs);
          t_ok = __all_sync(0xffffffffu, t_ok);
          if (!t_ok) {
            if (lane == 0) {
              atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
              sm.abort = 1;
            }
            break;
          }
          tc_fence_after();
        }
        uint32_t d0[4], d1[4];  // deep scores of the four ads for both users
        tmem_ld4(tl + tb * tcols + a0, d0);
        tmem_ld4(tl + tb * tcols + kWin + a0, d1);
        tmem_ld_wait();
        const unsigned long long thr0 = *((volatile unsigned long long *)&sm.thr_u[user0]);
        const unsigned long long thr1 = *((volatile unsigned long long *)&sm.thr_u[user1]);
        const float thr0_f = key_score(thr0), thr1_f = key_score(thr1);  // NaN: no bound yet
        // scores, and which of them pass the bitmap and the float test (bits
        // 0-3: user0's four ads, 4-7: user1's); a NaN score passes
        float sc[8];
        uint32_t pass = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const float sa_i = F8 ? __shfl_sync(0xffffffffu, sa_l, i) : 1.f;
          const float deep0 = F8 ? __uint_as_float(d0[i]) * (sa_i * usc0) : __uint_as_float(d0[i]);
          const float deep1 = F8 ? __uint_as_float(d1[i]) * (sa_i * usc1) : __uint_as_float(d1[i]);
          sc[i] = deep0 + acc.x[i].x;
          sc[4 + i] = deep1 + acc.x[i].y;
          pass |= (!(sc[i] < thr0_f) ? 1u << i : 0u) | (!(sc[4 + i] < thr1_f) ? 16u << i : 0u);
        }
        const uint32_t left = a.n_ads - min(a.n_ads, wbase + a0);  // ads of the four that exist
        const uint32_t exist = left >= 4 ? 0xFu : (1u << left) - 1u;
        pass &= ((bits0 >> c) & exist) | (((bits1 >> c) & exist) << 4);
        // one candidate per thread and turn: few threads have any, and hardly
        // one has two, so a turn or two do for the eight (one inlined copy
        // instead of eight that each run for a lane or two)
        while (__any_sync(0xffffffffu, pass != 0u)) {
          if (pass) {
            const uint32_t e = __ffs(pass) - 1;
            pass &= pass - 1;
            float score = sc[0], wide = acc.x[0].x;
#pragma unroll
            for (int i = 1; i < 8; i++)
              if (e == (uint32_t)i) {
                score = sc[i];
                wide = i < 4 ? acc.x[i & 3].x : acc.x[i & 3].y;
              }
            offer(e < 4 ? user0 : user1, e < 4 ? thr0 : thr1, score, wide, wbase + a0 + (e & 3));
          }
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sm.t_empty[tb]);
        if (!FWD) mbar_arrive(&sm.l_empty[lbuf]);
      }
      j++;
      if (!t_ok) {  // timed out above
        j = my_wins;
        break;
      }
      if ((ok0 && *((volatile uint32_t *)&sm.cnt_u[user0]) + 2 * kBWin > a.cap_u) ||
          (ok1 && *((volatile uint32_t *)&sm.cnt_u[user1]) + 2 * kBWin > a.cap_u))
        *((volatile uint32_t *)&sm.trim) = 1u;
      __syncwarp();
    }
    gsync();
    if (tid == 0) {
      sm.stop_epi = *((volatile uint32_t *)&sm.abort);
      sm.meet = sm.trim;
      sm.trim = 0;
    }
    gsync();
    if (sm.stop_epi || !sm.meet) break;
    // make room: drop what the running threshold excludes, then, if that is
    // not enough, keep the exact top-m by radix select
    for (uint32_t b = warp; b < nG; b += kEpiWarps) {
      const uint32_t n = min(sm.cnt_u[b], a.cap_u);
      if (n + 2 * kBWin <= a.cap_u) continue;
      const uint32_t kept = warp_compact(user_buf(b), n, sm.thr_u[b]);
      if (lane == 0) {
        sm.cnt_u[b] = kept;
        sm.trim_u[b] = kept + 3 * kBWin > a.cap_u && kept > a.m;
      }
    }
    gsync();
    trim_users();
    gsync();
    }
    if (FWD) cp_async_wait();  // nothing in flight (after an abort) when the CTA ends
    if (tid == 0) *((volatile uint32_t *)&sm.finished) = 1u;
    // at most m candidates per user for the merge (it reads grid * m): those
    // above the latest bound, and if they are more, the best m
    if (!sm.stop_epi) {
      for (uint32_t b = tid; b < nG; b += kEpiThreads)
        if (sm.cnt_u[b] > a.m) raise_threshold(a, sm, g0, b);
      gsync();
      for (uint32_t b = warp; b < nG; b += kEpiWarps) {
        const uint32_t n = min(sm.cnt_u[b], a.cap_u);
        if (n <= a.m) continue;
        const uint32_t kept = warp_compact(user_buf(b), n, sm.thr_u[b]);
        if (lane == 0) {
          sm.cnt_u[b] = kept;
          sm.trim_u[b] = kept > a.m;
        }
      }
      gsync();
      trim_users();
    }
    gsync();
    for (uint32_t b = tid; b < nG; b += kEpiThreads) {
      a.cand_n[(uint64_t)blockIdx.x * a.B + g0 + b] = min(sm.cnt_u[b], a.cap_u);
      a.cand_thr[(uint64_t)blockIdx.x * a.B + g0 + b] = sm.cut_u[b];
    }
  }
  // Drain before teardown (matters only after an abort): the last issued
  // tile loads must have landed and the last MMAs retired before the
  // shared memory and TMEM are released.
  __syncthreads();
  if (tid == 0) {
    const uint32_t ni = sm.n_issued, nm = sm.n_mma;
    bool ok = mbar_wait_bounded(&sm.u_full, 0, kWaitTimeoutNs);
    for (uint32_t j = ni > a.sa ? ni - a.sa : 0; ok && j < ni; j++)
      ok = mbar_wait_bounded(&sm.a_full[j % a.sa], (j / a.sa) & 1u, kWaitTimeoutNs);
    if (ok && nm) ok = mbar_wait_bounded(&sm.t_full[(nm - 1) % a.tb], ((nm - 1) / a.tb) & 1u, kWaitTimeoutNs);
    if (!ok) atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp) tmem_dealloc(tmem, ncols);
}

// Per user: the best R*K of the CTAs' candidate buffers (exact if no CTA's
// buffer threshold exceeds the selected cut), rescored in FP32, best K.
// One CTA per user, and what bounds it is the chain of its steps: reads of the
// candidates a warp per buffer (a thread per buffer, then buffer after buffer by
// all threads: 100 us), both selections by score bins, four rows in flight per
// warp in the rescoring.  Measured, 2000 of 280k FP8 ads for 152 users (4000
// rescored each) 311 us, now 87; 250 users, two rounds of CTAs, 610 and 174.
// (CTAs of 512 threads, two to an SM, for more users than SMs: no gain.)
// Dynamic shared memory: merge_smem(kscan, kout) for the largest of the batch.
constexpr int kMergeThreads = 1024;
constexpr uint32_t kMergeCap = 32768;  // approximate candidates gathered per user
static size_t merge_smem(uint32_t ks, uint32_t ko) { return ((size_t)ks + sel_buf(ko)) * 8; }

__global__ void __launch_bounds__(kMergeThreads) k_batch_merge(
    const CandEntry *__restrict__ cand, const uint32_t *__restrict__ cand_n,
    const unsigned long long *__restrict__ cand_thr, uint32_t grid, uint32_t B, uint32_t cap_u,
    const uint32_t *__restrict__ kscan, const uint32_t *__restrict__ kout, uint32_t kmax,
    const float *__restrict__ emb, uint32_t d, const float *__restrict__ h_u,
    uint64_t *__restrict__ scratch /* [B][kMergeCap] */, uint32_t *__restrict__ out_ids,
    float *__restrict__ out_scores, uint32_t *__restrict__ status /* [B] */,
    const uint32_t *__restrict__ B_dev, const uint32_t *__restrict__ slot_dev,
    uint64_t out_slot_stride, uint32_t status_slot_stride) {
  constexpr uint32_t NT = kMergeThreads, NW = NT / 32;
  extern __shared__ __align__(16) uint64_t s_v[];  // [kscan], then the sort's buffer
  __shared__ SelSmem s_sel;
  __shared__ uint32_t s_hist[256], s_misc[8], s_cnt, s_ncut;
  __shared__ uint64_t s_cut[kSelMaxBin], s_T;  // the keys of the cut's bin
  __shared__ float s_cutw[kSelMaxBin];
  __shared__ float s_h[128];
  const uint32_t b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a device-side loop: only the wave's active users, results into its ring slot
  if (B_dev && b >= *B_dev) return;
  if (slot_dev) {
    const uint32_t slot = *slot_dev;
    out_ids += slot * out_slot_stride;
    out_scores += slot * out_slot_stride;
    status += (uint64_t)slot * status_slot_stride;
  }
  const uint32_t ks = kscan[b], ko = kout[b];
  if (tid == 0) {
    s_cnt = 0;
    s_ncut = 0;
    s_T = 0;
  }
  const uint64_t hrow = user_row(b);  // the user table is in pair order
  for (uint32_t i = tid; i < d; i += NT) s_h[i] = h_u[hrow * d + i];
  // this user's candidates, a warp per CTA's buffer
  auto for_entries = [&](auto f) {
    for (uint32_t c = warp; c < grid; c += NW) {
      const uint32_t n = __ldg(cand_n + (uint64_t)c * B + b);
      const CandEntry *src = cand + ((uint64_t)c * B + b) * cap_u;
      for (uint32_t i = lane; i < n; i += 32)
        if (src[i].key) f(src + i);
    }
  };
  auto add = [&](uint64_t key, float wide) {  // one more to rescore: (wide, id)
    const uint32_t pos = atomicAdd(&s_cnt, 1u);
    if (pos < ks) s_v[pos] = ((uint64_t)__float_as_uint(wide) << 32) | key_id(key);
  };
  // 1. the best ks by approximate score (T = 0: all of them)
  const SelCut c1 = sel_cut<NT>(
      s_sel, ks, [&](auto f) { for_entries([&](const CandEntry *e) { f(e->key); }); });
  if (c1.real <= ks) {
    for_entries([&](const CandEntry *e) { add(e->key, e->wide); });
  } else if (!c1.crowded) {
    for_entries([&](const CandEntry *e) {
      const uint64_t x = e->key;
      const uint32_t bin = c1.bin(x);
      if (bin > c1.cut) {
        add(x, e->wide);
      } else if (bin == c1.cut) {
        const uint32_t pos = atomicAdd(&s_ncut, 1u);
        s_cut[pos] = x;
        s_cutw[pos] = e->wide;
      }
    });
    __syncthreads();
    const uint32_t n = s_ncut, need = ks - (c1.m - n);
    if (tid < n) {
      const uint64_t x = s_cut[tid];
      uint32_t rank = 0;
      for (uint32_t q = 0; q < n; q++) rank += s_cut[q] > x ? 1u : 0u;
      if (rank < need) add(x, s_cutw[tid]);
      if (rank == need - 1) s_T = x;
    }
  } else {
    uint64_t *keys = scratch + (uint64_t)b * kMergeCap;
    for_entries([&](const CandEntry *e) {
      const uint32_t pos = atomicAdd(&s_ncut, 1u);
      if (pos < kMergeCap) keys[pos] = e->key;
    });
    __syncthreads();
    const uint64_t T = cta_radix_select<NT>(keys, min(s_ncut, kMergeCap), ks, s_hist, s_misc);
    if (tid == 0) s_T = T;
    for_entries([&](const CandEntry *e) {
      if (e->key >= T) add(e->key, e->wide);
    });
  }
  __syncthreads();
  // Exactness: CTA c holds every one of its candidates with key >= its
  // threshold, so the union's best ks are the inventory's best ks when no
  // threshold lies above the selected cut T.
  uint32_t inexact = c1.real > kMergeCap;
  for (uint32_t c = tid; c < grid; c += NT)
    if (cand_thr[(uint64_t)c * B + b] > s_T) inexact = 1;
  if (inexact) atomicOr(&status[b], 1u);
  // 2. FP32 rescoring, a warp per candidate (coalesced rows), in place
  const uint32_t nres = min(s_cnt, ks);
  auto rescore = [&](auto d32, auto per) {  // d / 32, candidates in flight per warp
    constexpr int kT = decltype(d32)::value, kU = decltype(per)::value;
    for (uint32_t i0 = warp * kU; i0 < nres; i0 += NW * kU) {
      uint64_t e[kU];
      float x[kU][kT], dot[kU];
#pragma unroll
      for (int u = 0; u < kU; u++) {
        e[u] = s_v[i0 + u < nres ? i0 + u : i0];  // (this warp's own entries only)
        const float *row = emb + (uint64_t)(uint32_t)e[u] * (32 * kT) + lane;
#pragma unroll
        for (int t = 0; t < kT; t++) x[u][t] = __ldg(row + 32 * t);
      }
#pragma unroll
      for (int u = 0; u < kU; u++) {
        dot[u] = 0.f;
#pragma unroll
        for (int t = 0; t < kT; t++) dot[u] = fmaf(s_h[32 * t + lane], x[u][t], dot[u]);
      }
#pragma unroll
      for (int o = 16; o; o >>= 1)
#pragma unroll
        for (int u = 0; u < kU; u++) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
      __syncwarp();
#pragma unroll
      for (int u = 0; u < kU; u++)
        if (lane == (uint32_t)u && i0 + u < nres)
          s_v[i0 + u] = make_key(dot[u] + __uint_as_float((uint32_t)(e[u] >> 32)), (uint32_t)e[u]);
    }
  };
  if (d == 64)
    rescore(std::integral_constant<int, 2>(), std::integral_constant<int, 8>());
  else
    rescore(std::integral_constant<int, 4>(), std::integral_constant<int, 4>());
  __syncthreads();
  // 3. best ko, sorted
  uint64_t *buf = s_v + ks;
  auto for_resc = [&](auto f) {
    for (uint32_t i = tid; i < nres; i += NT) f(s_v[i]);
  };
  auto emit = [&](uint32_t r, uint64_t x) {
    out_ids[(uint64_t)b * kmax + r] = key_id(x);
    out_scores[(uint64_t)b * kmax + r] = key_score(x);
  };
  const SelCut c2 = sel_cut<NT>(s_sel, ko, for_resc);
  if (c2.take && !c2.crowded && c2.m <= sel_buf(ko)) {
    sel_sorted<NT>(s_sel, c2, buf, for_resc, emit);
  } else if (c2.take) {
    uint64_t T2 = 0;
    if (nres > ko) T2 = cta_radix_select<NT>(s_v, nres, ko, s_hist, s_misc);
    if (tid == 0) s_ncut = 0;
    __syncthreads();
    uint32_t p2 = 1;
    while (p2 < c2.take) p2 <<= 1;
    for_resc([&](uint64_t x) {
      if (x < T2) return;
      const uint32_t pos = atomicAdd(&s_ncut, 1u);
      if (pos < p2) buf[pos] = x;
    });
    __syncthreads();
    for (uint32_t i = c2.take + tid; i < p2; i += NT) buf[i] = 0ull;
    bitonic_sort_desc<NT>(buf, p2);
    for (uint32_t i = tid; i < c2.take; i += NT) emit(i, buf[i]);
  }
  for (uint32_t i = c2.take + tid; i < kmax; i += NT) {
    out_ids[(uint64_t)b * kmax + i] = 0xFFFFFFFFu;
    out_scores[(uint64_t)b * kmax + i] = -INFINITY;
  }
}

}  // namespace ebr

// =====================================================================
// Host side of the batched path
// =====================================================================
namespace ebr {

// Pointers of one request's inputs (device memory), gathered by
// k_stage_requests into the batch's contiguous arrays.
struct ReqSrc {
  const float *h_u;
  const uint32_t *vals;    // [n] user field values
  const uint64_t *filter;  // null: no filter
  const uint32_t *ptr;     // [f_u + 1] field offsets into vals; null: one value per field
  uint32_t n, base;        // values, and their first position in the batch's value array
};
constexpr uint32_t kStageWords = 8192;  // filter words per block of the gather

// Block (b, y): request b's user vector (to row user_row(b)), field
// values and field offsets (y == 0) and words [y * kStageWords, +kStageWords)
// of its filter.  With B_dev (a device-side loop launching Bq blocks), blocks
// past the wave's users zero their user row and stop.  With
// uptr set, the offsets are written (relative to the request's base, base[b]
// beside them) after a check that they start at 0, do not decrease and end
// at n; offsets that fail it are flagged and every field is left empty.
__global__ void __launch_bounds__(256) k_stage_requests(const ReqSrc *__restrict__ src,
                                                        uint32_t d, uint32_t fu, uint32_t words,
                                                        float *__restrict__ users,
                                                        uint32_t *__restrict__ vals,
                                                        uint32_t *__restrict__ uptr,
                                                        uint32_t *__restrict__ base,
                                                        uint64_t *__restrict__ filters,
                                                        uint32_t *__restrict__ flags,
                                                        const uint32_t *__restrict__ B_dev) {
  __shared__ uint32_t s_ok;
  const uint32_t b = blockIdx.x;
  if (B_dev && b >= *B_dev) {  // a device-side loop's wave has fewer users: zero the row
    if (blockIdx.y == 0)
      for (uint32_t t = threadIdx.x; t < d; t += blockDim.x)
        users[(size_t)user_row(b) * d + t] = 0.f;
    return;
  }
  const ReqSrc r = src[b];
  if (blockIdx.y == 0) {
    const size_t row = (size_t)user_row(b);
    for (uint32_t t = threadIdx.x; t < d; t += blockDim.x) users[row * d + t] = r.h_u[t];
    for (uint32_t t = threadIdx.x; t < r.n; t += blockDim.x) vals[(size_t)r.base + t] = r.vals[t];
    if (uptr) {
      if (threadIdx.x == 0) {
        uint32_t ok = 1;
        if (r.ptr) {
          uint32_t prev = 0;
          for (uint32_t i = 0; i <= fu; i++) {
            const uint32_t x = r.ptr[i];
            if ((i == 0 && x != 0) || x < prev || (i == fu && x != r.n)) ok = 0;
            prev = x;
          }
        }
        if (!ok) atomicOr(flags, DEVERR_BAD_USER);
        s_ok = ok;
        base[b] = r.base;
      }
      __syncthreads();
      for (uint32_t i = threadIdx.x; i <= fu; i += blockDim.x)
        uptr[(size_t)b * (fu + 1) + i] = !s_ok ? 0u : (r.ptr ? r.ptr[i] : i);
    }
  }
  if (r.filter) {
    const uint32_t w0 = blockIdx.y * kStageWords;
    const uint32_t w1 = min(words, w0 + kStageWords);
    for (uint32_t t = w0 + threadIdx.x; t < w1; t += blockDim.x)
      filters[(size_t)b * words + t] = r.filter[t];
  }
}

// Layout of the batch's user field values: request b's n[b] values start at
// base[b] (one value per field without user_ptr); returns the total.
static uint64_t user_vals_layout(const ebr_query *q, uint32_t B, uint32_t fu,
                                 std::vector<uint32_t> *n, std::vector<uint32_t> *base) {
  uint64_t t = 0;
  n->resize(B);
  base->resize(B);
  for (uint32_t b = 0; b < B; b++) {
    (*n)[b] = q[b].user_ptr ? q[b].n_user_vals : fu;
    (*base)[b] = (uint32_t)t;
    t += (*n)[b];
  }
  return t;
}

struct BatchPlan {
  uint32_t Bq, m, cap_u, sa, lb, tb, list_cap, tile_row, kb_n;
  int mode;  // kWalk, kForward, kForwardSw
  size_t smem;
};

// The batch rounded up to whole groups of users.
static uint32_t users_padded(uint32_t B) { return (B + kGroup - 1) / kGroup * kGroup; }

// Shared-memory layout of k_batch_window: a group's two M-tiles, `sa` ad
// stages, the key lists, the trims' histograms and, for a small key space, a
// group's slice of w^T.  One 256-ad stage (or two of 128) is enough, since the next window's MMAs
// wait for this window's accumulators to be read anyway, and what is left is
// L1 for the gathers.
constexpr size_t kBatchSmemBudget = 220 * 1024;
static bool plan_smem(const ebr_index *ix, uint32_t B, BatchPlan *p) {
  p->Bq = users_padded(B);
  p->list_cap = kBWin * ix->max_keys_per_ad;  // 8 runs x 32 ads x rows
  const uint32_t n_mt = 2;  // even and odd users
  const uint32_t win = ix->fwd ? kFwdWin : kBWin;
  p->tb = accum_bufs(ix->fwd != nullptr);
  p->sa = ix->fwd ? 2 : 1;
  const uint32_t row_bytes = ix->d * (ix->dtype == EBR_FP8E4M3 ? 1u : 2u);
  p->tile_row = row_bytes >= 128 ? 128u : 64u;
  p->kb_n = row_bytes / p->tile_row;
  const size_t u_bytes = (size_t)n_mt * p->kb_n * 128 * p->tile_row;
  const size_t a_stage = (size_t)p->kb_n * win * p->tile_row;
  const size_t hist = (size_t)kTrimWarps * 256 * 4;
  const size_t fixed = 1024 + u_bytes + p->sa * a_stage + hist;
  const uint32_t mq = ix->fwd_max_quads[0];
  const size_t raw = (size_t)mq * win * (ix->fwd_quad_bytes > 256u ? 12 : 8);
  if (ix->fwd) {
    const size_t wt = ((size_t)ix->n_keys + 1) * kGroup * 4;
    p->lb = 1;
    p->mode = kForwardSw;
    p->smem = fixed + raw + (size_t)mq * 4 * win * 2 + wt;
    if (ix->n_keys < 4096 && p->smem <= kBatchSmemBudget) return true;
    p->mode = kForward;
    p->smem = fixed + raw + (size_t)mq * 4 * win * 4;
    if (p->smem <= kBatchSmemBudget) return true;
    return false;
  }
  p->mode = kWalk;
  for (p->lb = 2; p->lb >= 1; p->lb--) {
    p->smem = fixed + p->lb * ((size_t)kListHdr + p->list_cap) * 4;
    if (p->smem <= kBatchSmemBudget) return true;
  }
  return false;
}

// (The last but one condition bounds w^T, 17 GB: a batch over a larger key space is served
// by single requests, whose scratch does not grow with the users.)
bool batch_index_ok(const ebr_index *ix, const ebr_cross *cross, uint32_t batch) {
  BatchPlan p;
  return (ix->dtype == EBR_BF16 || ix->dtype == EBR_FP8E4M3) && (ix->d == 64 || ix->d == 128) &&
         batch >= 2 && batch <= (uint32_t)kMaxUsers && cross && cross->n_keys == ix->n_keys &&
         ix->n_win > 0 && ix->ad_nkeys.p && ix->max_keys_per_ad > 0 &&
         ix->max_keys_per_ad <= kMaxBatchKeysPerAd &&
         ((uint64_t)ix->n_keys + 1) * users_padded(batch) < (1ull << 32) &&
         plan_smem(ix, batch, &p);
}

bool batch_qualifies(const ebr_index *ix, const ebr_cross *cross, const ebr_query *q,
                     uint32_t batch) {
  if (!batch_index_ok(ix, cross, batch)) return false;
  for (uint32_t b = 0; b < batch; b++) {
    if (!q[b].user_vals || (q[b].flags & EBR_QF_KEY_MAJOR)) return false;
    if ((uint64_t)q[b].k * ix->rescore_mult > 8192) return false;
  }
  return true;
}

static bool plan_batch(const ebr_index *ix, uint32_t B, uint32_t kscan_max, int grid,
                       BatchPlan *p) {
  if (!plan_smem(ix, B, p)) return false;
  const uint32_t per_cta = (kscan_max + grid - 1) / grid;
  p->m = std::max<uint32_t>(64, (2 * per_cta + 32 + 31) / 32 * 32);
  p->cap_u = 4 * p->m + 2 * kBWin;  // room for 4m entries and what the warps add before they meet
  return (uint64_t)grid * p->m <= kMergeCap;
}

// Device bytes of every buffer of one batched call (B users, scan depth up to
// kscan_max), in one place for the reservation below and the serving loop's
// memory budget.  The pinned host mirror holds [kscan B][kout B][has_filter B]
// [status B] words, then the request pointer table.
struct BatchSizes {
  BatchPlan pl;
  int grid;
  size_t users_f32, users_q, users_scale, user_vals, user_ptr, wT, filters, small, cand, cand_n,
      cand_thr, uhist, scratch, ctrl, req, host;
  size_t total() const {
    size_t t = 0;
    for (size_t b : {users_f32, users_q, users_scale, user_vals, user_ptr, wT, filters, small,
                     cand, cand_n, cand_thr, uhist, scratch, ctrl, req})
      t += (b + 255) / 256 * 256;
    return t;
  }
};

// Per-user score histograms, then their maps of bins in use (one memset clears both).
static size_t user_hist_bytes(uint32_t B) { return (size_t)B * (kUserBins + kMapWords) * 4; }

static size_t host_table_off(uint32_t B) { return ((size_t)4 * B * 4 + 15) / 16 * 16; }

// CTAs per group of users.  A large index has one per SM, group after group
// (64 users' weights at a time stay in L2); a small one, where a CTA would have
// few windows for its set-up and its own candidates, one wave over all groups.
// Scan, one wave against group after group, us: 54k ads x 161 users 208 and 269,
// 427k x 185 797 and 1177, 661k x 73 841 and 811, 5M x 256 9116 and 8493; the line is
// at 32 windows of 128 ads per CTA (622k ads).
static int batch_grid(const ebr_index *ix, uint32_t Bq) {
  const uint32_t n_win = (ix->n_ads + kFwdWin - 1) / kFwdWin;
  const bool one_wave = n_win < 32u * (uint32_t)ix->num_sms;
  const int ctas = one_wave ? ix->num_sms / (int)(Bq / kGroup) : ix->num_sms;
  return std::max(1, std::min<int>(ctas, (int)ix->n_win));
}

static bool batch_sizes(const ebr_index *ix, const ebr_cross *cross, uint32_t B,
                        uint32_t kscan_max, uint64_t n_vals, BatchSizes *z) {
  if (n_vals == 0) n_vals = (uint64_t)B * cross->f_u;
  // the serving loop's narrower waves use the same buffers
  size_t entries = 0, ctas = 0;
  for (uint32_t q = kGroup; q <= users_padded(B); q += kGroup) {
    z->grid = batch_grid(ix, q);
    if (!plan_batch(ix, q, kscan_max, z->grid, &z->pl)) return false;
    entries = std::max<size_t>(entries, (size_t)z->grid * z->pl.cap_u);
    ctas = std::max<size_t>(ctas, z->grid);
  }
  const size_t Bp = z->pl.Bq, d = ix->d, words = (ix->n_ads + 63) / 64;
  z->users_f32 = Bp * d * 4;
  z->users_q = Bp * d * 2;  // BF16 or FP8 users
  z->users_scale = Bp * 4;
  z->user_vals = (size_t)n_vals * 4;
  z->user_ptr = (size_t)B * (cross->f_u + 2) * 4;  // offsets [B][f_u + 1], then base [B]
  z->wT = ((size_t)ix->n_keys + 1) * Bp * 4;
  z->filters = (size_t)B * words * 8;
  z->small = small_bytes(B);
  z->cand = entries * B * sizeof(CandEntry);
  z->cand_n = ctas * B * 4;
  z->cand_thr = ctas * B * 8;
  z->uhist = user_hist_bytes(B);
  z->scratch = (size_t)B * kMergeCap * 8;
  z->ctrl = sizeof(Ctrl);
  z->req = (size_t)B * sizeof(ReqSrc);
  // after the words: the pointer table (device requests) or the packed user
  // vectors and field values (host requests)
  z->host = host_table_off(B) + std::max(z->req, Bp * d * 4 + z->user_ptr + z->user_vals);
  return true;
}

size_t batch_ws_bytes(const ebr_index *ix, const ebr_cross *cross, uint32_t B,
                      uint32_t kscan_max, uint64_t n_vals) {
  BatchSizes z;
  return batch_sizes(ix, cross, B, kscan_max, n_vals, &z) ? z.total() : 0;
}

int batch_ws_reserve(const ebr_index *ix, const ebr_cross *cross, uint32_t B,
                     uint32_t kscan_max, uint64_t n_vals, BatchWs &w) {
  BatchSizes z;
  if (!batch_sizes(ix, cross, B, kscan_max, n_vals, &z)) {
    set_error("batched scan: per-window key tables (%u keys per ad) do not fit shared memory",
              ix->max_keys_per_ad);
    return EBR_EINVAL;
  }
  EBR_TRY(dev_reserve(w.users_f32, z.users_f32));
  EBR_TRY(dev_reserve(w.users_bf16, z.users_q));
  EBR_TRY(dev_reserve(w.users_scale, z.users_scale));
  EBR_TRY(dev_reserve(w.user_vals, z.user_vals));
  EBR_TRY(dev_reserve(w.user_ptr, z.user_ptr));
  EBR_TRY(dev_reserve(w.wT, z.wT));
  EBR_TRY(dev_reserve(w.filters, z.filters));
  EBR_TRY(dev_reserve(w.small, z.small));
  EBR_TRY(dev_reserve(w.cand, z.cand));
  EBR_TRY(dev_reserve(w.cand_n, z.cand_n));
  EBR_TRY(dev_reserve(w.cand_thr, z.cand_thr));
  EBR_TRY(dev_reserve(w.uhist, z.uhist));
  EBR_TRY(dev_reserve(w.scratch, z.scratch));
  EBR_TRY(dev_reserve(w.ctrl, z.ctrl));
  EBR_TRY(dev_reserve(w.req, z.req));
  if (w.host_bytes < z.host) {
    if (w.host) cudaFreeHost(w.host);
    w.host = nullptr;
    w.host_bytes = 0;
    if (cudaMallocHost(&w.host, z.host) != cudaSuccess) {
      cudaGetLastError();
      set_error("batched scan: pinned host allocation of %zu bytes failed", z.host);
      return EBR_ENOMEM;
    }
    w.host_bytes = z.host;
  }
  return EBR_OK;
}

static int stage(void *dst, const void *src, size_t bytes, int io, cudaStream_t st) {
  if (!bytes) return EBR_OK;
  EBR_CUDA_TRY(cudaMemcpyAsync(dst, src, bytes,
                               io == EBR_IO_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                               st));
  return EBR_OK;
}

// The last row of every group's slice of w^T: the lists' padding key.  (The pitch
// may pass 2^31 bytes, 8.4 M keys: unlike a 2-D copy's it is not limited.)
static cudaError_t clear_zero_rows(const ebr_index *ix, BatchWs &w, uint32_t Bq, cudaStream_t st) {
  const size_t slice = ((size_t)ix->n_keys + 1) * kGroup * 4;
  return cudaMemset2DAsync((char *)w.wT.p + (size_t)ix->n_keys * kGroup * 4, slice, 0, kGroup * 4,
                           Bq / kGroup, st);
}

static void (*window_kernel(bool f8, int mode))(BatchArgs) {
  if (mode == kForwardSw)
    return f8 ? k_batch_window<true, kForwardSw> : k_batch_window<false, kForwardSw>;
  if (mode == kForward)
    return f8 ? k_batch_window<true, kForward> : k_batch_window<false, kForward>;
  return f8 ? k_batch_window<true, kWalk> : k_batch_window<false, kWalk>;
}

// The window kernel's arguments for a batch of B users (B: the candidate
// buffers' user stride; B_dev: the active users, read on the device, or null).
static int fill_batch_args(ebr_index *ix, uint32_t B, const BatchPlan &pl, BatchWs &w,
                           const uint32_t *kscan, const uint32_t *has_filter, Ctrl *ctrl,
                           const uint32_t *B_dev, BatchArgs *out) {
  const bool f8 = ix->dtype == EBR_FP8E4M3;
  const uint32_t eb = f8 ? 1u : 2u, d = ix->d, Bp = pl.Bq;
  if (!w.tmap_ready || w.tmap_for != ix->emb_q.p) {
    EBR_TRY(make_tmap_2d(reinterpret_cast<CUtensorMap *>(w.tmap_bytes), ix->emb_q.p, ix->n_ads, d,
                         eb, 128));
    w.tmap_ready = true;
    w.tmap_for = ix->emb_q.p;
  }
  BatchArgs &a = *out;
  memset(&a, 0, sizeof(a));
  memcpy(&a.ta, w.tmap_bytes, sizeof(CUtensorMap));
  EBR_TRY(make_tmap_2d(&a.tu, w.users_bf16.p, Bp, d, eb, kGroup / 2));
  a.tile_row = pl.tile_row;
  a.kb_n = pl.kb_n;
  a.ad_scale = f8 ? (const float *)ix->emb_scale.p : nullptr;
  a.user_scale = f8 ? (const float *)w.users_scale.p : nullptr;
  for (int g = 0; g < kGroups; g++) {
    a.wkey[g] = ix->wkey[g];
    a.wvals[g] = ix->wvals[g];
    a.win_ptr[g] = ix->win_ptr[g];
  }
  a.ad_nkeys = (const uint16_t *)ix->ad_nkeys.p;
  a.fwd = ix->fwd;
  a.fwd_off = ix->fwd_off;
  a.quad_bytes = ix->fwd_quad_bytes;
  a.max_quads = ix->fwd_max_quads[0];
  a.wT = (const float *)w.wT.p;
  a.filters = (const uint64_t *)w.filters.p;
  a.has_filter = has_filter;
  a.n_ads = ix->n_ads;
  a.n_win = pl.mode == kWalk ? ix->n_win : (ix->n_ads + kFwdWin - 1) / kFwdWin;
  a.B = B;
  a.B_dev = B_dev;
  a.wt_rows = ix->n_keys + 1;
  a.d = d;
  a.m = pl.m;
  a.cap_u = pl.cap_u;
  a.list_cap = pl.list_cap;
  a.zero_row = ix->n_keys * (kGroup / 2);  // in 8-byte pair units
  a.words = (ix->n_ads + 63) / 64;
  a.sa = pl.sa;
  a.lb = pl.lb;
  a.tb = pl.tb;
  a.cand = (CandEntry *)w.cand.p;
  a.cand_n = (uint32_t *)w.cand_n.p;
  a.cand_thr = (unsigned long long *)w.cand_thr.p;
  a.uhist = (uint32_t *)w.uhist.p;
  a.umap = a.uhist + (size_t)B * kUserBins;
  a.kscan = kscan;
  a.ctrl = ctrl;
  return EBR_OK;
}

// Stages the batch's requests into w, launches expansion, the window scan and
// the merge on st, and queues the copies of the per-user status and the
// control block to w's pinned mirror.  Nothing here waits for the device.
int batch_launch(ebr_index *ix, const ebr_cross *cross, const ebr_query *q, uint32_t B,
                 uint32_t *d_ids, float *d_scores, uint32_t kmax, int io, BatchWs &w,
                 cudaStream_t st) {
  const uint32_t d = ix->d, fu = cross->f_u, words = (ix->n_ads + 63) / 64;
  uint32_t kscan_max = 1;
  for (uint32_t b = 0; b < B; b++)
    kscan_max = std::max(kscan_max, std::min<uint32_t>(q[b].k * ix->rescore_mult, ix->n_ads));
  std::vector<uint32_t> nv, vbase;
  const uint64_t n_vals = user_vals_layout(q, B, fu, &nv, &vbase);
  bool multi = false;
  for (uint32_t b = 0; b < B; b++) multi |= q[b].user_ptr != nullptr;
  if (io == EBR_IO_HOST)  // offsets of host requests are checked here, before anything is queued
    for (uint32_t b = 0; b < B; b++) {
      const uint32_t *p = q[b].user_ptr;
      if (!p) continue;
      for (uint32_t i = 0; i <= fu; i++)
        if ((i == 0 && p[0] != 0) || (i > 0 && p[i] < p[i - 1]) || (i == fu && p[i] != nv[b])) {
          set_error("ebr_score_topk: request %u: user_ptr must start at 0, not decrease and end "
                    "at n_user_vals",
                    b);
          return EBR_EDATA;
        }
    }
  if (n_vals >= (1ull << 32)) {
    set_error("batched scan: %llu user values in one batch", (unsigned long long)n_vals);
    return EBR_EINVAL;
  }
  // profiling events (ebr_profile_enable): before staging, before the scan,
  // after the scan, after the merge
  std::array<cudaEvent_t, 5> ev{};
  const bool prof = ix->prof;
  if (prof) {
    if (!ix->prof_pool.empty()) {
      ev = ix->prof_pool.back();
      ix->prof_pool.pop_back();
    } else {
      for (auto &e : ev) EBR_CUDA_TRY(cudaEventCreate(&e));
    }
    EBR_CUDA_TRY(cudaEventRecord(ev[0], st));
  }
  EBR_TRY(batch_ws_reserve(ix, cross, B, kscan_max, n_vals, w));
  BatchSizes z;
  batch_sizes(ix, cross, B, kscan_max, n_vals, &z);
  const int grid = z.grid;
  const BatchPlan pl = z.pl;
  const uint32_t Bp = pl.Bq;
  // pinned host mirror: [kscan B][kout B][has_filter B] in, then [status B]
  // out, then the request table
  uint32_t *h_in = reinterpret_cast<uint32_t *>(w.host);
  for (uint32_t b = 0; b < B; b++) {
    h_in[b] = std::min<uint32_t>(q[b].k * ix->rescore_mult, ix->n_ads);
    h_in[B + b] = q[b].k;
    h_in[2 * B + b] = q[b].filter ? 1u : 0u;
  }
  uint32_t *kk = (uint32_t *)w.small.p;
  uint32_t *has_filter = kk + 2 * B;
  uint32_t *status = (uint32_t *)((char *)w.small.p + small_status_off(B));
  Ctrl *ctrl = (Ctrl *)w.ctrl.p;
  EBR_CUDA_TRY(cudaMemsetAsync(ctrl, 0, sizeof(Ctrl), st));
  EBR_CUDA_TRY(cudaMemcpyAsync(kk, h_in, (size_t)3 * B * 4, cudaMemcpyHostToDevice, st));
  EBR_CUDA_TRY(cudaMemsetAsync(status, 0, B * 4, st));
  EBR_CUDA_TRY(cudaMemsetAsync(w.uhist.p, 0, user_hist_bytes(B), st));
  // request inputs: device-resident requests are gathered by one kernel
  // through a table of their pointers; host requests are packed into the
  // pinned mirror and copied in two transfers (filters one per request)
  // user vectors in pair order (user_row); rows of absent users stay zero
  if (Bp > B) EBR_CUDA_TRY(cudaMemsetAsync(w.users_f32.p, 0, (size_t)Bp * d * 4, st));
  bool any_filter = false;
  for (uint32_t b = 0; b < B; b++) any_filter |= q[b].filter != nullptr;
  uint32_t *d_uptr = multi ? (uint32_t *)w.user_ptr.p : nullptr;
  uint32_t *d_base = multi ? d_uptr + (size_t)B * (fu + 1) : nullptr;
  if (io == EBR_IO_HOST) {
    // [user vectors Bq x d, pair order][offsets B x (f_u + 1)][base B][values]
    float *hu = reinterpret_cast<float *>((char *)w.host + host_table_off(B));
    uint32_t *hp = reinterpret_cast<uint32_t *>(hu + (size_t)Bp * d);
    uint32_t *hv = hp + (size_t)B * (fu + 2);
    if (Bp > B) memset(hu, 0, (size_t)Bp * d * 4);
    for (uint32_t b = 0; b < B; b++) {
      memcpy(hu + (size_t)user_row(b) * d, q[b].h_u, (size_t)d * 4);
      memcpy(hv + vbase[b], q[b].user_vals, (size_t)nv[b] * 4);
      if (!multi) continue;
      uint32_t *up = hp + (size_t)b * (fu + 1);
      for (uint32_t i = 0; i <= fu; i++) up[i] = q[b].user_ptr ? q[b].user_ptr[i] : i;
      hp[(size_t)B * (fu + 1) + b] = vbase[b];
    }
    EBR_CUDA_TRY(cudaMemcpyAsync(w.users_f32.p, hu, (size_t)Bp * d * 4, cudaMemcpyHostToDevice, st));
    if (multi)
      EBR_CUDA_TRY(cudaMemcpyAsync(d_uptr, hp, (size_t)B * (fu + 2) * 4, cudaMemcpyHostToDevice, st));
    EBR_CUDA_TRY(cudaMemcpyAsync(w.user_vals.p, hv, n_vals * 4, cudaMemcpyHostToDevice, st));
    for (uint32_t b = 0; b < B; b++)
      if (q[b].filter)
        EBR_TRY(stage((uint64_t *)w.filters.p + (size_t)b * words, q[b].filter, words * 8, io, st));
  } else {
    ReqSrc *tab = reinterpret_cast<ReqSrc *>((char *)w.host + host_table_off(B));
    for (uint32_t b = 0; b < B; b++)
      tab[b] = ReqSrc{q[b].h_u, q[b].user_vals, q[b].filter, q[b].user_ptr, nv[b], vbase[b]};
    EBR_CUDA_TRY(cudaMemcpyAsync(w.req.p, tab, (size_t)B * sizeof(ReqSrc), cudaMemcpyHostToDevice,
                                 st));
    const uint32_t ys = any_filter ? (words + kStageWords - 1) / kStageWords : 1u;
    k_stage_requests<<<dim3(B, ys), 256, 0, st>>>((const ReqSrc *)w.req.p, d, fu, words,
                                                  (float *)w.users_f32.p,
                                                  (uint32_t *)w.user_vals.p, d_uptr, d_base,
                                                  (uint64_t *)w.filters.p, &ctrl->flags, nullptr);
    EBR_CUDA_TRY(cudaGetLastError());
    ix->launches += 1;
  }
  const bool f8 = ix->dtype == EBR_FP8E4M3;
  if (f8)  // users as FP8 with a scale per user (kind::f8f6f4 takes both operands in FP8)
    EBR_TRY(launch_quantize_rows_fp8((const float *)w.users_f32.p, Bp, d, (uint8_t *)w.users_bf16.p,
                                     (float *)w.users_scale.p, st));
  else
    EBR_TRY(launch_quantize((const float *)w.users_f32.p, (uint64_t)Bp * d, EBR_BF16,
                            w.users_bf16.p, st));
  EBR_TRY(expand_transposed(cross, (const uint32_t *)w.user_vals.p, d_uptr, d_base, B, Bp,
                            (float *)w.wT.p, &ctrl->flags, ix->num_sms, st, nullptr,
                            ix->key_id));
  EBR_CUDA_TRY(clear_zero_rows(ix, w, Bp, st));
  BatchArgs a;
  EBR_TRY(fill_batch_args(ix, B, pl, w, kk, has_filter, ctrl, nullptr, &a));
  auto kern = window_kernel(f8, pl.mode);
  EBR_CUDA_TRY(allow_smem(kern, kBatchSmemBudget));
  if (prof) EBR_CUDA_TRY(cudaEventRecord(ev[1], st));
  kern<<<dim3(grid, Bp / kGroup), batch_threads(pl.mode), pl.smem, st>>>(a);
  EBR_CUDA_TRY(cudaGetLastError());
  if (prof) EBR_CUDA_TRY(cudaEventRecord(ev[2], st));
  const size_t msm = merge_smem(kscan_max, kmax);
  EBR_CUDA_TRY(allow_smem(k_batch_merge, merge_smem(8192, 8192)));
  k_batch_merge<<<B, kMergeThreads, msm, st>>>(
      (const CandEntry *)w.cand.p, (const uint32_t *)w.cand_n.p,
      (const unsigned long long *)w.cand_thr.p, (uint32_t)grid, B, pl.cap_u, kk, kk + B, kmax,
      (const float *)ix->emb_f32.p, d, (const float *)w.users_f32.p,
      (uint64_t *)w.scratch.p, d_ids, d_scores, status, nullptr, nullptr, 0, 0);
  EBR_CUDA_TRY(cudaGetLastError());
  if (prof) {
    EBR_CUDA_TRY(cudaEventRecord(ev[3], st));
    ix->bprof_pending.push_back(ev);
  }
  ix->launches += 4;
  ix->batched += B;
  // status and flags back to the pinned mirror
  uint32_t *h_status = h_in + 3 * B;
  EBR_CUDA_TRY(cudaMemcpyAsync(h_status, status, B * 4, cudaMemcpyDeviceToHost, st));
  return EBR_OK;
}

// Waits for a batch started by batch_launch, checks the device flags and
// recomputes on the single-request scan every user whose candidate buffers
// could not prove exactness (outputs rewritten in place on st).
int batch_finish(ebr_index *ix, const ebr_cross *cross, const ebr_query *q, uint32_t B,
                 uint32_t *d_ids, float *d_scores, uint32_t kmax, BatchWs &w, cudaStream_t st) {
  const uint32_t d = ix->d, fu = cross->f_u, words = (ix->n_ads + 63) / 64;
  Ctrl hc;
  EBR_CUDA_TRY(cudaMemcpyAsync(&hc, w.ctrl.p, sizeof(Ctrl), cudaMemcpyDeviceToHost, st));
  EBR_CUDA_TRY(cudaStreamSynchronize(st));
  EBR_TRY(check_device_flags(hc.flags, "ebr_score_topk (batched)"));
  const uint32_t *h_status = reinterpret_cast<const uint32_t *>(w.host) + 3 * B;
  std::vector<uint32_t> nv, vbase;
  user_vals_layout(q, B, fu, &nv, &vbase);
  for (uint32_t b = 0; b < B; b++) {
    if (!h_status[b]) continue;
    ebr_query dq = q[b];
    dq.h_u = (const float *)w.users_f32.p + (size_t)user_row(b) * d;
    dq.user_vals = (const uint32_t *)w.user_vals.p + vbase[b];
    // the checked offsets staged for the batch (device memory)
    dq.user_ptr = q[b].user_ptr ? (const uint32_t *)w.user_ptr.p + (size_t)b * (fu + 1) : nullptr;
    dq.n_user_vals = nv[b];
    dq.filter = q[b].filter ? (const uint64_t *)w.filters.p + (size_t)b * words : nullptr;
    EBR_TRY(ws_prepare_one(ix, ix->n_keys, 8192));
    EBR_TRY(query_one(ix, cross, dq, d_ids + (size_t)b * kmax, d_scores + (size_t)b * kmax, kmax,
                      st));
    ix->fallbacks += 1;
    EBR_CUDA_TRY(cudaMemcpyAsync(&hc, ix->ws.ctrl.p, sizeof(Ctrl), cudaMemcpyDeviceToHost, st));
    EBR_CUDA_TRY(cudaStreamSynchronize(st));
    EBR_TRY(check_device_flags(hc.flags, "ebr_score_topk (single-request recompute)"));
  }
  return EBR_OK;
}

void batch_ws_free(BatchWs &w) {
  for (DevBuf *b : {&w.users_f32, &w.users_bf16, &w.users_scale, &w.user_vals, &w.user_ptr, &w.wT,
                    &w.filters, &w.small, &w.cand, &w.cand_n, &w.cand_thr, &w.uhist, &w.scratch, &w.res,
                    &w.ctrl, &w.req})
    dev_free(*b);
  if (w.host) cudaFreeHost(w.host);
  w.host = nullptr;
  w.host_bytes = 0;
  w.tmap_ready = false;
}

int query_batch(ebr_index *ix, const ebr_cross *cross, const ebr_query *q, uint32_t B,
                uint32_t *out_ids, float *out_scores, uint32_t kmax, int io, cudaStream_t st) {
  BatchWs &w = ix->bws;
  uint32_t *d_ids = out_ids;
  float *d_scores = out_scores;
  if (io == EBR_IO_HOST) {
    EBR_TRY(dev_reserve(w.res, (size_t)B * kmax * 8 + 256));
    d_ids = (uint32_t *)w.res.p;
    d_scores = (float *)((char *)w.res.p + (((size_t)B * kmax * 4 + 255) / 256 * 256));
  }
  EBR_TRY(batch_launch(ix, cross, q, B, d_ids, d_scores, kmax, io, w, st));
  EBR_TRY(batch_finish(ix, cross, q, B, d_ids, d_scores, kmax, w, st));
  if (io == EBR_IO_HOST) {
    EBR_CUDA_TRY(cudaMemcpyAsync(out_ids, d_ids, (size_t)B * kmax * 4, cudaMemcpyDeviceToHost, st));
    EBR_CUDA_TRY(
        cudaMemcpyAsync(out_scores, d_scores, (size_t)B * kmax * 4, cudaMemcpyDeviceToHost, st));
    EBR_CUDA_TRY(cudaStreamSynchronize(st));
  }
  return EBR_OK;
}

// =====================================================================
// Device-resident serving loop
// =====================================================================
// Wave descriptor (one ring slot, written by the host, copied to `cur` by
// the fetch kernel): [B, pad x3][kscan Bmax][kout Bmax][has_filter Bmax]
// [ReqSrc Bmax, 16-byte aligned].
static size_t desc_src_off(uint32_t Bmax) { return (16 + (size_t)12 * Bmax + 15) / 16 * 16; }
static size_t desc_bytes_for(uint32_t Bmax) {
  return (desc_src_off(Bmax) + (size_t)Bmax * sizeof(ReqSrc) + 15) / 16 * 16;
}

struct LoopArgs {
  LoopShared *sh;              // mapped host words
  const uint8_t *desc;         // mapped [R][desc_bytes]
  uint32_t *flags_out;         // mapped [R]
  uint32_t *status_out;        // mapped [R][Bmax]
  uint8_t *cur;                // device copy of the current descriptor
  uint32_t *slot;
  unsigned long long *seq, *idle_ns;
  Ctrl *ctrl;
  uint32_t *status;            // [R][Bmax]
  uint32_t R, Bmax, desc_bytes;
  unsigned long long poll_ns, idle_exit_ns;
  cudaGraphConditionalHandle handle;  // the WHILE node's
  cudaGraphConditionalHandle sw;      // the SWITCH node's: which user-table width runs
  uint32_t nsw, bq[3];                // widths (users) of the switch's cases, ascending
};

__device__ __forceinline__ unsigned long long ld_acquire_sys(const volatile unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_sys(volatile unsigned long long *p,
                                               unsigned long long v) {
  asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// First node of the loop body.  Thread 0 waits, for at most poll_ns, for a
// wave the host posted whose result slot the host has freed, or for stop.
// A wave: its descriptor is copied into `cur`, its control block and status
// zeroed, and the SWITCH node that follows is told which user-table width
// (the narrowest that holds the wave's users) to run.  No wave: cur.B = 0
// (every later node of this iteration returns at once), and after
// idle_exit_ns without a wave, or on stop, the loop's condition is cleared
// so that this iteration is the last.
__global__ void __launch_bounds__(256) k_loop_fetch(LoopArgs a) {
  __shared__ uint32_t s_state, s_slot;
  if (threadIdx.x == 0) {
    const unsigned long long seq = *a.seq;
    const uint64_t t0 = global_timer_ns();
    uint32_t st = 0;  // 0: no wave, 1: a wave, 2: leave the loop
    for (;;) {
      if (a.sh->stop) {
        st = 2;
        break;
      }
      const unsigned long long posted = ld_acquire_sys(&a.sh->posted);
      if (posted > seq && seq < a.sh->freed + a.R) {
        st = 1;
        break;
      }
      if (global_timer_ns() - t0 >= a.poll_ns) break;
      __nanosleep(1000);
    }
    if (st == 0) {
      *a.idle_ns += global_timer_ns() - t0;
      if (*a.idle_ns >= a.idle_exit_ns) st = 2;
    } else if (st == 1) {
      *a.idle_ns = 0;
    }
    if (st == 2) cudaGraphSetConditional(a.handle, 0u);
    if (st == 1) {  // the narrowest user table that holds the wave
      const uint32_t B = reinterpret_cast<const volatile uint32_t *>(
          a.desc + (size_t)(seq % a.R) * a.desc_bytes)[0];
      uint32_t c = 0;
      while (c + 1 < a.nsw && B > a.bq[c]) c++;
      cudaGraphSetConditional(a.sw, c);
    }
    s_state = st;
    s_slot = (uint32_t)(seq % a.R);
    *a.slot = s_slot;
  }
  __syncthreads();
  if (s_state != 1) {
    if (threadIdx.x == 0) *reinterpret_cast<uint32_t *>(a.cur) = 0u;
    return;
  }
  const volatile uint32_t *src =
      reinterpret_cast<const volatile uint32_t *>(a.desc + (size_t)s_slot * a.desc_bytes);
  uint32_t *dst = reinterpret_cast<uint32_t *>(a.cur);
  for (uint32_t i = threadIdx.x; i < a.desc_bytes / 4; i += blockDim.x) dst[i] = src[i];
  for (uint32_t i = threadIdx.x; i < sizeof(Ctrl) / 4; i += blockDim.x)
    reinterpret_cast<uint32_t *>(a.ctrl)[i] = 0u;
  for (uint32_t i = threadIdx.x; i < a.Bmax; i += blockDim.x) a.status[s_slot * a.Bmax + i] = 0u;
}

// Last node of the loop body: a wave's flags and per-user status go to the
// mapped result words, then (system-scope release) done = waves finished.
__global__ void k_loop_publish(LoopArgs a) {
  const uint32_t B = *reinterpret_cast<const uint32_t *>(a.cur);
  if (B == 0) return;
  const uint32_t slot = *a.slot;
  for (uint32_t b = threadIdx.x; b < B; b += blockDim.x)
    a.status_out[slot * a.Bmax + b] = a.status[slot * a.Bmax + b];
  __syncthreads();
  if (threadIdx.x == 0) {
    a.flags_out[slot] = a.ctrl->flags;
    __threadfence_system();
    const unsigned long long seq = *a.seq + 1;
    *a.seq = seq;
    st_release_sys(&a.sh->done, seq);
  }
}

static void loop_dev_sizes(uint32_t R, uint32_t Bmax, uint32_t kmax, size_t *cur_b, size_t *st_b,
                           size_t *out_b, size_t *ctl_b) {
  *cur_b = (desc_bytes_for(Bmax) + 255) / 256 * 256;
  *st_b = ((size_t)R * Bmax * 4 + 255) / 256 * 256;
  *out_b = ((size_t)R * Bmax * kmax * 4 + 255) / 256 * 256;
  *ctl_b = (256 + sizeof(Ctrl) + 255) / 256 * 256;
}

size_t loop_dev_bytes(uint32_t Bmax, uint32_t kmax) {
  size_t cur_b, st_b, out_b, ctl_b;
  loop_dev_sizes(LoopBufs{}.R, Bmax, kmax, &cur_b, &st_b, &out_b, &ctl_b);
  return cur_b + st_b + 2 * out_b + ctl_b;
}

int loop_alloc(LoopBufs &L, uint32_t Bmax, uint32_t kmax) {
  L.Bmax = Bmax;
  L.kmax = kmax;
  L.desc_bytes = (uint32_t)desc_bytes_for(Bmax);
  const size_t sh_b = 256, desc_b = (size_t)L.R * L.desc_bytes, fl_b = (size_t)L.R * 4;
  const size_t host_b = sh_b + desc_b + fl_b + (size_t)L.R * Bmax * 4;
  if (cudaHostAlloc(&L.host, host_b, cudaHostAllocMapped) != cudaSuccess) {
    cudaGetLastError();
    L.host = nullptr;
    set_error("serving loop: mapped host allocation of %zu bytes failed", host_b);
    return EBR_ENOMEM;
  }
  memset(L.host, 0, host_b);
  void *dp = nullptr;
  EBR_CUDA_TRY(cudaHostGetDevicePointer(&dp, L.host, 0));
  if (dp != L.host) {  // every pointer below is used on both sides
    set_error("serving loop: mapped host memory has a different device address");
    return EBR_EINVAL;
  }
  uint8_t *h = (uint8_t *)L.host;
  L.sh = (LoopShared *)h;
  L.desc = h + sh_b;
  L.flags_out = (uint32_t *)(h + sh_b + desc_b);
  L.status_out = (uint32_t *)(h + sh_b + desc_b + fl_b);
  size_t cur_b, st_b, out_b, ctl_b;
  loop_dev_sizes(L.R, Bmax, kmax, &cur_b, &st_b, &out_b, &ctl_b);
  EBR_TRY(dev_alloc(L.dev, cur_b + st_b + 2 * out_b + ctl_b));
  uint8_t *d = (uint8_t *)L.dev.p;
  L.cur = d;
  L.status = (uint32_t *)(d + cur_b);
  L.out_ids = (uint32_t *)(d + cur_b + st_b);
  L.out_scores = (float *)(d + cur_b + st_b + out_b);
  uint8_t *c = d + cur_b + st_b + 2 * out_b;
  L.slot = (uint32_t *)c;
  L.seq = (unsigned long long *)(c + 8);
  L.idle_ns = (unsigned long long *)(c + 16);
  L.ctrl = (Ctrl *)(c + 256);
  EBR_CUDA_TRY(cudaMemset(L.dev.p, 0, L.dev.bytes));
  return EBR_OK;
}

void loop_free(LoopBufs &L) {
  if (L.exec) cudaGraphExecDestroy(L.exec);
  L.exec = nullptr;
  dev_free(L.dev);
  if (L.host) cudaFreeHost(L.host);
  L.host = nullptr;
}

int loop_fill(LoopBufs &L, uint64_t wave, const ebr_index *ix, const ebr_cross *cross,
              const ebr_query *q, uint32_t B) {
  if (B == 0 || B > L.Bmax) {
    set_error("serving loop: a wave of %u users (at most %u)", B, L.Bmax);
    return EBR_EINVAL;
  }
  uint8_t *p = L.desc + (size_t)(wave % L.R) * L.desc_bytes;
  uint32_t *w32 = (uint32_t *)p;
  w32[0] = B;
  uint32_t *ks = (uint32_t *)(p + 16), *ko = ks + L.Bmax, *hf = ko + L.Bmax;
  ReqSrc *src = (ReqSrc *)(p + desc_src_off(L.Bmax));
  uint32_t base = 0;
  for (uint32_t b = 0; b < B; b++) {
    ks[b] = std::min<uint32_t>(q[b].k * ix->rescore_mult, ix->n_ads);
    ko[b] = q[b].k;
    hf[b] = q[b].filter ? 1u : 0u;
    const uint32_t n = q[b].user_ptr ? q[b].n_user_vals : cross->f_u;
    src[b] = ReqSrc{q[b].h_u, q[b].user_vals, q[b].filter, q[b].user_ptr, n, base};
    base += n;
  }
  return EBR_OK;
}

// Builds the loop graph for index ix: a WHILE node whose body is
//   fetch -> SWITCH { one case per user-table width 64, 128, 256 (up to the
//   server's batch): staging, quantiser, expansion, window scan, merge }
//   -> publish,
// so a wave of a few users runs on the narrowest table that holds it.  The
// batch plan (candidate buffers, shared memory) is the same for every width.
int loop_build(ebr_index *ix, const ebr_cross *cross, uint32_t max_user_vals, BatchWs &w,
               LoopBufs &L, cudaStream_t st) {
  if (L.exec) {
    cudaGraphExecDestroy(L.exec);
    L.exec = nullptr;
  }
  const uint32_t Bmax = L.Bmax, d = ix->d, fu = cross->f_u, words = (ix->n_ads + 63) / 64;
  const uint32_t kscan_max = std::min<uint32_t>(L.kmax * ix->rescore_mult, ix->n_ads);
  EBR_TRY(batch_ws_reserve(ix, cross, Bmax, kscan_max, (uint64_t)Bmax * max_user_vals, w));
  BatchSizes z;
  batch_sizes(ix, cross, Bmax, kscan_max, (uint64_t)Bmax * max_user_vals, &z);
  const BatchPlan pl = z.pl;
  const bool f8 = ix->dtype == EBR_FP8E4M3;
  uint8_t *cur = L.cur;
  const uint32_t *B_dev = (const uint32_t *)cur;
  const uint32_t *ks = (const uint32_t *)(cur + 16), *ko = ks + Bmax, *hf = ko + Bmax;
  const ReqSrc *srcs = (const ReqSrc *)(cur + desc_src_off(Bmax));
  uint32_t *d_uptr = (uint32_t *)w.user_ptr.p;
  uint32_t *d_base = d_uptr + (size_t)Bmax * (fu + 1);
  auto kern = window_kernel(f8, pl.mode);
  EBR_CUDA_TRY(allow_smem(kern, kBatchSmemBudget));
  const size_t msm = merge_smem(kscan_max, L.kmax);
  EBR_CUDA_TRY(allow_smem(k_batch_merge, merge_smem(8192, 8192)));
  LoopArgs la;
  memset(&la, 0, sizeof(la));
  la.nsw = 0;  // 64, 128, ... and, last, the table's own width
  for (uint32_t q = kGroup; q < pl.Bq; q <<= 1) la.bq[la.nsw++] = q;
  la.bq[la.nsw++] = pl.Bq;
  cudaGraph_t g = nullptr;
  EBR_CUDA_TRY(cudaGraphCreate(&g, 0));
  int rc = EBR_OK;
  const char *what = "conditional graph nodes";
  cudaError_t e = cudaGraphConditionalHandleCreate(&la.handle, g, 1u, cudaGraphCondAssignDefault);
  cudaGraphNodeParams wp = {}, sp = {};
  cudaGraphNode_t wnode, fnode, snode;
  if (e == cudaSuccess) {
    wp.type = cudaGraphNodeTypeConditional;
    wp.conditional.handle = la.handle;
    wp.conditional.type = cudaGraphCondTypeWhile;
    wp.conditional.size = 1;
    e = cudaGraphAddNode(&wnode, g, nullptr, nullptr, 0, &wp);
  }
  cudaGraph_t body = e == cudaSuccess ? wp.conditional.phGraph_out[0] : nullptr;
  if (e == cudaSuccess)
    e = cudaGraphConditionalHandleCreate(&la.sw, body, 0u, cudaGraphCondAssignDefault);
  la.sh = L.sh;
  la.desc = L.desc;
  la.flags_out = L.flags_out;
  la.status_out = L.status_out;
  la.cur = cur;
  la.slot = L.slot;
  la.seq = L.seq;
  la.idle_ns = L.idle_ns;
  la.ctrl = L.ctrl;
  la.status = L.status;
  la.R = L.R;
  la.Bmax = Bmax;
  la.desc_bytes = L.desc_bytes;
  la.poll_ns = L.poll_ns;
  la.idle_exit_ns = L.idle_exit_ns;
  // fetch
  if (e == cudaSuccess) {
    what = "capture of the fetch node";
    e = cudaStreamBeginCaptureToGraph(st, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
    if (e == cudaSuccess) {
      k_loop_fetch<<<1, 256, 0, st>>>(la);
      cudaGraph_t cap = nullptr;
      e = cudaStreamEndCapture(st, &cap);
    }
    size_t nn = 1;
    if (e == cudaSuccess) e = cudaGraphGetNodes(body, &fnode, &nn);
    if (e == cudaSuccess && nn != 1) e = cudaErrorInvalidValue;
  }
  // the switch and its cases
  if (e == cudaSuccess) {
    what = "switch node";
    sp.type = cudaGraphNodeTypeConditional;
    sp.conditional.handle = la.sw;
    sp.conditional.type = cudaGraphCondTypeSwitch;
    sp.conditional.size = la.nsw;
    e = cudaGraphAddNode(&snode, body, &fnode, nullptr, 1, &sp);
  }
  for (uint32_t c = 0; e == cudaSuccess && rc == EBR_OK && c < la.nsw; c++) {
    what = "capture of a wave";
    const uint32_t Bp = la.bq[c];
    const int grid = batch_grid(ix, Bp);
    BatchPlan pc;
    if (!plan_batch(ix, Bp, kscan_max, grid, &pc)) {
      rc = EBR_EINVAL;
      break;
    }
    BatchArgs ba;
    rc = fill_batch_args(ix, Bmax, pc, w, ks, hf, L.ctrl, B_dev, &ba);
    if (rc != EBR_OK) break;
    e = cudaStreamBeginCaptureToGraph(st, sp.conditional.phGraph_out[c], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) break;
    const uint32_t ys = (words + kStageWords - 1) / kStageWords;
    k_stage_requests<<<dim3(Bp, ys), 256, 0, st>>>(srcs, d, fu, words,
                                                   (float *)w.users_f32.p,
                                                   (uint32_t *)w.user_vals.p, d_uptr, d_base,
                                                   (uint64_t *)w.filters.p, &L.ctrl->flags, B_dev);
    if (f8)
      rc = launch_quantize_rows_fp8((const float *)w.users_f32.p, Bp, d,
                                    (uint8_t *)w.users_bf16.p, (float *)w.users_scale.p, st);
    else
      rc = launch_quantize((const float *)w.users_f32.p, (uint64_t)Bp * d, EBR_BF16,
                           w.users_bf16.p, st);
    if (rc == EBR_OK)
      rc = expand_transposed(cross, (const uint32_t *)w.user_vals.p, d_uptr, d_base,
                             std::min(Bmax, Bp), Bp, (float *)w.wT.p, &L.ctrl->flags,
                             ix->num_sms, st, B_dev, ix->key_id);
    if (rc == EBR_OK) e = clear_zero_rows(ix, w, Bp, st);
    if (rc == EBR_OK && e == cudaSuccess) e = cudaMemsetAsync(w.uhist.p, 0, user_hist_bytes(Bmax), st);
    if (rc == EBR_OK && e == cudaSuccess) {
      kern<<<dim3(grid, Bp / kGroup), batch_threads(pl.mode), pl.smem, st>>>(ba);
      k_batch_merge<<<std::min(Bmax, Bp), kMergeThreads, msm, st>>>(
          (const CandEntry *)w.cand.p, (const uint32_t *)w.cand_n.p,
          (const unsigned long long *)w.cand_thr.p, (uint32_t)grid, Bmax, pc.cap_u, ks, ko,
          L.kmax, (const float *)ix->emb_f32.p, d, (const float *)w.users_f32.p,
          (uint64_t *)w.scratch.p, L.out_ids, L.out_scores, L.status, B_dev, L.slot,
          (uint64_t)Bmax * L.kmax, Bmax);
    }
    cudaGraph_t cap = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(st, &cap);
    if (e == cudaSuccess) e = e2;
  }
  // publish, after the switch
  if (e == cudaSuccess && rc == EBR_OK) {
    what = "capture of the publish node";
    e = cudaStreamBeginCaptureToGraph(st, body, &snode, nullptr, 1, cudaStreamCaptureModeRelaxed);
    if (e == cudaSuccess) {
      k_loop_publish<<<1, 256, 0, st>>>(la);
      cudaGraph_t cap = nullptr;
      e = cudaStreamEndCapture(st, &cap);
    }
  }
  if (e == cudaSuccess && rc == EBR_OK) {
    what = "graph instantiation";
    e = cudaGraphInstantiate(&L.exec, g, 0);
  }
  cudaGraphDestroy(g);
  if (rc != EBR_OK) return rc;
  if (e != cudaSuccess) {
    L.exec = nullptr;
    cudaGetLastError();
    set_error("serving loop: %s: %s", what, cudaGetErrorString(e));
    return EBR_ECUDA;
  }
  return EBR_OK;
}

}  // namespace ebr
