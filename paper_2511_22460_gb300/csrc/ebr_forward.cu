// Streaming scan over the forward key table: one request against every ad.
//
// The forward table (built with the index, ebr_index.cu) holds, for every run
// of 32 consecutive ads, the ads' keys row by row: row r is the r-th key (in
// the order of the window-major view) of each of the 32 ads, four rows to a
// quad, short ads padded with the key n_keys whose term is zero.  It is the same binary
// feature->ad matrix L as the compressed lists of Algorithm 1 (Sec. 3.4),
// transposed.  With it a warp evaluates the wide term of the HitMatch equation
// (Sec. 3.3) for its 32 ads in registers, one ad per lane: two or three
// shared-memory reads give a lane four keys, four gathers their packed
// fixed-point terms (pack_term), and integer additions the class sums.  No
// block is decoded, nothing is added in shared memory and no warp waits for
// another one's part, which is what bounded the block-wise decode
// (k_fused_window, ebr_fused.cu: 10.2 k warp instructions per 256 ads of 16
// keys, 5.1 k here, waits included).  The integer sums are the block-wise scan's
// bits, and so are the whole scores of FP32 rows (their additions are in its
// order, but for the TREE form); BF16 and FP8 rows are summed on the tensor
// pipe, no further off than by its FP32 multiply-adds (kChain).
//
// One persistent CTA per SM over a contiguous range of ads:
//   producer (1 warp): stages of 32 to 256 ads -- their embedding rows and
//       their runs' keys, two bulk copies (cp.async.bulk, L2 evict-first);
//   consumers (8 to 22 warps): one run of 32 ads at a time: its keys into
//       registers, its inner products (FP32: a thread per row, two for
//       128-element rows, h_u permuted in registers so that neighbouring rows
//       read other banks; BF16 and FP8: mma.sync with h_u in three 16-bit
//       pieces), the stage handed back, then the terms; candidates go
//       to a per-CTA buffer, which the warps meet to trim (radix select) only
//       when it fills;
//   threshold (1 warp): adds the CTA's candidate counts to the histogram all
//       CTAs share and raises the CTA's running threshold from it.
// The table names keys by popularity rank, and the terms of the first 8 k ranks
// (0.90 of the gathers of the 2M-ad inventory) are copied to shared memory:
// gathers of hot terms from global memory all went to the same few L2 slices
// (ncu, 2M ads: the busiest slice at 82 % of its tag rate, the average at 38 %;
// 39 and 30 % now), and a shared-memory gather of 32 random words takes about
// four cycles.
// What bounds it: 2M FP32 ads (512 MB of rows, 97 MB of keys) the stream, 111 us
// = 5.5 TB/s (the block-wise scan: 152 us); 10M FP8 ads with 32 keys each (1.32
// GB) instruction issue, 72 % of the slots, 298 us (block-wise: 814 us).
// Every wait is bounded (2 s).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ebr_device.cuh"
#include "ebr_internal.cuh"

namespace ebr {

namespace {

// Consumer warps, and the quads of a run whose keys are read into registers at
// once.  FP32 rows of 64 and 128 elements keep 64 registers of h_u per thread
// (narrower ones d of them; they have the same eight warps, not tuned apart), BF16
// and FP8 rows (on mma.sync) 8 or 16.  Measured scans: 2M FP32 ads (d = 64, 16 keys) 8 warps 111
// us, 10 warps 113-134 us, 14 warps 183 us (they spill); 1M BF16 ads (d = 128,
// 24 keys) 14 warps keeping 8 quads 70 us, 18 keeping 4 77 us; 10M FP8 ads (d =
// 64, 32 keys) 22 warps 302 us, 18 313 us, 14 345 us.
template <typename Elt>
constexpr int cons_warps() {
  return std::is_same<Elt, float>::value ? 8 : (std::is_same<Elt, Fp8Tag>::value ? 22 : 14);
}
template <typename Elt>
constexpr int keep_quads() {
  return std::is_same<Elt, Bf16Tag>::value ? 8 : 4;
}
constexpr int kMaxConsWarps = 22;
constexpr int kFwdMaxStages = 24;
// Candidate buffer: a trim is asked for at trim_at entries; every warp may
// still append one run (32) before it sees that.
constexpr uint32_t kTrimSlack = 3072;

struct FwdArgs {
  const void *emb;
  const float *scale;        // FP8 row scales, or null
  const float *h_u;
  const uint32_t *wq;        // [n_keys + 1] packed terms by key id, the last one 0
  const uint8_t *fwd;        // forward table; null: the wide term is wide_in or absent
  const uint32_t *fwd_off;   // [n_runs + 1] first quad of each run
  const uint32_t *filter;    // targeting bitmap as 32-bit words (one per run), or null
  uint32_t n_ads, n_stages;  // stages of stage_ads ads in the whole inventory
  uint32_t workers;          // consumer warps that take runs (at most stages * runs per stage)
  uint32_t k, cap, trim_at, stages, lg_runs, stage_ads, stage_bytes, emb_bytes;
  uint32_t quad_bytes;       // 256 (16-bit keys) or 384 (24-bit keys)
  uint32_t smem_terms;       // first entries of wq, copied to shared memory
  uint64_t *cand_out;
  uint64_t *cand_g;          // if set: the CTAs' candidate buffers, else they are in shared memory
  Ctrl *ctrl;
  float *all_out;            // if set: every score is written here and nothing selected
  uint32_t direct;           // every ad's key to cand_out[ad] (0: filtered out)
  float *wide_out;           // if set: the per-ad wide term is written here
  uint32_t *hist;            // [kCandBins + 1] candidate-score histogram + top bin
  const int *fx_word;        // F of the packed terms
  const float *wide_in;      // if set: the wide term, already summed
  const uint32_t *route;     // if set: *route != 0 ignores wide_in and uses the table after all
  int cls_shift;
};

template <typename Elt, int D>
struct FwdShape {
  static constexpr int kRowBytes = D * EltTraits<Elt>::kBytes;
  static constexpr int kTPR = D > 64 ? D / 64 : 1;   // threads per row
  static constexpr int kCPT = kRowBytes / 16 / kTPR;  // 16-byte chunks per thread
  static constexpr int kRowsPer128 = kRowBytes >= 128 ? 1 : 128 / kRowBytes;
  static constexpr int kHPT = kCPT * EltTraits<Elt>::kVec;
  static_assert(kTPR <= 2 && (kCPT & (kCPT - 1)) == 0 && kHPT <= 64, "row split");
  // mma.sync form (BF16, FP8): steps of four 16-byte chunks per row
  static constexpr int kChunks = kRowBytes / 16;
  static constexpr int kSteps = kChunks >= 4 ? kChunks / 4 : 1;
  static constexpr int kMmas = EltTraits<Elt>::kVec / 4;  // per step: 16 elements of k each
  // Products summed in one accumulator before FP32 additions take over: the tensor
  // pipe drops what lies below the largest of its addends.  Rms error in 2^-24 of the
  // sum of the products' sizes, 200k ads, normal user vectors and (second) ones that
  // fall off to 1e-5 from the first element to the last: BF16 d = 128 all eight
  // 0.30, 1.47, four 0.20, 0.70, two 0.16, 0.43, FP32 multiply-adds 0.26, 0.63; d = 16 both
  // 0.29, 1.04, one 0.28, 0.74, multiply-adds 0.40, 0.78; FP8 d = 64 all four 0.23, 1.09,
  // two 0.20, 0.67, multiply-adds 0.36, 0.86.  One at a time throughout costs 1 % of a
  // request on 10M FP8 ads (354 -> 358 us), two nothing.
  static constexpr int kChain = kSteps * kMmas > 2 ? 2 : 1;
};

// The inner products of BF16 and FP8 rows on the tensor pipe: 16 rows x 16
// elements per mma.sync, FP32 accumulators.  h_u is split into 16-bit pieces,
// one to a column: three BF16 pieces of 8 bits each for BF16 rows (exact for
// |h_u| of 2^-109 and more, below which the last one loses bits); for FP8 rows,
// whose elements are FP16 values, FP16 pieces of 11 bits, h_u scaled by a power of two
// so that its largest element is near 1 and piece n by 2^11n.  Three of those hold
// 24 bits of an element down to 2^-22 of the largest (an element of 2^-32 of it
// would keep 15, of 2^-40 seven); the other five columns, which the instruction
// multiplies anyway, carry it on to 2^-77.  Every product is exact
// in FP32, and their sum is no further off than the one of FP32 multiply-adds
// (kChain).
// A thread's 16-byte chunk supplies the elements of its own k positions (the
// order of the sum over k is free), so rows are read as they lie.
__device__ __forceinline__ void mma_16816(float *d, uint32_t a0, uint32_t a1, uint32_t a2,
                                          uint32_t a3, uint32_t b0, uint32_t b1, bool f16) {
  if (f16)
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 16 bits of piece n of h (BF16: 0, 1, 2, else 0).  A value that is not finite
// is its own first piece.
__device__ __forceinline__ uint32_t piece_bf16(float h, int n) {
  float r = h;
  uint32_t bits = 0;
  for (int i = 0; i < 3; i++) {
    const float x = __uint_as_float(__float_as_uint(r) & 0xFFFF0000u);  // towards zero: 8 bits
    if (i == n) bits = __float_as_uint(x) >> 16;
    r = fabsf(h) < INFINITY ? r - x : 0.f;
  }
  return bits;
}
template <int PIECES>
__device__ __forceinline__ uint32_t piece_f16(float h, int n) {
  float r = h;
  uint32_t bits = 0;
#pragma unroll
  for (int i = 0; i < PIECES; i++) {
    const __half x = __float2half_rn(r);
    if (i == n) bits = (uint32_t)__half_as_ushort(x);
    r = fabsf(h) < INFINITY ? (r - __half2float(x)) * 2048.f : 0.f;
  }
  return bits;
}
__device__ __forceinline__ uint32_t e4m3x2_f16x2(uint32_t w, bool high) {
  uint32_t r;
  if (high)
    asm("{\n .reg .b16 lo, hi;\n mov.b32 {lo, hi}, %1;\n cvt.rn.f16x2.e4m3x2 %0, hi;\n}"
        : "=r"(r) : "r"(w));
  else
    asm("{\n .reg .b16 lo, hi;\n mov.b32 {lo, hi}, %1;\n cvt.rn.f16x2.e4m3x2 %0, lo;\n}"
        : "=r"(r) : "r"(w));
  return r;
}

struct FwdSmem {
  uint64_t full[kFwdMaxStages], empty[kFwdMaxStages], terms;
  uint32_t chist[kCandBins];
  uint32_t hist[256], misc[8], wtot[2][kMaxConsWarps];
  unsigned long long thr;
  uint32_t n, n_seen, abort, stop, top_bin;
  uint32_t above;   // candidates of the CTA at or above the last bound
  uint32_t issued;  // stages whose copies the producer has issued
  uint32_t trim, meet, finished;  // trim asked for; what a meeting of the warps is for; all done
};

__device__ __forceinline__ uint2 lds_v2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_1(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

// Class sums of one ad's terms (see pack_term): all = classes 0 and 1
// together (modulo 2^32), c1, c2 and the FP32 remainder.
struct TermSum {
  int all = 0, c1 = 0, c2 = 0;
  float fp = 0.f;
  __device__ __forceinline__ void add4(uint32_t p0, uint32_t p1, uint32_t p2, uint32_t p3) {
    const uint32_t p[4] = {p0, p1, p2, p3};
    if (((p0 | p1 | p2 | p3) & 2u) == 0u) {  // classes 0 and 1 only: nearly always
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const int t = (int)p[i] >> 2;
        all += t;
        c1 += (int)(p[i] & 1u) * t;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const int t = (int)p[i] >> 2;
        const uint32_t c = p[i] & 3u;
        if (c < 2u) all += t;
        if (c == 1u) c1 += t;
        if (c == 2u) c2 += t;
        if (c == 3u) fp += __uint_as_float(p[i] & ~3u);
      }
    }
  }
};

// Wait for stage j, which is in ring slot s = j % S on turn j / S.  A warp may
// get here while the turn before is still being read, where a barrier's parity
// alone would pass for this turn's: it waits for the producer's count to say
// that stage j is issued.  From then on the full barrier's parity is not ambiguous
// (the next turn is not issued before this warp hands the slot back).  While
// the stage is not issued, warps that are to read the slot's turn before may
// have gone to a meeting (sm.trim), which this warp then has to join.
enum { kStageFail = 0, kStageReady = 1, kStageMeet = 2 };
__device__ __forceinline__ uint32_t wait_stage(FwdSmem &sm, uint32_t s, uint32_t turn, uint32_t j) {
  if (*((volatile uint32_t *)&sm.issued) <= j) {
    const uint64_t t0 = global_timer_ns();
    do {
      if (*((volatile uint32_t *)&sm.trim)) return kStageMeet;
      if (*((volatile uint32_t *)&sm.abort) || global_timer_ns() - t0 > kWaitTimeoutNs)
        return kStageFail;
      __nanosleep(32);
    } while (*((volatile uint32_t *)&sm.issued) <= j);
  }
  __threadfence_block();
  return mbar_wait_bounded(&sm.full[s], turn & 1u, kWaitTimeoutNs) ? kStageReady : kStageFail;
}

// Sum over the chunks congruent to I modulo S: pairs S apart ... first, so
// S = 1 is the order of a butterfly reduction over one lane per chunk.
template <int I, int S, int N, typename F>
__device__ __forceinline__ float tree_sum(F leaf) {
  if constexpr (S == N)
    return leaf(I);
  else
    return tree_sum<I, 2 * S, N>(leaf) + tree_sum<I + S, 2 * S, N>(leaf);
}

// TREE (FP32 only): the additions of the inner product in the order of the
// allocation-free scan, a chain of four multiply-adds per chunk and a tree over
// the chunks.  (The chunks are visited in the order i ^ rot here too: an XOR
// only swaps the sides of the tree's additions.)
// ALL: every term is in shared memory; else those with id < hot are.
template <typename Elt, int D, bool ALL, bool TREE>
__global__ void __launch_bounds__((cons_warps<Elt>() + 2) * 32, 1)
    k_forward(const __grid_constant__ FwdArgs a) {
  constexpr int kConsWarps = cons_warps<Elt>(), kConsThreads = kConsWarps * 32;
  constexpr int kKeep = keep_quads<Elt>();
  constexpr int kThrWarp = kConsWarps, kProdWarp = kConsWarps + 1;
  constexpr int kFwdThreads = (kProdWarp + 1) * 32;
  constexpr bool kMma = !std::is_same<Elt, float>::value;
  constexpr bool kF8 = std::is_same<Elt, Fp8Tag>::value;
  using Sh = FwdShape<Elt, D>;
  using Tr = EltTraits<Elt>;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ FwdSmem sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t S = a.stages, runs = 1u << a.lg_runs;
  uint32_t *s_terms = reinterpret_cast<uint32_t *>(smem + (size_t)S * a.stage_bytes);
  float *s_h = reinterpret_cast<float *>(s_terms + (a.smem_terms + 3) / 4 * 4);
  uint64_t *cand = a.cand_g ? a.cand_g + (size_t)blockIdx.x * a.cap
                            : reinterpret_cast<uint64_t *>(s_h + (D + 3) / 4 * 4);
  const uint32_t st0 = (uint32_t)(((uint64_t)a.n_stages * blockIdx.x) / gridDim.x);
  const uint32_t my_stages =
      (uint32_t)(((uint64_t)a.n_stages * (blockIdx.x + 1)) / gridDim.x) - st0;

  pdl_trigger();  // the final selection may be scheduled behind this grid
  for (int i = tid; i < D; i += kFwdThreads) s_h[i] = a.h_u[i];
  for (int i = tid; i < kCandBins; i += kFwdThreads) sm.chist[i] = 0;
  if (tid == 0) {
    sm.n = 0;
    sm.abort = 0;
    sm.issued = 0;
    sm.thr = 0ull;
    sm.top_bin = 0;
    sm.trim = 0;
    sm.finished = 0;
    mbar_init(&sm.terms, 1);
    for (uint32_t q = 0; q < S; q++) {
      mbar_init(&sm.full[q], 1);
      mbar_init(&sm.empty[q], runs);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == kProdWarp) {
    // ------------------------------------------------------------ producer
    // The lanes read the runs' offsets of 32 stages at a time; lane 0 issues.
    bool keys = a.fwd != nullptr;
    if (a.route) {  // the device decides whether the keys are needed at all
      pdl_wait();
      keys = keys && *a.route != 0u;
    } else if (a.wide_in) {
      keys = false;
    }
    const uint64_t pol = l2_evict_first_policy();
    uint32_t seq = 0;
    bool stop = false;
    for (uint32_t j0 = 0; j0 < my_stages && !stop; j0 += 32) {
      uint32_t q_lo = 0, q_hi = 0;  // quads of stage j0 + lane
      if (keys && j0 + lane < my_stages) {
        const uint32_t r = (st0 + j0 + lane) * runs;
        q_lo = __ldg(a.fwd_off + r);
        q_hi = __ldg(a.fwd_off + r + runs);
      }
      for (uint32_t i = 0; i < 32 && j0 + i < my_stages; i++) {
        const uint32_t k0 = __shfl_sync(0xffffffffu, q_lo, i);
        const uint32_t k1 = __shfl_sync(0xffffffffu, q_hi, i);
        if (lane == 0) {
          const uint32_t s = seq % S;
          if (seq >= S && !mbar_wait_bounded(&sm.empty[s], ((seq / S) - 1) & 1u, kWaitTimeoutNs)) {
            atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
            sm.abort = 1;
          }
          stop = *((volatile uint32_t *)&sm.abort) != 0u;
          if (!stop) {
            const uint32_t row0 = (st0 + seq) * a.stage_ads;
            const uint32_t rows = row0 < a.n_ads ? min(a.stage_ads, a.n_ads - row0) : 0u;
            const uint32_t eb = rows * Sh::kRowBytes, kb = (k1 - k0) * a.quad_bytes;
            uint8_t *dst = smem + (size_t)s * a.stage_bytes;
            mbar_arrive_expect_tx(&sm.full[s], eb + kb);
            if (eb)
              bulk_g2s_hint(dst,
                            reinterpret_cast<const uint8_t *>(a.emb) + (uint64_t)row0 * Sh::kRowBytes,
                            eb, &sm.full[s], pol);
            if (kb)
              bulk_g2s_hint(dst + a.emb_bytes, a.fwd + (uint64_t)k0 * a.quad_bytes, kb,
                            &sm.full[s], pol);
            __threadfence_block();
            *((volatile uint32_t *)&sm.issued) = seq + 1;
          }
        }
        stop = __shfl_sync(0xffffffffu, (int)stop, 0) != 0;
        if (stop) break;
        seq++;
      }
    }
    if (stop && lane == 0)  // stopped early: wait (bounded) for the copies still in flight
      for (uint32_t q = (seq > S ? seq - S : 0); q < seq; q++)
        mbar_wait_bounded(&sm.full[q % S], (q / S) & 1u, kWaitTimeoutNs / 4);
    return;
  }

  if (warp == kThrWarp) {
    // ----------------------------------------------------------- threshold
    if (a.all_out || a.direct) return;
    pdl_wait();  // the histogram and the control block are zeroed before this kernel
    while (!*((volatile uint32_t *)&sm.finished) && !*((volatile uint32_t *)&sm.abort)) {
      // counts below the known bound cannot raise it
      const uint32_t b0 =
          (uint32_t)(*((volatile unsigned long long *)&sm.thr) >> kBinShift);
      const uint32_t top = *((volatile uint32_t *)&sm.top_bin);
      for (uint32_t i = b0 + lane; i <= top; i += 32)
        if (*((volatile uint32_t *)&sm.chist[i]))
          atomicAdd(a.hist + i, atomicExch(&sm.chist[i], 0u));
      if (lane == 0 && top) atomicMax(a.hist + kCandBins, top);
      const unsigned long long h = hist_top_threshold(a.hist, b0, a.k);
      if (lane == 0) {
        const unsigned long long g = *((volatile unsigned long long *)&a.ctrl->thr);
        if (max(g, h) > *((volatile unsigned long long *)&sm.thr)) atomicMax(&sm.thr, max(g, h));
      }
      __syncwarp();
      __nanosleep(500);
    }
    return;
  }

  // -------------------------------------------------------------- consumers
  const GroupSync gsync{1, kConsThreads};
  // FP32: this thread's row part and its permuted copy of h_u
  const int qd = lane % Sh::kTPR;
  const uint32_t rot = (lane / Sh::kRowsPer128) % Sh::kCPT;
  float hreg[kMma ? 1 : Sh::kHPT];
  // BF16, FP8: this thread's part of the columns of pieces (column
  // lane / 4, chunk 4 step + lane % 4), and the weights of columns 2 (lane % 4)
  // and 2 (lane % 4) + 1
  uint32_t breg[kMma ? Sh::kSteps * Sh::kMmas * 2 : 1];
  float cw0 = 0.f, cw1 = 0.f;
  if constexpr (!kMma) {
#pragma unroll
    for (int i = 0; i < Sh::kCPT; i++) {
      const uint32_t c = TREE ? (i ^ rot) * Sh::kTPR + qd : qd * Sh::kCPT + (i ^ rot);
#pragma unroll
      for (int e = 0; e < Tr::kVec; e++) hreg[i * Tr::kVec + e] = s_h[c * Tr::kVec + e];
    }
  } else {
    float sc = 1.f, inv = 1.f;
    bool spread = false;  // elements that three FP16 pieces do not hold
    if (kF8) {  // the largest finite |h_u| to [1, 4); both powers of two are normal numbers
      float mx = 0.f, mn = INFINITY;
      for (int i = lane; i < D; i += 32) {
        const float x = fabsf(s_h[i]);
        mx = fmaxf(mx, x < INFINITY ? x : 0.f);
        mn = fminf(mn, x > 0.f ? x : INFINITY);
      }
      for (int o = 16; o; o >>= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      }
      const int e = mx > 0.f ? max(-126, min(126, (int)(__float_as_uint(mx) >> 23) - 127)) : 0;
      sc = pow2f(-e);
      inv = pow2f(e);
      spread = mn * sc < pow2f(-22);
    }
    const int t = lane & 3, n = lane >> 2;
    // FP8: column n weighs inv x 2^-11n, down to 0 where a piece has nothing left
    cw0 = kF8 ? inv : (t < 2 ? 1.f : 0.f);
    for (int i = 0; kF8 && i < 2 * t; i++) cw0 *= pow2f(-11);
    cw1 = kF8 ? cw0 * pow2f(-11) : (t == 0 ? 1.f : 0.f);
    auto split = [&](auto pieces) {
      constexpr int P = decltype(pieces)::value;
#pragma unroll
      for (int j = 0; j < Sh::kSteps; j++)
#pragma unroll
        for (int i = 0; i < Sh::kMmas * 2; i++) {
          const int c = 4 * j + t;
          uint32_t w = 0;
          if (c < Sh::kChunks) {
            const float x = s_h[c * Tr::kVec + 2 * i] * sc, y = s_h[c * Tr::kVec + 2 * i + 1] * sc;
            w = kF8 ? piece_f16<P>(x, n) | (piece_f16<P>(y, n) << 16)
                    : piece_bf16(x, n) | (piece_bf16(y, n) << 16);
          }
          breg[j * Sh::kMmas * 2 + i] = w;
        }
    };
    // (all eight for every vector: 827k FP8 ads of 128 elements 72.2 -> 75.8 us)
    if (kF8 && spread)
      split(std::integral_constant<int, 8>());
    else
      split(std::integral_constant<int, 3>());
  }
  pdl_wait();  // the packed terms, their exponent and the route are visible from here on
  const bool pre = a.wide_in != nullptr && !(a.route && *a.route);
  const bool keys = a.fwd != nullptr && !pre;
  const bool hi24 = a.quad_bytes > 256u;
  if (keys && a.smem_terms) {  // one bulk copy (a multiple of 16 bytes; both ends aligned)
    if (tid == 0) {
      const uint32_t bytes = (a.smem_terms + 3) / 4 * 16;
      mbar_arrive_expect_tx(&sm.terms, bytes);
      bulk_g2s(s_terms, a.wq, bytes, &sm.terms);
      if (!mbar_wait_bounded(&sm.terms, 0, kWaitTimeoutNs)) {
        atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
        sm.abort = 1;
      }
    }
    gsync();
    mbar_try_wait(&sm.terms, 0);  // per-thread acquire
  }
  const uint32_t s_terms_a = smem_u32(s_terms);
  const int fx_e = keys ? *a.fx_word : 0;
  const float u0 = pow2f(-fx_e), u1 = pow2f(-fx_e - a.cls_shift),
              u2 = pow2f(-fx_e - 2 * a.cls_shift);
  const uint32_t hot = a.smem_terms;
  auto term = [&](uint32_t id) -> uint32_t {
    if (ALL) return lds_1(s_terms_a + 4u * id);
    // No branch: lanes read their term from one place or the other.  (Not .nc:
    // the kernel before writes wq while this one already runs, and that path is
    // for memory that nothing writes as long as the kernel lives.)
    uint32_t v;
    asm volatile(
        "{\n .reg .pred p;\n setp.lt.u32 p, %1, %2;\n @p ld.shared.u32 %0, [%3];\n"
        " @!p ld.global.u32 %0, [%4];\n}"
        : "=r"(v)
        : "r"(id), "r"(hot), "r"(s_terms_a + 4u * id), "l"(a.wq + id));
    return v;
  };
  // this lane's four keys of the quad at ka: 16 low bits each, then 8 high bits each
  struct Quad {
    uint2 lo;
    uint32_t hi;
  };
  auto load_quad = [&](uint32_t ka) {
    Quad q;
    q.lo = lds_v2(ka + lane * 8u);
    q.hi = hi24 ? lds_1(ka + 256u + lane * 4u) : 0u;
    return q;
  };
  auto quad_terms = [&](const Quad &q, uint32_t *p) {
    const uint32_t ha = q.hi & 0x00FF00FFu, hb = (q.hi >> 8) & 0x00FF00FFu;
    p[0] = term(__byte_perm(q.lo.x, ha, 0x5410));
    p[1] = term(__byte_perm(q.lo.x, hb, 0x5432));
    p[2] = term(__byte_perm(q.lo.y, ha, 0x7610));
    p[3] = term(__byte_perm(q.lo.y, hb, 0x7632));
  };

  // A run's side inputs, loaded a run ahead: their latency would otherwise
  // hold the run's stage.
  struct Side {
    uint32_t o0, o1, os, fword;
    float wide, scale;
  };
  const uint32_t slots = my_stages << a.lg_runs;
  auto load_side = [&](uint32_t u) {
    Side d{0u, 0u, 0u, 0xFFFFFFFFu, 0.f, 1.f};
    const uint32_t run = (st0 << a.lg_runs) + u;
    const uint32_t ad = run * 32u + lane;
    if (u < slots) {
      if (keys) {
        d.os = __ldg(a.fwd_off + (run & ~(runs - 1u)));
        d.o0 = __ldg(a.fwd_off + run);
        d.o1 = __ldg(a.fwd_off + run + 1);
      }
      if (ad < a.n_ads) {
        if (pre) d.wide = __ldcg(a.wide_in + ad);  // (the kernel before's; see term)
        if (a.scale) d.scale = __ldg(a.scale + ad);
        if (a.filter) d.fword = __ldg(a.filter + run);
      }
    }
    return d;
  };
  uint32_t u = warp < (int)a.workers ? warp : slots;  // this warp's run within the CTA's range
  Side next = load_side(u);
  for (;;) {
    // (one lane's view of the flag: the whole warp goes on or stops)
    while (u < slots && !__shfl_sync(0xffffffffu, *((volatile uint32_t *)&sm.trim), 0)) {
      const uint32_t j = u >> a.lg_runs, rs = u & (runs - 1u);
      const uint32_t s = j % S, turn = j / S;
      // (FP32: before the wait, 118 -> 114 us for 1M ads of 128 elements; the others
      // have no registers to hold it meanwhile, a request on 10M FP8 ads 384 against 359 us)
      Side ahead;
      if (!kMma) ahead = load_side(u + a.workers);
      uint32_t staged = kStageFail;
      if (lane == 0 && !*((volatile uint32_t *)&sm.abort)) staged = wait_stage(sm, s, turn, j);
      staged = __shfl_sync(0xffffffffu, staged, 0);
      if (staged == kStageMeet) break;
      if (staged == kStageFail) {
        if (lane == 0 && !*((volatile uint32_t *)&sm.abort)) {
          atomicOr(&a.ctrl->flags, DEVERR_TIMEOUT);
          sm.abort = 1;
        }
        u = slots;
        break;
      }
      const Side sd = next;
      next = kMma ? load_side(u + a.workers) : ahead;
      const uint32_t run = (st0 << a.lg_runs) + u;
      const uint32_t ad = run * 32u + lane;
      u += a.workers;
      const bool in = ad < a.n_ads;
      mbar_try_wait(&sm.full[s], turn & 1u);  // per-thread acquire
      const uint8_t *stage = smem + (size_t)s * a.stage_bytes;
      const uint32_t ka = smem_u32(stage) + a.emb_bytes + (sd.o0 - sd.os) * a.quad_bytes;
      const uint32_t nq = sd.o1 - sd.o0;
      // the keys of the first kKeep quads, kept in registers
      Quad kq[kKeep];
#pragma unroll
      for (int q = 0; q < kKeep; q++)
        if (q < nq) kq[q] = load_quad(ka + q * a.quad_bytes);
      float dot = 0.f;
      if constexpr (kMma) {
        float d[2][4];
        const int t = lane & 3, g = lane >> 2;
#pragma unroll
        for (int m = 0; m < 2; m++) {
          const uint8_t *row = stage + (size_t)(rs * 32u + 16 * m + g) * Sh::kRowBytes;
          float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int j = 0; j < Sh::kSteps; j++) {
            uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
            if (4 * j + t < Sh::kChunks) {
              lo = *reinterpret_cast<const uint4 *>(row + (4 * j + t) * 16);
              hi = *reinterpret_cast<const uint4 *>(row + 8 * Sh::kRowBytes + (4 * j + t) * 16);
            }
            const uint32_t l[4] = {lo.x, lo.y, lo.z, lo.w}, h[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
            for (int i = 0; i < Sh::kMmas; i++) {
              const uint32_t *bb = breg + (j * Sh::kMmas + i) * 2;
              if (kF8)
                mma_16816(part, e4m3x2_f16x2(l[i], false), e4m3x2_f16x2(h[i], false),
                          e4m3x2_f16x2(l[i], true), e4m3x2_f16x2(h[i], true), bb[0], bb[1], true);
              else
                mma_16816(part, l[2 * i], h[2 * i], l[2 * i + 1], h[2 * i + 1], bb[0], bb[1], false);
              const int done = j * Sh::kMmas + i + 1;
              if (done % Sh::kChain == 0 || done == Sh::kSteps * Sh::kMmas) {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                  d[m][q] = done <= Sh::kChain ? part[q] : d[m][q] + part[q];
                  part[q] = 0.f;
                }
              }
            }
          }
        }
        // rows g, 8 + g, 16 + g, 24 + g: this thread's two columns weighted,
        // then summed over the quad so that thread t holds row 8 t + g
        float y[4] = {d[0][0] * cw0 + d[0][1] * cw1, d[0][2] * cw0 + d[0][3] * cw1,
                      d[1][0] * cw0 + d[1][1] * cw1, d[1][2] * cw0 + d[1][3] * cw1};
        const bool up = t >= 2, odd = t & 1;
        const float r0 = __shfl_xor_sync(0xffffffffu, up ? y[0] : y[2], 2);
        const float r1 = __shfl_xor_sync(0xffffffffu, up ? y[1] : y[3], 2);
        const float z0 = (up ? y[2] : y[0]) + r0, z1 = (up ? y[3] : y[1]) + r1;
        const float z = (odd ? z1 : z0) + __shfl_xor_sync(0xffffffffu, odd ? z0 : z1, 1);
        dot = __shfl_sync(0xffffffffu, z, 4 * (lane & 7) + (lane >> 3));
      } else {
        // with two threads per row, rows 16 ps .. 16 ps + 15
#pragma unroll
        for (int ps = 0; ps < Sh::kTPR; ps++) {
          const uint32_t rw = Sh::kTPR == 1 ? lane : 16 * ps + lane / 2;
          const uint8_t *row = stage + (size_t)(rs * 32u + rw) * Sh::kRowBytes;
          float2 d2 = make_float2(0.f, 0.f);
          if (TREE) {
            d2.x = tree_sum<0, 1, Sh::kCPT>([&](int i) {
              const float4 f = *reinterpret_cast<const float4 *>(
                  row + ((i ^ rot) * Sh::kTPR + qd) * 16);
              return fmaf(hreg[4 * i + 3], f.w,
                          fmaf(hreg[4 * i + 2], f.z,
                               fmaf(hreg[4 * i + 1], f.y, fmaf(hreg[4 * i], f.x, 0.f))));
            });
          } else if (run * 32u + rw < a.n_ads) {
#pragma unroll
            for (int i = 0; i < Sh::kCPT; i++) {
              const uint32_t c = qd * Sh::kCPT + (i ^ rot);
              const float4 f = *reinterpret_cast<const float4 *>(row + c * 16);
              d2 = __ffma2_rn(make_float2(hreg[4 * i], hreg[4 * i + 1]), make_float2(f.x, f.y), d2);
              d2 = __ffma2_rn(make_float2(hreg[4 * i + 2], hreg[4 * i + 3]), make_float2(f.z, f.w),
                              d2);
            }
          }
          float dd = TREE ? d2.x : d2.x + d2.y;
          if (Sh::kTPR == 2) {
            dd += __shfl_xor_sync(0xffffffffu, dd, 1);
            const float mine = __shfl_sync(0xffffffffu, dd, 2 * (lane & 15));
            if ((lane >> 4) == ps) dot = mine;
          } else {
            dot = dd;
          }
        }
      }
      // The stage goes back as soon as its rows and keys are read, before the
      // gathers: what a stage is held for counts against the bytes in flight.
      if (nq <= (uint32_t)kKeep) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.empty[s]);
      }
      TermSum ts;
#pragma unroll
      for (int q0 = 0; q0 < kKeep; q0 += 4) {
        if (q0 < nq) {
          uint32_t p[16];
#pragma unroll
          for (int q = 0; q < 4; q++) {
            p[4 * q] = p[4 * q + 1] = p[4 * q + 2] = p[4 * q + 3] = 0u;
            if (q0 + q < nq) quad_terms(kq[q0 + q], p + 4 * q);
          }
#pragma unroll
          for (int q = 0; q < 4; q++)
            if (q0 + q < nq) ts.add4(p[4 * q], p[4 * q + 1], p[4 * q + 2], p[4 * q + 3]);
        }
      }
      if (nq > (uint32_t)kKeep) {
        for (uint32_t q = kKeep; q < nq; q++) {
          uint32_t p[4];
          quad_terms(load_quad(ka + q * a.quad_bytes), p);
          ts.add4(p[0], p[1], p[2], p[3]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.empty[s]);
      }
      float wide = sd.wide;
      if (keys)
        wide = ((float)(ts.all - ts.c1) * u0 + (float)ts.c1 * u1) + ((float)ts.c2 * u2 + ts.fp);
      if constexpr (kMma && !kF8) {
        // An infinite element times a piece or a column that is zero is NaN,
        // which a sum with h_u itself need not be: such rows are summed again
        // by FP32 multiply-adds (E4M3 has no infinities).  Here and from global
        // memory, so that the stage and the gathers do not wait for the sum (1M ads
        // of 128 elements from host buffers 201 us with that, 197 us so).
        if (__any_sync(0xffffffffu, in && !(fabsf(dot) < INFINITY))) {
          if (in && !(fabsf(dot) < INFINITY)) {
            const uint4 *row = reinterpret_cast<const uint4 *>(a.emb) + (uint64_t)ad * Sh::kChunks;
            dot = 0.f;
#pragma unroll 1
            for (int c = 0; c < Sh::kChunks; c++) {
              float f[Tr::kVec];
              Tr::load(__ldg(row + c), f);
#pragma unroll
              for (int e = 0; e < Tr::kVec; e++) dot = fmaf(s_h[c * Tr::kVec + e], f[e], dot);
            }
          }
          __syncwarp();
        }
      }
      float score = dot;
      if (a.scale) score *= sd.scale;
      score += wide;
      if (a.wide_out && keys && in) a.wide_out[ad] = wide;
      if (a.all_out) {
        if (in) a.all_out[ad] = score;
        continue;
      }
      bool keep = in && ((sd.fword >> lane) & 1u);
      if (a.direct) {
        if (in) a.cand_out[ad] = keep ? make_key(score, ad) : 0ull;
        continue;
      }
      uint64_t kk = 0;
      if (keep) {
        kk = make_key(score, ad);
        keep = kk >= *((volatile unsigned long long *)&sm.thr);
      }
      if (__any_sync(0xffffffffu, keep)) {
        const uint32_t pos = warp_append(keep, &sm.n);
        if (keep) {
          cand[pos] = kk;
          const uint32_t bin = (uint32_t)(kk >> kBinShift);
          atomicAdd(&sm.chist[bin], 1u);
          if (bin > *((volatile uint32_t *)&sm.top_bin)) atomicMax(&sm.top_bin, bin);
          if (pos >= a.trim_at) *((volatile uint32_t *)&sm.trim) = 1u;
        }
        __syncwarp();
      }
    }
    if (a.all_out || a.direct) return;
    // The warps meet: to trim the buffer, or because every warp is done (a
    // warp without runs waits here and takes part in the trims of the others).
    gsync();
    if (tid == 0) {
      sm.n_seen = sm.n;
      sm.stop = *((volatile uint32_t *)&sm.abort);
      sm.meet = sm.trim;
      sm.trim = 0;
      if (!sm.meet || sm.stop) *((volatile uint32_t *)&sm.finished) = 1u;
    }
    gsync();
    if (sm.stop) return;
    if (!sm.meet) break;
    // trim to the K best: radix select, then a stable in-place compaction
    const uint32_t n = sm.n_seen;
    const uint64_t cut =
        group_radix_select<kConsThreads>(cand, n, a.k, sm.hist, sm.misc, tid, gsync);
    uint32_t kept = 0;
    for (uint32_t b0 = 0, rnd = 0; b0 < n; b0 += kConsThreads, rnd++) {
      const uint32_t i = b0 + tid;
      const uint64_t x = i < n ? cand[i] : 0ull;
      const bool kp = i < n && x >= cut;
      const uint32_t bal = __ballot_sync(0xffffffffu, kp);
      if (lane == 0) sm.wtot[rnd & 1][warp] = __popc(bal);
      gsync();
      uint32_t before = kept, round_total = 0;
#pragma unroll
      for (int q2 = 0; q2 < kConsWarps; q2++) {
        const uint32_t t2 = sm.wtot[rnd & 1][q2];
        before += (q2 < warp) ? t2 : 0u;
        round_total += t2;
      }
      if (kp) cand[before + __popc(bal & ((1u << lane) - 1u))] = x;
      kept += round_total;
    }
    gsync();
    if (tid == 0) {
      sm.n = kept;
      const unsigned long long g = atomicMax(&a.ctrl->thr, (unsigned long long)cut);
      atomicMax(&sm.thr, max((unsigned long long)cut, g));
    }
    gsync();
  }
  const uint32_t n = sm.n_seen;
  // the last counts, then the bound of all CTAs' counts so far: it nearly
  // always leaves fewer than K candidates, and the selection is not needed
  for (int i = tid; i < kCandBins; i += kConsThreads)
    if (sm.chist[i]) atomicAdd(a.hist + i, atomicExch(&sm.chist[i], 0u));
  if (tid == 0) {
    atomicMax(a.hist + kCandBins, sm.top_bin);
    sm.above = 0;  // (not n_seen: no barrier lies between the other warps' read of it and here)
  }
  gsync();
  if (warp == 0) {
    const unsigned long long h = hist_top_threshold(a.hist, (uint32_t)(sm.thr >> kBinShift), a.k);
    if (lane == 0) atomicMax(&sm.thr, max(*((volatile unsigned long long *)&a.ctrl->thr), h));
  }
  gsync();
  {
    const uint64_t thr = sm.thr;
    uint32_t above = 0;
    for (uint32_t i = tid; i < n; i += kConsThreads) above += cand[i] >= thr ? 1u : 0u;
    above = __reduce_add_sync(0xffffffffu, above);
    if (lane == 0 && above) atomicAdd(&sm.above, above);
  }
  gsync();
  if (sm.above > a.k) {
    const uint64_t cut =
        group_radix_select<kConsThreads>(cand, n, a.k, sm.hist, sm.misc, tid, gsync);
    if (tid == 0) {
      atomicMax(&a.ctrl->thr, (unsigned long long)cut);
      atomicMax(&sm.thr, (unsigned long long)cut);
    }
  }
  gsync();
  const uint64_t fin = sm.thr;
  for (uint32_t b0 = 0; b0 < n; b0 += kConsThreads) {
    const uint32_t i = b0 + tid;
    const uint64_t x = i < n ? cand[i] : 0ull;
    const bool kp = i < n && x >= fin;
    const uint32_t pos = warp_append(kp, &a.ctrl->n_cand);
    if (kp) a.cand_out[pos] = x;
  }
}

constexpr size_t kFwdSmemBudget = 227 * 1024 - sizeof(FwdSmem) - 512;
// Bytes of one stage: larger copies stream faster (2M FP32 ads without keys:
// stages of 16 KB 104 us, 32 KB 89 us, 64 KB 91 us).
constexpr uint32_t kStageTarget = 40 * 1024;
// Bytes of the stage ring: more did not help (2M FP32: 200 KB 111 us, 160 KB 111
// us), less did harm (10M FP8: 120 KB 445 us against 361 us at that revision),
// and what is left is L1 for the gathers of rare terms.
constexpr size_t kRingTarget = 160 * 1024;
// Packed terms held in shared memory: 4 k, 8 k and 16 k entries give the 2M FP32
// scan the same time within 2 us, 24 k leave too small a ring (182 us).
constexpr uint32_t kSmemTermsMax = 8 * 1024;
constexpr uint32_t kSmemCandMax = 5 * 1024;       // candidate buffer entries in shared memory

template <typename Elt, int D>
int launch_t(const FwdCall &c, FwdArgs a, cudaStream_t st) {
  using Sh = FwdShape<Elt, D>;
  // Ads per stage: a power of two of runs, near kStageTarget bytes, and few
  // enough that every SM gets some stages of a small inventory.
  uint32_t runs = 1;
  auto bytes_of = [&](uint32_t lg) {
    return (32u << lg) * (uint32_t)Sh::kRowBytes + (c.max_quads ? c.max_quads[lg] : 0u) * a.quad_bytes;
  };
  uint32_t lg = 0;
  while (lg < 3 && bytes_of(lg + 1) <= kStageTarget &&
         (uint64_t)c.sms * 4 * (64u << lg) <= a.n_ads)
    lg++;
  runs = 1u << lg;
  a.lg_runs = lg;
  a.stage_ads = 32 * runs;
  a.emb_bytes = a.stage_ads * Sh::kRowBytes;
  a.stage_bytes = (bytes_of(lg) + 127) / 128 * 128;
  a.n_stages = (a.n_ads + a.stage_ads - 1) / a.stage_ads;
  const int grid = (int)std::min<uint32_t>((uint32_t)c.sms, a.n_stages);
  a.trim_at = a.k + kTrimSlack;
  a.cap = a.all_out || a.direct ? 0 : (a.trim_at + 64 * cons_warps<Elt>() + 255) / 256 * 256;
  a.cand_g = nullptr;
  if (a.cap > kSmemCandMax && (size_t)grid * a.cap <= c.cta_cand_entries) a.cand_g = c.cta_cand;
  // Terms in shared memory: the copy is worth its read where the CTA gathers
  // about four times as many.
  a.smem_terms = 0;
  if (a.fwd)
    a.smem_terms = (uint32_t)std::min<uint64_t>(
        std::min<uint32_t>(c.n_keys + 1, kSmemTermsMax), (uint64_t)c.total_quads * 32 / grid);
  const bool sw = a.fwd && a.smem_terms == c.n_keys + 1;
  const size_t fixed = (size_t)(a.smem_terms + 3) / 4 * 16 + (D + 3) / 4 * 16 +
                       (a.cand_g ? 0 : (size_t)a.cap * 8);
  uint32_t stages = 2;
  // (no rare terms, no L1 for them: a ring of few runs, 128-element FP32 rows,
  // gets more; 1M ads with 450 keys 145 -> 122 us)
  const size_t ring = sw && a.stage_bytes / runs > 16 * 1024 ? 200 * 1024 : kRingTarget;
  while (stages < (uint32_t)kFwdMaxStages && (size_t)(stages + 1) * a.stage_bytes <= ring &&
         fixed + (size_t)(stages + 1) * a.stage_bytes <= kFwdSmemBudget)
    stages++;
  const size_t smem = fixed + (size_t)stages * a.stage_bytes;
  if (smem > kFwdSmemBudget) {
    set_error("forward scan: k = %u needs %zu bytes of shared memory", a.k, smem);
    return EBR_EINVAL;
  }
  a.stages = stages;
  a.workers = std::min<uint32_t>(cons_warps<Elt>(), stages << lg);
  auto kern = sw ? k_forward<Elt, D, true, false> : k_forward<Elt, D, false, false>;
  if constexpr (std::is_same<Elt, float>::value) {
    if (c.tree) kern = k_forward<float, D, false, true>;
  }
  EBR_CUDA_TRY(allow_smem(kern, kFwdSmemBudget));
  EBR_CUDA_TRY(launch_pdl(kern, grid, (cons_warps<Elt>() + 2) * 32, smem, st, a));
  return EBR_OK;
}

template <typename Elt>
int launch_d(const FwdCall &c, const FwdArgs &a, cudaStream_t st) {
  switch (c.d) {
    case 4: if constexpr (EltTraits<Elt>::kVec <= 4) return launch_t<Elt, 4>(c, a, st); break;
    case 8: if constexpr (EltTraits<Elt>::kVec <= 8) return launch_t<Elt, 8>(c, a, st); break;
    case 16: return launch_t<Elt, 16>(c, a, st);
    case 32: return launch_t<Elt, 32>(c, a, st);
    case 64: return launch_t<Elt, 64>(c, a, st);
    case 128: return launch_t<Elt, 128>(c, a, st);
  }
  set_error("embedding dimension %u unsupported for this dtype", c.d);
  return EBR_EINVAL;
}

}  // namespace

int launch_forward(const FwdCall &c, cudaStream_t st) {
  FwdArgs a;
  memset(&a, 0, sizeof(a));
  a.emb = c.emb;
  a.scale = c.scale;
  a.h_u = c.h_u;
  a.wq = c.wq;
  a.fwd = c.fwd;
  a.fwd_off = c.fwd_off;
  a.filter = reinterpret_cast<const uint32_t *>(c.filter);
  a.n_ads = c.n_ads;
  a.k = c.k;
  a.quad_bytes = c.quad_bytes;
  a.cand_out = c.cand_out;
  a.ctrl = c.ctrl;
  a.all_out = c.all_out;
  a.direct = c.direct;
  a.wide_out = c.wide_out;
  a.hist = c.hist;
  a.fx_word = reinterpret_cast<const int *>(&c.ctrl->fx);
  a.wide_in = c.wide_in;
  a.route = c.route;
  a.cls_shift = c.cls_shift;
  if (c.dtype == EBR_F32) return launch_d<float>(c, a, st);
  if (c.dtype == EBR_BF16) return launch_d<Bf16Tag>(c, a, st);
  return launch_d<Fp8Tag>(c, a, st);
}

}  // namespace ebr
