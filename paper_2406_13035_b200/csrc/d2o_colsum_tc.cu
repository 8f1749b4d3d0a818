// Column sums of the causal prompt attention (Section 4.1, Eq. 4; Eq. 6 case 1) for 16-bit Q/K on the
// 5th-generation tensor cores.  The P x P probability matrix is never stored: two sweeps recompute the
// logits tile by tile with tcgen05.mma (fp32 accumulators in tensor memory) and reduce them on the fly.
//
//   sweep 1 (rows)     lse2_i = log2 sum_{j<=i} 2^{c q_i.k_j},  c = log2(e)/sqrt(d); stored negated
//                      A = 256 query rows of one head (resident), B = key tiles 0 .. diagonal (streamed)
//   sweep 2 (columns)  s_j = sum_{i>=j} 2^{c q_i.k_j - lse2_i}
//                      A = 256 keys (resident), B = query tiles diagonal .. end (streamed, with their lse2)
// In both sweeps the quantity that is reduced belongs to an A row, i.e. to one tensor-memory lane, i.e.
// to one thread of the epilogue, and the reduction runs over that thread's registers: no shuffles, no
// atomics, a fixed order, bit-reproducible.  Across jobs the per-thread partials are added in fp64
// (sweep 2) so that a column which receives up to P probabilities keeps full fp32 accuracy.
//
// One item = (head, 256 A rows); a CTA per SM works through its items (see CsItem), so that one item's first loads and
// products run beside the epilogue of the one before it (one CTA per item: the prologue and the last combination, about
// 4 us of every CTA, were most of a short prompt's time: 32 layers of 1200 tokens 976 -> 724 us for both sweeps, eight
// layers of 4096 tokens with the caller's normalisers 811 -> 730).  One job = one streamed tile of 128 B rows against both 128-row A
// tiles: two 128 x 128 x d MMAs whose accumulators fill one of two 256-column tensor-memory buffers.
//   warp 0      TMA producer (A once; B tiles and, in sweep 2, their lse2 through a 4-stage ring)
//   warp 1      tensor-memory allocation, MMA issue
//   warps 2-17  epilogue: four warps per quarter of the lanes; warp parts 0,1 take the first A tile
//               (B rows 0-63 / 64-127), parts 2,3 the second
//
// What bounds a job: one exponential per logit.  The special-function unit takes 8 cycles for a warp's 32 of them, 2048
// cycles per job and SM quarter, twice the job's tensor-pipe time; and the instructions around them, so scale, sum and
// the normaliser's addition are packed (two logits per issue slot) and masked tiles (the diagonal, the end of the prompt)
// have a path of their own.  One pair of logits in four takes a polynomial on the FMA pipe instead (exp2_poly_pair): more
// and the issue slots become the limit.  P = 8192, 32 fp16 heads, us per sweep (ncu): 482 / 417 with scalar arithmetic
// and the mask inside the loop, 369 / 370 with every exponential on the special-function unit, 337 / 348 with every fourth
// pair as a polynomial (xu 67 %, issue 61 %, tensor 44 %).  Two layers of 32768 tokens: 24.0, 20.7 and 20.2 ms (power cap).
#include <math.h>

#include <algorithm>

#include <cuda/std/type_traits>

#include "d2o_common.cuh"
#include "d2o_tc.cuh"

namespace d2o {

constexpr int kCsEpiWarps = 16;
constexpr int kCsThreads = (2 + kCsEpiWarps) * 32;
constexpr int kCsTile = 128;                 // rows per MMA operand tile (M and N)
constexpr int kCsStages = 4;                 // B ring
enum { kSweepRows = 0, kSweepCols = 1, kSweepColsGiven = 2 };    // Given: with the caller's normalisers

struct ColsumTcArgs {
  float* neg_lse2;                           // [layers][B * Hq][lse_row(P)] negated log2-domain row normalisers (sweep 1 -> sweep 2)
  float* colsum;                             // [layers][B, Hq, P] (sweep 2)
  size_t lse_stride;                         // floats between the normalisers of two layers
  int n_items, n_pairs;                      // items of the launch; pairs of tiles of the longest prompt
  uint32_t* sched;                           // [2] items handed out beyond the first of every CTA; CTAs done (both 0 between launches)
  uint32_t* status;                          // NULL: no error word (the allocation-free entry point)
  const int32_t* plen;                       // [B] prompt length of every sequence (<= P); NULL: all P
  int P, Hq, group, BHq;                     // P: the length the tensors are laid out for; BHq: (sequence, head) pairs of a layer
  unsigned long long wait_ns;                // limit of every wait
  int stop_job;                              // failure-detection tests: no copy from this streamed tile of a CTA on (-1: never)
};

// Layers of one launch: a short prompt's layer alone (32 heads, 1200 tokens: 160 items) is little more than one item per
// SM.
struct ColsumTcMaps {
  CUtensorMap q[kColsumLayers], k[kColsumLayers];
};

// Row stride of the normalisers: the bulk copies of sweep 2 start on 16-byte boundaries whatever the prompt length.
__host__ __device__ __forceinline__ size_t lse_row(int P) { return (size_t)((P + 3) & ~3); }

constexpr int kPolyPairs = 0x11;             // of eight pairs of logits, those whose exponentials go to the FMA pipe

namespace tc {
// two fp32 lanes in one 64-bit register, and the packed operations on them (one issue slot each)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// maximum and minimum that keep a NaN
__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// global -> this CTA's shared memory, 16-byte aligned on both sides, size a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// 2^x on the special-function unit (one instruction; results below 2^-126 flush to zero)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// maximum of three; a NaN operand is ignored
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
}  // namespace tc

// acc += (2^x, 2^y) on the FMA pipe.  x = n + f with n the nearest integer and |f| <= 1/2 (adding 1.5 * 2^23 rounds to
// the nearest integer and leaves n in the low mantissa bits), 2^f by the polynomial of degree 5 with constant term 1
// whose largest relative error on [-1/2, 1/2] is smallest (9.1e-8; found as a linear program over 4001 Chebyshev points;
// 1.7e-7 with the fp32 roundings of Horner's rule, the same size as the special-function unit's), 2^n as exponent bits.
// Exponents below -127 count as -127, whose exponent bits are those of zero: such a term is 0.  A NaN stays one.  HIGH:
// exponents that round to 128 and more count as 128, whose exponent bits are those of infinity (normalisers that the caller
// made too low, or -inf); the sweeps' own normalisers leave none above 0, but for rounding, and skip it.
template <bool HIGH>
__device__ __forceinline__ tc::f32x2 exp2_poly_pair(tc::f32x2 xy, tc::f32x2 acc) {
  const float kRound = 12582912.0f;
  float x, y;
  tc::unpack2(xy, x, y);
  x = tc::max_nan(x, -127.f); y = tc::max_nan(y, -127.f);
  if (HIGH) { x = tc::min_nan(x, 128.f); y = tc::min_nan(y, 128.f); }
  xy = tc::pack2(x, y);
  const tc::f32x2 t = tc::add2(xy, tc::pack2(kRound, kRound));
  const tc::f32x2 n = tc::add2(t, tc::pack2(-kRound, -kRound));
  const tc::f32x2 f = tc::fma2(n, tc::pack2(-1.f, -1.f), xy);                 // exact
  tc::f32x2 p = tc::pack2(0.001326472731307149f, 0.001326472731307149f);
  p = tc::fma2(p, f, tc::pack2(0.009671512991189957f, 0.009671512991189957f));
  p = tc::fma2(p, f, tc::pack2(0.05550733581185341f, 0.05550733581185341f));
  p = tc::fma2(p, f, tc::pack2(0.24022242426872253f, 0.24022242426872253f));
  p = tc::fma2(p, f, tc::pack2(0.6931470036506653f, 0.6931470036506653f));
  p = tc::fma2(p, f, tc::pack2(1.f, 1.f));
  float t0, t1;
  tc::unpack2(t, t0, t1);
  const tc::f32x2 s = tc::pack2(__uint_as_float((__float_as_uint(t0) << 23) + 0x3f800000u),
                                __uint_as_float((__float_as_uint(t1) << 23) + 0x3f800000u));
  return tc::fma2(p, s, acc);
}

// Which pairs of 64 logits take the polynomial.
__host__ __device__ constexpr bool poly_pair(int k) { return (kPolyPairs >> (k & 7)) & 1; }

// Sum of 2^{c s_i + b_i} over the 64 logits s_i of one accumulator row (in two register blocks).  Rows: every b_i is
// `b`; columns: b_i comes from shared memory (the negated normalisers of the 64 streamed rows).
template <bool PER_ROW, bool HIGH>
__device__ __forceinline__ float exp_sum_64(const uint32_t (&ra)[32], const uint32_t (&rb)[32], float c, float b,
                                            const float* s_b) {
  const tc::f32x2 c2 = tc::pack2(c, c), b2 = tc::pack2(b, b);
  tc::f32x2 acc[2] = {0ull, 0ull}, pac[2] = {0ull, 0ull};
#pragma unroll
  for (int i4 = 0; i4 < 8; ++i4) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      tc::f32x2 bb[2] = {b2, b2};
      if (PER_ROW) {
        const float4 v = *reinterpret_cast<const float4*>(s_b + half * 32 + i4 * 4);
        bb[0] = tc::pack2(v.x, v.y); bb[1] = tc::pack2(v.z, v.w);
      }
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int i = i4 * 4 + w * 2;
        const tc::f32x2 s = half == 0 ? tc::pack2(__uint_as_float(ra[i]), __uint_as_float(ra[i + 1]))
                                      : tc::pack2(__uint_as_float(rb[i]), __uint_as_float(rb[i + 1]));
        const tc::f32x2 x = tc::fma2(s, c2, bb[w]);
        if (poly_pair(i4 * 4 + half * 2 + w)) {
          pac[w] = exp2_poly_pair<HIGH>(x, pac[w]);
        } else {
          float x0, x1;
          tc::unpack2(x, x0, x1);
          acc[w] = tc::add2(acc[w], tc::pack2(tc::ex2(x0), tc::ex2(x1)));
        }
      }
    }
  }
  const tc::f32x2 t = tc::add2(tc::add2(acc[0], acc[1]), tc::add2(pac[0], pac[1]));
  float lo, hi;
  tc::unpack2(t, lo, hi);
  return lo + hi;
}

// One item: 256 A rows of one (layer, sequence, head).  Items of a layer are numbered heaviest first (sweep 1: the last
// rows see the most keys; sweep 2: the first keys see the most rows), all heads of a pair of tiles next to one another so
// that the CTAs at work share the streamed tiles in L2, the layers one after another.  CTA i begins with item i and takes
// the next free one from a counter from then on.
template <int SWEEP>
struct CsItem {
  int layer, bh, P, a0, bt0, n_jobs;                         // n_jobs = 0: the sequence has no such rows
  __device__ __forceinline__ void decode(const ColsumTcArgs& a, int i) {
    n_jobs = 0;
    bh = i % a.BHq;
    const int y = i / a.BHq % a.n_pairs;
    layer = i / a.BHq / a.n_pairs;
    P = a.plen ? a.plen[bh / a.Hq] : a.P;                    // this sequence's prompt; rows beyond it are padding
    const int n_pairs = (P + 2 * kCsTile - 1) / (2 * kCsTile), n_tiles = (P + kCsTile - 1) / kCsTile;
    if (y >= n_pairs) return;                                // the numbering is for the longest prompt
    a0 = (SWEEP == kSweepRows ? n_pairs - 1 - y : y) * 2 * kCsTile;          // first A row (query or key position)
    // streamed tiles: sweep 1 keys [0, a0 + 256), sweep 2 queries [a0, P)
    bt0 = SWEEP == kSweepRows ? 0 : a0 / kCsTile;
    n_jobs = (SWEEP == kSweepRows ? min(n_tiles, (a0 + 2 * kCsTile) / kCsTile) : n_tiles) - bt0;
  }
  // Has A tile t any valid logit with the streamed tile of a job?  Not beyond the diagonal, nor past the prompt.
  __device__ __forceinline__ bool valid(int t, int job) const {
    const int at = a0 / kCsTile + t;
    return at * kCsTile < P && (SWEEP == kSweepRows ? bt0 + job <= at : bt0 + job >= at);
  }
  __device__ __forceinline__ int q_base(const ColsumTcArgs& a) const { return bh * a.P; }     // first row of the head in the views
  __device__ __forceinline__ int k_base(const ColsumTcArgs& a) const {
    return (bh / a.Hq * (a.Hq / a.group) + bh % a.Hq / a.group) * a.P;
  }
};

template <int D, int FMT, int SWEEP>
__global__ void __launch_bounds__(kCsThreads, 1)
attn_tc_kernel(ColsumTcArgs a, const __grid_constant__ ColsumTcMaps maps) {
  constexpr int KB = D / 64;                                 // 64-element (128-byte) blocks along d
  constexpr int BLOCK = kCsTile * 128;                       // bytes of one k-block of one 128-row tile
  constexpr int TILE = KB * BLOCK;                           // bytes of one 128-row tile
  constexpr uint32_t IDESC = make_idesc(FMT, kCsTile, kCsTile);
  const float c = (D == 64 ? 0.125f : 0.08838834764831845f) * kLog2e;

  extern __shared__ __align__(1024) unsigned char cs_smem[];
  unsigned char* sA = cs_smem;                               // [2 tiles][KB][128 rows][128 B]
  unsigned char* sB = cs_smem + 2 * TILE;                    // [stages][KB][128 rows][128 B]
  float* s_lse = reinterpret_cast<float*>(sB + kCsStages * TILE);   // [stages][128] negated lse2 of the B rows (sweep 2)
  float* s_comb = s_lse + kCsStages * kCsTile;               // [2][2][2][128] partner values for the final combination
  __shared__ unsigned long long a_full, a_empty, b_full[kCsStages], b_empty[kCsStages], tm_full[2], tm_empty[2], it_full[2], it_empty[2];
  __shared__ int s_item[2];                                  // the CTA's current and next item, -1: no more
  __shared__ int s_now[2], s_lost;                           // the epilogue's current item; taken after a wait had run out
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if ((tc::smem_u32(cs_smem) & 1023u) != 0u) {               // swizzled tiles need 1024-byte aligned shared memory
    if (tid == 0 && a.status) report_error(a.status, D2O_ERR_STATE, 0xC5C10000u);
    return;
  }

  if (tid == 0) {
    s_fail = 0; s_lost = s_item[0] = s_item[1] = -1;
    tc::mbar_init(&a_full, 1); tc::mbar_init(&a_empty, 1);
    for (int s = 0; s < kCsStages; ++s) { tc::mbar_init(&b_full[s], 1); tc::mbar_init(&b_empty[s], 1 + kCsEpiWarps); }
    for (int i = 0; i < 2; ++i) { tc::mbar_init(&tm_full[i], 1); tc::mbar_init(&tm_empty[i], kCsEpiWarps);
                                  tc::mbar_init(&it_full[i], 1); tc::mbar_init(&it_empty[i], 2); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {                                           // 512 columns: two buffers of 2 x (128 x 128) fp32
    tc::tmem_alloc(&s_tmem, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem_base = s_tmem;
  auto wait = [&](unsigned long long* bar, uint32_t parity) { return tc::mbar_wait(bar, parity, a.wait_ns); };
  // The set-up above ran beside the tail of the kernel ahead (both sweeps and the densities of 32 heads of 300 tokens 26.7 ->
  // 20.5 us, three layers of 32 heads of 1100 tokens, d = 64, 71.9 -> 66.8; large calls as before).
  wait_for_prior_grid();

  // The k-th item of this CTA as its two consumers see it (the MMA thread, one thread of the epilogue); -1: no more.
  auto next_item = [&](int k) {
    if (!wait(&it_full[k & 1], (uint32_t)((k >> 1) & 1))) { s_fail = 1; return -1; }
    const int i = s_item[k & 1];
    tc::mbar_arrive(&it_empty[k & 1]);
    return i;
  };
  int jb_copies = 0, ia_copies = 0;                          // the producer's streamed tiles and items with copies

  if (warp == 0) {
    // ======================================================================= TMA producer
    if (lane == 0) {
      if (SWEEP != kSweepRows) asm volatile("fence.proxy.async.global;" ::: "memory");    // normalisers: stored by the kernel ahead, copied in bulk here
      CsItem<SWEEP> it{};
      int jb = 0, ia = 0;                                    // jobs and items so far
      int item = (int)blockIdx.x;
      for (int k = 0;; ++k) {
        if (k >= 2 && !wait(&it_empty[k & 1], (uint32_t)(((k >> 1) - 1) & 1))) s_fail = 1;
        if (s_fail) { s_lost = item; break; }                // the consumers find no further item and leave
        s_item[k & 1] = item < a.n_items ? item : -1;
        tc::mbar_arrive(&it_full[k & 1]);
        if (item >= a.n_items) { start_dependents(); break; }  // the next kernel may set itself up during the last items
        it.decode(a, item);
        const CUtensorMap* map_a = SWEEP == kSweepRows ? &maps.q[it.layer] : &maps.k[it.layer];
        const CUtensorMap* map_b = SWEEP == kSweepRows ? &maps.k[it.layer] : &maps.q[it.layer];
        const int a_row = (SWEEP == kSweepRows ? it.q_base(a) : it.k_base(a)) + it.a0;
        const int b_base = SWEEP == kSweepRows ? it.k_base(a) : it.q_base(a);
        const float* neg_lse2 = a.neg_lse2 + it.layer * a.lse_stride + it.bh * lse_row(a.P);
        for (int job = 0; job < it.n_jobs; ++job, ++jb) {
          // the first streamed tile goes ahead of the resident ones: its stage is free earlier than they are
          const int s = jb % kCsStages;
          if (jb >= kCsStages && !s_fail && !wait(&b_empty[s], (uint32_t)(((jb / kCsStages) - 1) & 1))) s_fail = 1;
          if (s_fail || jb == a.stop_job) break;
          const int r0 = (it.bt0 + job) * kCsTile;           // first B row of the tile
          // 16-byte granules: up to three entries past the prompt come from the row's padding and are masked
          const int n_lse = SWEEP != kSweepRows ? min(kCsTile, ((it.P + 3) & ~3) - r0) : 0;
          tc::mbar_expect_tx(&b_full[s], (uint32_t)(TILE + n_lse * 4));
          for (int kb = 0; kb < KB; ++kb)
            tc::tma_load_2d(sB + s * TILE + kb * BLOCK, map_b, kb * 64, b_base + r0, &b_full[s]);
          if (n_lse > 0) tc::bulk_g2s(s_lse + s * kCsTile, neg_lse2 + r0, (uint32_t)(n_lse * 4), &b_full[s]);
          if (job == 0) {
            if (ia >= 1 && !wait(&a_empty, (uint32_t)((ia - 1) & 1))) { s_fail = 1; ++jb; break; }
            tc::mbar_expect_tx(&a_full, (uint32_t)(2 * TILE));
            for (int t = 0; t < 2; ++t)
              for (int kb = 0; kb < KB; ++kb)
                tc::tma_load_2d(sA + t * TILE + kb * BLOCK, map_a, kb * 64, a_row + t * kCsTile, &a_full);
            ++ia;
          }
        }
        if (jb == a.stop_job) break;
        // Not earlier: this thread is up to four tiles ahead of the epilogue, which covers the counter's latency, and an
        // item taken at the beginning of a long one would wait while other CTAs run out of work (2048 tokens, 32 heads:
        // 80 us instead of 62).
        item = (int)(gridDim.x + atomicAdd(&a.sched[0], 1u));
      }
      jb_copies = jb; ia_copies = ia;
    }
  } else if (warp == 1) {
    // ======================================================================= MMA issuer
    if (lane == 0) {
      CsItem<SWEEP> it;
      int jb = 0, ia = 0;
      for (int k = 0;; ++k) {
      const int item = next_item(k);
      if (item < 0) break;
      it.decode(a, item);
      if (it.n_jobs == 0) continue;
      if (!s_fail && !wait(&a_full, (uint32_t)(ia & 1))) s_fail = 1;
      ++ia;
      for (int job = 0; job < it.n_jobs && !s_fail; ++job, ++jb) {
        const int s = jb % kCsStages, buf = jb & 1;
        if (!s_fail && !wait(&b_full[s], (uint32_t)((jb / kCsStages) & 1))) s_fail = 1;
        // the epilogue must have drained this buffer (the first use of each buffer passes at once)
        if (!s_fail && !wait(&tm_empty[buf], (uint32_t)(((jb >> 1) & 1) ^ 1))) s_fail = 1;
        if (s_fail) break;
        tc::fence_after_sync();
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (!it.valid(t, job)) continue;
          const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256 + t * kCsTile);
#pragma unroll
          for (int kb = 0; kb < KB; ++kb) {
            const uint64_t adesc = tc::smem_desc_sw128(tc::smem_u32(sA + t * TILE + kb * BLOCK));
            const uint64_t bdesc = tc::smem_desc_sw128(tc::smem_u32(sB + s * TILE + kb * BLOCK));
#pragma unroll
            for (int k = 0; k < 4; ++k)                      // 16 elements = 32 bytes along d per instruction
              tc::mma_f16(d_tmem, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), IDESC, (kb | k) != 0 ? 1u : 0u);
          }
        }
        tc::mma_commit(&tm_full[buf]);
        tc::mma_commit(&b_empty[s]);                         // one of the 17 arrivals that free the stage
        if (job == it.n_jobs - 1) tc::mma_commit(&a_empty);  // the resident tiles have been read
      }
      }
      if (s_fail)                                            // tensor memory is freed behind the last products
        for (int j = max(0, jb - 2); j < jb; ++j) (void)wait(&tm_full[j & 1], (uint32_t)((j >> 1) & 1));
    }
  } else {
    // ======================================================================= epilogue warps
    const int e = warp - 2;
    const int quarter = warp & 3;                            // tensor-memory lanes this warp may read: 32*quarter ..
    const int part = e >> 2;                                 // 0,1: first A tile, B rows 0-63 / 64-127; 2,3: second A tile
    const int at = part >> 1, bhalf = part & 1;
    CsItem<SWEEP> it;
    int jb = 0;
    // One thread looks at the next item, for all, ahead of the barrier that ends the one before: warps that waited for it each
    // by itself could run out of time apart, and those that stayed would wait at the barrier for good.
    auto end_item = [&](int k) {
      if (e == 0 && lane == 0) s_now[(k + 1) & 1] = next_item(k + 1);
      __syncwarp();
      asm volatile("bar.sync 1, %0;" ::"n"(kCsEpiWarps * 32) : "memory");
    };
    end_item(-1);
#pragma unroll 1
    for (int k = 0;; ++k) {
    const int item = s_now[k & 1];
    if (item < 0) break;
    it.decode(a, item);
    if (it.n_jobs == 0) { end_item(k); continue; }
    const int n_jobs = __any_sync(0xffffffffu, s_fail != 0) ? 0 : it.n_jobs;     // after a wait that ran out: NaN, at once
    const int P = it.P, w0 = it.a0 + at * kCsTile + quarter * 32;        // first A row of this warp
    const int arow = w0 + lane;                              // position of this thread's A row (query or key)
    // sweep 1: running maximum m of the log2-domain logits and sum of 2^{c s - m}; sweep 2: column sum
    float m_run = -INFINITY, l_run = 0.f;
    double col_acc = 0.0;
#pragma unroll 1
    for (int job = 0; job < n_jobs; ++job, ++jb) {
      const int s = jb % kCsStages, buf = jb & 1;
      const int brow0 = (it.bt0 + job) * kCsTile + bhalf * 64;   // position of the first B row this warp looks at
      if (!__all_sync(0xffffffffu, wait(&tm_full[buf], (uint32_t)((jb >> 1) & 1)))) { s_fail = 1; break; }
      tc::fence_after_sync();
      // Each of the paths below loads the accumulator's block into registers of its own, and products that no path needs are
      // not made (CsItem::valid).  us, one set for masked and unmasked paths and all products / so: 32 heads of 300 tokens
      // 20.3 / 18.5; four layers of 2 x 16 heads of 1700 tokens, d = 64, 142.4 / 136.9; four layers of 2 x 32 heads of 600 tokens with
      // the caller's normalisers 39.1 / 38.3; long prompts run at the power cap and take the same time (two layers of 6001
      // tokens 714 - 726 / 716 - 719).
      auto drained = [&]() {                                   // hand the accumulator back to the MMA warp
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&tm_empty[buf]);
      };
      auto load = [&](uint32_t (&ra)[32], uint32_t (&rb)[32]) {
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * 256 + at * kCsTile + bhalf * 64);
        tc::tmem_ld32_issue(taddr, ra);
        tc::tmem_ld32_issue(taddr + 32u, rb);
        tc::tmem_ld_wait(ra);
        tc::tmem_ld_wait(rb);
        drained();
      };
      if (SWEEP == kSweepRows) {
        // B rows are keys: valid iff key <= query (keys >= P are > every stored query)
        auto rows = [&](auto diagonal) {
          uint32_t ra[32], rb[32];
          load(ra, rb);
          if (decltype(diagonal)::value) {
            const int last = arow - brow0;                     // the row's last valid column of the 64
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              if (i > last) ra[i] = 0xff800000u;
              if (i + 32 > last) rb[i] = 0xff800000u;
            }
          }
          // four independent chains of three-input maxima: the block maximum is on every thread's critical path
          float bmx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int i = 0; i < 32; ++i) bmx[i & 3] = tc::max3(bmx[i & 3], __uint_as_float(ra[i]), __uint_as_float(rb[i]));
          const float bm = fmaxf(fmaxf(bmx[0], bmx[1]), fmaxf(bmx[2], bmx[3])) * c;     // in the log2 domain, rounded once
          if (bm > m_run) { l_run *= exp2f(m_run - bm); m_run = bm; }            // exp2f(-inf) = 0 on the first block
          const float sum = exp_sum_64<false, false>(ra, rb, c, m_run > -INFINITY ? -m_run : 0.f, nullptr);
          if (m_run > -INFINITY) l_run += sum;
        };
        if (brow0 > w0 + 31 || w0 >= P) drained();             // warp-uniform: nothing of this warp's block is valid
        else if (brow0 + 63 > w0) rows(cuda::std::true_type{});
        else rows(cuda::std::false_type{});
      } else {
        // B rows are queries: valid iff query >= key and query < P
        const float* ls = s_lse + s * kCsTile + bhalf * 64;
        if (brow0 + 63 < w0 || brow0 >= P) {                   // warp-uniform: nothing is valid
          drained();
        } else if (brow0 >= w0 + 31 && brow0 + 64 <= P) {      // warp-uniform: nothing is masked
          uint32_t ra[32], rb[32];
          load(ra, rb);
          col_acc += (double)exp_sum_64<true, SWEEP == kSweepColsGiven>(ra, rb, c, 0.f, ls);
        } else {
          uint32_t ra[32], rb[32];
          load(ra, rb);
          const int first = arow - brow0, end = P - brow0;     // the row's valid columns of the 64
          float p0 = 0.f, p1 = 0.f;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float x = tc::ex2(fmaf(__uint_as_float(ra[i]), c, ls[i]));
            const float y = tc::ex2(fmaf(__uint_as_float(rb[i]), c, ls[32 + i]));
            p0 += i >= first && i < end ? x : 0.f;
            p1 += i + 32 >= first && i + 32 < end ? y : 0.f;
          }
          col_acc += (double)(p0 + p1);
        }
      }
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&b_empty[s]);           // this warp is done with the stage (sweep 2: its normalisers)
    }
    // combine the two warps that share an A row (B-row halves), fixed order; after a wait that ran out: NaN.  The exchange
    // area alternates between items: whoever writes it again has passed the barrier of the item in between.
    const int r = quarter * 32 + lane;
    float* comb = s_comb + (k & 1) * 4 * kCsTile;
    if (SWEEP == kSweepRows) {
      if (bhalf == 1) { comb[(at * 2 + 0) * kCsTile + r] = m_run; comb[(at * 2 + 1) * kCsTile + r] = l_run; }
      end_item(k);
      if (bhalf == 0 && arow < P) {
        const float m2 = comb[(at * 2 + 0) * kCsTile + r], l2 = comb[(at * 2 + 1) * kCsTile + r];
        const float mm = fmaxf(m_run, m2);
        const float ll = (m_run > -INFINITY ? l_run * exp2f(m_run - mm) : 0.f) +
                         (m2 > -INFINITY ? l2 * exp2f(m2 - mm) : 0.f);
        a.neg_lse2[it.layer * a.lse_stride + it.bh * lse_row(a.P) + arow] = s_fail ? NAN : -(mm + log2f(ll));
      }
    } else {
      double* dcomb = reinterpret_cast<double*>(comb);
      if (bhalf == 1) dcomb[at * kCsTile + r] = col_acc;
      end_item(k);
      if (bhalf == 0 && arow < P)
        a.colsum[((size_t)it.layer * a.BHq + it.bh) * a.P + arow] = s_fail ? NAN : (float)(col_acc + dcomb[at * kCsTile + r]);
    }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem_base, 512);
  }
  if (s_fail) {
    if (tid == 0) {                                          // see the copies on their way land before the CTA may end
      for (int i = max(0, jb_copies - kCsStages); i < jb_copies; ++i)
        if (!wait(&b_full[i % kCsStages], (uint32_t)((i / kCsStages) & 1))) break;
      if (ia_copies > 0) (void)wait(&a_full, (uint32_t)((ia_copies - 1) & 1));
    }
    // NaN for the items this CTA had in hand, and for those that nobody has taken
    for (int n = 0;; ++n) {
      if (tid == 0) s_now[0] = n < 2 ? s_item[n] : n == 2 ? s_lost : (int)(gridDim.x + atomicAdd(&a.sched[0], 1u));
      __syncthreads();
      const int i = s_now[0];
      __syncthreads();
      if (i >= a.n_items && n > 2) break;
      if (i < 0 || i >= a.n_items) continue;
      CsItem<SWEEP> it;
      it.decode(a, i);
      if (it.n_jobs == 0) continue;
      for (int r = it.a0 + tid; r < min(it.P, it.a0 + 2 * kCsTile); r += kCsThreads) {
        if (SWEEP == kSweepRows) a.neg_lse2[it.layer * a.lse_stride + it.bh * lse_row(a.P) + r] = NAN;
        else a.colsum[((size_t)it.layer * a.BHq + it.bh) * a.P + r] = NAN;
      }
    }
  }
  if (tid == 0) {                                            // the last CTA leaves the counters at zero for the next launch
    __threadfence();
    if (atomicAdd(&a.sched[1], 1u) == gridDim.x - 1) { a.sched[0] = 0u; a.sched[1] = 0u; }
  }
  if (tid == 0 && s_fail && a.status) report_error(a.status, D2O_ERR_TIMEOUT, 0xC5C00000u | (uint32_t)(blockIdx.x & 0xfffff));
}

// natural-log row normalisers supplied by the caller -> negated log2 domain, padded rows; one (sequence, head) per
// blockIdx.x, one layer per blockIdx.z
struct LseIn { const float* p[kColsumLayers]; };
__global__ void lse_to_log2_kernel(LseIn lse, float* __restrict__ neg_lse2, size_t lse_stride, int P) {
  const int i = blockIdx.y * blockDim.x + threadIdx.x;
  if (i < P)
    neg_lse2[blockIdx.z * lse_stride + blockIdx.x * lse_row(P) + i] = -(lse.p[blockIdx.z][(size_t)blockIdx.x * P + i] * kLog2e);
}

size_t colsum_tc_lse_bytes(int batch, int n_q_heads, int P) { return (size_t)batch * n_q_heads * lse_row(P) * 4; }

// Column sums of n <= kColsumLayers layers of 16-bit Q, K on the tensor cores.  `lse_in` (natural log; NULL, or a pointer
// per layer) replaces sweep 1; `neg_lse2` is scratch of n times colsum_tc_lse_bytes(), `lse_stride` bytes apart; `colsum` of
// the layers lies one after another; `plen` (DEVICE, may be NULL) holds every sequence's prompt length, `status` (may be
// NULL) the error word, `sched` two words that are zero between launches; `wait_ns` (0: one second) and `stop_job` are for the
// failure-detection tests.  Any prompt length: the rows of a TMA box need no alignment.  (Lengths that are not a multiple of
// four used to take the FFMA kernels: 17.5 ms instead of 1.0 for two layers of 6001 tokens.)
cudaError_t launch_colsum_tc(int dtype, int D, int B, int Hq, int Hkv, int P, int n, const void* const* Q,
                             const void* const* K, const float* const* lse_in, float* neg_lse2, size_t lse_stride,
                             float* colsum, const int32_t* plen, uint32_t* status, uint32_t* sched, cudaStream_t st,
                             unsigned long long wait_ns, int stop_job) {
  ColsumTcMaps maps;
  LseIn lse;
  for (int l = 0; l < n; ++l) {
    if (!encode_rows_2d(&maps.q[l], dtype, Q[l], (uint64_t)B * Hq * P, D, kCsTile)) return cudaErrorNotSupported;
    if (!encode_rows_2d(&maps.k[l], dtype, K[l], (uint64_t)B * Hkv * P, D, kCsTile)) return cudaErrorNotSupported;
    if (lse_in) lse.p[l] = lse_in[l];
  }
  ColsumTcArgs a;
  a.neg_lse2 = neg_lse2;
  a.lse_stride = lse_stride / sizeof(float);
  a.colsum = colsum;
  a.status = status;
  a.sched = sched;
  a.wait_ns = wait_ns > 0 ? wait_ns : kTcWaitNs; a.stop_job = stop_job;
  a.P = P; a.Hq = Hq; a.group = Hq / Hkv; a.BHq = B * Hq;
  a.plen = plen;
  const int KB = D / 64;
  const size_t smem = (size_t)(2 + kCsStages) * KB * kCsTile * 128 + (size_t)kCsStages * kCsTile * 4 + 8 * kCsTile * 4;
  a.n_pairs = (P + 2 * kCsTile - 1) / (2 * kCsTile);
  const long items = (long)n * B * Hq * a.n_pairs;
  if (items >= (1l << 30)) return cudaErrorInvalidValue;
  a.n_items = (int)items;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return cudaGetLastError();
  const dim3 grid((unsigned)std::min(items, (long)sms));     // one CTA per SM (shared and tensor memory)
  const int fmt = dtype == D2O_F16 ? 0 : 1;
  cudaError_t e;
#define D2O_LAUNCH_CS(DD, FF, SW)                                                                                  \
  do {                                                                                                             \
    e = cudaFuncSetAttribute(attn_tc_kernel<DD, FF, SW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);  \
    if (e != cudaSuccess) return e;                                                                                \
    e = launch_behind(attn_tc_kernel<DD, FF, SW>, grid, kCsThreads, smem, st, a, maps);                            \
    if (e != cudaSuccess) return e;                                                                                \
  } while (0)
#define D2O_LAUNCH_CS_ALL(SW)                                                                    \
  do {                                                                                           \
    if (D == 128) { if (fmt == 0) D2O_LAUNCH_CS(128, 0, SW); else D2O_LAUNCH_CS(128, 1, SW); }   \
    else          { if (fmt == 0) D2O_LAUNCH_CS(64, 0, SW); else D2O_LAUNCH_CS(64, 1, SW); }     \
  } while (0)
  if (lse_in) {
    lse_to_log2_kernel<<<dim3((unsigned)(B * Hq), (unsigned)((P + 255) / 256), (unsigned)n), 256, 0, st>>>(lse, neg_lse2, a.lse_stride, P);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    D2O_LAUNCH_CS_ALL(kSweepColsGiven);
  } else {
    D2O_LAUNCH_CS_ALL(kSweepRows);
    D2O_LAUNCH_CS_ALL(kSweepCols);
  }
#undef D2O_LAUNCH_CS_ALL
#undef D2O_LAUNCH_CS
  return cudaSuccess;
}

}  // namespace d2o
