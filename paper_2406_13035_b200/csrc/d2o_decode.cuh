// Pieces shared by the two decode kernels (d2o_decode.cu: one CTA per slice; d2o_decode_split.cu: one cluster per
// slice): launch arguments, mbarrier and bulk-copy wrappers with bounded waits, packed fp32 arithmetic, the mma.sync steps.
#pragma once

#include <cuda/std/type_traits>

#include "d2o_common.cuh"
#include "d2o_tc.cuh"

namespace d2o {

constexpr unsigned long long kWaitNs = 1000000000ull;   // an mbarrier wait gives up after 1 s
constexpr uint32_t kSuspendNs = 4000u;                  // a waiting thread may stay suspended this long before it looks again

// 16-bit caches with several query heads per KV head take the tensor-core path (more registers per thread, fewer
// instructions per row); the weights enter its value pass as two 16-bit terms.  With one head the FMA loops are as fast, use
// every warp, and keep the weights in fp32.
constexpr int kTensorMinG = 2;
__host__ __device__ constexpr bool tensor_path(int elem_size, int G) { return elem_size == 2 && G >= kTensorMinG; }

struct DecodeArgs {
  const int32_t* budgets; const int32_t* windows; const int64_t* row_off;   // [B, L, Hkv]
  int32_t* pos; float* score; float* rnorm;                                  // pool-wide
  int32_t* len; float* tau;                                                  // [L, B, Hkv]
  unsigned long long* counters; uint32_t* status;
  const int32_t* plen;              // [B] prompt length of every sequence
  int L, l0, B, Hkv, T, step;       // step = number of tokens generated before this one: its position is plen[b] + step
  float beta, tau_override;
  int row_cap;                      // rows of a slice whose logits / probabilities live in shared memory (multiple of 8)
  float* spill;                     // the same for rows >= row_cap: [(row0 + 8 slice) G + g (stride(S) + 8) + row], stays in L2
  int stages;                       // stages of the ring
  int l2_hints;                     // 1: the streamed rows are marked evict-first in L2 (each is read once per step)
  const int32_t* order;             // NULL: CTAs take (layer, b, h) in index order; else (layer * B + b) per group of Hkv CTAs
  int pair_base;                    // first entry of `order` this launch works on
  int average;                      // 1: average merge (both rows weigh 1/2) instead of the weights of Eq. 12
  unsigned long long wait_ns;       // a wait for a stage gives up after this long
  int stop_stage;                   // failure-detection tests: the producer issues no copy from this stage on (-1: never)
  long long pool_rows;              // rows of the cache pool (bounds of the checked build)
  int32_t* steps_done;              // [L, B, Hkv] decode steps completed on the slice: written as a CTA's last act
  int chained;                      // 1: the previous step's grids may still be running (see slice_ready)
  int early;                        // decode_split_kernel: 1: the slice may be read (once slice_ready) before the grid ahead is done.
                                    // Only behind a step that published the counter: a compression's grids may still be writing
                                    // the slice, and until they are done the counter may be an earlier conversation's
  int publish;                      // 1: the CTA (cluster) publishes the slice's step counter at its end: a chained step follows, or
                                    // (decode_split_kernel) the next call is likely to work on the same layers
  int pub_first, pub_count, pub_step;   // decode_split_kernel: slices of the call before whose counters this grid writes, and their value
};

// d2o_decode_split.cu
void decode_split_places(int* clusters);
int decode_split_cluster(const d2o_ctx* c, int n_slices, int max_rows, double total_rows);
cudaError_t launch_decode_split(const d2o_ctx* c, DecodeArgs a, int C, int n_slices, int max_rows, const void* q,
                                const void* k, const void* v, void* out, void* kpool, void* vpool, cudaStream_t st);

// ----------------------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long global_ns() { unsigned long long t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs) : "memory");
  return ok != 0;
}
// Wait for a stage in the kernel's loops: one probe when the phase is already complete (the common case); otherwise
// poll until it completes, another thread has recorded a timeout, or this one does.
__device__ __forceinline__ void stage_wait(unsigned long long* bar, uint32_t parity, volatile int* timeout,
                                           unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return;
  const unsigned long long t0 = global_ns();
  while (*timeout == 0) {
    if (mbar_try_wait(bar, parity)) return;
    if (global_ns() - t0 > limit_ns) { *timeout = 2; return; }
  }
}
// The same without giving up early when another thread has recorded a timeout: used by the producer to see its own
// copies land before it leaves.  false = the limit ran out.
__device__ __forceinline__ bool landed_wait(unsigned long long* bar, uint32_t parity, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}
// Waits, with a limit, until the slice's step counter has reached `want`: the CTA that ran the slice's previous
// decode step has finished and its stores are visible.  0: ready; 1: an anomaly was recorded meanwhile (the state is
// no longer trusted); 2: the wait ran out.
__device__ __forceinline__ int slice_ready(const int32_t* flag, int want, const uint32_t* status, unsigned long long limit_ns) {
  const unsigned long long t0 = global_ns();
  for (;;) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= want) return 0;
    if (*reinterpret_cast<const volatile uint32_t*>(status) != 0u) return 1;
    if (global_ns() - t0 > limit_ns) return 2;
    __nanosleep(200);
  }
}
// Similarity as an ordered key: -0 (a zero-norm row times a negative dot product) must count as +0, or equal
// similarities would not tie.
__device__ __forceinline__ uint32_t sim_ord(float u) { return float_ord(__fadd_rn(u, 0.f)); }
// d = a * b + c on two fp32 lanes at once (one issue slot instead of two)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<const unsigned long long*>(&a)), "l"(*reinterpret_cast<const unsigned long long*>(&b)),
        "l"(*reinterpret_cast<const unsigned long long*>(&c)));
  return *reinterpret_cast<float2*>(&d);
}
// dot product of two pieces of N floats each, accumulated in two interleaved fp32 chains
template <int N>
__device__ __forceinline__ float dot_pairs(const float (&a)[N], const float (&b)[N]) {
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < N; i += 2) acc = ffma2(make_float2(a[i], a[i + 1]), make_float2(b[i], b[i + 1]), acc);
  return acc.x + acc.y;
}
// next slot of the ring; the parity flips on wrap-around
__device__ __forceinline__ void ring_next(int& slot, uint32_t& ph, int stages) {
  if (++slot == stages) { slot = 0; ph ^= 1u; }
}
// global -> this CTA's shared memory, 16-byte aligned on both sides, size a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void bulk_g2s_hint(void* dst, const void* src, uint32_t bytes, unsigned long long* bar,
                                              unsigned long long policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy) : "memory");
}

// Sums four values, each spread over the LPR lanes of a row group, with 3 + log2(LPR/4) shuffles instead of
// 4*log2(LPR): lanes trade halves of the batch first.  Lane `lig` returns the total of value lig / (LPR/4).
// All 32 lanes of the warp must call it.
template <int LPR>
__device__ __forceinline__ float reduce4(float s0, float s1, float s2, float s3, int lig) {
  const bool hi = (lig & (LPR / 2)) != 0;
  float k0 = hi ? s2 : s0, k1 = hi ? s3 : s1;
  const float t0 = hi ? s0 : s2, t1 = hi ? s1 : s3;
  k0 += __shfl_xor_sync(0xffffffffu, t0, LPR / 2);
  k1 += __shfl_xor_sync(0xffffffffu, t1, LPR / 2);
  const bool hi2 = (lig & (LPR / 4)) != 0;
  float k = hi2 ? k1 : k0;
  const float t = hi2 ? k0 : k1;
  k += __shfl_xor_sync(0xffffffffu, t, LPR / 4);
#pragma unroll
  for (int o = LPR / 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  return k;
}

// 2-D tiled load with an L2 eviction-priority hint; x = innermost coordinate (elements), y = row
__device__ __forceinline__ void tma_load_2d_hint(void* dst, const CUtensorMap* map, int x, int y, unsigned long long* bar,
                                                 unsigned long long policy) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;"
               ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(policy) : "memory");
}

// One warp-level tensor-core step for the logits of 16 rows against up to 8 heads: acc (16 x 8, fp32) += A (16 rows x
// 16 elements of d, from the row-major stage) * B (16 elements x 8 heads, the queries).  Both operands take their
// 16-byte pieces from the same offsets of their rows, so the order of the elements inside a step is free and a
// thread's piece is one contiguous vector load.
// the same step with a zero accumulator on input: d = a * b
template <typename T>
__device__ __forceinline__ void mma_16x8x16_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                 uint32_t b0, uint32_t b1) {
  if constexpr (sizeof(T) == 2 && !cuda::std::is_same<T, __nv_bfloat16>::value) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
  } else {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
  }
}
template <typename T>
__device__ __forceinline__ void mma_16x8x16(float (&acc)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                            uint32_t b0, uint32_t b1) {
  if constexpr (sizeof(T) == 2 && !cuda::std::is_same<T, __nv_bfloat16>::value) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  } else {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
}

// (hi, lo) 16-bit pairs of two fp32 weights, hi + lo carrying 16 (bf16) or 22 (fp16) significant bits: x -> low half
template <typename T>
__device__ __forceinline__ void split_pair(float x, float y, uint32_t& hi, uint32_t& lo) {
  if constexpr (cuda::std::is_same<T, __nv_bfloat16>::value) {
    // hi = the upper 16 bits (the subtraction is then exact), lo = the remainder rounded
    const uint32_t xb = __float_as_uint(x) & 0xffff0000u, yb = __float_as_uint(y) & 0xffff0000u;
    hi = (xb >> 16) | yb;
    const __nv_bfloat162 l = __floats2bfloat162_rn(x - __uint_as_float(xb), y - __uint_as_float(yb));
    lo = *reinterpret_cast<const uint32_t*>(&l);
  } else {
    const __half xh = __float2half_rn(x), yh = __float2half_rn(y);
    const __half2 h = __halves2half2(xh, yh);
    const __half2 l = __halves2half2(__float2half_rn(x - __half2float(xh)), __float2half_rn(y - __half2float(yh)));
    hi = *reinterpret_cast<const uint32_t*>(&h); lo = *reinterpret_cast<const uint32_t*>(&l);
  }
}
// four 8x8 16-bit matrices, transposed on the way into registers (value rows become the A operand's columns)
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t saddr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(saddr) : "memory");
}

// Dot products of the 16 rows of tile `tile` of a swizzled stage ([d half][SR rows][128 bytes], 16-byte chunk c of
// row r at chunk c ^ (r & 7)) with the (up to 8) vectors whose fragments are in `qb`.  Thread (gid, tig) reads chunk
// 2 tig + (j & 1) of half j / 2 of rows gid and gid + 8 in step j: with the swizzle the eight lanes of a quarter-warp
// hit eight different bank groups.  The order of the elements inside a step is free as long as both operands agree,
// so a thread's piece is one vector load; `qb[j]` holds the same chunk of vector gid.
// acc[0], acc[1] = row gid of the tile against vectors 2 tig, 2 tig + 1; acc[2], acc[3] = row gid + 8.
template <typename T, int D, int SR>
__device__ __forceinline__ void tile_dots(const unsigned char* stage, int tile, const uint4 (&qb)[D / 32], float (&acc)[4]) {
  const int gid = (threadIdx.x & 31) >> 2, tig = threadIdx.x & 3;
  // all fragments first, then one tensor-core step per 16 elements of d, each into its own accumulator: neither
  // the loads nor the steps wait for one another
  uint4 A0[D / 32], A1[D / 32];
#pragma unroll
  for (int j = 0; j < D / 32; ++j) {
    const unsigned char* row = stage + (size_t)(j >> 1) * SR * 128 + (size_t)(tile * 16 + gid) * 128 +
                               (((2 * tig + (j & 1)) ^ gid) << 4);
    A0[j] = *reinterpret_cast<const uint4*>(row);
    A1[j] = *reinterpret_cast<const uint4*>(row + 8 * 128);
  }
  float part[D / 16][4];
#pragma unroll
  for (int j = 0; j < D / 32; ++j) {
    mma_16x8x16_zero<T>(part[2 * j], A0[j].x, A1[j].x, A0[j].y, A1[j].y, qb[j].x, qb[j].y);
    mma_16x8x16_zero<T>(part[2 * j + 1], A0[j].z, A1[j].z, A0[j].w, A1[j].w, qb[j].z, qb[j].w);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < D / 16; ++i) t += part[i][e];
    acc[e] = t;
  }
}

}  // namespace d2o
