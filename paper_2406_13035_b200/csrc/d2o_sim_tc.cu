// Nearest-neighbour matching at the prompt stage (Section 4.2, Eq. 9) for 16-bit keys on the
// 5th-generation tensor cores: U = K_e K_c^T as tcgen05.mma (kind::f16, fp32 accumulators in tensor
// memory), fused with the scaling by the inverse key norms and the row max / arg-max.
//
// The evicted keys are most of the prompt (80 - 95 % at the cache ratios of interest), in prompt
// order.  Instead of gathering them, the kernel multiplies ALL prompt rows of a slice with the
// retained keys and lets the consumer pick the evicted positions: the A operand is then a plain
// tiled TMA load of 128 consecutive prompt rows, and the few retained rows among them cost
// S/P extra work.
//
// One CTA = one work item = (slice, chunk of up to 384 retained rows, range of 128-row prompt tiles); the host
// cuts every (slice, chunk) into ranges of about equal work once the budgets are known (sim_tc_build_items).
//   warp 0      TMA producer: the retained chunk once (B operand, stays in shared memory), then the prompt tiles
//               (A operand) into four slots, one per part; 128-byte swizzled K-major tiles
//   warp 1      allocates tensor memory, issues tcgen05.mma: one job = 128 x 128 x d (d/16 instructions) into the
//               part's own 128-column accumulator, the parts in turn
//   warps 2-17  epilogue: four parts of four warps.  A part owns every fourth prompt tile; each of its threads owns
//               one row (tensor-memory lane) of that tile and scans all retained columns of it, job after job:
//               tcgen05.ld of the accumulator, times 1/|k_c| per column, running max and arg-max (ties -> lowest
//               slot) in registers.  No exchange between warps and no barrier per tile; while one part drains its
//               accumulator the tensor cores work for the other three.
// Output: for every prompt position of the tile range and this chunk, the packed key
// (ordered max_j k_i.k_j/|k_j|, 0x7fffffff - slot).  neighbour_reduce_kernel takes the maximum over
// the chunks at the evicted positions and multiplies by 1/|k_i|.
#include <cuda.h>
#include <limits.h>
#include <math.h>
#include <stdlib.h>

#include <algorithm>
#include <cuda/std/type_traits>
#include <utility>
#include <vector>

#include "d2o_common.cuh"
#include "d2o_tc.cuh"

namespace d2o {

constexpr int kTcEpiWarps = 16;             // four per quarter of the tensor-memory lanes
constexpr int kTcThreads = (2 + kTcEpiWarps) * 32;
constexpr int kTileM = 128;                 // prompt rows per A tile
constexpr int kJobN = 128;                  // retained rows per MMA job (one 128 x 128 fp32 accumulator)
constexpr int kChunkN = 384;                // retained rows resident per CTA (96 KB for d = 128)
constexpr int kBBoxRows = 64;               // rows per TMA box of the B operand
constexpr int kParts = 4;                   // prompt tiles in flight: each with its own accumulator and four epilogue warps

struct SimTcArgs {
  const int32_t* budgets; const int64_t* row_off;
  const float* rnorm;                       // pool-wide 1/|k_c|
  unsigned long long* part_key;             // [slices][n_chunks_max][P]
  float* prompt_rn;                         // [slices][P] 1/|k| of the prompt rows (written with chunk 0)
  size_t stride;                            // bytes between two layers' part_key, prompt_rn
  uint32_t* status;
  const int32_t* plen;                      // [B] prompt length of every sequence; P is the row stride per slice
  const int4* items;                        // work lists of the layers of the launch: (slice, chunk, first tile, end tile) per CTA
  int item0[kCompressLayers];               // first item of every layer
  int n, L, layer0, Hkv, P, n_chunks_max;
};
struct SimTcMaps {
  CUtensorMap k[kCompressLayers], pool;     // prompt rows per layer; the cache rows
};

// Retained rows per chunk for a slice of S rows: ceil(S / kChunkN) chunks of equal size, rounded up to the MMA's
// column granularity.
__host__ __device__ __forceinline__ int chunk_columns(int S) {
  const int n_chunks = (S + kChunkN - 1) / kChunkN;
  return (((S + n_chunks - 1) / n_chunks) + 15) & ~15;
}

// (x0, x1) = (a0 * b0, a1 * b1), each product rounded to nearest as a single multiply would.
__device__ __forceinline__ void mul_pair(float a0, float a1, float b0, float b1, float& x0, float& x1) {
  unsigned long long a, b, d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(a0), "f"(a1));
  asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(b0), "f"(b1));
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(d));
}

// Maximum of three; a NaN operand is ignored.
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Running maximum over the columns of a job, for one row.  Columns go in pairs (2i, 2i + 1): one packed multiply, one three-input
// maximum against the running value, one compare and two selects per pair.  A chain remembers the winning pair and that pair's
// first value, from which the column inside the pair follows at the end.  Two chains (pairs i mod 2) keep them short.  max.f32
// drops a NaN operand, as a compare would.
struct JobMax {
  float pb[2], plo[2]; int pi[2];
  __device__ __forceinline__ void start() {
#pragma unroll
    for (int w = 0; w < 2; ++w) { pb[w] = plo[w] = -INFINITY; pi[w] = w; }
  }
  // Block `b` of 32 columns of the job: accumulators r times 1/|k_c| (s_rn: those of the block).  MASK: columns from `n` on hold other
  // slices' rows.
  template <bool MASK>
  __device__ __forceinline__ void block(const uint32_t (&r)[32], const float* s_rn, int b, int n) {
    const float4* rn4 = reinterpret_cast<const float4*>(s_rn);
#pragma unroll
    for (int i4 = 0; i4 < 8; ++i4) {
      const float4 q = rn4[i4];
      const float rv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int at = i4 * 4 + 2 * w;
        float x0, x1;
        mul_pair(__uint_as_float(r[at]), __uint_as_float(r[at + 1]), rv[2 * w], rv[2 * w + 1], x0, x1);
        if (MASK) { x0 = at < n ? x0 : -INFINITY; x1 = at + 1 < n ? x1 : -INFINITY; }
        const float m = max3(pb[w], x0, x1);
        const bool up = m > pb[w];
        pi[w] = up ? b * 16 + i4 * 2 + w : pi[w];
        plo[w] = up ? x0 : plo[w];
        pb[w] = m;
      }
    }
  }
  // Merged into the row's (best, best_col); col0: the job's first column.  The later chain wins only with a larger value or an
  // equal one from an earlier pair; equal values inside a pair go to the lower column; the first of equal jobs stays.
  __device__ __forceinline__ void finish(int col0, float& best, int& best_col) {
    if (pb[1] > pb[0] || (pb[1] == pb[0] && pi[1] < pi[0])) { pb[0] = pb[1]; pi[0] = pi[1]; plo[0] = plo[1]; }
    if (pb[0] > best) { best = pb[0]; best_col = col0 + 2 * pi[0] + (plo[0] == pb[0] ? 0 : 1); }
  }
};

template <typename T, int D, int FMT>
__global__ void __launch_bounds__(kTcThreads, 1)
sim_tc_kernel(SimTcArgs a, const __grid_constant__ SimTcMaps maps) {
  constexpr int KB = D / 64;                                 // 64-element (128-byte) blocks along d
  constexpr int A_BLOCK = kTileM * 128;                      // bytes of one A k-block
  constexpr int A_TILE = KB * A_BLOCK;
  constexpr int B_BLOCK = kChunkN * 128;                     // bytes of one B k-block (all chunk rows)

  extern __shared__ __align__(1024) unsigned char tc_smem[];
  unsigned char* sB = tc_smem;                               // [KB][kChunkN rows][128 B]
  unsigned char* sA = tc_smem + KB * B_BLOCK;                // [kParts][KB][128 rows][128 B]: the prompt tile of each part
  float* s_rn = reinterpret_cast<float*>(sA + kParts * A_TILE);                    // [kChunkN] 1/|k_c| of the chunk
  __shared__ unsigned long long b_full, a_full[kParts], a_empty[kParts], tm_full[kParts], tm_empty[kParts];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // No start_dependents: the reduction's CTAs would wait in the SMs for all of this kernel's run, and it is the slower for it
  // (32 slices of 5000 tokens, two layers, all of the compression: 159 us instead of 143).
  wait_for_prior_grid();
  const int4 item = a.items[blockIdx.x];
  int z = 0;                                                 // layer of the launch
  while (z + 1 < a.n && (int)blockIdx.x >= a.item0[z + 1]) ++z;
  const int layer = a.layer0 + z;
  const int slice = item.x;
  const int nc = item.y;
  const int b = slice / a.Hkv, h = slice % a.Hkv;
  const int S = a.budgets[slice_entry(b, layer, h, a.L, a.Hkv)];
  const int chunk_cols = chunk_columns(S);                   // the retained rows are split evenly over the chunks
  const int c0 = nc * chunk_cols;                            // first retained slot of the chunk
  const int Pb = a.plen[b];                                  // this sequence's prompt length
  if (c0 >= S || Pb - S <= 0) return;                        // uniform for the CTA: nothing to do
  const int n_cols = min(chunk_cols, S - c0);
  const int n_j = (n_cols + kJobN - 1) / kJobN;              // MMA column tiles (jobs) per prompt tile: 1 .. 3
  const int job_w = ((n_cols + n_j - 1) / n_j + 31) & ~31;   // columns of a job: about the same for all
  const int n_last = (n_cols - (n_j - 1) * job_w + 15) & ~15;    // of the last one's MMA (multiple of 16)
  const int n_tiles_all = (Pb + kTileM - 1) / kTileM;
  const int t0 = item.z;
  const int t1 = min(n_tiles_all, item.w);
  if (t0 >= t1) return;
  const int n_t = t1 - t0;                                     // prompt tiles of this CTA; part p takes tiles p, p + 4, ...
  const int64_t row0 = a.row_off[slice_entry(b, layer, h, a.L, a.Hkv)];
  if ((tc::smem_u32(tc_smem) & 1023u) != 0u) {               // swizzled tiles need 1024-byte aligned shared memory
    if (tid == 0) report_error(a.status, D2O_ERR_STATE, 0x51C10000u);
    return;
  }

  if (tid == 0) {
    s_fail = 0;
    tc::mbar_init(&b_full, 1);
    for (int p = 0; p < kParts; ++p) {
      tc::mbar_init(&a_full[p], 1); tc::mbar_init(&a_empty[p], nc == 0 ? 1 + kTcEpiWarps / kParts : 1);
      tc::mbar_init(&tm_full[p], 1); tc::mbar_init(&tm_empty[p], kTcEpiWarps / kParts);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {                                           // 512 columns: one 128 x 128 fp32 accumulator per part
    tc::tmem_alloc(&s_tmem, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem_base = s_tmem;

  if (warp == 0) {
    // ======================================================================= TMA producer
    if (lane == 0) {
      const int n_box = (n_cols + kBBoxRows - 1) / kBBoxRows;    // rows past the slice's S are other slices' rows: never used
      tc::mbar_expect_tx(&b_full, (uint32_t)(KB * n_box * kBBoxRows * 128));
      for (int kb = 0; kb < KB; ++kb)
        for (int j = 0; j < n_box; ++j)
          tc::tma_load_2d(sB + kb * B_BLOCK + j * kBBoxRows * 128, &maps.pool, kb * 64, (int)(row0 + c0 + j * kBBoxRows), &b_full);
      for (int i = 0; i < n_t; ++i) {                            // tile i goes to part i % 4, its k-th tile with k = i / 4
        const int p = i % kParts, k = i / kParts;
        if (k >= 1 && !s_fail && !tc::mbar_wait(&a_empty[p], (uint32_t)((k - 1) & 1))) s_fail = 1;
        tc::mbar_expect_tx(&a_full[p], (uint32_t)A_TILE);
        for (int kb = 0; kb < KB; ++kb)
          tc::tma_load_2d(sA + p * A_TILE + kb * A_BLOCK, &maps.k[z], kb * 64, slice * a.P + (t0 + i) * kTileM, &a_full[p]);
      }
    }
  } else if (warp == 1) {
    // ======================================================================= MMA issuer
    // Jobs are issued part by part in turn, so that while one part's epilogue drains its accumulator the tensor
    // cores work for the other three.
    if (lane == 0) {
      if (!tc::mbar_wait(&b_full, 0)) s_fail = 1;
      const int rounds = (n_t + kParts - 1) / kParts;
      for (int k = 0; k < rounds; ++k)
        for (int j = 0; j < n_j; ++j)
          for (int p = 0; p < kParts; ++p) {
            if (k * kParts + p >= n_t) continue;
            if (j == 0 && !s_fail && !tc::mbar_wait(&a_full[p], (uint32_t)(k & 1))) s_fail = 1;
            const int cnt = k * n_j + j;                         // jobs issued to this part before this one
            // the part's epilogue must have drained its accumulator (the first use passes at once)
            if (!s_fail && !tc::mbar_wait(&tm_empty[p], (uint32_t)((cnt & 1) ^ 1))) s_fail = 1;
            tc::fence_after_sync();
            const uint32_t d_tmem = tmem_base + (uint32_t)(p * kJobN);
            const uint32_t idesc = make_idesc(FMT, kTileM, j == n_j - 1 ? (uint32_t)n_last : (uint32_t)job_w);
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
              const uint64_t adesc = tc::smem_desc_sw128(tc::smem_u32(sA + p * A_TILE + kb * A_BLOCK));
              const uint64_t bdesc = tc::smem_desc_sw128(tc::smem_u32(sB + kb * B_BLOCK + j * job_w * 128));
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)                     // 16 elements = 32 bytes along K per instruction
                tc::mma_f16(d_tmem, adesc + (uint64_t)(2 * kk), bdesc + (uint64_t)(2 * kk), idesc, (kb | kk) != 0 ? 1u : 0u);
            }
            tc::mma_commit(&tm_full[p]);
            if (j == n_j - 1) tc::mma_commit(&a_empty[p]);       // the tile's slot is free once its MMAs have read it
          }
    }
  } else {
    // ======================================================================= epilogue warps
    // Four warps per part, one per quarter of the tensor-memory lanes: a thread owns one row of its part's prompt
    // tile and scans all retained columns of it, job after job, so that the row's maximum never leaves its registers
    // (no exchange between warps, no barrier per tile).
    const int e = warp - 2;
    const int quarter = warp & 3;                            // tensor-memory lanes this warp may read: 32*quarter ..
    const int p = e >> 2;                                    // part
    const int row = quarter * 32 + lane;                     // row of the prompt tile owned by this thread
    for (int i = tid - 64; i < kChunkN; i += kTcEpiWarps * 32)
      s_rn[i] = i < n_cols ? a.rnorm[row0 + c0 + i] : 0.f;
    asm volatile("bar.sync 1, %0;" ::"n"(kTcEpiWarps * 32) : "memory");
    unsigned long long* out_keys = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(a.part_key) + a.stride * z) +
                                   ((size_t)slice * a.n_chunks_max + nc) * a.P;
    float* out_rn = reinterpret_cast<float*>(reinterpret_cast<char*>(a.prompt_rn) + a.stride * z) + (size_t)slice * a.P;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(p * kJobN);
    const int n_tp = p < n_t ? (n_t - p + kParts - 1) / kParts : 0;   // tiles of this part
    // every load of a job has landed in registers: hand the accumulator back to the MMA warp
    auto release = [&]() {
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&tm_empty[p]);
    };
#pragma unroll 1
    for (int k = 0; k < n_tp; ++k) {
      float best = -INFINITY; int best_col = 0x7fffffff;
      const int pos = (t0 + k * kParts + p) * kTileM + row;
      if (nc == 0) {
        // 1/|k| of this thread's prompt row, from the tile itself (16-byte segment c of a row at c ^ (row & 7)), while the
        // tensor cores work on it: the reduction then reads 4 bytes per evicted row instead of its key.  One sum per segment
        // and then the tree of gather_kernel: both sides of a cosine round alike, with less error than one chain of 128 terms
        // (1/|k| of random bf16 rows, d = 128: 4.0e-8 rms, the chain 9.9e-8).
        if (!s_fail && !tc::mbar_wait(&a_full[p], (uint32_t)(k & 1))) s_fail = 1;
        float seg[8];
#pragma unroll
        for (int kb = 0; kb < KB; ++kb) {
          const unsigned char* r = sA + p * A_TILE + kb * A_BLOCK + row * 128;
#pragma unroll
          for (int cc = 0; cc < 8; ++cc) {
            float f[8], ss = 0.f;
            Elem<T>::unpack(*reinterpret_cast<const uint4*>(r + ((cc ^ (row & 7)) << 4)), f);
#pragma unroll
            for (int i = 0; i < 8; ++i) ss = fmaf(f[i], f[i], ss);
            seg[cc] = kb == 0 ? ss : seg[cc] + ss;
          }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&a_empty[p]);
        const float ss = ((seg[0] + seg[4]) + (seg[2] + seg[6])) + ((seg[1] + seg[5]) + (seg[3] + seg[7]));
        if (pos < Pb) out_rn[pos] = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
      }
#pragma unroll 1
      for (int j = 0; j < n_j; ++j) {
        const int cnt = k * n_j + j;
        if (!s_fail && !tc::mbar_wait(&tm_full[p], (uint32_t)(cnt & 1))) s_fail = 1;
        tc::fence_after_sync();
        const int cl = j * job_w;                              // chunk-local column of the job's first block
        const int cols = min(job_w, n_cols - cl);              // its columns with retained rows: up to four blocks of 32
        // One straight path per number of blocks, with registers of its own; loads run one block ahead of the scan.  us of
        // compression, conditional loads into shared registers, a merge per block and jobs of 128 columns and a rest / so: three
        // layers of 48 slices of 5000 tokens, d = 64, 293 / 278; two of 32 slices of 3000 tokens 145.7 / 142.4; 32 layers of 32 slices of
        // 1200 tokens, the whole prompt stage, 1149 / 1135; four of 128 slices of 8192 tokens 1703 / 1704 and 1691 / 1682.
        auto job = [&](auto blocks) {
          constexpr int NB = decltype(blocks)::value;
          uint32_t r[2][32];
          JobMax mx;
          mx.start();
          tc::tmem_ld32_issue(lane_base, r[0]);
          tc::tmem_ld_wait(r[0]);
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            if (b + 1 < NB) tc::tmem_ld32_issue(lane_base + (uint32_t)(b + 1) * 32u, r[(b + 1) & 1]); else release();
            if (b + 1 < NB || cols == NB * 32) mx.block<false>(r[b & 1], s_rn + cl + b * 32, b, 32);
            else mx.block<true>(r[b & 1], s_rn + cl + b * 32, b, cols - b * 32);
            if (b + 1 < NB) tc::tmem_ld_wait(r[(b + 1) & 1]);
          }
          mx.finish(c0 + cl, best, best_col);
        };
        switch ((cols + 31) / 32) {
          case 4: job(cuda::std::integral_constant<int, 4>()); break;
          case 3: job(cuda::std::integral_constant<int, 3>()); break;
          case 2: job(cuda::std::integral_constant<int, 2>()); break;
          default: job(cuda::std::integral_constant<int, 1>()); break;
        }
      }
      // (ordered value, inverted slot): larger is better, ties go to the lower slot; -0 counts as +0
      if (best == 0.f) best = 0.f;
      const unsigned long long key = best > -INFINITY
          ? (((unsigned long long)float_ord(best) << 32) | (uint32_t)(0x7fffffff - best_col)) : 0ull;
      if (pos < Pb) out_keys[pos] = key;
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem_base, 512);
  }
  if (tid == 0 && s_fail) report_error(a.status, D2O_ERR_TIMEOUT, 0x51C00000u | (uint32_t)(slice & 0xfffff));
}

// mx_i = 1/|k_i| * max over the chunks of the partial maxima, nn_i = its slot, for the evicted positions.
struct NnReduceArgs {
  const int32_t* budgets; const int64_t* row_off;
  const int32_t* evict_idx;
  const unsigned long long* part_key;
  const float* prompt_rn;                   // 1/|k| of the prompt rows
  const float* rnorm;                       // pool-wide 1/|k_c|
  float* evict_mx; int32_t* evict_nn;
  size_t stride;                            // bytes between two layers' working arrays
  uint32_t* status;
  const int32_t* plen;
  int L, layer0, Hkv, P, n_chunks_max;
  const void* K[kCompressLayers];
};

// One evicted row per thread: the positions ascend, so that neighbouring threads read neighbouring entries.  (With 16 lanes
// per row, which read the row's key for its norm, the kernel took 138 us on 128 slices of 8192 tokens; the chain position ->
// key and partial maxima is what it waited for.)
template <typename T, int D>
__global__ void __launch_bounds__(256)
neighbour_reduce_kernel(NnReduceArgs a, const T* kpool) {
  constexpr int EPV = Elem<T>::kPerVec;
  start_dependents();
  wait_for_prior_grid();
  const int slice = blockIdx.y, z = blockIdx.z, layer = a.layer0 + z;
  const int b = slice / a.Hkv, h = slice % a.Hkv;
  const int S = a.budgets[slice_entry(b, layer, h, a.L, a.Hkv)];
  const int Pb = a.plen[b];
  const int Le = Pb - S;
  if ((int)(blockIdx.x * blockDim.x) >= Le) return;
  auto lane_of = [&](const void* p) { return reinterpret_cast<const char*>(p) + a.stride * z; };
  const int32_t* evict_idx = reinterpret_cast<const int32_t*>(lane_of(a.evict_idx)) + (size_t)slice * a.P;
  const unsigned long long* part_key = reinterpret_cast<const unsigned long long*>(lane_of(a.part_key)) + (size_t)slice * a.n_chunks_max * a.P;
  const float* prompt_rn = reinterpret_cast<const float*>(lane_of(a.prompt_rn)) + (size_t)slice * a.P;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const int n_chunks = (S + kChunkN - 1) / kChunkN;
  int pos = i < Le ? evict_idx[i] : -1;
  if (pos >= 0 && !D2O_GUARD(pos < Pb, a.status, 0xC4EC0008u)) pos = -1;
  unsigned long long key = 0ull;
  float rn = 0.f;
  if (pos >= 0) {
    rn = prompt_rn[pos];
    for (int c = 0; c < n_chunks; ++c) {
      const unsigned long long k2 = part_key[(size_t)c * a.P + pos];
      key = k2 > key ? k2 : key;
    }
  }
  int slot = 0x7fffffff - (int)(uint32_t)(key & 0xffffffffu);
  float mx = ord_float((uint32_t)(key >> 32)) * rn;
  // No chunk reported a maximum (no finite similarity in the row: non-finite keys).  The row is redone by the whole warp in
  // fp32, all retained rows in slot order (the first maximum stays); without any finite similarity it gets maximum -inf and
  // neighbour 0 and is never merged.
  unsigned redo = __ballot_sync(0xffffffffu, pos >= 0 && !(key != 0ull && (unsigned)slot < (unsigned)S));
  while (redo) {
    const int src = __ffs(redo) - 1;
    redo &= redo - 1;
    const int rp = __shfl_sync(0xffffffffu, pos, src);
    const float rr = __shfl_sync(0xffffffffu, rn, src);
    const T* row = (const T*)a.K[z] + ((size_t)slice * a.P + rp) * D;
    const int64_t row0 = a.row_off[slice_entry(b, layer, h, a.L, a.Hkv)];
    float best = -INFINITY; int bj = 0;
    for (int j = 0; j < S; ++j) {
      float dot = 0.f;
      if (lane < D / EPV) {
        float f[EPV], g[EPV];
        Elem<T>::unpack(ld_global_v4(row + lane * EPV), f);
        Elem<T>::unpack(ld_global_v4(kpool + (row0 + j) * D + lane * EPV), g);
#pragma unroll
        for (int e = 0; e < EPV; ++e) dot = fmaf(f[e], g[e], dot);
      }
      dot = warp_sum(dot);
      const float u = __fadd_rn(dot * rr * a.rnorm[row0 + j], 0.f);
      if (u > best) { best = u; bj = j; }
    }
    if (lane == src) { mx = best; slot = bj; }
  }
  if (pos >= 0) {
    (reinterpret_cast<float*>(reinterpret_cast<char*>(a.evict_mx) + a.stride * z) + (size_t)slice * a.P)[i] = mx;
    (reinterpret_cast<int32_t*>(reinterpret_cast<char*>(a.evict_nn) + a.stride * z) + (size_t)slice * a.P)[i] = slot;
  }
}

// ------------------------------------------------------------------------------------ host side
// The driver's tensor-map encoder, looked up through the runtime so that the library has no link-time dependency
// on the driver (it must load, and reject calls with status codes, on machines without one).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

bool encode_rows_2d(CUtensorMap* map, int dtype, const void* base, uint64_t rows, int d, int box_rows) {
  EncodeTiledFn encode = encode_tiled_fn();
  if (!encode) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1u, 1u};
  const CUtensorMapDataType dt = dtype == D2O_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  return encode(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Upper bound of the work items of one layer: one per (slice, chunk) plus the splits into tile ranges.
size_t sim_tc_max_items(const d2o_config* cfg, int max_budget) {
  const size_t chunks = ((size_t)max_budget + kChunkN - 1) / kChunkN;
  return (size_t)cfg->batch * cfg->n_kv_heads * chunks + 2048;
}

// The work lists of all layers, built on the host once the budgets are known: every (slice, chunk of retained rows)
// is cut into ranges of prompt tiles of about equal work (tiles x columns), so that one launch is several full waves
// of CTAs of the same length whatever the spread of the budgets; longest first.  The lists lie one after another in
// `items` (room for n_layers * sim_tc_max_items() entries); `count[layer]` and `first[layer]` describe each.  Returns the
// entries of all layers.
size_t sim_tc_build_items(const d2o_ctx* c, int n_sms, int4* items, int32_t* count, int32_t* first) {
  const d2o_config& g = c->cfg;
  const int B = g.batch, Hkv = g.n_kv_heads, L = g.n_layers;
  const size_t cap = sim_tc_max_items(&g, c->max_budget);
  struct Piece { int slice, chunk, tiles, cols; };
  std::vector<Piece> pieces;
  std::vector<std::pair<double, int4>> list;
  size_t n = 0;
  for (int layer = 0; layer < L; ++layer) {
    pieces.clear();
    list.clear();
    double total = 0.0;
    for (int b = 0; b < B; ++b)
      for (int h = 0; h < Hkv; ++h) {
        const int S = c->h_budgets[((size_t)b * L + layer) * Hkv + h];
        const int P = c->h_plen[b];
        if (P - S <= 0) continue;
        const int n_chunks = (S + kChunkN - 1) / kChunkN, cc = chunk_columns(S);
        const int tiles = (P + kTileM - 1) / kTileM;
        for (int nc = 0; nc < n_chunks; ++nc) {
          const int cols = min(cc, S - nc * cc);
          if (cols <= 0) continue;
          pieces.push_back({b * Hkv + h, nc, tiles, cols});
          total += (double)tiles * (cols + 64);                // + a per-tile cost that does not depend on the columns
        }
      }
    // Aim at two waves of equal items per layer (the layers of a launch follow one another), at least eight tiles each: a CTA
    // costs about 10 us before its first and after its last tile (128 slices of 8192 tokens, four layers, compression as a
    // whole: 1900 us with five waves, 1860 with three, 1850 with two).
    const double target = total / ((double)n_sms * 2.0);
    for (size_t i = 0; i < pieces.size(); ++i) {
      const Piece& p = pieces[i];
      const double work = (double)p.tiles * (p.cols + 64);
      int k = (int)(work / target + 0.5);
      k = max(1, min(k, max(1, p.tiles / 8)));
      if (list.size() + k + (pieces.size() - i) > cap) k = 1;  // never more entries than the list holds
      for (int j = 0; j < k; ++j) {
        const int t0 = (int)((long long)p.tiles * j / k), t1 = (int)((long long)p.tiles * (j + 1) / k);
        if (t1 > t0) list.push_back({(double)(t1 - t0) * (p.cols + 64), make_int4(p.slice, p.chunk, t0, t1)});
      }
    }
    // longest first; ties keep the slice order
    std::stable_sort(list.begin(), list.end(),
                     [](const std::pair<double, int4>& x, const std::pair<double, int4>& y) { return x.first > y.first; });
    first[layer] = (int32_t)n;
    count[layer] = (int32_t)list.size();
    for (const auto& e : list) items[n++] = e.second;
  }
  return n;
}

size_t sim_tc_part_key_bytes(const d2o_config* cfg, int max_budget) {
  const size_t chunks = ((size_t)max_budget + kChunkN - 1) / kChunkN;
  return (size_t)cfg->batch * cfg->n_kv_heads * chunks * cfg->prompt_len * 8;
}

// Layers [layer, layer + n) in one launch per kernel.  Returns cudaErrorNotSupported if the tensor maps cannot be built.
cudaError_t launch_similarity_tc(const d2o_ctx* c, int layer, int n, const void* const* K, int max_evicted, cudaStream_t st) {
  const d2o_config& g = c->cfg;
  const int B = g.batch, Hkv = g.n_kv_heads, P = g.prompt_len, D = g.d_head;
  const int n_slices = B * Hkv;
  char* S = c->state; char* X = c->scratch;
  SimTcMaps maps;
  // the retained rows of the same kind: K_c, or V_c when the similarity is taken on the values
  char* pool = S + (g.sim_feature ? c->lay.vpool : c->lay.kpool);
  if (!encode_rows_2d(&maps.pool, g.dtype, pool, (uint64_t)c->pool_rows, D, kBBoxRows)) return cudaErrorNotSupported;
  SimTcArgs a;
  NnReduceArgs r;
  int n_items = 0;
  for (int l = 0; l < n; ++l) {
    if (!encode_rows_2d(&maps.k[l], g.dtype, K[l], (uint64_t)n_slices * P, D, kTileM)) return cudaErrorNotSupported;
    a.item0[l] = n_items;
    n_items += c->h_sim_count[layer + l];
    r.K[l] = K[l];
  }
  if (n_items == 0) return cudaSuccess;                      // nothing was evicted in these layers
  a.budgets = (const int32_t*)(S + c->lay.budgets); a.row_off = (const int64_t*)(S + c->lay.row_off);
  a.rnorm = (const float*)(S + c->lay.rnorm);
  a.part_key = (unsigned long long*)(X + c->slay.part_key);
  a.prompt_rn = (float*)(X + c->slay.prompt_rn);
  a.stride = c->slay.lane_stride;
  a.status = (uint32_t*)(S + c->lay.status);
  a.plen = (const int32_t*)(S + c->lay.plen);
  a.n = n; a.L = g.n_layers; a.layer0 = layer; a.Hkv = Hkv; a.P = P; a.n_chunks_max = (c->max_budget + kChunkN - 1) / kChunkN;
  a.items = (const int4*)(S + c->lay.sim_items) + c->h_sim_off[layer];
  const int KB = D / 64;
  const size_t smem = (size_t)KB * kChunkN * 128 + (size_t)kParts * KB * kTileM * 128 + kChunkN * 4;
  dim3 grid((unsigned)n_items);
  cudaError_t e;
#define D2O_LAUNCH_TC(TT, DD, FF)                                                                                     \
  do {                                                                                                                \
    e = cudaFuncSetAttribute(sim_tc_kernel<TT, DD, FF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);      \
    if (e != cudaSuccess) return e;                                                                                   \
    e = launch_behind(sim_tc_kernel<TT, DD, FF>, grid, kTcThreads, smem, st, a, maps);                                \
    if (e != cudaSuccess) return e;                                                                                   \
  } while (0)
  if (D == 128) { if (g.dtype == D2O_F16) D2O_LAUNCH_TC(__half, 128, 0); else D2O_LAUNCH_TC(__nv_bfloat16, 128, 1); }
  else          { if (g.dtype == D2O_F16) D2O_LAUNCH_TC(__half, 64, 0); else D2O_LAUNCH_TC(__nv_bfloat16, 64, 1); }
#undef D2O_LAUNCH_TC

  r.budgets = a.budgets; r.row_off = a.row_off; r.rnorm = a.rnorm; r.status = a.status; r.plen = a.plen;
  r.evict_idx = (const int32_t*)(X + c->slay.evict_idx); r.part_key = a.part_key; r.prompt_rn = a.prompt_rn;
  r.evict_mx = (float*)(X + c->slay.evict_mx); r.evict_nn = (int32_t*)(X + c->slay.evict_nn); r.stride = a.stride;
  r.L = g.n_layers; r.layer0 = layer; r.Hkv = Hkv; r.P = P; r.n_chunks_max = a.n_chunks_max;
  dim3 rgrid((unsigned)((max_evicted + 255) / 256), (unsigned)n_slices, (unsigned)n);
  if (g.dtype == D2O_F16) {
    if (D == 128) e = launch_behind(neighbour_reduce_kernel<__half, 128>, rgrid, 256, 0, st, r, (const __half*)pool);
    else e = launch_behind(neighbour_reduce_kernel<__half, 64>, rgrid, 256, 0, st, r, (const __half*)pool);
  } else {
    if (D == 128) e = launch_behind(neighbour_reduce_kernel<__nv_bfloat16, 128>, rgrid, 256, 0, st, r, (const __nv_bfloat16*)pool);
    else e = launch_behind(neighbour_reduce_kernel<__nv_bfloat16, 64>, rgrid, 256, 0, st, r, (const __nv_bfloat16*)pool);
  }
  return e;
}

}  // namespace d2o
