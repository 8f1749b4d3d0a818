// Layer-level operation (Section 4.1): column sums of the causal prompt attention (Eq. 4 / Eq. 6
// case 1), the density F_v = Var(s) per query head, and the inverse-variance-softmax budgets
// (Eq. 5, Appendix A.2).
//
// Kernels in this file
//   sweep_kernel    row normalisers log sum_j exp(q_i.k_j/sqrt(d)) of the causal attention, and the
//                   column sums s_j = sum_{i>=j} exp(q_i.k_j/sqrt(d) - lse_i)
//   colsum_stored_kernel  the same column sums from dot products that the row sweep stored (fp32 caches)
//   density_kernel  warp-shuffle mean / variance of s per query head (double accumulation)
//   budget_kernel   Eq. 5 with clamping and exact-sum integerisation, one CTA per sequence
// The two attention sweeps here are the generic FFMA implementation (any dtype, fp32 math);
// 16-bit inputs take the tensor-core path of d2o_colsum_tc.cu.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "d2o_common.cuh"

namespace d2o {

namespace cg = cooperative_groups;

// Both sweeps multiply 64 x 64 tiles of the causal triangle: one tile stays (a row tile of Q for the normalisers, a column
// tile of K for the column sums), those of the other operand stream past it, and the reduction runs along the stream.
//
// A triangle of nT tiles has long and short strips.  Strips u and nT - 1 - u are nT + 1 tiles together for every u, so a
// pair is the unit of work; a cluster of C CTAs divides the pair's tiles evenly and combines its 128 results through
// distributed shared memory in rank order (no atomics, no scratch, the same bits every time).  With one CTA per strip the
// last of 16 strips was the launch.
//
// 128 threads hold 8 x 4 results each as two partial sums over the even and odd elements (fma.rn.f32x2 on operands as they
// lie in memory); tiles are copied as they are (cp.async, two buffers, one barrier per slab) into rows of d + 4 floats,
// which keeps the 16-byte reads of both operands free of bank conflicts.  The FMA pipe is busy 55 - 60 % of the time (twelve
// warps per SM wait for shared memory); 8 x 8 results on 64 threads were no faster for d = 64 and 25 % slower for d = 128.
// fp32, both sweeps (no products stored) and the densities, one CTA per strip -> so: 8 heads of 1024 tokens 132 -> 66 us, of 100
// tokens 29 -> 22; 16 heads of 1500 tokens, d = 128, 675 -> 334.
constexpr int kTile = 64;             // rows and columns per tile
constexpr int kStatThreads = 128;
constexpr int kStripA = 8, kStripB = 4;   // results per thread: rows of the resident tile x rows of the streaming tile
constexpr int kSlab = 64;                 // elements of d per streamed copy
constexpr int kMaxSweepCtas = 8;          // CTAs per cluster at most

template <int D> struct SweepSmem {
  static constexpr int kLdX = D + 4, kLdY = kSlab + 4;
  float x[kTile * kLdX], y[2][kTile * kLdY], yl[2][kTile];
  double res[2][2][kTile];            // column sums, or (maximum, sum) as two floats: [strip of the pair][half of the warps]
};

// Elements [0, W) of rows [row0, row0 + 64) of a [n_rows, D] matrix into shared memory; rows past the end are zero.  fp32
// rows travel asynchronously (the caller commits and waits), 16-bit rows are converted on the way.
template <typename T, int D, int W>
__device__ __forceinline__ void load_tile(float* t, const T* base, int row0, int n_rows) {
  constexpr int EPV = Elem<T>::kPerVec, VPR = W / EPV, LD = W + 4;
#pragma unroll 4
  for (int i = threadIdx.x; i < kTile * VPR; i += kStatThreads) {
    const int r = i / VPR, v = i % VPR;
    const bool in = row0 + r < n_rows;
    const T* src = base + (size_t)(in ? row0 + r : 0) * D + v * EPV;
    float* dst = t + r * LD + v * EPV;
    if (sizeof(T) == 4) {
      const uint32_t to = (uint32_t)__cvta_generic_to_shared(dst);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(src), "r"(in ? 16 : 0) : "memory");
    } else {
      float f[EPV];
      if (in) Elem<T>::unpack(ld_global_v4(src), f);
#pragma unroll
      for (int e = 0; e < EPV; ++e) dst[e] = in ? f[e] : 0.f;
    }
  }
}

// 2^x; terms below 2^-126 count as zero
__device__ __forceinline__ float exp2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (m, l) <- log2-domain maximum and sum of 2^(x - m) over two sets
__device__ __forceinline__ void combine_lse(float& m, float& l, float mo, float lo) {
  const float mn = fmaxf(m, mo);
  const float a = m > -INFINITY ? l * exp2f(m - mn) : 0.f;
  const float b = mo > -INFINITY ? lo * exp2f(mo - mn) : 0.f;
  l = a + b;
  m = mn;
}

// log2(e) / sqrt(d)
__host__ __device__ constexpr float logit_scale(int d) { return (d == 64 ? 0.125f : 0.08838834764831845f) * kLog2e; }

// tiles of the causal triangle of P rows
__host__ __device__ __forceinline__ size_t triangle_tiles(int P) { const size_t n = (size_t)(P + kTile - 1) / kTile; return n * (n + 1) / 2; }

// kSum: colsum_j = sum_{i >= j} exp(q_i.k_j / sqrt(d) - lse_i); else lse_i = log sum_{j <= i} exp(q_i.k_j / sqrt(d)).
template <typename T, int D, bool kSum>
__global__ void __launch_bounds__(kStatThreads, 3)
sweep_kernel(const T* Q, const T* K, const float* lse_in, float* __restrict__ out,    // inputs: see wait_for_prior_grid
             int Pmax, int Hq, int group, const int32_t* __restrict__ plen, int head0, float4* __restrict__ logits) {
  extern __shared__ __align__(16) unsigned char sweep_smem[];
  SweepSmem<D>& sm = *reinterpret_cast<SweepSmem<D>*>(sweep_smem);
  constexpr int LDX = SweepSmem<D>::kLdX, LDY = SweepSmem<D>::kLdY, kSlabs = D / kSlab;
  // The first kernel of a call: what is ahead of it may be writing Q and K, or reading the scratch of the call before.  Only its
  // launch overlaps with that (8 heads of 100 tokens 22.6 -> 20.6 us a call, of 1024 tokens 49.9 -> 49.6).  The kernel behind it
  // starts after this wait: the column sweep requests tiles of Q and K ahead of its own.
  if (!kSum) wait_for_prior_grid();
  start_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int u = blockIdx.x / C;
  const int bh = head0 + (int)blockIdx.y, b = bh / Hq, hq = bh % Hq;
  const int P = plen ? plen[b] : Pmax;                 // this sequence's prompt length; tensors are laid out for Pmax
  const int nT = (P + kTile - 1) / kTile;
  if (2 * u >= nT + (nT & 1)) return;                  // the whole cluster
  const T* q = Q + (size_t)bh * Pmax * D;
  const T* k = K + ((size_t)b * (Hq / group) + hq / group) * (size_t)Pmax * D;
  const float* ls = kSum ? lse_in + (size_t)bh * Pmax : nullptr;
  // strip `part` of the pair: its resident tile and its number of streamed tiles
  const int n0 = nT - u, n = u != nT - 1 - u ? nT + 1 : n0;
  auto resident = [&](int part) { return (part == 0) == kSum ? u : nT - 1 - u; };
  const int s0 = rank * n / C, s1 = (rank + 1) * n / C;
  // resident rows ty + 8 r, streamed rows tx + 16 c; a warp is 4 x 8 threads, the CTA 2 x 2 warps
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = warp >> 1;
  const int ty = (warp & 1) * 4 + (lane >> 3), tx = half * 8 + (lane & 7);
  const float mul = logit_scale(D);

#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    const int at = resident(part), from = part == 0 ? 0 : n0;
    const int i0 = max(s0, from) - from, i1 = min(s1, part == 0 ? n0 : n) - from;   // streamed tiles of this CTA
    float m[kStripA], l[kStripA];
    double acc[kStripA];
#pragma unroll
    for (int r = 0; r < kStripA; ++r) { m[r] = -INFINITY; l[r] = 0.f; acc[r] = 0.0; }
    auto request = [&](int step) {                    // slab `step` of the stream into its buffer
      const int i = i0 + step / kSlabs, row0 = (kSum ? at + i : i) * kTile, buf = step & 1;
      load_tile<T, D, kSlab>(sm.y[buf], (kSum ? q : k) + (step % kSlabs) * kSlab, row0, P);
      if (kSum && step == 0) wait_for_prior_grid();   // the normalisers
      if (kSum && step % kSlabs == kSlabs - 1 && threadIdx.x < kTile) {
        const bool in = row0 + (int)threadIdx.x < P;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(&sm.yl[buf][threadIdx.x])),
                       "l"(ls + (in ? row0 + (int)threadIdx.x : 0)), "r"(in ? 4 : 0) : "memory");
      }
    };
    if (i0 < i1) {
      load_tile<T, D, D>(sm.x, kSum ? k : q, at * kTile, P);
      request(0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int n_steps = (i1 - i0) * kSlabs;
    unsigned long long s[kStripA][kStripB];
#pragma unroll 1
    for (int step = 0; step < n_steps; ++step) {
      const int i = i0 + step / kSlabs, slab = step % kSlabs, buf = step & 1;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();                                // the slab is there; every warp is done with the one before it
      if (step + 1 < n_steps) request(step + 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (slab == 0) {
#pragma unroll
        for (int r = 0; r < kStripA; ++r)
#pragma unroll
          for (int c = 0; c < kStripB; ++c) s[r][c] = 0ull;
      }
      const float* xr = sm.x + ty * LDX + slab * kSlab;
      const float* yr = sm.y[buf] + tx * LDY;
#pragma unroll 4
      for (int e = 0; e < kSlab; e += 4) {
        ulonglong2 yv[kStripB];
#pragma unroll
        for (int c = 0; c < kStripB; ++c) yv[c] = *reinterpret_cast<const ulonglong2*>(yr + c * 16 * LDY + e);
#pragma unroll
        for (int r = 0; r < kStripA; ++r) {
          const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(xr + r * 8 * LDX + e);
#pragma unroll
          for (int c = 0; c < kStripB; ++c) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s[r][c]) : "l"(xv.x), "l"(yv[c].x));
#pragma unroll
          for (int c = 0; c < kStripB; ++c) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s[r][c]) : "l"(xv.y), "l"(yv[c].y));
        }
      }
      if (slab < kSlabs - 1) continue;
      // the tile on the diagonal, and the last rows of the prompt, need a mask
      const int res0 = at * kTile + ty, str0 = (kSum ? at + i : i) * kTile + tx;
      const bool masked = (kSum ? i == 0 : i == at) || (kSum && (at + i + 1) * kTile > P);
      float lr[kStripB];
#pragma unroll
      for (int c = 0; c < kStripB; ++c) lr[c] = kSum ? sm.yl[buf][tx + 16 * c] * kLog2e : 0.f;
#pragma unroll
      for (int r = 0; r < kStripA; ++r) {
        float x[kStripB];
#pragma unroll
        for (int c = 0; c < kStripB; ++c) {
          float lo, hi;
          asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(s[r][c]));
          x[c] = lo + hi;
        }
        if (!kSum && logits)                          // for colsum_stored_kernel, in the order of the threads
          logits[(blockIdx.y * triangle_tiles(Pmax) + (size_t)at * (at + 1) / 2 + i) * (kTile * kTile / 4) + r * kStatThreads + threadIdx.x] =
              make_float4(x[0], x[1], x[2], x[3]);
#pragma unroll
        for (int c = 0; c < kStripB; ++c) x[c] = fmaf(x[c], mul, -lr[c]);
        if (masked) {
#pragma unroll
          for (int c = 0; c < kStripB; ++c) {
            const int row = kSum ? str0 + 16 * c : res0 + 8 * r, col = kSum ? res0 + 8 * r : str0 + 16 * c;
            if (col > row || (kSum && row >= P)) x[c] = -INFINITY;
          }
        }
        if (kSum) {
          acc[r] += (double)((exp2_ftz(x[0]) + exp2_ftz(x[1])) + (exp2_ftz(x[2]) + exp2_ftz(x[3])));
        } else {
          const float mx = fmaxf(m[r], fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])));
          if (mx > -INFINITY) {
            l[r] = l[r] * exp2_ftz(m[r] - mx) +
                   ((exp2_ftz(x[0] - mx) + exp2_ftz(x[1] - mx)) + (exp2_ftz(x[2] - mx) + exp2_ftz(x[3] - mx)));
            m[r] = mx;
          }
        }
      }
    }
    __syncthreads();                                  // the next strip uses the same buffers
    if (i0 >= i1) {                                   // nothing of this strip here
      if (kSum) sm.res[part][0][threadIdx.x] = 0.0;
      else reinterpret_cast<float2*>(sm.res[part][0])[threadIdx.x] = make_float2(-INFINITY, 0.f);
      continue;
    }
    // the 8 lanes that share a resident row; the other half of the warps has the rest of it
#pragma unroll
    for (int r = 0; r < kStripA; ++r) {
      if (kSum) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
        if ((lane & 7) == 0) sm.res[part][half][ty + 8 * r] = acc[r];
      } else {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
          combine_lse(m[r], l[r], __shfl_xor_sync(0xffffffffu, m[r], o), __shfl_xor_sync(0xffffffffu, l[r], o));
        if ((lane & 7) == 0) reinterpret_cast<float2*>(sm.res[part][half])[ty + 8 * r] = make_float2(m[r], l[r]);
      }
    }
  }
  cluster.sync();
  const int share = 2 * kTile / C;                    // results this CTA writes
  for (int i = threadIdx.x; i < share; i += kStatThreads) {
    const int e = rank * share + i, part = e / kTile, row = resident(part) * kTile + e % kTile;
    // Added in fp64 under the final maximum; the exponentials and products that bring the halves to it are fp32.  One fp32 combination
    // after another had errors of the column sums against fp64 of 8.8e-8 (32 heads, 500 tokens; relative, rms) and 9.4e-8 (16, 900); so:
    // 8.4e-8 and 8.9e-8.  The halves are read once, all at a time: the same 39.7 us at 16 x 700 and 139 us at 128 x 500 as one after another.
    double t = 0.0;
    float m = -INFINITY;
    if (kSum) {
      for (int c = 0; c < 2 * C; ++c) t += cluster.map_shared_rank(&sm, c >> 1)->res[part][c & 1][e % kTile];
    } else {
      float2 o[2 * kMaxSweepCtas];                    // maximum and sum of every half
#pragma unroll
      for (int c = 0; c < 2 * kMaxSweepCtas; ++c) {
        o[c] = make_float2(-INFINITY, 0.f);
        if (c < 2 * C) o[c] = *reinterpret_cast<const float2*>(&cluster.map_shared_rank(&sm, c >> 1)->res[part][c & 1][e % kTile]);
      }
#pragma unroll
      for (int c = 0; c < 2 * kMaxSweepCtas; ++c) m = fmaxf(m, o[c].x);
#pragma unroll
      for (int c = 0; c < 2 * kMaxSweepCtas; ++c)
        if (o[c].x > -INFINITY) t += (double)(o[c].y * exp2f(o[c].x - m));
    }
    if (row < P && (part == 0 || n > n0))
      out[(size_t)bh * Pmax + row] = kSum ? (float)t : (m + log2f((float)t)) * 0.6931471805599453f;
  }
  cluster.sync();                                     // no CTA ends while another reads its results
}

// Column sums from the dot products that the row sweep left in `logits` (whole tiles; those of rows >= P are not looked at: zeros
// times a key that is not finite are NaN), one pair of column tiles per cluster as above.  A thread holds the entries that it
// computed there: rows ty + 8 r, columns tx + 16 c.  The sums run in the order of sweep_kernel, so that the bits are the same
// whoever computes them: groups of rows 16 apart in fp32 (r even: group ty, r odd: group ty + 8), the tiles of a CTA, and the
// groups as its butterfly takes them (4 apart, 2, 1).
//
// The row sweep is bound by its FMAs (one per element of d and logit); repeating them for the column sums took half of the call.
// A logit costs 8 bytes of traffic instead (kStoredLogits: how many are kept at a time).  Row sweep, column sums and densities,
// us, repeated / stored: 8 heads of 1024 tokens, d = 64, 65.8 / 48.7, of 100 tokens 21.7 / 19.3; 32 heads of 1999 tokens 525 / 365, 16 of
// 1500, d = 128, 334 / 202; six layers of these 1686 / 1022.
__global__ void __launch_bounds__(kStatThreads)
colsum_stored_kernel(const float4* logits, const float* lse, float* __restrict__ out, int Pmax, int Hq, const int32_t* __restrict__ plen,
                     int head0, float mul) {
  __shared__ double res[2][2][kTile];                  // [strip of the pair][groups below 8, from 8 on][column]
  __shared__ double upper[2 * kStripB][kStatThreads / 2];           // of the warps with groups 4 to 7 and 12 to 15
  start_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int u = blockIdx.x / C, bh = head0 + (int)blockIdx.y;
  const int P = plen ? plen[bh / Hq] : Pmax;
  const int nT = (P + kTile - 1) / kTile;
  wait_for_prior_grid();
  if (2 * u >= nT + (nT & 1)) return;                  // the whole cluster
  const int n0 = nT - u, n = u != nT - 1 - u ? nT + 1 : n0;
  const int s0 = rank * n / C, s1 = (rank + 1) * n / C;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ty = (warp & 1) * 4 + (lane >> 3), tx = (warp >> 1) * 8 + (lane & 7);
  logits += blockIdx.y * triangle_tiles(Pmax) * (kTile * kTile / 4) + threadIdx.x;
  lse += (size_t)bh * Pmax;
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    const int col = part == 0 ? u : nT - 1 - u, from = part == 0 ? 0 : n0;            // column tile
    const int i0 = max(s0, from) - from, i1 = min(s1, part == 0 ? n0 : n) - from;     // its row tiles of this CTA, from the diagonal on
    double acc[2][kStripB] = {};
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
      const int at = col + i;
      const float4* t = logits + ((size_t)at * (at + 1) / 2 + col) * (kTile * kTile / 4);
      float4 x[kStripA];
      float l[kStripA];
#pragma unroll
      for (int r = 0; r < kStripA; ++r) {
        x[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (at * kTile + ty + 8 * r < P) x[r] = t[r * kStatThreads];
      }
#pragma unroll
      for (int r = 0; r < kStripA; ++r) { const int row = at * kTile + ty + 8 * r; l[r] = row < P ? -(lse[row] * kLog2e) : -INFINITY; }
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        float p[4][kStripB];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = 2 * q + g;
          const float d[kStripB] = {x[r].x, x[r].y, x[r].z, x[r].w};
#pragma unroll
          for (int c = 0; c < kStripB; ++c) {
            const float e = exp2_ftz(fmaf(d[c], mul, l[r]));
            p[q][c] = i == 0 && tx + 16 * c > ty + 8 * r ? 0.f : e;                   // the tile on the diagonal
          }
        }
#pragma unroll
        for (int c = 0; c < kStripB; ++c) acc[g][c] += (double)((p[0][c] + p[1][c]) + (p[2][c] + p[3][c]));
      }
    }
    const int peer = (warp >> 1) * 32 + lane;
    if (warp & 1) {
#pragma unroll
      for (int k = 0; k < 2 * kStripB; ++k) upper[k][peer] = acc[k / kStripB][k % kStripB];
    }
    __syncthreads();
    if (!(warp & 1)) {
#pragma unroll
      for (int k = 0; k < 2 * kStripB; ++k) {
        double t = acc[k / kStripB][k % kStripB] + upper[k][peer];
        t += __shfl_xor_sync(0xffffffffu, t, 16);
        t += __shfl_xor_sync(0xffffffffu, t, 8);
        if (lane < 8) res[part][k / kStripB][tx + 16 * (k % kStripB)] = t;
      }
    }
    __syncthreads();                                   // `upper` is used again
  }
  cluster.sync();
  const int share = 2 * kTile / C;                     // results this CTA writes
  for (int i = threadIdx.x; i < share; i += kStatThreads) {
    const int e = rank * share + i, part = e / kTile, col = (part == 0 ? u : nT - 1 - u) * kTile + e % kTile;
    double t = 0.0;
    for (int c = 0; c < 2 * C; ++c) t += cluster.map_shared_rank(&res[0][0][0], c >> 1)[(part * 2 + (c & 1)) * kTile + e % kTile];
    if (col < P && (part == 0 || n > n0)) out[(size_t)bh * Pmax + col] = (float)t;
  }
  cluster.sync();                                      // no CTA ends while another reads its results
}

// CTAs per cluster of a sweep over `heads` heads: as many as give every SM its CTAs (three fit, four leave a short second round);
// past that only while every CTA keeps four tiles, because the copies that start a strip weigh as much as a tile or two, or
// eight in sweeps of several rounds, so that the last one is a small part of the launch (32 heads of 1999 tokens, d = 64: 4.67 ms
// with four tiles per CTA, 4.20 with eight).  us, two rounds of CTAs with one or two tiles / one round: 16 heads of 700 tokens 48.3 /
// 39.7, four layers of 32 heads of 500 tokens 183 / 139, of 16 heads of 900 tokens 199 / 174; 16 heads of 1024 tokens 72.4 / 73.4
// (by itself 78.9 / 74.8); but 24 heads of 1000 tokens, two rounds of four tiles / one round 87.3 / 89.2.
// Sums depend on it, so it is that of all heads of a call also where they go in groups.
static int sweep_ctas(int P, int heads, int sms) {
  const int nT = (P + kTile - 1) / kTile, pairs = (nT + 1) / 2;
  const long long units = (long long)pairs * heads;
  int C = 1;
  while (C < kMaxSweepCtas && 2 * C <= nT + 1 &&
         (units * 2 * C <= 4 * sms || (units * C < 4 * sms && nT + 1 >= 8 * C) || (units * C < 16 * sms && nT + 1 >= 16 * C)))
    C *= 2;
  return C;
}

// The same for the column sweep by itself (the caller's normalisers): of the sizes 1, 2, 4 and 8 the one whose rounds are shortest.  A
// round takes as long as the tiles of a CTA do (1.5 and 1.7 times as long with two and three CTAs per SM as with one) and 1.5
// tiles to start and end.  us with the rule above / so: 32 heads of 896 tokens, where that leaves four CTAs for a second round,
// 71.8 / 65.7, 22 of 896, d = 128, 102 / 87.7, 48 of 640, d = 128, 102 / 90.6, 12 of 1500 74.2 / 65.2, 32 of 1999 263 / 239, 28 of 832 51.3 / 51.3;
// two layers side by side 12 of 1500 127 / 114, but 22 of 896 88 / 92 and 16 of 900 71 / 77.
static int given_ctas(int P, int heads, int sms) {
  const int nT = (P + kTile - 1) / kTile;
  const long long units = (long long)((nT + 1) / 2) * heads;
  static const int tile10[4] = {0, 10, 15, 17};
  int best = 1;
  long long shortest = -1;
  for (int C = 1; C <= kMaxSweepCtas && (C == 1 || C <= nT + 1); C *= 2) {
    const long long rounds = units * C / (3 * sms), rest = units * C % (3 * sms), tiles = (nT + C) / C;
    const long long t = rounds * (17 * tiles + 15) + (rest > 0 ? tile10[(rest + sms - 1) / sms] * tiles + 15 : 0);
    if (shortest < 0 || t < shortest) { shortest = t; best = C; }
  }
  return best;
}

// Bytes of logits that one of `lanes` lanes keeps: whole heads, for all lanes at most kStoredLogits; 0 where one head's
// triangle is larger.  Fewer heads at a time mean more launches with a start and an end each, which weighs more than keeping
// the logits in L2: 32 heads of 1999 tokens, one lane, 517 us with 32 MB, 437 with 64, 367 with 256 (in another order of the sums).
constexpr size_t kStoredLogits = (size_t)256 << 20;
constexpr int kB200Sms = 148;             // the size of the scratch does not depend on the current device
static size_t stored_head_bytes(int P) { return triangle_tiles(P) * kTile * kTile * sizeof(float); }

// Are the dot products of `heads` heads better stored than computed twice, with room for `fit` heads and `lanes` layers at a time?
// Heads that all fit: always.  In groups, one launch after another, only where the CTAs in flight come near to filling the GPU as
// those of all heads do: its places are three per SM, and a group on half of them takes as long as both sweeps over all heads at
// once.  ms, twice / stored, d = 64: 448 CTAs and more 0.53 / 0.37 (32 heads of 2000 tokens) to 3.46 / 2.92 (16 of 8000); 376 1.99 /
// 1.73; 366 2.65 / 2.46; 344 3.29 / 3.06; 336 2.90 / 2.95; 320 5.09 / 5.66 and 1.43 / 1.45; 288 1.91 / 2.12; 252 6.39 / 8.21; 160 5.26 /
// 8.31 (64 heads of 5000 tokens); clusters of four, two CTAs to an SM, are as good again: 288 2.26 / 2.25, 284 4.41 / 3.95, but 300
// 3.70 / 3.97, 252 3.47 / 4.26.  A logit of d = 128 is twice the products: 344 6.12 / 5.45; 320 4.03 / 3.64; 288 3.72 / 3.62 and
// 4.40 / 4.07; 252 6.80 / 7.36; 188 14.1 / 18.5.
static bool stored_pays(int P, int D, int heads, int fit, int lanes, int sms) {
  if (fit >= heads) return true;
  if (fit < 1) return false;
  const int groups = (heads + fit - 1) / fit, pairs = ((P + kTile - 1) / kTile + 1) / 2, C = sweep_ctas(P, heads, sms);
  const long long ctas = (long long)lanes * heads * pairs * C / groups;
  return 10 * ctas >= 19 * sms && (D == 128 || 10 * ctas >= 23 * sms || (C >= 4 && ctas <= 2 * sms));
}

size_t stored_logits_bytes(int heads, int P, int D, int lanes) {
  const size_t head = stored_head_bytes(P);
  const int fit = (int)std::min<size_t>(heads, kStoredLogits / lanes / head), all = (int)std::min<size_t>(heads, lanes * (size_t)fit);
  // layers side by side, or one at a time in the room of all lanes
  return stored_pays(P, D, heads, fit, lanes, kB200Sms) || stored_pays(P, D, heads, all, 1, kB200Sms) ? fit * head : 0;
}

static cudaError_t launch_colsum_stored(const float4* logits, const float* lse, float* colsum, int P, int D, int head0, int n_heads, int Hq,
                                        const int32_t* plen, cudaStream_t st, int C) {
  const int pairs = ((P + kTile - 1) / kTile + 1) / 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pairs * C), (unsigned)n_heads); cfg.blockDim = dim3(kStatThreads); cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, colsum_stored_kernel, logits, lse, colsum, P, Hq, plen, head0, logit_scale(D));
}

// One sweep over `n_heads` heads from `head0` on.
template <typename T, int D, bool kSum>
static cudaError_t launch_sweep(const T* Q, const T* K, const float* lse_in, float* out, int P, int n_heads, int Hq, int group,
                                const int32_t* plen, cudaStream_t st, bool overlap, int C, int head0 = 0, float4* logits = nullptr) {
  const int pairs = ((P + kTile - 1) / kTile + 1) / 2;
  const size_t smem = sizeof(SweepSmem<D>);
  cudaError_t e = cudaFuncSetAttribute(sweep_kernel<T, D, kSum>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pairs * C), (unsigned)n_heads);
  cfg.blockDim = dim3(kStatThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = overlap ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, sweep_kernel<T, D, kSum>, Q, K, lse_in, out, P, Hq, group, plen, head0, logits);
}

__global__ void density_kernel(const float* colsum, double* __restrict__ density, int Pmax, int Hq, int L, int layer0,
                               const int32_t* __restrict__ plen, uint32_t* sched);
constexpr int kDensityThreads = 512;

// Row normalisers (unless the caller has them), column sums and densities of one layer, one of `lanes` side by side.  Each kernel may start beside the
// tail of the one before it: only what this call wrote is waited for inside the kernels.
template <typename T, int D>
static cudaError_t launch_sweeps(const T* Q, const T* K, const float* lse, float* lse_buf, float* colsum, double* density, int P,
                                 int B, int Hq, int group, int L, int layer, const int32_t* plen, cudaStream_t st, float4* logits,
                                 size_t logits_bytes, int lanes) {
  const bool own = lse == nullptr;
  int dev = 0, sms = kB200Sms;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) (void)cudaGetLastError();
  const int heads = B * Hq, C = own ? sweep_ctas(P, heads, sms) : given_ctas(P, heads, sms);
  const int fit = (int)std::min<size_t>(heads, logits_bytes / stored_head_bytes(P));
  cudaError_t e;
  if (own && stored_pays(P, D, heads, fit, lanes, sms)) {
    // as many heads at a time as leave their logits behind, in groups of about the same size
    const int groups = (heads + fit - 1) / fit;
    for (int i = 0; i < groups; ++i) {
      const int h0 = (int)((long long)heads * i / groups), n = (int)((long long)heads * (i + 1) / groups) - h0;
      e = launch_sweep<T, D, false>(Q, K, nullptr, lse_buf, P, n, Hq, group, plen, st, true, C, h0, logits);
      if (e != cudaSuccess) return e;
      e = launch_colsum_stored(logits, lse_buf, colsum, P, D, h0, n, Hq, plen, st, C);
      if (e != cudaSuccess) return e;
    }
  } else {
    if (own) {
      e = launch_sweep<T, D, false>(Q, K, nullptr, lse_buf, P, heads, Hq, group, plen, st, true, C);
      if (e != cudaSuccess) return e;
      lse = lse_buf;
    }
    e = launch_sweep<T, D, true>(Q, K, lse, colsum, P, heads, Hq, group, plen, st, own, C);
    if (e != cudaSuccess) return e;
  }
  return launch_behind(density_kernel, dim3((unsigned)(B * Hq)), kDensityThreads, 0, st, (const float*)colsum, density, P, Hq, L, layer, plen,
                       (uint32_t*)nullptr);
}

// F[b, layer, hq] = (1/P) sum_j (s_j - mean)^2, mean = (1/P) sum_j s_j   (Eq. 4; population variance)
// One CTA per (sequence, head) and layer (blockIdx.y).  Two passes in fp64; a thread keeps its values of the first pass in
// registers (up to 8, P <= 4096) or reads them again (8192 tokens, 32 heads: 21.6 us with 256 threads that read everything
// twice and one value at a time; the kernel is a chain of load latencies).
__global__ void __launch_bounds__(kDensityThreads)
density_kernel(const float* colsum, double* __restrict__ density, int Pmax, int Hq, int L, int layer0,
               const int32_t* __restrict__ plen, uint32_t* sched) {
  constexpr int kKeep = 8, kWarps = kDensityThreads / 32;
  __shared__ double part[kWarps];
  const int bh = blockIdx.x, layer = layer0 + (int)blockIdx.y;
  const int b = bh / Hq, hq = bh % Hq;
  start_dependents();
  wait_for_prior_grid();
  // The column sums' work counter (NULL: there is none) is zero for the next call whatever became of it in this one, so that
  // calls that overlap on the GPU against the rules spoil their own results only.
  if (sched && bh == 0 && blockIdx.y == 0 && threadIdx.x < 2) sched[threadIdx.x] = 0u;
  const int P = plen ? plen[b] : Pmax;
  const float* s = colsum + ((size_t)blockIdx.y * gridDim.x + bh) * Pmax;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto block_total = [&](double t) {                                 // every thread gets it
    t = warp_sum(t);
    __syncthreads();
    if (lane == 0) part[warp] = t;
    __syncthreads();
    t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += part[w];
    return t;
  };
  float v[kKeep];
  double t = 0.0;
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    const int j = threadIdx.x + i * kDensityThreads;
    v[i] = j < P ? s[j] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < kKeep; ++i) t += (double)v[i];
  for (int j0 = threadIdx.x + kKeep * kDensityThreads; j0 < P; j0 += 4 * kDensityThreads) {
    float f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = j0 + i * kDensityThreads < P ? s[j0 + i * kDensityThreads] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) t += (double)f[i];
  }
  const double mean = block_total(t) / (double)P;
  t = 0.0;
#pragma unroll
  for (int i = 0; i < kKeep; ++i)
    if (threadIdx.x + i * kDensityThreads < P) { const double dlt = (double)v[i] - mean; t += dlt * dlt; }
  for (int j0 = threadIdx.x + kKeep * kDensityThreads; j0 < P; j0 += 4 * kDensityThreads) {
    float f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = j0 + i * kDensityThreads < P ? s[j0 + i * kDensityThreads] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (j0 + i * kDensityThreads < P) { const double dlt = (double)f[i] - mean; t += dlt * dlt; }
  }
  t = block_total(t);
  if (threadIdx.x == 0) density[((size_t)b * L + layer) * Hq + hq] = t / (double)P;
}

// Cache sizes from the densities.  budget_rule 0 (Eq. 5): S_l = clip(lambda * w_l, S_min, S_max) with
// sum_l S_l = S_tot, then floor + largest remainder; rule 1 (per-head sizes of Appendix A.5): the same over the
// (layer, KV head) units; rule 2 (exponential-decay allocation of the ablation): S_l = round(mean_h exp(-F/gamma) P),
// clamped, no fixed total.  Output tables are [B, L, Hkv]; the per-layer rules give every KV head of a layer the same size.
//
// One CTA per sequence.  The integers must not depend on how the work is divided, so every sum runs in one thread in the
// order of the units; what runs side by side are different sums: the weights of different units, the totals at different
// values of lambda (all kinks at once, or a many-way search where there are more of them than threads), the rank of every
// remainder.
constexpr int kBudgetThreads = 256;
__device__ inline double clipd(double v, double lo, double hi) { return v < lo ? lo : (v > hi ? hi : v); }

// minimum over the CTA; every thread gets it
__device__ inline double block_min(double v, double* part) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { const double t = __shfl_xor_sync(0xffffffffu, v, o); v = t < v ? t : v; }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  v = part[0];
  for (int w = 1; w < kBudgetThreads / 32; ++w) v = part[w] < v ? part[w] : v;
  return v;
}

__global__ void __launch_bounds__(kBudgetThreads)
budget_kernel(const double* __restrict__ density, int L, int H, int Hkv, int Pmax, double rho, int min_budget,
              int max_budget_cfg, double gamma, int head_reduce, int budget_rule, int n_sink, int window, double nm_ratio,
              int32_t* __restrict__ budgets, int32_t* __restrict__ windows, uint32_t* status_word,
              const int32_t* __restrict__ plen) {
  extern __shared__ __align__(16) double dsm[];
  const int n = budget_rule == 1 ? L * Hkv : L;                       // allocation units
  const int G = H / Hkv;
  int n_pad = 2;                                                      // kinks, padded for the sort
  while (n_pad < 2 * n) n_pad *= 2;
  double* w = dsm;              // [n] weights
  double* x = w + n;            // [n] scaled sizes, then remainders
  double* kinks = x + n;        // [n_pad]
  __shared__ double part[kBudgetThreads / 32], s_lam;
  __shared__ int s_lo, s_hi, s_open;
  __shared__ long long s_left;
  const int tid = threadIdx.x, b = blockIdx.x;
  const double lo = (double)min_budget;
  const int P = plen ? plen[b] : Pmax;                                // this sequence's prompt length
  const int max_budget = max_budget_cfg > 0 ? max_budget_cfg : P;     // no clamp given: a layer cannot hold more than the prompt
  const double hi = (double)max_budget;
  const long long S_tot = (long long)floor(rho * (double)n * (double)P + 0.5);
  const double* F = density + (size_t)b * L * H;
  int32_t* bud = budgets + (size_t)b * L * Hkv;
  // unit u -> its (first) entry of the [L, Hkv] table
  auto slot_of = [&](int u) { return budget_rule == 1 ? u : u * Hkv; };
  if (budget_rule == 2) {
    for (int l = tid; l < L; l += kBudgetThreads) {
      double a = 0.0;
      for (int h = 0; h < H; ++h) a = __dadd_rn(a, exp(-__ddiv_rn(F[l * H + h], gamma)));
      const double s = floor(__dadd_rn(__dmul_rn(__ddiv_rn(a, (double)H), (double)P), 0.5));
      bud[l * Hkv] = (int32_t)clipd(s, lo, hi);
    }
  } else {
    if (budget_rule == 1 || head_reduce == 0) {
      double fmin = INFINITY;
      for (int i = tid; i < L * H; i += kBudgetThreads) fmin = F[i] < fmin ? F[i] : fmin;
      fmin = block_min(fmin, part);
      const int heads = budget_rule == 1 ? G : H;                     // query heads of a unit
      for (int u = tid; u < n; u += kBudgetThreads) {
        double a = 0.0;
        for (int g = 0; g < heads; ++g) a = __dadd_rn(a, exp(-__ddiv_rn(__dadd_rn(F[u * heads + g], -fmin), gamma)));
        w[u] = a;
      }
    } else if (head_reduce == 2) {
      // reciprocal of the variance, per head (a zero variance counts as the smallest positive one)
      for (int l = tid; l < L; l += kBudgetThreads) {
        double a = 0.0;
        for (int h = 0; h < H; ++h) {
          const double f = F[l * H + h];
          a = __dadd_rn(a, __ddiv_rn(1.0, f > 1e-300 ? f : 1e-300));
        }
        w[l] = a;
      }
    } else {
      double fmin = INFINITY;
      for (int l = tid; l < L; l += kBudgetThreads) {
        double a = 0.0;
        for (int h = 0; h < H; ++h) a = __dadd_rn(a, F[l * H + h]);
        x[l] = __ddiv_rn(a, (double)H);
        fmin = fmin < x[l] ? fmin : x[l];
      }
      fmin = block_min(fmin, part);
      for (int l = tid; l < L; l += kBudgetThreads) {                 // x[l] was written by this thread
        if (head_reduce == 1) w[l] = exp(-__ddiv_rn(__dadd_rn(x[l], -fmin), gamma));
        else w[l] = __ddiv_rn(1.0, x[l] > 1e-300 ? x[l] : 1e-300);
      }
    }
    // kinks of the piecewise-linear total(lambda), ascending
    for (int u = tid; u < n; u += kBudgetThreads) {
      w[u] = w[u] > 1e-300 ? (w[u] < 1e300 ? w[u] : 1e300) : 1e-300;
      kinks[2 * u] = __ddiv_rn(lo, w[u]);
      kinks[2 * u + 1] = __ddiv_rn(hi, w[u]);
    }
    for (int i = 2 * n + tid; i < n_pad; i += kBudgetThreads) kinks[i] = INFINITY;
    for (int k = 2; k <= n_pad; k *= 2)                               // bitonic sort
      for (int j = k / 2; j > 0; j /= 2) {
        __syncthreads();
        for (int i = tid; i < n_pad; i += kBudgetThreads) {
          const int o = i ^ j;
          if (o > i) {
            const double p = kinks[i], q = kinks[o];
            if ((p > q) == ((i & k) == 0)) { kinks[i] = q; kinks[o] = p; }
          }
        }
      }
    const int nk = 2 * n;
    auto total = [&](double lam) {
      double t = 0.0;
      for (int u = 0; u < n; ++u) t = __dadd_rn(t, clipd(__dmul_rn(lam, w[u]), lo, hi));
      return t;
    };
    // total() is non-decreasing: the first kink that reaches S_tot, in [s_lo, s_hi]
    if (tid == 0) { s_lo = 0; s_hi = nk; }
    __syncthreads();
    while (s_lo < s_hi) {                                             // uniform: written before a barrier
      const int from = s_lo, to = s_hi, step = (to - from + kBudgetThreads - 1) / kBudgetThreads;
      const int at = min(from + (tid + 1) * step - 1, to - 1);        // last kink of this thread's stretch
      const bool below = from + tid * step < to && total(kinks[at]) < (double)S_tot;
      // stretches whose last kink stays below the total are passed over; the next one holds the answer
      const int passed = __syncthreads_count(below);
      if (tid == 0) {
        s_lo = min(from + passed * step, to);
        s_hi = step == 1 ? s_lo : min(s_lo + step - 1, to);
      }
      __syncthreads();
    }
    if (tid == 0) {
      const int k = s_lo;
      double lam;
      if (k == 0) lam = kinks[0];
      else if (k == nk) lam = kinks[nk - 1];
      else {
        const double a = kinks[k - 1], bb = kinks[k];
        const double mid = __dmul_rn(0.5, __dadd_rn(a, bb));
        double fixed = 0.0, wf = 0.0;
        for (int u = 0; u < n; ++u) {
          const double v = __dmul_rn(mid, w[u]);
          if (v > lo && v < hi) wf = __dadd_rn(wf, w[u]);
          else fixed = __dadd_rn(fixed, clipd(v, lo, hi));
        }
        lam = wf > 0.0 ? __ddiv_rn(__dadd_rn((double)S_tot, -fixed), wf) : bb;
        lam = lam < a ? a : (lam > bb ? bb : lam);
      }
      s_lam = lam;
      s_left = S_tot;
      s_open = 0;
    }
    __syncthreads();
    const double lam = s_lam;
    for (int u = tid; u < n; u += kBudgetThreads) {
      const double v = clipd(__dmul_rn(lam, w[u]), lo, hi), fl = floor(v);
      bud[slot_of(u)] = (int32_t)fl;
      x[u] = (int32_t)fl < max_budget ? v - fl : -1.0;                // remainder; a unit at the upper clamp takes no further row
      if (x[u] >= 0.0) atomicAdd(&s_open, 1);
      atomicAdd((unsigned long long*)&s_left, (unsigned long long)(-(long long)fl));
    }
    __syncthreads();
    long long left = s_left;
    if (left < 0 || left > n) {
      if (tid == 0) report_error(status_word, D2O_ERR_STATE, 0xB0000000u | (uint32_t)b);
      left = 0;
    }
    if (left > s_open && tid == 0) report_error(status_word, D2O_ERR_STATE, 0xB1000000u | (uint32_t)b);
    // largest remainder first, ties -> lower unit: the first `left` in that order get one more row
    if (left > 0)
      for (int u = tid; u < n; u += kBudgetThreads) {
        const double xu = x[u];
        if (xu < 0.0) continue;
        int rank = 0;
        for (int v = 0; v < n; ++v) rank += x[v] > xu || (x[v] == xu && v < u) ? 1 : 0;
        if (rank < left) bud[slot_of(u)] += 1;
      }
  }
  __syncthreads();                                                    // the CTA's own writes to `bud` are read below
  for (int i = tid; i < L * Hkv; i += kBudgetThreads) {
    const int S = budget_rule == 1 ? bud[i] : bud[i / Hkv * Hkv];     // one size per layer: every KV head gets it
    if (budget_rule != 1 && i % Hkv != 0) bud[i] = S;
    if (windows) {
      const int T = n_sink < S ? n_sink : S;
      int M = window > 0 ? window : (int)floor((double)(S - T) / (1.0 + nm_ratio) + 0.5);
      M = M < 0 ? 0 : (M > S - T ? S - T : M);
      windows[(size_t)b * L * Hkv + i] = M;
    }
  }
}

// First cache row of every slice: rows are laid out layer-major, then sequence, then head.
__global__ void __launch_bounds__(1024)
row_offset_kernel(const int32_t* __restrict__ budgets, int B, int L, int Hkv, int64_t* __restrict__ row_off) {
  __shared__ long long s_warp[32], s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_base = 0;
  const int n = L * B * Hkv;
  for (int i0 = 0; i0 < n; i0 += 1024) {
    const int i = i0 + threadIdx.x;
    const int l = i / (B * Hkv), b = i / Hkv % B, h = i % Hkv;
    const size_t e = ((size_t)b * L + l) * Hkv + h;
    const long long v = i < n ? (long long)slice_stride(budgets[e]) : 0;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const long long t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    long long before = s_base;
    for (int k = 0; k < warp; ++k) before += s_warp[k];
    if (i < n) row_off[e] = before + inc - v;
    __syncthreads();
    if (threadIdx.x == 1023) s_base = before + inc;
    __syncthreads();
  }
}

template <typename T, int D>
static cudaError_t run_stats(const d2o_ctx* c, int layer, const void* Q, const void* K, const float* lse_in,
                             cudaStream_t st, int lane, int lanes) {
  const d2o_config& g = c->cfg;
  const int P = g.prompt_len, Hq = g.n_q_heads, B = g.batch;
  float* colsum = (float*)(c->state + c->lay.colsum) + (size_t)layer * B * Hq * P;
  double* density = (double*)(c->state + c->lay.density);
  const int32_t* plen = (const int32_t*)(c->state + c->lay.plen);
  return launch_sweeps<T, D>((const T*)Q, (const T*)K, lse_in, (float*)(c->scratch + c->slay.lse + (size_t)lane * c->slay.lse_stride),
                             colsum, density, P, B, Hq, c->group, g.n_layers, layer, plen, st,
                             (float4*)(c->scratch + c->slay.logits + (size_t)lane * c->slay.logits_stride),
                             // a layer by itself has the room of all lanes
                             (lanes == 1 ? std::min(g.n_layers, kStatsLanes) : 1) * c->slay.logits_stride, lanes);
}

cudaError_t launch_layer_stats_tc(const d2o_ctx* c, int layer, int n, const void* const* Q, const void* const* K,
                                  const float* const* lse, cudaStream_t st) {
  const d2o_config& g = c->cfg;
  const int P = g.prompt_len, Hq = g.n_q_heads, B = g.batch;
  float* colsum = (float*)(c->state + c->lay.colsum) + (size_t)layer * B * Hq * P;
  const int32_t* plen = (const int32_t*)(c->state + c->lay.plen);
  cudaError_t e = launch_colsum_tc(g.dtype, g.d_head, B, Hq, g.n_kv_heads, P, n, Q, K, lse, (float*)(c->scratch + c->slay.lse),
                                   c->slay.lse_stride, colsum, plen, (uint32_t*)(c->state + c->lay.status),
                                   (uint32_t*)(c->state + c->lay.colsum_sched), st,
                                   (unsigned long long)c->wait_limit_us * 1000ull, c->producer_stop_stage);
  if (e != cudaSuccess) return e;
  return launch_behind(density_kernel, dim3((unsigned)(B * Hq), (unsigned)n), kDensityThreads, 0, st, (const float*)colsum,
                       (double*)(c->state + c->lay.density), P, Hq, g.n_layers, layer, plen,
                       (uint32_t*)(c->state + c->lay.colsum_sched));
}

cudaError_t launch_layer_stats(const d2o_ctx* c, int layer, const void* Q, const void* K, const float* lse,
                               cudaStream_t st, int lane, int lanes) {
  if (c->stats_path == 0 && c->cfg.dtype != D2O_F32) return launch_layer_stats_tc(c, layer, 1, &Q, &K, lse ? &lse : nullptr, st);
  const int d = c->cfg.d_head;
  switch (c->cfg.dtype) {
    case D2O_F32: return d == 64 ? run_stats<float, 64>(c, layer, Q, K, lse, st, lane, lanes) : run_stats<float, 128>(c, layer, Q, K, lse, st, lane, lanes);
    case D2O_F16: return d == 64 ? run_stats<__half, 64>(c, layer, Q, K, lse, st, lane, lanes) : run_stats<__half, 128>(c, layer, Q, K, lse, st, lane, lanes);
    default: return d == 64 ? run_stats<__nv_bfloat16, 64>(c, layer, Q, K, lse, st, lane, lanes)
                            : run_stats<__nv_bfloat16, 128>(c, layer, Q, K, lse, st, lane, lanes);
  }
}

cudaError_t launch_budgets(const double* density, int B, int L, int H, int Hkv, int P, float rho, int min_budget,
                           int max_budget, float gamma, int head_reduce, int budget_rule, int n_sink, int window,
                           float nm_ratio, int32_t* budgets, int32_t* windows, int64_t* row_off, uint32_t* status_word,
                           const int32_t* plen, cudaStream_t st) {
  const size_t n = budget_rule == 1 ? (size_t)L * Hkv : (size_t)L;
  size_t n_pad = 2;
  while (n_pad < 2 * n) n_pad *= 2;
  const size_t sm = (2 * n + n_pad) * sizeof(double);
  if (sm > 200 * 1024) return cudaErrorInvalidValue;          // more allocation units than the work arrays hold
  cudaError_t e = cudaFuncSetAttribute(budget_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  budget_kernel<<<B, kBudgetThreads, sm, st>>>(density, L, H, Hkv, P, (double)rho, min_budget, max_budget, (double)gamma,
                                               head_reduce, budget_rule, n_sink, window, (double)nm_ratio, budgets, windows,
                                               status_word, plen);
  if (row_off) row_offset_kernel<<<1, 1024, 0, st>>>(budgets, B, L, Hkv, row_off);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------ allocation-free variant
// Scratch for the row normalisers of d2o_layer_stats_static: part of the library image, one copy per GPU.  The
// tensor-core kernels pad every (sequence, head) row to a multiple of four floats.
constexpr int kStaticMaxRows = 65535;                // (sequence, head) pairs: one grid row of the generic kernels each
// The two words behind them are its work counter (zero in the image, and left at zero by every call).
constexpr size_t kStaticFloats = (size_t)D2O_STATIC_LSE_FLOATS + 3 * kStaticMaxRows + 1;
static __device__ __align__(256) float g_static_lse[kStaticFloats + 2];
constexpr int kMaxDevices = 64;
static float* g_static_lse_addr[kMaxDevices];        // device address of g_static_lse, per device (host-side cache)

template <typename T, int D>
static cudaError_t run_stats_static(int dtype, const void* Q, const void* K, float* lse_buf, float* colsum, double* density,
                                    int B, int Hq, int group, int P, cudaStream_t st) {
  if (sizeof(T) == 2) {
    uint32_t* sched = (uint32_t*)(lse_buf + kStaticFloats);
    cudaError_t e = launch_colsum_tc(dtype, D, B, Hq, Hq / group, P, 1, &Q, &K, nullptr, lse_buf, 0, colsum, nullptr, nullptr,
                                     sched, st);
    if (e != cudaSuccess) return e;
    return launch_behind(density_kernel, dim3((unsigned)(B * Hq)), kDensityThreads, 0, st, (const float*)colsum, density, P, Hq, 1, 0,
                         nullptr, sched);
  }
  return launch_sweeps<T, D>((const T*)Q, (const T*)K, nullptr, lse_buf, colsum, density, P, B, Hq, group, 1, 0, nullptr, st, nullptr, 0, 1);
}

}  // namespace d2o

extern "C" d2o_status d2o_layer_stats_static(int32_t dtype, int32_t d_head, int32_t batch, int32_t n_q_heads,
                                             int32_t n_kv_heads, int32_t prompt_len, const void* Q, const void* K,
                                             float* colsum, double* density, void* stream) {
  using namespace d2o;
  if (dtype != D2O_F32 && dtype != D2O_F16 && dtype != D2O_BF16) return D2O_ERR_UNSUPPORTED;
  if (d_head != 64 && d_head != 128) return D2O_ERR_UNSUPPORTED;
  if (batch < 1 || n_q_heads < 1 || n_kv_heads < 1 || prompt_len < 1 || n_q_heads % n_kv_heads != 0)
    return D2O_ERR_INVALID_ARG;
  auto aligned16 = [](const void* p) { return p && (((uintptr_t)p & 15) == 0); };
  if (!aligned16(Q) || !aligned16(K) || !aligned16(colsum) || !density || ((uintptr_t)density & 7)) return D2O_ERR_INVALID_ARG;
  if ((unsigned long long)batch * n_q_heads * prompt_len > (unsigned long long)D2O_STATIC_LSE_FLOATS)
    return D2O_ERR_TOO_LARGE;
  if ((long long)batch * n_q_heads > kStaticMaxRows) return D2O_ERR_TOO_LARGE;      // one grid row per (sequence, head)
  // set-up, once per device: in host code `g_static_lse` is only a handle, the kernels need its device address
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return record_cuda_error(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return D2O_ERR_UNSUPPORTED;
  float* lse_buf = __atomic_load_n(&g_static_lse_addr[dev], __ATOMIC_ACQUIRE);
  if (!lse_buf) {
    e = cudaGetSymbolAddress((void**)&lse_buf, g_static_lse);
    if (e != cudaSuccess || !lse_buf) return record_cuda_error(e, "cudaGetSymbolAddress(g_static_lse)");
    __atomic_store_n(&g_static_lse_addr[dev], lse_buf, __ATOMIC_RELEASE);     // every thread would store the same value
  }
  const int group = n_q_heads / n_kv_heads;
  cudaStream_t st = (cudaStream_t)stream;
  switch (dtype) {
    case D2O_F32:
      e = d_head == 64 ? run_stats_static<float, 64>(dtype, Q, K, lse_buf, colsum, density, batch, n_q_heads, group, prompt_len, st)
                       : run_stats_static<float, 128>(dtype, Q, K, lse_buf, colsum, density, batch, n_q_heads, group, prompt_len, st);
      break;
    case D2O_F16:
      e = d_head == 64 ? run_stats_static<__half, 64>(dtype, Q, K, lse_buf, colsum, density, batch, n_q_heads, group, prompt_len, st)
                       : run_stats_static<__half, 128>(dtype, Q, K, lse_buf, colsum, density, batch, n_q_heads, group, prompt_len, st);
      break;
    default:
      e = d_head == 64 ? run_stats_static<__nv_bfloat16, 64>(dtype, Q, K, lse_buf, colsum, density, batch, n_q_heads, group, prompt_len, st)
                       : run_stats_static<__nv_bfloat16, 128>(dtype, Q, K, lse_buf, colsum, density, batch, n_q_heads, group, prompt_len, st);
  }
  if (e != cudaSuccess) return record_cuda_error(e, "d2o_layer_stats_static launch");
  return D2O_OK;
}
