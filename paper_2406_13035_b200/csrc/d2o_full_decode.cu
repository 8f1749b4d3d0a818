// Uncompressed decode attention (Section 3, Eq. 2-3): the comparison kernel for the compressed path.
//
// One thread-block cluster handles one slice = (sequence, KV head) with its G query heads; the len+1 rows (cache + the
// new token) are split evenly over the CTAs of the cluster and, row by row, over the row groups of their warps.  Every
// row group walks through its rows on its own with a running softmax (maximum, sum, un-normalised output), keys and
// values of several rows in flight at a time; at the end the groups, the warps and (through distributed shared memory,
// by rank 0) the CTAs of a cluster are combined.  The new token's row is appended at row `len`.
//
// Bound by HBM.  An earlier form read all keys of a CTA before its values, reduced every row's dot product with four
// shuffles and had 512 CTAs of 1032 rows for 256 slices (1.15 waves): 83 us for 256 slices of 2049 fp16 rows, now 46.7
// (0.88 of the copy bandwidth).
#include <cooperative_groups.h>
#include <math.h>

#include "d2o_common.cuh"
#include "d2o_decode.cuh"

namespace cg = cooperative_groups;

namespace d2o {

constexpr int kFullThreads = 256;
constexpr int kFullWarps = kFullThreads / 32;
constexpr int kFullMaxCluster = 8;

struct FullArgs {
  int capacity, len;
};

template <int G, int D>
struct alignas(16) FullExchange {    // the part of shared memory that peer CTAs read
  float m[G];
  float l[G];
  float acc[G][D];
};

// rows of a row group in flight, and CTAs per SM the registers are capped for
__host__ __device__ constexpr int full_rows(int G) { return G <= 2 ? 8 : 4; }
__host__ __device__ constexpr int full_ctas(int G) { return G <= 4 ? 2 : 1; }

template <typename T, int D, int G>
__global__ void __launch_bounds__(kFullThreads, full_ctas(G))
full_decode_kernel(FullArgs a, const T* q_in, const T* k_in, const T* v_in,      // the grid ahead may still be writing them: see wait_for_prior_grid
                   T* __restrict__ out, T* __restrict__ kcache, T* __restrict__ vcache) {
  constexpr int EPV = Elem<T>::kPerVec;
  constexpr int LPR = D / EPV;                  // lanes that share one row (16-byte segment each)
  constexpr int NGRP = kFullThreads / LPR;      // row groups of the CTA
  constexpr int QL = LPR / 4;                   // lanes that end up with the same row total after reduce4
  constexpr int U = full_rows(G);
  using Xch = FullExchange<G, D>;

  // launched with programmatic stream serialisation: the CTAs move in while the grid ahead drains
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int sl = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = tid / LPR, lig = tid % LPR;

  const int64_t row0 = (int64_t)sl * a.capacity;
  const int n_old = a.len;
  const int n = n_old + 1;
  const int chunk = (n + C - 1) / C;
  const int r0 = min(n, rank * chunk), r1 = min(n, r0 + chunk);

  extern __shared__ __align__(16) unsigned char dsm[];
  Xch* xch = reinterpret_cast<Xch*>(dsm);
  float* red = reinterpret_cast<float*>(dsm + sizeof(Xch));        // [warps][G][D]
  __shared__ float s_m[kFullWarps][G], s_l[kFullWarps][G];

  const T* k_new = k_in + (size_t)sl * D;
  const T* v_new = v_in + (size_t)sl * D;

  float qf[G][EPV];
  {
    const float mul = (D == 64 ? 0.125f : 0.08838834764831845f) * kLog2e;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      Elem<T>::unpack(ld_global_v4(q_in + ((size_t)sl * G + g) * D + lig * EPV), qf[g]);
#pragma unroll
      for (int e = 0; e < EPV; ++e) qf[g][e] *= mul;
    }
  }
  float m[G], l[G], acc[G][EPV];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    m[g] = -INFINITY; l[g] = 0.f;
#pragma unroll
    for (int e = 0; e < EPV; ++e) acc[g][e] = 0.f;
  }
  // rows base + u * NGRP + grp; all groups of a warp take part in every iteration (their shuffles name all lanes)
  for (int base = r0; base < r1; base += U * NGRP) {
    uint4 kv[U], vv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = base + u * NGRP + grp;
      kv[u] = make_uint4(0, 0, 0, 0);
      if (r < r1) kv[u] = ld_stream_v4((r < n_old ? kcache + (row0 + r) * D : k_new) + lig * EPV);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = base + u * NGRP + grp;
      vv[u] = make_uint4(0, 0, 0, 0);
      if (r < r1) vv[u] = ld_stream_v4((r < n_old ? vcache + (row0 + r) * D : v_new) + lig * EPV);
    }
    float x[G][U / 4];                                               // logit of this lane's row of every four
#pragma unroll
    for (int b = 0; b < U / 4; ++b) {
      float dot[G][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float f[EPV];
        Elem<T>::unpack(kv[b * 4 + u], f);
#pragma unroll
        for (int g = 0; g < G; ++g) dot[g][u] = dot_pairs<EPV>(qf[g], f);
      }
      const bool in = base + (b * 4 + lig / QL) * NGRP + grp < r1;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float t = reduce4<LPR>(dot[g][0], dot[g][1], dot[g][2], dot[g][3], lig);
        x[g][b] = in ? t : -INFINITY;
      }
    }
    float f[U][EPV];
#pragma unroll
    for (int u = 0; u < U; ++u) Elem<T>::unpack(vv[u], f[u]);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float mx = x[g][0];
#pragma unroll
      for (int b = 1; b < U / 4; ++b) mx = fmaxf(mx, x[g][b]);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, QL));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2 * QL));
      const float mn = fmaxf(m[g], mx);
      const float old = mn > -INFINITY ? exp2f(m[g] - mn) : 0.f;
      m[g] = mn;
      const float base = mn > -INFINITY ? mn : 0.f;                  // rows past the end, and logits of -inf: 0; a NaN stays one
      float p[U / 4], s = 0.f;
#pragma unroll
      for (int b = 0; b < U / 4; ++b) { p[b] = exp2f(x[g][b] - base); s += p[b]; }
      l[g] = fmaf(l[g], old, s);                                     // this lane's rows only: summed over the group at the end
#pragma unroll
      for (int e = 0; e < EPV; ++e) acc[g][e] *= old;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float w = __shfl_sync(0xffffffffu, p[u / 4], (u & 3) * QL, LPR);
#pragma unroll
        for (int e = 0; e < EPV; e += 2) {
          const float2 t = ffma2(make_float2(w, w), make_float2(f[u][e], f[u][e + 1]), make_float2(acc[g][e], acc[g][e + 1]));
          acc[g][e] = t.x; acc[g][e + 1] = t.y;
        }
      }
    }
  }
  // ---- combine the row groups of a warp, then the warps
#pragma unroll
  for (int g = 0; g < G; ++g) {
    float ls = l[g];                                                 // QL lanes hold the same rows
    ls += __shfl_xor_sync(0xffffffffu, ls, QL);
    ls += __shfl_xor_sync(0xffffffffu, ls, 2 * QL);
    float mw = m[g];
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, o));
    const float w = mw > -INFINITY ? exp2f(m[g] - mw) : 0.f;
    ls *= w;
#pragma unroll
    for (int e = 0; e < EPV; ++e) acc[g][e] *= w;
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
      ls += __shfl_xor_sync(0xffffffffu, ls, o);
#pragma unroll
      for (int e = 0; e < EPV; ++e) acc[g][e] += __shfl_xor_sync(0xffffffffu, acc[g][e], o);
    }
    if (lane == 0) { s_m[warp][g] = mw; s_l[warp][g] = ls; }
    if (lane < LPR) {
#pragma unroll
      for (int e = 0; e < EPV; ++e) red[(warp * G + g) * D + lane * EPV + e] = acc[g][e];
    }
  }
  __syncthreads();
  for (int i = tid; i < G * D; i += kFullThreads) {
    const int g = i / D;
    float mc = s_m[0][g];
#pragma unroll
    for (int w = 1; w < kFullWarps; ++w) mc = fmaxf(mc, s_m[w][g]);
    float t = 0.f, lc = 0.f;
#pragma unroll
    for (int w = 0; w < kFullWarps; ++w) {
      const float c = mc > -INFINITY ? exp2f(s_m[w][g] - mc) : 0.f;
      t = fmaf(red[w * G * D + i], c, t);
      lc = fmaf(s_l[w][g], c, lc);
    }
    if (C == 1) { out[(size_t)sl * G * D + i] = Elem<T>::from_float(t / lc); continue; }
    xch->acc[g][i % D] = t;
    if (i % D == 0) { xch->m[g] = mc; xch->l[g] = lc; }
  }
  if (C > 1) {
    cluster.sync();                                                  // (max, sum, partial outputs) of every CTA are visible
    if (rank == 0) {
      for (int i = tid; i < G * D; i += kFullThreads) {
        const int g = i / D, dd = i % D;
        float ms = -INFINITY;
        for (int r = 0; r < C; ++r) ms = fmaxf(ms, cluster.map_shared_rank(xch, r)->m[g]);
        float ls = 0.f, num = 0.f;
        for (int r = 0; r < C; ++r) {
          const Xch* x = cluster.map_shared_rank(xch, r);
          const float w = exp2f(x->m[g] - ms);
          ls = fmaf(x->l[g], w, ls);
          num = fmaf(x->acc[g][dd], w, num);
        }
        out[(size_t)sl * G * D + i] = Elem<T>::from_float(num / ls);
      }
    }
  }
  // append the new token's row
  if (rank == n_old / chunk && grp == 0) {
    *reinterpret_cast<uint4*>(kcache + (row0 + n_old) * D + lig * EPV) = ld_global_v4(k_new + lig * EPV);
    *reinterpret_cast<uint4*>(vcache + (row0 + n_old) * D + lig * EPV) = ld_global_v4(v_new + lig * EPV);
  }
  if (C > 1) cluster.sync();                                         // rank 0 may still read our exchange area
}

// ------------------------------------------------------------------------------------ launch
template <typename T, int D, int G>
static cudaError_t launch_one(const FullArgs& a, int n_slices, int C, const void* q, const void* k, const void* v,
                              void* out, void* kc, void* vc, cudaStream_t st) {
  const size_t smem = sizeof(FullExchange<G, D>) + (size_t)kFullWarps * G * D * 4;
  auto kern = full_decode_kernel<T, D, G>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_slices * C));
  cfg.blockDim = dim3(kFullThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, a, (const T*)q, (const T*)k, (const T*)v, (T*)out, (T*)kc, (T*)vc);
}

template <typename T, int D>
static cudaError_t launch_g(int G, const FullArgs& a, int n_slices, int C, const void* q, const void* k,
                            const void* v, void* out, void* kc, void* vc, cudaStream_t st) {
  switch (G) {
    case 1: return launch_one<T, D, 1>(a, n_slices, C, q, k, v, out, kc, vc, st);
    case 2: return launch_one<T, D, 2>(a, n_slices, C, q, k, v, out, kc, vc, st);
    case 4: return launch_one<T, D, 4>(a, n_slices, C, q, k, v, out, kc, vc, st);
    default: return launch_one<T, D, 8>(a, n_slices, C, q, k, v, out, kc, vc, st);
  }
}

cudaError_t launch_full_decode(int dtype, int d, int n_slices, int group, int capacity, int len, void* kc, void* vc,
                               const void* q, const void* k, const void* v, void* out, cudaStream_t st,
                               d2o_status* why) {
  (void)why;
  FullArgs a = {};
  a.capacity = capacity; a.len = len;
  int sms = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return cudaGetLastError();
  // One wave: as many CTAs per slice as there are places for (measured: 256 slices of 2049 fp16 rows 46.7 us with one CTA
  // each, 51 with two, 59 with four; 64 slices of 2001 rows with four heads 24.6 us with four CTAs each, 30 with eight).
  int C = 1;
  while (2 * C <= kFullMaxCluster && (long)n_slices * 2 * C <= (long)full_ctas(group) * sms && len + 1 >= 48 * 2 * C) C *= 2;
  if (dtype == D2O_F32)
    return d == 64 ? launch_g<float, 64>(group, a, n_slices, C, q, k, v, out, kc, vc, st)
                   : launch_g<float, 128>(group, a, n_slices, C, q, k, v, out, kc, vc, st);
  if (dtype == D2O_F16)
    return d == 64 ? launch_g<__half, 64>(group, a, n_slices, C, q, k, v, out, kc, vc, st)
                   : launch_g<__half, 128>(group, a, n_slices, C, q, k, v, out, kc, vc, st);
  return d == 64 ? launch_g<__nv_bfloat16, 64>(group, a, n_slices, C, q, k, v, out, kc, vc, st)
                 : launch_g<__nv_bfloat16, 128>(group, a, n_slices, C, q, k, v, out, kc, vc, st);
}

}  // namespace d2o
