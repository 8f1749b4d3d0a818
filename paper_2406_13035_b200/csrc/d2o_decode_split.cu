// Token generation (Section 3, Eq. 2-3; Section 4.2, Eq. 6-12) when a call has fewer slices than the GPU has room for:
// one thread-block cluster per slice = (layer, sequence, KV head) instead of one CTA (d2o_decode.cu).
//
// A model that calls layer by layer hands over one layer's slices per call: 8 for one sequence of a grouped-query model.
// With one CTA per slice 140 of the 148 SMs idle while eight CTAs walk through their rows.  Here the rows of a slice are
// divided over the C CTAs of a cluster; every CTA requests its keys and values at once and keeps both in shared memory,
// and what concerns the whole slice travels through distributed shared memory around three cluster barriers:
//
//   keys     logits of the G heads; local maximum and sum per head            -> barrier 1 (softmax normaliser)
//   values   local outputs, between arriving at barrier 1 and waiting for it
//   scores   AttnScore += probabilities (Eq. 6); local victim (Eq. 7-8); scaled partial outputs
//                                                                              -> barrier 2 (victim, outputs, failures)
//   cosines  victim's key with the resident keys (Eq. 9), local neighbour      -> barrier 3 (neighbour)
//   merge    tau_t, merge or discard, the new token's row (Eq. 10-12), by the CTA that holds the neighbour
//
// Launched with programmatic stream serialisation: the grid starts beside the one before it on the stream, loads the
// slice's state as soon as the slice's step counter shows that the previous step on the slice is complete (the state
// depends on nothing else), and only then waits for the grid before it, whose outputs the queries may be.
//
// A CTA writes into another's shared memory only before a barrier that both wait for, and reads from another's only
// before barrier 3.  Nothing of the slice is written before barrier 2 has shown that no CTA's wait ran out.
#include <cooperative_groups.h>
#include <math.h>

#include "d2o_common.cuh"
#include "d2o_decode.cuh"

namespace cg = cooperative_groups;

namespace d2o {

constexpr int kSplitThreads = 256;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kSplitMaxCluster = 16;
constexpr int kSplitPiece = 64;                          // rows per bulk copy
constexpr int kSplitMaxRows = 512;                       // rows per CTA: two per thread
constexpr int kSplitPieces = kSplitMaxRows / kSplitPiece;

__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// What the CTAs of a cluster tell one another; entry r comes from rank r.
template <int G>
struct SplitExchange {
  float m[kSplitMaxCluster][G], l[kSplitMaxCluster][G];          // barrier 1: maximum and sum of the rank's rows
  unsigned long long vkey[kSplitMaxCluster], nkey[kSplitMaxCluster];   // barriers 2, 3: best victim / neighbour
  int vli[kSplitMaxCluster], nli[kSplitMaxCluster];              // and its row in the slice
  int bad1[kSplitMaxCluster], bad2[kSplitMaxCluster];            // a wait ran out, or an anomaly was recorded before
  float new_score;                                               // of the new token, from the rank that holds it
};

// Extremum of n <= 32 keys in shared memory and its row; every lane of the calling warp gets it.
template <bool MIN>
__device__ __forceinline__ unsigned long long keys_extreme(const unsigned long long* key, const int* li, int n, int* out_li) {
  const int lane = threadIdx.x & 31;
  const unsigned long long k = lane < n ? key[lane] : (MIN ? ~0ull : 0ull);
  const unsigned long long w = MIN ? warp_min_u64(k) : warp_max_u64(k);
  const int src = __ffs(__ballot_sync(0xffffffffu, k == w)) - 1;
  *out_li = __shfl_sync(0xffffffffu, lane < n ? li[lane] : -1, src);
  return w;
}

// `a.row_cap`: rows per CTA the shared arrays are sized for.
template <typename T, int D, int G>
__global__ void __launch_bounds__(kSplitThreads, G <= 4 ? 2 : 1)
decode_split_kernel(DecodeArgs a, const T* __restrict__ q_in, const T* __restrict__ k_in, const T* __restrict__ v_in,
                    T* __restrict__ out, T* __restrict__ kpool, T* __restrict__ vpool) {
  constexpr int EPV = Elem<T>::kPerVec;
  constexpr int LPR = D / EPV;                            // lanes that share one row (16-byte segment each)
  constexpr int NGRP = kSplitThreads / LPR;               // row groups
  constexpr int BLK = 4 * NGRP;                           // rows per pass over the groups: four per group
  constexpr int QL = LPR / 4;                             // lanes that end up with the same row total after reduce4
  constexpr int ROWB = D * (int)sizeof(T);
  constexpr int R = kSplitMaxRows / kSplitThreads;        // rows whose score a thread keeps
  constexpr int OUT = (G * D + kSplitThreads - 1) / kSplitThreads;

  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = tid / LPR, lig = tid % LPR;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- which slice
  const int item = (int)blockIdx.x / C;
  const int h = item % a.Hkv;
  const int layer = a.l0 + item / (a.B * a.Hkv), b = (item / a.Hkv) % a.B;
  const int sl = ((layer - a.l0) * a.B + b) * a.Hkv + h;
  const int sidx = (layer * a.B + b) * a.Hkv + h;
  const T* k_new = k_in + (size_t)sl * D;
  const T* v_new = v_in + (size_t)sl * D;

  // ---- shared memory
  extern __shared__ __align__(128) unsigned char dsm[];
  const int cap = a.row_cap;
  uint4* sK = reinterpret_cast<uint4*>(dsm);                              // [cap][LPR]
  uint4* sV = sK + (size_t)cap * LPR;                                     // [cap][LPR]
  float* red = reinterpret_cast<float*>(sV + (size_t)cap * LPR);          // [warps][G][D]
  float* part = red + kSplitWarps * G * D;                                // [C][G * D / C] partial outputs of this rank's share
  float* pl = part + G * D;                                               // [G][cap] logits, then 2^{x - local maximum}
  float* s_rn = pl + (size_t)G * cap;                                     // [cap] 1/|k|
  int* s_ps = reinterpret_cast<int*>(s_rn + cap);                         // [cap] positions
  __shared__ SplitExchange<G> xch;
  __shared__ unsigned long long s_k[kSplitPieces], s_v[kSplitPieces];
  __shared__ volatile int s_timeout;                                      // 1: nothing may be done; 2: a wait of this CTA ran out
  __shared__ float s_red[2][kSplitWarps][G], s_fac[G], s_new_rn;
  __shared__ unsigned long long s_key[kSplitWarps];
  __shared__ int s_li[kSplitWarps];

  if (tid == 0) {
    for (int i = 0; i < kSplitPieces; ++i) { mbar_init(&s_k[i], 1); mbar_init(&s_v[i], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  // barrier 0: every CTA of the cluster has started before anything is written into its shared memory
  cluster_arrive();
  if (!a.early) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == 0) {
    int stop = *reinterpret_cast<volatile uint32_t*>(a.status) != 0u;
    if (!stop && a.early) {
      stop = slice_ready(a.steps_done + sidx, a.step, a.status, a.chained ? a.wait_ns : 20000ull);
      if (stop == 2 && !a.chained) {                                      // not soon: behind the grid ahead it is certain
        asm volatile("griddepcontrol.wait;" ::: "memory");
        stop = slice_ready(a.steps_done + sidx, a.step, a.status, a.wait_ns);
      }
      // rows that the previous step's cluster wrote with ordinary stores are read here by bulk copies
      asm volatile("fence.proxy.async.global;" ::: "memory");
    }
    s_timeout = stop;
  }
  // ---- slice parameters that do not change from step to step
  const int e = slice_entry(b, layer, h, a.L, a.Hkv);
  const int t_pos = a.plen[b] + a.step;
  const int S = a.budgets[e], M = a.windows[e];
  const int64_t row0 = a.row_off[e];
  const int Tn = a.T < S ? a.T : S;
  __syncthreads();
  // ---- the rows [r0, r0 + cnt) of the n = n_old + 1 (the new token is row n_old) of this rank
  const int n_old = a.len[sidx];
  const float tau_old = a.tau[sidx];
  const int n = n_old + 1;
  const bool evict = n > S;
  const int chunk = (n + C - 1) / C;
  const int r0 = min(rank * chunk, n);
  const int cnt = min(n, r0 + chunk) - r0;
  const int new_li = n_old - r0;                                          // local row of the new token, if within [0, cnt)
  const bool has_new = new_li >= 0 && new_li < cnt;
  if (tid == 0 && s_timeout == 0) {
    if (chunk > cap) { report_error(a.status, D2O_ERR_STATE, 0xDEC30000u | (uint32_t)(sl & 0xffff)); s_timeout = 1; }
    if (!D2O_GUARD(S >= 1 && n_old >= 0 && n_old <= S && row0 >= 0 && row0 + slice_stride(S) <= a.pool_rows, a.status, 0xC4EC0010u))
      s_timeout = 1;
  }
  const bool run = __syncthreads_or(s_timeout != 0) == 0;                 // if not: nothing is loaded, the cluster leaves after barrier 1
  const int n_pc = run ? (cnt + kSplitPiece - 1) / kSplitPiece : 0;

  // ---- all keys, then all values; the new token's row follows once the inputs may be read
  int issued = 0;                                                         // thread 0
  if (tid == 0) {
    unsigned long long drop = 0;
    if (a.l2_hints) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(drop));
    for (int i = 0; i < 2 * n_pc; ++i) {
      if (a.stop_stage >= 0 && i >= a.stop_stage) break;                  // failure-detection tests: never arrives
      issued = i + 1;
      const bool is_v = i >= n_pc;
      const int a0 = (is_v ? i - n_pc : i) * kSplitPiece;
      const int np = min(min(cnt, a0 + kSplitPiece), new_li) - a0;        // cache rows: all but the new token's, the last of the slice
      unsigned long long* bar = is_v ? &s_v[i - n_pc] : &s_k[i];
      mbar_expect_tx(bar, (uint32_t)(max(np, 0) * ROWB));
      if (np > 0) {
        uint4* dst = (is_v ? sV : sK) + (size_t)a0 * LPR;
        const T* src = (is_v ? vpool : kpool) + (row0 + r0 + a0) * D;
        if (a.l2_hints) bulk_g2s_hint(dst, src, (uint32_t)(np * ROWB), bar, drop);
        else bulk_g2s(dst, src, (uint32_t)(np * ROWB), bar);
      }
    }
  }
  // ---- per-row state, while the rows are on their way
  float sc[R]; int ps[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int li = tid + r * kSplitThreads;
    sc[r] = 0.f; ps[r] = t_pos;
    if (run && li < cnt) {
      if (li != new_li) {
        sc[r] = a.score[row0 + r0 + li];
        ps[r] = a.pos[row0 + r0 + li];
        s_rn[li] = a.rnorm[row0 + r0 + li];
      }
      s_ps[li] = ps[r];
    }
  }
  // ---- from here on the inputs: the grid ahead on the stream must be done (unless the call promised them complete)
  if (a.early && !a.chained) asm volatile("griddepcontrol.wait;" ::: "memory");
  const float qscale = (D == 64 ? 0.125f : 0.08838834764831845f) * kLog2e;   // log2(e)/sqrt(d)
  float qf[G][EPV];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    Elem<T>::unpack(ld_global_v4(q_in + ((size_t)sl * G + g) * D + lig * EPV), qf[g]);
#pragma unroll
    for (int i = 0; i < EPV; ++i) qf[g][i] *= qscale;
  }
  if (warp == 0) {
    const uint4 kn = lane < LPR ? ld_global_v4(k_new + lane * EPV) : make_uint4(0, 0, 0, 0);
    const uint4 vn = lane < LPR ? ld_global_v4(v_new + lane * EPV) : make_uint4(0, 0, 0, 0);
    float f[EPV];
    Elem<T>::unpack(kn, f);
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < EPV; ++i) ss = fmaf(f[i], f[i], ss);
    ss = warp_sum(ss);
    const float rn = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;                   // 1/|k| of the new token
    if (lane == 0) {
      s_new_rn = rn;
      if (run && has_new) s_rn[new_li] = rn;
    }
    if (run && has_new && lane < LPR) { sK[(size_t)new_li * LPR + lane] = kn; sV[(size_t)new_li * LPR + lane] = vn; }
  }
  __syncthreads();

  // ---- pass K: logits
  float mx[G];
#pragma unroll
  for (int g = 0; g < G; ++g) mx[g] = -INFINITY;
  if (run) {
    int seen = 0;
    for (int base = 0; base < cnt; base += BLK) {
      for (const int end = min(cnt, base + BLK); seen * kSplitPiece < end; ++seen) stage_wait(&s_k[seen], 0u, &s_timeout, a.wait_ns);
      __syncwarp();
      uint4 raw[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int li = base + u * NGRP + grp;
        raw[u] = li < cnt ? sK[(size_t)li * LPR + lig] : make_uint4(0, 0, 0, 0);
      }
      float dot[G][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float f[EPV];
        Elem<T>::unpack(raw[u], f);
#pragma unroll
        for (int g = 0; g < G; ++g) dot[g][u] = dot_pairs<EPV>(qf[g], f);
      }
      const int li = base + (lig / QL) * NGRP + grp;                      // the row whose total this lane receives
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float x = reduce4<LPR>(dot[g][0], dot[g][1], dot[g][2], dot[g][3], lig);
        if (li < cnt) {
          mx[g] = fmaxf(mx[g], x);
          if (lig % QL == 0) pl[(size_t)g * cap + li] = x;
        }
      }
    }
  }
  // ---- local softmax statistics -> barrier 1
#pragma unroll
  for (int g = 0; g < G; ++g) { const float w = warp_max(mx[g]); if (lane == 0) s_red[0][warp][g] = w; }
  __syncthreads();
#pragma unroll
  for (int g = 0; g < G; ++g) {
    float t = s_red[0][0][g];
#pragma unroll
    for (int w = 1; w < kSplitWarps; ++w) t = fmaxf(t, s_red[0][w][g]);
    mx[g] = t;
  }
  {
    float sum[G];
#pragma unroll
    for (int g = 0; g < G; ++g) sum[g] = 0.f;
    if (run)
      for (int li = tid; li < cnt; li += kSplitThreads) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const float p = exp2f(pl[(size_t)g * cap + li] - mx[g]);
          pl[(size_t)g * cap + li] = p;
          sum[g] += p;
        }
      }
#pragma unroll
    for (int g = 0; g < G; ++g) { const float w = warp_sum(sum[g]); if (lane == 0) s_red[1][warp][g] = w; }
  }
  cluster_wait();                                                         // barrier 0
  __syncthreads();
  if (warp == 0 && lane < C) {
    SplitExchange<G>* x = cluster.map_shared_rank(&xch, lane);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float t = 0.f;
#pragma unroll
      for (int w = 0; w < kSplitWarps; ++w) t += s_red[1][w][g];
      x->m[rank][g] = mx[g];
      x->l[rank][g] = t;
    }
    x->bad1[rank] = s_timeout;
  }
  cluster_arrive();                                                       // barrier 1

  // ---- pass V: un-normalised outputs of this rank's rows
  float o[OUT];
#pragma unroll
  for (int i = 0; i < OUT; ++i) o[i] = 0.f;
  {
    float acc[G][EPV];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int i = 0; i < EPV; ++i) acc[g][i] = 0.f;
    if (run) {
      int seen = 0;
      for (int base = 0; base < cnt; base += BLK) {
        for (const int end = min(cnt, base + BLK); seen * kSplitPiece < end; ++seen) stage_wait(&s_v[seen], 0u, &s_timeout, a.wait_ns);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int li = base + u * NGRP + grp;
          if (li < cnt) {
            float f[EPV];
            Elem<T>::unpack(sV[(size_t)li * LPR + lig], f);
#pragma unroll
            for (int g = 0; g < G; ++g) {
              const float p = pl[(size_t)g * cap + li];
#pragma unroll
              for (int i = 0; i < EPV; i += 2) {
                const float2 t = ffma2(make_float2(p, p), make_float2(f[i], f[i + 1]), make_float2(acc[g][i], acc[g][i + 1]));
                acc[g][i] = t.x; acc[g][i + 1] = t.y;
              }
            }
          }
        }
      }
    }
#pragma unroll
    for (int s = LPR; s < 32; s <<= 1)
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int i = 0; i < EPV; ++i) acc[g][i] += __shfl_xor_sync(0xffffffffu, acc[g][i], s);
    if (lane < LPR) {
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int i = 0; i < EPV; i += 4)
          *reinterpret_cast<float4*>(&red[(warp * G + g) * D + lane * EPV + i]) =
              make_float4(acc[g][i], acc[g][i + 1], acc[g][i + 2], acc[g][i + 3]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < OUT; ++i) {
      const int at = tid + i * kSplitThreads;
      if (at < G * D) {
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) o[i] += red[w * G * D + at];
      }
    }
  }

  // A chained grid must not be complete before its predecessor (whatever the stream runs next is ordered behind this
  // grid only): one CTA that stays until then is enough.
  auto hold = [&]() { if (a.chained && blockIdx.x == gridDim.x - 1) asm volatile("griddepcontrol.wait;" ::: "memory"); };
  // A CTA must not end while copies are on their way into its shared memory; a cluster that gives up sees its own land.
  auto leave = [&](uint32_t detail) {
    if (tid == 0) {
      if (s_timeout == 2) report_error(a.status, D2O_ERR_TIMEOUT, detail | (uint32_t)(sl & 0xffff));
      for (int i = 0; i < issued; ++i)
        if (!landed_wait(i < n_pc ? &s_k[i] : &s_v[i - n_pc], 0u, a.wait_ns)) break;
    }
    hold();
  };
  cluster_wait();                                                         // barrier 1
  // a CTA found an anomaly, or its keys did not arrive: the whole cluster leaves, nothing has been written
  int bad = 0;
  for (int r = 0; r < C; ++r) bad |= xch.bad1[r];
  if (bad) { leave(0xDEC10000u); return; }
  if (warp < G) {
    const float all = warp_max(lane < C ? xch.m[lane][warp] : -INFINITY);
    const float l = warp_sum(lane < C ? xch.l[lane][warp] * exp2f(xch.m[lane][warp] - all) : 0.f);
    // turns this rank's 2^{x - local maximum} into probabilities; 0 for a rank without rows
    if (lane == 0) s_fac[warp] = exp2f(xch.m[rank][warp] - all) / l;
  }
  __syncthreads();

  // ---- accumulated attention (Eq. 6 case 2), local victim (Eq. 7-8), scaled outputs -> barrier 2
  unsigned long long best = ~0ull; int best_li = -1;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int li = tid + r * kSplitThreads;
    if (li < cnt) {
      float p = 0.f;
#pragma unroll
      for (int g = 0; g < G; ++g) p = fmaf(pl[(size_t)g * cap + li], s_fac[g], p);
      sc[r] += p;
      if (ps[r] >= Tn && ps[r] <= t_pos - M) {                            // lowest score, ties -> latest position
        const unsigned long long key = ((unsigned long long)float_ord(sc[r]) << 32) | (uint32_t)(0x7fffffff - ps[r]);
        if (key < best) { best = key; best_li = r0 + li; }
      }
      if (li == new_li)
        for (int t = 0; t < C; ++t) cluster.map_shared_rank(&xch, t)->new_score = sc[r];
    }
  }
  auto block_key = [&](unsigned long long key, int li, bool lowest) {      // per-warp extremum into s_key, s_li
    const unsigned long long w = lowest ? warp_min_u64(key) : warp_max_u64(key);
    const int src = __ffs(__ballot_sync(0xffffffffu, key == w)) - 1;
    const int wli = __shfl_sync(0xffffffffu, li, src);
    if (lane == 0) { s_key[warp] = w; s_li[warp] = wli; }
  };
  __syncwarp();
  block_key(best, best_li, true);
  const int share = G * D / C;                                            // outputs a rank finishes
#pragma unroll
  for (int i = 0; i < OUT; ++i) {
    const int at = tid + i * kSplitThreads;
    if (at < G * D) cluster.map_shared_rank(part, at / share)[rank * share + at % share] = o[i] * s_fac[at / D];
  }
  __syncthreads();
  if (warp == 0) {
    int wli;
    const unsigned long long w = keys_extreme<true>(s_key, s_li, kSplitWarps, &wli);
    if (lane < C) {
      SplitExchange<G>* x = cluster.map_shared_rank(&xch, lane);
      x->vkey[rank] = w; x->vli[rank] = wli;
      x->bad2[rank] = s_timeout;
    }
  }
  cluster_arrive();                                                       // barrier 2
  cluster_wait();
  for (int r = 0; r < C; ++r) bad |= xch.bad2[r];
  if (bad) { leave(0xDEC10000u); return; }                                // the values did not arrive: nothing written yet

  // ---- the neighbour of the victim: its key with the resident keys (Eq. 9) -> barrier 3
  int vic_li = -1;
  const unsigned long long vbest = keys_extreme<true>(xch.vkey, xch.vli, C, &vic_li);
  const bool none = evict && vbest == ~0ull;                              // S_l < T + M: nothing may be evicted
  float kvic[EPV];
  uint4 vvic = make_uint4(0, 0, 0, 0);
  if (evict && !none) {
    if (!D2O_GUARD(vic_li >= 0 && vic_li <= n_old, a.status, 0xC4EC0011u)) vic_li = n_old;
    const int vr = vic_li / chunk, vl = vic_li % chunk;                   // who holds it
    Elem<T>::unpack(cluster.map_shared_rank(sK, vr)[(size_t)vl * LPR + lig], kvic);
    const float vic_rn = cluster.map_shared_rank(s_rn, vr)[vl];
    if (warp == 0 && lane < LPR) vvic = cluster.map_shared_rank(sV, vr)[(size_t)vl * LPR + lane];
    best = 0ull; best_li = -1;
    for (int base = 0; base < cnt; base += BLK) {
      float dot[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int li = base + u * NGRP + grp;
        float f[EPV];
        Elem<T>::unpack(li < cnt ? sK[(size_t)li * LPR + lig] : make_uint4(0, 0, 0, 0), f);
        dot[u] = dot_pairs<EPV>(kvic, f);
      }
      const float x = reduce4<LPR>(dot[0], dot[1], dot[2], dot[3], lig);
      const int li = base + (lig / QL) * NGRP + grp;
      if (lig % QL == 0 && li < cnt && r0 + li != vic_li) {               // max similarity, ties -> earliest position
        const unsigned long long key = ((unsigned long long)sim_ord(x * vic_rn * s_rn[li]) << 32) | (uint32_t)(0x7fffffff - s_ps[li]);
        if (key > best) { best = key; best_li = r0 + li; }
      }
    }
    __syncwarp();
    block_key(best, best_li, false);
    __syncthreads();
    if (warp == 0) {
      int wli;
      const unsigned long long w = keys_extreme<false>(s_key, s_li, kSplitWarps, &wli);
      if (lane < C) {
        SplitExchange<G>* x = cluster.map_shared_rank(&xch, lane);
        x->nkey[rank] = w; x->nli[rank] = wli;
      }
    }
  }
  // ---- scores of this rank's rows; the new token's goes with its row, wherever that ends up
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int li = tid + r * kSplitThreads;
    if (li < cnt && (li != new_li || !evict)) a.score[row0 + r0 + li] = sc[r];
  }
  cluster_arrive();                                                       // barrier 3
  // ---- this rank's share of the outputs (Eq. 3)
  if (!none) {
    for (int i = tid; i < share; i += kSplitThreads) {
      float t = 0.f;
      for (int r = 0; r < C; ++r) t += part[r * share + i];
      out[(size_t)sl * G * D + rank * share + i] = Elem<T>::from_float(t);
    }
  }
  hold();
  cluster_wait();
  if (none) {
    // report, drop the new token, keep the cache as it is
    if (rank == 0 && tid == 0) report_error(a.status, D2O_ERR_STATE, 0xDEC00000u | (uint32_t)(sl & 0xfffff));
    return;
  }

  // ---- threshold, merge or discard (Eq. 10-12), the new token's row: by the CTA that holds the neighbour (or, while
  // the cache still fills, the new token)
  if (warp != 0) return;
  int nn_li = -1;
  const unsigned long long nbest = evict ? keys_extreme<false>(xch.nkey, xch.nli, C, &nn_li) : 0ull;
  if ((evict ? max(nn_li, 0) : n_old) / chunk != rank) return;
  if (!evict) {
    if (lane < LPR) {
      *reinterpret_cast<uint4*>(kpool + (row0 + n_old) * D + lane * EPV) = sK[(size_t)new_li * LPR + lane];
      *reinterpret_cast<uint4*>(vpool + (row0 + n_old) * D + lane * EPV) = sV[(size_t)new_li * LPR + lane];
    }
    if (lane == 0) { a.pos[row0 + n_old] = t_pos; a.rnorm[row0 + n_old] = s_new_rn; a.len[sidx] = n; }
  } else {
    const float u = ord_float((uint32_t)(nbest >> 32));
    const float tau_new = a.beta * u + (1.0f - a.beta) * tau_old;
    const float thr = isnan(a.tau_override) ? tau_new : a.tau_override;
    bool merge = u >= thr && nn_li >= 0;
    if (!D2O_GUARD(nn_li >= 0 && nn_li <= n_old && nn_li != vic_li, a.status, 0xC4EC0012u)) merge = false;
    const bool nn_is_new = nn_li == n_old;
    const float ew = expf(u);
    const float w_e = a.average ? 0.5f : ew / (ew + kEuler);
    const float w_c = a.average ? 0.5f : kEuler / (ew + kEuler);
    if (lane < LPR) {
      uint4 kslot = ld_global_v4(k_new + lane * EPV), vslot = ld_global_v4(v_new + lane * EPV);
      float rn_slot = s_new_rn;
      if (merge) {
        float fk[EPV], fv[EPV], vv[EPV];
        Elem<T>::unpack(sK[(size_t)(nn_li - r0) * LPR + lane], fk);
        Elem<T>::unpack(sV[(size_t)(nn_li - r0) * LPR + lane], fv);
        Elem<T>::unpack(vvic, vv);
#pragma unroll
        for (int i = 0; i < EPV; ++i) { fk[i] = w_c * fk[i] + w_e * kvic[i]; fv[i] = w_c * fv[i] + w_e * vv[i]; }
        const uint4 kn = Elem<T>::pack(fk), vn = Elem<T>::pack(fv);
        Elem<T>::unpack(kn, fk);                                          // norm of what is stored
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < EPV; ++i) ss = fmaf(fk[i], fk[i], ss);
        ss = group_sum<LPR>(ss, group_mask<LPR>());
        const float rnew = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
        if (nn_is_new) { kslot = kn; vslot = vn; rn_slot = rnew; }
        else {
          *reinterpret_cast<uint4*>(kpool + (row0 + nn_li) * D + lane * EPV) = kn;
          *reinterpret_cast<uint4*>(vpool + (row0 + nn_li) * D + lane * EPV) = vn;
          if (lane == 0) a.rnorm[row0 + nn_li] = rnew;
        }
      }
      if (vic_li != n_old) {
        *reinterpret_cast<uint4*>(kpool + (row0 + vic_li) * D + lane * EPV) = kslot;
        *reinterpret_cast<uint4*>(vpool + (row0 + vic_li) * D + lane * EPV) = vslot;
        if (lane == 0) {
          a.pos[row0 + vic_li] = t_pos;
          a.score[row0 + vic_li] = xch.new_score;
          a.rnorm[row0 + vic_li] = rn_slot;
        }
      }
    }
    if (lane == 0) {
      a.tau[sidx] = tau_new;
      atomicAdd(&a.counters[kCntEvictions], 1ull);
      atomicAdd(&a.counters[merge ? kCntMerges : kCntDiscards], 1ull);
    }
  }
  if (lane == 0) atomicAdd(&a.counters[kCntDecodeSteps], 1ull);
  // every other CTA's stores to the state were ordered before barrier 3, this warp's before the release
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncwarp();
  if (lane == 0) asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.steps_done + sidx), "r"(a.step + 1) : "memory");
}

// ------------------------------------------------------------------------------------ launch
// shared memory of a CTA with room for `rows` rows
static size_t split_smem(int rows, int G, int D, int esz) {
  return (size_t)rows * (2 * D * esz + G * 4 + 8) + (size_t)(kSplitWarps + 1) * G * D * 4;
}

#ifndef SPLIT_BYTES
#define SPLIT_BYTES (24l << 20)
#endif

// CTAs per slice, or 0 when one CTA per slice (decode_kernel) is the better choice or the rows do not fit.
int decode_split_cluster(const d2o_ctx* c, int n_slices, int max_rows) {
  const d2o_config& g = c->cfg;
  if ((long)n_slices * max_rows * 2 * g.d_head * c->elem_size > SPLIT_BYTES) return 0;
#ifdef SPLIT_FORCE
  int C = SPLIT_FORCE;
#else
  int C = 1;
  while (2 * C <= c->max_cluster && 2L * C * g.batch * g.n_kv_heads <= c->n_sms) C *= 2;
  if (C == 1) return 0;
#endif
  const size_t room = 227 * 1024 - 4096;                                  // 4 KB for the static shared arrays
  for (; C <= c->max_cluster; C *= 2) {
    const int rows = (max_rows + C - 1) / C;
    if (rows <= kSplitMaxRows && split_smem(rows, c->group, g.d_head, c->elem_size) <= room) return C;
  }
  return 0;
}

// Largest cluster the kernels can be launched with on the current device (8 is always possible).
int decode_split_max_cluster() {
  auto kern = decode_split_kernel<float, 128, 8>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kSplitMaxCluster); cfg.blockDim = dim3(kSplitThreads); cfg.dynamicSmemBytes = 220 * 1024;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kSplitMaxCluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 8;
  }
  return n > 0 ? kSplitMaxCluster : 8;
}

template <typename T, int D, int G>
static cudaError_t launch_one(const DecodeArgs& a, int C, int n_slices, const void* q, const void* k, const void* v,
                              void* out, void* kpool, void* vpool, cudaStream_t st) {
  const size_t smem = split_smem(a.row_cap, G, D, (int)sizeof(T));
  auto kern = decode_split_kernel<T, D, G>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_slices * C)); cfg.blockDim = dim3(kSplitThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, a, (const T*)q, (const T*)k, (const T*)v, (T*)out, (T*)kpool, (T*)vpool);
}

template <typename T, int D>
static cudaError_t launch_g(int G, const DecodeArgs& a, int C, int n_slices, const void* q, const void* k, const void* v,
                            void* out, void* kpool, void* vpool, cudaStream_t st) {
  switch (G) {
    case 1: return launch_one<T, D, 1>(a, C, n_slices, q, k, v, out, kpool, vpool, st);
    case 2: return launch_one<T, D, 2>(a, C, n_slices, q, k, v, out, kpool, vpool, st);
    case 4: return launch_one<T, D, 4>(a, C, n_slices, q, k, v, out, kpool, vpool, st);
    default: return launch_one<T, D, 8>(a, C, n_slices, q, k, v, out, kpool, vpool, st);
  }
}

// One step of `n_slices` slices (in index order) with `C` CTAs each.  `a.chained`, `a.publish`: see launch_decode;
// `a.early`: the step counters of the slices are kept up to date, so the kernel may look at them.
cudaError_t launch_decode_split(const d2o_ctx* c, DecodeArgs a, int C, int n_slices, int max_rows, const void* q,
                                const void* k, const void* v, void* out, void* kpool, void* vpool, cudaStream_t st) {
  const d2o_config& g = c->cfg;
  a.row_cap = (max_rows + C - 1) / C;
  if (g.dtype == D2O_F32)
    return g.d_head == 64 ? launch_g<float, 64>(c->group, a, C, n_slices, q, k, v, out, kpool, vpool, st)
                          : launch_g<float, 128>(c->group, a, C, n_slices, q, k, v, out, kpool, vpool, st);
  if (g.dtype == D2O_F16)
    return g.d_head == 64 ? launch_g<__half, 64>(c->group, a, C, n_slices, q, k, v, out, kpool, vpool, st)
                          : launch_g<__half, 128>(c->group, a, C, n_slices, q, k, v, out, kpool, vpool, st);
  return g.d_head == 64 ? launch_g<__nv_bfloat16, 64>(c->group, a, C, n_slices, q, k, v, out, kpool, vpool, st)
                        : launch_g<__nv_bfloat16, 128>(c->group, a, C, n_slices, q, k, v, out, kpool, vpool, st);
}

}  // namespace d2o
