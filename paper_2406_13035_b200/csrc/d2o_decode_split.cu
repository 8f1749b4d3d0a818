// Token generation (Section 3, Eq. 2-3; Section 4.2, Eq. 6-12) when a call has fewer slices than the GPU has room for:
// one thread-block cluster per slice = (layer, sequence, KV head) instead of one CTA (d2o_decode.cu).
//
// A model that calls layer by layer hands over one layer's slices per call: 8 for one sequence of a grouped-query model.
// With one CTA per slice 140 of the 148 SMs idle while eight CTAs walk through their rows.  Here the rows of a slice are
// divided over the C CTAs of a cluster; every CTA requests its keys and values at once and keeps both in shared memory,
// and what concerns the whole slice travels through distributed shared memory around cluster barriers:
//
//   guess    the row with the lowest score as it stands before the step, among those that may be evicted, is nearly
//            always the victim (see d2o_decode.cu)                              -> barrier G
//            its key with the resident keys (Eq. 9), best neighbour
//   ----- up to here only the slice's state is read, nothing of the step's inputs -----
//   keys     logits of the G heads; maximum and sum per head                    -> barrier 1 (softmax normaliser)
//   values   un-normalised outputs, between arriving at barrier 1 and waiting for it
//   scores   AttnScore += probabilities (Eq. 6); victim (Eq. 7-8); partial outputs -> barrier 2 (victim, outputs, failures)
//            a wrong guess: cosines of the true victim, one more barrier
//   outputs, merge: tau_t, merge or discard, the new token's row (Eq. 10-12), by the CTA that holds the neighbour
//
// The kernel is bound by this chain of latencies, not by bandwidth or arithmetic, so a warp works alone wherever it can:
// it owns every eighth tile of 16 rows from the logits to the cosines and writes its own entries (maximum and sum, best
// victim, best neighbour) into every CTA of the cluster; the only block-wide step is the sum of the warps' outputs.
// 16-bit caches with several heads per slice run both passes and the cosines on mma.sync (d2o_decode.cu describes the
// layout), fp32 caches and single heads on FMAs (tensor_path).
//
// Launched with programmatic stream serialisation: the grid starts beside the one before it on the stream, loads the
// slice's state as soon as the slice's step counter shows that the previous step on the slice is complete (from the second
// step after a compression on the state depends on nothing else), and only then waits for the grid before it, whose outputs
// the queries may be.  The first step after a compression waits for the grids ahead before it reads anything: the counter
// says nothing about the prompt stage, whose last kernels may still be at work.
//
// Who writes the step counter.  A step that tells by itself that a slice is complete has to collect the stores of the whole
// cluster first: one more cluster barrier and a release, 1.5 us of every call.  Where calls alternate between layers the next
// call does it instead: behind its wait for the grid ahead that grid's stores are all visible, and a warp of its last CTA writes
// the counters (DecodeArgs::pub_first).  A chained step, one that follows a step on the same layers, and one whose next call is
// likely to take decode_kernel (launch_decode) writes its own.
// Calls layer by layer, us a call, with the barrier / so: 32 layers of 8 slices of 1640 bf16 rows, four heads, 11.5 / 10.7; 24 layers of
// 32 fp16 slices of 450 rows, one head, 10.2 / 9.5; 5 layers of 24 fp32 slices of 180 rows 7.8 / 7.0.  (A release by every rank in
// the place of the barrier: 11.4 and 9.9.)
//
// A CTA writes into another's shared memory only before it arrives at a barrier that the other waits for before it ends (on the
// way out after a wait that ran out there is a barrier for that), and reads from another's only before such a barrier.
// Nothing of the slice is written before barrier 2 has shown that no CTA's wait ran out.
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include "d2o_common.cuh"
#include "d2o_decode.cuh"

namespace cg = cooperative_groups;

namespace d2o {

constexpr int kSplitThreads = 256;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kSplitMaxCluster = 16;
constexpr int kSplitPiece = 32;                          // rows per copy: two tiles of 16
constexpr int kSplitMaxRows = 512;                       // rows per CTA: two per thread, four tiles per warp
constexpr int kSplitPieces = kSplitMaxRows / kSplitPiece;
constexpr int kSplitEntries = kSplitMaxCluster * kSplitWarps;

__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// What the warps of a cluster tell one another; entry 8 r + w comes from warp w of rank r.
template <int G>
struct SplitExchange {
  float m[kSplitEntries][G], l[kSplitEntries][G];                // barrier 1: maximum and sum over the warp's rows
  unsigned long long vkey[kSplitEntries], nkey[kSplitEntries];   // best victim (guess, then barrier 2) / its neighbour
  int vli[kSplitEntries], nli[kSplitEntries];                    // and its row in the slice
  int bad1[kSplitEntries], bad2[kSplitEntries];                  // a wait ran out, or an anomaly was recorded before
  float new_score;                                               // of the new token, from the warp that holds it
  unsigned long long new_nkey;                                   // and its cosine with the guessed victim
};

// Extremum of n keys in shared memory and its row; every lane of the calling warp gets it.
template <bool MIN>
__device__ __forceinline__ unsigned long long keys_extreme(const unsigned long long* key, const int* li, int n, int* out_li) {
  const int lane = threadIdx.x & 31;
  unsigned long long k = MIN ? ~0ull : 0ull;
  int kl = -1;
#pragma unroll
  for (int i = 0; i < kSplitEntries / 32; ++i)
    if (i * 32 + lane < n) {
      const unsigned long long t = key[i * 32 + lane];
      if (MIN ? t < k : t > k) { k = t; kl = li[i * 32 + lane]; }
    }
  const unsigned long long w = MIN ? warp_min_u64(k) : warp_max_u64(k);
  const int src = __ffs(__ballot_sync(0xffffffffu, k == w)) - 1;
  *out_li = __shfl_sync(0xffffffffu, kl, src);
  return w;
}

// `a.row_cap`: rows per CTA the shared arrays are sized for (a multiple of kSplitPiece).
// kPublish (DecodeArgs::publish): the step writes its own counters.  Compiled for either: with both paths in one kernel, and the
// inputs asked into L2 for both, repeated and chained steps were slower (8 steps of 4 layers of 8 bf16 slices of 410 rows 100.7 -> 103.7
// us, chained 99.4 -> 101.4; so 101.8 and 100.2; layer by layer, four tokens of 32 layers, 1370 -> 1345).
template <typename T, int D, int G, bool kPublish>
__global__ void __launch_bounds__(kSplitThreads, G <= 4 ? 2 : 1)
decode_split_kernel(DecodeArgs a, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const T* q_in, const T* k_in, const T* v_in, T* __restrict__ out,
                    T* __restrict__ kpool, T* __restrict__ vpool) {
  constexpr bool kTensor = tensor_path((int)sizeof(T), G);      // both passes and the cosines on mma.sync
  constexpr int EPV = Elem<T>::kPerVec;
  constexpr int LPR = D / EPV;                            // 16-byte segments of a row; lanes that share a row
  constexpr int WG = 32 / LPR;                            // rows a warp's lanes cover at a time
  constexpr int QL = LPR / 4;                             // lanes that end up with the same row total after reduce4
  constexpr int ROWB = D * (int)sizeof(T);
  constexpr int NH = kTensor ? ROWB / 128 : 1;            // 128-byte halves of a row
  constexpr int R = kSplitMaxRows / kSplitThreads;        // rows whose score a lane keeps
  constexpr int OUT = (G * D + kSplitThreads - 1) / kSplitThreads;

  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lig = lane % LPR, wg = lane / LPR, gid = lane >> 2, tig = lane & 3;
  if (a.early) start_dependents();

  // ---- which slice
  const int item = (int)blockIdx.x / C;
  const int h = item % a.Hkv;
  const int layer = a.l0 + item / (a.B * a.Hkv), b = (item / a.Hkv) % a.B;
  const int sl = ((layer - a.l0) * a.B + b) * a.Hkv + h;
  const int sidx = (layer * a.B + b) * a.Hkv + h;
  const T* k_new = k_in + (size_t)sl * D;
  const T* v_new = v_in + (size_t)sl * D;
  // The inputs may still be on their way from the grid ahead and are not read before it is done, but their lines can be in L2 by
  // then.
  if (!kPublish && a.early) {
    constexpr int kQ = G * D * (int)sizeof(T) / 128, kR = D * (int)sizeof(T) / 128;            // lines of the queries, of a row
    const char* line = tid < kQ ? reinterpret_cast<const char*>(q_in + (size_t)sl * G * D) + tid * 128
                     : tid < kQ + kR ? reinterpret_cast<const char*>(k_new) + (tid - kQ) * 128
                                     : reinterpret_cast<const char*>(v_new) + (tid - kQ - kR) * 128;
    if (tid < kQ + 2 * kR) asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
  }

  // ---- shared memory.  Keys and values lie as the copies bring them: on the tensor path in pieces of [half][32 rows][128 B]
  // with the 128-byte swizzle (16-byte segment c of row r at c ^ (r & 7)), else rows one after another.
  extern __shared__ __align__(1024) unsigned char dsm[];
  const int cap = a.row_cap;
  uint4* sK = reinterpret_cast<uint4*>(dsm);                              // [cap][LPR]
  uint4* sV = sK + (size_t)cap * LPR;                                     // [cap][LPR]
  float* red = reinterpret_cast<float*>(sV + (size_t)cap * LPR);          // [warps][G][D] the warps' outputs
  float* part = red + kSplitWarps * G * D;                                // [C][G * D / C] partial outputs of this rank's share
  float* pl = part + G * D;                                               // [G][cap] logits, then 2^{x - the warp's maximum}
  float* s_rn = pl + (size_t)G * cap;                                     // [cap] 1/|k|
  int* s_ps = reinterpret_cast<int*>(s_rn + cap);                         // [cap] positions
  auto seg = [](int row, int c) -> int {                                  // where segment c of a row is, in uint4
    if (kTensor) return ((row / kSplitPiece * NH + (c >> 3)) * kSplitPiece + row % kSplitPiece) * 8 + ((c & 7) ^ (row & 7));
    return row * LPR + c;
  };
  __shared__ SplitExchange<G> xch;
  __shared__ unsigned long long s_k[kSplitPieces], s_v[kSplitPieces];
  __shared__ volatile int s_timeout;                                      // 1: nothing may be done; 2: a wait of this CTA ran out
  __shared__ float s_fac[kSplitWarps][G], s_new_rn;

  if (tid == 0) {
    for (int i = 0; i < kSplitPieces; ++i) { mbar_init(&s_k[i], 1); mbar_init(&s_v[i], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  // barrier 0: every CTA of the cluster has started before anything is written into its shared memory
  cluster_arrive();
  if (!a.early) {
    // the grids ahead may still write the slice (the end of the prompt stage): its next step, which looks at the step
    // counter alone, must not start before they are done either
    wait_for_prior_grid();
    start_dependents();
  }
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
  const int new_li = n_old >= r0 && n_old < r0 + cnt ? n_old - r0 : -1;   // local row of the new token, the last of the slice
  const int old_cnt = new_li >= 0 ? cnt - 1 : cnt;                        // cache rows
  if (tid == 0 && s_timeout == 0) {
    if (chunk > cap) { report_error(a.status, D2O_ERR_STATE, 0xDEC30000u | (uint32_t)(sl & 0xffff)); s_timeout = 1; }
    if (!D2O_GUARD(S >= 1 && n_old >= 0 && n_old <= S && row0 >= 0 && row0 + slice_stride(S) <= a.pool_rows, a.status, 0xC4EC0010u))
      s_timeout = 1;
  }
  const bool run = __syncthreads_or(s_timeout != 0) == 0;                 // if not: nothing is loaded, the cluster leaves after barrier 1
  const int n_pc = run ? (cnt + kSplitPiece - 1) / kSplitPiece : 0;
  const int n_tiles = run ? (cnt + 15) / 16 : 0;

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
      const int np = max(0, min(old_cnt, a0 + kSplitPiece) - a0);
      unsigned long long* bar = is_v ? &s_v[i - n_pc] : &s_k[i];
      uint4* dst = (is_v ? sV : sK) + (size_t)a0 * LPR;
      if (kTensor) {
        // whole boxes: rows past the slice are masked (keys) or zeroed (values) by whoever reads the tile
        mbar_expect_tx(bar, np > 0 ? (uint32_t)(kSplitPiece * ROWB) : 0u);
        if (np > 0) {
          const CUtensorMap* map = is_v ? &map_v : &map_k;
#pragma unroll
          for (int hf = 0; hf < NH; ++hf) {
            void* to = reinterpret_cast<unsigned char*>(dst) + hf * kSplitPiece * 128;
            if (a.l2_hints) tma_load_2d_hint(to, map, hf * 64, (int)(row0 + r0 + a0), bar, drop);
            else tc::tma_load_2d(to, map, hf * 64, (int)(row0 + r0 + a0), bar);
          }
        }
      } else {
        mbar_expect_tx(bar, (uint32_t)(np * ROWB));
        if (np > 0) {
          const T* src = (is_v ? vpool : kpool) + (row0 + r0 + a0) * D;
          if (a.l2_hints) bulk_g2s_hint(dst, src, (uint32_t)(np * ROWB), bar, drop);
          else bulk_g2s(dst, src, (uint32_t)(np * ROWB), bar);
        }
      }
    }
  }
  // ---- per-row state, while the rows are on their way.  Lane l keeps rows l % 16 of the tiles of its warp (tiles
  // warp, warp + 8, ...), two tiles per register.
  auto row_of = [&](int r) { return (warp + kSplitWarps * (2 * r + (lane >> 4))) * 16 + (lane & 15); };
  float sc[R]; int ps[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int li = row_of(r);
    sc[r] = 0.f; ps[r] = t_pos;
    if (run && li < old_cnt) {
      sc[r] = a.score[row0 + r0 + li];
      ps[r] = a.pos[row0 + r0 + li];
      s_rn[li] = a.rnorm[row0 + r0 + li];
    }
    if (run && li < cnt) s_ps[li] = ps[r];
  }
  // Dot products of the 16 rows of tile t with the vectors in `vf` / `vb`: put(g, row, value), each value by one lane.
  auto dots = [&](int t, auto& vf, auto& vb, auto n_vec, auto put) {
    constexpr int NV = decltype(n_vec)::value;
    if constexpr (kTensor) {
      float acc[4];
      tile_dots<T, D, kSplitPiece>(reinterpret_cast<const unsigned char*>(sK + (size_t)(t >> 1) * kSplitPiece * LPR), t & 1, vb, acc);
      if (2 * tig < NV) { put(2 * tig, t * 16 + gid, acc[0]); put(2 * tig, t * 16 + gid + 8, acc[2]); }
      if (2 * tig + 1 < NV) { put(2 * tig + 1, t * 16 + gid, acc[1]); put(2 * tig + 1, t * 16 + gid + 8, acc[3]); }
    } else {
#pragma unroll
      for (int bt = 0; bt < 4 / WG; ++bt) {
        float dot[NV][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int row = t * 16 + (bt * 4 + u) * WG + wg;
          float f[EPV];
          Elem<T>::unpack(row < cnt ? sK[seg(row, lig)] : make_uint4(0, 0, 0, 0), f);
#pragma unroll
          for (int g = 0; g < NV; ++g) dot[g][u] = dot_pairs<EPV>(vf[g], f);
        }
#pragma unroll
        for (int g = 0; g < NV; ++g) {
          const float x = reduce4<LPR>(dot[g][0], dot[g][1], dot[g][2], dot[g][3], lig);
          if (lig % QL == 0) put(g, t * 16 + (bt * 4 + lig / QL) * WG + wg, x);
        }
      }
    }
  };

  // the warp's extremum, for every rank
  auto push_key = [&](unsigned long long key, int li, bool lowest, bool victim) {
    const unsigned long long w = lowest ? warp_min_u64(key) : warp_max_u64(key);
    const int src = __ffs(__ballot_sync(0xffffffffu, key == w)) - 1;
    const int wli = __shfl_sync(0xffffffffu, li, src);
    if (lane < C) {
      SplitExchange<G>* to = cluster.map_shared_rank(&xch, lane);
      const int at = rank * kSplitWarps + warp;
      (victim ? to->vkey : to->nkey)[at] = w;
      (victim ? to->vli : to->nli)[at] = wli;
    }
  };
  const int entries = C * kSplitWarps;
  cluster_wait();                                                         // barrier 0
  // ---- the guess of the victim
  unsigned long long best = ~0ull; int best_li = -1;
  if (run && evict) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (row_of(r) < old_cnt && ps[r] >= Tn && ps[r] <= t_pos - M) {      // lowest score, ties -> latest position
        const unsigned long long key = ((unsigned long long)float_ord(sc[r]) << 32) | (uint32_t)(0x7fffffff - ps[r]);
        if (key < best) { best = key; best_li = r0 + row_of(r); }
      }
    }
  }
  __syncwarp();
  push_key(best, best_li, true, true);
  cluster_arrive();                                                       // barrier G
  cluster_wait();
  int cand_li = -1;                                                       // -1: no row of the cache may be evicted
  float cand_rn = 0.f;
  float cf[1][EPV];
  uint4 cb[D / 32];
  uint4 kvic = make_uint4(0, 0, 0, 0), vvic = make_uint4(0, 0, 0, 0);     // the victim's rows: warp 0 and the new token's warp
  const bool own_new = new_li >= 0 && ((new_li >> 4) % kSplitWarps) == warp;  // this warp's tile holds the new token
  (void)keys_extreme<true>(xch.vkey, xch.vli, entries, &cand_li);
  if (!run || !evict || !D2O_GUARD(cand_li >= -1 && cand_li < n_old, a.status, 0xC4EC0013u)) cand_li = -1;
  best = 0ull; best_li = -1;
  // cosines of this warp's rows (below `rows`) with the vector in cf / cb
  auto cosines = [&](int vic, float vic_rn, int rows) {
    for (int t = warp; t < n_tiles; t += kSplitWarps) {
      stage_wait(&s_k[t >> 1], 0u, &s_timeout, a.wait_ns);
      __syncwarp();
      dots(t, cf, cb, cuda::std::integral_constant<int, 1>(), [&](int, int row, float x) {
        if (row < rows && r0 + row != vic) {                              // max similarity, ties -> earliest position
          const unsigned long long key = ((unsigned long long)sim_ord(x * vic_rn * s_rn[row]) << 32) | (uint32_t)(0x7fffffff - s_ps[row]);
          if (key > best) { best = key; best_li = r0 + row; }
        }
      });
    }
    __syncwarp();
  };
  if (cand_li >= 0) {
    const uint4* ck = reinterpret_cast<const uint4*>(kpool + (row0 + cand_li) * D);
    cand_rn = a.rnorm[row0 + cand_li];
    if (lane < LPR && (warp == 0 || own_new)) {
      kvic = ck[lane];
      vvic = *reinterpret_cast<const uint4*>(vpool + (row0 + cand_li) * D + lane * EPV);
    }
    if constexpr (kTensor) {
#pragma unroll
      for (int j = 0; j < D / 32; ++j) cb[j] = gid == 0 ? ck[(j >> 1) * 8 + 2 * tig + (j & 1)] : make_uint4(0, 0, 0, 0);
    } else {
      Elem<T>::unpack(ck[lig], cf[0]);
    }
    cosines(cand_li, cand_rn, old_cnt);
  }
  push_key(best, best_li, false, false);
  // ---- from here on the inputs: the grid ahead on the stream must be done (unless the call promised them complete)
  if (a.early && !a.chained) asm volatile("griddepcontrol.wait;" ::: "memory");
  // A wait of the grids ahead that ran out while this one waited for them: looked at again below, beside the key pass.  (Other
  // anomalies concern one slice and may be those of another cluster of this launch: its own token is dropped, no other.)
  const uint32_t word = a.early && !a.chained && tid == 0 ? *reinterpret_cast<volatile uint32_t*>(a.status) : 0u;
  if (a.pub_count > 0 && warp == kSplitWarps - 1 && blockIdx.x == gridDim.x - 1) {
    // the slices of the call before: its grid is done
    for (int i = lane; i < a.pub_count; i += 32)
      asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.steps_done + a.pub_first + i), "r"(a.pub_step) : "memory");
  }
  const float qscale = (D == 64 ? 0.125f : 0.08838834764831845f) * kLog2e;   // log2(e)/sqrt(d)
  float qf[kTensor ? 1 : G][EPV];
  uint4 qb[D / 32];                                                       // tensor path: this lane's pieces of query gid
  if constexpr (kTensor) {
#pragma unroll
    for (int j = 0; j < D / 32; ++j)
      qb[j] = gid < G ? ld_global_v4(q_in + ((size_t)sl * G + gid) * D + ((j >> 1) * 8 + 2 * tig + (j & 1)) * 8)
                      : make_uint4(0, 0, 0, 0);
  } else {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      Elem<T>::unpack(ld_global_v4(q_in + ((size_t)sl * G + g) * D + lig * EPV), qf[g]);
#pragma unroll
      for (int i = 0; i < EPV; ++i) qf[g][i] *= qscale;
    }
  }
  uint4 knew = make_uint4(0, 0, 0, 0), vnew = make_uint4(0, 0, 0, 0);
  if ((warp == 0 || own_new) && lane < LPR) { knew = ld_global_v4(k_new + lane * EPV); vnew = ld_global_v4(v_new + lane * EPV); }

  // ---- pass K: logits of the warp's tiles, their maximum and sum -> barrier 1
  auto key_tile = [&](int t) {                                            // tile t is there, the new token's row included
    stage_wait(&s_k[t >> 1], 0u, &s_timeout, a.wait_ns);
    __syncwarp();
    if (own_new && t == new_li >> 4) {
      if (lane < LPR) sK[seg(new_li, lane)] = knew;
      __syncwarp();
    }
  };
  const int my_entry = rank * kSplitWarps + warp;
  if constexpr (kTensor) {
    // a lane's accumulators are rows gid, gid + 8 against heads 2 tig, 2 tig + 1: the row sums are three shuffles
    constexpr int TW = kSplitMaxRows / 16 / kSplitWarps;                  // tiles per warp
    float acc[TW][4], m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
#pragma unroll
    for (int i = 0; i < TW; ++i) {
      const int t = warp + i * kSplitWarps;
      if (t >= n_tiles) break;
      key_tile(t);
      tile_dots<T, D, kSplitPiece>(reinterpret_cast<const unsigned char*>(sK + (size_t)(t >> 1) * kSplitPiece * LPR), t & 1, qb, acc[i]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j] = t * 16 + gid + (j >> 1) * 8 < cnt ? acc[i][j] * qscale : -INFINITY;
        if (j & 1) m1 = fmaxf(m1, acc[i][j]); else m0 = fmaxf(m0, acc[i][j]);
      }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
      m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
    // a warp whose logits are all -inf: weights 0, as against the slice's maximum
    const float b0 = m0 > -INFINITY ? m0 : 0.f, b1 = m1 > -INFINITY ? m1 : 0.f;
#pragma unroll
    for (int i = 0; i < TW; ++i) {
      const int t = warp + i * kSplitWarps;
      if (t >= n_tiles) break;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = t * 16 + gid + (j >> 1) * 8 < cnt ? exp2f(acc[i][j] - ((j & 1) ? b1 : b0)) : 0.f;
        if (j & 1) l1 += p; else l0 += p;
        if (2 * tig + (j & 1) < G) pl[(size_t)(2 * tig + (j & 1)) * cap + t * 16 + gid + (j >> 1) * 8] = p;
      }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      l0 += __shfl_xor_sync(0xffffffffu, l0, o);
      l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    }
    if (2 * tig < G)
      for (int to_rank = gid; to_rank < C; to_rank += 8) {
        SplitExchange<G>* to = cluster.map_shared_rank(&xch, to_rank);
        to->m[my_entry][2 * tig] = m0; to->l[my_entry][2 * tig] = l0;
        if (2 * tig + 1 < G) { to->m[my_entry][2 * tig + 1] = m1; to->l[my_entry][2 * tig + 1] = l1; }
      }
    __syncwarp();
  } else {
    for (int t = warp; t < n_tiles; t += kSplitWarps) {
      key_tile(t);
      dots(t, qf, qb, cuda::std::integral_constant<int, G>(), [&](int g, int row, float x) { pl[(size_t)g * cap + row] = x; });
    }
    __syncwarp();
    float x[R][G], mw[G], lw[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      mw[g] = -INFINITY;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        x[r][g] = run && row_of(r) < cnt ? pl[(size_t)g * cap + row_of(r)] : -INFINITY;
        mw[g] = fmaxf(mw[g], x[r][g]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int g = 0; g < G; ++g) mw[g] = fmaxf(mw[g], __shfl_xor_sync(0xffffffffu, mw[g], o));
#pragma unroll
    for (int g = 0; g < G; ++g) {
      lw[g] = 0.f;
      const float base = mw[g] > -INFINITY ? mw[g] : 0.f;                 // all -inf: weights 0, as against the slice's maximum
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float p = run && row_of(r) < cnt ? exp2f(x[r][g] - base) : 0.f;
        if (run && (row_of(r) >> 4) < n_tiles) pl[(size_t)g * cap + row_of(r)] = p;       // 0 past the last row
        lw[g] += p;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int g = 0; g < G; ++g) lw[g] += __shfl_xor_sync(0xffffffffu, lw[g], o);
    if (lane < C) {
      SplitExchange<G>* to = cluster.map_shared_rank(&xch, lane);
#pragma unroll
      for (int g = 0; g < G; ++g) { to->m[my_entry][g] = mw[g]; to->l[my_entry][g] = lw[g]; }
    }
  }
  if (word == D2O_ERR_TIMEOUT && s_timeout == 0) s_timeout = 1;
  __syncwarp();
  if (lane < C) cluster.map_shared_rank(&xch, lane)->bad1[my_entry] = s_timeout;
  cluster_arrive();                                                       // barrier 1
  if (warp == 0 || own_new) {
    // 1/|k| of the new token, its cosine with the guessed victim
    float f[EPV], g[EPV];
    Elem<T>::unpack(knew, f);
    Elem<T>::unpack(kvic, g);
    float ss = 0.f, x = 0.f;
#pragma unroll
    for (int i = 0; i < EPV; ++i) { ss = fmaf(f[i], f[i], ss); x = fmaf(f[i], g[i], x); }
    ss = warp_sum(ss);
    x = warp_sum(x);
    const float rn = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
    if (lane == 0 && warp == 0) s_new_rn = rn;
    if (own_new) {
      if (lane == 0 && run) s_rn[new_li] = rn;
      const unsigned long long key = ((unsigned long long)sim_ord(x * cand_rn * rn) << 32) | (uint32_t)(0x7fffffff - t_pos);
      if (lane < C) cluster.map_shared_rank(&xch, lane)->new_nkey = key;
    }
  }

  // ---- pass V: un-normalised outputs of the warp's rows
  if constexpr (kTensor) {
    // out^T (d x heads) = V^T (d x rows) P (rows x heads); the weights in two 16-bit terms
    float acc[NH][4][4];
#pragma unroll
    for (int i = 0; i < NH * 16; ++i) acc[i / 16][(i >> 2) & 3][i & 3] = 0.f;
    const int krow = (lane & 7) + ((lane >> 4) & 1) * 8;
    const int gw = gid < G ? gid : 0;                                     // lanes past the heads: their columns are never used
    const uint32_t v_u32 = smem_u32(sV);
    for (int t = warp; t < n_tiles; t += kSplitWarps) {
      stage_wait(&s_v[t >> 1], 0u, &s_timeout, a.wait_ns);
      __syncwarp();
      if (t * 16 + 16 > old_cnt) {
        // the new token's row; rows past the slice (its padding, the next slice, or nothing) count as zero
        for (int i = lane; i < 16 * LPR; i += 32) {
          const int row = t * 16 + i / LPR;
          if (row >= cnt) sV[seg(row, i % LPR)] = make_uint4(0, 0, 0, 0);
        }
        if (own_new && t == new_li >> 4 && lane < LPR) sV[seg(new_li, lane)] = vnew;
        __syncwarp();
      }
      const float2 w0 = *reinterpret_cast<const float2*>(pl + (size_t)gw * cap + t * 16 + 2 * tig);
      const float2 w1 = *reinterpret_cast<const float2*>(pl + (size_t)gw * cap + t * 16 + 2 * tig + 8);
      uint32_t bh0, bl0, bh1, bl1;
      split_pair<T>(w0.x, w0.y, bh0, bl0);
      split_pair<T>(w1.x, w1.y, bh1, bl1);
#pragma unroll
      for (int hf = 0; hf < NH; ++hf) {
        const uint32_t tile = v_u32 + (uint32_t)((((t >> 1) * NH + hf) * kSplitPiece + (t & 1) * 16) * 128);
        uint32_t fa[4][4];
#pragma unroll
        for (int mt = 0; mt < 4; ++mt)
          ldmatrix_x4_trans(tile + (uint32_t)(krow * 128 + (((mt * 2 + ((lane >> 3) & 1)) ^ (lane & 7)) << 4)),
                            fa[mt][0], fa[mt][1], fa[mt][2], fa[mt][3]);
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) mma_16x8x16<T>(acc[hf][mt], fa[mt][0], fa[mt][1], fa[mt][2], fa[mt][3], bh0, bh1);
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) mma_16x8x16<T>(acc[hf][mt], fa[mt][0], fa[mt][1], fa[mt][2], fa[mt][3], bl0, bl1);
      }
    }
#pragma unroll
    for (int hf = 0; hf < NH; ++hf)
#pragma unroll
      for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int g = 2 * tig + (i & 1);
          if (g < G) red[(warp * G + g) * D + hf * 64 + mt * 16 + gid + (i >> 1) * 8] = acc[hf][mt][i];
        }
  } else {
    float acc[G][EPV];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int i = 0; i < EPV; ++i) acc[g][i] = 0.f;
    for (int t = warp; t < n_tiles; t += kSplitWarps) {
      stage_wait(&s_v[t >> 1], 0u, &s_timeout, a.wait_ns);
      __syncwarp();
      if (own_new && t == new_li >> 4) {
        if (lane < LPR) sV[seg(new_li, lane)] = vnew;
        __syncwarp();
      }
#pragma unroll 4
      for (int u = 0; u < 16 / WG; ++u) {
        const int row = t * 16 + u * WG + wg;
        if (row < cnt) {
          float f[EPV];
          Elem<T>::unpack(sV[seg(row, lig)], f);
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float p = pl[(size_t)g * cap + row];
#pragma unroll
            for (int i = 0; i < EPV; i += 2) {
              const float2 s = ffma2(make_float2(p, p), make_float2(f[i], f[i + 1]), make_float2(acc[g][i], acc[g][i + 1]));
              acc[g][i] = s.x; acc[g][i + 1] = s.y;
            }
          }
        }
      }
      __syncwarp();
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
        for (int i = 0; i < EPV; ++i) red[(warp * G + g) * D + lane * EPV + i] = acc[g][i];
    }
  }

  // A chained grid must not be complete before its predecessor (whatever the stream runs next is ordered behind this
  // grid only): one CTA that stays until then is enough.
  auto hold = [&]() { if (a.chained && blockIdx.x == gridDim.x - 1) asm volatile("griddepcontrol.wait;" ::: "memory"); };
  // A CTA must not end while copies are on their way into its shared memory (a cluster that gives up sees its own land), nor
  // while a peer that has arrived at the barrier before may still store into it: one more barrier.  The flags are the same in
  // every CTA, so all of them come here or none.
  auto leave = [&](uint32_t detail) {
    cluster_arrive();
    cluster_wait();
    if (tid == 0) {
      if (s_timeout == 2) report_error(a.status, D2O_ERR_TIMEOUT, detail | (uint32_t)(sl & 0xffff));
      for (int i = 0; i < issued; ++i)
        if (!landed_wait(i < n_pc ? &s_k[i] : &s_v[i - n_pc], 0u, a.wait_ns)) break;
    }
    hold();
  };
  auto any_bad = [&](const int* flags) {
    int f = 0;
    for (int i = lane; i < entries; i += 32) f |= flags[i];
    return __any_sync(0xffffffffu, f != 0) != 0;
  };
  cluster_wait();                                                         // barrier 1
  // a CTA found an anomaly, or its keys did not arrive: the whole cluster leaves, nothing has been written
  if (any_bad(xch.bad1)) { leave(0xDEC10000u); return; }
  if (warp < G) {
    float m[kSplitEntries / 32], mx = -INFINITY, l = 0.f;
#pragma unroll
    for (int i = 0; i < kSplitEntries / 32; ++i) {
      m[i] = i * 32 + lane < entries ? xch.m[i * 32 + lane][warp] : -INFINITY;
      mx = fmaxf(mx, m[i]);
    }
    mx = warp_max(mx);
#pragma unroll
    for (int i = 0; i < kSplitEntries / 32; ++i)
      if (i * 32 + lane < entries) l += xch.l[i * 32 + lane][warp] * exp2f(m[i] - mx);
    l = warp_sum(l);
    // turns a warp's 2^{x - its maximum} into probabilities; 0 for a warp without rows
    if (lane < kSplitWarps) s_fac[lane][warp] = exp2f(xch.m[rank * kSplitWarps + lane][warp] - mx) / l;
  }
  __syncthreads();

  // ---- accumulated attention (Eq. 6 case 2), the warp's victim (Eq. 7-8) -> barrier 2
  best = ~0ull; best_li = -1;
  float fac[G];
#pragma unroll
  for (int g = 0; g < G; ++g) fac[g] = s_fac[warp][g];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int li = row_of(r);
    if (li < cnt) {
      float p = 0.f;
#pragma unroll
      for (int g = 0; g < G; ++g) p = fmaf(pl[(size_t)g * cap + li], fac[g], p);
      sc[r] += p;
      if (ps[r] >= Tn && ps[r] <= t_pos - M) {                            // lowest score, ties -> latest position
        const unsigned long long key = ((unsigned long long)float_ord(sc[r]) << 32) | (uint32_t)(0x7fffffff - ps[r]);
        if (key < best) { best = key; best_li = r0 + li; }
      }
    }
  }
  __syncwarp();
  push_key(best, best_li, true, true);
  if (lane < C) cluster.map_shared_rank(&xch, lane)->bad2[my_entry] = s_timeout;
  if (own_new) {
    const int tl = (new_li >> 4) / kSplitWarps;                           // which of the warp's tiles
    const float ns = __shfl_sync(0xffffffffu, (tl >> 1) == 0 ? sc[0] : sc[R - 1], (tl & 1) * 16 + (new_li & 15));
    if (lane < C) cluster.map_shared_rank(&xch, lane)->new_score = ns;
  }
  // scaled outputs, each to the rank that finishes it: read behind the cluster's last barrier
  const int share = G * D / C;                                            // outputs a rank finishes
  auto send_outputs = [&]() {
#pragma unroll
    for (int i = 0; i < OUT; ++i) {
      const int at = tid + i * kSplitThreads;
      if (at < G * D) {
        float o = 0.f;
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) o = fmaf(red[w * G * D + at], s_fac[w][at / D], o);
        cluster.map_shared_rank(part, at / share)[rank * share + at % share] = o;
      }
    }
  };
  if (!kPublish) send_outputs();
  cluster_arrive();                                                       // barrier 2
  if (kPublish) send_outputs();                                           // beside the barrier: there is another one
  cluster_wait();
  if (any_bad(xch.bad2)) { leave(0xDEC10000u); return; }                  // the values did not arrive: nothing written yet

  // ---- the victim and its neighbour
  int vic_li = -1, nn_li = -1;
  unsigned long long nbest = 0ull;
  const unsigned long long vbest = keys_extreme<true>(xch.vkey, xch.vli, entries, &vic_li);
  const bool none = evict && vbest == ~0ull;                              // S_l < T + M: nothing may be evicted
  // ---- this rank's share of the outputs (Eq. 3)
  auto write_outputs = [&](int first) {
    if (none) return;
    for (int i = first; i < share; i += kSplitThreads) {
      float t = 0.f;
      for (int r = 0; r < C; ++r) t += part[r * share + i];
      out[(size_t)sl * G * D + rank * share + i] = Elem<T>::from_float(t);
    }
  };
  if (!kPublish) write_outputs(kSplitThreads - 1 - tid);                  // the first warp goes on to the merge
  if (!evict) vic_li = -1;
  if (evict && !none) {
    if (!D2O_GUARD(vic_li >= 0 && vic_li <= n_old, a.status, 0xC4EC0011u)) vic_li = n_old;
    if (vic_li != cand_li) {
      // the guess was wrong: the cosines once more
      if (rank == 0 && tid == 0) atomicAdd(&a.counters[kCntGuessMisses], 1ull);
      const int vr = vic_li / chunk, vl = vic_li % chunk;                 // who holds the victim
      const uint4* rK = cluster.map_shared_rank(sK, vr);
      if (lane < LPR && warp == 0) { kvic = rK[seg(vl, lane)]; vvic = cluster.map_shared_rank(sV, vr)[seg(vl, lane)]; }
      if constexpr (kTensor) {
#pragma unroll
        for (int j = 0; j < D / 32; ++j)
          cb[j] = gid == 0 ? rK[seg(vl, (j >> 1) * 8 + 2 * tig + (j & 1))] : make_uint4(0, 0, 0, 0);
      } else {
        Elem<T>::unpack(rK[seg(vl, lig)], cf[0]);
      }
      best = 0ull; best_li = -1;
      cosines(vic_li, cluster.map_shared_rank(s_rn, vr)[vl], cnt);
      push_key(best, best_li, false, false);
      cluster_arrive();
      cluster_wait();
    }
    nbest = keys_extreme<false>(xch.nkey, xch.nli, entries, &nn_li);
    if (vic_li == cand_li && xch.new_nkey > nbest) { nbest = xch.new_nkey; nn_li = n_old; }
  }
  // ---- scores of this rank's rows; the new token's goes with its row, wherever that ends up
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int li = row_of(r);
    if ((li < old_cnt && r0 + li != vic_li) || (li == new_li && !evict)) a.score[row0 + r0 + li] = sc[r];
  }
  if (kPublish) cluster_arrive();                                         // barrier 3
  // ---- threshold, merge or discard (Eq. 10-12), the new token's row: by the CTA that holds the neighbour (or, while
  // the cache still fills, the new token)
  const bool writer = warp == 0 && !none && (evict ? max(nn_li, 0) : n_old) / chunk == rank;
  if (writer) {
    if (!evict) {
      if (lane < LPR) {
        *reinterpret_cast<uint4*>(kpool + (row0 + n_old) * D + lane * EPV) = sK[seg(new_li, lane)];
        *reinterpret_cast<uint4*>(vpool + (row0 + n_old) * D + lane * EPV) = sV[seg(new_li, lane)];
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
        uint4 kslot = knew, vslot = vnew;
        float rn_slot = s_new_rn;
        if (merge) {
          float fk[EPV], fv[EPV], kv[EPV], vv[EPV];
          Elem<T>::unpack(sK[seg(nn_li - r0, lane)], fk);
          Elem<T>::unpack(sV[seg(nn_li - r0, lane)], fv);
          Elem<T>::unpack(kvic, kv);
          Elem<T>::unpack(vvic, vv);
  #pragma unroll
          for (int i = 0; i < EPV; ++i) { fk[i] = w_c * fk[i] + w_e * kv[i]; fv[i] = w_c * fv[i] + w_e * vv[i]; }
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
  }
  if (none && rank == 0 && tid == 0)                                      // drop the new token, keep the cache as it is
    report_error(a.status, D2O_ERR_STATE, 0xDEC00000u | (uint32_t)(sl & 0xfffff));
  hold();
  if (kPublish) cluster_wait();                                           // barrier 3
  if (writer) {
    asm volatile("fence.proxy.async.global;" ::: "memory");
    __syncwarp();
    // every other CTA's stores to the state were ordered before barrier 3, this warp's before the release
    if (kPublish && lane == 0)
      asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.steps_done + sidx), "r"(a.step + 1) : "memory");
  }
  if (kPublish) write_outputs(tid);
}

// ------------------------------------------------------------------------------------ launch
// rows per CTA the shared arrays are sized for
static int split_rows(int max_rows, int C) { return ((max_rows + C - 1) / C + kSplitPiece - 1) / kSplitPiece * kSplitPiece; }

// shared memory of a CTA with room for `rows` rows
static size_t split_smem(int rows, int G, int D, int esz) {
  return (size_t)rows * (2 * D * esz + G * 4 + 8) + (size_t)(kSplitWarps + 1) * G * D * 4;
}

// CTAs per slice, or 0 when one CTA per slice (decode_kernel) is the better choice or the rows do not fit.
//
// What counts here is how quickly one slice is done, and how many rounds of resident clusters the call takes: about 11 us
// for one and less for those behind it, plus the time for the longest slice's rows, which the one-CTA kernel pays in full (us
// per call, this kernel / decode_kernel: 8 fp16 slices of 1640 rows, one head, 13.8 / 37, 32 of 820 rows 13.8 / 25, 72 of 160
// bf16 rows, four heads, 12.7 / 14.5).  One round of clusters is the better choice, also for short slices: repeated steps on
// 24 slices of 40 rows and one head take 11.9 / 10.4, but in a model that calls layer by layer the clusters of one call start
// beside those of the call before (56 fp32 slices of 172 rows 8.7 / 9.9).  Rows are long where one layer holds most of the
// budget, and then shared memory admits one CTA per SM: 144 slices of which the longest has 1460 rows are four rounds of four
// CTAs or eight of eight, 99 / 27; 100 slices of 320 rows are two rounds, 21.8 / 16.5; but 64 slices of up to 1345 rows in two
// rounds 21.5 / 26.  Larger clusters shorten the passes, but every barrier and every exchange takes longer: two CTAs, four for
// longer slices while there is an SM for each (32 slices of 800 rows 12.9 us with four, 14.2 with two, 17 with eight), more
// only where the rows do not fit otherwise, two where four would take a second round (36 slices of 640 rows 15.6 instead of
// 19.9).  From 20 MB of keys and values on, the passes count more than the chain of steps (96 of 800 rows (39 MB) 36 / 31).
int decode_split_cluster(const d2o_ctx* c, int n_slices, int max_rows, double total_rows) {
  const d2o_config& g = c->cfg;
  const int G = c->group;
  if (total_rows * 2 * g.d_head * c->elem_size > 20e6 || n_slices > c->n_sms) return 0;
  const size_t fixed = (size_t)G * 1024 + 5 * 1024;                       // static shared arrays
  // rounds of resident clusters; 0: the rows do not fit
  auto rounds = [&](int i) {
    const int rows = split_rows(max_rows, 2 << i);
    const size_t smem = split_smem(rows, G, g.d_head, c->elem_size) + fixed + 1024;
    if (c->split_clusters[i] == 0 || rows > kSplitMaxRows || smem > 227 * 1024) return 0;
    const int resident = c->split_clusters[i] * (G <= 4 && 2 * smem <= 228 * 1024 ? 2 : 1);
    return (n_slices + resident - 1) / resident;
  };
  int i = max_rows > 320 && 4 * n_slices <= c->n_sms ? 1 : 0, n = 0;
  while (i < kSplitSizes && (n = rounds(i)) == 0) ++i;
  if (n == 0) return 0;
  if (n > 1 && i == 1 && rounds(0) == 1) { i = 0; n = 1; }
  if (n == 1) return 2 << i;
  const double row_us = 3.1e-5 * 2 * g.d_head * c->elem_size * max_rows;  // the longest slice in one CTA
  const double one_us = (G == 1 ? 10.0 : G <= 4 ? 12.3 : 16.0) + row_us;
  const double split_us = 11.5 + 9.5 * (n - 1) + row_us / (2 << i);
  return split_us < one_us ? 2 << i : 0;
}

// Clusters of 2, 4, 8 and 16 CTAs that the current device holds at one CTA per SM.
void decode_split_places(int* clusters) {
  auto kern = decode_split_kernel<float, 128, 8, true>;
  const size_t smem = 150 * 1024;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  for (int i = 0; i < kSplitSizes; ++i) {
    const int C = 2 << i;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C); cfg.blockDim = dim3(kSplitThreads); cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    clusters[i] = 0;
    if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess || cudaOccupancyMaxActiveClusters(&clusters[i], kern, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      clusters[i] = 0;
    }
  }
}

template <typename T, int D, int G>
static cudaError_t launch_one(const DecodeArgs& a, const CUtensorMap* maps, int C, int n_slices, const void* q, const void* k,
                              const void* v, void* out, void* kpool, void* vpool, cudaStream_t st) {
  const size_t smem = split_smem(a.row_cap, G, D, (int)sizeof(T));
  auto kern = a.publish ? decode_split_kernel<T, D, G, true> : decode_split_kernel<T, D, G, false>;
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
  return cudaLaunchKernelEx(&cfg, kern, a, maps[0], maps[1], (const T*)q, (const T*)k, (const T*)v, (T*)out, (T*)kpool, (T*)vpool);
}

template <typename T, int D>
static cudaError_t launch_g(int G, const DecodeArgs& a, const CUtensorMap* maps, int C, int n_slices, const void* q,
                            const void* k, const void* v, void* out, void* kpool, void* vpool, cudaStream_t st) {
  switch (G) {
    case 1: return launch_one<T, D, 1>(a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
    case 2: return launch_one<T, D, 2>(a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
    case 4: return launch_one<T, D, 4>(a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
    default: return launch_one<T, D, 8>(a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
  }
}

// One step of `n_slices` slices (in index order) with `C` CTAs each.  `a.chained`, `a.publish`: see launch_decode;
// `a.early`: see DecodeArgs.
cudaError_t launch_decode_split(const d2o_ctx* c, DecodeArgs a, int C, int n_slices, int max_rows, const void* q,
                                const void* k, const void* v, void* out, void* kpool, void* vpool, cudaStream_t st) {
  const d2o_config& g = c->cfg;
  a.row_cap = split_rows(max_rows, C);
  CUtensorMap maps[2];
  memset(maps, 0, sizeof(maps));
  if (tensor_path(c->elem_size, c->group) && (!encode_rows_2d(&maps[0], g.dtype, kpool, (uint64_t)c->pool_rows, g.d_head, kSplitPiece) ||
                            !encode_rows_2d(&maps[1], g.dtype, vpool, (uint64_t)c->pool_rows, g.d_head, kSplitPiece)))
    return cudaErrorNotSupported;
  if (g.dtype == D2O_F32)
    return g.d_head == 64 ? launch_g<float, 64>(c->group, a, maps, C, n_slices, q, k, v, out, kpool, vpool, st)
                          : launch_g<float, 128>(c->group, a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
  if (g.dtype == D2O_F16)
    return g.d_head == 64 ? launch_g<__half, 64>(c->group, a, maps, C, n_slices, q, k, v, out, kpool, vpool, st)
                          : launch_g<__half, 128>(c->group, a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
  return g.d_head == 64 ? launch_g<__nv_bfloat16, 64>(c->group, a, maps, C, n_slices, q, k, v, out, kpool, vpool, st)
                        : launch_g<__nv_bfloat16, 128>(c->group, a, maps, C, n_slices, q, k, v, out, kpool, vpool, st);
}

}  // namespace d2o
