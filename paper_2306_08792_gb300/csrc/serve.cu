// Re-ranking against a resident gallery (serving form of GCR, Sec. IV-F2: the gallery's graphs
// are computed and stored in advance).
//
// The gallery state holds the layers G_0..G_T of offline GCR on the gallery alone and, per
// layer t < T, the degrees of that layer's gallery graph. A batch of queries then runs, for
// t = 1..T, the certified kNN search against G_{t-1} (column-split streaming pools, merged),
// and one row of the operator per query with the gallery frozen and no query-query edges:
//   symmetric (Eq. 7): y = x_q / D_q + sum_j (w_qj / 2) g_j / sqrt(D_q D_j),
//                      D_q = (1 + sum_j w_qj + 1) / 2
//   asymmetric (Eq. 6): y = x_q / sqrt(r_q) + sum_j w_qj g_j / sqrt(r_q Dc_j), r_q = 1 + sum w
// x_q <- normalise(y); finally the certified top-K of the gallery on G_T. Every step is per
// query row, so a query's result does not depend on the other queries of its batch.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "pool.cuh"

namespace gcr {
namespace {

// Merges the sorted list held by a warp (b, bi: KP entries, entry p*32 + lane) with the sorted
// KP-entry list at (lv, li) (shared or global memory), keeping the KP best. Chunks of a sorted
// list are sorted, so the merge stops at the first chunk whose best cannot enter.
template <int KP>
__device__ __forceinline__ void merge_list(float (&b)[KP / 32], int (&bi)[KP / 32], const float* lv, const int* li,
                                           int lane) {
  constexpr int P = KP / 32;
#pragma unroll
  for (int c = 0; c < P; ++c) {
    float a = lv[c * 32 + lane];
    int ai = li[c * 32 + lane];
    const float worst = __shfl_sync(GCR_FULL, b[P - 1], 31);
    const int worst_i = __shfl_sync(GCR_FULL, bi[P - 1], 31);
    const float best = __shfl_sync(GCR_FULL, a, 0);
    const int best_i = __shfl_sync(GCR_FULL, ai, 0);
    if (!better(best, best_i, worst, worst_i)) break;
    const float ar = __shfl_sync(GCR_FULL, a, 31 - lane);
    const int ari = __shfl_sync(GCR_FULL, ai, 31 - lane);
    if (better(ar, ari, b[P - 1], bi[P - 1])) { b[P - 1] = ar; bi[P - 1] = ari; }
#pragma unroll
    for (int stride = KP / 2; stride >= 32; stride >>= 1) {
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const int q2 = p ^ (stride >> 5);
        if (q2 > p && better(b[q2], bi[q2], b[p], bi[p])) {
          float tv = b[p]; b[p] = b[q2]; b[q2] = tv;
          int ti = bi[p]; bi[p] = bi[q2]; bi[q2] = ti;
        }
      }
    }
#pragma unroll
    for (int p = 0; p < P; ++p) warp_merge32_desc(b[p], bi[p], lane);
  }
}

// The pool of (kind, row) w = kind * na + row among [kinds][out_rows], the rows from row0 on.
__device__ __forceinline__ size_t out_row(long w, int na, int out_rows, int row0) {
  const long kind = w >= na ? 1 : 0;  // at most two graphs
  return (size_t)(kind * out_rows + row0 + (w - kind * na));
}

// Merge S sorted pools per (kind, row) into one: pools [S][kinds][na][KP] -> [kinds][out_rows][KP].
// One block of 8 warps per (kind, row): warp w merges splits w, w + 8, ..., then warp 0 merges
// the 8 partial lists (the strict order makes the result independent of the merge order).
template <int KP>
__global__ void __launch_bounds__(256) merge_splits_kernel(const float* __restrict__ pv, const int* __restrict__ pi,
                                                           int S, int kinds, int na, float* __restrict__ ov,
                                                           int* __restrict__ oi, int out_rows, int row0) {
  constexpr int P = KP / 32;
  __shared__ float sv[8][KP];
  __shared__ int si[8][KP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long w = blockIdx.x;  // (kind, row)
  float b[P];
  int bi[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const bool has = warp < S;
    b[p] = has ? pv[((size_t)warp * kinds * na + w) * KP + p * 32 + lane] : -CUDART_INF_F;
    bi[p] = has ? pi[((size_t)warp * kinds * na + w) * KP + p * 32 + lane] : -1;
  }
  for (int s = warp + 8; s < S; s += 8) {
    const size_t base = ((size_t)s * kinds * na + w) * KP;
    merge_list<KP>(b, bi, pv + base, pi + base, lane);
  }
#pragma unroll
  for (int p = 0; p < P; ++p) {
    sv[warp][p * 32 + lane] = b[p];
    si[warp][p * 32 + lane] = bi[p];
  }
  __syncthreads();
  if (warp != 0) return;
  for (int v = 1; v < 8 && v < S; ++v) merge_list<KP>(b, bi, sv[v], si[v], lane);
  const size_t out = out_row(w, na, out_rows, row0) * KP;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    ov[out + p * 32 + lane] = b[p];
    oi[out + p * 32 + lane] = bi[p];
  }
}

// Merges 32 entries (one per lane, any order) into the sorted list held by the warp.
template <int KP>
__device__ __forceinline__ void merge_chunk(float (&b)[KP / 32], int (&bi)[KP / 32], float a, int ai, int lane) {
  constexpr int P = KP / 32;
  warp_sort32_desc(a, ai, lane);
  const float ar = __shfl_sync(GCR_FULL, a, 31 - lane);
  const int ari = __shfl_sync(GCR_FULL, ai, 31 - lane);
  if (better(ar, ari, b[P - 1], bi[P - 1])) { b[P - 1] = ar; bi[P - 1] = ari; }
#pragma unroll
  for (int stride = KP / 2; stride >= 32; stride >>= 1) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const int q2 = p ^ (stride >> 5);
      if (q2 > p && better(b[q2], bi[q2], b[p], bi[p])) {
        float tv = b[p]; b[p] = b[q2]; b[q2] = tv;
        int ti = bi[p]; bi[p] = bi[q2]; bi[q2] = ti;
      }
    }
  }
#pragma unroll
  for (int p = 0; p < P; ++p) warp_merge32_desc(b[p], bi[p], lane);
}

// The selection buffers of a (kind, row)'s S splits sorted into its pool, a warp per row (few
// splits). The warp streams its entries (the next 32 in flight while 32 are tested): those that
// would enter its list so far are staged in shared memory and merged 32 at a time, so past the
// first few splits most entries cost one comparison. The strict order makes the result independent
// of the merge order.
template <int KP>
__global__ void __launch_bounds__(256) pool_finish_kernel(const float* __restrict__ pv, const int* __restrict__ pi,
                                                          const int* __restrict__ cnt, int S, long rows, int cap,
                                                          float* __restrict__ ov, int* __restrict__ oi, int part_rows,
                                                          int out_rows, int row0, Gate gate) {
  if (gate_shut(gate)) return;
  constexpr int P = KP / 32;
  __shared__ float stv[8][64];
  __shared__ int sti[8][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long w = (long)blockIdx.x * 8 + warp;  // (kind, row)
  if (w >= rows) return;
  float b[P];
  int bi[P];
#pragma unroll
  for (int p = 0; p < P; ++p) { b[p] = -CUDART_INF_F; bi[p] = -1; }
  float worst = -CUDART_INF_F;
  int worst_i = -1, staged = 0;
  auto merge_staged = [&](int take) {
    const float a = lane < take ? stv[warp][lane] : -CUDART_INF_F;
    const int ai = lane < take ? sti[warp][lane] : -1;
    const float rv = stv[warp][32 + lane];
    const int ri = sti[warp][32 + lane];
    __syncwarp();
    stv[warp][lane] = rv;
    sti[warp][lane] = ri;
    __syncwarp();
    staged -= take;
    merge_chunk<KP>(b, bi, a, ai, lane);
    worst = __shfl_sync(GCR_FULL, b[P - 1], 31);
    worst_i = __shfl_sync(GCR_FULL, bi[P - 1], 31);
  };
  auto test = [&](float a, int ai) {
    const bool in = ai >= 0 && (worst_i < 0 || better(a, ai, worst, worst_i));
    const unsigned m = __ballot_sync(GCR_FULL, in);
    if (!m) return;
    if (in) {
      const int at = staged + __popc(m & ((1u << lane) - 1u));
      stv[warp][at] = a;
      sti[warp][at] = ai;
    }
    staged += __popc(m);
    __syncwarp();
    if (staged >= 32) merge_staged(32);
  };
  float na = 0.f;  // the next chunk, in flight
  int ni = -1;
  for (int s0 = 0; s0 < S; s0 += 32) {  // 32 splits: a lane holds each count
    const int sl = s0 + lane;
    const int cl = sl < S ? min(max(cnt[(size_t)sl * rows + w], 0), cap) : 0;
    for (int l = 0; l < 32 && s0 + l < S; ++l) {
      const int c = __shfl_sync(GCR_FULL, cl, l);
      const size_t base = ((size_t)(s0 + l) * rows + w) * cap;
      for (int e0 = 0; e0 < c; e0 += 32) {
        const int e = e0 + lane;
        const float a = e < c ? pv[base + e] : 0.f;
        const int ai = e < c ? pi[base + e] : -1;
        test(na, ni);
        na = a;
        ni = ai;
      }
    }
  }
  test(na, ni);
  if (staged > 0) merge_staged(staged);
  const size_t out = out_row(w, part_rows, out_rows, row0) * KP;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    ov[out + p * 32 + lane] = b[p];
    oi[out + p * 32 + lane] = bi[p];
  }
}

// The same from many splits' buffers, a block per row: the entries as 64-bit keys (score's image,
// complement of the column: the strict order) in shared memory, narrowed to at most kSelKeep by
// histograms of 256 equal parts of the keys' range (usually two or three), and these ranked by
// counting. Merging sorted lists pairwise took about 110 shuffles per 32 entries and was bound by
// them: 512 rows, 128-entry pools of 38 splits 139 -> 23 us, one row of 152 splits 46 -> 15 us (32
// entries: 31 -> 14 and 20 -> 10).
// Splits are taken in groups that fit the buffer; the best KP so far stay at its front.
constexpr int kSelKeep = 256;
constexpr int kSelThreads = 512;

template <int KP>
__global__ void __launch_bounds__(kSelThreads) pool_select_kernel(const float* __restrict__ pv,
                                                                  const int* __restrict__ pi,
                                                                  const int* __restrict__ cnt, int S, long rows,
                                                                  int cap, int group, float* __restrict__ ov,
                                                                  int* __restrict__ oi, int part_rows, int out_rows,
                                                                  int row0, Gate gate) {
  static_assert(KP <= kSelKeep, "the kept entries hold the pool");
  if (gate_shut(gate)) return;
  extern __shared__ __align__(16) unsigned long long ent[];  // [KP + group * cap]
  __shared__ unsigned long long keep[kSelKeep], s_min, s_max;
  __shared__ int hist[256], part[kSelThreads], s_total, s_kept, s_bin, s_over;
  constexpr int NW = kSelThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long w = blockIdx.x;  // (kind, row)
  const size_t out = out_row(w, part_rows, out_rows, row0) * KP;
  int have = 0;
  for (int s0 = 0; s0 < S; s0 += group) {
    const int s1 = min(S, s0 + group);
    if (tid == 0) { s_total = have; s_kept = 0; s_min = ~0ull; s_max = 0ull; }
    __syncthreads();
    unsigned long long mn = ~0ull, mx = 0ull;
    for (int e = tid; e < have; e += kSelThreads) { mn = min(mn, ent[e]); mx = max(mx, ent[e]); }
    for (int sb = s0 + warp; sb < s1; sb += NW * 32) {  // up to 32 splits of the warp: a lane holds each count
      const int sl = sb + NW * lane;
      const int cl = sl < s1 ? min(max(cnt[(size_t)sl * rows + w], 0), cap) : 0;
      int inc = cl;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(GCR_FULL, inc, o);
        if (lane >= o) inc += y;
      }
      int at0 = 0;
      if (lane == 31) at0 = atomicAdd(&s_total, inc);
      at0 = __shfl_sync(GCR_FULL, at0, 31);
      for (int l = 0; l < 32 && sb + NW * l < s1; ++l) {
        const int c = __shfl_sync(GCR_FULL, cl, l), at = at0 + __shfl_sync(GCR_FULL, inc, l) - c;
        const size_t base = ((size_t)(sb + NW * l) * rows + w) * cap;
        for (int e = lane; e < c; e += 32) {
          const unsigned long long key = ((unsigned long long)float_to_ordered(pv[base + e] + 0.f) << 32) |
                                         (uint32_t)~pi[base + e];
          ent[at + e] = key;
          mn = min(mn, key);
          mx = max(mx, key);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn = min(mn, __shfl_xor_sync(GCR_FULL, mn, o));
      mx = max(mx, __shfl_xor_sync(GCR_FULL, mx, o));
    }
    if (lane == 0) { atomicMin(&s_min, mn); atomicMax(&s_max, mx); }
    __syncthreads();
    const int E = s_total;
    unsigned long long lo = s_min, hi = s_max;
    if (E > kSelKeep) {
      int need = KP, over = 0;  // the KP best: `over` above hi, `need` of those in [lo, hi]
      for (;;) {                // block-uniform; every pass takes 8 bits off the range
        const int shift = max(0, 56 - __clzll((long long)(hi - lo)));
        if (tid < 256) hist[tid] = 0;
        __syncthreads();
        for (int e = tid; e < E; e += kSelThreads) {
          const unsigned long long k = ent[e];
          if (k >= lo && k <= hi) atomicAdd(&hist[(int)((k - lo) >> shift)], 1);
        }
        __syncthreads();
        if (warp == 0) {  // the part that holds the need-th from above; lane l holds 8 parts
          int c[8], tot = 0;
#pragma unroll
          for (int x = 0; x < 8; ++x) { c[x] = hist[255 - 8 * lane - x]; tot += c[x]; }
          int inc = tot;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(GCR_FULL, inc, o);
            if (lane >= o) inc += y;
          }
          int run = inc - tot;
          if (run < need && inc >= need) {  // one lane
            bool done = false;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
              if (!done && run + c[x] >= need) { s_bin = 255 - 8 * lane - x; s_over = run; done = true; }
              run += c[x];
            }
          }
        }
        __syncthreads();
        const int bin = s_bin, in = hist[bin];
        need -= s_over;
        over += s_over;
        lo += (unsigned long long)bin << shift;
        const unsigned long long width = (1ull << shift) - 1ull;
        if (hi - lo > width) hi = lo + width;
        if (over + in <= kSelKeep || shift == 0) break;
        __syncthreads();  // hist and the result are read before the next pass clears them
      }
    }
    // (E <= kSelKeep: lo is the smallest key and all are kept)
    for (int e = tid; e < E; e += kSelThreads) {
      const unsigned long long k = ent[e];
      if (k >= lo) {
        const int at = atomicAdd(&s_kept, 1);
        if (at < kSelKeep) keep[at] = k;
      }
    }
    __syncthreads();
    const int n = min(s_kept, kSelKeep), half = (n + 1) / 2;
    const int i = tid & (kSelKeep - 1), j0 = (tid >> 8) * half, j1 = min(n, j0 + half);
    const unsigned long long k = i < n ? keep[i] : 0ull;
    int r = 0;
    if (i < n)
      for (int j = j0; j < j1; ++j) r += keep[j] > k;
    part[tid] = r;
    __syncthreads();
    have = min(n, KP);
    if (tid < n) {
      r = part[tid] + part[tid + kSelKeep];
      if (r < KP) {
        if (s1 < S) {
          ent[r] = k;
        } else {
          ov[out + r] = ordered_to_float((uint32_t)(k >> 32));
          oi[out + r] = (int)~(uint32_t)k;
        }
      }
    }
    __syncthreads();
  }
  for (int r = have + tid; r < KP; r += kSelThreads) { ov[out + r] = -CUDART_INF_F; oi[out + r] = -1; }
}

// One warp per query: the query's row of the operator against the frozen layer, normalised. Lanes
// fetch 32 neighbours' indices, distances and degrees at once and the rows are gathered U at a time:
// neighbour by neighbour, each step waited for three dependent loads (one query, k = 20, d = 256:
// 28 -> 8 us). Sums keep the neighbours' order.
template <int VPL>
__global__ void __launch_bounds__(256) query_step_kernel(const float* __restrict__ xq, int b, int d,
                                                         const float* __restrict__ G, const float* __restrict__ deg,
                                                         const int32_t* __restrict__ nbr,
                                                         const float* __restrict__ d2, int k, float gamma,
                                                         int symmetric, float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int q = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (q >= b) return;
  constexpr int U = VPL <= 2 ? 8 : VPL <= 4 ? 4 : VPL <= 8 ? 2 : 1;
  float wsum = 0.f;
  for (int s0 = 0; s0 < k; s0 += 32) {
    const int s = s0 + lane;
    const int j = s < k ? nbr[(size_t)q * k + s] : -1;
    const float w = j >= 0 ? expf(-d2[(size_t)q * k + s] / gamma) : 0.f;
    for (unsigned m = __ballot_sync(GCR_FULL, j >= 0); m; m &= m - 1) wsum += __shfl_sync(GCR_FULL, w, __ffs(m) - 1);
  }
  const float Dq = symmetric ? 0.5f * (1.f + wsum + 1.f) : 1.f + wsum;
  const float cself = symmetric ? 1.f / Dq : 1.f / sqrtf(Dq);
  float4 acc[VPL];
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int off = v * 128 + lane * 4;
    acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (off < d) {
      const float4 x = *reinterpret_cast<const float4*>(xq + (size_t)q * d + off);
      acc[v] = make_float4(cself * x.x, cself * x.y, cself * x.z, cself * x.w);
    }
  }
  for (int s0 = 0; s0 < k; s0 += 32) {
    const int s = s0 + lane;
    const int j = s < k ? nbr[(size_t)q * k + s] : -1;
    float c = 0.f;
    if (j >= 0) {
      const float w = expf(-d2[(size_t)q * k + s] / gamma);
      c = symmetric ? 0.5f * w / sqrtf(Dq * deg[j]) : w / sqrtf(Dq * deg[j]);
    }
    if constexpr (U == 1) {  // long rows: the columns of one neighbour are loads enough in flight
      for (unsigned m = __ballot_sync(GCR_FULL, j >= 0); m; m &= m - 1) {
        const float cu = __shfl_sync(GCR_FULL, c, __ffs(m) - 1);
        const float* g = G + (size_t)__shfl_sync(GCR_FULL, j, __ffs(m) - 1) * d;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int off = v * 128 + lane * 4;
          if (off < d) {
            const float4 y = *reinterpret_cast<const float4*>(g + off);
            acc[v].x = fmaf(cu, y.x, acc[v].x); acc[v].y = fmaf(cu, y.y, acc[v].y);
            acc[v].z = fmaf(cu, y.z, acc[v].z); acc[v].w = fmaf(cu, y.w, acc[v].w);
          }
        }
      }
    } else {
      for (unsigned m = __ballot_sync(GCR_FULL, j >= 0); m;) {
        float4 y[U][VPL];
        float cu[U];
        int nu = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int l = m ? __ffs(m) - 1 : 0;
          nu += m != 0;
          m &= m - 1;  // (0 stays 0)
          cu[u] = __shfl_sync(GCR_FULL, c, l);
          const int ju = __shfl_sync(GCR_FULL, j, l);
#pragma unroll
          for (int v = 0; v < VPL; ++v) {
            const int off = v * 128 + lane * 4;
            if (u < nu && off < d) y[u][v] = *reinterpret_cast<const float4*>(G + (size_t)ju * d + off);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (u < nu) {
#pragma unroll
            for (int v = 0; v < VPL; ++v)
              if (v * 128 + lane * 4 < d) {
                acc[v].x = fmaf(cu[u], y[u][v].x, acc[v].x); acc[v].y = fmaf(cu[u], y[u][v].y, acc[v].y);
                acc[v].z = fmaf(cu[u], y[u][v].z, acc[v].z); acc[v].w = fmaf(cu[u], y[u][v].w, acc[v].w);
              }
          }
      }
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int v = 0; v < VPL; ++v)
    ss += acc[v].x * acc[v].x + acc[v].y * acc[v].y + acc[v].z * acc[v].z + acc[v].w * acc[v].w;
  ss = warp_sum(ss);
  const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int off = v * 128 + lane * 4;
    if (off < d)
      *reinterpret_cast<float4*>(out + (size_t)q * d + off) =
          make_float4(acc[v].x * inv, acc[v].y * inv, acc[v].z * inv, acc[v].w * inv);
  }
}

// Symmetric degree D = (D_r + D_c) / 2, or D_c for the asymmetric operator.
__global__ void layer_degree_kernel(const float* __restrict__ dr, const float* __restrict__ dc, int n, int symmetric,
                                    float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = symmetric ? 0.5f * (dr[i] + dc[i]) : dc[i];
}

}  // namespace

cudaError_t launch_merge_splits(const float* pv, const int* pi, int S, int kinds, int na, int kp, float* ov, int* oi,
                                int out_rows, int row0, cudaStream_t st) {
  dim3 grid((unsigned)((long)kinds * na));  // one block per (kind, row)
  if (kp == 32) merge_splits_kernel<32><<<grid, 256, 0, st>>>(pv, pi, S, kinds, na, ov, oi, out_rows, row0);
  else if (kp == 64) merge_splits_kernel<64><<<grid, 256, 0, st>>>(pv, pi, S, kinds, na, ov, oi, out_rows, row0);
  else if (kp == 128) merge_splits_kernel<128><<<grid, 256, 0, st>>>(pv, pi, S, kinds, na, ov, oi, out_rows, row0);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

template <int KP>
static cudaError_t pool_finish(const float* pv, const int* pi, const int* cnt, int S, int kinds, int na, int cap,
                               float* ov, int* oi, int out_rows, int row0, cudaStream_t st, Gate gate) {
  const long rows = (long)kinds * na;
  if (S <= 8) {  // a warp per row
    pool_finish_kernel<KP><<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(pv, pi, cnt, S, rows, cap, ov, oi, na, out_rows,
                                                                        row0, gate);
    return cudaGetLastError();
  }
  // a block per row: room for every split's buffer where a block has an SM to itself, for 6,144
  // entries (four blocks per SM) where rows share one
  const int room = rows <= kSMs ? 24576 : 6144;
  const int group = std::max(1, std::min(S, room / cap));
  const size_t smem = sizeof(unsigned long long) * ((size_t)KP + (size_t)group * cap);
  cudaError_t e = cudaFuncSetAttribute(pool_select_kernel<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  pool_select_kernel<KP><<<(unsigned)rows, kSelThreads, smem, st>>>(pv, pi, cnt, S, rows, cap, group, ov, oi, na,
                                                                     out_rows, row0, gate);
  return cudaGetLastError();
}

cudaError_t launch_pool_finish(const float* pv, const int* pi, const int* cnt, int S, int kinds, int na, int cap, int kp,
                               float* ov, int* oi, int out_rows, int row0, cudaStream_t st, Gate gate) {
  if (kp == 32) return pool_finish<32>(pv, pi, cnt, S, kinds, na, cap, ov, oi, out_rows, row0, st, gate);
  if (kp == 64) return pool_finish<64>(pv, pi, cnt, S, kinds, na, cap, ov, oi, out_rows, row0, st, gate);
  if (kp == 128) return pool_finish<128>(pv, pi, cnt, S, kinds, na, cap, ov, oi, out_rows, row0, st, gate);
  return cudaErrorInvalidValue;
}

cudaError_t launch_query_step(const float* xq, int b, int d, const float* G, const float* deg, const int32_t* nbr,
                              const float* d2, int k, float gamma, int symmetric, float* out, cudaStream_t st) {
  dim3 grid((b + 7) / 8);
  const int vpl = (d + 127) / 128;
  if (vpl <= 1) query_step_kernel<1><<<grid, 256, 0, st>>>(xq, b, d, G, deg, nbr, d2, k, gamma, symmetric, out);
  else if (vpl <= 2) query_step_kernel<2><<<grid, 256, 0, st>>>(xq, b, d, G, deg, nbr, d2, k, gamma, symmetric, out);
  else if (vpl <= 4) query_step_kernel<4><<<grid, 256, 0, st>>>(xq, b, d, G, deg, nbr, d2, k, gamma, symmetric, out);
  else if (vpl <= 8) query_step_kernel<8><<<grid, 256, 0, st>>>(xq, b, d, G, deg, nbr, d2, k, gamma, symmetric, out);
  else if (vpl <= 16) query_step_kernel<16><<<grid, 256, 0, st>>>(xq, b, d, G, deg, nbr, d2, k, gamma, symmetric, out);
  else if (vpl <= 32) query_step_kernel<32><<<grid, 256, 0, st>>>(xq, b, d, G, deg, nbr, d2, k, gamma, symmetric, out);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_layer_degree(const float* dr, const float* dc, int n, int symmetric, float* out, cudaStream_t st) {
  layer_degree_kernel<<<(n + 255) / 256, 256, 0, st>>>(dr, dc, n, symmetric, out);
  return cudaGetLastError();
}

}  // namespace gcr
