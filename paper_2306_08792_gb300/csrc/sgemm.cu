// FP32 similarity GEMM on CUDA cores (the plain FP32 reference path of the kNN search).
//
// s_ij = x_i . x_j (Sec. III-B: on unit rows ||x_i - x_j||^2 = 2 - 2 s_ij, so the k nearest
// samples are the k largest scores) computed in 128 x 128 tiles, 128 threads, 8 x 16
// outputs per thread, each output a plain sequential FMA chain over d. That fixes the
// error bound used by the certified refinement: |s^ - s| <= gamma_d * ||x_i|| ||x_j||,
// gamma_d = d u / (1 - d u), u = 2^-24.
//
// Three epilogues share the tile loop:
//   POOL  a CTA owns 128 rows and sweeps the column tiles of its split; the scores above a row's
//         threshold go from the accumulators into the row's selection buffer (pool.cuh).
//   BAND  one CTA owns a column tile and loops over blocks of gathered rows; every score
//         at or above the row's threshold is appended to that row's band buffer.
//   DIST  one CTA per (row tile, column tile): writes ||x_q||^2 + ||x_g||^2 - 2 s_qg.
#include <algorithm>
#include <climits>
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "pool.cuh"
#include "sgemm_tile.cuh"

namespace gcr {

using namespace simt;

// ---------------------------------------------------------------------------------- POOL
// S = A . B^T; rows of A own pools, columns are the rows of B. grid = (row blocks, splits): the
// part_rows rows from r0 on, split y sweeps column tiles [y * tps, (y + 1) * tps). GLOBAL / CROSS: which
// graphs' pools it keeps; buffers [split][kind][part_rows][cap], kind0 the first of its kinds among
// them. With self_excl
// (A == B) the diagonal is skipped; the cross-camera graph needs A == B.
//
// Every thread tests its 128 scores of a tile against the rows' thresholds in shared memory and
// appends those above (a slot by atomicAdd); few pass once the thresholds have risen. Then the
// rows' owners (a lane per row and graph) compact the buffers that are nearly full. Scores that
// found a buffer full are tested again after that, so a round always makes room or progress: a
// compaction leaves at least three quarters of CAP - KP slots free. Two CTAs per SM (but for the
// largest pools), so that one's epilogue runs beside the other's FMAs; the earlier kernel kept
// one CTA per SM, one per 128 rows, and passed every score through shared memory to one thread per
// row: 13,290 rows of d = 2048 32.2 -> 14.7 ms, 2,500 rows of d = 256 1.40 -> 0.23 ms.
template <int KP, bool GLOBAL, bool CROSS>
struct SimtPool {
  static constexpr int kinds = (GLOBAL ? 1 : 0) + (CROSS ? 1 : 0);
  static constexpr int cap = SelCap<KP, kinds == 2>::cap;
  static constexpr size_t buf = (size_t)kinds * cap * BM * (sizeof(float) + sizeof(uint16_t));
  static constexpr size_t smem = sizeof(TileSmem) + buf + sizeof(int) * BM * (3 * kinds + 2);
  static constexpr int ctas = 2 * (smem + 1024) <= 228 * 1024 ? 2 : 1;
};

template <int KP, bool GLOBAL, bool CROSS>
__global__ void __launch_bounds__(NT, SimtPool<KP, GLOBAL, CROSS>::ctas)
sgemm_pool_kernel(const float* __restrict__ A, int na, const float* __restrict__ B, int nb, int d,
                  const int* __restrict__ cam, int self_excl, int tps, int r0, int part_rows, int kinds_total, int kind0,
                  float* __restrict__ part_v, int* __restrict__ part_i, int* __restrict__ part_cnt,
                  uint32_t* __restrict__ tau_x) {
  using P = SimtPool<KP, GLOBAL, CROSS>;
  constexpr int KINDS = P::kinds, CAP = P::cap;
  extern __shared__ __align__(16) unsigned char dyn[];
  TileSmem& sm = *reinterpret_cast<TileSmem*>(dyn);
  unsigned char* buf = dyn + sizeof(TileSmem);   // scores [kind][slot][row], then column offsets
  int* cnt_s = reinterpret_cast<int*>(buf + P::buf);          // [kind][row]
  float* tau_s = reinterpret_cast<float*>(cnt_s + KINDS * BM);  // [kind][row]
  int* camr_s = reinterpret_cast<int*>(tau_s + KINDS * BM);     // [row], [column]
  int* camc_s = camr_s + BM;

  const int tid = threadIdx.x;
  const int row0 = r0 + blockIdx.x * BM;
  const int arows = min(BM, na - row0);
  const int ntiles = (nb + BN - 1) / BN;
  const int t0 = blockIdx.y * tps, t1 = min(ntiles, t0 + tps);
  const uint32_t bv = static_cast<uint32_t>(__cvta_generic_to_shared(buf));
  const uint32_t bi = bv + (uint32_t)(KINDS * CAP * BM * sizeof(float));
  // thread r owns row r, of every graph
  const bool valid = tid < arows;
  float tau[KINDS], lo[KINDS], pub[KINDS];
#pragma unroll
  for (int q = 0; q < KINDS; ++q) {
    tau[q] = valid ? -CUDART_INF_F : CUDART_INF_F;
    lo[q] = pub[q] = -CUDART_INF_F;
    cnt_s[q * BM + tid] = 0;
    tau_s[q * BM + tid] = tau[q];
  }
  if (CROSS) camr_s[tid] = tid < arows ? cam[row0 + tid] : -1;

  float acc[TM][TN];
  for (int t = t0; t < t1; ++t) {
    const int col0 = t * BN;
    const int brows = min(BN, nb - col0);
#pragma unroll
    for (int q = 0; q < KINDS; ++q) {
      const uint32_t x = (valid && tau_x) ? __ldcg(tau_x + (size_t)(kind0 + q) * na + row0 + tid) : 0u;
      if (x) tau_s[q * BM + tid] = tau[q] = fmaxf(tau[q], ordered_to_float(x));
    }
    if (CROSS) camc_s[tid] = tid < brows ? cam[col0 + tid] : -1;
    tile_mma(sm, A + (size_t)row0 * d, arows, nullptr, B + (size_t)col0 * d, brows, d, acc);
    // (its barriers also publish the owners' thresholds and counts)
    if (brows < BN || (self_excl && row0 < col0 + BN && col0 < row0 + BM)) {
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int cc = acc_col(tid, j);
          if (cc >= brows || (self_excl && col0 + cc == row0 + acc_row(tid, i))) acc[i][j] = -CUDART_INF_F;
        }
    }
    const int off0 = (t - t0) * BN;
    uint32_t done[KINDS][TM];  // per row a bit for each of its columns already appended
#pragma unroll
    for (int q = 0; q < KINDS; ++q)
#pragma unroll
      for (int i = 0; i < TM; ++i) done[q][i] = 0u;
    for (;;) {
      bool full = false;
#pragma unroll
      for (int q = 0; q < KINDS; ++q) {
        const bool cross_kind = q == 1 || !GLOBAL;
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const int r = acc_row(tid, i);
          const float th = tau_s[q * BM + r];
          float m = acc[i][0];
#pragma unroll
          for (int j = 1; j < TN; ++j) m = fmaxf(m, acc[i][j]);
          if (m > th) {
#pragma unroll
            for (int j = 0; j < TN; ++j) {
              const int cc = acc_col(tid, j);
              if (acc[i][j] > th && !((done[q][i] >> j) & 1u) && !(cross_kind && camc_s[cc] == camr_s[r])) {
                const int pos = atomicAdd(&cnt_s[q * BM + r], 1);
                if (pos < CAP) {
                  sel_st(bv + (uint32_t)(((q * CAP + pos) * BM + r) * sizeof(float)),
                         bi + (uint32_t)(((q * CAP + pos) * BM + r) * sizeof(uint16_t)), acc[i][j], off0 + cc);
                  done[q][i] |= 1u << j;
                } else {
                  full = true;
                }
              }
            }
          }
        }
      }
      const int again = __syncthreads_or(full ? 1 : 0);
#pragma unroll
      for (int q = 0; q < KINDS; ++q) {
        int n = min(cnt_s[q * BM + tid], CAP);
        if (__any_sync(GCR_FULL, n > (again ? KP : CAP - (CAP - KP) / 2))) {
          const SelState ss = sel_compact<KP, CAP, false>(bv + (uint32_t)((q * CAP * BM + tid) * sizeof(float)),
                                                          bi + (uint32_t)((q * CAP * BM + tid) * sizeof(uint16_t)),
                                                          SelState{tau[q], lo[q], pub[q], 0.f, n});
          n = ss.cnt;
          lo[q] = ss.lo;
          tau[q] = ss.tau;
          if (valid && tau_x && ss.pub > pub[q])
            atomicMax(tau_x + (size_t)(kind0 + q) * na + row0 + tid, float_to_ordered(ss.pub));
          pub[q] = ss.pub;
        }
        cnt_s[q * BM + tid] = n;
        // Where ties were cut the threshold is their score, lo just below it. Within the tile lo holds:
        // its scores do not come in column order, and an equal one of a smaller column may follow. A
        // later tile's cannot enter. (With lo for good, each tile's ties were buffered and cut again: the
        // sweep of 13,290 rows of d = 64 that are copies of 8 took 5.7 ms, 1.7 so.)
        if (valid) tau_s[q * BM + tid] = again ? fmaxf(tau_s[q * BM + tid], lo[q]) : tau[q];
      }
      if (!again) break;
      __syncthreads();
    }
  }
  if (!valid) return;
  const int c0 = t0 * BN;
#pragma unroll
  for (int q = 0; q < KINDS; ++q) {
    const int cnt = cnt_s[q * BM + tid];
    const size_t row = ((size_t)blockIdx.y * kinds_total + kind0 + q) * part_rows + row0 - r0 + tid;
    part_cnt[row] = cnt;
    float4* ov = reinterpret_cast<float4*>(part_v + row * CAP);
    int4* oi = reinterpret_cast<int4*>(part_i + row * CAP);
    for (int s = 0; s < cnt; s += 4) {  // (slots past the count: never read)
      const uint32_t va = bv + (uint32_t)(((q * CAP + s) * BM + tid) * sizeof(float));
      const uint32_t ia = bi + (uint32_t)(((q * CAP + s) * BM + tid) * sizeof(uint16_t));
      ov[s >> 2] = make_float4(sel_ldv(va), sel_ldv(va + kSelV), sel_ldv(va + 2 * kSelV), sel_ldv(va + 3 * kSelV));
      oi[s >> 2] = make_int4(c0 + (int)sel_ldi(ia), c0 + (int)sel_ldi(ia + kSelI), c0 + (int)sel_ldi(ia + 2 * kSelI),
                             c0 + (int)sel_ldi(ia + 3 * kSelI));
    }
  }
}

// ---------------------------------------------------------------------------------- BAND
// Rows to rescan: band_row[u] (sample index), band_kind[u], band_thr[u], u < *count.
// grid.x = ceil(n / 128) column tiles; each CTA loops over the row blocks.
__global__ void __launch_bounds__(NT, 2)
sgemm_band_kernel(const float* __restrict__ X, const float* __restrict__ Bm, int n, int d,
                  const int* __restrict__ cam, int self_excl,
                  const int* __restrict__ count, int cap, const int* __restrict__ band_row,
                  const int* __restrict__ band_kind, const float* __restrict__ band_thr,
                  int bcap, int* __restrict__ band_cnt, float* __restrict__ band_v,
                  int* __restrict__ band_i) {
  __shared__ TileSmem sm;
  const int tid = threadIdx.x;
  const int col0 = blockIdx.x * BN;
  const int brows = min(BN, n - col0);
  const int U = min(*count, cap);
  float acc[TM][TN];
  for (int u0 = 0; u0 < U; u0 += BM) {
    const int arows = min(BM, U - u0);
    tile_mma(sm, X, arows, band_row + u0, Bm + (size_t)col0 * d, brows, d, acc);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int ur = acc_row(tid, i);
      if (ur >= arows) continue;
      const int u = u0 + ur;
      const int row = band_row[u];
      const int kind = band_kind[u];
      const float thr = band_thr[u];
      const int rc = cam ? cam[row] : 0;
      // the row's hits first, then one atomic for all of them (see the BAND mode of umma.cu)
      uint32_t hit = 0u;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int cc = acc_col(tid, j);
        const int col = col0 + cc;
        if (cc >= brows || (self_excl && col == row) || acc[i][j] < thr) continue;
        if (kind == 1 && cam[col] == rc) continue;
        hit |= 1u << j;
      }
      if (!hit) continue;
      int pos = atomicAdd(&band_cnt[u], __popc(hit));
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if ((hit >> j) & 1u) {
          if (pos < bcap) {
            band_v[(size_t)u * bcap + pos] = acc[i][j];
            band_i[(size_t)u * bcap + pos] = col0 + acc_col(tid, j);
          }
          ++pos;
        }
    }
  }
}

// ---------------------------------------------------------------------------------- DIST
// D[q][g] = nq[q] + ng[g] - 2 s_qg (squared Euclidean distance), grid = (ceil(ng/128), ceil(nq/128)).
__global__ void __launch_bounds__(NT, 2)
sgemm_dist_kernel(const float* __restrict__ Xq, int nq, const float* __restrict__ Xg, int ng,
                  int d, const float* __restrict__ nrm_q, const float* __restrict__ nrm_g,
                  float* __restrict__ D) {
  __shared__ TileSmem sm;
  const int tid = threadIdx.x;
  const int q0 = blockIdx.y * BM, g0 = blockIdx.x * BN;
  const int arows = min(BM, nq - q0), brows = min(BN, ng - g0);
  float acc[TM][TN];
  tile_mma(sm, Xq + (size_t)q0 * d, arows, nullptr, Xg + (size_t)g0 * d, brows, d, acc);
  // four consecutive columns of a row at a time, as one 16-byte store where the rows allow it
  const bool wide = (ng & 3) == 0 && (reinterpret_cast<uintptr_t>(D) & 15) == 0;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int qr = acc_row(tid, i);
    if (qr >= arows) continue;
    const float a = nrm_q[q0 + qr];
    float* out = D + (size_t)(q0 + qr) * ng + g0;
#pragma unroll
    for (int h = 0; h < TN / 4; ++h) {
      const int gc = acc_col(tid, 4 * h);
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = gc + j < brows ? a + nrm_g[g0 + gc + j] - 2.f * acc[i][4 * h + j] : 0.f;
      if (wide && gc + 4 <= brows) {
        *reinterpret_cast<float4*>(out + gc) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (gc + j < brows) out[gc + j] = v[j];
      }
    }
  }
}

// ---------------------------------------------------------------------------------- launchers
// CTAs of the sweep an SM holds (SimtPool::ctas), by pool size and graphs.
static int simt_ctas(int kp, bool cross) { return kp == 128 || (kp == 64 && cross) ? 1 : 2; }

// As pool_plan: splits whose CTAs fill the SMs evenly. A tile takes about 2 * 128 * 128 * d FMAs
// at the SM's share; set-up, the first tile's rounds and the write-out about 20 us.
constexpr long kFewRowsBytes = 9l << 20;
constexpr int kFewRows = 3 * BM;

static int simt_cap(int kp, bool cross) {
  return kp == 32 ? (cross ? SelCap<32, true>::cap : SelCap<32, false>::cap)
         : kp == 64 ? (cross ? SelCap<64, true>::cap : SelCap<64, false>::cap)
                    : SelCap<128, false>::cap;
}

PoolPlan simt_pool_plan(int na, int nb, int d, int kp, bool cross, int max_splits) {
  PoolPlan p{};
  p.sel = true;
  const bool two = kp == 128 && cross;  // two graphs of 128-entry pools: a sweep for each
  p.cap = simt_cap(kp, cross);
  const int ntiles = (nb + BN - 1) / BN, rblocks = (na + BM - 1) / BM;
  const int slots = kSMs * simt_ctas(kp, cross && !two);
  const double tile_us = d * 0.15, around = 20.0 / tile_us;
  int best = 1;
  double best_t = 1e300;
  // the smallest s of each tps (others of the same tps make the same cut): about 2 sqrt(ntiles) of them,
  // 3 us where all s of one query against 500,000 rows took 40
  for (int s = 1, tps = ntiles; s <= std::min(ntiles, max_splits); s = tps > 1 ? (ntiles + tps - 2) / (tps - 1) : INT_MAX) {
    tps = (ntiles + s - 1) / s;
    if (s > 1 && (long)rblocks * (s - 1) > 16 * slots) break;
    // up to three row blocks (a search of few queries): buffers of at most kFewRowsBytes, so that
    // the workspace stays within what callers with fixed scratch had for such problems
    if (s > 1 && na <= kFewRows && (long)s * na * p.cap * 8 > kFewRowsBytes) break;
    if ((long)tps * BN > kSelMaxCols) continue;
    const long ctas = (long)rblocks * ((ntiles + tps - 1) / tps);
    const double t = std::ceil((double)ctas / slots) * (tps + around);
    if (t < best_t * 0.97) {
      best_t = t;
      best = s;
    }
  }
  while ((long)((ntiles + best - 1) / best) * BN > kSelMaxCols) ++best;
  p.tps = (ntiles + best - 1) / best;
  p.splits = (ntiles + p.tps - 1) / p.tps;
  p.rows = pool_sweep_rows(p, na, cross);
  return p;
}

// The splits of few rows depend on the row count, not on its blocks alone: a smaller search can need
// more. Its buffers are within kFewRowsBytes or what the 16-bit column offsets force, its splits at
// most the column tiles and, up to two row blocks, the places on the chip (which one and two
// blocks divide evenly: no cut of more waves is shorter).
size_t simt_part_rows_bound(int na, int nb, int kp, bool cross) {
  const long few = std::min(na, kFewRows), ntiles = (nb + BN - 1) / BN;
  const long slots = kSMs * simt_ctas(kp, cross && kp != 128), forced = ((long)nb + kSelMaxCols - 1) / kSelMaxCols + 1;
  long rows = std::min(kFewRowsBytes / (simt_cap(kp, cross) * 8), ntiles * few);
  if (few <= 2 * BM) rows = std::min(rows, slots * std::min<long>(few, BM));
  return (size_t)std::max(rows, std::min(forced, ntiles) * few);
}

namespace {
template <int KP, bool GLOBAL, bool CROSS>
cudaError_t launch_simt(const PoolPlan& p, const float* A, int na, const float* B, int nb, int d, const int* cam,
                        int self_excl, int r0, int rows, int kinds_total, int kind0, const PoolParts& parts, uint32_t* tau,
                        cudaStream_t st) {
  using P = SimtPool<KP, GLOBAL, CROSS>;
  auto fn = sgemm_pool_kernel<KP, GLOBAL, CROSS>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::smem);
  if (e != cudaSuccess) return e;
  fn<<<dim3((rows + BM - 1) / BM, p.splits), NT, P::smem, st>>>(A, na, B, nb, d, cam, self_excl, p.tps, r0, rows,
                                                                 kinds_total, kind0, parts.v, parts.i, parts.cnt, tau);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_sgemm_pool(const float* A, int na, const float* B, int nb, int d, const int* cam, int kp,
                              bool cross, int self_excl, const PoolParts& parts, float* pool_v, int* pool_i,
                              cudaStream_t st) {
  const PoolPlan& p = parts.plan;
  const int kinds = cross ? 2 : 1;
  uint32_t* tau = nullptr;
  cudaError_t e = cudaSuccess;
  if (p.splits > 1) {
    tau = parts.tau;
    e = cudaMemsetAsync(tau, 0, sizeof(uint32_t) * kinds * (size_t)na, st);
    if (e != cudaSuccess) return e;
  }
  for (int r0 = 0; r0 < na; r0 += p.rows) {
    const int rows = std::min(p.rows, na - r0);
#define GCR_SIMT(KPV, G, C, K0) \
  launch_simt<KPV, G, C>(p, A, na, B, nb, d, cam, self_excl, r0, rows, kinds, K0, parts, tau, st)
    if (kp == 32) e = cross ? GCR_SIMT(32, true, true, 0) : GCR_SIMT(32, true, false, 0);
    else if (kp == 64) e = cross ? GCR_SIMT(64, true, true, 0) : GCR_SIMT(64, true, false, 0);
    else if (kp == 128) {
      e = GCR_SIMT(128, true, false, 0);
      if (e == cudaSuccess && cross) e = GCR_SIMT(128, false, true, 1);
    } else return cudaErrorInvalidValue;
#undef GCR_SIMT
    if (e != cudaSuccess) return e;
    e = launch_pool_finish(parts.v, parts.i, parts.cnt, p.splits, kinds, rows, p.cap, kp, pool_v, pool_i, na, r0, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_sgemm_band(const float* X, const float* Bm, int n, int d, const int* cam, int self_excl,
                              const int* count, int cap, const int* band_row, const int* band_kind,
                              const float* band_thr, int bcap, int* band_cnt, float* band_v, int* band_i,
                              cudaStream_t st) {
  dim3 grid((n + BN - 1) / BN);
  sgemm_band_kernel<<<grid, NT, 0, st>>>(X, Bm, n, d, cam, self_excl, count, cap, band_row, band_kind, band_thr,
                                          bcap, band_cnt, band_v, band_i);
  return cudaGetLastError();
}

cudaError_t launch_sgemm_dist(const float* Xq, int nq, const float* Xg, int ng, int d,
                              const float* nrm_q, const float* nrm_g, float* D, cudaStream_t st) {
  dim3 grid((ng + BN - 1) / BN, (nq + BM - 1) / BM);
  sgemm_dist_kernel<<<grid, NT, 0, st>>>(Xq, nq, Xg, ng, d, nrm_q, nrm_g, D);
  return cudaGetLastError();
}

}  // namespace gcr
