// Affinity weights, degrees and the propagation operator (Eq. 4-9).
//
// From the kNN lists (ELL: row i lists N_i) this builds, per graph (global, cross-camera):
//   w_ij = exp(-||x_i - x_j||^2 / gamma) for j in N_i        (Eq. 4 / Eq. 8; A~_ii = 1)
//   D_r(i) = 1 + sum_{j in N_i} w_ij,  D_c(j) = 1 + sum_{i: j in N_i} w_ij       (Eq. 5)
// and then one CSR matrix M_mix that a propagation layer applies:
//   symmetric (Eq. 7, Eq. 2): M = D^{-1/2} (A~ + A~^T)/2 D^{-1/2}, D = (D_r + D_c)/2
//   asymmetric (Eq. 6):       M = D_r^{-1/2} A~ D_c^{-1/2}
//   M_mix = alpha M + (1 - alpha) M^cr (Eq. 9); alpha = 1 without the cross-camera graph.
// The transpose A~^T is built by a counting sort whose segments are then sorted by source
// row, so every sum (degrees, operator rows) runs in a fixed order: results are
// bit-reproducible run to run. Operator rows are sorted by column with duplicate columns
// (mutual neighbours, overlapping graphs) merged into one entry.
#include "common.cuh"
#include "kernels.h"

namespace gcr {
namespace {

// The two graphs' arrays, indexed by blockIdx.y (graph 0 the global one): the graphs are
// independent until the operator is assembled, and one launch serves both.
struct PairArgs {
  int n, k;
  float gamma;
  const int32_t* nbr[2];
  const float* d2[2];
  float* w[2];
  float* deg_r[2];
  float* deg_c[2];
  int* cnt[2];       // in-degrees
  int* tptr[2];      // their scan: transposed row pointers
  int* fill[2];
  int* src_tmp[2];   // unsorted transpose
  float* w_tmp[2];
  int* src[2];       // the transpose, each row sorted by source
  float* tw[2];
  int* long_list[2];
  int* long_count;   // [2]
};

// One warp per row: weights, the in-degree counts, and D_r summed in list order.
__global__ void weights_kernel(PairArgs a) {
  const int q = blockIdx.y, lane = threadIdx.x & 31, k = a.k;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= a.n) return;
  float acc = 1.0f;  // A~_ii = 1
  for (int s0 = 0; s0 < k; s0 += 32) {
    const int s = s0 + lane;
    const size_t at = (size_t)i * k + s;
    float wij = 0.f;
    if (s < k) {
      const int j = a.nbr[q][at];
      if (j >= 0) {
        wij = expf(-a.d2[q][at] / a.gamma);
        atomicAdd(&a.cnt[q][j], 1);
      }
      a.w[q][at] = wij;
    }
    const int m = min(32, k - s0);
    for (int t = 0; t < m; ++t) acc += __shfl_sync(GCR_FULL, wij, t);
  }
  if (lane == 0) a.deg_r[q][i] = acc;
}

// Exclusive scan of in[0, n) into out[0, n] (out[n] = total), one block.
__global__ void __launch_bounds__(1024) scan_kernel(const int* __restrict__ in, int* __restrict__ out, int n) {
  const int total = block_scan_1024(n, [&](int i) { return in[i]; }, [&](int i, int p, int) { out[i] = p; });
  if (threadIdx.x == 0) out[n] = total;
}
__global__ void __launch_bounds__(1024) scan_pair_kernel(PairArgs a) {
  const int q = blockIdx.y;
  const int total = block_scan_1024(a.n, [&](int i) { return a.cnt[q][i]; }, [&](int i, int p, int) { a.tptr[q][i] = p; });
  if (threadIdx.x == 0) a.tptr[q][a.n] = total;
}

__global__ void scatter_kernel(PairArgs a) {
  const int q = blockIdx.y;
  const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long)a.n * a.k) return;
  const int i = (int)(t / a.k);
  const int j = a.nbr[q][t];
  if (j < 0) return;
  const int pos = a.tptr[q][j] + atomicAdd(&a.fill[q][j], 1);
  a.src_tmp[q][pos] = i;
  a.w_tmp[q][pos] = a.w[q][t];
}

// Sorting keys held P per lane (element e = p*32 + lane), ascending, payload float.
template <int P, typename Key>
__device__ __forceinline__ void warp_sort_keys(Key (&key)[P], float (&pay)[P], int lane) {
  constexpr int N = 32 * P;
#pragma unroll
  for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= 32) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const int q = p ^ (stride >> 5);
          if (q > p) {
            const int s = p * 32 + lane;
            const bool asc = (s & size) == 0;
            const bool sw = asc ? key[q] < key[p] : key[q] > key[p];
            if (sw) {
              const Key tk = key[p]; key[p] = key[q]; key[q] = tk;
              float tp = pay[p]; pay[p] = pay[q]; pay[q] = tp;
            }
          }
        }
      } else {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const Key ok = __shfl_xor_sync(GCR_FULL, key[p], stride);
          const float op = __shfl_xor_sync(GCR_FULL, pay[p], stride);
          const int s = p * 32 + lane;
          const bool asc = (s & size) == 0;
          const bool lower = (s & stride) == 0;
          const bool take = (lower == asc) ? ok < key[p] : ok > key[p];
          if (take) { key[p] = ok; pay[p] = op; }
        }
      }
    }
  }
}

// Ascending sort of 32-bit keys alone, as above.
template <int P>
__device__ __forceinline__ void warp_sort_u32(uint32_t (&key)[P], int lane) {
  constexpr int N = 32 * P;
#pragma unroll
  for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll
      for (int p = 0; p < P; ++p) {
        if (stride >= 32) {
          const int q = p ^ (stride >> 5);
          if (q > p) {
            const bool asc = ((p * 32 + lane) & size) == 0;
            const uint32_t lo = min(key[p], key[q]), hi = max(key[p], key[q]);
            key[p] = asc ? lo : hi;
            key[q] = asc ? hi : lo;
          }
        } else {
          const uint32_t ok = __shfl_xor_sync(GCR_FULL, key[p], stride);
          const int s = p * 32 + lane;
          key[p] = (((s & stride) == 0) == ((s & size) == 0)) ? min(key[p], ok) : max(key[p], ok);
        }
      }
    }
  }
}

// Sort one transposed segment by source row (register bitonic for <= 32*P entries).
template <int P>
__device__ void tseg_sort_regs(int beg, int len, const int* __restrict__ src_tmp, const float* __restrict__ w_tmp,
                               int* __restrict__ src, float* __restrict__ tw, int lane) {
  uint32_t key[P];
  float pay[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    key[p] = e < len ? (uint32_t)src_tmp[beg + e] : ~0u;
    pay[p] = e < len ? w_tmp[beg + e] : 0.f;
  }
  warp_sort_keys<P>(key, pay, lane);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    if (e < len) { src[beg + e] = (int)key[p]; tw[beg + e] = pay[p]; }
  }
}

constexpr int kLongSeg = 256;  // longer transposed segments (in-degree hubs) go to tsort_long_kernel

// One warp per transposed row j: sort its entries by source, then D_c(j) = 1 + sum. Longer rows
// are listed (in arbitrary order, each is processed on its own) for tsort_long_kernel, which
// sorts them and sets their D_c.
__global__ void tsort_kernel(PairArgs a) {
  const int q = blockIdx.y, lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= a.n) return;
  const int beg = a.tptr[q][j], len = a.tptr[q][j + 1] - beg;
  const int* st = a.src_tmp[q];
  const float* wt = a.w_tmp[q];
  int* src = a.src[q];
  float* tw = a.tw[q];
  if (len <= 32) tseg_sort_regs<1>(beg, len, st, wt, src, tw, lane);
  else if (len <= 64) tseg_sort_regs<2>(beg, len, st, wt, src, tw, lane);
  else if (len <= 128) tseg_sort_regs<4>(beg, len, st, wt, src, tw, lane);
  else if (len <= kLongSeg) tseg_sort_regs<8>(beg, len, st, wt, src, tw, lane);
  else {
    if (lane == 0) a.long_list[q][atomicAdd(a.long_count + q, 1)] = j;
    return;
  }
  __syncwarp();
  float acc = 1.0f;  // A~_jj = 1, then the weights in order
  for (int e0 = 0; e0 < len; e0 += 32) {
    const float x = e0 + lane < len ? tw[beg + e0 + lane] : 0.f;
    const int m = min(32, len - e0);
    for (int t = 0; t < m; ++t) acc += __shfl_sync(GCR_FULL, x, t);
  }
  if (lane == 0) a.deg_c[q][j] = acc;
}

// One CTA per long transposed segment (a persistent loop over the list): a stable LSD radix
// sort of the segment by source row (8-bit digits, nbits = bits of the largest row index),
// chunk by chunk through global memory in segment order, so the work is linear in the
// segment's length (an in-degree hub can hold tens of thousands of entries). Within a chunk
// each warp ranks its keys slot by slot (lanes with equal digits found by ballots); a running
// per-digit offset carries the order from chunk to chunk. The weights follow their keys. Then D_c(j) = 1 + sum
// of the weights, reduced in a fixed order.
template <int IPT>
__global__ void __launch_bounds__(256) tsort_long_kernel(PairArgs a, int nbits) {
  constexpr int NT = 256, NW = NT / 32, CH = NT * IPT;
  __shared__ uint32_t dbase[256];       // running offset of each digit in the segment
  __shared__ uint32_t wcnt[NW][257];    // per-warp digit counts of a chunk (column 256: past the end)
  __shared__ float red[NW];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int q = blockIdx.y;
  const int* __restrict__ tptr = a.tptr[q];
  const int* __restrict__ list = a.long_list[q];
  int *src_tmp = a.src_tmp[q], *src = a.src[q];
  float *w_tmp = a.w_tmp[q], *tw = a.tw[q], *deg_c = a.deg_c[q];
  const int total = a.long_count[q];
  for (int li = blockIdx.x; li < total; li += gridDim.x) {
    const int j = list[li];
    const int beg = tptr[j], L = tptr[j + 1] - beg;
    int* ka = src_tmp + beg;
    float* va = w_tmp + beg;
    int* kb = src + beg;
    float* vb = tw + beg;
    for (int shift = 0; shift < nbits; shift += 8) {
      for (int v = t; v < 256; v += NT) dbase[v] = 0;
      __syncthreads();
      for (int e = t; e < L; e += NT) atomicAdd(&dbase[((uint32_t)ka[e] >> shift) & 255u], 1u);
      __syncthreads();
      if (w == 0) {  // exclusive scan of the 256 digit counts
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) { c[u] = dbase[lane * 8 + u]; sum += c[u]; }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(GCR_FULL, inc, o);
          if (lane >= o) inc += y;
        }
        uint32_t run = inc - sum;
#pragma unroll
        for (int u = 0; u < 8; ++u) { dbase[lane * 8 + u] = run; run += c[u]; }
      }
      __syncthreads();
      for (int c0 = 0; c0 < L; c0 += CH) {
        for (int v = t; v < NW * 257; v += NT) (&wcnt[0][0])[v] = 0;
        __syncthreads();
        uint32_t key[IPT], off[IPT], dg[IPT];
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
          const int e = c0 + w * 32 * IPT + i * 32 + lane;
          key[i] = e < L ? (uint32_t)ka[e] : 0u;
          dg[i] = e < L ? ((key[i] >> shift) & 255u) : 256u;
          const unsigned peers = warp_peers(dg[i], 9);  // digits 0..256 (256: past the end)
          const uint32_t base = wcnt[w][dg[i]];
          __syncwarp();
          if ((peers & lt) == 0) wcnt[w][dg[i]] = base + (uint32_t)__popc(peers);  // the lowest peer updates
          __syncwarp();
          off[i] = base + (uint32_t)__popc(peers & lt);
        }
        __syncthreads();
        {  // digit t: offsets of each warp's keys in (digit, warp) order, then the running base
          uint32_t run = dbase[t];
#pragma unroll
          for (int ww = 0; ww < NW; ++ww) {
            const uint32_t cc = wcnt[ww][t];
            wcnt[ww][t] = run;
            run += cc;
          }
          dbase[t] = run;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
          const int e = c0 + w * 32 * IPT + i * 32 + lane;
          if (e < L) {
            const uint32_t dst = wcnt[w][dg[i]] + off[i];
            kb[dst] = (int)key[i];
            vb[dst] = va[e];
          }
        }
        __syncthreads();
      }
      int* tk = ka; ka = kb; kb = tk;
      float* tv = va; va = vb; vb = tv;
    }
    if (ka != src + beg) {  // an even number of passes leaves the result in the scratch
      for (int e = t; e < L; e += NT) { src[beg + e] = ka[e]; tw[beg + e] = va[e]; }
      __syncthreads();
    }
    float sum = 0.f;
    for (int e = t; e < L; e += NT) sum += tw[beg + e];
    sum = warp_sum(sum);
    if (lane == 0) red[w] = sum;
    __syncthreads();
    if (t == 0) {
      float acc = 1.0f;  // A~_jj = 1
      for (int ww = 0; ww < NW; ++ww) acc += red[ww];
      deg_c[j] = acc;
    }
    __syncthreads();
  }
}

struct OpArgs {
  int n, k, kinds, symmetric;
  float coef[2];          // alpha, 1 - alpha
  const int32_t* nbr[2];
  const float* w[2];
  const float* deg_r[2];
  const float* deg_c[2];
  const int* tptr[2];
  const int* tsrc[2];
  const float* tw[2];
  const double* inv_r[2];  // per graph: 1/sqrt(D_i) (Eq. 7, D the mean of row and column
  const double* inv_c[2];  // degrees) in both, or 1/sqrt(D_r,i) and 1/sqrt(D_c,i) (Eq. 6)
  const int* rowptr;
  int* len;
  int* col;
  float* val;
  int* raw_col;
  float* raw_val;
};

// Per row: the inverse square roots of its degrees, per graph (FP64: every operator entry is then
// a product, without a square root or division per entry), and its raw operator entries.
__global__ void op_prepare_kernel(OpArgs a, double* __restrict__ inv, int* __restrict__ cnt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  int c = 1;
  for (int g = 0; g < a.kinds; ++g) {
    double* inv_r = inv + (size_t)(2 * g) * a.n;
    double* inv_c = inv_r + a.n;
    if (a.symmetric) {
      const double r = 1.0 / sqrt(0.5 * ((double)a.deg_r[g][i] + (double)a.deg_c[g][i]));
      inv_r[i] = r;
      inv_c[i] = r;
    } else {
      inv_r[i] = 1.0 / sqrt((double)a.deg_r[g][i]);
      inv_c[i] = 1.0 / sqrt((double)a.deg_c[g][i]);
    }
    c += a.k;
    if (a.symmetric) c += a.tptr[g][i + 1] - a.tptr[g][i];
  }
  cnt[i] = c;
}

// Raw entries of operator row i in a fixed generation order: self, then per graph its
// N_i entries (rank order) and, when symmetric, its transposed entries (by source).
__device__ __forceinline__ void gen_entry(const OpArgs& a, int i, int e, int& col, double& v) {
  // e == 0: self loop
  // self loop: A~_ii = 1, scaled by 1/D_i (Eq. 7) or 1/sqrt(D_r,i D_c,i) (Eq. 6)
  if (e == 0) {
    double s = 0.0;
    for (int g = 0; g < a.kinds; ++g) s += a.coef[g] * (a.inv_r[g][i] * a.inv_c[g][i]);
    col = i;
    v = s;
    return;
  }
  const double half = a.symmetric ? 0.5 : 1.0;  // (A~ + A~^T) / 2 in Eq. 7
  int r = e - 1;
  for (int g = 0; g < a.kinds; ++g) {
    if (r < a.k) {
      const int j = a.nbr[g][(size_t)i * a.k + r];
      const double wij = a.w[g][(size_t)i * a.k + r];
      if (j < 0) { col = -1; v = 0.0; return; }
      col = j;
      v = a.coef[g] * half * wij * (a.inv_r[g][i] * a.inv_c[g][j]);
      return;
    }
    r -= a.k;
    if (a.symmetric) {
      const int tb = a.tptr[g][i], tl = a.tptr[g][i + 1] - tb;
      if (r < tl) {
        const int s = a.tsrc[g][tb + r];
        const double wsi = a.tw[g][tb + r];
        col = s;
        v = a.coef[g] * 0.5 * wsi * (a.inv_r[g][i] * a.inv_c[g][s]);
        return;
      }
      r -= tl;
    }
  }
  col = -1;
  v = 0.0;
}

// Rows of up to 128 entries: one 32-bit key (column, generation position) per entry is sorted
// alone and its value fetched from shared memory after, and runs of equal columns are merged
// there (against 64-bit keys with their values, staged through global memory: 133 -> 93 us per
// build on 19,281 rows of about 60 entries). n <= 2^24, so column and 7-bit position fit below the empty key.
template <int P>
__device__ __forceinline__ void op_row_small(const OpArgs& a, int i, int beg, int L, int lane, uint32_t* skey,
                                             float* sval) {
  uint32_t key[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    int c = -1;
    double v = 0.0;
    if (e < L) gen_entry(a, i, e, c, v);
    key[p] = c >= 0 ? ((uint32_t)c << 7 | (uint32_t)e) : ~0u;
    sval[e] = (float)v;
  }
  warp_sort_u32<P>(key, lane);
  __syncwarp();
  float val[P];
#pragma unroll
  for (int p = 0; p < P; ++p) val[p] = key[p] != ~0u ? sval[key[p] & 127u] : 0.f;
  __syncwarp();
#pragma unroll
  for (int p = 0; p < P; ++p) {
    skey[p * 32 + lane] = key[p] == ~0u ? ~0u : key[p] >> 7;
    sval[p * 32 + lane] = val[p];
  }
  __syncwarp();
  int written = 0;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    const uint32_t c = skey[e];
    const bool head = c != ~0u && (e == 0 || skey[e - 1] != c);
    float v = 0.f;
    if (head) {
      v = sval[e];
      for (int f = e + 1; f < 32 * P && skey[f] == c; ++f) v += sval[f];
    }
    const unsigned hm = __ballot_sync(GCR_FULL, head);
    if (head) {
      const int pos = written + __popc(hm & ((1u << lane) - 1));
      a.col[beg + pos] = (int)c;
      a.val[beg + pos] = v;
    }
    written += __popc(hm);
  }
  if (lane == 0) a.len[i] = written;
}

template <int P>
__device__ void op_row_regs(const OpArgs& a, int i, int beg, int L, int lane) {
  unsigned long long key[P];
  float pay[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    int c = -1;
    double v = 0.0;
    if (e < L) gen_entry(a, i, e, c, v);
    // key: column, then generation position (invalid entries sort last)
    key[p] = c >= 0 ? (((unsigned long long)(unsigned)c << 32) | (unsigned)e) : ~0ull;
    pay[p] = (float)v;
  }
  warp_sort_keys<P>(key, pay, lane);
  // stage sorted entries in the raw buffer, then merge runs of equal columns
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    if (e < L) {
      a.raw_col[beg + e] = key[p] == ~0ull ? -1 : (int)(key[p] >> 32);
      a.raw_val[beg + e] = pay[p];
    }
  }
  __syncwarp();
  int written = 0;
  for (int e0 = 0; e0 < L; e0 += 32) {
    const int e = e0 + lane;
    int c = e < L ? a.raw_col[beg + e] : -1;
    const bool head = c >= 0 && (e == 0 || a.raw_col[beg + e - 1] != c);
    float v = 0.f;
    if (head) {
      v = a.raw_val[beg + e];
      for (int f = e + 1; f < L && a.raw_col[beg + f] == c; ++f) v += a.raw_val[beg + f];
    }
    const unsigned hm = __ballot_sync(GCR_FULL, head);
    if (head) {
      const int pos = written + __popc(hm & ((1u << lane) - 1));
      a.col[beg + pos] = c;
      a.val[beg + pos] = v;
    }
    written += __popc(hm);
  }
  if (lane == 0) a.len[i] = written;
}

// One warp per operator row.
__global__ void __launch_bounds__(256) op_fill_kernel(OpArgs a) {
  __shared__ uint32_t skey[8][128];
  __shared__ float sval[8][128];
  const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
  const int i = blockIdx.x * 8 + wb;
  if (i >= a.n) return;
  const int beg = a.rowptr[i], L = a.rowptr[i + 1] - beg;
  if (L <= 32) op_row_small<1>(a, i, beg, L, lane, skey[wb], sval[wb]);
  else if (L <= 64) op_row_small<2>(a, i, beg, L, lane, skey[wb], sval[wb]);
  else if (L <= 128) op_row_small<4>(a, i, beg, L, lane, skey[wb], sval[wb]);
  else if (L <= 256) op_row_regs<8>(a, i, beg, L, lane);
  else {
    // very long row (hub): keep the entries unmerged, in generation order
    int written = 0;
    for (int e0 = 0; e0 < L; e0 += 32) {
      const int e = e0 + lane;
      int c = -1;
      double v = 0.0;
      if (e < L) gen_entry(a, i, e, c, v);
      const unsigned hm = __ballot_sync(GCR_FULL, c >= 0);
      if (c >= 0) {
        const int pos = written + __popc(hm & ((1u << lane) - 1));
        a.col[beg + pos] = c;
        a.val[beg + pos] = (float)v;
      }
      written += __popc(hm);
    }
    if (lane == 0) a.len[i] = written;
  }
}

}  // namespace

cudaError_t launch_scan(const int* in, int* out, int n, cudaStream_t st) {
  scan_kernel<<<1, 1024, 0, st>>>(in, out, n);
  return cudaGetLastError();
}

cudaError_t launch_build_operator(const GraphArgs& g, cudaStream_t st) {
  const int n = g.n, k = g.k;
  const unsigned kinds = (unsigned)g.kinds;
  PairArgs t;
  t.n = n; t.k = k; t.gamma = g.gamma; t.long_count = g.long_count;
  for (int q = 0; q < 2; ++q) {
    const int s = q < g.kinds ? q : 0;
    t.nbr[q] = g.nbr[s]; t.d2[q] = g.d2[s]; t.w[q] = g.w[s];
    t.deg_r[q] = g.deg_r[s]; t.deg_c[q] = g.deg_c[s];
    t.cnt[q] = g.cnt[s]; t.fill[q] = g.fill[s];
    t.tptr[q] = s ? g.scan_tmp2 : g.scan_tmp;
    // unsorted transposes: the operator's buffers and the raw ones, unused until it is filled
    t.src_tmp[q] = s ? g.raw_col : g.op_col;
    t.w_tmp[q] = s ? g.raw_val : g.op_val;
    t.src[q] = g.t_src[s]; t.tw[q] = g.t_w[s];
    t.long_list[q] = s ? g.long_list2 : g.long_list;
  }
  cudaError_t e = cudaMemsetAsync(g.zero, 0, sizeof(int) * g.zero_n, st);  // counts, fills, hub counts
  if (e != cudaSuccess) return e;
  weights_kernel<<<dim3((n + 7) / 8, kinds), 256, 0, st>>>(t);
  scan_pair_kernel<<<dim3(1, kinds), 1024, 0, st>>>(t);
  if ((long)n * k > 0) scatter_kernel<<<dim3((unsigned)(((long)n * k + 255) / 256), kinds), 256, 0, st>>>(t);
  tsort_kernel<<<dim3((n + 7) / 8, kinds), 256, 0, st>>>(t);
  int nbits = 0;
  while (nbits < 31 && ((long)1 << nbits) < (long)n) ++nbits;
  tsort_long_kernel<8><<<dim3(2 * kSMs, kinds), 256, 0, st>>>(t, nbits);

  OpArgs a;
  a.n = n; a.k = k; a.kinds = g.kinds; a.symmetric = g.symmetric;
  a.coef[0] = g.kinds == 2 ? g.alpha : 1.0f;
  a.coef[1] = 1.0f - g.alpha;
  for (int q = 0; q < 2; ++q) {
    const int qq = q < g.kinds ? q : 0;
    a.nbr[q] = g.nbr[qq]; a.w[q] = g.w[qq]; a.deg_r[q] = g.deg_r[qq]; a.deg_c[q] = g.deg_c[qq];
    a.tptr[q] = t.tptr[qq]; a.tsrc[q] = g.t_src[qq]; a.tw[q] = g.t_w[qq];
    a.inv_r[q] = g.inv + (size_t)(2 * qq) * n;
    a.inv_c[q] = g.inv + (size_t)(2 * qq + 1) * n;
  }
  a.rowptr = g.op_rowptr; a.len = g.op_len; a.col = g.op_col; a.val = g.op_val;
  a.raw_col = g.raw_col; a.raw_val = g.raw_val;
  op_prepare_kernel<<<(n + 255) / 256, 256, 0, st>>>(a, g.inv, g.op_cnt);
  scan_kernel<<<1, 1024, 0, st>>>(g.op_cnt, g.op_rowptr, n);
  op_fill_kernel<<<(n + 7) / 8, 256, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace gcr
