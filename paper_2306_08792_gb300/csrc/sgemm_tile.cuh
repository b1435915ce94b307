// 128 x 128 FP32 tile product on CUDA cores, shared by the kernels of sgemm.cu.
//
// acc = A_tile . B_tile^T with A, B row-major along K (K contiguous), 128 threads, 8 x 16
// outputs per thread, BK = 16 slices double-buffered through shared memory, two CTAs per SM.
// Each output is one sequential FMA chain over K, which fixes its error bound:
// gamma_K * sum |a_k b_k|.
//
// Bound by FP32 FMA issue and, close behind, by the shared-memory pipe: 8 x 16 outputs read six
// 16-byte operands per 128 FMAs (8 x 8: four per 64). Two neighbouring columns of a thread share
// one packed instruction (fma.rn.f32x2: the same IEEE operation on each half, so the results are
// those of fmaf), which halves the FMA issue slots and leaves room for the operand loads. Four
// lanes load 64 consecutive bytes of a row (a lane per row takes one cache line per lane).
// 1,980 x 11,310 x 2,048 products: 1.96 ms as 8 x 8 outputs of 256 threads with scalar FMAs, 2.11
// with packed ones, 1.73 so (53 of the 75 TFLOP/s that a loop of FMAs alone reaches); scalar FMAs
// in this shape 2.11, operands loaded a step ahead 1.79.
#pragma once
#include "common.cuh"

namespace gcr {
namespace simt {

constexpr int BM = 128, BN = 128, BK = 16, NT = 128;
constexpr int TM = 8, TN = 16;  // outputs of a thread

// Slices lie k-major, [k][row ^ swz(k)]: the swizzle moves groups of 8 rows so that the scalar
// stores of a warp (8 rows x 16 k) hit 32 banks; 16-byte reads stay contiguous.
struct TileSmem {
  float As[2][BK][BM];
  float Bs[2][BK][BN];
};
__device__ __forceinline__ constexpr int swz(int k) { return ((k >> 2) & 3) << 3; }

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ void unpack2(f32x2 p, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(p));
}

// A thread's share of the slice [k0, k0 + 16) of 128 rows: 4 columns of 4 rows, 32 rows apart.
struct Slice {
  float4 v[4];
};
__device__ __forceinline__ void load_slice(Slice& s, const float* __restrict__ base, int nrows,
                                           const int* __restrict__ rowmap, int d, int k0, int tid) {
  const int r = tid >> 2, kk = k0 + ((tid & 3) << 2);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = r + 32 * q;
    s.v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < nrows && kk < d)
      s.v[q] = *reinterpret_cast<const float4*>(base + (size_t)(rowmap ? rowmap[row] : row) * d + kk);
  }
}
__device__ __forceinline__ void store_slice(float (*S)[BM], const Slice& s, int tid) {
  const int k = (tid & 3) << 2, r = (tid >> 2) ^ swz(k);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    S[k + 0][r + 32 * q] = s.v[q].x;
    S[k + 1][r + 32 * q] = s.v[q].y;
    S[k + 2][r + 32 * q] = s.v[q].z;
    S[k + 3][r + 32 * q] = s.v[q].w;
  }
}

// Output (i, j) of a thread: row acc_row(tid, i), column acc_col(tid, j) of the tile. A warp
// covers 64 x 64 outputs as 8 x 4 threads.
__device__ __forceinline__ int acc_row(int tid, int i) {
  return ((tid >> 6) << 6) + (((tid & 31) >> 2) << 2) + (i & 3) + ((i >> 2) << 5);
}
__device__ __forceinline__ int acc_col(int tid, int j) {
  return (((tid >> 5) & 1) << 6) + ((tid & 3) << 2) + (j & 3) + ((j >> 2) << 4);
}

// acc[i][j] = sum_k A[row_i][k] * B[col_j][k]. A rows: abase[(rowmap ? rowmap[r] : r)],
// r < arows; B rows: bbase[c], c < brows; rows past those read as zero.
__device__ __forceinline__ void tile_mma(TileSmem& sm, const float* __restrict__ abase, int arows,
                                         const int* __restrict__ rowmap,
                                         const float* __restrict__ bbase, int brows, int d,
                                         float acc[TM][TN]) {
  const int tid = threadIdx.x;
  const int r0 = acc_row(tid, 0), c0 = acc_col(tid, 0);
  f32x2 p[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) p[i][j] = 0ull;

  Slice ra, rb;
  load_slice(ra, abase, arows, rowmap, d, 0, tid);
  load_slice(rb, bbase, brows, nullptr, d, 0, tid);
  __syncthreads();  // previous users of the staging buffers are done
  store_slice(sm.As[0], ra, tid);
  store_slice(sm.Bs[0], rb, tid);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < d; k0 += BK) {
    const bool more = k0 + BK < d;
    if (more) {
      load_slice(ra, abase, arows, rowmap, d, k0 + BK, tid);
      load_slice(rb, bbase, brows, nullptr, d, k0 + BK, tid);
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&sm.As[buf][kk][r0 ^ swz(kk)]);
      const float4 a1 = *reinterpret_cast<const float4*>(&sm.As[buf][kk][(r0 ^ swz(kk)) + 32]);
      f32x2 b[TN / 2];
#pragma unroll
      for (int j = 0; j < TN / 4; ++j) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(&sm.Bs[buf][kk][(c0 + 16 * j) ^ swz(kk)]);
        b[2 * j] = t.x;
        b[2 * j + 1] = t.y;
      }
      const float a[TM] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      f32x2 aa[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) aa[i] = pack2(a[i], a[i]);
#pragma unroll
      for (int j = 0; j < TN / 2; ++j)
#pragma unroll
        for (int i = 0; i < TM; ++i) fma2(p[i][j], aa[i], b[j]);
    }
    if (more) {
      store_slice(sm.As[buf ^ 1], ra, tid);
      store_slice(sm.Bs[buf ^ 1], rb, tid);
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) unpack2(p[i][j], acc[i][2 * j], acc[i][2 * j + 1]);
}

}  // namespace simt
}  // namespace gcr
