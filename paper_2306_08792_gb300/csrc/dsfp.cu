// DSFP: decentralized and synchronous feature propagation (Algorithm 1, Sec. III-B).
//
// For image i the local node set is L = {i} u N_i (m = 1 + |N_i| <= kDsfpMaxK + 1 nodes,
// local index 0 is i). Algorithm 1 builds the symmetric local similarity matrix
// A_uv = exp(-||x_u - x_v||^2 / gamma) over every pair of L, its degrees D_u = sum_v A_uv,
// M = D^{-1/2} A D^{-1/2}, and iterates X_{t+1} = M X_t on the m x d local features (each
// iteration followed by the row L2 normalisation, as in the global method). The output for
// image i is its own row of X_T.
//
// Every local row stays a combination of the input rows: X_t = P_t X_0 with P_t an m x m
// matrix, so the iterations run in the m x m space:
//   Y = M P_t,  ||row u of Y X_0||^2 = (Y G Y^T)_uu with G = X_0 X_0^T (the local Gram),
//   P_{t+1} = diag(1 / ||row u||) Y.
// G is also all that A needs (||x_u - x_v||^2 = G_uu + G_vv - 2 G_uv). So one CTA per image
// computes G over d in staged column chunks (the only pass over the m rows besides the
// output), runs the small recurrence, and writes sum_v Y_0v x_v / ||.|| for the last
// iteration's Y, the norm again from G. FP32 throughout; the Gram and the output are plain
// FP32 dot products.
// A chunk is staged row-major (a straight float4 copy).
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace gcr {
namespace {

constexpr int kDsfpThreads = 128;
constexpr int kCh = 128;   // columns per staged chunk
// Gram register tile of dsfp_kernel (kTl x kTl entries per thread and job).
constexpr int kTl = 3;
constexpr int kTT = kTl * kTl;
constexpr int kMaxGroups = 4;   // column-quad groups per tile pair (measured: 4 beats 6 and 8)

struct DsfpLayout {
  int mp;      // m rounded up to kTl (rows of the staged chunk)
  int cs;      // row stride of the chunk, kCh + 4 (float4-aligned, staggers the banks)
  int tiles;   // mp / kTl
  int tp;      // tile pairs (a <= b)
  int groups;  // column-quad groups per tile pair (<= kMaxGroups)
  int jobs;    // tp * groups (<= 2 * kDsfpThreads)
  size_t chunk_off, parts_off, mat_off, bytes;
};

__host__ __device__ inline DsfpLayout dsfp_layout(int m_max) {
  DsfpLayout L;
  L.mp = (m_max + kTl - 1) / kTl * kTl;
  L.cs = kCh + 4;
  L.tiles = L.mp / kTl;
  L.tp = L.tiles * (L.tiles + 1) / 2;
  // column-quad groups: as many as one job per thread allows (two jobs per thread past 128
  // tile pairs). Consecutive lanes take consecutive quads of the same tile pair, so a warp's
  // float4 reads mostly hit distinct banks (lanes on different 4-row tiles would alias: tiles
  // are 528 floats apart)
  L.groups = L.tp >= kDsfpThreads ? 1 : (kDsfpThreads / L.tp < kMaxGroups ? kDsfpThreads / L.tp : kMaxGroups);
  L.jobs = L.tp * L.groups;
  L.chunk_off = 0;
  L.parts_off = L.chunk_off + sizeof(float) * (size_t)2 * L.mp * L.cs;  // two chunk buffers
  L.mat_off = L.parts_off + sizeof(float) * (size_t)L.jobs * kTl * kTl;
  // G, M, P, Y (each mp x mp), then the row norms and degrees
  L.bytes = L.mat_off + sizeof(float) * ((size_t)4 * L.mp * L.mp + 2 * L.mp);
  return L;
}

// Asynchronous 16-byte global -> shared copy (zero-fill when !valid; src must still be a
// valid address), its group commit and wait.
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Copies columns [c0, c0 + kCh) of the local rows into a chunk buffer (rows >= m and columns
// >= d read as zero).
__device__ __forceinline__ void stage_chunk(float* buf, const float* __restrict__ X, const int* loc, int m, int mp,
                                            int cs, int d, int c0) {
  for (int e = threadIdx.x; e < mp * (kCh / 4); e += kDsfpThreads) {
    const int r = e / (kCh / 4), c4 = (e % (kCh / 4)) * 4;
    const bool ok = r < m && c0 + c4 < d;  // d % 4 == 0: a quad is wholly in or out
    cp_async16(buf + r * cs + c4, ok ? X + (size_t)loc[r] * d + c0 + c4 : X, ok);
  }
}

// The small m x m algebra from G (rows of mp floats): leaves the output weights in deg.
template <int THREADS>
__device__ __forceinline__ void dsfp_local(const float* G, float* M, float* P, float* Y, float* nrm, float* deg, int m,
                                           int mp, float gamma, int T) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // ---- A, degrees, M = D^{-1/2} A D^{-1/2} (steps 3 and 5): one warp per row u, lanes
  // over the columns v, row sums by warp reduction
  for (int u = warp; u < m; u += THREADS / 32) {
    float s = 0.f;
    for (int v = lane; v < m; v += 32) {
      const float d2 = fmaxf(0.f, G[u * mp + u] + G[v * mp + v] - 2.f * G[u * mp + v]);
      const float a = u == v ? 1.f : expf(-d2 / gamma);
      M[u * mp + v] = a;
      s += a;
    }
    s = warp_sum(s);
    if (lane == 0) deg[u] = 1.f / sqrtf(s);
  }
  __syncthreads();
  for (int u = warp; u < m; u += THREADS / 32)
    for (int v = lane; v < m; v += 32) {
      const float a = M[u * mp + v] * (deg[u] * deg[v]);
      M[u * mp + v] = a;
      Y[u * mp + v] = a;  // Y_1 = M P_0 = M
    }
  __syncthreads();

  // ---- step 6 in the m x m space: per iteration ||row u of Y X_0||^2 = sum_w (Y G)_uw Y_uw,
  // P = diag(1/||row u||) Y, Y <- M P
  for (int t = 1;; ++t) {
    const int rows = t < T ? m : 1;  // the last iteration needs the norm of row 0 only
    for (int u = warp; u < rows; u += THREADS / 32) {
      float s = 0.f;
      for (int w = lane; w < m; w += 32) {
        float z = 0.f;
        for (int v = 0; v < m; ++v) z = fmaf(Y[u * mp + v], G[v * mp + w], z);
        s = fmaf(z, Y[u * mp + w], s);
      }
      s = warp_sum(s);
      if (lane == 0) nrm[u] = s > 0.f ? 1.f / sqrtf(s) : 0.f;
    }
    __syncthreads();
    if (t == T) break;
    for (int u = warp; u < m; u += THREADS / 32)
      for (int v = lane; v < m; v += 32) P[u * mp + v] = Y[u * mp + v] * nrm[u];
    __syncthreads();
    for (int u = warp; u < m; u += THREADS / 32)
      for (int v = lane; v < m; v += 32) {
        float s = 0.f;
        for (int w = 0; w < m; ++w) s = fmaf(M[u * mp + w], P[w * mp + v], s);
        Y[u * mp + v] = s;
      }
    __syncthreads();
  }
  // output weights: row 0 of the last Y, scaled by the norm of that row's combination
  if (tid < m) deg[tid] = Y[tid] * nrm[0];
  __syncthreads();
}

// out = sum_v w_v x_v over the local rows, a column quad per thread: the m loads of a quad are
// independent of each other and of any barrier (staged through shared memory chunk by chunk, each
// chunk waited for the one before).
template <int THREADS>
__device__ __forceinline__ void dsfp_output(const float* __restrict__ X, int d, const int* loc, const float* w, int m,
                                            float* __restrict__ out) {
  for (int c = threadIdx.x * 4; c < d; c += THREADS * 4) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int v = 0; v < m; ++v) {
      const float4 x = __ldcg(reinterpret_cast<const float4*>(X + (size_t)loc[v] * d + c));
      const float wv = w[v];
      s.x = fmaf(wv, x.x, s.x);
      s.y = fmaf(wv, x.y, s.y);
      s.z = fmaf(wv, x.z, s.z);
      s.w = fmaf(wv, x.w, s.w);
    }
    *reinterpret_cast<float4*>(out + c) = s;
  }
}

// Local node set: i, then its valid neighbours in list order (warp 0).
__device__ __forceinline__ void dsfp_nodes(const int32_t* __restrict__ nbr, int i, int k, int* loc, int* s_m) {
  const int lane = threadIdx.x & 31;
  int cnt = 1;
  if (lane == 0) loc[0] = i;
  for (int s0 = 0; s0 < k; s0 += 32) {
    const int s = s0 + lane;
    const int j = s < k ? nbr[(size_t)i * k + s] : -1;
    const unsigned vm = __ballot_sync(GCR_FULL, j >= 0);
    if (j >= 0) loc[cnt + __popc(vm & ((1u << lane) - 1))] = j;
    cnt += __popc(vm);
  }
  if (lane == 0) *s_m = cnt;
}

__device__ __forceinline__ void dsfp_copy_row(const float* __restrict__ X, int i, int d, float* __restrict__ out,
                                              int threads) {
  for (int c4 = threadIdx.x; c4 < (d >> 2); c4 += threads)
    reinterpret_cast<float4*>(out + (size_t)i * d)[c4] = reinterpret_cast<const float4*>(X + (size_t)i * d)[c4];
}

// grid = n CTAs (one per image), kDsfpThreads threads, dynamic shared memory = layout.bytes.
// The Gram streams column chunks through two buffers: chunk c + 1 is in flight while chunk c is
// used. For more than 32 local rows; up to 32, dsfp_tile_kernel.
__global__ void __launch_bounds__(kDsfpThreads) dsfp_kernel(const float* __restrict__ X, int n, int d,
                                                            const int32_t* __restrict__ nbr, int k, float gamma,
                                                            int T, int m_max, float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int loc[kDsfpMaxK + 1];
  __shared__ int s_m;
  const DsfpLayout L = dsfp_layout(m_max);
  float* buf0 = reinterpret_cast<float*>(smem + L.chunk_off);   // [2][mp][cs]
  float* parts = reinterpret_cast<float*>(smem + L.parts_off);  // [jobs][kTT]
  float* G = reinterpret_cast<float*>(smem + L.mat_off);         // [mp][mp]
  float* M = G + L.mp * L.mp;
  float* P = M + L.mp * L.mp;
  float* Y = P + L.mp * L.mp;
  float* nrm = Y + L.mp * L.mp;                                  // [mp]
  float* deg = nrm + L.mp;                                       // [mp]
  const int tid = threadIdx.x, warp = tid >> 5;
  const int i = blockIdx.x;
  const int mp = L.mp, cs = L.cs;
  const int nch = (d + kCh - 1) / kCh;
  const int bufsz = mp * cs;

  if (T == 0) {  // the (already normalised) input row
    dsfp_copy_row(X, i, d, out, kDsfpThreads);
    return;
  }
  if (warp == 0) dsfp_nodes(nbr, i, k, loc, &s_m);
  __syncthreads();
  const int m = s_m;

  // ---- local Gram G = X_L X_L^T over d
  float acc[2][kTl][kTl];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int a = 0; a < kTl; ++a)
#pragma unroll
      for (int b = 0; b < kTl; ++b) acc[q][a][b] = 0.f;
  // job j = (tile pair j / groups, column-quad group j % groups); thread tid takes jobs tid
  // and tid + 128
  int ta[2], tb[2], tg[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int j = tid + q * kDsfpThreads;
    int pr = j < L.jobs ? j / L.groups : 0;
    tg[q] = j < L.jobs ? j % L.groups : -1;
    int a = 0;
    while (pr >= L.tiles - a) { pr -= L.tiles - a; ++a; }
    ta[q] = a;
    tb[q] = a + pr;
  }
  stage_chunk(buf0, X, loc, m, mp, cs, d, 0);
  cp_async_commit();
  for (int ci = 0; ci < nch; ++ci) {
    if (ci + 1 < nch) stage_chunk(buf0 + ((ci + 1) & 1) * bufsz, X, loc, m, mp, cs, d, (ci + 1) * kCh);
    cp_async_commit();  // (an empty group on the last chunk keeps the count uniform)
    cp_async_wait_prev();
    __syncthreads();
    const float* chunk = buf0 + (ci & 1) * bufsz;
    const int cw = min(kCh, d - ci * kCh);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (tg[q] < 0) continue;
      const float* ra = chunk + ta[q] * kTl * cs;
      const float* rb = chunk + tb[q] * kTl * cs;
      for (int c4 = tg[q] * 4; c4 < cw; c4 += L.groups * 4) {
        float4 u[kTl], v[kTl];
#pragma unroll
        for (int a = 0; a < kTl; ++a) {
          u[a] = *reinterpret_cast<const float4*>(ra + a * cs + c4);
          v[a] = *reinterpret_cast<const float4*>(rb + a * cs + c4);
        }
#pragma unroll
        for (int a = 0; a < kTl; ++a)
#pragma unroll
          for (int b = 0; b < kTl; ++b) {
            float t = acc[q][a][b];
            t = fmaf(u[a].x, v[b].x, t);
            t = fmaf(u[a].y, v[b].y, t);
            t = fmaf(u[a].z, v[b].z, t);
            t = fmaf(u[a].w, v[b].w, t);
            acc[q][a][b] = t;
          }
      }
    }
    __syncthreads();  // the buffer is refilled by the next iteration's copy
  }
  // fold the column groups in a fixed order (the result does not depend on the schedule)
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int j = tid + q * kDsfpThreads;
    if (j < L.jobs)
#pragma unroll
      for (int a = 0; a < kTl; ++a)
#pragma unroll
        for (int b = 0; b < kTl; ++b) parts[(size_t)j * kTT + a * kTl + b] = acc[q][a][b];
  }
  __syncthreads();
  for (int e2 = tid; e2 < L.tp * kTT; e2 += kDsfpThreads) {
    const int pr = e2 / kTT, e = e2 % kTT;
    int a = 0, r = pr;
    while (r >= L.tiles - a) { r -= L.tiles - a; ++a; }
    const int b = a + r;
    float s = 0.f;
    for (int g = 0; g < L.groups; ++g) s += parts[((size_t)pr * L.groups + g) * kTT + e];
    const int u = a * kTl + e / kTl, v = b * kTl + e % kTl;
    G[u * mp + v] = s;
    G[v * mp + u] = s;
  }
  __syncthreads();

  dsfp_local<kDsfpThreads>(G, M, P, Y, nrm, deg, m, mp, gamma, T);
  dsfp_output<kDsfpThreads>(X, d, loc, deg, m, out + (size_t)i * d);
}

// Up to 32 local rows: NT tiles of R rows, one warp per tile pair (a <= b), R x R outputs per lane
// over the column pairs lane, lane + 32, ... of each chunk. The 3 x 3 form above reads 6 x 16 bytes
// of shared memory per 36 FMA and was bound by that pipe (its lanes also meet in the same banks);
// here a pair of columns costs 2R x 8 bytes per 2R^2 FMA (half of it on the diagonal), every read
// is a contiguous 256 bytes, and what remains is the gather of the rows through L2 (twice m x 4d
// bytes per image, 5.2 TB/s). 19,281 images of d = 2048, k = 20: 1.78 -> 1.27 ms. Three buffers,
// one barrier per chunk.
constexpr int kStagesT = 3;

__host__ __device__ constexpr int dsfp_tile_threads(int nt) { return 32 * (nt * (nt + 1) / 2); }
__host__ __device__ constexpr size_t dsfp_tile_bytes(int mp) {
  return sizeof(float) * ((size_t)kStagesT * mp * kCh + (size_t)4 * mp * mp + 2 * mp);
}

// Sums the 64 values of v over the warp, halving them at each step: lane l ends with the totals of
// values 2l and 2l + 1 in v[0] and v[1].
__device__ __forceinline__ void warp_sum_many(float (&v)[64], int lane) {
#pragma unroll
  for (int off = 16, h = 32; off > 0; off >>= 1, h >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (e < h) {
        const float send = up ? v[e] : v[e + h];
        const float keep = up ? v[e + h] : v[e];
        v[e] = keep + __shfl_xor_sync(GCR_FULL, send, off);
      }
  }
}

template <int R, int NT>
__global__ void __launch_bounds__(dsfp_tile_threads(NT), NT == 3 ? (R == 8 ? 3 : 4) : 2)
    dsfp_tile_kernel(const float* __restrict__ X, int n, int d, const int32_t* __restrict__ nbr, int k, float gamma,
                     int T, float* __restrict__ out) {
  constexpr int MP = R * NT, THREADS = dsfp_tile_threads(NT), NW = THREADS / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int loc[MP];
  __shared__ int s_m;
  float* buf = reinterpret_cast<float*>(smem);  // [kStagesT][MP][kCh]
  float* G = buf + kStagesT * MP * kCh;         // [MP][MP] each
  float* M = G + MP * MP;
  float* P = M + MP * MP;
  float* Y = P + MP * MP;
  float* nrm = Y + MP * MP;
  float* deg = nrm + MP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i = blockIdx.x;
  if (T == 0) {
    dsfp_copy_row(X, i, d, out, THREADS);
    return;
  }
  if (warp == 0) dsfp_nodes(nbr, i, k, loc, &s_m);
  __syncthreads();
  const int m = s_m;
  const int nch = (d + kCh - 1) / kCh;
  int ta = 0, tb = warp;
  while (tb >= NT - ta) { tb -= NT - ta; ++ta; }
  tb += ta;

  // a row per warp and step, a column quad per lane; rows past m and columns past d read as zero
  auto stage = [&](int ci) {
    const int c = ci * kCh + lane * 4;
    float* dst = buf + (ci % kStagesT) * (MP * kCh) + lane * 4;
    for (int r = warp; r < MP; r += NW) {
      const bool ok = r < m && c < d;
      cp_async16(dst + r * kCh, ok ? X + (size_t)loc[r] * d + c : X, ok);
    }
  };
  float acc[64];
#pragma unroll
  for (int e = 0; e < 64; ++e) acc[e] = 0.f;
  stage(0);
  cp_async_commit();
  if (nch > 1) stage(1);
  cp_async_commit();
  for (int ci = 0; ci < nch; ++ci) {
    cp_async_wait_prev();
    __syncthreads();  // chunk ci is here, and nobody reads chunk ci - 1 any more
    if (ci + 2 < nch) stage(ci + 2);
    cp_async_commit();
    const float* ra = buf + (ci % kStagesT) * (MP * kCh) + ta * R * kCh;
    const float* rb = buf + (ci % kStagesT) * (MP * kCh) + tb * R * kCh;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = h * 64 + lane * 2;
      float2 u[R];
#pragma unroll
      for (int a = 0; a < R; ++a) u[a] = *reinterpret_cast<const float2*>(ra + a * kCh + c);
      if (ta == tb) {
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
          for (int b = a; b < R; ++b) acc[a * R + b] = fmaf(u[a].y, u[b].y, fmaf(u[a].x, u[b].x, acc[a * R + b]));
      } else {
#pragma unroll
        for (int b = 0; b < R; ++b) {
          const float2 v = *reinterpret_cast<const float2*>(rb + b * kCh + c);
#pragma unroll
          for (int a = 0; a < R; ++a) acc[a * R + b] = fmaf(u[a].y, v.y, fmaf(u[a].x, v.x, acc[a * R + b]));
        }
      }
    }
  }
  warp_sum_many(acc, lane);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int e = 2 * lane + h;
    const int a = e / R, b = e % R;
    if (e < R * R && (ta != tb || a <= b)) {
      const int u = ta * R + a, v = tb * R + b;
      G[u * MP + v] = acc[h];
      G[v * MP + u] = acc[h];
    }
  }
  __syncthreads();
  dsfp_local<THREADS>(G, M, P, Y, nrm, deg, m, MP, gamma, T);
  dsfp_output<THREADS>(X, d, loc, deg, m, out + (size_t)i * d);
}

template <int R, int NT>
cudaError_t launch_tile(const float* X, int n, int d, const int32_t* nbr, int k, float gamma, int T, float* out,
                        cudaStream_t st) {
  const size_t bytes = dsfp_tile_bytes(R * NT);
  cudaError_t e = cudaFuncSetAttribute(dsfp_tile_kernel<R, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  dsfp_tile_kernel<R, NT><<<n, dsfp_tile_threads(NT), bytes, st>>>(X, n, d, nbr, k, gamma, T, out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dsfp(const float* X, int n, int d, const int32_t* nbr, int k, float gamma, int T, float* out,
                        cudaStream_t st) {
  if (n < 1 || k < 0 || k > kDsfpMaxK || d < 4 || d > kMaxD || d % 4 || T < 0) return cudaErrorInvalidValue;
  // tiles that pad the k + 1 rows least (19,281 images of d = 2048: k = 25 2.26 ms in tiles of 8, 1.94
  // in tiles of 7, 2.61 in 3 x 3 tiles; k = 32, in 3 x 3 tiles, 3.95)
  if (k < 12) return launch_tile<4, 3>(X, n, d, nbr, k, gamma, T, out, st);
  if (k < 18) return launch_tile<6, 3>(X, n, d, nbr, k, gamma, T, out, st);
  if (k < 21) return launch_tile<7, 3>(X, n, d, nbr, k, gamma, T, out, st);
  if (k < 24) return launch_tile<8, 3>(X, n, d, nbr, k, gamma, T, out, st);
  if (k < 28) return launch_tile<7, 4>(X, n, d, nbr, k, gamma, T, out, st);
  if (k < 32) return launch_tile<8, 4>(X, n, d, nbr, k, gamma, T, out, st);
  const DsfpLayout L = dsfp_layout(k + 1);
  if (L.jobs > 2 * kDsfpThreads) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(dsfp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.bytes);
  if (e != cudaSuccess) return e;
  dsfp_kernel<<<n, kDsfpThreads, L.bytes, st>>>(X, n, d, nbr, k, gamma, T, k + 1, out);
  return cudaGetLastError();
}

}  // namespace gcr
