// Similarity GEMM on the 5th-generation tensor cores (tcgen05), sm_103a.
//
// S = A . B^T with A, B row-major (K = d contiguous, "K-major"), BF16 or scaled FP16 rows or FP32
// rows rounded to TF32: A holds 128 rows of X, B 256 rows. Per CTA:
//   warp 0        TMA producer: 128-byte K blocks (64 16-bit or 32 TF32 elements) of A (128 rows)
//                 and B (256 rows) into a 2- to 4-stage shared-memory ring (128-byte
//                 swizzle; as many stages as the pools leave room for), mbarrier transaction
//                 counts;
//   warp 1        allocates 512 TMEM columns (two 128 x 256 FP32 accumulators) and, from one
//                 thread, issues tcgen05.mma (kind::f16 with K=16, or kind::tf32 with K=8;
//                 M=128, N=256) for each K block,
//                 committing stage releases and "accumulator full" to mbarriers;
//   warps 2..5    epilogue for the global graph, warps 6..9 for the cross-camera graph:
//                 tcgen05.ld.32x32b gives each thread one accumulator row (32 columns per
//                 load); the scores go into the streaming per-row pool (pool.cuh), or are
//                 appended to the band buffer, or written out as distances.
// The accumulator is double-buffered so the MMAs of column tile j+1 overlap the epilogue of
// tile j. Every mbarrier wait is bounded (2 s of %globaltimer); on a timeout the CTA raises a
// shared abort flag that every role polls, waits (bounded) for its in-flight MMAs, frees TMEM
// and returns; the timeout is counted in a device word that gcr_sync reports.
#include <algorithm>
#include <cmath>
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"
#include "pool.cuh"

namespace gcr {

__device__ int g_umma_timeouts;  // bounded waits that ran out since the last gcr_sync

namespace {

constexpr int BM = 128;            // rows of A per tile (UMMA M)
constexpr int BN = 256;            // rows of B per tile (UMMA N)
constexpr int BKB = 128;           // K bytes per stage (one swizzle row): 64 BF16 / 32 TF32
constexpr int NST_MAX = 4;         // pipeline stages where nothing else needs shared memory
constexpr int A_BYTES = BM * BKB;
constexpr int B_BYTES = BN * BKB;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr uint32_t TMEM_COLS = 512;
constexpr unsigned long long kTimeoutNs = 2000000000ull;

enum Mode { POOL = 0, BAND = 1, DIST = 2, GRAM = 3, MUL = 4, GPOOL = 5 };

// POOL runs on selection buffers, except cross-camera pools of 128 entries (two graphs' buffers
// of 160 slots would leave room for one stage only): those, and GPOOL, keep sorted lists.
template <int MODE, int KP, bool CROSS, bool DEEP>
struct Cfg {
  static constexpr bool kSel = MODE == POOL && !(KP == 128 && CROSS);
  static constexpr bool kPool = MODE == POOL || MODE == GPOOL;
  // ring stages: what the pools leave of the 227 KB
  static constexpr int kStages = !kPool ? NST_MAX
                                 : !kSel ? 3
                                 : KP == 32 ? (DEEP ? 4 : 3)
                                 : KP == 64 ? (CROSS ? 2 : 3)
                                            : 2;
};

// ------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false when the CTA is aborting (or this wait ran out and started the abort).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long limit_ns = kTimeoutNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63) == 0) {
      if (*abort_flag) return false;
      if (globaltimer() - t0 > limit_ns) {
        *abort_flag = 1;
        atomicAdd(&g_umma_timeouts, 1);
        return false;
      }
    }
  }
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major tile of rows of 128 bytes, 128-byte swizzle,
// 8-row core groups 1024 bytes apart (SBO), tile base 1024-byte aligned.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);          // start address
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset
  d |= (uint64_t)1 << 46;                          // descriptor version (sm_100 family)
  d |= (uint64_t)2 << 61;                          // layout: 128-byte swizzle
  return d;
}
// Instruction descriptors: D = F32 (bits 4-5 = 1), A and B formats (bits 7-9, 10-12: F16 = 0 and
// BF16 = 1 under kind::f16, TF32 = 2 under kind::tf32), both K-major, N >> 3 (bits 17-22), M >> 4
// (bits 24-28); N = 256, M = 128.
constexpr uint32_t kIdescShape = ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
constexpr uint32_t kIdescBf16 = (1u << 4) | (1u << 7) | (1u << 10) | kIdescShape;
constexpr uint32_t kIdescF16 = (1u << 4) | kIdescShape;
constexpr uint32_t kIdescTf32 = (1u << 4) | (2u << 7) | (2u << 10) | kIdescShape;

__device__ __forceinline__ void umma_16bit(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum));
}
__device__ __forceinline__ void umma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(kIdescTf32), "r"(accum));
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// Asynchronous TMEM load of 32 columns (one accumulator row per thread) ...
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// ... and the wait for it; the registers are passed through the wait so that no use of them
// can be scheduled before the load has landed.
__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  tmem_ld32_async(taddr, r);
  tmem_wait32(r);
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// ------------------------------------------------------------------------ kernel
struct UmmaArgs {
  int mode;
  int tf32;       // operands: 0 16-bit (kind::f16), 1 TF32 held as FP32 (kind::tf32)
  uint32_t idesc; // instruction descriptor of 16-bit operands
  int n;          // rows of B (columns of S)
  int d;
  int a_rows;     // rows of A (POOL: rows owning pools; DIST: nq; BAND: band capacity)
  int self_excl;  // skip column j == row i (A and B are the same matrix)
  int tps;        // POOL: column tiles per split
  const int* cam;
  // POOL
  float* pool_v;      // sorted lists [split][kind][part_rows][KP], or selection buffers
  int* pool_i;        //   [split][kind][part_rows][cap] with part_cnt entries each
  int* part_cnt;      // [split][kind][part_rows]
  int row0;           // the launch's rows of A: [row0, row0 + part_rows), row0 a multiple of BM
  int part_rows;
  // per row of A (stride seed_ld), or NULL: KP of the row's scores are at or above it, so every
  // split keeps only scores at or above it (-inf: no floor)
  const float* seed;
  int seed_ld;
  // BAND
  const int* count;
  int cap;
  const int* band_row;
  const int* band_kind;
  const float* band_thr;
  int bcap;
  int* band_cnt;
  float* band_v;       // may be NULL (indices only)
  int* band_i;
  const int* band_off; // NULL: row u writes at u * bcap; else at band_off[u]
  const int* band_lim; // NULL: bcap entries per row; else band_lim[u]
  // DIST
  const float* nrm_q;
  const float* nrm_g;
  float* D;
  // GRAM: G_s = Z_s Z_s^T + lambda n_s I per camera s = blockIdx.z, Z = the transposed,
  // normalised frames (feature rows, frame columns) split as hi + lo in BF16; K blocks of 64
  // frames [gram_kstart[s], + gram_knum[s]) give hi.hi, hi.lo and lo.hi each
  const int64_t* gram_kstart;
  const int64_t* gram_knum;
  const int64_t* gram_nf;  // n_s
  float gram_lambda;
  float* G;                // [ncam][d][d]
  // MUL: Q = P G_s for each 128-row block of P (camera s = mul_rowcam[block], < 0: skipped);
  // TF32 operands split hi + lo (hi.hi + hi.lo + lo.hi); G stacked as ncam * d rows of d
  const int* mul_rowcam;
  int dist_nrb;    // row tiles of the distance matrix
  int dist_tiles;  // all tiles; CTA b takes tiles b, b + grid, ... in column-major tile order,
                   // so the CTAs at work share the (small) query blocks and stream each gallery
                   // column tile once
  // GPOOL: pools of the rows of a gathered matrix against column ranges of the same matrix.
  // Work item w = {first row, rows (<= BM), first column, columns}; CTA b takes the items
  // b, b + grid, ... of the *n_items; a pool entry holds s - col_bias[j]; column j == row is
  // skipped when self_excl; cam (may be NULL) is indexed by gathered position.
  const int4* items;
  const int* n_items;
  const float* col_bias;
  // POOL: splits of one row block next to each other in the grid (grid.x = splits, grid.y = row
  // blocks): they run at the same time, and fewer row blocks are at work, whose A rows then stay
  // in L2. Otherwise grid.x = row blocks, so the first split of every block runs first.
  int split_first;
  // POOL with more than one split: per (kind, row) the order-preserving image of the best bound
  // any split has published (KP of the row's scores are strictly above it; 0: none yet). Every
  // split reads it before a tile and raises its own threshold to it.
  uint32_t* tau_x;
  Gate gate;       // POOL, BAND: whether this launch runs
};

struct __align__(8) Bars {
  uint64_t full[NST_MAX];
  uint64_t empty[NST_MAX];
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
};

// GPOOL walk over a CTA's work items and their column tiles: every role keeps its own cursor
// and advances it once per tile, so all roles see the same sequence.
struct ItemCursor {
  int item, ct, nt;
  int4 w;
  __device__ void load(const UmmaArgs& a, int nitems) {
    w = item < nitems ? a.items[item] : make_int4(0, 0, 0, 0);
    nt = (w.w + BN - 1) / BN;
  }
  __device__ void start(const UmmaArgs& a, int nitems) {
    item = blockIdx.x;
    ct = 0;
    load(a, nitems);
  }
  __device__ void advance(const UmmaArgs& a, int nitems) {
    if (++ct >= nt) {
      item += gridDim.x;
      ct = 0;
      load(a, nitems);
    }
  }
};

// Work list of a CTA: tiles (row block of A, column tile of B) in order.
template <int MODE>
struct Tiles {
  int count;
  int rb, split;  // POOL: row block and column split of this CTA
  __device__ int row0(const UmmaArgs& a, int t) const {
    if (MODE == POOL) return rb * BM;
    if (MODE == GRAM || MODE == MUL) return blockIdx.y * BM;
    if (MODE == BAND) return (blockIdx.y + t * gridDim.y) * BM;  // row tiles strided over grid.y
    return (((int)blockIdx.x + t * (int)gridDim.x) % a.dist_nrb) * BM;
  }
  __device__ int col0(const UmmaArgs& a, int t) const {
    if (MODE == POOL) return (split * a.tps + t) * BN;
    if (MODE == GRAM || MODE == MUL) return blockIdx.x * BN;
    if (MODE == BAND) return blockIdx.x * BN;
    return (((int)blockIdx.x + t * (int)gridDim.x) / a.dist_nrb) * BN;
  }
};

// Eligible scores of the tile above f (elig: a bit per column, all ones for most chunks).
__device__ __forceinline__ int tile_count(uint32_t taddr, int ncol, const uint32_t (&elig)[BN / 32], float f) {
  int cnt = 0;
#pragma unroll
  for (int ch = 0; ch < BN / 32; ++ch) {
    if (ch * 32 < ncol) {
      float v[32];
      tmem_ld32(taddr + ch * 32, v);
      if (__all_sync(GCR_FULL, elig[ch] == GCR_FULL)) {
#pragma unroll
        for (int c = 0; c < 32; ++c) cnt += v[c] > f ? 1 : 0;
      } else {
        uint32_t above = 0;
#pragma unroll
        for (int c = 0; c < 32; ++c) above |= (v[c] > f ? 1u : 0u) << c;
        cnt += __popc(above & elig[ch]);
      }
    }
  }
  return cnt;
}

// Upper quantile of the standard normal: z with P(Z > z) = q, to 3e-3 (Abramowitz and Stegun
// 26.2.22). Only used to guess thresholds that are then verified by counting.
__device__ __forceinline__ float normal_upper(float q) {
  const float u = fminf(fmaxf(fminf(q, 1.f - q), 1e-6f), 0.5f);
  const float t = sqrtf(-2.f * __logf(u));
  const float z = t - (2.30753f + 0.27061f * t) / (1.f + t * (0.99229f + 0.04481f * t));
  return q <= 0.5f ? z : -z;
}

// Admission floor of one row from the first column tile of its sweep. A pool starts empty, so
// without a floor every score of that tile would be buffered. A value f with at least KP of the
// tile's eligible scores above it is guessed from their mean and spread as if they were normal,
// verified by counting them in TMEM, and corrected by the count: the row's KP best scores of the
// whole sweep all lie above f, so scores at or below f can be dropped from the sweep. The counts
// use the same values and the same eligibility (column < n, not the row itself, another camera
// for the cross-camera pool) as the appends. -inf when the tile holds KP eligible scores or
// fewer. Most warps need two or three counts where a bisection takes six (800 rows of d = 128:
// 41,000 -> 25,000 cycles per CTA). All lanes run every step (the TMEM loads are warp-wide).
template <int KP, bool CAMCHK>
__device__ __noinline__ float warm_floor(uint32_t taddr, int cb0, int ncol, int n, int self_excl, int my_row,
                                         const int* __restrict__ cam, int my_cam, int lane) {
  uint32_t elig[BN / 32];
  float s1 = 0.f, s2 = 0.f, shift = 0.f, lo = CUDART_INF_F, hi = -CUDART_INF_F;
  int ne = 0;
#pragma unroll
  for (int ch = 0; ch < BN / 32; ++ch) {
    elig[ch] = 0u;
    if (ch * 32 < ncol) {
      float v[32];
      tmem_ld32(taddr + ch * 32, v);
      const int cb = cb0 + ch * 32;
      uint32_t e = cb + 32 <= n ? GCR_FULL : (1u << (n - cb)) - 1u;
      if (self_excl && my_row >= cb && my_row < cb + 32) e &= ~(1u << (my_row - cb));
      if (CAMCHK) {
        const int ccam = (cb + lane < n) ? cam[cb + lane] : -1;
        uint32_t same = 0;
#pragma unroll
        for (int c = 0; c < 32; ++c) same |= (__shfl_sync(GCR_FULL, ccam, c) == my_cam ? 1u : 0u) << c;
        e &= ~same;
      }
      elig[ch] = e;
      ne += __popc(e);
      if (ch == 0) shift = v[0];  // sums of v - shift: the spread can be far below the mean
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const bool ok = (e >> c) & 1u;
        const float x = v[c] - shift;
        s1 += ok ? x : 0.f;
        s2 += ok ? x * x : 0.f;
        lo = ok ? fminf(lo, v[c]) : lo;
        hi = ok ? fmaxf(hi, v[c]) : hi;
      }
    }
  }
  const bool active = ne > KP;
  const float inv = 1.f / (float)max(1, ne);
  const float mean = s1 * inv, sd = sqrtf(fmaxf(0.f, s2 * inv - mean * mean));
  const float goal = fminf(KP * 1.1f + 1.f, 0.5f * (float)(KP + ne));
  const float zg = normal_upper(goal * inv);
  float f = -CUDART_INF_F, x = mean + shift + zg * sd;
  bool more = active;
#pragma unroll 1
  for (int it = 0; it < 6 && __any_sync(GCR_FULL, more); ++it) {
    if (!(x > lo && x < hi)) x = 0.5f * lo + 0.5f * hi;
    const int c = tile_count(taddr, ncol, elig, x);
    if (more) {
      if (c >= KP) {
        f = lo = x;
        more = c > KP + KP / 4;
      } else {
        hi = x;
      }
      x += (zg - normal_upper((float)max(c, 1) * inv)) * sd;
    }
  }
  return f;
}

// MODE is a template parameter (not only a field of UmmaArgs) so that each mode's epilogue is
// compiled alone, without mode branches per value: when it was introduced, on pools of sorted lists,
// the similarity GEMM on crosscam went from 2.72 to 2.65 ms per TF32 launch and from 2.75 to 2.48 in
// BF16. One CTA per SM leaves room for the 128 to 196 registers a thread that the selection buffers
// take (they are compacted in registers); two graphs of 64 entries, at the 168 that 320 threads
// leave, spill 40 bytes.
template <int MODE, int KP, bool CROSS, bool DEEP = false>
__global__ void __launch_bounds__(CROSS ? 320 : 192, 1)
umma_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
            const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2, UmmaArgs a) {
  extern __shared__ __align__(1024) unsigned char dyn_raw[];
  // aligned by an offset from the shared array itself, so that every pointer derived from it
  // stays known as shared memory (queue appends compile to shared stores, not generic ones)
  unsigned char* dyn = dyn_raw + ((1024u - (smem_u32(dyn_raw) & 1023u)) & 1023u);
  constexpr int NS = Cfg<MODE, KP, CROSS, DEEP>::kStages;                   // ring stages
  unsigned char* stages = dyn;                                        // NS * STAGE_BYTES
  float2* qs = reinterpret_cast<float2*>(dyn + NS * STAGE_BYTES);    // [2][BM][kQCap] queues of the sorted lists
  constexpr bool SEL = Cfg<MODE, KP, CROSS, DEEP>::kSel;                    // selection buffers instead
  constexpr int CAP = SEL ? SelCap<KP, CROSS, DEEP>::cap : 1;
  constexpr int KINDS = CROSS ? 2 : 1;
  __shared__ Bars bars;

  if ((MODE == POOL || MODE == BAND) && gate_shut(a.gate)) return;  // (every CTA alike, before any barrier)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bk = a.tf32 ? BKB / 4 : BKB / 2;  // K elements per stage
  // K blocks per tile (GRAM, MUL: the hi operands' and the lo operands' of each block in turn)
  const int gram_kn = MODE == GRAM ? (int)a.gram_knum[blockIdx.z] : (a.d + bk - 1) / bk;
  const int kb_count = (MODE == GRAM || MODE == MUL) ? 2 * gram_kn : (a.d + bk - 1) / bk;
  // MUL: rows of camera s's G_s in the stacked G
  const int mul_b0 = MODE == MUL ? max(0, a.mul_rowcam[blockIdx.y]) * a.n : 0;

  Tiles<MODE> tl;
  tl.rb = ((MODE == POOL && a.split_first) ? (int)blockIdx.y : (int)blockIdx.x) + (MODE == POOL ? a.row0 / BM : 0);
  tl.split = (MODE == POOL && a.split_first) ? (int)blockIdx.x : (int)blockIdx.y;
  int nitems = 0;
  if (MODE == GPOOL) {
    nitems = *a.n_items;
    if ((int)blockIdx.x >= nitems) return;  // nothing to do: leave before any barrier or TMEM use
    tl.count = 0;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) tl.count += (a.items[it].w + BN - 1) / BN;
  } else if (MODE == POOL) tl.count = max(0, min(a.tps, (a.n + BN - 1) / BN - tl.split * a.tps));
  else if (MODE == BAND) {
    const int U = min(*a.count, a.cap);
    const int tiles = (U + BM - 1) / BM;
    tl.count = max(0, (tiles - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y);
    if (tl.count == 0) return;  // no rows for this CTA: leave before any barrier or TMEM use
  } else if (MODE == GRAM) {
    // G_s is symmetric: tiles wholly below the diagonal (every column < every row) are mirrored
    tl.count = ((int)blockIdx.x + 1) * BN <= (int)blockIdx.y * BM ? 0 : 1;
  } else if (MODE == MUL) {
    tl.count = a.mul_rowcam[blockIdx.y] >= 0 ? 1 : 0;
  } else {
    tl.count = max(0, (a.dist_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x);
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&bars.full[s], 1);
      mbar_init(&bars.empty[s], 1);
    }
    const int epi_warps = CROSS ? 8 : 4;
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars.tfull[b], 1);
      mbar_init(&bars.tempty[b], epi_warps);
    }
    mbar_init(&bars.drain, 1);
    bars.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars.tmem_base)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_base;
  volatile int* abort_flag = &bars.abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int it = 0;
      ItemCursor cur;
      if (MODE == GPOOL) cur.start(a, nitems);
      for (int t = 0; t < tl.count && !*abort_flag; ++t) {
        const int r0 = MODE == GPOOL ? cur.w.x : tl.row0(a, t);
        const int c0 = MODE == GPOOL ? cur.w.z + cur.ct * BN : tl.col0(a, t);
        if (MODE == GPOOL) cur.advance(a, nitems);
        for (int kb = 0; kb < kb_count; ++kb, ++it) {
          const int s = it % NS;
          const uint32_t round = it / NS;
          if (!mbar_wait(&bars.empty[s], (round & 1) ^ 1, abort_flag)) break;
          unsigned char* sa = stages + s * STAGE_BYTES;
          mbar_arrive_expect_tx(&bars.full[s], STAGE_BYTES);
          if (MODE == GRAM || MODE == MUL) {
            // even K blocks: the hi operands, odd ones: the lo operands of the same elements
            const int x = MODE == GRAM ? (int)((a.gram_kstart[blockIdx.z] + (kb >> 1)) * bk) : (kb >> 1) * bk;
            tma_load_2d(sa, (kb & 1) ? &tmA2 : &tmA, &bars.full[s], x, r0);
            tma_load_2d(sa + A_BYTES, (kb & 1) ? &tmB2 : &tmB, &bars.full[s], x, mul_b0 + c0);
          } else {
            tma_load_2d(sa, &tmA, &bars.full[s], kb * bk, r0);
            tma_load_2d(sa + A_BYTES, &tmB, &bars.full[s], kb * bk, c0);
          }
        }
      }
      // in-flight loads land before the CTA can exit: wait for the last armed stages
      if (*abort_flag) {
        for (int back = 1; back <= NS && back <= it; ++back) {
          const int j = it - back;
          const unsigned long long t0 = globaltimer();
          while (!mbar_try_wait(&bars.full[j % NS], (j / NS) & 1) && globaltimer() - t0 < kTimeoutNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = 0; t < tl.count && ok; ++t) {
        const int buf = t & 1;
        const uint32_t use = t >> 1;
        if (!mbar_wait(&bars.tempty[buf], (use & 1) ^ 1, abort_flag)) break;
        tc_fence_after();
        const uint32_t dcol = tmem + buf * BN;
        for (int kb = 0; kb < kb_count; ++kb, ++it) {
          const int s = it % NS;
          if (!mbar_wait(&bars.full[s], (it / NS) & 1, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(stages + s * STAGE_BYTES);
          const uint64_t ad = smem_desc(sa), bd = smem_desc(sa + A_BYTES);
          // four MMAs per stage, +32 bytes (16 16-bit elements or K=8 TF32) inside the swizzle row
          auto mma4 = [&](uint64_t da, uint64_t db, bool accum) {
            if (a.tf32) {
#pragma unroll
              for (int k = 0; k < 4; ++k) umma_tf32(dcol, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), accum || k);
            } else {
#pragma unroll
              for (int k = 0; k < 4; ++k)
                umma_16bit(dcol, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), a.idesc, accum || k);
            }
          };
          if (MODE == GRAM || MODE == MUL) {
            // hi.hi as soon as the hi operands have landed; hi.lo and lo.hi with the lo ones, after
            // which both stages are free: two operand loads per three products
            static_assert(!(MODE == GRAM || MODE == MUL) || NS % 2 == 0, "hi and lo stages in pairs");
            if (!(kb & 1)) {
              mma4(ad, bd, kb != 0);
              continue;
            }
            const uint32_t sh = smem_u32(stages + (s - 1) * STAGE_BYTES);
            mma4(smem_desc(sh), bd, true);
            mma4(ad, smem_desc(sh + A_BYTES), true);
            umma_commit(&bars.empty[s - 1]);
            umma_commit(&bars.empty[s]);
            continue;
          }
          mma4(ad, bd, kb != 0);
          umma_commit(&bars.empty[s]);
        }
        if (ok) umma_commit(&bars.tfull[buf]);
      }
      // all issued MMAs complete before TMEM is released
      umma_commit(&bars.drain);
      const unsigned long long t0 = globaltimer();
      while (!mbar_try_wait(&bars.drain, 0) && globaltimer() - t0 < kTimeoutNs) {
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps
    const int ew = warp - 2;                 // 0..7
    const int kind = ew >> 2;                // 0: global graph, 1: cross-camera graph
    const int quad = warp & 3;               // TMEM lanes 32*quad .. 32*quad+31
    const int r = quad * 32 + lane;          // row of the accumulator owned by this thread
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    PoolOwner me;
    int my_row = -1, my_cam = 0;
    float my_thr = 0.f, my_nq = 0.f;
    int my_kind = 0;
    const int qrow = kind * BM + r;
    const int sw = qrow & 31;
    // selection buffers: scores [kind][slot][row], then column offsets
    const uint32_t sva0 = smem_u32(dyn + NS * STAGE_BYTES) + (uint32_t)((kind * CAP * BM + r) * sizeof(float));
    const uint32_t sia0 = smem_u32(dyn + NS * STAGE_BYTES) + (uint32_t)(KINDS * CAP * BM * sizeof(float)) +
                         (uint32_t)((kind * CAP * BM + r) * sizeof(uint16_t));
    uint32_t sva = sva0, sia = sia0;                       // the next free slot
    const uint32_t sva_end = sva0 + (CAP - 4) * kSelV;     // past it a group of four may not fit
    float ssum = 0.f;                                      // sum of the buffered scores
    float pub = -CUDART_INF_F, pub_sent = -CUDART_INF_F;  // bound for the other splits
    const bool idle = SEL && tl.rb * BM + quad * 32 >= a.a_rows;  // no row of this warp exists
    // of the launch's rows, indexed by the row of A
    const ptrdiff_t part0 = (ptrdiff_t)((MODE == POOL ? tl.split : 0) * KINDS + kind) * a.part_rows - a.row0;
    float* pv = a.pool_v ? a.pool_v + part0 * (SEL ? CAP : KP) : nullptr;
    int* pi = a.pool_i ? a.pool_i + part0 * (SEL ? CAP : KP) : nullptr;
    if (MODE == POOL) {
      my_row = tl.rb * BM + r;
      const bool valid = my_row < a.a_rows;
      float floor = -CUDART_INF_F;
      if (valid && a.seed) floor = a.seed[(size_t)my_row * a.seed_ld];
      // strictly above the value below the floor
      pool_init(me, valid, floor > -CUDART_INF_F ? float_below(floor) : floor);
      if (CROSS && valid) my_cam = a.cam[my_row];
    }
    ItemCursor cur;
    if (MODE == GPOOL) cur.start(a, nitems);
    bool g_valid = false;        // GPOOL: this thread's row belongs to the current item
    int g_row0 = 0, g_cend = 0;  // GPOOL: first row of the item, end of its columns
    uint32_t* const tx = (SEL && a.tau_x && my_row >= 0 && my_row < a.a_rows) ? a.tau_x + (size_t)kind * a.a_rows + my_row : nullptr;
    for (int t = 0; t < tl.count; ++t) {
      const int buf = t & 1;
      const uint32_t use = t >> 1;
      const uint32_t tau_other = tx ? __ldcg(tx) : 0u;
      // the lanes stay together: one may find the tile ready while another finds the CTA aborting, and
      // what follows (TMEM loads, votes, merges) needs the whole warp
      if (!__all_sync(GCR_FULL, mbar_wait(&bars.tfull[buf], use & 1, abort_flag))) break;
      tc_fence_after();
      const int r0 = MODE == GPOOL ? cur.w.x : tl.row0(a, t);
      const int c0 = MODE == GPOOL ? cur.w.z + cur.ct * BN : tl.col0(a, t);
      const bool g_first = MODE == GPOOL && cur.ct == 0;
      const bool g_last = MODE == GPOOL && cur.ct == cur.nt - 1;
      if (g_first) {
        g_row0 = cur.w.x;
        g_cend = cur.w.z + cur.w.w;
        g_valid = r < cur.w.y;
        my_row = g_row0 + r;
        pool_init(me, g_valid);
        if (CROSS && g_valid) my_cam = a.cam[my_row];
      }
      if (MODE == GPOOL) cur.advance(a, nitems);
      int u = -1;
      if (MODE == BAND) {
        u = r0 + r;
        const int U = min(*a.count, a.cap);
        if (u < U) {
          my_row = a.band_row[u];
          my_kind = a.band_kind[u];
          my_thr = a.band_thr[u];
          if (a.cam) my_cam = a.cam[my_row];
        } else {
          u = -1;
        }
      } else if (MODE == DIST) {
        my_row = r0 + r;
        my_nq = my_row < a.a_rows ? a.nrm_q[my_row] : 0.f;
      } else if (MODE == MUL) {
        my_row = r0 + r;
      } else if (MODE == GRAM) {
        my_row = r0 + r;
        my_nq = a.gram_lambda * (float)a.gram_nf[blockIdx.z];  // lambda n_s, added on the diagonal
      }
      const int cend = MODE == GPOOL ? g_cend : a.n;  // end of this tile's valid columns
      const int ncol = min(BN, cend - c0);
      if (MODE == POOL && t == 0 && !idle) {
        const uint32_t ta = tmem + lane_addr + buf * BN;
        const float f = (CROSS && kind == 1)
                            ? warm_floor<KP, true>(ta, c0, ncol, a.n, a.self_excl, my_row, a.cam, my_cam, lane)
                            : warm_floor<KP, false>(ta, c0, ncol, a.n, a.self_excl, my_row, a.cam, my_cam, lane);
        me.floor = fmaxf(me.floor, f);
        me.tau = fmaxf(me.tau, f);
        if (my_row < a.a_rows) pub = f;
      }
      if (tau_other) me.tau = fmaxf(me.tau, ordered_to_float(tau_other));
      // cross-camera pools: the column cameras of chunk ch + 1 are loaded while chunk ch is
      // processed, so one load latency per tile is exposed instead of one per chunk
      int cam_next = 0;
      if (MODE == POOL && CROSS && kind == 1) cam_next = (c0 + lane < a.n) ? a.cam[c0 + lane] : -1;
      for (int ch = 0; ch < BN / 32; ++ch) {
        if (ch * 32 >= ncol || idle) break;
        float v[32];
        tmem_ld32(tmem + lane_addr + buf * BN + ch * 32, v);
        const int cb = c0 + ch * 32;
        int cam_cur = 0;
        if (MODE == POOL && CROSS && kind == 1) {
          cam_cur = cam_next;
          if ((ch + 1) * 32 < ncol) cam_next = (cb + 32 + lane < a.n) ? a.cam[cb + 32 + lane] : -1;
        }
        if (MODE == GPOOL) {
          if (kind == 0 || CROSS) {
            int ccam = 0;
            if (CROSS && kind == 1) ccam = (cb + lane < cend) ? a.cam[cb + lane] : -1;
            const float hb = (cb + lane < cend) ? a.col_bias[cb + lane] : 0.f;
            float2* myq = qs + qrow * kQCap;
#pragma unroll
            for (int c = 0; c < 32; ++c) v[c] -= __shfl_sync(GCR_FULL, hb, c);  // biased scores
            const int r0w = g_row0 + quad * 32;  // first row of this warp (rows are not 32-aligned)
            if (cb + 32 > cend || (a.self_excl && cb < r0w + 32 && cb + 32 > r0w)) {
#pragma unroll
              for (int c = 0; c < 32; ++c)
                if (cb + c >= cend || (a.self_excl && cb + c == my_row)) v[c] = -CUDART_INF_F;
            }
            // four values at a time, as in the POOL mode
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const float m4 = fmaxf(fmaxf(v[4 * g], v[4 * g + 1]), fmaxf(v[4 * g + 2], v[4 * g + 3]));
              if (__any_sync(GCR_FULL, m4 > me.tau)) {
                pool_make_room<KP>(4, lane, me, r0w, kind * BM + quad * 32, qs, pv, pi);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  const int cc = g * 4 + c;
                  const int cj = (CROSS && kind == 1) ? __shfl_sync(GCR_FULL, ccam, cc) : 0;
                  const bool eligible = !(CROSS && kind == 1) || cj != my_cam;
                  if (eligible && v[cc] > me.tau) {
                    myq[me.qcnt ^ sw] = make_float2(v[cc], __int_as_float(cb + cc));
                    ++me.qcnt;
                  }
                }
              }
            }
          }
        } else if (MODE == POOL) {
          // Most groups of four scores fall below every row's threshold (floors from the first
          // tile and from the other splits; thresholds only rise): one vote over the warp skips
          // them. The chunk on the warp's diagonal (each row meets itself) and the ragged last
          // chunk first get their excluded columns set to -inf; the global pool's warps compare
          // against a camera no column has.
          const int r0w = tl.rb * BM + quad * 32;  // first row of this warp
          if (cb + 32 > a.n || (a.self_excl && cb == r0w)) {
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (cb + c >= a.n || (a.self_excl && cb + c == my_row)) v[c] = -CUDART_INF_F;
          }
          const int ccam = (CROSS && kind == 1) ? cam_cur : 0;
          const int cmp_cam = (CROSS && kind == 1) ? my_cam : -2;
          const int off0 = cb - tl.split * a.tps * BN;  // 16-bit column offset of the chunk
          float2* myq = qs + qrow * kQCap;
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const float m4 = fmaxf(fmaxf(v[4 * g], v[4 * g + 1]), fmaxf(v[4 * g + 2], v[4 * g + 3]));
            if (!__any_sync(GCR_FULL, m4 > me.tau)) continue;
            if constexpr (SEL) {
              if (__any_sync(GCR_FULL, sva > sva_end)) {
                const SelState ss = sel_compact<KP, CAP>(
                    sva0, sia0, SelState{me.tau, me.floor, pub, ssum, (int)((sva - sva0) / kSelV)});
                me.tau = ss.tau;
                me.floor = ss.lo;
                sva = sva0 + ss.cnt * kSelV;
                sia = sia0 + ss.cnt * kSelI;
                pub = ss.pub;
                ssum = ss.sum;
              }
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const int cc = g * 4 + c;
                const int cj = CROSS ? __shfl_sync(GCR_FULL, ccam, cc) : 0;
                if (cj != cmp_cam && v[cc] > me.tau) {
                  sel_st(sva, sia, v[cc], off0 + cc);
                  sva += kSelV;
                  sia += kSelI;
                  ssum += v[cc];
                }
              }
            } else {
              pool_make_room<KP>(4, lane, me, r0w, kind * BM + quad * 32, qs, pv, pi);
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const int cc = g * 4 + c;
                const int cj = CROSS ? __shfl_sync(GCR_FULL, ccam, cc) : 0;
                if (cj != cmp_cam && v[cc] > me.tau) {
                  myq[me.qcnt ^ sw] = make_float2(v[cc], __int_as_float(cb + cc));
                  ++me.qcnt;
                }
              }
            }
          }
        } else if (MODE == BAND) {
          if (kind == 0) {
            int ccam = 0;
            if (a.cam) ccam = (cb + lane < a.n) ? a.cam[cb + lane] : -1;
            // the chunk's hits first, then one atomic for all of them: an atomic per hit waits for
            // each in turn, and the lanes' rows meet their columns apart
            uint32_t hit = 0u;
#pragma unroll
            for (int cc = 0; cc < 32; ++cc) {
              const int j = cb + cc;
              const int cjv = __shfl_sync(GCR_FULL, ccam, cc);
              const int cj = a.cam ? cjv : 0;
              if (u < 0 || j >= a.n || (a.self_excl && j == my_row) || v[cc] < my_thr) continue;
              if (my_kind == 1 && cj == my_cam) continue;
              hit |= 1u << cc;
            }
            if (hit) {
              const int lim = a.band_lim ? a.band_lim[u] : a.bcap;
              int pos = atomicAdd(&a.band_cnt[u], __popc(hit));
              const size_t base = a.band_off ? (size_t)a.band_off[u] : (size_t)u * a.bcap;
              if (pos >= lim) {
                if (a.band_v) my_thr = CUDART_INF_F;  // past the band: what more there is need not be counted
              } else {
#pragma unroll
                for (int cc = 0; cc < 32; ++cc)
                  if ((hit >> cc) & 1u) {
                    if (pos < lim) {
                      if (a.band_v) a.band_v[base + pos] = v[cc];
                      a.band_i[base + pos] = cb + cc;
                    }
                    ++pos;
                  }
              }
            }
          }
        } else if (MODE == MUL) {
          if (kind == 0 && my_row < a.a_rows) {
            float* out = a.D + (size_t)my_row * a.n + cb;
#pragma unroll
            for (int cc = 0; cc < 32; ++cc)
              if (cb + cc < a.n) out[cc] = v[cc];
          }
        } else if (MODE == GRAM) {
          if (kind == 0 && my_row < a.a_rows) {
            float* out = a.G + ((size_t)blockIdx.z * a.a_rows + my_row) * a.n + cb;
            const bool none = gram_kn == 0;  // a camera without frames: no MMA wrote the accumulator
#pragma unroll
            for (int cc = 0; cc < 32; ++cc)
              if (cb + cc < a.n) out[cc] = (none ? 0.f : v[cc]) + (cb + cc == my_row ? my_nq : 0.f);
          }
        } else {
          if (kind == 0) {
            const float ngv = (cb + lane < a.n) ? a.nrm_g[cb + lane] : 0.f;
            const bool row_ok = my_row < a.a_rows;
            float* out = a.D + (size_t)(row_ok ? my_row : 0) * a.n + cb;
#pragma unroll
            for (int cc = 0; cc < 32; ++cc) {
              const float g = __shfl_sync(GCR_FULL, ngv, cc);
              if (row_ok && cb + cc < a.n) out[cc] = my_nq + g - 2.f * v[cc];
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars.tempty[buf]);
      if (tx && pub > pub_sent) {
        atomicMax(tx, float_to_ordered(pub));
        pub_sent = pub;
      }
      if (g_last && (kind == 0 || CROSS))
        pool_flush<KP>(lane, g_valid, me, g_row0 + quad * 32, kind * BM + quad * 32, qs, pv, pi);
    }
    // After a wait that ran out too: every count and list of the launch is written (with what was
    // swept), so that what reads them stays within them; gcr_sync reports the timeout.
    if (MODE == GPOOL && (kind == 0 || CROSS)) {
      for (; cur.item < nitems; cur.item += gridDim.x, cur.load(a, nitems)) {  // items not finished: empty lists
        if (r >= cur.w.y) continue;
        for (int e = 0; e < KP; ++e) {
          pv[(size_t)(cur.w.x + r) * KP + e] = -CUDART_INF_F;
          pi[(size_t)(cur.w.x + r) * KP + e] = -1;
        }
      }
    }
    if (MODE == POOL) {
      if constexpr (SEL) {
        if (my_row < a.a_rows) {
          const int col0 = tl.split * a.tps * BN;
          const int cnt = (int)((sva - sva0) / kSelV);
          a.part_cnt[part0 + my_row] = cnt;
          float4* ov = reinterpret_cast<float4*>(pv + (size_t)my_row * CAP);
          int4* oi = reinterpret_cast<int4*>(pi + (size_t)my_row * CAP);
          for (int s = 0; s < cnt; s += 4) {  // (slots past the count: never read)
            const uint32_t va = sva0 + s * kSelV, ia = sia0 + s * kSelI;
            ov[s >> 2] = make_float4(sel_ldv(va), sel_ldv(va + kSelV), sel_ldv(va + 2 * kSelV), sel_ldv(va + 3 * kSelV));
            oi[s >> 2] = make_int4(col0 + (int)sel_ldi(ia), col0 + (int)sel_ldi(ia + kSelI),
                                   col0 + (int)sel_ldi(ia + 2 * kSelI), col0 + (int)sel_ldi(ia + 3 * kSelI));
          }
        }
      } else {
        pool_flush<KP>(lane, my_row < a.a_rows, me, tl.rb * BM + quad * 32, kind * BM + quad * 32, qs, pv, pi);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

// Self-test of the bounded wait: one warp waits on an mbarrier that nothing signals; the wait
// gives up after limit_ns, counts a timeout (reported by gcr_sync) and the kernel returns.
__global__ void wait_probe_kernel(unsigned long long limit_ns, int* result) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait(&bar, 0, &abort_flag, limit_ns);
  __syncthreads();
  if (threadIdx.x == 0 && result) *result = ok ? 1 : 0;
}

// ------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Row-major matrix [rows][d] (BF16, or TF32 held as FP32) viewed as a 2-D tensor, box = 128
// bytes of K x box_rows; K past d reads as zero. step: every step-th row of the matrix.
cudaError_t make_map(CUtensorMap* m, const void* base, Elt elt, int rows, int d, int box_rows, int step = 1) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const size_t es = elt_bytes(elt);
  if ((reinterpret_cast<uintptr_t>(base) & 15) || ((size_t)d * es) % 16) return cudaErrorInvalidValue;
  cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)step * d * es};
  cuuint32_t box[2] = {(cuuint32_t)(BKB / es), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m,
                  elt == Elt::TF32  ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                  : elt == Elt::F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                    : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                  const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int MODE, int KP, bool CROSS, bool DEEP>
constexpr size_t smem_bytes() {
  using C = Cfg<MODE, KP, CROSS, DEEP>;
  size_t s = 1024 + (size_t)C::kStages * STAGE_BYTES;
  if constexpr (C::kSel)
    s += (size_t)(CROSS ? 2 : 1) * SelCap<KP, CROSS, DEEP>::cap * BM * (sizeof(float) + sizeof(uint16_t));
  else if (C::kPool)
    s += 2 * BM * kQCap * (sizeof(float) + sizeof(int));
  return s;
}

template <int MODE, int KP, bool CROSS, bool DEEP = false>
cudaError_t launch(const CUtensorMap& ta, const CUtensorMap& tb, const UmmaArgs& a, dim3 grid, cudaStream_t st,
                   const CUtensorMap* ta2 = nullptr, const CUtensorMap* tb2 = nullptr) {
  auto fn = umma_kernel<MODE, KP, CROSS, DEEP>;
  constexpr size_t smem = smem_bytes<MODE, KP, CROSS, DEEP>();
  static_assert(smem + sizeof(Bars) <= 232448, "shared memory of a CTA");
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fn<<<grid, CROSS ? 320 : 192, smem, st>>>(ta, tb, ta2 ? *ta2 : ta, tb2 ? *tb2 : tb, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_wait_probe(unsigned long long limit_ns, cudaStream_t st) {
  wait_probe_kernel<<<1, 32, 0, st>>>(limit_ns, nullptr);
  return cudaGetLastError();
}

int umma_read_and_clear_timeouts() {
  int h = 0, z = 0;
  if (cudaMemcpyFromSymbol(&h, g_umma_timeouts, sizeof(int)) != cudaSuccess) return -1;
  if (h) cudaMemcpyToSymbol(g_umma_timeouts, &z, sizeof(int));
  return h;
}

// A sweep's time in units of a column tile, per CTA: its tiles and the set-up, first-tile floor
// and write-out around them (about 12 us against d / 64 * 0.25 us per tile, at least 0.8).
// The 16-bit column offsets force a split per 65,536 columns, and the buffers of all splits of a row
// wait for its pool: kept for all rows at once they grow with n^2 (4,000,000 rows of d = 64, 62
// splits: 190 GB, where everything else takes 28). So the rows are swept in chunks whose buffers
// share kPartBytes, which still hold 2,000 CTAs and more. 201,000 rows of d = 512 with four splits
// of 64-entry pools (617 MB, three chunks), the whole three-layer call: 221.2 ms at once, 221.5 so.
constexpr long kPartBytes = 256l << 20;
int pool_sweep_rows(const PoolPlan& p, int na, bool cross) {
  const long per_row = 8l * std::max(p.splits, p.sample_splits) * (cross ? 2 : 1) * p.cap;
  const long most = std::max<long>(BM, kPartBytes / per_row / BM * BM);
  if (na <= most) return na;
  const long chunks = (na + most - 1) / most, rows = (na + chunks - 1) / chunks;
  return (int)((rows + BM - 1) / BM * BM);
}

PoolPlan pool_plan(int na, int nb, int d, Elt elt, int kp, bool cross, int max_splits) {
  PoolPlan p;
  p.sel = !(kp == 128 && cross);
  // eight K blocks or fewer per tile: a three-stage ring covers them
  p.deep = kp == 32 && !cross && d * elt_bytes(elt) > 8 * BKB;
  p.cap = !p.sel ? kp : kp == 32 ? (cross ? SelCap<32, true>::cap : p.deep ? SelCap<32, false, true>::cap : SelCap<32, false>::cap)
                      : kp == 64 ? (cross ? SelCap<64, true>::cap : SelCap<64, false>::cap)
                                 : SelCap<128, false>::cap;
  const int ntiles = (nb + BN - 1) / BN, rblocks = (na + BM - 1) / BM;
  const double tile_us = std::max(0.8, d * (double)elt_bytes(elt) / 128.0 * 0.25);
  const double around = 12.0 / tile_us;
  auto tps_of = [&](int s) { return (ntiles + s - 1) / s; };
  int best = 1;
  double best_t = 1e300;
  for (int s = 1; s <= std::min(std::min(ntiles, kSMs), max_splits); ++s) {
    const int tps = tps_of(s);
    if (s > 1 && (long)rblocks * (s - 1) > 16 * kSMs) break;  // past 16 waves nothing is left to even out
    if (p.sel && (long)tps * BN > kSelMaxCols) continue;  // 16-bit column offsets
    const int used = (ntiles + tps - 1) / tps;
    const double waves = std::ceil((double)rblocks * used / kSMs);
    const double t = waves * (tps + around);
    if (t < best_t * 0.999) {
      best_t = t;
      best = s;
    }
  }
  // more splits than SMs only for the 16-bit offsets (over kSelMaxCols columns per SM)
  if (p.sel)
    while ((long)tps_of(best) * BN > kSelMaxCols) ++best;
  // Where one A block per SM would not fit in half the L2 (151 blocks of 128 x 2048 TF32 rows:
  // 151 MB, re-read for every column tile), two CTAs sweep the halves of each block at the same
  // time, so half as many blocks are at work.
  const double live_a = (double)std::min(rblocks, kSMs) * BM * d * (double)elt_bytes(elt);
  p.split_first = false;
  if (best == 1 && std::min(ntiles, max_splits) >= 2 && live_a > 0.5 * kL2Bytes) {
    best = 2;
    p.split_first = true;
  }
  p.tps = tps_of(best);
  p.splits = (ntiles + p.tps - 1) / p.tps;  // no split is left without a column tile
  // Many splits over long ranges (few rows against many columns): each split alone would admit
  // about kp (1 + ln(its columns / kp)) scores a row. A sweep of an evenly spaced sample of the
  // columns first bounds every row at about the (kp / share)-th best of all its scores, which
  // leaves a split a handful: no compactions, and little for pool_finish to read. Sample tiles
  // from 1/16 of the columns, 16 to 64 of them. Three searches of 512 queries over 500,000 rows
  // of d = 256: 2.2 ms with floors from 4,096 rows re-scored per query in FP32 (0.85 of them for
  // the floors), 2.3 without floors, 1.42 so; of 37 queries over 50,000 rows 0.48 -> 0.38.
  p.sample_tiles = 0;
  if (p.sel && !cross && p.splits >= 8 && p.tps >= 4) p.sample_tiles = std::max(16, std::min(64, ntiles / 16));
  if (p.sample_tiles * 2 > ntiles) p.sample_tiles = 0;
  p.sample_splits = 0;
  if (p.sample_tiles) {  // about one sample tile per CTA
    const int tps = std::max((int)(((long)p.sample_tiles * rblocks + kSMs - 1) / kSMs),
                             1 + (p.sample_tiles - 1) / max_splits);
    p.sample_splits = (p.sample_tiles + tps - 1) / tps;
  }
  p.rows = pool_sweep_rows(p, na, cross);
  return p;
}

size_t pool_part_rows(const PoolPlan& p, int na, bool cross) {
  return (size_t)std::max(p.splits, p.sample_splits) * (cross ? 2 : 1) * std::min(na, p.rows);
}

template <typename... T>
static cudaError_t launch_pool_sweep(int kp, bool cross, bool deep, T&&... t) {
  if (kp == 32)
    return cross  ? launch<POOL, 32, true>(t...)
           : deep ? launch<POOL, 32, false, true>(t...)
                  : launch<POOL, 32, false>(t...);
  if (kp == 64) return cross ? launch<POOL, 64, true>(t...) : launch<POOL, 64, false>(t...);
  if (kp == 128) return cross ? launch<POOL, 128, true>(t...) : launch<POOL, 128, false>(t...);
  return cudaErrorInvalidValue;
}

cudaError_t launch_umma_pool(const void* Ab, int na, const void* Bb, int nb, int d, Elt elt,
                             const int* cam, bool cross, int self_excl, int kp, const PoolParts& parts,
                             float* pool_v, int* pool_i, cudaStream_t st, Gate gate, int a_step) {
  CUtensorMap ta, tb, sb;
  cudaError_t e = make_map(&ta, Ab, elt, na, d, BM, a_step);
  if (e != cudaSuccess) return e;
  e = make_map(&tb, Bb, elt, nb, d, BN);
  if (e != cudaSuccess) return e;
  const PoolPlan& p = parts.plan;
  const int kinds = cross ? 2 : 1;
  UmmaArgs a{};
  a.mode = POOL;
  a.tf32 = elt == Elt::TF32;
  a.idesc = elt == Elt::F16 ? kIdescF16 : kIdescBf16;
  a.n = nb;
  a.d = d;
  a.a_rows = na;
  a.self_excl = self_excl;
  a.tps = p.tps;
  a.cam = cam;
  a.pool_v = parts.v;
  a.pool_i = parts.i;
  a.part_cnt = parts.cnt;
  a.split_first = p.split_first;
  a.gate = gate;
  // every step-th row; the sample's pools end in pool_v, whose last entries are the floors
  const bool sample = p.sample_tiles && !self_excl;
  UmmaArgs sa = a;
  if (sample) {
    sa.n = p.sample_tiles * BN;
    sa.split_first = 0;
    sa.tps = (p.sample_tiles + p.sample_splits - 1) / p.sample_splits;
    e = make_map(&sb, Bb, elt, sa.n, d, BN, nb / sa.n);
    if (e != cudaSuccess) return e;
    a.seed = pool_v + kp - 1;
    a.seed_ld = kp;
  }
  if (p.sel && p.splits > 1) {
    a.tau_x = parts.tau;
    e = cudaMemsetAsync(parts.tau, 0, sizeof(uint32_t) * kinds * (size_t)na, st);
    if (e != cudaSuccess) return e;
  }
  for (int r0 = 0; r0 < na; r0 += p.rows) {
    const int rows = std::min(p.rows, na - r0), rblocks = (rows + BM - 1) / BM;
    a.row0 = sa.row0 = r0;
    a.part_rows = sa.part_rows = rows;
    if (sample) {
      e = launch_pool_sweep(kp, false, p.deep, ta, sb, sa, dim3(rblocks, p.sample_splits), st);
      if (e == cudaSuccess)
        e = launch_pool_finish(parts.v, parts.i, parts.cnt, p.sample_splits, 1, rows, p.cap, kp, pool_v, pool_i, na, r0,
                               st, gate);
      if (e != cudaSuccess) return e;
    }
    e = launch_pool_sweep(kp, cross, p.deep, ta, tb, a, p.split_first ? dim3(p.splits, rblocks) : dim3(rblocks, p.splits),
                          st);
    if (e != cudaSuccess) return e;
    e = p.sel ? launch_pool_finish(parts.v, parts.i, parts.cnt, p.splits, kinds, rows, p.cap, kp, pool_v, pool_i, na, r0,
                                   st, gate)
              : launch_merge_splits(parts.v, parts.i, p.splits, kinds, rows, kp, pool_v, pool_i, na, r0, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_umma_gpool(const void* Y, int rows, int d, Elt elt, const int* gcam, bool cross, int self_excl,
                              int kp, const int4* items, const int* n_items, int max_items, const float* col_bias,
                              float* pool_v, int* pool_i, cudaStream_t st) {
  if (rows < 1 || max_items < 1) return cudaSuccess;
  CUtensorMap ta, tb;
  cudaError_t e = make_map(&ta, Y, elt, rows, d, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&tb, Y, elt, rows, d, BN);
  if (e != cudaSuccess) return e;
  UmmaArgs a{};
  a.mode = GPOOL;
  a.tf32 = elt == Elt::TF32;
  a.idesc = elt == Elt::F16 ? kIdescF16 : kIdescBf16;
  a.n = rows;
  a.d = d;
  a.a_rows = rows;
  a.self_excl = self_excl;
  a.cam = gcam;
  a.pool_v = pool_v;
  a.pool_i = pool_i;
  a.part_rows = rows;
  a.items = items;
  a.n_items = n_items;
  a.col_bias = col_bias;
  // persistent: one CTA per SM (the POOL shared memory allows one), items strided over the grid
  dim3 grid((unsigned)std::max(1, std::min(max_items, 152)));
  if (kp == 32) return cross ? launch<GPOOL, 32, true>(ta, tb, a, grid, st) : launch<GPOOL, 32, false>(ta, tb, a, grid, st);
  if (kp == 64) return cross ? launch<GPOOL, 64, true>(ta, tb, a, grid, st) : launch<GPOOL, 64, false>(ta, tb, a, grid, st);
  if (kp == 128) return cross ? launch<GPOOL, 128, true>(ta, tb, a, grid, st) : launch<GPOOL, 128, false>(ta, tb, a, grid, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_umma_band(const void* Xb, int n, int d, Elt elt, const int* cam, int self_excl,
                             const void* Ab, const int* count, int cap, const int* band_row,
                             const int* band_kind, const float* band_thr, int bcap, int* band_cnt, float* band_v,
                             int* band_i, cudaStream_t st, const int* band_off, const int* band_lim, Gate gate) {
  CUtensorMap ta, tb;
  cudaError_t e = make_map(&ta, Ab, elt, cap, d, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&tb, Xb, elt, n, d, BN);
  if (e != cudaSuccess) return e;
  UmmaArgs a{};
  a.mode = BAND;
  a.tf32 = elt == Elt::TF32;
  a.idesc = elt == Elt::F16 ? kIdescF16 : kIdescBf16;
  a.n = n;
  a.d = d;
  a.a_rows = cap;
  a.self_excl = self_excl;
  a.cam = cam;
  a.count = count;
  a.cap = cap;
  a.band_row = band_row;
  a.band_kind = band_kind;
  a.band_thr = band_thr;
  a.bcap = bcap;
  a.band_cnt = band_cnt;
  a.band_v = band_v;
  a.band_i = band_i;
  a.band_off = band_off;
  a.band_lim = band_lim;
  a.gate = gate;
  // the row tiles (known only on the device) are strided over grid.y so that the grid covers
  // the GPU about twice even when the columns give few tiles
  const int gx = (n + BN - 1) / BN;
  const int gy = std::max(1, std::min(8, (2 * 152 + gx - 1) / gx));
  dim3 grid(gx, gy);
  return launch<BAND, 64, false>(ta, tb, a, grid, st);
}

cudaError_t launch_umma_dist(const __nv_bfloat16* Qb, int nq, const __nv_bfloat16* Gb, int ng, int d,
                             const float* nrm_q, const float* nrm_g, float* D, cudaStream_t st) {
  CUtensorMap ta, tb;
  cudaError_t e = make_map(&ta, Qb, Elt::BF16, nq, d, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&tb, Gb, Elt::BF16, ng, d, BN);
  if (e != cudaSuccess) return e;
  UmmaArgs a{};
  a.mode = DIST;
  a.idesc = kIdescBf16;
  a.n = ng;
  a.d = d;
  a.a_rows = nq;
  a.nrm_q = nrm_q;
  a.nrm_g = nrm_g;
  a.D = D;
  // persistent: one CTA per SM walks its tiles, so the MMAs of a tile overlap the epilogue of
  // the previous one (double-buffered accumulators)
  a.dist_nrb = (nq + BM - 1) / BM;
  a.dist_tiles = a.dist_nrb * ((ng + BN - 1) / BN);
  dim3 grid((unsigned)std::max(1, std::min(a.dist_tiles, 152)));
  return launch<DIST, 64, false>(ta, tb, a, grid, st);
}

cudaError_t launch_umma_gram(const __nv_bfloat16* zt_hi, const __nv_bfloat16* zt_lo, int d, int64_t cols,
                             const int64_t* kstart, const int64_t* knum, const int64_t* nf, int ncam, float lambda,
                             float* G, cudaStream_t st) {
  if (cols > INT32_MAX || cols % 8) return cudaErrorInvalidValue;
  CUtensorMap ta, tb, ta2, tb2;
  cudaError_t e = make_map(&ta, zt_hi, Elt::BF16, d, (int)cols, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&tb, zt_hi, Elt::BF16, d, (int)cols, BN);
  if (e != cudaSuccess) return e;
  e = make_map(&ta2, zt_lo, Elt::BF16, d, (int)cols, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&tb2, zt_lo, Elt::BF16, d, (int)cols, BN);
  if (e != cudaSuccess) return e;
  UmmaArgs a{};
  a.mode = GRAM;
  a.idesc = kIdescBf16;
  a.n = d;
  a.d = 64;  // unused: the K extent of a tile comes from gram_knum
  a.a_rows = d;
  a.gram_kstart = kstart;
  a.gram_knum = knum;
  a.gram_nf = nf;
  a.gram_lambda = lambda;
  a.G = G;
  dim3 grid((d + BN - 1) / BN, (d + BM - 1) / BM, ncam);
  return launch<GRAM, 64, false>(ta, tb, a, grid, st, &ta2, &tb2);
}

cudaError_t launch_umma_mul(const float* p_hi, const float* p_lo, int rows, const float* g_hi, const float* g_lo,
                            int ncam, int d, const int* rowcam, float* Q, cudaStream_t st) {
  CUtensorMap ta, tb, ta2, tb2;
  cudaError_t e = make_map(&ta, p_hi, Elt::TF32, rows, d, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&ta2, p_lo, Elt::TF32, rows, d, BM);
  if (e != cudaSuccess) return e;
  e = make_map(&tb, g_hi, Elt::TF32, ncam * d, d, BN);
  if (e != cudaSuccess) return e;
  e = make_map(&tb2, g_lo, Elt::TF32, ncam * d, d, BN);
  if (e != cudaSuccess) return e;
  UmmaArgs a{};
  a.mode = MUL;
  a.tf32 = 1;
  a.n = d;
  a.d = d;
  a.a_rows = rows;
  a.mul_rowcam = rowcam;
  a.D = Q;
  dim3 grid((d + BN - 1) / BN, (rows + BM - 1) / BM);
  return launch<MUL, 64, false>(ta, tb, a, grid, st, &ta2, &tb2);
}

}  // namespace gcr
