// Streaming per-row candidate pool for the kNN search of Eq. 4 / Eq. 8.
//
// The similarity tile S = X_rows . X_cols^T is produced column tile by column tile and
// never stored. Each row has one owning thread (lane r of a warp owns row warp_row0 + r).
// Two forms. Selection buffers (SelCap and below, second half of this file) serve the searches.
// Sorted lists, first, serve the ball search's groups and two graphs of 128-entry pools on the
// tensor-core path; their owner holds three registers:
//   tau   admission threshold: the KP-th best score seen so far (-inf until KP seen),
//   qcnt  survivors queued in shared memory,
//   len   entries in the row's list.
// A column value v enters the row's queue only if v > tau. Once a queue may overflow,
// the warp merges it (all 32 lanes on one row at a time) into the row's sorted list of
// KP (score, index) pairs, kept in global memory (L2-resident). After the last column
// tile the list holds the row's KP best scores, and every score left out is <= its
// last entry. The certified refinement consumes exactly that guarantee.
#pragma once
#include "common.cuh"

namespace gcr {

// Queue layout in shared memory: float2 entries (score, index bits); for CTA-local row r,
// slot s lives at r*kQCap + (s ^ (r & 31)), so that the owner's 8-byte appends and the warp's
// reads during a merge are both conflict-free.
struct PoolOwner {
  float tau;
  float floor;  // admission floor (or -inf): scores at or below it are dropped, so tau never
                // drops below it; the caller bounds what was dropped by it
  int qcnt;
  int len;
};

__device__ __forceinline__ void pool_init(PoolOwner& o, bool valid, float floor) {
  o.floor = floor;
  o.tau = valid ? floor : CUDART_INF_F;
  o.qcnt = 0;
  o.len = 0;
}
__device__ __forceinline__ void pool_init(PoolOwner& o, bool valid) { pool_init(o, valid, -CUDART_INF_F); }

// Warp-cooperative merge of the queue of the row owned by lane `owner` into its list.
// qv_row/qi_row: that row's queue; lv/li: that row's list (KP entries) in global memory.
// Kept out of line (the merge is rare and large); takes and returns plain values so that the
// caller's owner state stays in registers. Returns the new list length and its last score.
struct MergeResult {
  int len;
  float last;
};

template <int KP>
__device__ __noinline__ MergeResult pool_merge_row(int owner, int lane, float* lv, int* li,
                                                   const float2* q_row, int sw, int my_qcnt, int my_len) {
  __syncwarp();  // the owner's queue writes must be visible to the whole warp
  int q = __shfl_sync(GCR_FULL, my_qcnt, owner);
  int L = __shfl_sync(GCR_FULL, my_len, owner);
  float a = -CUDART_INF_F;
  int ai = -1;
  if (lane < q) {
    const float2 e = q_row[lane ^ sw];
    a = e.x;
    ai = __float_as_int(e.y);
  }
  // the list loads (L2 latency) are issued before the queue sort so that the two overlap
  static_assert(KP == 32 || KP == 64 || KP == 128, "pool size must be 32, 64 or 128");
  constexpr int P = KP / 32;  // list entries per lane: entry e = p*32 + lane
  float b[P];
  int bi[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int e = p * 32 + lane;
    b[p] = e < L ? lv[e] : -CUDART_INF_F;
    bi[p] = e < L ? li[e] : -1;
  }
  warp_sort32_desc(a, ai, lane);
  float ar = __shfl_sync(GCR_FULL, a, 31 - lane);
  int ari = __shfl_sync(GCR_FULL, ai, 31 - lane);
  // Top KP of (list, descending) U (queue, descending): C[s] = max(B[s], Q[KP-1-s]) with Q
  // padded by -inf past 32 entries is a bitonic sequence holding exactly those KP; only the
  // last 32 entries can change. A bitonic merge then sorts it.
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
  for (int p = 0; p < P; ++p) {
    warp_merge32_desc(b[p], bi[p], lane);
    lv[p * 32 + lane] = b[p];
    li[p * 32 + lane] = bi[p];
  }
  const float last = __shfl_sync(GCR_FULL, b[P - 1], 31);
  __syncwarp();  // queue slots are reused only after every lane has read them
  return MergeResult{min(KP, L + q), last};
}

template <int KP>
__device__ __forceinline__ void pool_merge_apply(int owner, int lane, float* lv, int* li, const float2* q_row,
                                                 int sw, PoolOwner& me) {
  const MergeResult r = pool_merge_row<KP>(owner, lane, lv, li, q_row, sw, me.qcnt, me.len);
  if (lane == owner) {
    me.len = r.len;
    me.qcnt = 0;
    me.tau = (r.len == KP) ? fmaxf(r.last, me.floor) : me.floor;
  }
}

// Merge every row of this warp whose queue could not take `room` more entries.
// row_of_lane0: global row of lane 0; qrow0: CTA-local queue row of lane 0.
template <int KP>
__device__ __forceinline__ void pool_make_room(int room, int lane, PoolOwner& me, int row_of_lane0,
                                               int qrow0, float2* q, float* pool_v, int* pool_i) {
  unsigned m = __ballot_sync(GCR_FULL, me.qcnt >= kQCap - room);
  while (m) {
    int o = __ffs(m) - 1;
    m &= m - 1;
    int qr = qrow0 + o;
    size_t grow = (size_t)(row_of_lane0 + o);
    pool_merge_apply<KP>(o, lane, pool_v + grow * KP, pool_i + grow * KP, q + qr * kQCap, qr & 31, me);
  }
}

// Final merge of every valid row of the warp (writes the list even if nothing is queued).
template <int KP>
__device__ __forceinline__ void pool_flush(int lane, bool valid, PoolOwner& me, int row_of_lane0,
                                           int qrow0, float2* q, float* pool_v, int* pool_i) {
  unsigned m = __ballot_sync(GCR_FULL, valid);
  while (m) {
    int o = __ffs(m) - 1;
    m &= m - 1;
    int qr = qrow0 + o;
    size_t grow = (size_t)(row_of_lane0 + o);
    pool_merge_apply<KP>(o, lane, pool_v + grow * KP, pool_i + grow * KP, q + qr * kQCap, qr & 31, me);
  }
}

// ---------------------------------------------------------------- selection buffers
// The pools of the tensor-core sweep (POOL mode of umma.cu). A row's candidates sit unsorted in
// a buffer of CAP > KP slots in shared memory, owned by one lane: every score above the row's
// threshold is appended, and when any lane of the warp runs short of room all its lanes compact
// their buffers at once: a search over the buffered scores finds a value f with at least KP of
// them above it, the others are dropped and f becomes the threshold. KP of the row's scores lie
// above f, so nothing dropped at or below it can be among the row's KP best; after the sweep the
// buffer holds all of them (and up to CAP - KP more), and pool_finish sorts and cuts it.
// What bounds the sweep is the feed of the tensor core where rows are long, and the admissions
// (about KP (1 + ln(columns / KP)) a row) where they are short. A heap, which these buffers
// replaced for 32-entry pools, pays a chain of dependent shared-memory reads per admission; the
// sorted lists of the larger pools paid a warp-wide merge through L2 per row and 28 admissions.
// With column splits that fill the chip (pool_plan), similarity stage before and after: 201,000
// rows of d = 512, 64-entry pools, 238 -> 180 ms for three layers; 7,001 rows of d = 1000 in
// BF16, two graphs, 1.43 -> 0.57 ms; 800 rows of d = 128, two graphs, 150 -> 65 us; 512 queries
// against 500,000 rows of d = 256, the 128-entry pools, 1.98 -> 0.57 ms.
// Scores and columns are slot-major, [slot][128 rows], so a warp's lanes touch 32 different banks
// whatever slot each is at; columns are 16-bit offsets from the split's first.
// More slots, fewer compactions; what the ring (umma.cu) leaves. DEEP (32-entry pools of one
// graph): 44 slots and a four-stage ring, where long rows make the sweep bound by its feed;
// otherwise 96 slots and three stages.
template <int KP, bool CROSS, bool DEEP = false>
struct SelCap {
  static constexpr int cap = KP == 32 ? (CROSS ? 48 : DEEP ? 44 : 96) : KP == 64 ? (CROSS ? 80 : 96) : 160;
};
constexpr int kSelMaxCols = 65536;         // columns per split (16-bit offsets)
constexpr uint32_t kSelV = 128 * 4, kSelI = 128 * 2;  // bytes between consecutive slots

__device__ __forceinline__ float sel_ldv(uint32_t a) {
  float r;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(r) : "r"(a) : "memory");
  return r;
}
// Unordered load, for sel_compact alone: the appends precede its (out-of-line) call, and its own
// stores only go to slots it has read.
__device__ __forceinline__ float sel_ldv_any(uint32_t a) {
  float r;
  asm("ld.shared.f32 %0, [%1];" : "=f"(r) : "r"(a));
  return r;
}
__device__ __forceinline__ uint32_t sel_ldi(uint32_t a) {
  unsigned short r;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(r) : "r"(a) : "memory");
  return r;
}
__device__ __forceinline__ void sel_st(uint32_t va, uint32_t ia, float v, uint32_t i) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(va), "f"(v) : "memory");
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(ia), "h"((unsigned short)i) : "memory");
}

struct SelState {
  float tau;   // threshold: scores at or below it are dropped
  float lo;    // every buffered score is above it (tau, but for what other splits raised it by)
  float pub;   // a bound another split may drop at: KP of the row's scores are strictly above it
  float sum;   // of the buffered scores
  int cnt;
};

// The buffered scores of a lane as its compaction reads them: in registers (-inf past the count)
// up to 96 slots, else from shared memory 16 at a time. The tensor core's operand reads and the
// TMA's writes take most of the shared memory's bandwidth while a compaction runs, so every
// pass that stays in registers counts (15,000 cycles per compaction of 44 slots when each pass
// read them again).
template <int CAP, bool REGS = (CAP <= 96)>
struct SelScores {
  float v[CAP];
  __device__ __forceinline__ void load(uint32_t va, int cnt) {
#pragma unroll
    for (int s = 0; s < CAP; ++s) v[s] = sel_ldv_any(va + s * kSelV);
#pragma unroll
    for (int s = 0; s < CAP; ++s) v[s] = s < cnt ? v[s] : -CUDART_INF_F;
  }
  // scores above p and their sum
  __device__ __forceinline__ void count(float p, int& c, float& t) const {
    int c4[4] = {0, 0, 0, 0};
    float t4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s = 0; s < CAP; ++s) {
      const bool in = v[s] > p;
      c4[s & 3] += in ? 1 : 0;
      t4[s & 3] += in ? v[s] : 0.f;
    }
    c = (c4[0] + c4[1]) + (c4[2] + c4[3]);
    t = (t4[0] + t4[1]) + (t4[2] + t4[3]);
  }
  // the smallest and the largest score in (a, b]
  __device__ __forceinline__ void range(float a, float b, float& mn, float& mx) const {
#pragma unroll
    for (int s = 0; s < CAP; ++s)
      if (v[s] > a && v[s] <= b) {
        mn = fminf(mn, v[s]);
        mx = fmaxf(mx, v[s]);
      }
  }
  // bit s & 31 of word w = s >> 5: score s is above f (EQ: is f)
  template <bool EQ = false>
  __device__ __forceinline__ void above(float f, uint32_t (&m)[(CAP + 31) / 32]) const {
#pragma unroll
    for (int w = 0; w < (CAP + 31) / 32; ++w) m[w] = 0u;
#pragma unroll
    for (int s = 0; s < CAP; ++s) m[s >> 5] |= ((EQ ? v[s] == f : v[s] > f) ? 1u : 0u) << (s & 31);
  }
};
template <int CAP>
struct SelScores<CAP, false> {
  uint32_t va;
  int cnt;
  __device__ __forceinline__ void load(uint32_t a, int n) { va = a; cnt = n; }
  __device__ __forceinline__ void count(float p, int& c, float& t) const {
    int c4[4] = {0, 0, 0, 0};
    float t4[4] = {0.f, 0.f, 0.f, 0.f};
    static_assert(CAP % 16 == 0, "whole steps");
#pragma unroll 1
    for (int s0 = 0; s0 < CAP; s0 += 16) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = sel_ldv_any(va + (s0 + u) * kSelV);
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const bool in = v[u] > p && s0 + u < cnt;
        c4[u & 3] += in ? 1 : 0;
        t4[u & 3] += in ? v[u] : 0.f;
      }
    }
    c = (c4[0] + c4[1]) + (c4[2] + c4[3]);
    t = (t4[0] + t4[1]) + (t4[2] + t4[3]);
  }
  __device__ __forceinline__ void range(float a, float b, float& mn, float& mx) const {
#pragma unroll 8
    for (int s = 0; s < CAP; ++s) {
      const float v = sel_ldv_any(va + s * kSelV);
      if (s < cnt && v > a && v <= b) {
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
      }
    }
  }
  template <bool EQ = false>
  __device__ __forceinline__ void above(float f, uint32_t (&m)[(CAP + 31) / 32]) const {
#pragma unroll
    for (int w = 0; w < CAP / 32; ++w) {
      uint32_t x = 0;
#pragma unroll(EQ ? 4 : 32)
      for (int u = 0; u < 32; ++u) {
        const float v = sel_ldv_any(va + (w * 32 + u) * kSelV);
        x |= ((EQ ? v == f : v > f) && w * 32 + u < cnt ? 1u : 0u) << u;
      }
      m[w] = x;
    }
  }
};

// The kept entries past slot `kept` fill the holes before it.
template <int W>
__device__ __forceinline__ void sel_close(uint32_t (&keep)[W], int kept, uint32_t va, uint32_t ia) {
  uint32_t hole = 0, mover = 0;  // what is left of the words being walked
  int hw = -1, mw = -1;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int below = min(max(kept - 32 * w, 0), 32);
    const uint32_t in = below == 32 ? GCR_FULL : (1u << below) - 1u;
    const uint32_t h = ~keep[w] & in, m = keep[w] & ~in;
    keep[w] = h | m;  // holes below slot `kept`, movers from it on
  }
  auto next = [&](uint32_t& word, int& w, bool holes) -> int {
    while (word == 0u) {
      ++w;
      if (w >= W) return -1;
      const int below = min(max(kept - 32 * w, 0), 32);
      const uint32_t in = below == 32 ? GCR_FULL : (1u << below) - 1u;
      uint32_t x = 0;
#pragma unroll
      for (int q = 0; q < W; ++q)
        if (q == w) x = keep[q];
      word = holes ? (x & in) : (x & ~in);
    }
    const int b = __ffs(word) - 1;
    word &= word - 1u;
    return 32 * w + b;
  };
  for (;;) {
    const int h = next(hole, hw, true);
    if (h < 0) break;
    const int m = next(mover, mw, false);
    if (m < 0) break;
    sel_st(va + h * kSelV, ia + h * kSelI, sel_ldv(va + m * kSelV), sel_ldi(ia + m * kSelI));
  }
  __syncwarp();
}

// The scores a compaction's threshold lies among, (a, b]: ca of the entries are above a (ca >= KP), cb
// above b (cb < KP); ta, tb are the sums of those.
struct SelRange {
  float a, b, ta, tb;
  int ca, cb;
};

// The rest of a compaction whose pivots left some lane more than KP + kSlack entries: ties, or
// infinities. The range is cut to the scores in it, which ends at once if they are all equal, and
// halved by their order-preserving images, down to a threshold or to the score that the KP-th
// largest ties with; of the entries equal to it those of the smallest columns are kept up to KP, as a
// sorted list would, found by counting their columns' digits. A function of its own, so that the
// pivots keep their registers. (By a binary search for the score and one for the column, each step
// through shared memory, such a compaction cost many usual ones: the sweep of 13,290 rows of d = 512 with two non-zeros
// each, nearly all scores tied, took 4.5 ms in TF32, 0.7 so, and 8.3 and 4.3 in FP32; of random rows 0.5
// and 3.9.)
template <int KP, int CAP>
__device__ __noinline__ SelState sel_compact_ties(uint32_t va, uint32_t ia, SelState st, SelRange g) {
  constexpr int kSlack = (CAP - KP) / 4, W = (CAP + 31) / 32;
  const int cnt = st.cnt;
  const bool act = cnt > KP;
  SelScores<CAP> sc;
  sc.load(va, cnt);
  bool more = act && g.ca > KP + kSlack;
  if (more) {
    float mn = CUDART_INF_F, mx = -CUDART_INF_F;
    sc.range(g.a, g.b, mn, mx);
    g.a = float_below(mn);
    g.b = mx;
  }
  while (__any_sync(GCR_FULL, more)) {
    const uint32_t ka = float_to_ordered(g.a), kb = float_to_ordered(g.b);  // (a < b: also as images)
    if (kb - ka <= 1u) more = false;  // KP entries at b or above, fewer above it
    const float p = ordered_to_float(ka + ((kb - ka) >> 1));
    int c;
    float t;
    sc.count(p, c, t);
    if (more) {
      if (c >= KP) {
        more = c > KP + kSlack;
        g.a = p;
        g.ca = c;
        g.ta = t;
      } else {
        g.b = p;
        g.cb = c;
        g.tb = t;
      }
    }
  }
  const bool ex = act && g.ca > KP + kSlack;
  const float f = ex ? g.b : g.a;
  uint32_t keep[W], eq[W];
  sc.above(act ? f : -CUDART_INF_F, keep);
  sc.template above<true>(f, eq);
  int need = ex ? KP - g.cb : 0;  // of the entries equal to f, those of the smallest columns
  uint32_t col = 0;               // the digits, from the top, of the largest of these columns
  for (int shift = 12; shift >= 0; shift -= 4) {
    unsigned long long n0 = 0, n1 = 0;  // entries of each digit, 8 bits a count
#pragma unroll
    for (int w = 0; w < W; ++w)
#pragma unroll 8
      for (int u = 0; u < (CAP - 32 * w < 32 ? CAP - 32 * w : 32); ++u) {
        const uint32_t c = sel_ldi(ia + (32 * w + u) * kSelI) >> shift;
        if (((eq[w] >> u) & 1u) && c >> 4 == col) {
          const unsigned long long one = 1ull << (8u * (c & 7u));
          if (c & 8u) n1 += one;
          else n0 += one;
        }
      }
    uint32_t dg = 0;
    for (; dg < 15u; ++dg) {
      const int c = (int)((dg < 8u ? n0 >> (8u * dg) : n1 >> (8u * (dg - 8u))) & 255u);
      if (c >= need) break;
      need -= c;
    }
    col = col << 4 | dg;
  }
  if (ex) {
#pragma unroll
    for (int w = 0; w < W; ++w)
#pragma unroll 8
      for (int u = 0; u < (CAP - 32 * w < 32 ? CAP - 32 * w : 32); ++u)
        keep[w] |= (sel_ldi(ia + (32 * w + u) * kSelI) <= col ? eq[w] : 0u) & (1u << u);
  }
  if (act) {
    st.lo = ex ? float_below(f) : f;  // (every tied entry kept is above the value below f)
    st.cnt = ex ? KP : g.ca;
    st.sum = ex ? g.tb + (float)(KP - g.cb) * f : g.ta;
    st.tau = fmaxf(st.tau, f);  // another split may have raised it further
    st.pub = fmaxf(st.pub, st.lo);
  }
  sel_close(keep, st.cnt, va, ia);
  return st;
}

// Compacts the buffers of the warp's lanes (slot 0 at va / ia, cnt entries): a lane with more
// than KP entries keeps KP to KP + kSlack of them (in any order), the others keep all. Every
// lane of the warp calls it. The threshold is searched by pivots: the scores of a row's best few
// hundred fall off about exponentially, so the first pivot is the quantile of an exponential
// with their mean above the old threshold; the next ones are the mean of the scores still in
// question, which splits them whatever their spread (a midpoint takes many more steps when a
// few scores lie far above the rest). Five or six passes settle most warps; what a mean does not
// split is left to sel_compact_ties.
// SUM: st.sum is given; else it is taken from the buffer.
template <int KP, int CAP, bool SUM = true>
__device__ __noinline__ SelState sel_compact(uint32_t va, uint32_t ia, SelState st) {
  constexpr int kSlack = (CAP - KP) / 4, W = (CAP + 31) / 32;
  constexpr float kTarget = KP + 0.5f * kSlack;
  const int cnt = st.cnt;
  const bool act = cnt > KP;
  SelScores<CAP> sc;
  sc.load(va, cnt);
  SelRange g{st.lo, CUDART_INF_F, st.sum, 0.f, cnt, 0};
  if constexpr (!SUM) {
    int c;
    sc.count(-CUDART_INF_F, c, g.ta);
  }
  bool more = act;
  for (int it = 0; it < 12 && __any_sync(GCR_FULL, more); ++it) {
    float p = (g.ta - g.tb) / (float)max(1, g.ca - g.cb);
    if (it == 0) {
      const float q = g.a + (p - g.a) * __logf((float)g.ca / kTarget);
      if (q > g.a && q < p) p = q;
    }
    int c;
    float t;
    sc.count(p, c, t);
    if (more) {
      if (c >= KP) {
        more = c > KP + kSlack && (it == 0 || c < g.ca);
        if (p > g.a) {
          g.a = p;
          g.ca = c;
          g.ta = t;
        }
      } else {
        more = it == 0 || c > g.cb;
        if (p < g.b) {
          g.b = p;
          g.cb = c;
          g.tb = t;
        }
      }
    }
  }
  if (__any_sync(GCR_FULL, act && g.ca > KP + kSlack)) return sel_compact_ties<KP, CAP>(va, ia, st, g);
  uint32_t keep[W];
  sc.above(act ? g.a : -CUDART_INF_F, keep);
  if (act) {
    st.lo = g.a;
    st.cnt = g.ca;
    st.sum = g.ta;  // (a lane that keeps all keeps its sum)
    st.tau = fmaxf(st.tau, g.a);  // another split may have raised it further
    st.pub = fmaxf(st.pub, g.a);
  }
  sel_close(keep, st.cnt, va, ia);
  return st;
}

}  // namespace gcr
