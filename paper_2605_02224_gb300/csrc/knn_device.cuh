// Device-side body of one k-NN query: Algorithm 1 (successor-list descent
// collecting transition sites) then Algorithm 2 (expansion over the
// successor lists of the nearest sites found so far), Sec. 4.
//
// One query is served by a group of G lanes (G = 4, 8, 16 or 32) of a
// warp. The group reads G consecutive successor entries at a time
// (coalesced), gathers their float4 coordinates through the read-only
// path, and decides with warp votes.
//
// Candidate list N: capacity K = G * S, sorted by the key (d, rank),
// distributed over the group: lane l, slot s holds position s * G + l. An
// insertion counts the keys below the new one with S votes, shifts the
// tail by one position with S shuffles per field and drops position k.
// Bit 31 of a stored rank marks an entry whose list has been expanded.
//
// Readings of the paper (see the design notes for the full list):
//  * descent: the scan of L_curr moves to the FIRST entry (lowest rank) that
//    is strictly closer than p_curr and restarts at the head of the new
//    list; every site moved to is inserted into N (all transition sites are
//    candidates, Sec. 4.2);
//  * "strictly closer" is decided in float32 with a guard band; inside the
//    band both distances are recomputed in float64 in the oracle's order,
//    so the descent follows the exact prefix minima of Eq. (2);
//  * expansion: the nearest not-yet-expanded entry among the first k-1 of
//    N is expanded until none is left (equal to Alg. 2's loop in exact
//    arithmetic, robust to float32 reordering of near-equal distances);
//  * prefix bound m (Sec. 4.2): rows are ascending, so a scan stops at the
//    first entry >= m.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "hub_index.h"

namespace mknn {

constexpr uint32_t kRankMask = 0x7fffffffu;
constexpr uint32_t kDoneBit = 0x80000000u;
constexpr uint32_t kPadRank = 0xffffffffu;
// |d32 - D| <= 5 * 2^-24 * D for the float32 evaluation below; the guard
// band is three times wider than the sum of two such errors.
constexpr float kGuard = 2e-6f;
// Below this the float32 distance may be subnormal; decide in float64.
constexpr float kTiny = 1e-30f;
// Entries of a list with a tree that the descent reads in rank order before
// it turns to the tree: the first strictly closer entry is often among the
// first few (the low ranks are spread over the whole cloud), and a walk
// that must prove its rank the lowest costs more than a chunk. On the patch
// clouds of the batching mix 0 / 32 / 64 / 128 entries took 104 / 98 / 100
// / 102 ms with the hand-over.
constexpr int kHubScanFirst = 32;

struct CloudDev {
  const float4* __restrict__ pts;
  const int2* __restrict__ rows;     // (first, end) of each successor row
  const int32_t* __restrict__ succ;
  int32_t n;
  // succ with each entry's site inlined: (x, y, z, rank bits), one 16-byte
  // load per entry instead of an index load and a dependent point load
  const float4* __restrict__ ent;
  // box trees over the long lists (NULL hub_of: none); read by the one-warp
  // kernel only. hub_of[i]: the tree of site i's list or -1; hub_desc:
  // (first entry, list length, first node, levels); hub_ent: the list's
  // entries along a Morton curve in chunks of 32; hub_node: two float4 per
  // node, (low corner, smallest rank's bits) and (high corner, largest
  // rank's bits), levels stored from the chunks' boxes up
  const int32_t* __restrict__ hub_of = nullptr;
  const int4* __restrict__ hub_desc = nullptr;
  const float4* __restrict__ hub_ent = nullptr;
  const float4* __restrict__ hub_node = nullptr;
};

// Squared distance in float32, fixed operation order (no reassociation).
__device__ __forceinline__ float sqd32(float qx, float qy, float qz, float4 p) {
  const float dx = __fsub_rn(qx, p.x);
  const float dy = __fsub_rn(qy, p.y);
  const float dz = __fsub_rn(qz, p.z);
  float d = __fmul_rn(dx, dx);
  d = __fmaf_rn(dy, dy, d);
  d = __fmaf_rn(dz, dz, d);
  return d;
}

// Squared distance in float64: ((dx*dx + dy*dy) + dz*dz), no fusion.
__device__ __forceinline__ double sqd64(float qx, float qy, float qz, float px, float py,
                                        float pz) {
  const double dx = __dsub_rn((double)qx, (double)px);
  const double dy = __dsub_rn((double)qy, (double)py);
  const double dz = __dsub_rn((double)qz, (double)pz);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__device__ __forceinline__ bool key_lt(float da, uint32_t ra, float db, uint32_t rb) {
  return da < db || (da == db && ra < rb);
}

template <int G>
struct Grp {
  uint32_t lane, base, mask;
  __device__ __forceinline__ Grp() {
    const uint32_t l = threadIdx.x & 31u;
    lane = l & (G - 1);
    base = l & ~(uint32_t)(G - 1);
    mask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << base);
  }
  __device__ __forceinline__ uint32_t ballot(bool p) const {
    const uint32_t b = __ballot_sync(mask, p);
    return (G == 32) ? b : ((b >> base) & ((1u << G) - 1u));
  }
  template <class T>
  __device__ __forceinline__ T shfl(T v, int src) const {
    return __shfl_sync(mask, v, src, G);
  }
};

template <int G, int S>
struct TopK {
  float d[S];
  uint32_t r[S];
  int cnt;
  float kd;     // key of position k-1 (a pad while fewer than k entries)
  uint32_t kr;
};

template <int G, int S>
__device__ __forceinline__ void topk_init(TopK<G, S>& T) {
#pragma unroll
  for (int s = 0; s < S; ++s) {
    T.d[s] = __int_as_float(0x7f800000);
    T.r[s] = kPadRank;
  }
  T.cnt = 0;
  T.kd = __int_as_float(0x7f800000);
  T.kr = kRankMask;
}

// Inserts (cd, cr) unless an equal key is present; keeps k entries.
template <int G, int S>
__device__ __forceinline__ void topk_insert(TopK<G, S>& T, const Grp<G>& g, float cd, uint32_t cr,
                                            int k) {
  int less = 0;
  bool eq = false;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const uint32_t rr = T.r[s] & kRankMask;
    less += __popc(g.ballot(key_lt(T.d[s], rr, cd, cr)));
    eq |= (T.d[s] == cd) & (rr == cr);
  }
  if (g.ballot(eq) || less >= k) return;
  const int pos = less;
  const int src = (int)((g.lane + G - 1) & (G - 1));
  float ud[S];
  uint32_t ur[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    ud[s] = g.shfl(T.d[s], src);
    ur[s] = g.shfl(T.r[s], src);
  }
#pragma unroll
  for (int s = S - 1; s >= 0; --s) {
    const int p = s * G + (int)g.lane;
    float pd;
    uint32_t pr;
    if (g.lane == 0) {
      pd = (s > 0) ? ud[s > 0 ? s - 1 : 0] : 0.f;
      pr = (s > 0) ? ur[s > 0 ? s - 1 : 0] : 0u;
    } else {
      pd = ud[s];
      pr = ur[s];
    }
    if (p >= k) {
      T.d[s] = __int_as_float(0x7f800000);
      T.r[s] = kPadRank;
    } else if (p > pos) {
      T.d[s] = pd;
      T.r[s] = pr;
    } else if (p == pos) {
      T.d[s] = cd;
      T.r[s] = cr;
    }
  }
  T.cnt = min(T.cnt + 1, k);
  const int kp = k - 1;
  const int ks = kp / G, kl = kp % G;
  float td = T.d[0];
  uint32_t tr = T.r[0];
#pragma unroll
  for (int s = 1; s < S; ++s)
    if (s == ks) {
      td = T.d[s];
      tr = T.r[s];
    }
  T.kd = g.shfl(td, kl);
  T.kr = g.shfl(tr, kl) & kRankMask;
}

struct QueryCounters {
  int rows, entries, coords, trans;
};

// One query by one group. m in [1, n]. Writes k results to oi / od.
template <int G, int S, bool COUNT>
__device__ __forceinline__ void knn_query(const CloudDev& C, const Grp<G>& g, float qx, float qy,
                                          float qz, int k, int m, int32_t* __restrict__ out_idx,
                                          float* __restrict__ out_d2, int32_t row,
                                          QueryCounters& qc) {
  const float INF = __int_as_float(0x7f800000);
  TopK<G, S> T;
  topk_init(T);

  // ---- Algorithm 1: descent from p_1 (rank 0), collecting transition sites
  // (the current site is held as a rank; its coordinates are reloaded only
  // for a float64 recheck)
  int curr = 0;
  float dcur = sqd32(qx, qy, qz, __ldg(C.pts));
  topk_insert(T, g, dcur, 0u, k);
  if (COUNT) {
    qc.coords = 1;
    qc.trans = 1;
  }
  for (;;) {
    const int2 rr = __ldg(C.rows + curr);
    const uint32_t beg = rr.x, end = rr.y;  // unsigned: no overflow of base + G
    if (COUNT) qc.rows++;
    bool moved = false;
    for (uint32_t base = beg; base < end; base += G) {
      const uint32_t e = base + g.lane;
      const bool valid = e < end;
      float4 ps = make_float4(0.f, 0.f, 0.f, 0.f);
      if (valid) ps = __ldg(C.ent + e);  // site and rank of the entry
      const int s = valid ? __float_as_int(ps.w) : 0x7fffffff;
      const bool inr = valid && s < m;
      const float d = inr ? sqd32(qx, qy, qz, ps) : INF;
      bool sure, maybe;
      if (dcur >= kTiny) {
        sure = inr && d < dcur * (1.f - kGuard);
        maybe = inr && !sure && d <= dcur * (1.f + kGuard);
      } else {
        sure = false;
        maybe = inr && d <= 2.f * kTiny;
      }
      uint32_t closer = g.ballot(sure);
      if (g.ballot(maybe)) {
        bool c64 = false;
        if (maybe) {
          const float4 pc = __ldg(C.pts + curr);
          c64 = sqd64(qx, qy, qz, ps.x, ps.y, ps.z) < sqd64(qx, qy, qz, pc.x, pc.y, pc.z);
        }
        closer |= g.ballot(c64);
      }
      const uint32_t stop = g.ballot(valid && !inr);
      if (closer) {
        const int w = __ffs(closer) - 1;
        if (COUNT) {
          qc.entries += w + 1;
          qc.coords += w + 1;
          qc.trans++;
        }
        curr = g.shfl(s, w);
        dcur = g.shfl(d, w);
        topk_insert(T, g, dcur, (uint32_t)curr, k);
        moved = true;
        break;
      }
      if (COUNT) {
        if (stop) {
          const int t = __ffs(stop) - 1;
          qc.entries += t + 1;
          qc.coords += t;
        } else {
          const int nv = min(G, (int)(end - base));
          qc.entries += nv;
          qc.coords += nv;
        }
      }
      if (stop) break;
    }
    if (!moved) break;
  }

  // ---- Algorithm 2: expand the nearest unexpanded entry among the first k-1
  for (;;) {
    const int lim = min(T.cnt, k - 1);
    int pos = -1;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int p = s * G + (int)g.lane;
      const uint32_t b = g.ballot(p < lim && !(T.r[s] & kDoneBit));
      if (b && pos < 0) pos = s * G + __ffs(b) - 1;
    }
    if (pos < 0) break;
    const int psl = pos / G, pln = pos % G;
    uint32_t rsel = T.r[0];
#pragma unroll
    for (int s = 1; s < S; ++s)
      if (s == psl) rsel = T.r[s];
    const int site = (int)(g.shfl(rsel, pln) & kRankMask);
    if ((int)g.lane == pln) {
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (s == psl) T.r[s] |= kDoneBit;
    }
    const int2 rr = __ldg(C.rows + site);
    const uint32_t beg = rr.x, end = rr.y;
    if (COUNT) qc.rows++;
    for (uint32_t base = beg; base < end; base += G) {
      const uint32_t e = base + g.lane;
      const bool valid = e < end;
      float4 ps = make_float4(0.f, 0.f, 0.f, 0.f);
      if (valid) ps = __ldg(C.ent + e);
      const int s = valid ? __float_as_int(ps.w) : 0x7fffffff;
      const bool inr = valid && s < m;
      const float d = inr ? sqd32(qx, qy, qz, ps) : INF;
      bool pass = inr && key_lt(d, (uint32_t)s, T.kd, T.kr);
      uint32_t b = g.ballot(pass);
      while (b) {
        const int w = __ffs(b) - 1;
        const float cd = g.shfl(d, w);
        const uint32_t cr = g.shfl((uint32_t)s, w);
        topk_insert(T, g, cd, cr, k);
        pass = pass && ((int)g.lane > w) && key_lt(d, (uint32_t)s, T.kd, T.kr);
        b = g.ballot(pass);
      }
      const uint32_t stop = g.ballot(valid && !inr);
      if (COUNT) {
        if (stop) {
          const int t = __ffs(stop) - 1;
          qc.entries += t + 1;
          qc.coords += t;
        } else {
          const int nv = min(G, (int)(end - base));
          qc.entries += nv;
          qc.coords += nv;
        }
      }
      if (stop) break;
    }
  }

  // ---- output: sorted (d, rank), padded with (-1, +inf)
  int32_t* oi = out_idx + (int64_t)row * k;
  float* od = out_d2 + (int64_t)row * k;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int p = s * G + (int)g.lane;
    if (p < k) {
      const uint32_t rr = T.r[s] & kRankMask;
      const bool real = rr != kRankMask;
      __stcs(oi + p, real ? (int32_t)rr : -1);
      __stcs(od + p, real ? T.d[s] : INF);
    }
  }
}

// ---------------------------------------------------------------------------
// One query per thread. The candidate list N is an unsorted array of K
// register slots holding the best min(k, seen) keys, with the worst of them
// tracked as the admission threshold once the list is full. The order the
// algorithm needs is recovered on demand: the nearest not-yet-expanded
// entry among "the first k-1" is the smallest unexpanded key other than the
// worst one (when the list is full). No lane talks to another, so a warp
// serves 32 queries with no votes or shuffles; with locality-sorted
// queries the 32 descents share most of their path.
template <int K>
struct TopT {
  float d[K];
  uint32_t r[K];  // rank, bit 31 = expanded
  int cnt;
  int worst;      // slot of the worst key, valid when cnt == k
  float wd;       // worst key (threshold); (+inf, kRankMask) while cnt < k
  uint32_t wr;
};

template <int K>
__device__ __forceinline__ void topt_init(TopT<K>& T) {
#pragma unroll
  for (int i = 0; i < K; ++i) {
    T.d[i] = __int_as_float(0x7f800000);
    T.r[i] = kPadRank;
  }
  T.cnt = 0;
  T.worst = 0;
  T.wd = __int_as_float(0x7f800000);
  T.wr = kRankMask;
}

// Inserts (cd, cr) unless present. Caller checks key_lt(cd, cr, wd, wr).
template <int K>
__device__ __forceinline__ void topt_insert(TopT<K>& T, float cd, uint32_t cr, int k) {
  bool dup = false;
#pragma unroll
  for (int i = 0; i < K; ++i) dup |= (T.d[i] == cd) & ((T.r[i] & kRankMask) == cr);
  if (dup) return;
  int slot;
  if (T.cnt < k) {
    slot = T.cnt++;
  } else {
    slot = T.worst;
  }
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (i == slot) {
      T.d[i] = cd;
      T.r[i] = cr;
    }
  if (T.cnt == k) {
    float wd = -1.f;
    uint32_t wr = 0;
    int w = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const uint32_t ri = T.r[i] & kRankMask;
      if (i < k && key_lt(wd, wr, T.d[i], ri)) {
        wd = T.d[i];
        wr = ri;
        w = i;
      }
    }
    T.worst = w;
    T.wd = wd;
    T.wr = wr;
  }
}

template <int K, bool COUNT>
__device__ __forceinline__ void knn_query_thread(const CloudDev& C, float qx, float qy, float qz,
                                                 int k, int m, int32_t* __restrict__ oi,
                                                 float* __restrict__ od, QueryCounters& qc) {
  const float INF = __int_as_float(0x7f800000);
  TopT<K> T;
  topt_init(T);

  // ---- Algorithm 1
  int curr = 0;
  float4 pc = __ldg(C.pts);
  float dcur = sqd32(qx, qy, qz, pc);
  topt_insert(T, dcur, 0u, k);
  if (COUNT) {
    qc.coords = 1;
    qc.trans = 1;
  }
  for (;;) {
    const int2 rr = __ldg(C.rows + curr);
    int e = rr.x;
    const int end = rr.y;
    if (COUNT) qc.rows++;
    bool moved = false;
    for (; e < end; ++e) {
      const int s = __ldg(C.succ + e);
      if (COUNT) qc.entries++;
      if (s >= m) break;
      const float4 ps = __ldg(C.pts + s);
      const float d = sqd32(qx, qy, qz, ps);
      if (COUNT) qc.coords++;
      bool closer;
      if (dcur >= kTiny && d < dcur * (1.f - kGuard)) {
        closer = true;
      } else if ((dcur >= kTiny && d > dcur * (1.f + kGuard)) || (dcur < kTiny && d > 2.f * kTiny)) {
        closer = false;
      } else {
        closer = sqd64(qx, qy, qz, ps.x, ps.y, ps.z) < sqd64(qx, qy, qz, pc.x, pc.y, pc.z);
      }
      if (closer) {
        curr = s;
        dcur = d;
        pc = ps;
        if (key_lt(d, (uint32_t)s, T.wd, T.wr)) topt_insert(T, d, (uint32_t)s, k);
        if (COUNT) qc.trans++;
        moved = true;
        break;
      }
    }
    if (!moved) break;
  }

  // ---- Algorithm 2
  for (;;) {
    float bd = INF;
    uint32_t br = kRankMask;
    int bi = -1;
    const bool full = T.cnt == k;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const uint32_t ri = T.r[i] & kRankMask;
      const bool ok = (i < T.cnt) && !(T.r[i] & kDoneBit) && !(full && i == T.worst);
      if (ok && key_lt(T.d[i], ri, bd, br)) {
        bd = T.d[i];
        br = ri;
        bi = i;
      }
    }
    if (bi < 0) break;
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (i == bi) T.r[i] |= kDoneBit;
    const int site = (int)br;
    const int2 rr = __ldg(C.rows + site);
    int e = rr.x;
    const int end = rr.y;
    if (COUNT) qc.rows++;
    for (; e < end; ++e) {
      const int s = __ldg(C.succ + e);
      if (COUNT) qc.entries++;
      if (s >= m) break;
      const float d = sqd32(qx, qy, qz, __ldg(C.pts + s));
      if (COUNT) qc.coords++;
      if (key_lt(d, (uint32_t)s, T.wd, T.wr)) topt_insert(T, d, (uint32_t)s, k);
    }
  }

  // ---- output: position of each entry = number of smaller keys
#pragma unroll
  for (int i = 0; i < K; ++i) {
    if (i < T.cnt) {
      const uint32_t ri = T.r[i] & kRankMask;
      int pos = 0;
#pragma unroll
      for (int j = 0; j < K; ++j) pos += key_lt(T.d[j], T.r[j] & kRankMask, T.d[i], ri) ? 1 : 0;
      oi[pos] = (int32_t)ri;
      od[pos] = T.d[i];
    }
  }
  for (int p = T.cnt; p < k; ++p) {
    oi[p] = -1;
    od[p] = INF;
  }
}

// ---------------------------------------------------------------------------
// One query per thread with the candidate list N in shared memory: entry i
// of the lane's list at col[i * 32] (a warp's lists interleaved, so any mix
// of positions across the lanes is bank-conflict free). An entry is one
// 64-bit key, the float bits of the squared distance above the rank plus
// one: distances are never negative, so the integer order of the keys is
// the (distance, rank) order and a comparison, a load or a move is one or
// two instructions. Slots not yet filled hold a pad key above every real
// one, so the search for an insertion position is a fixed sequence of
// halving steps with no bound to track. The search also finds an equal key,
// so the membership test of Alg. 2 costs nothing extra. The nearest not-yet-
// expanded entry among the first k-1 is one bit scan of the expanded mask;
// the output comes out in order. The list takes no registers, which leaves
// room for more resident warps.
//
// The lanes of a warp run in step, so the warp pays for the insertion code
// whenever any of its lanes inserts: insertion is kept to a short sequence
// with no data-dependent loop where that pays.
//  * PermList<8> (k <= 8), PermList<16> (k <= 16): keys stay where they were
//    written, a register holds their order.
//  * PermList32 (k <= 32): two such registers, for the nearer 16 and the
//    others.
//  * SortedList (k > 32): keys kept in position order; an insertion shifts
//    the tail by one slot (a loop as long as the longest shift among the
//    lanes inserting).
__device__ __forceinline__ uint64_t pack_key(float d, uint32_t r) {
  return ((uint64_t)__float_as_uint(d) << 32) | r;
}

// above every real key (real keys have the sign bit of the distance clear)
constexpr uint64_t kPadKey = ~0ull;

// Expanded flags, one bit per list position, in W 32-bit words: W = 1 for
// k <= 32 (one 32-bit register), 2 for k <= 64 (one 64-bit), 4 for k <= 128
// (two 64-bit).
template <int W>
struct Flags {
  uint64_t lo = 0, hi = 0;
};
template <>
struct Flags<1> {
  uint32_t lo = 0;
};

// Opens a clear flag at bit pos of one word: bits at pos and above move up.
template <typename T>
__device__ __forceinline__ T flags_open(T f, int pos) {
  const T low = pos ? (f & (~T(0) >> (8 * sizeof(T) - pos))) : T(0);
  return low | ((f >> pos) << 1 << pos);
}

// Opens a clear flag at list position pos (an insertion there).
template <int W>
__device__ __forceinline__ void flags_insert(Flags<W>& F, int pos) {
  if constexpr (W == 4) {
    if (pos < 64) {
      F.hi = (F.hi << 1) | (F.lo >> 63);
      F.lo = flags_open(F.lo, pos);
    } else {
      F.hi = flags_open(F.hi, pos - 64);
    }
  } else {
    F.lo = flags_open(F.lo, pos);
  }
}

// Position of the first entry among the first lim not yet expanded, or -1.
template <int W>
__device__ __forceinline__ int flags_first_clear(const Flags<W>& F, int lim) {
  if constexpr (W == 1) {
    const uint32_t c = ~F.lo & ((1u << lim) - 1u);  // lim <= 31
    return c ? __ffs((int)c) - 1 : -1;
  } else {
    const int l0 = min(lim, 64);
    const uint64_t c0 = ~F.lo & (l0 == 64 ? ~0ull : ((1ull << l0) - 1ull));
    if (c0) return __ffsll((long long)c0) - 1;
    if constexpr (W == 4) {
      if (lim > 64) {
        const uint64_t c1 = ~F.hi & ((1ull << (lim - 64)) - 1ull);
        if (c1) return 64 + __ffsll((long long)c1) - 1;
      }
    }
    return -1;
  }
}

template <int W>
__device__ __forceinline__ void flags_set(Flags<W>& F, int pos) {
  if constexpr (W == 1) {
    F.lo |= 1u << pos;
  } else if constexpr (W == 2) {
    F.lo |= 1ull << pos;
  } else {
    if (pos < 64)
      F.lo |= 1ull << pos;
    else
      F.hi |= 1ull << (pos - 64);
  }
}

// A one-lane list's key: the rank is stored plus one, so that 0 is below
// every real key.
__device__ __forceinline__ uint64_t lane_key(float d, int s) { return pack_key(d, (uint32_t)s + 1u); }

// Keys in position order. KS: the search size (a power of two >= the
// list's capacity cap); positions in [cap, KS) read as pads without a load.
template <int KS, int W>
struct SortedList {
  static constexpr int kVoteEvery = 1;  // see knn_query_smem
  uint64_t* col;
  int cap;
  int cnt;
  Flags<W> done;   // bit i: entry at position i expanded
  uint64_t worst;  // key of position k-1 (a pad while cnt < k)

  __device__ __forceinline__ void init(uint64_t* c, int k) {
    col = c;
    cap = k;
    cnt = 0;
    done = Flags<W>{};
    worst = kPadKey;
    for (int i = 0; i < cap; ++i) col[i * 32] = kPadKey;
  }
  __device__ __forceinline__ uint64_t key_at(int pos) const { return col[pos * 32]; }
  __device__ __forceinline__ uint64_t probe(int pos) const {
    return pos < cap ? col[pos * 32] : kPadKey;
  }
  // Inserts key c unless present; requires c < worst (then the position
  // found is below k <= cap).
  __device__ __forceinline__ void insert(uint64_t c, int k) {
    int pos = 0;
#pragma unroll
    for (int step = KS / 2; step >= 1; step >>= 1)
      if (probe(pos + step - 1) < c) pos += step;
    if (pos >= k || col[pos * 32] == c) return;
    for (int i = min(cnt, k - 1); i > pos; --i) col[i * 32] = col[(i - 1) * 32];
    col[pos * 32] = c;
    flags_insert(done, pos);
    if (cnt < k) cnt++;
    if (cnt == k) worst = col[(k - 1) * 32];
  }
  // Marks the nearest entry among the first k-1 not yet expanded and
  // returns its rank, or -1 when there is none.
  __device__ __forceinline__ int next(int k) {
    const int pos = flags_first_clear(done, min(cnt, k - 1));
    if (pos < 0) return -1;
    flags_set(done, pos);
    return (int)((uint32_t)col[pos * 32] - 1u);
  }
};

template <int S>
struct PermWord;
template <>
struct PermWord<8> {
  using T = uint32_t;
  static constexpr T identity = 0x76543210u;
};
template <>
struct PermWord<16> {
  using T = uint64_t;
  static constexpr T identity = 0xFEDCBA9876543210ull;
};

// S = 8 (k <= 8) or 16 (k <= 16) slots: keys stay in the slot they were
// written to; a register holds the slot of each position, four bits each.
// The list's k positions are the last k of S: the first S - k hold key 0
// (below every real key, marked expanded), so the position that drops out
// is always S - 1 and no step depends on k. An insertion writes the new key
// into the slot of position S - 1 and moves that slot's four bits to the
// insertion position: no key moves, a fixed instruction sequence.
template <int S>
struct PermList {
  static constexpr int kVoteEvery = 2;  // see knn_query_smem
  using T = typename PermWord<S>::T;
  uint64_t* col;
  T perm;          // bits 4j..4j+3: the slot of position j
  uint32_t done;   // by position
  uint64_t worst;  // key of position S-1 (a pad while fewer than k entries)

  __device__ __forceinline__ void init(uint64_t* c, int k) {
    col = c;
    perm = PermWord<S>::identity;
    done = (1u << (S - k)) - 1u;
    worst = kPadKey;
#pragma unroll
    for (int i = 0; i < S; ++i) col[i * 32] = i < S - k ? 0ull : kPadKey;
  }
  // the key whose slot is the four bits of perm at bit sh
  __device__ __forceinline__ uint64_t at(int sh) const {
    return col[((uint32_t)(perm >> sh) & 15u) * 32];
  }
  __device__ __forceinline__ uint64_t key_at(int pos, int k) const { return at(4 * (S - k + pos)); }
  // Inserts key c unless present; requires c < worst.
  __device__ __forceinline__ void insert(uint64_t c, int) {
    int sh = 0;  // four times the number of keys below c
#pragma unroll
    for (int step = S / 2; step >= 1; step >>= 1)
      if (at(sh + 4 * (step - 1)) < c) sh += 4 * step;
    if (at(sh) == c) return;
    const uint32_t w = (uint32_t)(perm >> (4 * S - 4));  // the dropped key's slot (or a pad's)
    col[w * 32] = c;
    // positions from sh / 4 on move up by one, w goes to sh / 4
    const T low = perm & ((T(1) << sh) - 1);
    perm = low | ((perm ^ low) << 4) | (T(w) << sh);
    const uint32_t fl = done & ((1u << (sh >> 2)) - 1u);
    done = fl | ((done ^ fl) << 1);
    worst = at(4 * S - 4);
  }
  __device__ __forceinline__ int next(int) {
    const uint32_t c = ~done & ((1u << (S - 1)) - 1u);
    if (c == 0u) return -1;
    const int pos = __ffs((int)c) - 1;
    const uint64_t key = at(4 * pos);
    if (key == kPadKey) return -1;  // pads only from here on
    done |= 1u << pos;
    return (int)((uint32_t)key - 1u);
  }
};
// 17 <= k <= 32: two permutation words over 32 slots, one for the nearer 16
// positions (near) and one for the others (far). An insertion searches one of
// the halves; a key that drops out of the nearer one goes to the front of the
// other. As in PermList the k positions are the last k of 32, here without
// memory for the 32 - k unused slots: they are never read (the search takes
// their keys as below every other). 500k mixed queries on the 1M-site torus,
// k = 32: 2.73 ms with a sorted list and its shift loop, 2.53 ms now. What
// bounds it is the list's 256 bytes per thread: 24 warps per SM, so the block
// is held to three per SM and takes the registers it wants (72, no spills).
struct PermList32 {
  static constexpr int kVoteEvery = 1;  // see knn_query_smem
  uint64_t* col;      // slot s at col[s * 32], s >= 32 - k
  uint64_t near, far; // bits 4j..4j+3: the slot of position j (16 + j: less 16)
  uint32_t done;      // by position
  uint64_t worst;     // key of position 31 (a pad while fewer than k entries)

  __device__ __forceinline__ void init(uint64_t* c, int k) {
    col = c - (32 - k) * 32;
    near = far = PermWord<16>::identity;
    done = (1u << (32 - k)) - 1u;
    worst = kPadKey;
    for (int i = 0; i < k; ++i) c[i * 32] = kPadKey;
  }
  static __device__ __forceinline__ uint32_t slot(uint64_t perm, int sh) {
    return (uint32_t)(perm >> sh) & 15u;
  }
  static __device__ __forceinline__ uint64_t opened(uint64_t perm, int sh, uint32_t w) {
    const uint64_t low = perm & ((1ull << sh) - 1);
    return low | ((perm ^ low) << 4) | ((uint64_t)w << sh);
  }
  // key of position pos (one of the last k)
  __device__ __forceinline__ uint64_t at(int pos) const {
    const bool f = pos >= 16;
    return col[(slot(f ? far : near, 4 * (pos & 15)) + (f ? 16 : 0)) * 32];
  }
  __device__ __forceinline__ uint64_t key_at(int pos, int k) const { return at(32 - k + pos); }
  __device__ __forceinline__ void to_far(uint64_t key) {
    const uint32_t w = (uint32_t)(far >> 60);
    col[(16 + w) * 32] = key;
    far = (far << 4) | w;
  }
  // Inserts key c unless present; requires c < worst.
  __device__ __forceinline__ void insert(uint64_t c, int k) {
    const uint64_t top = col[(uint32_t)(near >> 60) * 32];  // position 15
    const bool f = c > top;
    const uint64_t perm = f ? far : near;
    uint64_t* half = f ? col + 16 * 32 : col;
    const int unused = f ? 0 : 4 * (32 - k);
    int sh = 0;  // four times the number of the half's keys below c
#pragma unroll
    for (int step = 8; step >= 1; step >>= 1) {
      const int at_sh = sh + 4 * (step - 1);
      if (at_sh < unused || half[slot(perm, at_sh) * 32] < c) sh += 4 * step;
    }
    if (half[slot(perm, sh) * 32] == c) return;
    const uint32_t w = (uint32_t)(perm >> 60);
    const uint64_t opn = opened(perm, sh, w);
    half[w * 32] = c;
    if (f) {
      far = opn;
    } else {
      near = opn;
      to_far(top);
    }
    const uint32_t fl = done & ((1u << ((sh >> 2) + (f ? 16 : 0))) - 1u);
    done = fl | ((done ^ fl) << 1);
    worst = col[(16 + (uint32_t)(far >> 60)) * 32];
  }
  __device__ __forceinline__ int next(int) {
    const uint32_t c = ~done & 0x7fffffffu;
    if (c == 0u) return -1;
    const int pos = __ffs((int)c) - 1;
    const uint64_t key = at(pos);
    if (key == kPadKey) return -1;  // pads only from here on
    done |= 1u << pos;
    return (int)((uint32_t)key - 1u);
  }
};
__device__ __forceinline__ uint64_t list_key(const PermList32& N, int p, int k) {
  return N.key_at(p, k);
}
template <int KS, int W>
__device__ __forceinline__ uint64_t list_key(const SortedList<KS, W>& N, int p, int) {
  return N.key_at(p);
}
template <int S>
__device__ __forceinline__ uint64_t list_key(const PermList<S>& N, int p, int k) {
  return N.key_at(p, k);
}

// Descent decision: is site s, at squared distance d, strictly closer than
// the current site cur, at dcur? float32 outside the guard band; inside it the
// coordinates are loaded and the distances compared in float64, in the
// oracle's order.
__device__ __forceinline__ bool strictly_closer_at(const CloudDev& C, float qx, float qy, float qz,
                                                   float d, int s, float dcur, int cur) {
  if (dcur >= kTiny) {
    if (d < dcur * (1.f - kGuard)) return true;
    if (d > dcur * (1.f + kGuard)) return false;
  } else if (d > 2.f * kTiny) {
    return false;
  }
  const float4 ps = __ldg(C.pts + s), pc = __ldg(C.pts + cur);
  return sqd64(qx, qy, qz, ps.x, ps.y, ps.z) < sqd64(qx, qy, qz, pc.x, pc.y, pc.z);
}

// Two consecutive entries of the inlined table (the first at an even index)
// in one 32-byte load.
__device__ __forceinline__ void load_pair(const float4* p, float4& a, float4& b) {
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
      : "l"(p));
}

// Algorithms 1 and 2 for the 32 queries of a warp, one per lane, in two
// alternating phases.
//
// Scan: every lane with nothing to do reads its row two entries at a time
// and stops at the first pair with something to do: an entry that passes
// the float32 bound thr (descent: it may be strictly closer; expansion: it
// may be below the k-th key), or the row's end. Event: all such lanes act
// together - the hit is decided exactly and inserted, the descent moves, the
// next list not yet expanded is opened.
//
// Why two phases: the kernel is bound by instruction issue and divergence.
// With one loop over entries (test, insertion and row switch in every
// iteration) a warp of the 4M-query torus batch ran the insertion code in
// 72% of its 586 iterations with about 7 lanes in it, and 10.3 of 32 lanes
// were active per instruction. Waiting until two thirds of the lanes have
// something to do runs the event code about 190 times with 16 or more
// lanes. A third to three quarters of the lanes measure within 5% of each
// other; a bounded number of scan steps keeps the waiting lanes from
// standing by while one lane reads a list of thousands (plan of 12 clouds:
// 4.50 ms with 8 steps, 5.97 ms unbounded; 3 / 5 / 8 / 16 steps on the
// torus batch: 6.19 / 6.07 / 6.04 / 6.05 ms). Lists of up to 16 vote on it
// every second step (6.04 to 5.97 ms; with longer lists, where fewer warps
// are resident, 2.53 to 2.60 ms at k = 32).
//
// Why pairs: entries come from the inlined table (site and rank in 16
// bytes), two in one 32-byte load at an even index, the next pair in flight
// while the current one is tested: half the load instructions and half the
// L1 lines touched (8,700 to 4,600 per warp; L1 takes about one line per
// cycle). A pair may begin before the row (skip) or reach past its end.
//
// 4M queries, 1M-site torus, k = 16: 9.12 ms with the one-loop form, 5.97 ms
// now; 1M queries, 300k-site bumpy sphere, k = 4: 0.98 to 0.58 ms. What binds
// now is latency: most pairs come from L2, and a row switch is two dependent
// loads. Loading the next pair only after a hit is decided (four registers
// fewer) takes 6.84 ms; asking for a moved-to row's bounds before the
// insertion (two registers more, spills) 6.21 ms; prefetching a row's second
// pair, or every next one, to L1 6.10 and 6.55 ms.
//
// DEFER (a cloud with box trees over its long lists, hub_of not NULL): a
// query gives up, with nothing written (the function returns true), when it
// would read a list with a tree through - the expansion of such a list, or
// a descent that finds no strictly closer entry among its first
// kHubScanFirst - so that the one-warp kernel, which walks the tree
// instead, answers it; the queries that never meet such a list (most of
// them) stay on one lane.
//
// Called by the whole warp; lanes without a query pass live = false.
template <class L, bool DEFER = false>
__device__ __forceinline__ bool knn_query_smem(const CloudDev& C, bool live, float qx, float qy,
                                               float qz, int k, int m, uint64_t* col,
                                               int32_t* __restrict__ out_idx,
                                               float* __restrict__ out_d2, int32_t row) {
  // a lane's event: hits of its last pair still to be decided, the end of
  // its row (handled once no hit is left); kIdle alone: no query (any more)
  constexpr uint32_t kHit0 = 1u, kHit1 = 2u, kRowEnd = 4u, kIdle = 8u;
  constexpr int kScanSteps = 8;
  L N;
  N.init(col, k);
  float dcur = sqd32(qx, qy, qz, __ldg(C.pts));
  N.insert(lane_key(dcur, 0), k);
  float thr = dcur >= kTiny ? dcur * (1.f + kGuard) : 2.f * kTiny;
  int cur = 0;         // the descent's current site, -1 once it is over
  // (its coordinates are loaded only for a float64 recheck, which is rare)
  bool gave_up = false;
  bool cut = false;    // DEFER: the current list has a tree and its scan stops early
  uint32_t ev = kIdle;
  int e = 0, end = 0, skip = 0;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
  float d0 = 0.f, d1 = 0.f;
  int s0 = 0, s1 = 0;
  int open = live ? 0 : -1;  // the site whose list is read next
  uint32_t act = __ballot_sync(0xffffffffu, live);
  const auto open_row = [&]() {
    int2 rr = __ldg(C.rows + open);
    if constexpr (DEFER) {
      cut = false;
      if (__ldg(C.hub_of + open) >= 0) {
        cut = rr.y > rr.x + kHubScanFirst;
        rr.y = min(rr.y, rr.x + kHubScanFirst);
      }
    }
    end = rr.y;
    e = rr.x & ~1;
    open = -1;
    ev = kRowEnd;
    if (rr.x < end) {
      load_pair(C.ent + e, a, b);
      skip = rr.x & 1;
      ev = 0u;
    }
  };
  if (open >= 0) open_row();
  while (act) {
    const int na = __popc(act);
    for (int step = 0; step < kScanSteps; step += L::kVoteEvery) {
      const uint32_t waiting = __ballot_sync(0xffffffffu, ev != 0u) & act;
      if (3 * __popc(waiting) >= 2 * na) break;
#pragma unroll
      for (int t = 0; t < L::kVoteEvery; ++t)
        if (ev == 0u) {
          d0 = sqd32(qx, qy, qz, a);
          d1 = sqd32(qx, qy, qz, b);
          s0 = __float_as_int(a.w);
          s1 = __float_as_int(b.w);
          const bool more = e + 2 < end && s1 < m;
          if (!skip && s0 < m && !(d0 > thr)) ev = kHit0;
          skip = 0;
          if (e + 1 < end && s1 < m && !(d1 > thr)) ev |= kHit1;
          if (more) {
            e += 2;
            load_pair(C.ent + e, a, b);
          } else {
            ev |= kRowEnd;
          }
        }
    }
    if (ev != 0u && ev != kIdle) {
      if (ev & (kHit0 | kHit1)) {
        const bool first = ev & kHit0;
        const float d = first ? d0 : d1;
        const int s = first ? s0 : s1;
        ev &= first ? ~kHit0 : ~kHit1;
        const uint64_t key = lane_key(d, s);
        bool offer = true;
        if (cur >= 0) {
          offer = strictly_closer_at(C, qx, qy, qz, d, s, dcur, cur);
          if (offer) {
            dcur = d;
            cur = s;
            open = s;
            ev = 0u;
            thr = dcur >= kTiny ? dcur * (1.f + kGuard) : 2.f * kTiny;
          }
        }
        if (offer && key < N.worst) {
          N.insert(key, k);
          if (cur < 0) thr = __uint_as_float((uint32_t)(N.worst >> 32));
        }
      }
      if (ev == kRowEnd) {
        bool stop = false;
        if constexpr (DEFER) {
          if (cut) stop = !((e + 1 < end ? s1 : s0) >= m);  // the descent's scan was cut short
        }
        if (!stop) {
          cur = -1;
          thr = __uint_as_float((uint32_t)(N.worst >> 32));
          open = N.next(k);
          if constexpr (DEFER) {
            if (open >= 0 && __ldg(C.hub_of + open) >= 0) stop = true;
          }
        }
        if (DEFER && stop) {
          gave_up = true;
          open = -1;
        }
        if (open < 0) ev = kIdle;
      }
      if (open >= 0) open_row();
    }
    act = __ballot_sync(0xffffffffu, ev != kIdle);
  }
  if (!live || gave_up) return gave_up;
  // the output row is addressed only now, from its 32-bit index (fewer
  // registers held through the loop); streaming stores, so that the rows
  // written do not push successor entries out of L2; four values per
  // 16-byte store when k is a multiple of 4 and both arrays are 16-byte
  // aligned (then every row is), else one value per store
  int32_t* oi = out_idx + (int64_t)row * k;
  float* od = out_d2 + (int64_t)row * k;
  const bool vec = ((k & 3) == 0) &&
                   ((((uintptr_t)out_idx) | ((uintptr_t)out_d2)) & 15) == 0;
  if (vec) {
    for (int p = 0; p < k; p += 4) {
      int iv[4];
      float dv[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint64_t key = list_key(N, p + t, k);
        const bool real = key != kPadKey;
        iv[t] = real ? (int32_t)((uint32_t)key - 1u) : -1;
        dv[t] = real ? __uint_as_float((uint32_t)(key >> 32)) : __int_as_float(0x7f800000);
      }
      __stcs(reinterpret_cast<int4*>(oi + p), make_int4(iv[0], iv[1], iv[2], iv[3]));
      __stcs(reinterpret_cast<float4*>(od + p), make_float4(dv[0], dv[1], dv[2], dv[3]));
    }
  } else {
    for (int p = 0; p < k; ++p) {
      const uint64_t key = list_key(N, p, k);
      const bool real = key != kPadKey;
      __stcs(oi + p, real ? (int32_t)((uint32_t)key - 1u) : -1);
      __stcs(od + p, real ? __uint_as_float((uint32_t)(key >> 32)) : __int_as_float(0x7f800000));
    }
  }
  return false;
}

// Slots of a thread's list column for k: 8 for k <= 8, 16 for k <= 16 (the
// lists search a power-of-two size), k above.
__host__ __device__ __forceinline__ int list_slots(int k) { return k <= 8 ? 8 : (k <= 16 ? 16 : k); }

// ---------------------------------------------------------------------------
// One warp per query with the candidate list N in shared memory (for large
// k, where one list per thread would leave a few warps per SM, and for
// launches with few queries). The list is the warp's KC keys (KC = 32, 64 or
// 128 >= k), ascending, pads in the unused positions; lane l owns positions
// l + 32 j. A key is the distance's bits above twice the rank; its lowest
// bit, set once the entry's list has been expanded, moves with it and does
// not change its place in the order. Pads have it set.
__device__ __forceinline__ uint64_t warp_key(float d, int s) {
  return pack_key(d, (uint32_t)s << 1);
}

template <int KC>
struct WarpList {
  static constexpr int J = KC / 32;
  uint64_t* L;          // the warp's KC keys in shared memory
  int from;             // every entry before this position has been expanded
  uint64_t worst;       // key of position k-1 (a pad while fewer than k entries)

  __device__ __forceinline__ void init(uint64_t* list, int lane) {
    L = list;
    from = 0;
#pragma unroll
    for (int j = 0; j < J; ++j) L[lane + 32 * j] = kPadKey;
    worst = kPadKey;
    __syncwarp();
  }
  __device__ __forceinline__ uint32_t low(int p) const { return ((const uint32_t*)L)[2 * p]; }
  __device__ __forceinline__ uint32_t high(int p) const { return ((const uint32_t*)L)[2 * p + 1]; }
  // Marks the nearest entry among the first k-1 not yet expanded and returns
  // its site, or -1 (the same in every lane).
  __device__ __forceinline__ int next(int k, int lane) {
    for (int p0 = from & ~31; p0 < k - 1; p0 += 32) {
      const uint32_t lo = low(p0 + lane);
      const uint32_t open = __ballot_sync(0xffffffffu, p0 + lane < k - 1 && !(lo & 1u));
      if (open == 0u) continue;
      const int w = __ffs((int)open) - 1;
      if (lane == w) ((uint32_t*)L)[2 * (p0 + lane)] = lo | 1u;
      from = p0 + w + 1;
      __syncwarp();
      return (int)(__shfl_sync(0xffffffffu, lo, w) >> 1);
    }
    from = k - 1;
    return -1;
  }
  // is key c (c < worst) in the list? pos: the number of keys below c
  // (called by any subset of lanes). The halving steps compare distances
  // alone: one word and one comparison each.
  __device__ __forceinline__ bool contains(uint64_t c, int& pos) const {
    const uint32_t ch = (uint32_t)(c >> 32), cl = (uint32_t)c;
    pos = 0;
#pragma unroll
    for (int step = KC / 2; step >= 1; step >>= 1)
      if (high(pos + step - 1) < ch) pos += step;
    uint32_t l = low(pos);
    if (high(pos) != ch) return false;
    while (l < cl) {  // equal distances in rank order; ends at the k-th key at the latest
      l = low(++pos);
      if (high(pos) != ch) return false;
    }
    return (l | 1u) == (cl | 1u);
  }
  // Merges the lanes' keys with `fresh` set (not in the list; positions from
  // contains) into the list in one pass: each key goes to its position plus
  // the number of fresh keys below it, each entry moves up by the number of
  // fresh keys below it, and what reaches position k drops out. Called by the
  // whole warp, with no two fresh keys equal.
  __device__ __forceinline__ void merge(bool fresh, uint64_t key, int pos, int k, int lane) {
    uint32_t b = __ballot_sync(0xffffffffu, fresh);
    if (b == 0u) return;
    int up[J], below = 0, lowest = KC;
#pragma unroll
    for (int j = 0; j < J; ++j) up[j] = 0;
    do {
      const int f = __ffs((int)b) - 1;
      const uint64_t kf = __shfl_sync(0xffffffffu, key, f);
      const int pf = __shfl_sync(0xffffffffu, pos, f);
      b &= b - 1u;
      below += kf < key ? 1 : 0;
      lowest = min(lowest, pf);
#pragma unroll
      for (int j = 0; j < J; ++j) up[j] += pf <= lane + 32 * j ? 1 : 0;
    } while (b);
    uint64_t v[J];
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (32 * j + 31 >= lowest) v[j] = L[lane + 32 * j];
    __syncwarp();  // every lane has read its entries
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (32 * j + 31 >= lowest) {
        const int p = lane + 32 * j + up[j];
        if (up[j] && p < k) L[p] = v[j];
      }
    if (fresh && pos + below < k) L[pos + below] = key;
    __syncwarp();
    from = min(from, lowest);
    worst = L[k - 1];
  }
  // Inserts key c (the same in every lane) unless present.
  __device__ __forceinline__ void insert(uint64_t c, int k, int lane) {
    int pos = 0;
    if (!(c < worst) || contains(c, pos)) return;
    merge(lane == 0, c, pos, k, lane);
  }
};

// The descent's sites: lane t holds the key of the t-th one. Each is closer
// than all before it, so they become the list in reverse, with no search and
// no shift; when they do not come in that order (float32 near-ties) or are
// more than 32, they go to the list and the rest is inserted there.
template <int KC>
struct DescentKeys {
  uint64_t mine, last;
  int n;  // keys held, or -1 once they are in the list

  __device__ __forceinline__ void add(uint64_t c, WarpList<KC>& N, int k, int lane) {
    if (n >= 0 && (n == 32 || (n > 0 && c >= last))) flush(N, k, lane);
    if (n < 0) {
      N.insert(c, k, lane);
      return;
    }
    if (lane == n) mine = c;
    last = c;
    ++n;
  }
  __device__ __forceinline__ void flush(WarpList<KC>& N, int k, int lane) {
    if (n < 0) return;
    const uint64_t c = __shfl_sync(0xffffffffu, mine, (n - 1 - lane) & 31);
    if (lane < min(n, k)) N.L[lane] = c;
    __syncwarp();
    N.worst = N.L[k - 1];
    n = -1;
  }
};

// Box trees over long lists (one warp; every lane passes the same arguments).

// Node count of one level of a tree over len entries, and the level's
// offset from the tree's first node (the chunks' level first).
__device__ __forceinline__ void hub_level_of(int len, int level, int& off, int& cnt) {
  int c = (len + 31) >> 5, o = 0;
  for (int l = 0; l < level; ++l) {
    o += c;
    c = (c + 31) >> 5;
  }
  off = o;
  cnt = c;
}

// Squared distance from q to the box [lo, hi] with sqd32's operations,
// applied to per-axis gaps that are never larger in magnitude than the gap
// to any point of the box. Subtraction, product and fused add are monotonic
// under round-to-nearest, so the result is at most sqd32(q, p) for every
// site p in the box: no rounding can make a box look farther than a site
// inside it.
__device__ __forceinline__ float box_sqd32(float qx, float qy, float qz, float4 lo, float4 hi) {
  const float dx = qx < lo.x ? __fsub_rn(qx, lo.x) : (qx > hi.x ? __fsub_rn(qx, hi.x) : 0.f);
  const float dy = qy < lo.y ? __fsub_rn(qy, lo.y) : (qy > hi.y ? __fsub_rn(qy, hi.y) : 0.f);
  const float dz = qz < lo.z ? __fsub_rn(qz, lo.z) : (qz > hi.z ? __fsub_rn(qz, hi.z) : 0.f);
  float d = __fmul_rn(dx, dx);
  d = __fmaf_rn(dy, dy, d);
  d = __fmaf_rn(dz, dz, d);
  return d;
}

// Depth-first walk of tree D. The children of a node are rated one per lane
// with rate(low, high): a priority below 0xffffffff for a child that may
// hold an entry of interest (the smaller, the sooner it is entered), else
// 0xffffffff. The kept children of each level wait in a bit mask, their
// priorities in the warp's shared memory; the one with the smallest
// priority is entered next if still(priority) holds then (the bounds
// tighten as chunks are handled), and a kept chunk (level 0) goes to
// leaf(chunk). Every decision is the same in all lanes, so the warp stays
// converged. stack: kHubStackWords 32-bit words of the warp's shared memory.
template <class Rate, class Still, class Leaf>
__device__ __forceinline__ void hub_walk(const CloudDev& C, int4 D, int lane, uint32_t* stack,
                                         Rate&& rate, Still&& still, Leaf&& leaf) {
  const int len = D.y, node0 = D.z, top = D.w - 1;
  // per level: the children not entered yet (pend), the index of their
  // first (first), and each child's priority (prio, one per lane)
  uint32_t* pend = stack;
  uint32_t* first = stack + kHubMaxLevels;
  uint32_t* prio = stack + 2 * kHubMaxLevels;
  int l = top, off, cnt;
  hub_level_of(len, l, off, cnt);
  uint32_t pr = 0xffffffffu;
  if (lane < cnt) {
    const int j = node0 + off + lane;
    pr = rate(__ldg(C.hub_node + 2 * j), __ldg(C.hub_node + 2 * j + 1));
  }
  prio[32 * l + lane] = pr;
  pend[l] = __ballot_sync(0xffffffffu, pr != 0xffffffffu);
  first[l] = 0;
  __syncwarp();
  for (;;) {
    const uint32_t pm = pend[l];
    if (pm == 0u) {
      if (++l > top) break;
      continue;
    }
    const uint32_t mine = ((pm >> lane) & 1u) ? prio[32 * l + lane] : 0xffffffffu;
    const uint32_t low = __reduce_min_sync(0xffffffffu, mine);
    const int c = __ffs((int)__ballot_sync(0xffffffffu, mine == low)) - 1;
    pend[l] = pm & ~(1u << c);
    const int node = (int)first[l] + c;
    if (!still(low)) continue;
    if (l == 0) {
      leaf(node);
      continue;
    }
    --l;
    hub_level_of(len, l, off, cnt);
    const int ch = 32 * node + lane;
    pr = 0xffffffffu;
    if (ch < cnt) {
      const int jc = node0 + off + ch;
      pr = rate(__ldg(C.hub_node + 2 * jc), __ldg(C.hub_node + 2 * jc + 1));
    }
    __syncwarp();  // every lane has read this level's old priorities
    prio[32 * l + lane] = pr;
    pend[l] = __ballot_sync(0xffffffffu, pr != 0xffffffffu);
    first[l] = (uint32_t)(32 * node);
    __syncwarp();
  }
}

// Algorithm 1's step on a list with a tree: the lowest rank below m whose
// site is strictly closer than the current one (rank cur, squared distance
// dcur) - the first such entry of the list in rank order - or -1; its
// squared distance goes to bd. A box is skipped when its nearest point is
// beyond the float32 distance above which strictly_closer_at says no, or its
// smallest rank is not below m or below the best found.
__device__ __forceinline__ int hub_first_closer(const CloudDev& C, int hub, float qx, float qy,
                                                float qz, float dcur, int cur, int m, int lane,
                                                uint32_t* stack, float& bd) {
  const int4 D = __ldg(C.hub_desc + hub);
  const float reach = dcur >= kTiny ? dcur * (1.f + kGuard) : 2.f * kTiny;
  int best = 0x7fffffff;
  float bestd = 0.f;
  hub_walk(
      C, D, lane, stack,
      [&](float4 lo, float4 hi) {
        const int r = __float_as_int(lo.w);
        return (r < m && r < best && !(box_sqd32(qx, qy, qz, lo, hi) > reach)) ? (uint32_t)r
                                                                               : 0xffffffffu;
      },
      [&](uint32_t r) { return (int)r < best; },
      [&](int chunk) {
        const float4 ps = __ldg(C.hub_ent + D.x + 32 * chunk + lane);
        const int s = __float_as_int(ps.w);  // pads: 0x7fffffff, never below m
        const float d = sqd32(qx, qy, qz, ps);
        const bool cl = s < m && s < best && strictly_closer_at(C, qx, qy, qz, d, s, dcur, cur);
        const int low = __reduce_min_sync(0xffffffffu, cl ? s : 0x7fffffff);
        if (low < best) {
          const int w = __ffs((int)__ballot_sync(0xffffffffu, cl && s == low)) - 1;
          best = low;
          bestd = __shfl_sync(0xffffffffu, d, w);
        }
      });
  bd = bestd;
  return best == 0x7fffffff ? -1 : best;
}

// Algorithm 2's offer of a list with a tree: every entry below m whose key
// is below the k-th key of N goes to N. A box is skipped when its nearest
// point is farther than the k-th key's distance (the pad key's distance is
// a NaN, which skips nothing) or its smallest rank is not below m. N ends
// as after the scan in rank order: the k smallest keys of N and the list.
template <int KC>
__device__ __forceinline__ void hub_offer(const CloudDev& C, int hub, float qx, float qy,
                                          float qz, int m, int k, WarpList<KC>& N, int lane,
                                          uint32_t* stack) {
  const int4 D = __ldg(C.hub_desc + hub);
  hub_walk(
      C, D, lane, stack,
      [&](float4 lo, float4 hi) {
        const float wd = __uint_as_float((uint32_t)(N.worst >> 32));
        const float bd = box_sqd32(qx, qy, qz, lo, hi);
        return (__float_as_int(lo.w) < m && !(bd > wd)) ? __float_as_uint(bd) : 0xffffffffu;
      },
      [&](uint32_t d) { return !(__uint_as_float(d) > __uint_as_float((uint32_t)(N.worst >> 32))); },
      [&](int chunk) {
        const float4 ps = __ldg(C.hub_ent + D.x + 32 * chunk + lane);
        const int s = __float_as_int(ps.w);
        const float d = sqd32(qx, qy, qz, ps);
        const uint64_t key = warp_key(d, s);
        int pos = 0;
        const bool fresh = s < m && key < N.worst && !N.contains(key, pos);
        N.merge(fresh, key, pos, k, lane);
      });
}

// 32-bit words of a warp's tree-walk stack: per level a mask, a first
// index and 32 priorities.
constexpr int kHubStackWords = 34 * kHubMaxLevels;
// 64-bit words of shared memory for one warp of knn_query_warp<KC>.
__host__ __device__ constexpr int kWarpListWords(int kc) { return kc + kHubStackWords / 2; }

// Resident 256-thread blocks per SM that the one-warp kernels are held to.
// Five (48 registers) hide more latency in large launches, four (64) run the
// single query faster; us with 4 / 5 blocks: 100,000 queries at k = 100 2530 /
// 2402, 64 queries 105 / 125; on a 300k-site torus 100,000 queries at k = 64
// 1532 / 1348, at k = 16 550 / 477, 64 queries the same; with trees, k = 32,
// 10,000 queries 276 / 292, 60,000 609 / 546.
// The bound costs spills (ptxas -v: 0 to 68 bytes in the plain kernels, 52 to
// 192 in the persistent and hand-over kernels, which keep the request too);
// left alone the latter take 64 to 104 registers and are slower but for small
// launches with trees. Plans on a 300k-site torus, us held / left alone:
// 20,000 queries at k = 8 88 / 92, k = 64 346 / 425, k = 128 721 / 826; 300,000
// at k = 32 on one warp each 2005 / 2188, k = 64 4027 / 5146, k = 100 7165 /
// 8350; on a 200k-site patch cloud with trees 20,000 at k = 8 202 / 189, k = 32
// 302 / 283, k = 100 802 / 1072; 60,000 at k = 32 605 / 715; 300,000 at k = 100
// 9958 / 13872; with the hand-over, 300,000 at k = 8 758 / 772.
constexpr int kWarpBlocks(int kc, bool trees) { return (kc == 128 || trees) ? 4 : 5; }

// One query by one warp (every lane calls it with the same query). The
// descent reads its list 32 entries at a time; the first strictly closer
// entry in list order is the lowest lane that votes closer. In the expansion
// each lane whose entry falls below the k-th key searches N for it, all at
// once (most are already in N: at k = 100, 781 of 948 per query on the 1M
// torus), and the new ones are merged in one pass.
//
// The kernel is bound by instruction issue. With each new key inserted by
// itself (the tail moved and four flag words shifted every time) and every
// site of the descent searched for its place, a query took 40k warp
// instructions at k = 100; 100,000 surface queries on the 1M torus took 4.01
// ms, 2.53 now; 10,007 queries at k = 8 79 us with the sort, 52 now (with
// the one-block sort); 64 queries 19 us, 15 now (there the chain of dependent loads binds: the next
// list's bounds are asked for before the site is put into the list). Reading
// the lists of two sites at once, 16 lanes each, took 2.36 ms at k = 100 and
// was slower up to k = 16; it can expand a site that would have dropped out
// by its turn, which changes rows whose distances all tie within float32
// rounding, so lists are read one at a time.
//
// With TREES (a cloud whose hub_of is not NULL) a list with a box tree is
// searched through the tree (after kHubScanFirst entries in the descent);
// the result is the same as the scan's. The walk's code costs registers
// and issue slots in the scan loop too, so clouds without trees run the
// instantiation without it. list: the warp's kWarpListWords(KC) words of
// shared memory (KC keys, then the tree walk's stack).
template <int KC, bool TREES>
__device__ __forceinline__ void knn_query_warp(const CloudDev& C, float qx, float qy, float qz,
                                               int k, int m, uint64_t* list,
                                               int32_t* __restrict__ out_idx,
                                               float* __restrict__ out_d2, int32_t row) {
  const int lane = (int)(threadIdx.x & 31u);
  const float4 kNone = make_float4(0.f, 0.f, 0.f, __int_as_float(0x7fffffff));
  WarpList<KC> N;
  N.init(list, lane);

  // ---- Algorithm 1
  {
    DescentKeys<KC> T;
    T.n = 0;
    T.mine = T.last = kPadKey;
    int2 rr = __ldg(C.rows);
    int hub = -1;  // the current list's tree, or -1
    if constexpr (TREES) hub = __ldg(C.hub_of);
    float dcur = sqd32(qx, qy, qz, __ldg(C.pts));
    int cur = 0;
    T.add(warp_key(dcur, 0), N, k, lane);
    uint32_t base = rr.x;  // unsigned: base + 63 does not overflow
    for (;;) {
      int to = -1;  // the site moved to
      float dto = 0.f;
      bool over = base >= (uint32_t)rr.y;
      if (TREES && hub >= 0 && (int)base - rr.x >= kHubScanFirst) {
        to = hub_first_closer(C, hub, qx, qy, qz, dcur, cur, m, lane, (uint32_t*)(list + KC), dto);
        over = true;
      } else if (!over) {
        const uint32_t e = base + lane;
        const float4 ps = e < (uint32_t)rr.y ? __ldg(C.ent + e) : kNone;
        const int s = __float_as_int(ps.w);
        const float d = sqd32(qx, qy, qz, ps);
        // rows ascend: past the first s >= m nothing is below m
        const bool cl = s < m && strictly_closer_at(C, qx, qy, qz, d, s, dcur, cur);
        const uint32_t b = __ballot_sync(0xffffffffu, cl);
        over = base + 32 >= (uint32_t)rr.y || __any_sync(0xffffffffu, s >= m);
        if (b) {
          const int w = __ffs((int)b) - 1;
          to = __shfl_sync(0xffffffffu, s, w);
          dto = __shfl_sync(0xffffffffu, d, w);
        }
        base += 32;
      }
      if (to >= 0) {
        rr = __ldg(C.rows + to);
        if constexpr (TREES) hub = __ldg(C.hub_of + to);
        cur = to;
        dcur = dto;
        T.add(warp_key(dto, to), N, k, lane);
        base = rr.x;
      } else if (over) {
        break;
      }
    }
    T.flush(N, k, lane);
  }

  // ---- Algorithm 2
  for (;;) {
    const int site = N.next(k, lane);
    if (site < 0) break;
    if constexpr (TREES) {
      const int hub = __ldg(C.hub_of + site);
      if (hub >= 0) {
        hub_offer(C, hub, qx, qy, qz, m, k, N, lane, (uint32_t*)(list + KC));
        continue;
      }
    }
    const int2 rr = __ldg(C.rows + site);
    const uint32_t end = rr.y;
    for (uint32_t e = rr.x + lane, base = rr.x; base < end; base += 32, e += 32) {
      const float4 ps = e < end ? __ldg(C.ent + e) : kNone;
      const int s = __float_as_int(ps.w);
      const float d = sqd32(qx, qy, qz, ps);
      const uint64_t key = warp_key(d, s);
      int pos = 0;
      const bool fresh = s < m && key < N.worst && !N.contains(key, pos);
      // the list's end, or its first entry out of the prefix
      const bool over = __any_sync(0xffffffffu, s >= m);
      N.merge(fresh, key, pos, k, lane);
      if (over) break;
    }
  }
  int32_t* oi = out_idx + (int64_t)row * k;
  float* od = out_d2 + (int64_t)row * k;
#pragma unroll
  for (int j = 0; j < KC / 32; ++j) {
    const int p = lane + 32 * j;
    if (p < k) {
      const uint64_t key = N.L[p];
      const bool real = key != kPadKey;
      __stcs(oi + p, real ? (int32_t)((uint32_t)key >> 1) : -1);
      __stcs(od + p, real ? __uint_as_float((uint32_t)(key >> 32)) : __int_as_float(0x7f800000));
    }
  }
  __syncwarp();
}

// Writes a padded row (-1, +inf) for a query that cannot be served.
template <int G>
__device__ __forceinline__ void pad_row(const Grp<G>& g, int k, int32_t* oi, float* od) {
  for (int p = (int)g.lane; p < k; p += G) {
    oi[p] = -1;
    od[p] = __int_as_float(0x7f800000);
  }
}

}  // namespace mknn
