// sample_device.cuh — device code for drawing one wedge and checking its
// closure (Sec. 3.2, Alg. Phase 3b), shared by the single-graph sampler and
// the batched persistent sampler. Two mappings:
//   thread: one thread draws one wedge; the centre from a guide, the row searched by interpolation.
//   warp:   the 32 lanes of a warp draw one wedge together; 33-way searches
//           (each step probes 32 positions at once), so a search of length n
//           takes about log33(n) dependent steps instead of log2(n).
// Both mappings produce the same wedge for the same (seed, stream, index).
#pragma once

#include "device.cuh"
#include "internal.h"

namespace wedge {

// One sampling stream: a bin of one graph (tag 0) or all of its wedges (tag 1).
// n, n_adj, n_L, n_guide and err are read only by the bounds-checked debug build
// (err == nullptr: unchecked).
struct GraphView {
  const int64_t* off;
  const int32_t* adj;
  const int32_t* L;
  const uint64_t* W;
  const uint32_t* guide;
  float ids_inv;  // 1 / n
  int64_t n = 0;
  int64_t n_adj = 0;
  int64_t n_L = 0;
  int64_t n_guide = 0;
  uint32_t* err = nullptr;
};

// u / d, in 32 bits where both fit (the degrees of all but the largest hubs):
// a 64-bit division is several times the instructions.
__device__ __forceinline__ uint64_t div_small(uint64_t u, uint64_t d) {
  if (((u | d) >> 32) == 0) return (uint32_t)u / (uint32_t)d;
  return u / d;
}

struct Wedge {
  int32_t v0, v1, v2;
  int64_t d0, d1, d2;
  bool closed;
};

// ---------------------------------------------------------------- thread --

// One aligned 32-byte sector (eight ids) in one load: a warp's loads from 32
// random places take as long as the sectors they touch, so a search that reads
// a sector per load reads eight ids for the price of one.
struct Sector {
  int32_t e[8];
};
__device__ __forceinline__ Sector load_sector(const int32_t* p) {
  Sector s;
  asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(s.e[0]), "=r"(s.e[1]), "=r"(s.e[2]), "=r"(s.e[3]), "=r"(s.e[4]), "=r"(s.e[5]), "=r"(s.e[6]),
                 "=r"(s.e[7])
               : "l"(p));
  return s;
}

// Search of x in an ascending row of adj. First by sectors, each where x would
// be if the ids were spread evenly: over [0, n) at first, then counted from the
// last sector read, which for ids without structure lands within a sector or
// two of the place. After a step that is sent further than even ids would send
// it, or the third, what is left is halved entry by entry (`lost` says so: a
// warp that often loses its guesses does better without). Rows of a thousand
// even ids take two sectors outside the caches, a binary search six or seven.
// The phases are loops of their own, so that the lanes of a warp do the same
// thing at the same time. With the binary search in its place the sampling
// kernel took 2.98 ms on Kronecker scale 24 (15.2 M samples) and 0.60 ms on
// scale 14 with unpermuted, skewed ids; with this one and the guide over W
// 1.35 and 0.47 ms.
struct RowSearch {
  const int32_t* p;     // adj from the sector in which the row starts
  uint32_t first, end;  // the row's entries, from p
  uint32_t l, h;        // entries not yet ruled out
  uint32_t g;           // guessed entry
  int32_t x;
  int32_t tries;        // sectors by interpolation left
  float rate;           // entries per id
  bool found, lost;

  // ids_inv: 1 / n. Rows start at any entry; adj is allocated in whole sectors.
  __device__ __forceinline__ void start(const int32_t* __restrict__ adj, int64_t lo, int64_t d, int32_t id,
                                        float ids_inv, bool guess) {
    const int64_t a0 = lo & ~int64_t(7);
    p = adj + a0;
    first = (uint32_t)(lo - a0);
    end = first + (uint32_t)d;  // d < 2^31
    l = first;
    h = end;
    x = id;
    tries = guess ? 3 : 0;
    rate = (float)d * ids_inv;
    found = lost = false;
    g = clamp((float)first + (float)id * rate);
  }
  __device__ __forceinline__ uint32_t clamp(float at) const {
    return max(l, min(h - 1u, __float2uint_rz(at)));  // (what is outside the range converts to its nearer end)
  }
  __device__ __forceinline__ bool open() const { return l < h; }
  __device__ __forceinline__ bool guessing() const { return l < h && tries > 0; }
  __device__ __forceinline__ Sector load() const { return load_sector(p + (g & ~7u)); }
  // Rules out what g's sector shows; the next g by interpolation.
  __device__ __forceinline__ void look(const Sector& q) {
    const uint32_t s = g & ~7u;
    bool after, before;
    if (s >= first && s + 8u <= end) {
      found = q.e[0] == x || q.e[1] == x || q.e[2] == x || q.e[3] == x || q.e[4] == x || q.e[5] == x || q.e[6] == x ||
              q.e[7] == x;
      after = x > q.e[7];
      before = x < q.e[0];
    } else {  // only some of its entries belong to the row
      uint32_t in = 0xffu, eq = 0, lt = 0;
      if (s < first) in &= 0xffu << (first - s);
      if (s + 8u > end) in &= 0xffu >> (s + 8u - end);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        eq |= (uint32_t)(q.e[k] == x) << k;
        lt |= (uint32_t)(q.e[k] < x) << k;
      }
      found = (eq & in) != 0;
      after = (lt & in) == in;
      before = (lt & in) == 0;
    }
    if (found || !(after || before)) {
      h = l;
      return;
    }
    const float away = (float)(after ? x - q.e[7] : q.e[0] - x) * rate;  // entries to the place, for even ids
    if (after) l = s + 8u;
    else h = max(s, first);
    g = clamp(after ? (float)l + away : (float)h - away);
    tries = away > 8.0f + 0.0625f * (float)(end - first) ? 0 : tries - 1;
    lost = tries == 0;
  }
  __device__ __forceinline__ uint32_t middle() const { return l + ((h - l) >> 1); }
  __device__ __forceinline__ void look_middle(int32_t y) {  // the entry at middle()
    const uint32_t m = middle();
    found = y == x;
    if (y < x) l = m + 1u;
    else h = found ? l : m;
  }
};

// guess: whether to guess; false on return if that was no use.
__device__ __forceinline__ bool row_contains(const int32_t* __restrict__ adj, int64_t lo, int64_t d, int32_t x,
                                             float ids_inv, bool& guess) {
  RowSearch r;
  r.start(adj, lo, d, x, ids_inv, guess);
  while (r.guessing()) r.look(r.load());
  while (r.open()) r.look_middle(__ldg(r.p + r.middle()));
  guess = guess && !r.lost;
  return r.found;
}

// Two searches in step: the loads of a step are issued before either is used.
__device__ __forceinline__ void row_contains2(RowSearch& a, RowSearch& b) {
  while (a.guessing() || b.guessing()) {
    const bool ra = a.guessing(), rb = b.guessing();
    Sector qa{}, qb{};
    if (ra) qa = a.load();
    if (rb) qb = b.load();
    if (ra) a.look(qa);
    if (rb) b.look(qb);
  }
  while (a.open() || b.open()) {
    const bool ra = a.open(), rb = b.open();
    const int32_t ya = ra ? __ldg(a.p + a.middle()) : 0, yb = rb ? __ldg(b.p + b.middle()) : 0;
    if (ra) a.look_middle(ya);
    if (rb) b.look_middle(yb);
  }
}

// Closure of (v1, v0, v2): search the larger-(degree, id) endpoint in the other's row.
__device__ __forceinline__ bool closed_wedge(const int32_t* __restrict__ adj, int32_t v1, int32_t v2, int64_t o1,
                                             int64_t d1, int64_t o2, int64_t d2, float ids_inv, bool& guess) {
  const bool first = d1 < d2 || (d1 == d2 && v1 < v2);
  return row_contains(adj, first ? o1 : o2, first ? d1 : d2, first ? v2 : v1, ids_inv, guess);
}

// Whether a warp goes on guessing, from its lanes' last searches (all lanes
// call it): not once a third of them lost theirs.
__device__ __forceinline__ bool warp_guesses(bool guess, bool lost) {
  return guess && __popc(__ballot_sync(FULL_MASK, lost)) <= 10;
}

// The bins a stream's centres lie in, as a range of the guide table (in shared
// memory): one bin, or all that hold vertices (the global stream).
struct GuideRange {
  const GuideBin* tab;
  uint32_t first, end;
};

// The entries of L between which the centre of wedge T lies, W[lo] <= T < W[hi]:
// the cell of T's bin, about two entries wide where degrees in a bin are alike.
__device__ __forceinline__ void centre_cell(const GraphView& g, const GuideRange& gr, uint64_t T, int64_t& lo,
                                            int64_t& hi) {
  uint32_t b = gr.first, e = gr.end;  // last bin with wlo <= T (an empty bin's wlo is the next one's)
  while (e - b > 1) {
    const uint32_t mid = (b + e) >> 1;
    if (gr.tab[mid].wlo <= T) b = mid; else e = mid;
  }
  const GuideBin t = gr.tab[b];
  const int64_t c = (int64_t)(t.at + ((T - t.wlo) >> t.shift));
  lo = checked_ldg(g.guide, c, g.n_guide, g.err);
  hi = (int64_t)checked_ldg(g.guide, c + 1, g.n_guide, g.err) + 1;
}

// Centre and endpoints (no closure) for random words r of a stream of the bins
// gr with wedge total p and prefix base wbase = W at their start; fills
// everything but closed and returns the endpoints' row starts.
__device__ __forceinline__ Wedge draw_pair_thread(const GraphView& g, const GuideRange& gr, uint64_t p, uint64_t wbase,
                                                  const Philox4& r, int64_t& o1, int64_t& o2) {
  Wedge w;
  const uint64_t t = mulhi64((uint64_t)r.r0 | ((uint64_t)r.r1 << 32), p);
  const uint64_t T = wbase + t;
  int64_t lo, hi;
  centre_cell(g, gr, T, lo, hi);
  while (hi - lo > 1) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (checked_ldg(g.W, mid, g.n_L + 1, g.err) <= T) lo = mid; else hi = mid;
  }
  w.v0 = checked_ldg(g.L, lo, g.n_L, g.err);
  const int64_t o0 = checked_ldg(g.off, w.v0, g.n + 1, g.err);
  w.d0 = checked_ldg(g.off, (int64_t)w.v0 + 1, g.n + 1, g.err) - o0;
  const uint64_t dm1 = (uint64_t)(w.d0 - 1);
  const uint64_t u = mulhi64((uint64_t)r.r2 | ((uint64_t)r.r3 << 32), (uint64_t)w.d0 * dm1);
  const uint64_t i = div_small(u, dm1);
  const uint64_t jp = u - i * dm1;
  const uint64_t j = jp + (jp >= i ? 1ULL : 0ULL);
  w.v1 = checked_ldg(g.adj, o0 + (int64_t)i, g.n_adj, g.err);
  w.v2 = checked_ldg(g.adj, o0 + (int64_t)j, g.n_adj, g.err);
  o1 = checked_ldg(g.off, w.v1, g.n + 1, g.err);
  w.d1 = checked_ldg(g.off, (int64_t)w.v1 + 1, g.n + 1, g.err) - o1;
  o2 = checked_ldg(g.off, w.v2, g.n + 1, g.err);
  w.d2 = checked_ldg(g.off, (int64_t)w.v2 + 1, g.n + 1, g.err) - o2;
  w.closed = false;
  return w;
}

// The wedge for random words r, with its closure.
__device__ __forceinline__ Wedge draw_wedge_thread(const GraphView& g, const GuideRange& gr, uint64_t p,
                                                   uint64_t wbase, const Philox4& r, bool& guess) {
  int64_t o1, o2;
  Wedge w = draw_pair_thread(g, gr, p, wbase, r, o1, o2);
  // the closure search stays inside the two rows, which must lie in adj
  const bool rows_ok = in_bounds((uint64_t)(o1 + w.d1), (uint64_t)g.n_adj + 1, g.err) &&
                       in_bounds((uint64_t)(o2 + w.d2), (uint64_t)g.n_adj + 1, g.err);
  w.closed = rows_ok && closed_wedge(g.adj, w.v1, w.v2, o1, w.d1, o2, w.d2, g.ids_inv, guess);
  return w;
}

// Two wedges of one stream drawn in lockstep by one thread: the same results
// as two draw_wedge_thread calls, with each step of the two searches issuing
// both loads before using either, so two dependent chains of random loads
// are in flight per thread instead of one. A centre search that has finished
// keeps loading a valid index (its current lower bound) until the other ends.
__device__ __forceinline__ void draw_wedge_thread2(const GraphView& g, const GuideRange& gr, uint64_t p,
                                                   uint64_t wbase, const Philox4& ra, const Philox4& rb, Wedge& wa,
                                                   Wedge& wb, bool& guess) {
  const uint64_t Ta = wbase + mulhi64((uint64_t)ra.r0 | ((uint64_t)ra.r1 << 32), p);
  const uint64_t Tb = wbase + mulhi64((uint64_t)rb.r0 | ((uint64_t)rb.r1 << 32), p);
  int64_t la, ha, lb, hb;
  centre_cell(g, gr, Ta, la, ha);
  centre_cell(g, gr, Tb, lb, hb);
  while (ha - la > 1 || hb - lb > 1) {
    const bool sa = ha - la > 1, sb = hb - lb > 1;
    const int64_t ma = sa ? la + ((ha - la) >> 1) : la;
    const int64_t mb = sb ? lb + ((hb - lb) >> 1) : lb;
    const uint64_t xa = checked_ldg(g.W, ma, g.n_L + 1, g.err), xb = checked_ldg(g.W, mb, g.n_L + 1, g.err);
    if (sa) {
      if (xa <= Ta) la = ma; else ha = ma;
    }
    if (sb) {
      if (xb <= Tb) lb = mb; else hb = mb;
    }
  }
  wa.v0 = checked_ldg(g.L, la, g.n_L, g.err);
  wb.v0 = checked_ldg(g.L, lb, g.n_L, g.err);
  const int64_t oa = checked_ldg(g.off, wa.v0, g.n + 1, g.err);
  const int64_t ob = checked_ldg(g.off, wb.v0, g.n + 1, g.err);
  wa.d0 = checked_ldg(g.off, (int64_t)wa.v0 + 1, g.n + 1, g.err) - oa;
  wb.d0 = checked_ldg(g.off, (int64_t)wb.v0 + 1, g.n + 1, g.err) - ob;
  const uint64_t dma = (uint64_t)(wa.d0 - 1), dmb = (uint64_t)(wb.d0 - 1);
  const uint64_t ua = mulhi64((uint64_t)ra.r2 | ((uint64_t)ra.r3 << 32), (uint64_t)wa.d0 * dma);
  const uint64_t ub = mulhi64((uint64_t)rb.r2 | ((uint64_t)rb.r3 << 32), (uint64_t)wb.d0 * dmb);
  const uint64_t ia = div_small(ua, dma), ib = div_small(ub, dmb);
  const uint64_t jpa = ua - ia * dma, jpb = ub - ib * dmb;
  const uint64_t ja = jpa + (jpa >= ia ? 1ULL : 0ULL), jb = jpb + (jpb >= ib ? 1ULL : 0ULL);
  wa.v1 = checked_ldg(g.adj, oa + (int64_t)ia, g.n_adj, g.err);
  wa.v2 = checked_ldg(g.adj, oa + (int64_t)ja, g.n_adj, g.err);
  wb.v1 = checked_ldg(g.adj, ob + (int64_t)ib, g.n_adj, g.err);
  wb.v2 = checked_ldg(g.adj, ob + (int64_t)jb, g.n_adj, g.err);
  const int64_t o1a = checked_ldg(g.off, wa.v1, g.n + 1, g.err);
  const int64_t o2a = checked_ldg(g.off, wa.v2, g.n + 1, g.err);
  const int64_t o1b = checked_ldg(g.off, wb.v1, g.n + 1, g.err);
  const int64_t o2b = checked_ldg(g.off, wb.v2, g.n + 1, g.err);
  wa.d1 = checked_ldg(g.off, (int64_t)wa.v1 + 1, g.n + 1, g.err) - o1a;
  wa.d2 = checked_ldg(g.off, (int64_t)wa.v2 + 1, g.n + 1, g.err) - o2a;
  wb.d1 = checked_ldg(g.off, (int64_t)wb.v1 + 1, g.n + 1, g.err) - o1b;
  wb.d2 = checked_ldg(g.off, (int64_t)wb.v2 + 1, g.n + 1, g.err) - o2b;
  const bool oka = in_bounds((uint64_t)(o1a + wa.d1), (uint64_t)g.n_adj + 1, g.err) &&
                   in_bounds((uint64_t)(o2a + wa.d2), (uint64_t)g.n_adj + 1, g.err);
  const bool okb = in_bounds((uint64_t)(o1b + wb.d1), (uint64_t)g.n_adj + 1, g.err) &&
                   in_bounds((uint64_t)(o2b + wb.d2), (uint64_t)g.n_adj + 1, g.err);
  // closure: the larger-(degree, id) endpoint searched in the other's row
  const bool a1 = wa.d1 < wa.d2 || (wa.d1 == wa.d2 && wa.v1 < wa.v2);
  const bool b1 = wb.d1 < wb.d2 || (wb.d1 == wb.d2 && wb.v1 < wb.v2);
  RowSearch sa, sb;
  sa.start(g.adj, a1 ? o1a : o2a, oka ? (a1 ? wa.d1 : wa.d2) : 0, a1 ? wa.v2 : wa.v1, g.ids_inv, guess);
  sb.start(g.adj, b1 ? o1b : o2b, okb ? (b1 ? wb.d1 : wb.d2) : 0, b1 ? wb.v2 : wb.v1, g.ids_inv, guess);
  row_contains2(sa, sb);
  guess = guess && !(sa.lost || sb.lost);
  const bool fa = sa.found, fb = sb.found;
  wa.closed = oka && fa;
  wb.closed = okb && fb;
}

// ------------------------------------------------------------------ warp --

// Largest j in [lo, hi) with W[j] <= T, given W[lo] <= T < W[hi]. Same
// result on every lane.
__device__ __forceinline__ int64_t warp_search_prefix(const uint64_t* __restrict__ W, int64_t lo, int64_t hi,
                                                      uint64_t T, int lane) {
  while (hi - lo > 33) {
    const int64_t span = hi - lo;
    const int64_t p = lo + ((int64_t)(lane + 1) * span) / 33;  // in (lo, hi)
    const uint32_t c = __ballot_sync(FULL_MASK, __ldg(W + p) <= T);
    const int m = __popc(c);  // probes at or below T form a prefix
    const int64_t nlo = m > 0 ? lo + ((int64_t)m * span) / 33 : lo;
    const int64_t nhi = m < 32 ? lo + ((int64_t)(m + 1) * span) / 33 : hi;
    lo = nlo;
    hi = nhi;
  }
  // at most 33 candidates left: lo and lo+1 .. hi-1
  const int64_t p = lo + 1 + lane;
  const bool le = p < hi && __ldg(W + p) <= T;
  return lo + __popc(__ballot_sync(FULL_MASK, le));
}

// Is x in the ascending row adj[lo, hi)? Same result on every lane.
__device__ __forceinline__ bool warp_row_contains(const int32_t* __restrict__ adj, int64_t lo, int64_t hi, int32_t x,
                                                  int lane) {
  while (hi - lo > 32) {
    const int64_t span = hi - lo;
    const int64_t p = lo + ((int64_t)(lane + 1) * span) / 33;
    const uint32_t c = __ballot_sync(FULL_MASK, __ldg(adj + p) <= x);
    const int m = __popc(c);
    const int64_t nlo = m > 0 ? lo + ((int64_t)m * span) / 33 : lo;
    const int64_t nhi = m < 32 ? lo + ((int64_t)(m + 1) * span) / 33 : hi;
    lo = nlo;
    hi = nhi;
  }
  const int64_t p = lo + lane;
  return __ballot_sync(FULL_MASK, p < hi && __ldg(adj + p) == x) != 0u;
}

__device__ __forceinline__ Wedge draw_wedge_warp(const GraphView& g, int64_t start, int64_t len, uint64_t p,
                                                 uint64_t wbase, const Philox4& r, int lane) {
  Wedge w;
  const uint64_t t = mulhi64((uint64_t)r.r0 | ((uint64_t)r.r1 << 32), p);
  const int64_t j0 = warp_search_prefix(g.W, start, start + len, wbase + t, lane);
  w.v0 = __ldg(g.L + j0);
  const int64_t o0 = __ldg(g.off + w.v0);
  w.d0 = __ldg(g.off + w.v0 + 1) - o0;
  const uint64_t dm1 = (uint64_t)(w.d0 - 1);
  const uint64_t u = mulhi64((uint64_t)r.r2 | ((uint64_t)r.r3 << 32), (uint64_t)w.d0 * dm1);
  const uint64_t i = div_small(u, dm1);
  const uint64_t jp = u - i * dm1;
  const uint64_t j = jp + (jp >= i ? 1ULL : 0ULL);
  w.v1 = __ldg(g.adj + o0 + (int64_t)i);
  w.v2 = __ldg(g.adj + o0 + (int64_t)j);
  const int64_t o1 = __ldg(g.off + w.v1);
  w.d1 = __ldg(g.off + w.v1 + 1) - o1;
  const int64_t o2 = __ldg(g.off + w.v2);
  w.d2 = __ldg(g.off + w.v2 + 1) - o2;
  if (w.d1 < w.d2 || (w.d1 == w.d2 && w.v1 < w.v2)) w.closed = warp_row_contains(g.adj, o1, o1 + w.d1, w.v2, lane);
  else w.closed = warp_row_contains(g.adj, o2, o2 + w.d2, w.v1, lane);
  return w;
}

}  // namespace wedge
