// exact.cu — exact triangle counts per bin on the device (wedge_exact).
//
// The quantities sampling estimates (Sec. 2.1, 2.2): t, t_i and p_{b,q}, the
// closed wedges centred in bin b whose endpoints have q - 1 vertices in b
// (Alg. Phase 4c's classes), so that c_b = (p_{b,1} + p_{b,2} + p_{b,3}) / p_b.
// The paper obtains them by enumeration on a CPU; here vertices are ranked by
// (degree, id), N+(u) are u's neighbours of higher rank, and every triangle
// u < v < w is found once, as the edge (u, v) and a w after v in N+(u) that is
// in N+(v):
//   1. ranks: a radix sort of the degrees;
//   2. exact_orient: counts, per vertex, the neighbours of lower and of higher
//      rank and marks the entries that go down; a scan gives the in-lists (the u of
//      every v) and the rows N+;
//   3. exact_edges: the oriented edges by v, in rank order; a stable radix sort
//      by u then yields the rows N+(u) in rank order, and exact_rows records
//      for every edge of an in-list how many entries of N+(u) come after v;
//   4. exact_hash_warp / exact_hash_cta: for every v, a hash table of N+(v) in
//      shared memory, and the tails of N+(u) after v streamed against it for
//      all u of v's in-list, a warp per tail.
// The tails of all edges are the pairs of N+(u), sum C(d+, 2); streaming the
// whole N+(v) of every v in N+(u) against a table of N+(u) instead reads 3.6
// times as many entries (Kronecker scale 20: 4.4e9 against 1.2e9; 34.4 ms in
// all that way, 5.2 ms this way; scale 24: 1.11 s and 0.25 s). The count is
// bound by instructions and, where N+ rows are short, by the chain of loads per
// vertex. Graphs that would pay the ranks and the sort for nothing stream whole rows
// (exact_rows.cu; the rule: takes_rows), as does one whose memory is refused.
// Vertices are taken in groups of at most 2^27 in-edges, highest ranks
// first, so that the edges' scratch is bounded; rows fill from their ends, and
// the tails that a group reads are there when it is counted.
//
// Symmetry of an imported CSR is its owner's promise. What the kernels rely on
// is less: that m entries go to a lower rank (`down` counts them). Every buffer of
// edges holds m, and the second look at the entries gives each the place that the
// first counted for it, so with m of them all places of in-lists and rows are
// filled, with ranks in order, in any CSR of strictly ascending rows. With
// another number nothing after the first look does anything (the sort finds its
// histograms empty and then writes to places below m), and the call fails.
#include <string.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "exact.cuh"

namespace wedge {
namespace {

constexpr int EX_THREADS = 256;
constexpr int EX_WARPS = EX_THREADS / 32;
constexpr int OR_STEPS = 16;                            // 32-entry steps of a warp at most

// Adds w to the counts of the digits of x, and a CTA's counts to the sort's histograms.
constexpr int DIGIT_COUNTS = 4 * 256;
__device__ __forceinline__ void count_digits(uint32_t* sh, int passes, uint32_t x, uint32_t w) {
  for (int p = 0; p < passes; ++p) atomicAdd(&sh[p * 256 + ((x >> (8 * p)) & 255u)], w);
}
__device__ __forceinline__ void add_counts(const uint32_t* sh, int passes, unsigned long long* __restrict__ hist) {
  for (int i = threadIdx.x; i < passes * 256; i += EX_THREADS)
    if (sh[i]) atomicAdd(&hist[i], (unsigned long long)sh[i]);
}

// Degrees as sort keys, with the sort's histograms.
__global__ __launch_bounds__(EX_THREADS) void k_degree_keys(const int32_t* __restrict__ deg, int32_t n, int passes,
                                                            uint64_t* __restrict__ keys,
                                                            unsigned long long* __restrict__ hist) {
  __shared__ uint32_t sh[DIGIT_COUNTS];
  for (int i = threadIdx.x; i < DIGIT_COUNTS; i += EX_THREADS) sh[i] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * EX_THREADS;
  for (int64_t v = (int64_t)blockIdx.x * EX_THREADS + threadIdx.x; v < n; v += stride) {
    const uint32_t d = (uint32_t)__ldg(deg + v);
    keys[v] = ((uint64_t)d << 32) | (uint64_t)v;
    count_digits(sh, passes, d, 1u);
  }
  __syncthreads();
  add_counts(sh, passes, hist);
}

// order[r] = the vertex of rank r, rank its inverse.
__global__ __launch_bounds__(EX_THREADS) void k_ranks(const uint64_t* __restrict__ sorted, int32_t n,
                                                      int32_t* __restrict__ order, int32_t* __restrict__ rank) {
  const int64_t r = (int64_t)blockIdx.x * EX_THREADS + threadIdx.x;
  if (r < n) {
    const int32_t v = (int32_t)(uint32_t)sorted[r];
    order[r] = v;
    rank[v] = (int32_t)r;
  }
}

// The ranks of few vertices, by comparing each with all: one launch instead of
// a sort's eight (9 us for 256 vertices, some 25 us less than the sort; at
// 8,192 the comparisons take about as long).
constexpr int32_t FEW_VERTICES = 8192;

__global__ __launch_bounds__(EX_THREADS) void k_ranks_few(const int32_t* __restrict__ deg, int32_t n,
                                                          int32_t* __restrict__ order, int32_t* __restrict__ rank) {
  // a CTA takes 32 vertices, one a lane; its warps share out the others
  __shared__ int32_t s_sum[EX_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t v = blockIdx.x * 32 + lane;
  const int32_t d = v < n ? __ldg(deg + v) : 0;
  int32_t less = 0;
  for (int32_t x0 = warp * 32; x0 < n; x0 += EX_THREADS) {
    const int32_t mine = x0 + lane < n ? __ldg(deg + x0 + lane) : INT32_MAX;
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
      const int32_t o = __shfl_sync(FULL_MASK, mine, j);
      less += o < d || (o == d && x0 + j < v);
    }
  }
  s_sum[warp][lane] = less;
  __syncthreads();
  if (warp == 0 && v < n) {
    int32_t r = 0;
    for (int w = 0; w < EX_WARPS; ++w) r += s_sum[w][lane];
    rank[v] = r;
    order[r] = v;
  }
}

struct OrientArgs {
  const int64_t* off;
  const int32_t* adj;
  const int32_t* rank;
  int32_t n;
  int64_t n_adj;
  int steps;              // 32-entry steps of a warp
  int32_t* lower;         // by rank: neighbours of lower rank (EMIT: taken so far)
  int32_t* higher;        // by rank: neighbours of higher rank
  uint32_t* kept;         // which entries go to a lower rank, a bit each
  unsigned long long* down;  // their number
  const int64_t* in_off;  // EMIT: in-list offsets by rank
  int32_t r0, r1;         // EMIT: the group's ranks
  uint64_t* keys;         // EMIT: u << 32 | place in the group's in-lists
  uint32_t* v_of;         // EMIT: v by place
  uint32_t* u_of;         // EMIT: u by place
  int64_t m;              // EMIT: places in all in-lists
  int64_t places;         // and room for a group's (checked by the debug build, as below)
  uint32_t* err;
};

// Every adjacency entry (v, u) with rank(u) < rank(v): counted for both ends and
// marked, or (EMIT) given a place in v's in-list, if v is of the group. A warp takes up to
// 512 consecutive entries, 32 at a time; the lanes of a row share one atomic.
template <bool EMIT>
__global__ __launch_bounds__(EX_THREADS) void k_orient(OrientArgs a) {
  const int lane = threadIdx.x & 31;
  const uint32_t le = lanemask_lt() | (1u << lane);
  const int64_t base = ((int64_t)blockIdx.x * EX_WARPS + (threadIdx.x >> 5)) * (32 * a.steps);
  if (base >= a.n_adj || (EMIT && *a.down != (unsigned long long)a.m)) return;
  uint32_t down = 0;
  int32_t x = row_of(a.off, a.n, min(base + lane, a.n_adj - 1)), rx = __ldg(a.rank + x);
  for (int i = 0; i < a.steps; ++i) {
    const int64_t e = base + i * 32 + lane;
    if (e - lane >= a.n_adj) break;  // the whole warp
    const uint32_t marked = EMIT ? __ldg(a.kept + (e >> 5)) : FULL_MASK;  // (e - lane is a multiple of 32)
    if (EMIT && marked == 0) continue;
    bool keep = false;
    int32_t ry = 0;
    if (e < a.n_adj) {
      if (e >= __ldg(a.off + x + 1)) {
        x = next_row(a.off, a.n, x, e);
        rx = __ldg(a.rank + x);
      }
      if (!EMIT || ((marked >> lane & 1u) && rx >= a.r0 && rx < a.r1)) {
        ry = __ldg(a.rank + __ldcs(a.adj + e));
        keep = ry < rx;
      }
    }
    const uint32_t kept = __ballot_sync(FULL_MASK, keep);
    if (!EMIT && lane == 0) a.kept[e >> 5] = kept;
    down += __popc(kept);
    if (kept == 0) continue;
    const int32_t before = __shfl_up_sync(FULL_MASK, rx, 1);
    const uint32_t starts = __ballot_sync(FULL_MASK, lane == 0 || before != rx);
    const int start = 31 - __clz(starts & le);
    const uint32_t later = starts & ~le;
    const uint32_t run = (later ? (1u << (__ffs(later) - 1)) - 1u : FULL_MASK) & ~((1u << start) - 1u);
    const uint32_t mine = kept & run;  // the row's kept entries among these 32
    int32_t at = 0;
    if (lane == start && mine) at = atomicAdd(a.lower + rx, __popc(mine));
    if (!EMIT) {
      if (keep) atomicAdd(a.higher + ry, 1);
    } else {
      at = __shfl_sync(FULL_MASK, at, start);
      if (keep) {
        const uint64_t pos = (uint64_t)(__ldg(a.in_off + rx) - __ldg(a.in_off + a.r0)) + (uint32_t)at +
                             __popc(mine & lanemask_lt());
        if (in_bounds(pos, (uint64_t)a.places, a.err)) {
          a.keys[pos] = ((uint64_t)(uint32_t)ry << 32) | pos;
          a.v_of[pos] = (uint32_t)rx;
          a.u_of[pos] = (uint32_t)ry;
        }
      }
    }
  }
  if (!EMIT && lane == 0 && down) atomicAdd(a.down, (unsigned long long)down);
}

// Last place of each u's run in the group's edges sorted by u.
__global__ __launch_bounds__(EX_THREADS) void k_run_ends(const uint64_t* __restrict__ keys, int64_t m,
                                                         uint32_t* __restrict__ run_end) {
  const int64_t i = (int64_t)blockIdx.x * EX_THREADS + threadIdx.x;
  if (i >= m) return;
  const uint32_t u = (uint32_t)(keys[i] >> 32);
  if (i + 1 == m || (uint32_t)(keys[i + 1] >> 32) != u) run_end[u] = (uint32_t)(i + 1);
}

// After a group: how many entries each row holds now.
__global__ __launch_bounds__(EX_THREADS) void k_run_add(const uint64_t* __restrict__ keys, int64_t m,
                                                        const uint32_t* __restrict__ run_end,
                                                        uint32_t* __restrict__ filled) {
  const int64_t i = (int64_t)blockIdx.x * EX_THREADS + threadIdx.x;
  if (i >= m) return;
  const uint32_t u = (uint32_t)(keys[i] >> 32);
  if (i == 0 || (uint32_t)(keys[i - 1] >> 32) != u) filled[u] += run_end[u] - (uint32_t)i;
}

// Rows N+(u), from their ends: sorted edge i (u, and by its place the v) goes
// before the entries of higher rank, and its in-list place learns how many
// these are (alone: 4 bytes to random places; with u beside it, 134 MB of 16.8 M
// edges, past L2, 529 us, so 305..323). WHOLE: the group is all there is, so i is the
// place in the rows, and whether all of it was filled is not known to the host.
template <bool WHOLE>
__global__ __launch_bounds__(EX_THREADS) void k_rows(const uint64_t* __restrict__ keys, int64_t m, uint32_t n,
                                                     const unsigned long long* __restrict__ down,
                                                     const uint32_t* __restrict__ v_of,
                                                     const int64_t* __restrict__ row_off,
                                                     const uint32_t* __restrict__ run_end,
                                                     const uint32_t* __restrict__ filled, uint32_t* __restrict__ rows,
                                                     int64_t row_base, uint32_t* __restrict__ tail_of,
                                                     uint32_t* err) {
  const int64_t i = (int64_t)blockIdx.x * EX_THREADS + threadIdx.x;
  if (i >= m || (WHOLE && *down != (unsigned long long)m)) return;
  const uint64_t key = __ldcs(keys + i);
  const uint32_t u = (uint32_t)(key >> 32), pos = (uint32_t)key;
  if (!in_bounds(u, n, err)) return;
  const int64_t row_end = __ldg(row_off + u + 1);
  const uint32_t after = WHOLE ? (uint32_t)(row_end - 1 - row_base - i)
                               : __ldg(filled + u) + (__ldg(run_end + u) - 1u - (uint32_t)i);
  const int64_t at = row_end - 1 - row_base - (int64_t)after;
  if (!in_bounds(pos, (uint64_t)m, err) || !in_bounds((uint64_t)at, (uint64_t)row_base, err)) return;
  rows[at] = __ldg(v_of + pos);
  tail_of[pos] = after;
}

// ----------------------------------------------------------------- count --

struct CountArgs {
  const int64_t* in_off;   // n + 1, by rank
  const int64_t* row_off;  // n + 1, by rank, from m on (the scan goes on from the in-lists)
  const uint32_t* rows;
  const uint32_t* u_of;    // the group's in-lists: u,
  const uint32_t* tail_of; // and entries of N+(u) after v
  const int32_t* order;
  const uint32_t* bin_lo;  // first rank of each bin, then n
  uint32_t nb;
  uint32_t n;
  int64_t m;               // entries of rows
  int64_t places;          // entries of u_of and tail_of (checked by the debug build)
  uint32_t grab;           // vertices a warp takes per ticket
  uint32_t map_ranks;      // most ranks of a bit map, and half the slots of a hash table, of the
  uint32_t table_row;      // CTA kernels (as they are sized, or less)
  int32_t r0, r1;          // the group's ranks
  unsigned long long* pbq; // [nb][4] (class 1..3 used)
  unsigned long long* t_i; // per-vertex closed wedges or nullptr
  const unsigned long long* down;  // entries that go to a lower rank
  uint32_t* err;           // DERR_BAD_ID: they are not m
  unsigned int* next;      // work counter of the warp kernel
  uint2* units;            // (v, part of its in-list) for the CTA kernels: medium rows from the front, long from the back
  uint32_t max_units;
  unsigned int* n_units;   // [0] medium, [1] long
};

// Times of the whole call in us, each constant alone changed, on Kronecker scale
// 20 / scale 16 / power law of 1 M, gamma 2.3, 20 a vertex / uniform, 16.8 M edges of 4 M:
//   as they are 5,124 / 535 / 1,774 / 3,013
//   WARP_IN 32: 5,510 / 510 / 1,944 / 3,009; 128: 5,152 / 751 / 1,708 / 3,022
//   MEMORY_ROW 4: 5,129 / 534 / 1,797 / 3,127; 16: 5,131 / 532 / 1,763 / 3,013 (and a ring
//     with 16 neighbours a side, nearly all of whose looks find: 4,446, 5,483 with 8, 8,427)
//   UNIT_IN 256: 5,635 / 529 / 1,852 / 3,014; 1,024: 4,870 / 541 / 1,755 / 3,016
constexpr int WARP_ROW = 128;        // rows N+(v) up to this length ...
constexpr int WARP_IN = 64;          // ... with in-lists up to this: one warp
constexpr int WARP_SLOTS = 512;
constexpr int MEMORY_ROW = 8;        // rows up to this length are searched where they are
constexpr int MID_ROW = 1024;        // longest row of the medium CTA kernel
constexpr int UNIT_IN = 512;         // in-edges of a unit of the CTA kernels
constexpr uint32_t GRAB = 8;         // vertices a warp takes per ticket at most

__device__ __forceinline__ uint32_t slot_of(uint32_t w, uint32_t mask) { return (w * 0x9E3779B1u) >> 7 & mask; }

__device__ __forceinline__ uint2 in_edge(const CountArgs& a, int64_t place) {
  if (!in_bounds((uint64_t)place, (uint64_t)a.places, a.err)) return make_uint2(0, 0);
  const uint2 r = make_uint2(__ldcs(a.u_of + place), __ldcs(a.tail_of + place));
  return in_bounds(r.x, a.n, a.err) ? r : make_uint2(0, 0);
}

// Insert key w (absent); the table has free slots (load <= 1/2).
__device__ __forceinline__ void insert_key(uint32_t* table, uint32_t mask, uint32_t w) {
  uint32_t h = slot_of(w, mask);
  while (atomicCAS(table + h, ~0u, w) != ~0u) h = (h + 1) & mask;
}

// Bin of a rank: ranks ascend by degree, so every bin is a range of them,
// lo[b] to lo[b + 1] (lo[nb] = n).
__device__ __forceinline__ uint32_t rank_bin(const uint32_t* lo, uint32_t nb, uint32_t r) {
  uint32_t b = 0, e = nb;  // last bin with lo <= r
  while (e - b > 1) {
    const uint32_t mid = (b + e) >> 1;
    if (lo[mid] <= r) b = mid; else e = mid;
  }
  return b;
}

// Which w are in N+(v), and the counter each has.
struct HashRow {  // a hash table; the counter is the slot
  const uint32_t* table;
  uint32_t mask;
  __device__ __forceinline__ bool find(uint32_t w, uint32_t& slot) const {
    uint32_t h = slot_of(w, mask);
    while (true) {
      const uint32_t x = table[h];
      slot = h;
      if (x == w) return true;
      if (x == ~0u) return false;
      h = (h + 1) & mask;
    }
  }
};
struct BitRow {  // one bit per rank above v; the counter is w's place in the row
  const uint32_t* bits;
  const uint16_t* before;  // row entries before the word's first
  uint32_t above;          // v + 1
  uint32_t range;          // ranks of the map (checked by the debug build)
  uint32_t* err;
  __device__ __forceinline__ bool find(uint32_t w, uint32_t& slot) const {
    if (!in_bounds(w - above, range, err)) return false;
    const uint32_t i = w - above, word = bits[i >> 5], rest = word >> (i & 31u);
    if (!(rest & 1u)) return false;
    slot = before[i >> 5] + __popc(word) - __popc(rest);
    return true;
  }
};
struct MemoryRow {  // a search of the row in memory; no counters
  const uint32_t* row;
  uint32_t d;
  __device__ __forceinline__ bool find(uint32_t w, uint32_t&) const {
    uint32_t lo = 0, hi = d;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1, x = __ldg(row + mid);
      if (x == w) return true;
      if (x < w) lo = mid + 1; else hi = mid;
    }
    return false;
  }
};

// The tails of up to 32 in-edges of v (one per lane; length 0: none) against
// N+(v). A found w closes the triangle u < v < w, one closed wedge centred at
// each vertex, of class 1 + (endpoints in the centre's bin): w's are added to
// its counter (low half: bin(u) != bin(w), high half: equal; at most one per
// in-edge, so the halves do not overflow) or, where there is none, to the
// histogram; u's and v's are summed per tail, kept by the lane whose in-edge it
// is, and added at the end by all lanes at once (cv: v's, by number of
// endpoints in v's bin). w > v > u, so w is in u's bin iff it lies below that
// bin's end.
// Long tails are streamed one after the other by the whole warp. Tails shorter
// than FLAT entries on average are taken as one list of their entries (a search
// by shuffles finds an entry's tail): a warp per tail left most lanes idle
// (uniform graph, 16 M edges, tails of 7: 1.7 ms, 0.9 so).
constexpr uint32_t FLAT = 24;

template <bool COUNTERS, typename Row>
__device__ __forceinline__ void count_tails(const CountArgs& a, const Row& nv, const uint32_t* s_lo,
                                            unsigned long long* hist, uint2 r, uint32_t bv, uint32_t* hits,
                                            uint32_t* seg, uint32_t (&cv)[3], int lane) {
  const uint32_t my_bin = r.y ? rank_bin(s_lo, a.nb, r.x) : 0u, my_end_u = s_lo[my_bin + 1];
  const int64_t my_row_end = r.y ? __ldg(a.row_off + r.x + 1) : 0;
  const uint64_t my_tail = (uint64_t)(my_row_end - a.m - r.y);
  const uint32_t end_v = s_lo[bv + 1];
  uint32_t found = 0, with_u = 0, with_v = 0;  // this lane's in-edge
  // w of a tail of a u whose bin ends at end_u: what it adds to found (low 10
  // bits), with_u (next 10) and with_v (the rest)
  auto look = [&](uint32_t w, uint32_t end_u) {
    uint32_t slot;
    if (!nv.find(w, slot)) return 0u;
    const bool in_u = w < end_u;
    if (COUNTERS) {
      atomicAdd(hits + slot, in_u ? 0x10000u : 1u);
    } else {
      const uint32_t bu = rank_bin(s_lo, a.nb, end_u - 1u), bw = rank_bin(s_lo, a.nb, w);
      atomicAdd(&hist[bw * 4 + 1 + (bu == bw) + (bv == bw)], 1ULL);
      if (a.t_i) atomicAdd(a.t_i + a.order[w], 1ULL);
    }
    return (in_u ? 1025u : 1u) + (w < end_v ? 1u << 20 : 0u);
  };
  uint32_t todo = __ballot_sync(FULL_MASK, r.y != 0);
  const uint32_t total = __reduce_add_sync(FULL_MASK, min(r.y, 2 * 32 * FLAT));
  if (total < FLAT * __popc(todo)) {
    uint32_t incl = r.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL_MASK, incl, o);
      if (lane >= o) incl += y;
    }
    const uint64_t my_first = my_tail - (incl - r.y);  // entry t of the list is a.rows[my_first + t]
    seg[lane] = 0;
    __syncwarp();
    for (uint32_t t0 = 0; t0 < total; t0 += 32) {
      const uint32_t t = min(t0 + lane, total - 1u);
      int l = 0;  // the first lane whose tails end after t
#pragma unroll
      for (int step = 16; step > 0; step >>= 1)
        if (__shfl_sync(FULL_MASK, incl, l + step - 1) <= t) l += step;
      const uint64_t first = __shfl_sync(FULL_MASK, my_first, l);
      const uint32_t end_u = __shfl_sync(FULL_MASK, my_end_u, l);
      if (t0 + lane < total) {
        const uint32_t add = look(checked_ldg(a.rows, (int64_t)(first + t), a.m, a.err), end_u);
        if (add) atomicAdd(seg + l, add);
      }
    }
    __syncwarp();
    found = seg[lane] & 1023u;
    with_u = (seg[lane] >> 10) & 1023u;
    with_v = seg[lane] >> 20;
    __syncwarp();
  } else {
    for (; todo; todo &= todo - 1) {
      const int l = __ffs(todo) - 1;
      const uint32_t len = __shfl_sync(FULL_MASK, r.y, l), end_u = __shfl_sync(FULL_MASK, my_end_u, l);
      const uint64_t at = __shfl_sync(FULL_MASK, my_tail, l);
      if (len && !in_bounds(at + len - 1, (uint64_t)a.m, a.err)) continue;  // (the whole warp)
      const uint32_t* tail = a.rows + at;
      for (uint32_t k0 = 0; k0 < len; k0 += 30 * 32) {  // (sums of 30 x 32 fit their 10 bits)
        uint32_t mine = 0;
        const uint32_t k1 = min(len, k0 + 30 * 32);
        for (uint32_t k = k0 + lane; k < k1; k += 64) {  // two loads in flight
          const bool two = k + 32 < k1;
          const uint32_t w0 = __ldg(tail + k), w1 = two ? __ldg(tail + k + 32) : 0u;
          mine += look(w0, end_u);
          if (two) mine += look(w1, end_u);
        }
        mine = __reduce_add_sync(FULL_MASK, mine);
        if (lane == l) {
          found += mine & 1023u;
          with_u += (mine >> 10) & 1023u;
          with_v += mine >> 20;
        }
      }
    }
  }
  if (found) {
    unsigned long long* hu = hist + my_bin * 4 + 1 + (bv == my_bin);
    if (found > with_u) atomicAdd(hu, (unsigned long long)(found - with_u));
    if (with_u) atomicAdd(hu + 1, (unsigned long long)with_u);
    if (a.t_i) atomicAdd(a.t_i + a.order[r.x], (unsigned long long)found);
    const uint32_t diff = found - with_v;
    if (my_bin == bv) {
      cv[1] += diff;
      cv[2] += with_v;
    } else {
      cv[0] += diff;
      cv[1] += with_v;
    }
  }
}

// v's closed wedges, summed over the warp.
__device__ __forceinline__ void flush_centre(const CountArgs& a, unsigned long long* hist, uint32_t v, uint32_t bv,
                                             uint32_t (&cv)[3], int lane) {
  for (int q = 0; q < 3; ++q) cv[q] = __reduce_add_sync(FULL_MASK, cv[q]);
  if (lane != 0) return;
  for (int q = 0; q < 3; ++q)
    if (cv[q]) atomicAdd(&hist[bv * 4 + 1 + q], (unsigned long long)cv[q]);
  const uint32_t all = cv[0] + cv[1] + cv[2];
  if (a.t_i && all) atomicAdd(a.t_i + a.order[v], (unsigned long long)all);
}

// Adds a counter (closed wedges centred at w) to the histogram and clears it.
__device__ __forceinline__ void fold_hit(const CountArgs& a, const uint32_t* s_lo, unsigned long long* hist,
                                         uint32_t* hit, uint32_t w, uint32_t bv) {
  const uint32_t x = *hit, same = x >> 16, diff = x & 0xffffu;
  *hit = 0;
  const uint32_t bw = rank_bin(s_lo, a.nb, w);
  unsigned long long* hw = hist + bw * 4 + 1 + (bv == bw);
  if (diff) atomicAdd(hw, (unsigned long long)diff);
  if (same) atomicAdd(hw + 1, (unsigned long long)same);
  if (a.t_i) atomicAdd(a.t_i + a.order[w], (unsigned long long)(same + diff));
}

// One warp per vertex v with a short row and a short in-list, highest ranks
// (the most work) first; the others are queued as units of UNIT_IN in-edges.
__global__ __launch_bounds__(EX_THREADS) void k_tri_hash_warp(CountArgs a) {
  __shared__ uint32_t s_lo[WEDGE_MAX_BINS + 1];
  __shared__ unsigned long long s_hist[WEDGE_MAX_BINS * 4];
  __shared__ uint32_t s_table[EX_WARPS][WARP_SLOTS];
  __shared__ uint32_t s_hits[EX_WARPS][WARP_SLOTS];
  __shared__ uint32_t s_seg[EX_WARPS][32];
  if (*a.down != (unsigned long long)a.m) {  // (then no unit is queued either)
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, DERR_BAD_ID);
    return;
  }
  for (int i = threadIdx.x; i <= (int)a.nb; i += EX_THREADS) s_lo[i] = a.bin_lo[i];
  for (int i = threadIdx.x; i < (int)a.nb * 4; i += EX_THREADS) s_hist[i] = 0;
  for (int i = threadIdx.x; i < EX_WARPS * WARP_SLOTS; i += EX_THREADS) (&s_hits[0][0])[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t* table = s_table[wid];
  uint32_t* hits = s_hits[wid];
  const int64_t in0 = __ldg(a.in_off + a.r0);
  const uint32_t count = (uint32_t)(a.r1 - a.r0);
  while (true) {
    unsigned int first = 0;
    if (lane == 0) first = atomicAdd(a.next, a.grab);
    first = __shfl_sync(FULL_MASK, first, 0);
    if (first >= count) break;
    const uint32_t last = min(count, first + a.grab);
    for (uint32_t i = first; i < last; ++i) {
      const uint32_t v = (uint32_t)a.r1 - 1u - i;
      const int64_t row = __ldg(a.row_off + v) - a.m, in = __ldg(a.in_off + v);
      const int64_t d = __ldg(a.row_off + v + 1) - a.m - row;
      const int64_t k = __ldg(a.in_off + v + 1) - in;
      if (d == 0 || k == 0) continue;
      if (d > WARP_ROW || k > WARP_IN) {
        const uint32_t parts = (uint32_t)((k + UNIT_IN - 1) / UNIT_IN);
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(a.n_units + (d > MID_ROW), parts);
        at = __shfl_sync(FULL_MASK, at, 0);
        for (uint32_t p = lane; p < parts; p += 32)
          if (at + p < a.max_units) a.units[d > MID_ROW ? a.max_units - 1 - (at + p) : at + p] = make_uint2(v, p);
        continue;
      }
      const uint32_t bv = rank_bin(s_lo, a.nb, v);
      uint32_t cv[3] = {0, 0, 0};
      auto tails = [&](int64_t j) {
        return j + lane < k ? in_edge(a, in - in0 + j + lane) : make_uint2(0, 0);
      };
      if (d <= MEMORY_ROW) {  // a few entries are found faster than they are entered into a table
        for (int64_t j = 0; j < k; j += 32)
          count_tails<false>(a, MemoryRow{a.rows + row, (uint32_t)d}, s_lo, s_hist, tails(j), bv, hits, s_seg[wid], cv,
                             lane);
        flush_centre(a, s_hist, v, bv, cv, lane);
        continue;
      }
      uint32_t slots = 32;
      while (slots < 4u * (uint32_t)d) slots <<= 1;  // at most WARP_SLOTS
      for (uint32_t j = lane; j < slots; j += 32) table[j] = ~0u;
      __syncwarp();
      for (uint32_t j = lane; j < (uint32_t)d; j += 32) insert_key(table, slots - 1, __ldg(a.rows + row + j));
      __syncwarp();
      for (int64_t j = 0; j < k; j += 32)
        count_tails<true>(a, HashRow{table, slots - 1}, s_lo, s_hist, tails(j), bv, hits, s_seg[wid], cv, lane);
      flush_centre(a, s_hist, v, bv, cv, lane);
      __syncwarp();
      for (uint32_t h = lane; h < slots; h += 32)
        if (hits[h]) fold_hit(a, s_lo, s_hist, hits + h, table[h], bv);
      __syncwarp();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (int)a.nb * 4; i += EX_THREADS)
    if (s_hist[i]) atomicAdd(a.pbq + i, s_hist[i]);
}

// One CTA per unit (by ticket); its warps take the unit's in-edges 32 at a
// time. N+(v) is a bit map in shared memory where v is among the MAP_BITS
// highest ranks (most of the work is: they have the long in-lists; six
// instructions and no loop per look), a hash table where SLOTS is at least
// twice the row, and else searched in memory (degree order bounds rows by about
// sqrt(2m), so this is rare).
template <int THREADS, int SLOTS, int MAP_BITS>
struct CtaSmem {
  union {
    uint32_t table[SLOTS];
    struct {
      uint32_t bits[MAP_BITS / 32];
      uint16_t before[MAP_BITS / 32];
    } map;
  };
  uint32_t hits[SLOTS];
};

template <int THREADS, int SLOTS, int MAP_BITS>
__global__ __launch_bounds__(THREADS) void k_tri_hash_cta(CountArgs a, const uint2* __restrict__ list, int dir,
                                                          const unsigned int* __restrict__ n_units,
                                                          unsigned int* ticket) {
  extern __shared__ __align__(16) unsigned char dyn[];
  CtaSmem<THREADS, SLOTS, MAP_BITS>& sm = *reinterpret_cast<CtaSmem<THREADS, SLOTS, MAP_BITS>*>(dyn);
  __shared__ uint32_t s_lo[WEDGE_MAX_BINS + 1];
  __shared__ unsigned long long s_hist[WEDGE_MAX_BINS * 4];
  __shared__ uint32_t s_seg[THREADS / 32][32];
  __shared__ uint32_t s_q, s_batch;
  for (int i = threadIdx.x; i <= (int)a.nb; i += THREADS) s_lo[i] = a.bin_lo[i];
  for (int i = threadIdx.x; i < (int)a.nb * 4; i += THREADS) s_hist[i] = 0;
  for (int i = threadIdx.x; i < SLOTS; i += THREADS) sm.hits[i] = 0;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t in0 = __ldg(a.in_off + a.r0);
  const uint32_t n_list = min(*n_units, a.max_units);
  while (n_list > 0) {
    __syncthreads();  // the previous unit is done with the table
    if (tid == 0) {
      s_q = atomicAdd(ticket, 1u);
      s_batch = 0;
    }
    __syncthreads();
    const uint32_t q = s_q;
    if (q >= n_list) break;
    const uint2 unit = list[(int64_t)dir * q];
    const uint32_t v = unit.x;
    const int64_t row_at = __ldg(a.row_off + v);
    const uint32_t* row = a.rows + (row_at - a.m);
    const uint32_t d = (uint32_t)(__ldg(a.row_off + v + 1) - row_at);
    const int64_t in = __ldg(a.in_off + v) + (int64_t)unit.y * UNIT_IN;
    const uint32_t k = (uint32_t)min((int64_t)UNIT_IN, __ldg(a.in_off + v + 1) - in);
    const uint32_t range = a.n - 1u - v;  // ranks above v
    const bool in_map = range <= min((uint32_t)MAP_BITS, a.map_ranks) && d <= (uint32_t)SLOTS;
    const bool in_table = !in_map && d <= min((uint32_t)SLOTS / 2u, a.table_row);
    uint32_t slots = 64;
    while (slots < 4u * d && slots < (uint32_t)SLOTS) slots <<= 1;
    if (in_map) {
      for (uint32_t i = tid; i < (range + 31u) / 32u; i += THREADS) sm.map.bits[i] = 0;
      __syncthreads();
      for (uint32_t i = tid; i < d; i += THREADS) {
        const uint32_t x = __ldg(row + i) - (v + 1u), y = i ? __ldg(row + i - 1) - (v + 1u) : ~0u;
        if (!in_bounds(x, range, a.err)) continue;
        atomicOr(&sm.map.bits[x >> 5], 1u << (x & 31u));
        if ((x >> 5) != (y >> 5)) sm.map.before[x >> 5] = (uint16_t)i;
      }
      __syncthreads();
    } else if (in_table) {
      for (uint32_t i = tid; i < slots; i += THREADS) sm.table[i] = ~0u;
      __syncthreads();
      for (uint32_t i = tid; i < d; i += THREADS) insert_key(sm.table, slots - 1, __ldg(row + i));
      __syncthreads();
    }
    const uint32_t bv = rank_bin(s_lo, a.nb, v);
    uint32_t cv[3] = {0, 0, 0};
    while (true) {
      uint32_t j = 0;
      if (lane == 0) j = atomicAdd(&s_batch, 32u);
      j = __shfl_sync(FULL_MASK, j, 0);
      if (j >= k) break;
      const uint2 r = j + lane < k ? in_edge(a, in - in0 + j + lane) : make_uint2(0, 0);
      if (in_map)
        count_tails<true>(a, BitRow{sm.map.bits, sm.map.before, v + 1u, range, a.err}, s_lo, s_hist, r, bv, sm.hits, s_seg[tid >> 5], cv, lane);
      else if (in_table)
        count_tails<true>(a, HashRow{sm.table, slots - 1}, s_lo, s_hist, r, bv, sm.hits, s_seg[tid >> 5], cv, lane);
      else count_tails<false>(a, MemoryRow{row, d}, s_lo, s_hist, r, bv, sm.hits, s_seg[tid >> 5], cv, lane);
    }
    flush_centre(a, s_hist, v, bv, cv, lane);
    __syncthreads();  // all hits counted
    if (in_map) {
      for (uint32_t i = tid; i < d; i += THREADS)
        if (sm.hits[i]) fold_hit(a, s_lo, s_hist, sm.hits + i, __ldg(row + i), bv);
    } else if (in_table) {
      for (uint32_t i = tid; i < slots; i += THREADS)
        if (sm.hits[i]) fold_hit(a, s_lo, s_hist, sm.hits + i, sm.table[i], bv);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (int)a.nb * 4; i += THREADS)
    if (s_hist[i]) atomicAdd(a.pbq + i, s_hist[i]);
}

constexpr int MID_THREADS = 256, MID_SLOTS = 2048, MID_BITS = 1 << 16;    // rows up to 1024
constexpr int BIG_THREADS = 512, BIG_SLOTS = 16384, BIG_BITS = 1 << 19;   // rows beyond (table up to 8192)

unsigned blocks_for(int64_t items) { return (unsigned)((items + EX_THREADS - 1) / EX_THREADS); }

// What the neighbours of higher rank say before the edges are looked at again: the
// digit histograms of the sort by u, and whether any rank has neighbours on both
// sides (any[0]) and any two of higher rank (any[1]): without both there is no tail to
// look up.
__global__ __launch_bounds__(EX_THREADS) void k_row_sums(const int32_t* __restrict__ lower,
                                                         const int32_t* __restrict__ higher, int32_t n, int passes,
                                                         const unsigned long long* __restrict__ down, int64_t m,
                                                         unsigned long long* __restrict__ hist,
                                                         uint32_t* __restrict__ any) {
  __shared__ uint32_t sh[DIGIT_COUNTS];
  if (*down != (unsigned long long)m) return;  // (no counts: see above)
  for (int i = threadIdx.x; i < DIGIT_COUNTS; i += EX_THREADS) sh[i] = 0;
  __syncthreads();
  bool both = false, two = false;
  const int64_t stride = (int64_t)gridDim.x * EX_THREADS;
  for (int64_t r = (int64_t)blockIdx.x * EX_THREADS + threadIdx.x; r < n; r += stride) {
    const int32_t h = __ldg(higher + r);
    if (h == 0) continue;
    both = both || __ldg(lower + r) > 0;
    two = two || h > 1;
    count_digits(sh, passes, (uint32_t)r, (uint32_t)h);
  }
  both = __syncthreads_or(both);
  two = __syncthreads_or(two);
  if (threadIdx.x == 0 && both) any[0] = 1u;
  if (threadIdx.x == 0 && two) any[1] = 1u;
  add_counts(sh, passes, hist);
}

// For a graph of this many entries the host waits for `any` (while the offsets
// are scanned) before its edges are looked at again: 20 M edges between 1,000 and
// 20,000 vertices 1,108 -> 327 us, 2 M between 20 and 100,000 364 -> 177.
constexpr int64_t ASK_ENTRIES = int64_t(1) << 20;

// A few words read back while later work runs.
struct ReadBack {
  cudaEvent_t done = nullptr;
  uint32_t* words = nullptr;
  static constexpr size_t BYTES = 64;
  ~ReadBack() {
    if (done) {
      cudaEventSynchronize(done);  // the copy is no longer under way
      cudaEventDestroy(done);
    }
    pinned_free(words, BYTES);
  }
  cudaError_t start(const uint32_t* from, size_t n, cudaStream_t s) {
    words = static_cast<uint32_t*>(pinned_alloc(BYTES));
    if (!words) return cudaErrorMemoryAllocation;
    cudaError_t e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaMemcpyAsync(words, from, n * sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaEventRecord(done, s);
    return e;
  }
  cudaError_t wait() { return cudaEventSynchronize(done); }
};

unsigned some_blocks(int64_t items) {
  const int64_t blocks = (items + EX_THREADS - 1) / EX_THREADS;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)sm_count() * 8));
}

}  // namespace

wedge_status exact_tails(const wedge_graph* g, const wedge_bins* b, unsigned long long* t_i, cudaStream_t s,
                         const ExactLimits& lim, unsigned long long* pbq_out) {
  const wedge_bins_info& inf = b->info;
  const int32_t n = g->n;
  const int64_t n_adj = g->n_adj;
  const int64_t m = n_adj / 2;
  if (n_adj / (EX_WARPS * 32 * OR_STEPS) >= (int64_t)INT32_MAX) return fail(WEDGE_EINVAL, "wedge_exact: graph too large");

  // edges are taken in groups of at most `cap`
  const int64_t cap = std::max<int64_t>(lim.group_edges, g->max_degree);
  const bool grouped = m > cap, few = n <= FEW_VERTICES;
  const int64_t most = std::min(m, cap);
  const size_t n_keys = (size_t)(few ? most : std::max<int64_t>(most, n));
  const uint32_t nb = inf.n_bins;
  const size_t n_cnt = (size_t)nb * 4;
  // ranks, vertices by rank, per rank: lower and higher neighbours, entries taken; with groups also row entries, run
  // ends; then a bit per adjacency entry
  const size_t n_words = (grouped ? 7 : 5) * (size_t)n + (size_t)((n_adj + 31) / 32);

  // control words (error bits, warp ticket, 2 unit counts, 2 CTA tickets, any[2]; entries down), pbq [nb*4], the
  // bins' first ranks
  unsigned long long* cnt = nullptr;
  int32_t* words = nullptr;
  int64_t* offs = nullptr;  // in-list, then row offsets by rank, one scan (2n + 1)
  uint64_t* keys = nullptr;
  uint64_t* alt = nullptr;
  char* scratch = nullptr;   // of a sort, then of the scan
  uint32_t* rows = nullptr;  // m, and v and u by place of a group's edges
  uint2* units = nullptr;
  ReadBack any;
  auto done = [&](wedge_status st) {
    dfree(cnt, s);
    dfree(words, s);
    dfree(offs, s);
    dfree(keys, s);
    dfree(alt, s);
    dfree(scratch, s);
    dfree(rows, s);
    dfree(units, s);
    return st;
  };
#define EXACT_TRY(expr)                                                        \
  do {                                                                         \
    const cudaError_t e__ = (expr);                                            \
    if (e__ != cudaSuccess) return done(cuda_fail(e__, "wedge_exact"));        \
  } while (0)
#define EXACT_DO(expr)                                     \
  do {                                                     \
    const wedge_status st__ = (expr);                      \
    if (st__ != WEDGE_OK) return done(st__);               \
  } while (0)

  const size_t sort_bytes = std::max(sort_scratch_bytes((int64_t)n_keys, (int)g->id_bits),
                                     few ? 0 : sort_scratch_bytes(n, 31));
  EXACT_DO(dalloc_n(&cnt, 5 + n_cnt + nb / 2 + 1, s, "wedge_exact"));
  EXACT_DO(dalloc_n(&words, n_words, s, "wedge_exact: ranks and counts"));
  EXACT_DO(dalloc_n(&keys, n_keys, s, "wedge_exact: edges"));
  EXACT_DO(dalloc_n(&alt, n_keys, s, "wedge_exact: edges"));
  EXACT_DO(dalloc(reinterpret_cast<void**>(&scratch), sort_bytes + scan_scratch_bytes(2 * (int64_t)n), s,
                  "wedge_exact"));
  const uint64_t max_units = (uint64_t)most / UNIT_IN + (uint64_t)most / WARP_IN + (uint64_t)m / WARP_ROW + 64;
  if (most > (int64_t)UINT32_MAX || max_units > UINT32_MAX)
    return done(fail(WEDGE_EINVAL, "wedge_exact: graph too large"));
  EXACT_TRY(cudaMemsetAsync(cnt, 0, (5 + n_cnt) * sizeof(unsigned long long), s));
  uint32_t* ctl = reinterpret_cast<uint32_t*>(cnt);
  unsigned long long* down = cnt + 4;
  unsigned long long* pbq = cnt + 5;
  int32_t* rank = words;
  int32_t* order = rank + n;
  int32_t* lower = order + n;
  int32_t* higher = lower + n;
  int32_t* taken = higher + n;  // of a vertex's in-list
  uint32_t* kept = reinterpret_cast<uint32_t*>(taken + n);
  uint32_t* fill = kept + (n_adj + 31) / 32;  // entries per row so far
  uint32_t* run_end = fill + n;
  void* scan_scratch = scratch + sort_bytes;

  // 1. ranks (launched before what comes later is allocated)
  uint64_t* sorted = nullptr;
  if (few) {
    EXACT_DO(launch("exact_ranks", s, [&] {
      k_ranks_few<<<(unsigned)((n + 31) / 32), EX_THREADS, 0, s>>>(g->deg, n, order, rank);
    }));
  } else {
    int deg_bits = 1;
    while (deg_bits < 31 && (g->max_degree >> deg_bits) != 0) ++deg_bits;
    EXACT_DO(sort_clear(scratch, n, s));
    EXACT_DO(launch("exact_ranks", s, [&] {
      k_degree_keys<<<some_blocks(n), EX_THREADS, 0, s>>>(g->deg, n, (deg_bits + 7) / 8, keys, sort_hist_area(scratch));
    }));
    EXACT_DO(radix_sort_u64(keys, alt, n, deg_bits, scratch, ctl, s, &sorted, SortScratch::cleared, 32));
    EXACT_DO(launch("exact_ranks", s, [&] { k_ranks<<<blocks_for(n), EX_THREADS, 0, s>>>(sorted, n, order, rank); }));
  }

  // the bins as ranges of ranks (bin_lo, n)
  std::vector<uint32_t> bin_lo(nb + 1, 0);  // bin 0: degree 0
  uint64_t below = (uint64_t)n;
  for (uint32_t k = 0; k < nb; ++k) below -= inf.n_b[k];
  for (uint32_t k = 1; k < nb; ++k) {
    bin_lo[k] = (uint32_t)below;
    below += inf.n_b[k];
  }
  bin_lo[nb] = (uint32_t)n;
  uint32_t* d_bin_lo = reinterpret_cast<uint32_t*>(pbq + n_cnt);
  EXACT_TRY(cudaMemcpyAsync(d_bin_lo, bin_lo.data(), (nb + 1) * sizeof(uint32_t), cudaMemcpyHostToDevice, s));

  // 2. neighbours of lower and higher rank, in-list and row offsets
  EXACT_DO(dalloc_n(&offs, 2 * (size_t)n + 1, s, "wedge_exact: offsets"));
  EXACT_DO(dalloc_n(&rows, (size_t)m + 2 * (size_t)most, s, "wedge_exact: rows"));
  EXACT_DO(dalloc_n(&units, (size_t)max_units, s, "wedge_exact: units"));
  int64_t* in_off = offs;
  int64_t* row_off = offs + n;  // (row_off[0] = in_off[n] = m)
  uint32_t* v_of = rows + m;
  uint32_t* u_of = v_of + most;
  EXACT_TRY(cudaMemsetAsync(lower, 0, 3 * (size_t)n * sizeof(int32_t), s));
  if (grouped) EXACT_TRY(cudaMemsetAsync(fill, 0, (size_t)n * sizeof(int32_t), s));
  // a warp takes fewer entries where there are too few for all warps
  const int steps = (int)std::max<int64_t>(1, std::min<int64_t>(OR_STEPS, n_adj / ((int64_t)sm_count() * 64 * 32)));
  const int64_t tile = (int64_t)EX_WARPS * 32 * steps;
  const unsigned tiles = (unsigned)((n_adj + tile - 1) / tile);
  OrientArgs oa{};
  oa.off = g->off;
  oa.adj = g->adj;
  oa.rank = rank;
  oa.n = n;
  oa.n_adj = n_adj;
  oa.steps = steps;
  oa.lower = lower;
  oa.higher = higher;
  oa.kept = kept;
  oa.down = down;
  EXACT_DO(launch("exact_orient", s, [&] { k_orient<false><<<tiles, EX_THREADS, 0, s>>>(oa); }));
  const int key_bits = (int)g->id_bits;
  if (!grouped) {
    EXACT_DO(sort_clear(scratch, m, s));
    EXACT_DO(launch("exact_row_sums", s, [&] {
      k_row_sums<<<some_blocks(n), EX_THREADS, 0, s>>>(lower, higher, n, (key_bits + 7) / 8, down, m,
                                                       sort_hist_area(scratch), ctl + 6);
    }));
  }
  const bool ask = !grouped && n_adj >= ASK_ENTRIES;
  if (ask) EXACT_TRY(any.start(ctl + 6, 4, s));
  EXACT_DO(scan_i32_to_i64(lower, offs, 2 * (int64_t)n, offs + 2 * (size_t)n, scan_scratch, ctl, s));
  if (ask) {
    EXACT_TRY(any.wait());
    const bool half = any.words[2] == (uint32_t)m && any.words[3] == (uint32_t)(m >> 32);
    if (half && (!any.words[0] || !any.words[1])) {
      std::fill(pbq_out, pbq_out + n_cnt, 0ULL);
      EXACT_TRY(cudaStreamSynchronize(s));
      return done(WEDGE_OK);
    }
  }
  oa.lower = taken;
  oa.m = m;
  oa.places = most;
  oa.err = ctl;

  // 3-4. groups of ranks, highest first
  {
    auto in_at = [&](int32_t r, int64_t* x) {  // in_off[r]
      cudaError_t e = cudaMemcpyAsync(x, in_off + r, sizeof(*x), cudaMemcpyDeviceToHost, s);
      return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
    };
    std::vector<std::pair<int32_t, int64_t>> cut{{n, m}};  // ends of the groups, from the top: rank, in_off there
    if (grouped) {
      int64_t all = 0;
      EXACT_TRY(in_at(n, &all));
      if (all != m) return done(exact_not_symmetric());
      while (cut.back().second > 0) {
        const int64_t top = cut.back().second;
        int32_t lo = 0, hi = cut.back().first - 1;  // least rank whose group [rank, end) is at most cap
        int64_t at = 0;
        while (lo < hi) {
          const int32_t mid = lo + (hi - lo) / 2;
          EXACT_TRY(in_at(mid, &at));
          if (top - at <= cap) hi = mid; else lo = mid + 1;
        }
        EXACT_TRY(in_at(lo, &at));
        cut.push_back({lo, at});
      }
    } else {
      cut.push_back({0, 0});
    }
    constexpr auto mid_kernel = k_tri_hash_cta<MID_THREADS, MID_SLOTS, MID_BITS>;
    constexpr auto big_kernel = k_tri_hash_cta<BIG_THREADS, BIG_SLOTS, BIG_BITS>;
    constexpr size_t mid_smem = sizeof(CtaSmem<MID_THREADS, MID_SLOTS, MID_BITS>);
    constexpr size_t big_smem = sizeof(CtaSmem<BIG_THREADS, BIG_SLOTS, BIG_BITS>);
    static OncePerDevice once;
    static CtasPerSm warp_occupancy, mid_occupancy, big_occupancy;
    EXACT_DO(once([&] { return allow_shared(big_kernel, big_smem, "wedge_exact: shared memory"); }));
    const int warp_ctas = warp_occupancy(k_tri_hash_warp, EX_THREADS, 0);
    const int mid_ctas = mid_occupancy(mid_kernel, MID_THREADS, mid_smem);
    const int big_ctas = big_occupancy(big_kernel, BIG_THREADS, big_smem);
    const int sms = sm_count();
    const int64_t longest = longest_row(inf, g->max_degree);
    for (size_t gi = 0; gi + 1 < cut.size(); ++gi) {
      const int32_t r1 = cut[gi].first, r0 = cut[gi + 1].first;
      const int64_t edges = cut[gi].second - cut[gi + 1].second;
      if (edges == 0) continue;
      oa.in_off = in_off;
      oa.r0 = r0;
      oa.r1 = r1;
      oa.keys = keys;
      oa.v_of = v_of;
      oa.u_of = u_of;
      EXACT_DO(launch("exact_edges", s, [&] { k_orient<true><<<tiles, EX_THREADS, 0, s>>>(oa); }));
      EXACT_DO(radix_sort_u64(keys, alt, edges, key_bits, scratch, ctl, s, &sorted,
                              grouped ? SortScratch::unused : SortScratch::cleared, 32));
      uint32_t* tail_of = reinterpret_cast<uint32_t*>(sorted == keys ? alt : keys);  // the sort's other buffer
      EXACT_DO(launch("exact_rows", s, [&] {
        const unsigned blocks = blocks_for(edges);
        if (edges == m) {
          k_rows<true><<<blocks, EX_THREADS, 0, s>>>(sorted, edges, (uint32_t)n, down, v_of, row_off, run_end, fill,
                                                     rows, m, tail_of, ctl);
        } else {
          k_run_ends<<<blocks, EX_THREADS, 0, s>>>(sorted, edges, run_end);
          k_rows<false><<<blocks, EX_THREADS, 0, s>>>(sorted, edges, (uint32_t)n, down, v_of, row_off, run_end, fill,
                                                      rows, m, tail_of, ctl);
          k_run_add<<<blocks, EX_THREADS, 0, s>>>(sorted, edges, run_end, fill);
        }
      }));
      CountArgs ca{};
      ca.in_off = in_off;
      ca.row_off = row_off;
      ca.rows = rows;
      ca.u_of = u_of;
      ca.places = most;
      ca.tail_of = tail_of;
      ca.order = order;
      ca.bin_lo = d_bin_lo;
      ca.nb = nb;
      ca.n = (uint32_t)n;
      ca.m = m;
      ca.r0 = r0;
      ca.r1 = r1;
      ca.pbq = pbq;
      ca.t_i = t_i;
      ca.down = down;
      ca.err = ctl;
      ca.next = ctl + 1;
      ca.map_ranks = lim.map_ranks;
      ca.table_row = lim.table_row;
      ca.units = units;
      ca.max_units = (uint32_t)max_units;
      ca.n_units = ctl + 2;
      ca.grab = vertices_per_ticket(r1 - r0, (int64_t)sms * warp_ctas * EX_WARPS, GRAB);
      if (gi > 0) EXACT_TRY(cudaMemsetAsync(ctl + 1, 0, 5 * sizeof(uint32_t), s));
      EXACT_DO(launch("exact_hash_warp", s, [&] { k_tri_hash_warp<<<sms * warp_ctas, EX_THREADS, 0, s>>>(ca); }));
      // (their work lists are on the device; not launched where nothing can be in them)
      if (g->max_degree > WARP_IN)
        EXACT_DO(launch("exact_hash_cta", s, [&] {
          mid_kernel<<<sms * mid_ctas, MID_THREADS, mid_smem, s>>>(ca, units, 1, ctl + 2, ctl + 4);
        }));
      if (longest > MID_ROW)
        EXACT_DO(launch("exact_hash_cta_long", s, [&] {
          big_kernel<<<sms * big_ctas, BIG_THREADS, big_smem, s>>>(ca, units + (max_units - 1), -1, ctl + 3, ctl + 5);
        }));
    }
  }
  uint32_t herr = 0;
  EXACT_TRY(cudaMemcpyAsync(pbq_out, pbq, n_cnt * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
  EXACT_TRY(cudaMemcpyAsync(&herr, ctl, sizeof(herr), cudaMemcpyDeviceToHost, s));
  EXACT_TRY(cudaStreamSynchronize(s));
#undef EXACT_TRY
#undef EXACT_DO
  if (herr & DERR_TIMEOUT) return done(fail(WEDGE_ETIMEOUT, "wedge_exact: a look-back wait gave up"));
  if (herr & DERR_BOUNDS) return done(exact_out_of_bounds());
  if (herr & DERR_BAD_ID) return done(exact_not_symmetric());
  return done(WEDGE_OK);
}

namespace {

// Entries of whole rows N+(v) that exact_rows would stream per edge (u, v), by the
// bins: in a bin of mean degree d (of its wedges), a vertex has about d / 2 edges from
// below and as many to above, but no more than there are vertices in its bin and
// those after.
double streamed_per_edge(const wedge_bins_info& inf, int64_t m) {
  double entries = 0, above = -1;
  for (uint32_t k = inf.n_bins; k-- > 1;) {
    const double n_b = (double)inf.n_b[k];
    if (n_b == 0) continue;
    above += n_b;
    const double d = k == 1 ? 1.0 : 0.5 * (1.0 + std::sqrt(1.0 + 8.0 * (double)inf.p_b[k] / n_b));
    entries += n_b * d * std::min(d, above) / 4.0;
  }
  return entries / (double)m;
}

// Whether whole rows are streamed (exact_rows.cu) and not tails. Whole rows need no
// ranks and no sort of the edges, about 80 ps an edge and 50 us, but twice
// the entries where degrees are alike and up to four times where they are not, and
// a found triangle costs more. Both forms, us (16.8 M edges unless stated):
//   next to nothing to stream (R <= 2.25 entries an edge): path of 4.2 M 390, 1,430; star
//     1,450, 4,450; grid of 9 M vertices 4,850, 4,840; ring of 1 M with 2 neighbours a side 760, 930;
//   few edges: 0.26 M, power law 3.0 (R = 5) 200, 257, ring (R = 8) 255, 266; 0.52 M, ring
//     (R = 8) 397, 370; uniform (R = 4.5) of 1 M 360, 364; all of 16.8 M 3,990, 3,010;
//   many, degrees alike, next to no triangles: uniform, R = 16 2,190, 2,370; R = 32 2,770, 3,105
//     (67 M 12,140, 15,240: rows, lists and tails are past L2); R = 8 2,630, 2,515. With triangles, a
//     ring of 16 neighbours a side, 13,380, 5,450: so these are asked first, 2,048
//     wedges for 40 us (the forms meet at about one closed in sixty).
bool takes_rows(const wedge_graph* g, const wedge_bins* b, wedge_stream stream) {
  const wedge_bins_info& inf = b->info;
  const int64_t m = g->n_adj / 2;
  const double per_edge = streamed_per_edge(inf, m);
  if (per_edge <= 2.25 || (per_edge <= 9.0 && m <= (1 << 19))) return true;
  const double pairs_per_edge = (double)inf.p_total / (double)m;  // twice R where degrees are alike
  if (m < (1 << 23) || per_edge < 12.0 || pairs_per_edge > 2.3 * per_edge) return false;
  wedge_sample_params sp;
  memset(&sp, 0, sizeof(sp));
  sp.k_global = 2048;
  sp.flags = WEDGE_FLAG_NO_BINS;
  wedge_counts c;
  if (wedge_sample(g, b, &sp, stream, &c) != WEDGE_OK) {
    clear_error();
    return false;
  }
  return c.closed_global <= 20;
}

}  // namespace
}  // namespace wedge

using namespace wedge;

// form: 0 by the rule, 1 tails, 2 whole rows.
static wedge_status exact_counts(const wedge_graph* g, const wedge_bins* b, uint64_t* t_i, wedge_stream stream, int form,
                                 const ExactLimits& lim, wedge_exact_counts* out) {
  clear_error();
  if (!g || !b || !out) return fail(WEDGE_EINVAL, "wedge_exact: NULL argument");
  if (b->graph_uid != g->uid) return fail(WEDGE_EINVAL, "wedge_exact: bins were built from another graph");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const wedge_bins_info& inf = b->info;
  memset(out, 0, sizeof(*out));
  out->n_bins = inf.n_bins;
  out->p_total = inf.p_total;
  for (uint32_t k = 0; k < inf.n_bins; ++k) out->p_b[k] = inf.p_b[k];
  if (t_i) WEDGE_CUDA_TRY(cudaMemsetAsync(t_i, 0, (size_t)g->n * sizeof(uint64_t), s), "wedge_exact");
  if (g->n_adj == 0) {
    for (uint32_t k = 0; k < inf.n_bins; ++k) out->pbq[k][0] = inf.p_b[k];
    return WEDGE_OK;
  }
  unsigned long long pbq[WEDGE_MAX_BINS * 4];
  unsigned long long* ti = reinterpret_cast<unsigned long long*>(t_i);
  const bool rows = form == 0 ? takes_rows(g, b, stream) : form == 2;
  wedge_status st = rows ? exact_rows(g, b, ti, s, pbq) : exact_tails(g, b, ti, s, lim, pbq);
  if (st == WEDGE_ENOMEM && !rows && form == 0) {  // the other form needs less
    clear_error();
    st = exact_rows(g, b, ti, s, pbq);
  }
  if (st != WEDGE_OK) return st;
  uint64_t closed = 0;
  for (uint32_t k = 0; k < inf.n_bins; ++k) {
    uint64_t sum = 0;
    for (int q = 1; q <= 3; ++q) {
      out->pbq[k][q] = pbq[(size_t)k * 4 + q];
      sum += out->pbq[k][q];
    }
    out->pbq[k][0] = inf.p_b[k] - sum;
    closed += sum;
  }
  out->triangles = closed / 3;
  return WEDGE_OK;
}

extern "C" wedge_status wedge_exact(const wedge_graph* g, const wedge_bins* b, uint64_t* t_i, wedge_stream stream,
                                    wedge_exact_counts* out) {
  return exact_counts(g, b, t_i, stream, 0, ExactLimits(), out);
}

extern "C" wedge_status wedge_test_exact(const wedge_graph* g, const wedge_bins* b, uint64_t* t_i, wedge_stream stream,
                                         int form, int64_t group_edges, uint32_t map_ranks, uint32_t table_row,
                                         wedge_exact_counts* out) {
  clear_error();
  if (form < 0 || form > 2 || group_edges < 1) return fail(WEDGE_EINVAL, "wedge_test_exact: form or group out of range");
  ExactLimits lim;
  lim.group_edges = std::min(group_edges, lim.group_edges);
  lim.map_ranks = map_ranks;
  lim.table_row = table_row;
  return exact_counts(g, b, t_i, stream, form, lim, out);
}
