// bins.cu — degree bins and per-bin wedge totals (wedge_bin).
//
// Sec. 4.2 defines the bins; Alg. Phase 1b sums, per bin, the vertex count
// n_b and the wedge count p_b = sum C(d,2). Here one pass over the degree
// array counts per (bin, tile) in shared memory, an exclusive scan over the
// bin-major (bin, tile) count matrix gives every tile its output position in
// each bin, and a second pass writes the vertices of degree >= 2 in (bin, id)
// order (L) beside their degrees; one exclusive scan of their C(d,2) gives the
// running wedge prefix W over L (W[j] - W[start of bin b] is the
// wedge prefix within bin b). W is what the sampler's inverse-CDF centre
// search runs on (Sec. 3.2).
#include <string.h>

#include <vector>

#include "device.cuh"
#include "internal.h"
#include "runtime.h"

namespace wedge {
namespace {

constexpr int BIN_THREADS = 256;
constexpr int BIN_WARPS = BIN_THREADS / 32;
// (bin, tile) counts that are read back as a whole: one copy instead of a strided
// one and another for the end (wedge_bin at scale 12 93 -> 85 us, 20 104 -> 99, 22
// with 20,000 counts 129 -> 126; more would be a quarter of a megabyte and up).
constexpr int64_t SMALL_MATRIX = 1 << 15;
constexpr int BIN_ITEMS = 16;
constexpr int BIN_TILE = BIN_THREADS * BIN_ITEMS;

// BinId by bit length: degrees of B significant bits lie in bins
// range[B] & 0xffff .. range[B] >> 16, of which there are one or two where
// bins grow by 2, so that one comparison finds the bin and not a search of the
// whole table (35 of the count pass's 86 instructions a warp and vertex).
struct DegreeBins {
  uint32_t lo[WEDGE_MAX_BINS];  // BinLoDeg, cut off at 2^31
  uint32_t range[33];

  __device__ __forceinline__ void load(const uint64_t* __restrict__ lo_g, uint32_t nb) {  // (all threads; synchronises)
    for (uint32_t i = threadIdx.x; i < nb; i += BIN_THREADS) lo[i] = (uint32_t)min(lo_g[i], (uint64_t)1 << 31);
    __syncthreads();
    if (threadIdx.x < 33) {
      const uint32_t least = threadIdx.x ? 1u << (threadIdx.x - 1) : 0u, most = threadIdx.x ? least - 1u + least : 0u;
      range[threadIdx.x] = search(least, 0, nb - 1) | (search(most, 0, nb - 1) << 16);
    }
    __syncthreads();
  }
  // Last k in [k, e] with lo[k] <= d, given lo[k] <= d.
  __device__ __forceinline__ uint32_t search(uint32_t d, uint32_t k, uint32_t e) const {
    while (k < e) {
      const uint32_t mid = (k + e + 1) >> 1;
      if (lo[mid] <= d) k = mid; else e = mid - 1;
    }
    return k;
  }
  __device__ __forceinline__ uint32_t of(int32_t d) const {  // d >= 0
    const uint32_t r = range[32 - __clz(d)];
    return search((uint32_t)d, r & 0xffffu, r >> 16);
  }
};

// Four degrees from vertex v (a multiple of 4) on; zeros past the end.
__device__ __forceinline__ int4 load_degrees(const int32_t* __restrict__ deg, int32_t n, int64_t v) {
  if (v + 4 <= n) return __ldg(reinterpret_cast<const int4*>(deg + v));
  int4 d = make_int4(0, 0, 0, 0);
  if (v < n) d.x = __ldg(deg + v);
  if (v + 1 < n) d.y = __ldg(deg + v + 1);
  if (v + 2 < n) d.z = __ldg(deg + v + 2);
  return d;
}

// Row of bin b in the (bin, tile) count matrix: the bins that L holds (2 and
// up) in order, then bin 1, so that one scan of the matrix gives both the
// places in L and every n_b. (Bin 0 is empty: degree-0 vertices have no bin.)
__host__ __device__ inline uint32_t mat_row(uint32_t b, uint32_t nb) { return b >= 2 ? b - 2 : nb - 2; }

// Counts the vertices of each (bin, tile). Most vertices lie in a few bins, so
// every lane has counters of its own. Degrees come four at a time. Bound by
// instructions (scale 24, 16.8 M vertices, tau = 2: 72 us with peers gathered
// per increment and bins searched over the table, 32 us so; reading the
// degrees takes 10).
__global__ __launch_bounds__(BIN_THREADS) void k_bin_count(const int32_t* __restrict__ deg, int32_t n,
                                                           const uint64_t* __restrict__ lo_g, uint32_t nb,
                                                           int64_t n_tiles, uint32_t* __restrict__ mat_cnt,
                                                           uint32_t* err) {
  __shared__ DegreeBins s_bins;
  extern __shared__ uint32_t s_n[];  // [bin][lane]
  const int tid = threadIdx.x;
  const int64_t tile = blockIdx.x;
  const int64_t tbase = tile * BIN_TILE;
  if (tile == 0 && tid == 0) *err = 0u;  // first in the stream: nothing has been reported yet
  int4 d[BIN_ITEMS / 4];
#pragma unroll
  for (int i = 0; i < BIN_ITEMS / 4; ++i) d[i] = load_degrees(deg, n, tbase + 4 * (i * BIN_THREADS + tid));
  for (int i = tid; i < (int)nb * 32; i += BIN_THREADS) s_n[i] = 0;
  s_bins.load(lo_g, nb);
  uint32_t* mine = s_n + (tid & 31);
#pragma unroll
  for (int i = 0; i < BIN_ITEMS / 4; ++i) {
    if (d[i].x > 0) atomicAdd(mine + 32 * s_bins.of(d[i].x), 1u);
    if (d[i].y > 0) atomicAdd(mine + 32 * s_bins.of(d[i].y), 1u);
    if (d[i].z > 0) atomicAdd(mine + 32 * s_bins.of(d[i].z), 1u);
    if (d[i].w > 0) atomicAdd(mine + 32 * s_bins.of(d[i].w), 1u);
  }
  __syncthreads();
  // (bins >= 2 hold exactly the vertices of degree >= 2: bin 1 is {1})
  for (uint32_t b = 1 + (tid >> 5); b < nb; b += BIN_WARPS) {
    const uint32_t c = __reduce_add_sync(FULL_MASK, s_n[32 * b + (tid & 31)]);
    if ((tid & 31) == 0) mat_cnt[mat_row(b, nb) * n_tiles + tile] = c;
  }
}

// Per bin the cells of its guide: as many as GUIDE_PER vertices share one (up
// to twice that, cells being powers of two wide), so a sample's centre is
// found by one look into the guide and two or three halvings instead of
// log2(n_b) (sampling kernel at Kronecker scale 22, 16.3 M samples: 1.24 to
// 1.05 ms; 2 or 1 vertices a cell: no faster).
constexpr int BOUND_THREADS = WEDGE_MAX_BINS + 32;

// W at the bin boundaries: bound[k] = W[start of bin k], k = 0 .. nb (bins 0
// and 1 hold no vertex of L; starts of the others from the scanned matrix), so
// p_b = bound[b + 1] - bound[b]; and the guide table. One thread per boundary.
__global__ __launch_bounds__(BOUND_THREADS) void k_bin_bounds(const int64_t* __restrict__ pos_base, int64_t n_tiles,
                                                              int64_t n2, uint32_t nb, const uint64_t* __restrict__ W,
                                                              unsigned long long* __restrict__ bound,
                                                              int64_t* __restrict__ starts,
                                                              GuideBin* __restrict__ gtab) {
  __shared__ unsigned long long s_bound[WEDGE_MAX_BINS + 1];
  __shared__ int64_t s_start[WEDGE_MAX_BINS + 1];
  const uint32_t k = threadIdx.x;
  if (k <= nb) {
    const int64_t start = k < 2 ? 0 : k < nb ? pos_base[mat_row(k, nb) * n_tiles] : n2;
    starts[k] = s_start[k] = start;
    bound[k] = s_bound[k] = W[start];
  }
  __syncthreads();
  if (k < nb) {
    const uint64_t p = s_bound[k + 1] - s_bound[k];
    const uint64_t cells = max((uint64_t)1, (uint64_t)(s_start[k + 1] - s_start[k]) / GUIDE_PER);
    uint32_t shift = 0;
    while (p > 0 && ((p - 1) >> shift) >= cells) ++shift;
    gtab[k] = GuideBin{s_bound[k], (uint32_t)(s_start[k] / GUIDE_PER + 2 * (int64_t)k), shift};
  }
}

// Fills the guide, four entries of L per thread: the cells that begin inside an
// entry's wedges. A vertex of far more wedges than its bin's others begins many cells;
// its warp then writes them together. A CTA takes GUIDE_CHUNK consecutive
// entries, which lie in one bin more often than not: it is looked up once.
constexpr int GUIDE_CHUNK = 4 * BIN_THREADS;

__device__ __forceinline__ uint32_t bin_at(const int64_t* starts, uint32_t nb, int64_t j) {
  uint32_t lo = 2, hi = nb;  // last bin with start <= j (an empty bin starts where the next does)
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (starts[mid] <= j) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ __launch_bounds__(BIN_THREADS) void k_bin_guide(const uint64_t* __restrict__ W, int64_t n2,
                                                           const int64_t* __restrict__ starts,
                                                           const GuideBin* __restrict__ gtab, uint32_t nb,
                                                           uint32_t* __restrict__ guide, uint64_t guide_len,
                                                           uint32_t* err) {
  __shared__ int64_t s_start[WEDGE_MAX_BINS + 1];
  __shared__ uint32_t s_bin[2];
  const int64_t base = (int64_t)blockIdx.x * GUIDE_CHUNK;
  const int64_t j0 = base + 4 * threadIdx.x;  // (W holds n2 + 1 entries)
  uint64_t w[5];
  if (j0 + 4 <= n2) {
    const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(W + j0));
    const ulonglong2 z = __ldg(reinterpret_cast<const ulonglong2*>(W + j0 + 2));
    w[0] = a.x;
    w[1] = a.y;
    w[2] = z.x;
    w[3] = z.y;
    w[4] = __ldg(W + j0 + 4);
  } else {
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = __ldg(W + min(j0 + i, n2));
  }
  for (int i = threadIdx.x; i <= (int)nb; i += BIN_THREADS) s_start[i] = starts[i];
  __syncthreads();
  if (threadIdx.x < 2) s_bin[threadIdx.x] = bin_at(s_start, nb, threadIdx.x ? min(n2, base + GUIDE_CHUNK) - 1 : base);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint32_t b0 = s_bin[0];
  const bool one_bin = b0 == s_bin[1];
  GuideBin t = gtab[b0];
  int64_t end = s_start[b0 + 1];
  uint64_t c1 = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t j = j0 + i;
    if (!one_bin && j < n2) {
      const uint32_t b = bin_at(s_start, nb, j);
      t = gtab[b];
      end = s_start[b + 1];
    }
    const uint64_t up = (1ULL << t.shift) - 1ULL;
    // its cells, as guide entries (the first is where the entry before ended)
    const uint64_t c0 = one_bin && i > 0 ? c1 : t.at + ((w[i] - t.wlo + up) >> t.shift);
    c1 = j < n2 ? t.at + ((w[i + 1] - t.wlo + up) >> t.shift) : c0;
    uint64_t c_end = j + 1 == end ? c1 + 1 : c1;  // the bin's last also fills the entry past the last cell
    if (j >= n2 || !in_bounds(c_end, guide_len + 1, err)) c_end = c0;
    const bool wide = c_end - c0 > 8;
    if (!wide)
      for (uint64_t c = c0; c < c_end; ++c) guide[c] = (uint32_t)j;
    for (uint32_t todo = __ballot_sync(FULL_MASK, wide); todo; todo &= todo - 1) {
      const int l = __ffs(todo) - 1;
      const uint64_t a = __shfl_sync(FULL_MASK, c0, l), z = __shfl_sync(FULL_MASK, c_end, l);
      const uint32_t v = __shfl_sync(FULL_MASK, (uint32_t)j, l);
      for (uint64_t c = a + lane; c < z; c += 32) guide[c] = v;
    }
  }
}

// Most bins that k_bin_scatter takes; k_bin_scatter_many takes more. In 24.6 KB
// and 522 bytes a bin, four CTAs of the first fit an SM up to 60 bins, and one at
// 256. Both forms, us (Kronecker scale 24 / 2 M vertices of alike degrees): 20
// bins 61, 69 (kron); 36 bins 103, 102 / 27, 27; 49 and 47 bins 129, 109 / 27,
// 31; 62 bins 156, 111 / 41, 33; 139 bins 299, 129; 249 bins 671, 141.
constexpr uint32_t SCATTER_BINS = 52;

// Shared memory of k_bin_scatter.
constexpr size_t scatter_smem(uint32_t nb) {
  return nb * (BIN_THREADS * sizeof(uint16_t) + sizeof(int64_t) + sizeof(uint16_t)) +
         BIN_TILE * (sizeof(int32_t) + sizeof(uint16_t));
}

// Second pass: the vertices of degree >= 2 of each (bin, tile) go to the
// tile's position in the bin, in id order, with their degrees beside them.
// Each thread takes 16 consecutive ids and has a counter of its own per bin;
// per bin, a scan of the threads' counts gives each thread its place, and the
// same counters then hand out the places (counting lane groups by ballots took
// three times the instructions; scale 24: 131 us, so 71 us). The tile is laid out in (bin, id) order in
// shared memory first, so that the writes are runs of a whole tile's bin.
__global__ __launch_bounds__(BIN_THREADS) void k_bin_scatter(const int32_t* __restrict__ deg, int32_t n,
                                                             const uint64_t* __restrict__ lo_g, uint32_t nb,
                                                             int64_t n_tiles, const int64_t* __restrict__ pos_base,
                                                             int32_t* __restrict__ L, int32_t* __restrict__ ldeg,
                                                             int64_t n2, uint32_t* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint16_t* s_cnt = reinterpret_cast<uint16_t*>(smem);                       // [bin][thread]
  int64_t* s_goff = reinterpret_cast<int64_t*>(s_cnt + nb * BIN_THREADS);    // bin's place in L minus its place in the tile
  int32_t* s_deg = reinterpret_cast<int32_t*>(s_goff + nb);                  // BIN_TILE, in (bin, id) order
  uint16_t* s_id = reinterpret_cast<uint16_t*>(s_deg + BIN_TILE);            // BIN_TILE
  uint16_t* s_start = s_id + BIN_TILE;                                       // bin's place in the tile
  __shared__ DegreeBins s_bins;
  __shared__ uint32_t s_total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tile = blockIdx.x;
  const int64_t tbase = tile * BIN_TILE;
  int32_t d[BIN_ITEMS];
#pragma unroll
  for (int i = 0; i < BIN_ITEMS / 4; ++i) {
    const int4 q = load_degrees(deg, n, tbase + tid * BIN_ITEMS + 4 * i);
    d[4 * i] = q.x;
    d[4 * i + 1] = q.y;
    d[4 * i + 2] = q.z;
    d[4 * i + 3] = q.w;
  }
  for (int i = tid; i < (int)nb * BIN_THREADS / 8; i += BIN_THREADS) reinterpret_cast<uint4*>(s_cnt)[i] = make_uint4(0, 0, 0, 0);
  s_bins.load(lo_g, nb);
  uint16_t* mine = s_cnt + tid;
#pragma unroll
  for (int i = 0; i < BIN_ITEMS; ++i)
    if (d[i] >= 2) ++mine[s_bins.of(d[i]) * BIN_THREADS];
  __syncthreads();
  // per bin the threads' places within it (eight threads a lane)
  for (uint32_t b = 2 + warp; b < nb; b += BIN_WARPS) {
    uint4* row = reinterpret_cast<uint4*>(s_cnt + b * BIN_THREADS) + lane;
    const uint4 q = *row;
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t at[8], sum = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      at[k] = sum;
      sum += (w[k / 2] >> (16 * (k & 1))) & 0xffffu;
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL_MASK, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t ex = incl - sum;
    *row = make_uint4((at[0] + ex) | (at[1] + ex) << 16, (at[2] + ex) | (at[3] + ex) << 16,
                      (at[4] + ex) | (at[5] + ex) << 16, (at[6] + ex) | (at[7] + ex) << 16);
    if (lane == 31) s_start[b] = (uint16_t)incl;  // the bin's size, for now
  }
  __syncthreads();
  if (warp == 0) {
    uint32_t run = 0;
    for (uint32_t b0 = 2; b0 < nb; b0 += 32) {
      const uint32_t b = b0 + lane;
      const uint32_t c = b < nb ? s_start[b] : 0u;
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t at = run + incl - c;
      run += __shfl_sync(FULL_MASK, incl, 31);
      if (b < nb) {
        s_start[b] = (uint16_t)at;
        s_goff[b] = pos_base[mat_row(b, nb) * n_tiles + tile] - (int64_t)at;
      }
    }
    if (lane == 0) s_total = run;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < BIN_ITEMS; ++i)
    if (d[i] >= 2) {
      const uint32_t b = s_bins.of(d[i]);
      const uint32_t pos = s_start[b] + mine[b * BIN_THREADS]++;
      s_deg[pos] = d[i];
      s_id[pos] = (uint16_t)(tid * BIN_ITEMS + i);
    }
  __syncthreads();
  const int total = (int)s_total;
  for (int i = tid; i < total; i += BIN_THREADS) {
    const int32_t x = s_deg[i];
    const int64_t at = s_goff[s_bins.of(x)] + i;
    if (in_bounds((uint64_t)at, (uint64_t)n2, err)) {
      L[at] = (int32_t)(tbase + s_id[i]);
      ldeg[at] = x;
    }
  }
}

// The same for many bins. The counters per thread are 512 bytes a bin to clear,
// scan and hold; here a warp takes 32 consecutive ids at a time, the lanes of a bin
// find each other, and a counter per warp and bin gives them their place.
__global__ __launch_bounds__(BIN_THREADS) void k_bin_scatter_many(const int32_t* __restrict__ deg, int32_t n,
                                                                  const uint64_t* __restrict__ lo_g, uint32_t nb,
                                                                  int64_t n_tiles, const int64_t* __restrict__ pos_base,
                                                                  int32_t* __restrict__ L, int32_t* __restrict__ ldeg,
                                                                  int64_t n2, uint32_t* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  int64_t* s_pos = reinterpret_cast<int64_t*>(smem);  // [warp][bin]: counts, then places in L
  __shared__ DegreeBins s_bins;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tile = blockIdx.x;
  const int64_t first = tile * BIN_TILE + warp * (32 * BIN_ITEMS) + lane;
  int32_t d[BIN_ITEMS];
#pragma unroll
  for (int i = 0; i < BIN_ITEMS; ++i) d[i] = first + 32 * i < n ? __ldg(deg + first + 32 * i) : 0;
  for (int i = tid; i < BIN_WARPS * (int)nb; i += BIN_THREADS) s_pos[i] = 0;
  s_bins.load(lo_g, nb);
  int64_t* mine = s_pos + warp * nb;
  const uint32_t lt = lanemask_lt();
  uint32_t bin[BIN_ITEMS], peers[BIN_ITEMS];
#pragma unroll
  for (int i = 0; i < BIN_ITEMS; ++i) {
    bin[i] = d[i] >= 2 ? s_bins.of(d[i]) : 0u;
    peers[i] = __match_any_sync(FULL_MASK, bin[i]);
    if (bin[i] && (peers[i] & lt) == 0) mine[bin[i]] += __popc(peers[i]);
    __syncwarp();
  }
  __syncthreads();
  for (uint32_t b = 2 + tid; b < nb; b += BIN_THREADS) {
    int64_t pos = pos_base[mat_row(b, nb) * n_tiles + tile];
    for (int w = 0; w < BIN_WARPS; ++w) {
      const int64_t c = s_pos[w * nb + b];
      s_pos[w * nb + b] = pos;
      pos += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < BIN_ITEMS; ++i) {
    const int64_t p0 = bin[i] ? mine[bin[i]] : 0;
    __syncwarp();
    if (bin[i]) {
      if ((peers[i] & lt) == 0) mine[bin[i]] = p0 + __popc(peers[i]);
      const int64_t at = p0 + __popc(peers[i] & lt);
      if (in_bounds((uint64_t)at, (uint64_t)n2, err)) {
        L[at] = (int32_t)(first + 32 * i);
        ldeg[at] = d[i];
      }
    }
    __syncwarp();
  }
}

// BinLoDeg table (Eq. BinLoDeg) in integer arithmetic: lo[k] = k for k <= tau,
// then lo[k] = lo[k-1] + omega^(k-1-tau). Saturates at UINT64_MAX.
std::vector<uint64_t> lodeg_table(uint32_t tau, uint64_t omega, uint64_t max_degree, uint32_t* n_bins) {
  std::vector<uint64_t> lo;
  lo.push_back(0);
  uint64_t step = 1;
  for (uint64_t k = 1;; ++k) {
    uint64_t v;
    if (k <= tau) {
      v = k;
    } else {
      const uint64_t prev = lo.back();
      v = (prev > UINT64_MAX - step) ? UINT64_MAX : prev + step;
      step = (step > UINT64_MAX / omega) ? UINT64_MAX : step * omega;
    }
    lo.push_back(v);
    if (v > max_degree || v == UINT64_MAX || lo.size() > WEDGE_MAX_BINS + 1) break;
  }
  // bin ids present: 0 .. last k with lo[k] <= max_degree
  uint32_t nbins = (uint32_t)lo.size() - 1;  // lo.back() > max_degree
  *n_bins = nbins < 2 ? 2 : nbins;
  while (lo.size() < (size_t)*n_bins + 1) lo.push_back(UINT64_MAX);
  return lo;
}

void free_bins(wedge_bins* b, cudaStream_t s) {
  if (!b) return;
  dfree(b->L, s);
  dfree(b->W, s);
  dfree(b->lo_dev, s);
  dfree(b->gtab, s);
  dfree(b->guide, s);
  delete b;
}

}  // namespace
}  // namespace wedge

using namespace wedge;

#define BIN_TRY(expr, what)                                    \
  do {                                                         \
    cudaError_t e__ = (expr);                                  \
    if (e__ != cudaSuccess) return bail(cuda_fail(e__, what)); \
  } while (0)

extern "C" wedge_status wedge_bin(const wedge_graph* g, const wedge_bin_params* bp, wedge_stream stream,
                                  wedge_bins** out) {
  clear_error();
  if (!out) return fail(WEDGE_EINVAL, "wedge_bin: out is NULL");
  *out = nullptr;
  if (!g || !bp) return fail(WEDGE_EINVAL, "wedge_bin: NULL argument");
  if (bp->tau < 1) return fail(WEDGE_EINVAL, "wedge_bin: tau must be >= 1");
  if (bp->omega < 2 || bp->omega >= (1ULL << 32)) return fail(WEDGE_EINVAL, "wedge_bin: omega must be in [2, 2^32)");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

  uint32_t nb = 0;
  std::vector<uint64_t> lo = lodeg_table(bp->tau, bp->omega, (uint64_t)(g->max_degree > 0 ? g->max_degree : 0), &nb);
  if (nb > WEDGE_MAX_BINS)
    return fail(WEDGE_EINVAL, "wedge_bin: max degree %d falls beyond bin id %d (tau=%u too large or omega too small)",
                g->max_degree, WEDGE_MAX_BINS - 1, bp->tau);
  // Wedge-count range check: p <= max_degree * m; keep every prefix below 2^58.
  {
    const unsigned __int128 bound = (unsigned __int128)(uint64_t)(g->max_degree > 0 ? g->max_degree : 0) *
                                    (unsigned __int128)(uint64_t)(g->n_adj / 2 + 1);
    if (bound >= ((unsigned __int128)1 << 58))
      return fail(WEDGE_EOVERFLOW, "wedge_bin: wedge count may exceed 2^58");
  }

  wedge_bins* b = new wedge_bins();
  memset(&b->info, 0, sizeof(b->info));
  b->device = g->device;
  b->graph_uid = g->uid;
  b->pow2 = (bp->tau == 1 && bp->omega == 2) ? 1u : 0u;
  b->L = nullptr;
  b->W = nullptr;
  b->lo_dev = nullptr;
  b->gtab = nullptr;
  b->guide = nullptr;
  uint32_t* mat_cnt = nullptr;
  int64_t* pos_base = nullptr;
  int32_t* ldeg = nullptr;  // degree per entry of L; its C(d,2) are scanned into W
  // (pos_base is followed by, in 8-byte words: the error word, W at the nb + 1
  // bin boundaries, the nb + 1 bin starts; what the host reads lies together)
  void* scratch = nullptr;
  auto release_tmp = [&]() {
    dfree(mat_cnt, s);
    dfree(pos_base, s);
    dfree(ldeg, s);
    dfree(scratch, s);
    mat_cnt = nullptr;
    pos_base = nullptr;
    ldeg = nullptr;
    scratch = nullptr;
  };
  auto bail = [&](wedge_status e) {
    release_tmp();
    free_bins(b, s);
    return e;
  };

  const int32_t n = g->n;
  const int64_t n_tiles = ((int64_t)n + BIN_TILE - 1) / BIN_TILE;
  const int64_t mat = (int64_t)(nb - 1) * n_tiles;  // nb >= 2
  wedge_status st;
  if ((st = dalloc_n(&b->lo_dev, nb, s, "wedge_bin")) != WEDGE_OK) return bail(st);
  if ((st = dalloc_n(&mat_cnt, (size_t)mat, s, "wedge_bin")) != WEDGE_OK) return bail(st);
  if ((st = dalloc_n(&pos_base, (size_t)mat + 2 * (size_t)nb + 4, s, "wedge_bin")) != WEDGE_OK) return bail(st);
  if ((st = dalloc(&scratch, scan_scratch_bytes(mat), s, "wedge_bin")) != WEDGE_OK) return bail(st);
  uint32_t* derr = reinterpret_cast<uint32_t*>(pos_base + mat + 1);
  unsigned long long* sums = reinterpret_cast<unsigned long long*>(pos_base + mat + 2);
  BIN_TRY(cudaMemcpyAsync(b->lo_dev, lo.data(), nb * sizeof(uint64_t), cudaMemcpyHostToDevice, s), "wedge_bin");

  st = launch("bin_count", s, [&] {
    k_bin_count<<<(unsigned)n_tiles, BIN_THREADS, nb * 32 * sizeof(uint32_t), s>>>(g->deg, n, b->lo_dev, nb, n_tiles, mat_cnt,
                                                                                     derr);
  });
  if (st != WEDGE_OK) return bail(st);
  if ((st = scan_u32_with_total(mat_cnt, pos_base, mat, scratch, derr, s)) != WEDGE_OK) return bail(st);

  // the matrix rows' starts (one entry a row), and the total
  std::vector<int64_t> rows(nb + 1);
  std::vector<unsigned long long> bound(nb + 2, 0);  // the error word, W at the bin boundaries
  if (mat <= SMALL_MATRIX) {  // one copy of all of it is shorter than two of parts
    std::vector<int64_t> all((size_t)mat + 2);
    BIN_TRY(cudaMemcpyAsync(all.data(), pos_base, all.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s), "wedge_bin");
    BIN_TRY(cudaStreamSynchronize(s), "wedge_bin");
    for (uint32_t r = 0; r < nb; ++r) rows[r] = all[(size_t)r * n_tiles];  // (nb - 1 rows, and the total)
    rows[nb] = all[(size_t)mat + 1];
  } else {
    BIN_TRY(cudaMemcpy2DAsync(rows.data(), sizeof(int64_t), pos_base, (size_t)n_tiles * sizeof(int64_t),
                              sizeof(int64_t), nb - 1, cudaMemcpyDeviceToHost, s),
            "wedge_bin");
    BIN_TRY(cudaMemcpyAsync(&rows[nb - 1], pos_base + mat, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, s), "wedge_bin");
    BIN_TRY(cudaStreamSynchronize(s), "wedge_bin");
  }
  uint32_t herr = (uint32_t)rows[nb];
  if (herr & DERR_TIMEOUT) return bail(fail(WEDGE_ETIMEOUT, "wedge_bin: a look-back wait gave up"));

  wedge_bins_info& inf = b->info;
  inf.n_bins = nb;
  inf.tau = bp->tau;
  inf.omega = bp->omega;
  int64_t n2 = 0;
  for (uint32_t k = 0; k < nb; ++k) {
    inf.lo_deg[k] = lo[k];
    inf.hi_deg[k] = lo[k + 1] == UINT64_MAX ? UINT64_MAX : lo[k + 1] - 1;
    inf.n_b[k] = k == 0 ? 0 : (uint64_t)(rows[mat_row(k, nb) + 1] - rows[mat_row(k, nb)]);
    inf.start[k] = n2;
    if (k >= 2) n2 += (int64_t)inf.n_b[k];
  }
  for (uint32_t k = nb; k <= WEDGE_MAX_BINS; ++k) inf.start[k] = n2;
  inf.n_wedge_vertices = n2;

  if ((st = dalloc_n(&b->L, (size_t)(n2 > 0 ? n2 : 1), s, "wedge_bin: L")) != WEDGE_OK) return bail(st);
  if ((st = dalloc_n(&b->W, (size_t)n2 + 1, s, "wedge_bin: W")) != WEDGE_OK) return bail(st);
  const size_t guide_len = guide_alloc(n2, nb);
  if ((st = dalloc_n(&b->guide, guide_len, s, "wedge_bin: guide")) != WEDGE_OK) return bail(st);
  if ((st = dalloc_n(&b->gtab, nb, s, "wedge_bin: guide")) != WEDGE_OK) return bail(st);
  if (n2 > 0) {
    if ((st = dalloc_n(&ldeg, (size_t)n2, s, "wedge_bin")) != WEDGE_OK) return bail(st);
    static OncePerDevice once;
    st = once([] { return allow_shared(k_bin_scatter, scatter_smem(SCATTER_BINS), "wedge_bin: shared memory"); });
    if (st != WEDGE_OK) return bail(st);
    const bool many = nb > SCATTER_BINS;
    const size_t smem = many ? BIN_WARPS * nb * sizeof(int64_t) : scatter_smem(nb);
    st = launch("bin_scatter", s, [&] {
      auto* kernel = many ? k_bin_scatter_many : k_bin_scatter;
      kernel<<<(unsigned)n_tiles, BIN_THREADS, smem, s>>>(g->deg, n, b->lo_dev, nb, n_tiles, pos_base, b->L, ldeg, n2,
                                                          derr);
    });
    if (st != WEDGE_OK) return bail(st);
    // W = exclusive prefix of the wedge counts over L, W[n2] = p
    if (scan_scratch_bytes(n2) > scan_scratch_bytes(mat)) {
      dfree(scratch, s);
      scratch = nullptr;
      if ((st = dalloc(&scratch, scan_scratch_bytes(n2), s, "wedge_bin")) != WEDGE_OK) return bail(st);
    }
    if ((st = scan_pairs_with_total(ldeg, b->W, n2, scratch, derr, s, "scan_bin_wedges")) != WEDGE_OK)
      return bail(st);
    int64_t* starts = reinterpret_cast<int64_t*>(sums + nb + 1);
    st = launch("bin_bounds", s, [&] {
      k_bin_bounds<<<1, BOUND_THREADS, 0, s>>>(pos_base, n_tiles, n2, nb, b->W, sums, starts, b->gtab);
    });
    if (st != WEDGE_OK) return bail(st);
    const int64_t gblocks = (n2 + GUIDE_CHUNK - 1) / GUIDE_CHUNK;
    st = launch("bin_guide", s, [&] {
      k_bin_guide<<<(unsigned)gblocks, BIN_THREADS, 0, s>>>(b->W, n2, starts, b->gtab, nb, b->guide, guide_len, derr);
    });
    if (st != WEDGE_OK) return bail(st);
    BIN_TRY(cudaMemcpyAsync(bound.data(), derr, (nb + 2) * sizeof(uint64_t), cudaMemcpyDeviceToHost, s), "wedge_bin");
  } else {
    BIN_TRY(cudaMemsetAsync(b->W, 0, sizeof(uint64_t), s), "wedge_bin");
  }
  BIN_TRY(cudaStreamSynchronize(s), "wedge_bin");
  herr = (uint32_t)bound[0];
  if (herr & DERR_TIMEOUT) return bail(fail(WEDGE_ETIMEOUT, "wedge_bin: a look-back wait gave up"));
  if (herr & DERR_BOUNDS) return bail(fail(WEDGE_ECUDA, "wedge_bin: an index outside its buffer (bounds-checked build)"));
  // p_b: the wedge prefix across bin b's stretch of L
  for (uint32_t k = 0; k < nb; ++k) inf.p_b[k] = bound[k + 2] - bound[k + 1];
  inf.p_total = bound[nb + 1];
  release_tmp();
  inf.L = b->L;
  inf.W = b->W;
  *out = b;
  return WEDGE_OK;
}

#undef BIN_TRY

extern "C" void wedge_bins_free(wedge_bins* b) {
  if (!b) return;
  cudaDeviceSynchronize();
  free_bins(b, nullptr);
}

extern "C" wedge_status wedge_bins_get_info(const wedge_bins* b, wedge_bins_info* out) {
  clear_error();
  if (!b || !out) return fail(WEDGE_EINVAL, "wedge_bins_get_info: NULL argument");
  *out = b->info;
  return WEDGE_OK;
}

extern "C" wedge_status wedge_bins_copy(const wedge_bins* b, int32_t* L, uint64_t* W, wedge_stream stream) {
  clear_error();
  if (!b) return fail(WEDGE_EINVAL, "wedge_bins_copy: NULL bins");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int64_t n2 = b->info.n_wedge_vertices;
  if (L && n2 > 0)
    WEDGE_CUDA_TRY(cudaMemcpyAsync(L, b->L, (size_t)n2 * sizeof(int32_t), cudaMemcpyDefault, s), "wedge_bins_copy");
  if (W)
    WEDGE_CUDA_TRY(cudaMemcpyAsync(W, b->W, ((size_t)n2 + 1) * sizeof(uint64_t), cudaMemcpyDefault, s),
                   "wedge_bins_copy");
  WEDGE_CUDA_TRY(cudaStreamSynchronize(s), "wedge_bins_copy");
  return WEDGE_OK;
}
