// exact.cuh — what the two forms of wedge_exact share (exact.cu, exact_rows.cu).
#pragma once

#include <algorithm>
#include <atomic>

#include "device.cuh"
#include "internal.h"
#include "runtime.h"

namespace wedge {

// Sizes of the tails' form that a test may lower, to take graphs of a few thousand
// edges through what else takes millions: in-edges of a group (unless one vertex
// has more), ranks of a CTA's bit map, entries of a row in a CTA's hash table (no
// more than the kernels' own).
struct ExactLimits {
  int64_t group_edges = int64_t(1) << 27;
  uint32_t map_ranks = ~0u;
  uint32_t table_row = ~0u;
};

// Enumerates the triangles: adds to t_i (device, zeroed; or nullptr) and fills
// pbq (host, [n_bins][4], classes 1 to 3). Both synchronise s; all of their device
// memory is allocated before anything is added to t_i.
wedge_status exact_tails(const wedge_graph* g, const wedge_bins* b, unsigned long long* t_i, cudaStream_t s,
                         const ExactLimits& lim, unsigned long long* pbq);
wedge_status exact_rows(const wedge_graph* g, const wedge_bins* b, unsigned long long* t_i, cudaStream_t s,
                        unsigned long long* pbq);

inline wedge_status exact_not_symmetric() {
  return fail(WEDGE_EINVAL, "wedge_exact: the graph's CSR is not symmetric");
}

inline wedge_status exact_out_of_bounds() {
  return fail(WEDGE_ECUDA, "wedge_exact: an index outside its buffer (bounds-checked build)");
}

// The most neighbours of higher (degree, id) that a vertex can have, by the bins.
inline int64_t longest_row(const wedge_bins_info& inf, int32_t max_degree) {
  int64_t longest = 0, above = -1;  // vertices of the bin and those after it, but for one
  for (uint32_t k = inf.n_bins; k-- > 1;) {
    above += (int64_t)inf.n_b[k];
    if (inf.n_b[k])
      longest = std::max(longest, std::min(above, (int64_t)std::min(inf.hi_deg[k], (uint64_t)max_degree)));
  }
  return longest;
}

// CTAs of a kernel that the current device's SMs hold, asked for once a device.
class CtasPerSm {
 public:
  template <typename F>
  int operator()(F* f, int threads, size_t smem) {
    int dev = -1, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) dev = 0;
    if ((n = n_[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, threads, smem) != cudaSuccess) {
      cudaGetLastError();
      return 1;
    }
    n = std::max(n, 1);
    n_[dev].store(n, std::memory_order_relaxed);
    return n;
  }

 private:
  std::atomic<int> n_[MAX_DEVICES] = {};
};

// Vertices that a warp takes per ticket: few where there are few for each warp.
inline uint32_t vertices_per_ticket(int64_t vertices, int64_t warps, int64_t most) {
  return (uint32_t)std::max<int64_t>(1, std::min<int64_t>(most, vertices / (4 * warps)));
}

// Largest u in [0, n) with off[u] <= e (off ascending, off[0] = 0 <= e).
__device__ __forceinline__ int32_t row_of(const int64_t* __restrict__ off, int32_t n, int64_t e) {
  int32_t lo = 0, hi = n;
  while (hi - lo > 1) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(off + mid) <= e) lo = mid; else hi = mid;
  }
  return lo;
}

// Row of entry e, given a row u with off[u] <= e: up to 32 steps forward
// over consecutive (cached) offsets, the common case even with isolated
// vertices, then a binary search, so a long run of empty rows costs O(log n)
// instead of one step each.
__device__ __forceinline__ int32_t next_row(const int64_t* __restrict__ off, int32_t n, int32_t u, int64_t e) {
#pragma unroll 1
  for (int t = 0; t < 32; ++t) {
    if (e < __ldg(off + u + 1)) return u;
    ++u;
  }
  int32_t lo = u, hi = n;  // off[lo] <= e < off[n]
  while (hi - lo > 1) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(off + mid) <= e) lo = mid; else hi = mid;
  }
  return lo;
}

}  // namespace wedge
