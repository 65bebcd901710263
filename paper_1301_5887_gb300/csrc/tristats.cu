// tristats.cu — statistics of sampled triangles (wedge_triangle_stats).
//
// Sec. 5.7 of the paper samples wedges from one bin of all degrees, keeps
// the closed ones — a uniform sample of triangles (Thm 3.4) — and studies
// degree assortativity: triangles are grouped by the bin (tau = 2, omega = 2)
// of their smallest degree, and for each group the distribution of the
// largest degree is summarised as a box plot. Here, on the device:
//   1. draw k wedges of the global stream with per-sample records;
//   2. append each closed wedge as two sort keys: (BinId22(d_min), d_max) and
//      the IEEE double d_max / d_min (its bit pattern orders like the value);
//   3. radix-sort both key arrays;
//   4. one CTA per d_min bin finds its range and reads off, by nearest rank,
//      the quartiles of d_max, the whiskers (most extreme values within
//      1.5 IQR of the box, in exact integer arithmetic) and the outlier
//      count; the ratio quartiles come from the sorted ratio array.
// Every statistic is an order statistic of integers or of correctly rounded
// divisions, so the result does not depend on the order of appends.
#include <string.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"
#include "runtime.h"

namespace wedge {
namespace {

constexpr int KEY_THREADS = 256;
constexpr int KEY_RECORDS = 8;  // of a thread at a time

// A CTA takes KEY_THREADS * KEY_RECORDS records at a time, whose `closed` words
// are all loaded before the first is looked at, and makes room for its closed
// ones with one atomic. They are few (one in sixty on Kronecker scale 24), so
// they are gathered first and their keys made by full warps: a double division
// occupies the few FP64 units as long for one lane as for 32. 5 M records (160
// MB): 75 us with an atomic and a division per warp and 32 records, 32 so.
__global__ __launch_bounds__(KEY_THREADS) void k_tri_keys(const wedge_record* __restrict__ rec, uint64_t k,
                                                          unsigned long long* __restrict__ n_closed,
                                                          uint64_t* __restrict__ bin_keys,
                                                          uint64_t* __restrict__ ratio_keys) {
  __shared__ uint2 s_degrees[KEY_THREADS * KEY_RECORDS];  // least, largest
  __shared__ uint32_t s_count[KEY_THREADS / 32];
  __shared__ uint32_t s_total;
  __shared__ unsigned long long s_base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr uint64_t TILE = (uint64_t)KEY_THREADS * KEY_RECORDS;
  for (uint64_t t0 = blockIdx.x * TILE; t0 < k; t0 += gridDim.x * TILE) {
    bool closed[KEY_RECORDS];
#pragma unroll
    for (int j = 0; j < KEY_RECORDS; ++j) {
      const uint64_t i = t0 + (uint64_t)j * KEY_THREADS + tid;
      closed[j] = i < k && __ldg(&rec[i].closed) != 0;
    }
    uint32_t mine = 0, bal[KEY_RECORDS];
#pragma unroll
    for (int j = 0; j < KEY_RECORDS; ++j) {
      bal[j] = __ballot_sync(FULL_MASK, closed[j]);
      mine += __popc(bal[j]);
    }
    if (lane == 0) s_count[warp] = mine;
    __syncthreads();
    if (tid == 0) {
      uint32_t total = 0;
      for (int w = 0; w < KEY_THREADS / 32; ++w) {
        const uint32_t c = s_count[w];
        s_count[w] = total;
        total += c;
      }
      s_total = total;
      s_base = total ? atomicAdd(n_closed, (unsigned long long)total) : 0ULL;
    }
    __syncthreads();
    uint32_t slot = s_count[warp];
    const uint32_t below = lanemask_lt();
#pragma unroll
    for (int j = 0; j < KEY_RECORDS; ++j) {
      if (closed[j]) {
        const wedge_record& r = rec[t0 + (uint64_t)j * KEY_THREADS + tid];
        const uint32_t d0 = (uint32_t)r.d0, d1 = (uint32_t)r.d1, d2 = (uint32_t)r.d2;
        s_degrees[slot + __popc(bal[j] & below)] = make_uint2(min(d0, min(d1, d2)), max(d0, max(d1, d2)));
      }
      slot += __popc(bal[j]);
    }
    __syncthreads();
    const uint64_t base = s_base;
    for (uint32_t i = tid; i < s_total; i += KEY_THREADS) {
      const uint2 d = s_degrees[i];
      bin_keys[base + i] = ((uint64_t)stat_bin(d.x) << 32) | d.y;
      ratio_keys[base + i] = (uint64_t)__double_as_longlong(__ddiv_rn((double)d.y, (double)d.x));
    }
    __syncthreads();  // the gathered degrees have been read
  }
}

// Index of the first key >= x in sorted keys[0, n), by a warp: 32 probes at a
// time. The same on every lane.
__device__ __forceinline__ uint64_t lower_bound_u64(const uint64_t* keys, uint64_t n, uint64_t x) {
  const uint32_t lane = threadIdx.x & 31u;
  uint64_t lo = 0, hi = n;  // the index lies in [lo, hi]
  while (lo < hi) {
    const uint64_t step = (hi - lo + 31) / 32;
    const uint64_t at = lo + lane * step;
    const uint32_t less = __ballot_sync(FULL_MASK, at < hi && keys[at] < x);  // lanes 0 .. m - 1
    const uint32_t m = __popc(less);
    if (m == 0) return lo;
    const uint64_t from = lo;
    lo = from + (m - 1) * step + 1;
    hi = min(hi, from + m * step);
  }
  return lo;
}

// Nearest rank: the ceil(p * n)-th smallest (1-based), p = num/den.
__device__ __forceinline__ uint64_t rank_index(uint64_t n, uint64_t num, uint64_t den) {
  uint64_t r = (num * n + den - 1) / den;
  if (r < 1) r = 1;
  return r - 1;
}

// One warp per bin.
__global__ __launch_bounds__(32) void k_tri_box(const uint64_t* __restrict__ keys, uint64_t n,
                                                wedge_triangle_box* __restrict__ out) {
  const uint32_t b = blockIdx.x;
  const uint64_t lo = lower_bound_u64(keys, n, (uint64_t)b << 32);
  const uint64_t hi = lower_bound_u64(keys, n, (uint64_t)(b + 1) << 32);
  wedge_triangle_box box = {};
  box.count = hi - lo;
  if (box.count > 0) {
    const uint64_t c = box.count;
    const uint64_t mask = 0xffffffffULL;
    box.min = keys[lo] & mask;
    box.max = keys[hi - 1] & mask;
    box.q1 = keys[lo + rank_index(c, 1, 4)] & mask;
    box.median = keys[lo + rank_index(c, 1, 2)] & mask;
    box.q3 = keys[lo + rank_index(c, 3, 4)] & mask;
    // whiskers: most extreme values v with 2v >= 2 q1 - 3 IQR and 2v <= 2 q3 + 3 IQR
    const int64_t iqr3 = 3 * ((int64_t)box.q3 - (int64_t)box.q1);
    const int64_t lo2 = 2 * (int64_t)box.q1 - iqr3;   // bound on 2v
    const int64_t hi2 = 2 * (int64_t)box.q3 + iqr3;
    const uint64_t lo_v = lo2 <= 0 ? 0 : (uint64_t)((lo2 + 1) / 2);   // smallest v with 2v >= lo2
    const uint64_t hi_v = (uint64_t)(hi2 / 2);                          // largest v with 2v <= hi2
    const uint64_t a = lower_bound_u64(keys + lo, c, ((uint64_t)b << 32) | lo_v);
    const uint64_t z = lower_bound_u64(keys + lo, c, ((uint64_t)b << 32) | (hi_v + 1));
    box.whisker_lo = a < c ? (keys[lo + a] & mask) : box.min;
    box.whisker_hi = z > 0 ? (keys[lo + z - 1] & mask) : box.max;
    box.outliers = a + (c - z);
  }
  if (threadIdx.x == 0) out[b] = box;
}

__global__ void k_tri_ratio(const uint64_t* __restrict__ keys, uint64_t n, double* __restrict__ q) {
  if (threadIdx.x != 0 || blockIdx.x != 0 || n == 0) return;
  q[0] = __longlong_as_double((long long)keys[0]);
  q[1] = __longlong_as_double((long long)keys[rank_index(n, 1, 4)]);
  q[2] = __longlong_as_double((long long)keys[rank_index(n, 1, 2)]);
  q[3] = __longlong_as_double((long long)keys[rank_index(n, 3, 4)]);
  q[4] = __longlong_as_double((long long)keys[n - 1]);
}

}  // namespace
}  // namespace wedge

using namespace wedge;

extern "C" wedge_status wedge_triangle_stats(const wedge_graph* g, const wedge_bins* b, uint64_t seed, uint64_t k,
                                             void* records, wedge_stream stream, wedge_triangle_summary* out) {
  clear_error();
  if (!g || !b || !out) return fail(WEDGE_EINVAL, "wedge_triangle_stats: NULL argument");
  if (b->graph_uid != g->uid) return fail(WEDGE_EINVAL, "wedge_triangle_stats: bins were built from another graph");
  if (k == 0) return fail(WEDGE_EINVAL, "wedge_triangle_stats: k must be positive");
  if (k > (1ULL << 34)) return fail(WEDGE_EINVAL, "wedge_triangle_stats: k > 2^34");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  memset(out, 0, sizeof(*out));
  out->k = k;

  wedge_record* own_rec = nullptr;
  uint64_t *bin_keys = nullptr, *bin_alt = nullptr, *ratio_keys = nullptr, *ratio_alt = nullptr;
  // what the host reads, in one block: appended keys, error bits, the ratio's
  // quartiles, the boxes
  struct Results {
    unsigned long long n_closed, err;
    double ratio_q[5];
    wedge_triangle_box box[WEDGE_STAT_BINS];
  };
  Results* res = nullptr;
  void* scratch = nullptr;
  auto cleanup = [&](wedge_status st) {
    dfree(own_rec, s);
    dfree(bin_keys, s);
    dfree(bin_alt, s);
    dfree(ratio_keys, s);
    dfree(ratio_alt, s);
    dfree(res, s);
    dfree(scratch, s);
    return st;
  };
  wedge_status st;
  wedge_record* rec = static_cast<wedge_record*>(records);
  if (!rec) {
    if ((st = dalloc_n(&own_rec, (size_t)k, s, "wedge_triangle_stats")) != WEDGE_OK) return cleanup(st);
    rec = own_rec;
  }

  // 1. samples [0, k) of the global stream, with records (synchronises s)
  wedge_sample_params sp;
  memset(&sp, 0, sizeof(sp));
  sp.seed = seed;
  sp.k_global = k;
  sp.flags = WEDGE_FLAG_NO_BINS;
  sp.records = rec;
  wedge_counts counts;
  if ((st = wedge_sample(g, b, &sp, stream, &counts)) != WEDGE_OK) return cleanup(st);
  const uint64_t n = counts.closed_global;
  out->closed = n;
  memcpy(out->hist, counts.stats, sizeof(out->hist));

  const size_t nk = (size_t)std::max<uint64_t>(n, 1);
  if ((st = dalloc_n(&bin_keys, nk, s, "wedge_triangle_stats")) != WEDGE_OK) return cleanup(st);
  if ((st = dalloc_n(&bin_alt, nk, s, "wedge_triangle_stats")) != WEDGE_OK) return cleanup(st);
  if ((st = dalloc_n(&ratio_keys, nk, s, "wedge_triangle_stats")) != WEDGE_OK) return cleanup(st);
  if ((st = dalloc_n(&ratio_alt, nk, s, "wedge_triangle_stats")) != WEDGE_OK) return cleanup(st);
  if ((st = dalloc_n(&res, 1, s, "wedge_triangle_stats")) != WEDGE_OK) return cleanup(st);
  if ((st = dalloc(&scratch, sort_scratch_bytes((int64_t)nk, 64), s, "wedge_triangle_stats")) != WEDGE_OK)
    return cleanup(st);
  uint32_t* derr = reinterpret_cast<uint32_t*>(&res->err);
  cudaError_t e = cudaMemsetAsync(res, 0, sizeof(Results), s);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "wedge_triangle_stats"));

  // 2. one (BinId(d_min), d_max) key and one ratio key per closed sample
  constexpr uint64_t tile = (uint64_t)KEY_THREADS * KEY_RECORDS;
  const unsigned blocks = (unsigned)std::min<uint64_t>((k + tile - 1) / tile, (uint64_t)sm_count() * 8);
  st = launch("triangle_keys", s,
              [&] { k_tri_keys<<<blocks, KEY_THREADS, 0, s>>>(rec, k, &res->n_closed, bin_keys, ratio_keys); });
  if (st != WEDGE_OK) return cleanup(st);

  // 3. sort: BinId(d_min) <= 32 sits in bits 32..37 above d_max < 2^31; a
  //    ratio >= 1 is a positive double, whose bits order like its value
  uint64_t* sorted_bins = bin_keys;
  uint64_t* sorted_ratio = ratio_keys;
  if ((st = radix_sort_u64(bin_keys, bin_alt, (int64_t)n, 38, scratch, derr, s, &sorted_bins)) != WEDGE_OK)
    return cleanup(st);
  if ((st = radix_sort_u64(ratio_keys, ratio_alt, (int64_t)n, 63, scratch, derr, s, &sorted_ratio)) != WEDGE_OK)
    return cleanup(st);

  // 4. box plot per BinId(d_min); ratio order statistics
  st = launch("triangle_box", s, [&] { k_tri_box<<<WEDGE_STAT_BINS, 32, 0, s>>>(sorted_bins, n, res->box); });
  if (st != WEDGE_OK) return cleanup(st);
  st = launch("triangle_ratio", s, [&] { k_tri_ratio<<<1, 32, 0, s>>>(sorted_ratio, n, res->ratio_q); });
  if (st != WEDGE_OK) return cleanup(st);
  Results h;
  e = cudaMemcpyAsync(&h, res, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "wedge_triangle_stats"));
  memcpy(out->box, h.box, sizeof(out->box));
  memcpy(out->ratio_q, h.ratio_q, sizeof(out->ratio_q));
  const uint32_t herr = (uint32_t)h.err;
  const unsigned long long appended = h.n_closed;
  if (herr & DERR_TIMEOUT) return cleanup(fail(WEDGE_ETIMEOUT, "wedge_triangle_stats: a look-back wait gave up"));
  if (appended != n)
    return cleanup(fail(WEDGE_ECUDA, "wedge_triangle_stats: %llu closed records for %llu closed samples", appended,
                        (unsigned long long)n));
  return cleanup(WEDGE_OK);
}
