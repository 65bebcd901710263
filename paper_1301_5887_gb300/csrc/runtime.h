// runtime.h — host-side runtime of the library: error reporting, the
// stream-ordered device memory pool, launch accounting and kernel timing.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>

#include "../../include/wedge.h"

namespace wedge {

// Record a failure message for wedge_last_error() and return `st`.
wedge_status fail(wedge_status st, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
void clear_error();

// Map a CUDA error to a status, recording where it happened.
wedge_status cuda_fail(cudaError_t e, const char* what);

#define WEDGE_CUDA_TRY(expr, what)              \
  do {                                          \
    cudaError_t e__ = (expr);                   \
    if (e__ != cudaSuccess) return cuda_fail(e__, what); \
  } while (0)

// Device memory from the library's pool on the current device (stream-ordered).
wedge_status dalloc(void** p, size_t bytes, cudaStream_t s, const char* what);
void dfree(void* p, cudaStream_t s);
wedge_status trim_pool();

template <typename T>
wedge_status dalloc_n(T** p, size_t n, cudaStream_t s, const char* what) {
  return dalloc(reinterpret_cast<void**>(p), n * sizeof(T), s, what);
}

int sm_count();

constexpr int MAX_DEVICES = 64;

// What a kernel needs done before its first launch on a device (its attributes
// belong to the device): run where it has not succeeded on the current device yet.
// Threads that come first at the same time all run it, so it sets constants:
// a kernel's shared memory limit, say, is that of its largest launch, never of
// one call's, which could come between another's limit and launch.
class OncePerDevice {
 public:
  template <typename F>
  wedge_status operator()(F&& f) {
    int dev = -1;
    WEDGE_CUDA_TRY(cudaGetDevice(&dev), "current device");
    return on(dev, std::forward<F>(f));
  }
  template <typename F>
  wedge_status on(int dev, F&& f) {
    const uint64_t bit = dev >= 0 && dev < MAX_DEVICES ? uint64_t(1) << dev : 0;
    if (done_.load(std::memory_order_acquire) & bit) return WEDGE_OK;
    const wedge_status st = f();
    if (st == WEDGE_OK) done_.fetch_or(bit, std::memory_order_release);
    return st;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

// Lets a kernel be launched with up to `bytes` of dynamic shared memory on the current device.
template <typename K>
wedge_status allow_shared(K* kernel, size_t bytes, const char* what) {
  WEDGE_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), what);
  return WEDGE_OK;
}

// Pinned host blocks, cached by power-of-two size class and reused (pinning
// and unpinning are slow and may synchronise the device).
void* pinned_alloc(size_t bytes);
void pinned_free(void* p, size_t bytes);

// Launch accounting: every kernel launch goes through launch(), which counts
// it and, when timing is enabled, brackets it with CUDA events on `s`.
struct LaunchMark {
  const char* name;
  cudaStream_t stream;
  cudaEvent_t start;
};
LaunchMark launch_begin(const char* name, cudaStream_t s);
wedge_status launch_end(const LaunchMark& m);

template <typename F>
wedge_status launch(const char* name, cudaStream_t s, F&& f) {
  LaunchMark m = launch_begin(name, s);
  std::forward<F>(f)();
  return launch_end(m);
}

// True if the pointer can be dereferenced by kernels on the current device.
bool device_accessible(const void* p);

uint32_t id_bits_for(int64_t n);

}  // namespace wedge
