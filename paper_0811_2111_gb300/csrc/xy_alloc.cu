// xy_alloc.cu -- the one device-allocation wrapper of the library, with a
// host-side failure hook for tests.
//
// Every cudaMalloc of the library's engines (contexts, batches, HMC, four
// replicas, record growth) goes through xyk::dev_malloc.  xy_debug_fail_alloc
// arms a countdown: the k-th allocation after the call fails with
// cudaErrorMemoryAllocation without reaching the driver, so the engines'
// out-of-memory paths (XY_ENOMEM, nothing leaked, the device still usable) can
// be exercised on a GPU without exhausting its memory.
//
// Also touch_pages: the first touch of a large output array that the caller has
// just allocated.
#include <cuda_runtime.h>
#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <thread>

#include "xy.h"
#include "xy_internal.h"

namespace {

// Allocations left before the armed failure (0: disarmed).
std::atomic<int> g_fail_countdown{0};

}  // namespace

namespace xyk {

cudaError_t dev_malloc_raw(void** p, size_t bytes) {
  int left = g_fail_countdown.load();
  while (left > 0) {
    if (g_fail_countdown.compare_exchange_weak(left, left - 1)) {
      if (left == 1) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
      }
      break;
    }
  }
  return cudaMalloc(p, bytes);
}

// A copy into pages that do not exist yet waits for the kernel to zero them one
// by one: 64 MB of a fresh numpy array took 3.3 ms, of touched pages 0.36 ms.
// Eight threads touching a byte of each page take 0.8 ms, and do so while the
// stream still works.  Nothing is done below kTouchBytes (the allocator hands
// such blocks out again, already touched) or where the pages are resident.
void touch_pages(void* p, size_t bytes) {
  constexpr size_t kTouchBytes = 8u << 20;
  constexpr int kThreads = 8;
  if (!p || bytes < kTouchBytes) return;
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  char* const base = static_cast<char*>(p);
  const uintptr_t first = (reinterpret_cast<uintptr_t>(p) + page - 1) / page * page;
  const size_t pages = (reinterpret_cast<uintptr_t>(p) + bytes - first) / page;
  bool resident = true;
  for (size_t i : {size_t(0), pages / 2, pages - 1}) {
    unsigned char in_core = 0;
    if (mincore(reinterpret_cast<void*>(first + i * page), page, &in_core) != 0) return;
    resident &= (in_core & 1) != 0;
  }
  if (resident) return;
  auto touch = [=](size_t lo, size_t hi) {
    for (size_t i = lo; i < hi; ++i)
      *reinterpret_cast<volatile char*>(base + (first - reinterpret_cast<uintptr_t>(base)) +
                                        i * page) = 0;
  };
  const size_t share = (pages + kThreads - 1) / kThreads;
  std::thread t[kThreads];
  for (int k = 0; k < kThreads; ++k) {
    const size_t lo = std::min(pages, k * share), hi = std::min(pages, lo + share);
    try {
      t[k] = std::thread(touch, lo, hi);
    } catch (...) {                      // no thread to be had: the copy touches the rest itself
    }
  }
  for (std::thread& x : t)
    if (x.joinable()) x.join();
}

}  // namespace xyk

extern "C" {

xy_status xy_debug_fail_alloc(int32_t k) {
  if (k < 0) return XY_EINVAL;
  g_fail_countdown.store(k);
  return XY_OK;
}

}  // extern "C"
