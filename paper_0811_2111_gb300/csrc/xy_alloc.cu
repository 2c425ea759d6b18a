// xy_alloc.cu -- the library's device-allocation and cooperative-launch wrappers,
// with host-side failure hooks for tests.
//
// Every cudaMalloc of the library's engines (contexts, batches, HMC, four
// replicas, record growth) goes through xyk::dev_malloc.  xy_debug_fail_alloc
// arms a countdown: the k-th allocation after the call fails with
// cudaErrorMemoryAllocation without reaching the driver, so the engines'
// out-of-memory paths (XY_ENOMEM, nothing leaked, the device still usable) can
// be exercised on a GPU without exhausting its memory.
//
// Every cooperative launch goes through xyk::coop_launch; xy_debug_fail_cooperative
// makes the next ones fail as a grid does that finds no room beside other work, so
// that the kernels which then take over can be exercised.
//
// Also xy_touch_pages: the first touch of a large array that the caller has just
// allocated.
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

// Cooperative launches still to fail.
std::atomic<int> g_fail_coop{0};

// MADV_POPULATE_WRITE (Linux 5.14; older headers do not name it).
constexpr int kPopulateWrite = 23;

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

cudaError_t coop_launch(const void* fn, int grid, int threads, void** args, size_t smem,
                        cudaStream_t stream) {
  int left = g_fail_coop.load();
  while (left > 0)
    if (g_fail_coop.compare_exchange_weak(left, left - 1)) return cudaErrorCooperativeLaunchTooLarge;
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, smem, stream);
}

}  // namespace xyk

extern "C" {

xy_status xy_debug_fail_alloc(int32_t k) {
  if (k < 0) return XY_EINVAL;
  g_fail_countdown.store(k);
  return XY_OK;
}

xy_status xy_debug_fail_cooperative(int32_t k) {
  if (k < 0) return XY_EINVAL;
  g_fail_coop.store(k);
  return XY_OK;
}

// A copy into pages that do not exist yet waits for the kernel to zero them one
// by one: 64 MB of a fresh numpy array took 3.3 ms, of touched pages 0.36 ms.
// Eight threads touching a byte of each page take 0.8 ms, and may do so while
// the stream still works.  (Touches that change no byte take longer than the copy
// saves: an atomic OR with zero 24 ms, its read mapping the zero page first;
// MADV_POPULATE_WRITE 2.4 ms, 3.2 with eight threads.  So the get_state calls,
// whose output is the caller's until they copy, touch nothing.)  Nothing is done
// below kTouchBytes (the allocator hands such blocks out again, already touched),
// where the pages are resident, or where the host may not write: three pages are
// asked of the kernel, which refuses where a touch would end the process.
xy_status xy_touch_pages(void* p, int64_t bytes) {
  constexpr int64_t kTouchBytes = 8 << 20;
  constexpr int kThreads = 8;
  if (bytes < 0) return XY_EINVAL;
  if (!p || bytes < kTouchBytes) return XY_OK;
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  char* const base = static_cast<char*>(p);
  char* const first = base + (page - reinterpret_cast<uintptr_t>(p) % page) % page;
  const size_t pages = (size_t)(base + bytes - first) / page;
  const size_t sample[3] = {0, pages / 2, pages - 1};
  bool resident = true;
  for (size_t i : sample) {
    unsigned char in_core = 0;
    if (mincore(first + i * page, page, &in_core) != 0) return XY_OK;
    resident &= (in_core & 1) != 0;
  }
  if (resident) return XY_OK;
  for (size_t i : sample)
    if (madvise(first + i * page, page, kPopulateWrite) != 0) return XY_OK;
  auto touch = [=](size_t lo, size_t hi) {
    for (size_t i = lo; i < hi; ++i) *reinterpret_cast<volatile char*>(first + i * page) = 0;
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
  return XY_OK;
}

}  // extern "C"
