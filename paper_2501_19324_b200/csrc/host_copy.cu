// Copies of megabytes from the device into memory of the caller's that is not page-locked.
// cudaMemcpy moves them through the driver's buffers with one thread, which also takes the faults of pages that nobody has touched: that thread is the bound,
// not the bus (50 GB/s).  Here the bus fills page-locked chunks of the context's while several threads empty them.  Milliseconds, cudaMemcpy / here:
//   new pages of 4 KB, 14.6 MB 6.6 / 1.3, 210 MB 92 / 13.8; of 2 MB 3.7 / 1.1, 43 / 11.3; pages already there, 2 MB 0.127 / 0.126, 16.8 MB 0.83 / 0.68, 134 MB 8.0 / 5.0.
// 14.6 MB into new 4 KB pages with 1 / 2 / 4 / 8 / 12 threads 4.4 / 2.8 / 2.0 / 1.3 / 1.1; chunks of 256 KB 1.5, of 1 MB 1.4.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <exception>
#include <thread>

#include "common.cuh"
#include "kernels.cuh"

namespace rsd {

namespace {
constexpr size_t kChunk = 512 << 10;
constexpr int kThreads = 8, kSlots = 16;      // chunks on the bus or being emptied
}  // namespace

size_t host_copy_staging_bytes() { return kChunk * kSlots; }

// Ordered like cudaMemcpy: everything goes through the default stream.  The threads call nothing of CUDA's.
cudaError_t copy_to_host(void* out, const void* src, size_t bytes, void* staging) {
  cudaPointerAttributes attr{};
  // Below 2 MB starting threads costs what they save where the pages are there.  Memory that the driver knows needs no chunks.
  if (!staging || bytes < 4 * kChunk || cudaPointerGetAttributes(&attr, out) != cudaSuccess || attr.type != cudaMemoryTypeUnregistered) {
    (void)cudaGetLastError();
    return cudaMemcpy(out, src, bytes, cudaMemcpyDeviceToHost);
  }
  const size_t n = (bytes + kChunk - 1) / kChunk;
  auto size = [&](size_t i) { return std::min(kChunk, bytes - i * kChunk); };
  auto slot = [&](size_t i) { return (char*)staging + i % kSlots * kChunk; };
  std::atomic<size_t> arrived{0}, next{0}, emptied[kSlots] = {};      // emptied: one more than the last chunk taken out of the slot
  std::atomic<bool> stop{false};
  auto work = [&] {
    for (size_t i; (i = next.fetch_add(1)) < n;) {
      while (arrived.load(std::memory_order_acquire) <= i) {
        if (stop.load()) return;
        std::this_thread::yield();
      }
      std::memcpy((char*)out + i * kChunk, slot(i), size(i));
      emptied[i % kSlots].store(i + 1, std::memory_order_release);
    }
  };
  cudaEvent_t ev[kSlots] = {};
  cudaError_t rc = cudaSuccess;
  for (int s = 0; s < kSlots && rc == cudaSuccess; ++s) rc = cudaEventCreateWithFlags(&ev[s], cudaEventDisableTiming);
  std::thread threads[kThreads];
  int n_threads = 0;
  if (rc == cudaSuccess) {
    const int want = (int)std::min<size_t>({(size_t)kThreads, n / 2, std::max(2u, std::thread::hardware_concurrency()) - 1});
    try {
      for (; n_threads < want; ++n_threads) threads[n_threads] = std::thread(work);
    } catch (const std::exception&) {          // those that there are take all the chunks
    }
    if (n_threads == 0) rc = cudaMemcpy(out, src, bytes, cudaMemcpyDeviceToHost);
  }
  for (size_t asked = 0, done = 0; n_threads > 0 && rc == cudaSuccess && done < n;) {
    for (; rc == cudaSuccess && asked < n && asked < done + kSlots; ++asked) {
      if (asked >= kSlots && emptied[asked % kSlots].load(std::memory_order_acquire) != asked - kSlots + 1) break;
      rc = cudaMemcpyAsync(slot(asked), (const char*)src + asked * kChunk, size(asked), cudaMemcpyDeviceToHost, cudaStreamLegacy);
      if (rc == cudaSuccess) rc = cudaEventRecord(ev[asked % kSlots], cudaStreamLegacy);
    }
    if (rc != cudaSuccess) break;
    if (done == asked) {                       // every slot is being emptied
      std::this_thread::yield();
      continue;
    }
    rc = cudaEventSynchronize(ev[done % kSlots]);
    if (rc == cudaSuccess) arrived.store(++done, std::memory_order_release);
  }
  if (rc == cudaSuccess && n_threads > 0) work();
  stop.store(true);
  for (int t = 0; t < n_threads; ++t) threads[t].join();
  if (rc != cudaSuccess) (void)cudaStreamSynchronize(cudaStreamLegacy);      // nothing is on its way to the chunks any more
  for (cudaEvent_t e : ev)
    if (e) cudaEventDestroy(e);
  return rc;
}

}  // namespace rsd
