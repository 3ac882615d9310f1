// host_lease.h -- page-locked host memory that kernels read and write in place, borrowed for
// the length of one call (kss_runtime.cu, kss_regrid.cu).  Host code only.
#pragma once

#include <cstddef>
#include <mutex>

#include <cuda_runtime_api.h>

namespace kss_rt {

// The first kMailBytes take the lattice's status block, the rest small arrays on their way
// from or to pageable memory.  A call that needs it takes a lease from a pool, shared by all
// threads and lattices, of at most kLeases buffers, made as they are first needed and kept.
// `p` is nullptr if all are borrowed or page-locked memory could not be had: the call then
// copies through the driver as for large arrays.  (Making and freeing a buffer in such a call
// would cost it more than the copies, and freeing one can wait for other streams' work.)
//
// Kernels of `stream` use the buffer until the call has waited for the stream (settled).  A
// call that returns before that, on an error, waits when the lease ends: the next borrower
// must not find a kernel still writing.  A buffer that cannot be waited for is not handed on.
struct HostLease {
  static constexpr size_t kMailBytes = 256, kBytes = size_t(1) << 20;
  static constexpr int kLeases = 8;
  unsigned char* p = nullptr;

  explicit HostLease(cudaStream_t stream, bool wanted = true) : stream_(stream) {
    if (!wanted) return;
    Pool& pool = the_pool();
    {
      std::lock_guard<std::mutex> lock(pool.mutex);
      if (pool.n > 0) {
        p = pool.kept[--pool.n];
        return;
      }
      if (pool.made == kLeases) return;
      ++pool.made;
    }
    // (another thread's stream capture is not disturbed by the allocation)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    void* q = nullptr;
    if (cudaHostAlloc(&q, kBytes, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
      cudaGetLastError();
      q = nullptr;
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    p = static_cast<unsigned char*>(q);
    if (!p) {
      std::lock_guard<std::mutex> lock(pool.mutex);
      --pool.made;
    }
  }
  ~HostLease() {
    if (!p) return;
    if (!settled_ && cudaStreamSynchronize(stream_) != cudaSuccess) return;
    Pool& pool = the_pool();
    std::lock_guard<std::mutex> lock(pool.mutex);
    pool.kept[pool.n++] = p;
  }
  HostLease(const HostLease&) = delete;
  HostLease& operator=(const HostLease&) = delete;

  // room for `bytes` of array data, or nullptr
  void* room(size_t bytes) const {
    return p && bytes <= kBytes - kMailBytes ? p + kMailBytes : nullptr;
  }
  // The call has waited for everything it queued on the stream.
  void settled() { settled_ = true; }

 private:
  struct Pool {
    std::mutex mutex;
    unsigned char* kept[kLeases] = {};
    int n = 0, made = 0;
  };
  static Pool& the_pool() {
    static Pool pool;
    return pool;
  }
  cudaStream_t stream_;
  bool settled_ = false;
};

}  // namespace kss_rt
