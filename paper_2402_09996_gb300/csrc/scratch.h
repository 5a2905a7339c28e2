// Device scratch of one call (the point updates' rate tables, the labelling's generators),
// stream-ordered from a pool that each device keeps.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

namespace rve {

// Bytes the pool of a device keeps between calls; more is given back at the next
// synchronisation.
constexpr uint64_t kScratchKeep = 64u << 20;

// The current device's pool (created on first use, kept until the process exits), or null.
inline cudaMemPool_t scratch_pool() {
  static std::mutex mu;
  static cudaMemPool_t pools[64] = {};
  static bool tried[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!tried[dev]) {
    tried[dev] = true;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = kScratchKeep;
    if (cudaMemPoolCreate(&pool, &props) == cudaSuccess &&
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess)
      pools[dev] = pool;
    else
      cudaGetLastError();
  }
  return pools[dev];
}

// An allocation for work on one stream, given back when it goes out of scope.  cudaMalloc and
// the device-wide wait of cudaFree took 150 us a call, as much as the small calls themselves;
// the default pool would map its memory again after each synchronisation.  Where the pool has
// none (or the stream is being captured) the memory comes from cudaMalloc.
class CallScratch {
 public:
  void* p = nullptr;
  CallScratch() = default;
  CallScratch(const CallScratch&) = delete;
  CallScratch& operator=(const CallScratch&) = delete;
  cudaError_t alloc(size_t bytes, cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
      cudaMemPool_t pool = scratch_pool();
      if (pool && cudaMallocFromPoolAsync(&p, bytes, pool, st) == cudaSuccess) {
        st_ = st;
        pooled_ = true;
        return cudaSuccess;
      }
    }
    cudaGetLastError();
    p = nullptr;
    return cudaMalloc(&p, bytes);
  }
  ~CallScratch() {
    if (!p) return;
    if (pooled_) cudaFreeAsync(p, st_);
    else cudaFree(p);
  }

 private:
  cudaStream_t st_ = nullptr;
  bool pooled_ = false;
};

}  // namespace rve
