// Device memory of the library's contexts: stream-ordered allocations from a memory pool the
// library owns, one per device. A freed block stays in the pool for the next context instead of
// going back to the driver: cudaFree waits for the whole device and unmaps the pages, and a
// context of the Si512 workload holds about forty buffers (several GB), so creating and
// releasing contexts one after another (benchmarks, batches, warm-started sequences that
// rebuild their setup) would otherwise pay for that every time.
#include "omm_internal.cuh"

#include <cstdint>
#include <map>
#include <mutex>
#include <new>

namespace omm {
namespace mem {
namespace {

std::mutex g_mu;
std::map<int, cudaMemPool_t> g_pools;          // contexts: freed memory is kept for the next one
std::map<int, cudaMemPool_t> g_scratch_pools;  // scratch of single calls: at most kScratchKeep stays reserved
constexpr uint64_t kScratchKeep = 2ull << 30;

cudaMemPool_t pool_of_current_device(std::map<int, cudaMemPool_t>& pools, uint64_t keep) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    throw std::bad_alloc();
  }
  std::lock_guard<std::mutex> lock(g_mu);
  auto it = pools.find(dev);
  if (it != pools.end()) return it->second;
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
    cudaGetLastError();
    throw std::bad_alloc();
  }
  // what is reserved beyond `keep` goes back to the driver at a synchronisation after its release (trim_scratch
  // does not leave that to the caller, whose next one may be far away)
  cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
  pools[dev] = pool;
  return pool;
}

void* alloc_from(cudaMemPool_t pool, size_t bytes, cudaStream_t st) {
  void* p = nullptr;
  if (cudaMallocFromPoolAsync(&p, bytes ? bytes : 1, pool, st) != cudaSuccess) {
    cudaGetLastError();
    throw std::bad_alloc();
  }
  return p;
}

}  // namespace

void* alloc(size_t bytes, cudaStream_t st) {
  return alloc_from(pool_of_current_device(g_pools, UINT64_MAX), bytes, st);
}

void* alloc_scratch(size_t bytes, cudaStream_t st) {
  return alloc_from(pool_of_current_device(g_scratch_pools, kScratchKeep), bytes, st);
}

void release(void* p, cudaStream_t st) {
  if (p == nullptr) return;
  if (cudaFreeAsync(p, st) != cudaSuccess) cudaGetLastError();
}

void trim_scratch(cudaStream_t st) noexcept {
  cudaMemPool_t pool = nullptr;
  try {
    pool = pool_of_current_device(g_scratch_pools, kScratchKeep);
  } catch (const std::bad_alloc&) {
    return;
  }
  uint64_t reserved = 0;
  if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  if (reserved <= kScratchKeep) return;
  if (cudaStreamSynchronize(st) != cudaSuccess || cudaMemPoolTrimTo(pool, kScratchKeep) != cudaSuccess)
    cudaGetLastError();
}

void release_unused() {
  OMM_CUDA_TRY(cudaDeviceSynchronize());  // pending releases are complete
  OMM_CUDA_TRY(cudaMemPoolTrimTo(pool_of_current_device(g_pools, UINT64_MAX), 0));
  OMM_CUDA_TRY(cudaMemPoolTrimTo(pool_of_current_device(g_scratch_pools, kScratchKeep), 0));
}

}  // namespace mem
}  // namespace omm
