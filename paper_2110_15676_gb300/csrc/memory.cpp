// Device and pinned host memory of the library.
//
// cudaFree and cudaFreeHost wait for everything that runs on the device.  A request server
// that released one finished problem so waited for the whole stationary solves of the others
// (one graph launch of tens of milliseconds each), with the driver's lock held: four solves
// on four streams ran one after another.  Device memory therefore comes from a stream-ordered
// pool per device, pinned memory from a list of small blocks.
//
// Safety.  An allocation is made on the calling thread's own stream, which is synchronised
// before the memory is handed out, so any stream may use it; a
// caller frees memory only when the work that uses it has finished (it has synchronised the
// streams that it was used on).  The runtime orders a reuse on another thread's stream after the
// free.
// Bounds.  The pool keeps at most kKeepBytes of free memory while problems, batches or servers live (a
// burst of eight served requests of 17 to 33 nodes a side holds 0.75 GB) and none once none does;
// afc_trim_memory gives it back at any time.  The pinned lists keep at most kKeepBlocks blocks each.
#include <cstdint>
#include <mutex>
#include <vector>

#include "afc_internal.h"

namespace afc {

namespace {

constexpr int kMaxDevices = 64;
constexpr uint64_t kKeepBytes = (uint64_t)2 << 30;
constexpr size_t kBlockBytes[2] = {4096, 65536};   // scalars of a problem; tables of a batch
constexpr size_t kKeepBlocks[2] = {256, 32};

std::mutex g_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};
int64_t g_live[kMaxDevices] = {};        // allocations not freed, and holders
std::vector<void*> g_blocks[2];          // free pinned blocks

cudaError_t pool_of(int device, cudaMemPool_t* out) {   // with g_mu held
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!g_pool[device]) {
    cudaMemPoolProps pr = {};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = device;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = cudaMemPoolCreate(&pool, &pr);
    if (e != cudaSuccess) return e;
    uint64_t keep = kKeepBytes;
    if ((e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
      cudaMemPoolDestroy(pool);
      return e;
    }
    g_pool[device] = pool;
  }
  *out = g_pool[device];
  return cudaSuccess;
}

}  // namespace

cudaError_t device_alloc(void** ptr, size_t bytes, bool zero) {
  *ptr = nullptr;
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if ((e = pool_of(device, &pool)) != cudaSuccess) return e;
    ++g_live[device];   // before the allocation: an idle trim does not run beside it
  }
  e = cudaMallocFromPoolAsync(ptr, bytes, pool, cudaStreamPerThread);
  if (e == cudaErrorMemoryAllocation) {   // once more without what the pool keeps in free pieces
    cudaGetLastError();
    *ptr = nullptr;
    cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(ptr, bytes, pool, cudaStreamPerThread);
  }
  if (e == cudaSuccess && zero) e = cudaMemsetAsync(*ptr, 0, bytes, cudaStreamPerThread);
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamPerThread);
  if (e != cudaSuccess) {
    if (*ptr) cudaFreeAsync(*ptr, cudaStreamPerThread);
    *ptr = nullptr;
    std::lock_guard<std::mutex> lk(g_mu);
    --g_live[device];
  }
  return e;
}

namespace {

// One allocation or holder less on `device`, which is current; the last one trims the pool.
void drop(int device) {
  bool idle = false;
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (device >= 0 && device < kMaxDevices) {
      idle = --g_live[device] == 0;
      pool = g_pool[device];
    }
  }
  if (idle && pool) {
    cudaStreamSynchronize(cudaStreamPerThread);
    cudaMemPoolTrimTo(pool, 0);
  }
}

}  // namespace

void device_free(void* ptr) {
  if (!ptr) return;
  cudaPointerAttributes at = {};
  int device = 0, now = 0;
  if (cudaPointerGetAttributes(&at, ptr) == cudaSuccess) device = at.device;
  else cudaGetDevice(&device);
  cudaGetDevice(&now);
  if (now != device) cudaSetDevice(device);
  cudaFreeAsync(ptr, cudaStreamPerThread);
  drop(device);
  if (now != device) cudaSetDevice(now);
}

void device_hold(int device, bool on) {
  if (device < 0 || device >= kMaxDevices) return;
  if (on) {
    std::lock_guard<std::mutex> lk(g_mu);
    ++g_live[device];
    return;
  }
  int now = 0;
  cudaGetDevice(&now);
  if (now != device) cudaSetDevice(device);
  drop(device);
  if (now != device) cudaSetDevice(now);
}

cudaError_t device_trim(int device) {
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
    pool = g_pool[device];
  }
  if (!pool) return cudaSuccess;   // nothing was allocated there yet
  // what other threads freed is free once their frees have run: wait for this thread's alone
  const cudaError_t e = cudaStreamSynchronize(cudaStreamPerThread);
  return e != cudaSuccess ? e : cudaMemPoolTrimTo(pool, 0);
}

// Pinned host memory in blocks of two sizes from the lists (larger: from the runtime).
cudaError_t pinned_alloc(void** ptr, size_t bytes) {
  *ptr = nullptr;
  const int c = bytes <= kBlockBytes[0] ? 0 : 1;
  if (bytes > kBlockBytes[1]) return cudaHostAlloc(ptr, bytes, cudaHostAllocPortable);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_blocks[c].empty()) {
      *ptr = g_blocks[c].back();
      g_blocks[c].pop_back();
      return cudaSuccess;
    }
  }
  return cudaHostAlloc(ptr, kBlockBytes[c], cudaHostAllocPortable);
}

void pinned_free(void* ptr, size_t bytes) {
  if (!ptr) return;
  if (bytes <= kBlockBytes[1]) {
    const int c = bytes <= kBlockBytes[0] ? 0 : 1;
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_blocks[c].size() < kKeepBlocks[c]) {
      g_blocks[c].push_back(ptr);
      return;
    }
  }
  cudaFreeHost(ptr);
}

}  // namespace afc
