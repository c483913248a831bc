// Device memory of the library's own objects, and words of pinned host memory that kernels report through.
//
// Objects live in one stream-ordered pool per device: a cudaMalloc / cudaFree pair of a layer's arrays takes hundreds
// of microseconds (encoding a 4096 x 4096 layer spent 1.9 of 2.2 ms in them), an allocation that the pool can serve
// about one.  The pool keeps at most kPoolKeepBytes of unused memory; what is above goes back to the system at the
// next synchronisation, all of it when an allocation fails, and whatever the caller asks for through gwq_trim_memory
// (other allocators of the process cannot reach it).
#include <mutex>
#include <vector>

#include "common.cuh"

namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kPoolKeepBytes = 256ull << 20;   // about eight 7B-shaped layers

std::mutex g_mutex;
cudaMemPool_t g_pool[kMaxDevices] = {nullptr};

cudaError_t pool_of_current_device(cudaMemPool_t* pool) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    e = cudaMemPoolCreate(&p, &props);
    if (e != cudaSuccess) return e;
    unsigned long long keep = kPoolKeepBytes;
    e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      (void)cudaMemPoolDestroy(p);
      return e;
    }
    g_pool[dev] = p;
  }
  *pool = g_pool[dev];
  return cudaSuccess;
}

// Pinned words: pages cut into slots that calls borrow and return; a further page only when every slot is borrowed.
constexpr int kSlotsPerPage = 64;
std::vector<void*> g_free_slots;

}  // namespace

cudaError_t gwq_dev_alloc(void** p, size_t bytes, cudaStream_t stream) {
  *p = nullptr;
  cudaMemPool_t pool = nullptr;
  cudaError_t e = pool_of_current_device(&pool);
  if (e != cudaSuccess) return e;
  e = cudaMallocFromPoolAsync(p, bytes, pool, stream);
  if (e == cudaErrorMemoryAllocation) {   // give back what the pool keeps, then try once more
    (void)cudaGetLastError();
    (void)cudaDeviceSynchronize();
    (void)cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(p, bytes, pool, stream);
  }
  return e;
}

extern "C" gwq_status gwq_trim_memory(size_t keep_bytes) {
  int dev = -1;
  cudaMemPool_t pool = nullptr;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return GWQ_ERR_CUDA;
  }
  if (dev >= 0 && dev < kMaxDevices) {
    std::lock_guard<std::mutex> lock(g_mutex);
    pool = g_pool[dev];
  }
  if (!pool) return GWQ_OK;   // nothing has been allocated on this device
  // what was freed in stream order is unused once the frees have been reached
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemPoolTrimTo(pool, keep_bytes) != cudaSuccess) {
    (void)cudaGetLastError();
    return GWQ_ERR_CUDA;
  }
  return GWQ_OK;
}

void gwq_dev_free_async(void* p, cudaStream_t stream) {
  if (p && cudaFreeAsync(p, stream) != cudaSuccess) (void)cudaGetLastError();
}

// As cudaFree: waits for the work of every stream of the device that holds p, so that an object may be released while
// a product with it is still running.
void gwq_dev_free(void* p) {
  if (!p) return;
  cudaPointerAttributes at = {};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return;
  }
  const bool move = at.device != dev;
  if (move) (void)cudaSetDevice(at.device);
  (void)cudaDeviceSynchronize();
  gwq_dev_free_async(p, cudaStreamLegacy);
  if (move) (void)cudaSetDevice(dev);
}

void* gwq_pinned_slot() {
  std::lock_guard<std::mutex> lock(g_mutex);
  if (g_free_slots.empty()) {
    void* page = nullptr;
    if (cudaHostAlloc(&page, kSlotsPerPage * GWQ_PINNED_SLOT_BYTES, cudaHostAllocPortable) != cudaSuccess) {
      (void)cudaGetLastError();
      return nullptr;
    }
    for (int i = kSlotsPerPage - 1; i >= 0; --i)
      g_free_slots.push_back(static_cast<unsigned char*>(page) + (size_t)i * GWQ_PINNED_SLOT_BYTES);
  }
  void* slot = g_free_slots.back();
  g_free_slots.pop_back();
  return slot;
}

void gwq_pinned_slot_return(void* slot) {
  if (!slot) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  g_free_slots.push_back(slot);
}

namespace {
// Up to eight arrays copied by one launch; starts are multiples of 16 bytes, ends need not be.
struct CopyArgs {
  const char* from[8];
  char* to[8];
  size_t bytes[8];
};
__global__ void __launch_bounds__(256) copy_kernel(const CopyArgs a) {
  const size_t stride = (size_t)gridDim.x * blockDim.x, first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const char* from = a.from[blockIdx.y];
  char* to = a.to[blockIdx.y];
  const size_t bytes = a.bytes[blockIdx.y], wide = bytes / 16;
  for (size_t i = first; i < wide; i += stride) reinterpret_cast<uint4*>(to)[i] = __ldcs(reinterpret_cast<const uint4*>(from) + i);
  for (size_t i = wide * 16 + first; i < bytes; i += stride) to[i] = from[i];
}
}  // namespace

// One launch instead of a cudaMemcpyAsync per array (six of a layer, about 5 us of the host's time each).
cudaError_t gwq_copy_arrays(int count, const void* const* from, void* const* to, const size_t* bytes, cudaStream_t stream) {
  CopyArgs a = {};
  size_t most = 0;
  if (count < 1 || count > 8) return cudaErrorInvalidValue;
  for (int i = 0; i < count; ++i) {
    a.from[i] = static_cast<const char*>(from[i]);
    a.to[i] = static_cast<char*>(to[i]);
    a.bytes[i] = bytes[i];
    if (bytes[i] > most) most = bytes[i];
  }
  size_t ctas = (most / 16 + 255) / 256;
  ctas = ctas < 1 ? 1 : (ctas > 1184 ? 1184 : ctas);
  copy_kernel<<<dim3((unsigned)ctas, (unsigned)count), 256, 0, stream>>>(a);
  return cudaGetLastError();
}
