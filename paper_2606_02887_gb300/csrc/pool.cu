// What the library keeps per device and context: the shared-memory limits of its kernels (SmemLimit), and
// device memory for the workspaces of calls that have no handle: stream-ordered allocations from a
// pool of the library's own on each device, which keeps up to kPoolKeep bytes between calls (a
// cudaMalloc and cudaFree of the kNN workspace took about a third of the call).  snmf_destroy gives back
// what the pool holds unused.  The runtime orders reuse over streams and threads.
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>

#include "common.cuh"

namespace snmf {
namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kPoolKeep = 128ull << 20;

// A pool lives as long as its context (a device reset ends both): it is known by the context's id.
struct DevicePool {
  cudaMemPool_t pool = nullptr;
  unsigned long long ctx = 0;
};
DevicePool g_pool[kMaxDevices];
std::mutex g_pool_mu;

template <typename F>
F entry(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    p = nullptr;
  return reinterpret_cast<F>(p);
}

// the current device's pool; nullptr without one (`make`: created when missing)
cudaMemPool_t device_pool(bool make) {
  int dev = 0;
  unsigned long long id = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices || (make && cudaFree(nullptr) != cudaSuccess) ||
      !context_id(&id))
    return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  DevicePool& d = g_pool[dev];
  if (d.pool && d.ctx == id) return d.pool;
  if (!make) return nullptr;
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t p = nullptr;
  if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  unsigned long long keep = kPoolKeep;
  cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
  d.pool = p;
  d.ctx = id;
  return p;
}

}  // namespace

bool context_id(unsigned long long* id) {
  static auto get_ctx = entry<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
  static auto get_id = entry<CUresult (*)(CUcontext, unsigned long long*)>("cuCtxGetId");
  CUcontext ctx = nullptr;
  return get_ctx && get_id && get_ctx(&ctx) == CUDA_SUCCESS && ctx && get_id(ctx, id) == CUDA_SUCCESS && *id;
}

cudaError_t raise_smem_limit(SmemLimit& l, const void* kernel, size_t bytes) {
  int dev = 0;
  unsigned long long id = 0;
  const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices && context_id(&id);
  if (known && l.ctx[dev].load(std::memory_order_relaxed) == id) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && known) l.ctx[dev].store(id, std::memory_order_relaxed);
  return e;
}

cudaError_t workspace_alloc(void** p, size_t bytes, cudaStream_t s) {
  cudaMemPool_t pool = device_pool(true);
  return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}

void workspace_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

void workspace_trim() {
  if (cudaMemPool_t pool = device_pool(false)) cudaMemPoolTrimTo(pool, 0);
}

}  // namespace snmf
