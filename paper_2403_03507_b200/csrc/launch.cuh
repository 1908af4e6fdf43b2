// Kernel launches: clusters, programmatic dependent launch, shared-memory opt-in.
#pragma once

#include <atomic>
#include <utility>

#include "common.cuh"

namespace galore {

// Device side of programmatic dependent launch.  A kernel that was launched "early" may run beside the end of the kernel
// before it: nothing that kernel wrote may be read, and nothing it reads may be written, before the wait.  Every kernel
// of a step waits before it lets its own successor start, so whatever came before its predecessor is complete.
// Inputs of such a kernel are no `const T* __restrict__` parameters: the compiler would read them as memory that does not
// change while the kernel runs (ld.global.nc), and until the wait the kernel before it may still write them.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// more than 48 KiB of dynamic shared memory for a kernel, once per device; `done` belongs to that kernel
inline galore_status_t allow_smem(std::atomic<uint64_t>& done, const void* kern, int bytes) {
  int dev = 0;
  GALORE_CUDA_TRY(cudaGetDevice(&dev));
  const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return GALORE_OK;
  GALORE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done.fetch_or(bit, std::memory_order_release);
  return GALORE_OK;
}

// early: the kernel calls grid_dependency_wait() where it needs the kernel before it
template <class... KArgs, class... Args>
galore_status_t launch_kernel(void (*kern)(KArgs...), dim3 grid, int threads, size_t smem, int cluster, bool early, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (early) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  GALORE_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
  count_launch();
  return GALORE_OK;
}

}  // namespace galore
