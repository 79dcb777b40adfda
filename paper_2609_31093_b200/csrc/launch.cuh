// Kernel launches of the latency-bound paths: programmatic dependent launch.
//
// Between two dependent kernels of a stream the GPU idles for 2 to 3 us (drain, launch, ramp up), a third of a short
// forward's time.  launch_dependent() marks a kernel as a programmatic dependent of whatever is before it in the stream: it
// may be placed on the SMs while that kernel drains.  A kernel launched this way calls grid_dependency() before it touches
// memory: it waits until the kernels before it have completed (and, because every one of them did the same, everything
// before those), then lets its own dependent be placed.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

#include "pisa_common.cuh"

namespace pisa {

__device__ __forceinline__ void grid_dependency() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Raises the kernel's dynamic shared memory limit to `smem` where it is lower (asked of the driver once per device and
// size; never lowered, so that threads using the kernel with different sizes do not undo one another's).
template <auto Kern>
cudaError_t allow_smem(size_t smem) {
  constexpr int kMaxDev = 64;
  static std::atomic<size_t> allowed[kMaxDev] = {};
  static std::mutex m;
  if (smem == 0) return cudaSuccess;        // (static and dynamic together may exceed the default 48 KB at any dynamic size)
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDev) return cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (smem <= allowed[dev].load(std::memory_order_acquire)) return cudaSuccess;
  std::lock_guard<std::mutex> lock(m);
  if (smem <= allowed[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) allowed[dev].store(smem, std::memory_order_release);
  return e;
}

template <auto Kern, typename... Args>
int launch_dependent(const char* what, dim3 grid, unsigned threads, size_t smem, cudaStream_t s, const Args&... args) {
  cudaError_t e = allow_smem<Kern>(smem);
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, Kern, args...);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    record_cuda_error(what, e);
    return PISA_ERR_CUDA;
  }
  return check_launch(what);
}

}  // namespace pisa
