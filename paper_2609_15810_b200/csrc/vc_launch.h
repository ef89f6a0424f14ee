// Kernel launches that may overlap the end of the kernel in front of them (programmatic dependent
// launch), and shared-memory limits raised once per kernel and device.
//
// Every kernel launched this way calls pdl_wait() before it touches anything an earlier kernel on
// the stream wrote or still reads: the call returns when the kernel in front has completed and its writes
// are visible.  Because each of them waits, and allows its successor only behind its own wait, whatever
// happened before the kernel in front is complete as well; a caller's own kernels, which allow nothing,
// are simply waited for.  What is gained is the gap between two kernels (about 1.5 us) and the
// successor's prologue.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace vc {

template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Lets KERNEL use up to the whole SM's shared memory.  One driver call per kernel and device for the
// life of the process (it used to be one per kernel and call).
template <auto KERNEL>
inline cudaError_t allow_smem() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_allow() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

}  // namespace vc
