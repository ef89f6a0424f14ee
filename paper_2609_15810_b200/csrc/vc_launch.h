// Kernel launches that may overlap the end of the kernel in front of them (programmatic dependent
// launch), and shared-memory limits raised once per kernel and context.
//
// What makes it sound:
//   - Every kernel launched this way calls pdl_wait() in front of whatever the kernel before it on the stream may
//     write or still read: the call returns when that kernel has completed and its writes are visible.
//   - A kernel allows its successor (pdl_allow) only behind its own wait.  So when a kernel starts, everything
//     in front of the kernel before it is complete, and a caller's own kernels, which allow nothing, are
//     simply waited for.  (One exception: the assignment of vc_group allows early.  Its successor, the update,
//     waits before it does anything.)
//   - Therefore a kernel may read, in front of its wait, what the kernel before it neither writes nor makes
//     late: the preprocessing passes read Q, K, V and the permutation, the assignment of vc_group reads V.  The
//     kernels before them (table, permutation check, passes, finalize; init, update) write none of these.  (The one launch
//     of short heads stands behind a caller's kernels and reads nothing in front of its wait.)  Another
//     kernel put in between has to keep to that, and has to wait before it allows.
// What is gained is the gap between two kernels (about 1.5 us) and the successor's prologue.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace vc {

template <typename... P, typename... A>
inline cudaError_t launch_clusters(void (*kernel)(P...), dim3 grid, int cluster, int threads, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
  return launch_clusters(kernel, grid, 1, threads, smem, s, args...);
}

// A number for the current context that no other context of the process gets, 0 if there is none yet.
inline uint64_t context_number() {
  typedef CUresult (*GetId)(CUcontext, unsigned long long*);
  static const GetId get = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult found;
    const bool ok = cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &found) == cudaSuccess && found == cudaDriverEntryPointSuccess;
    return ok ? reinterpret_cast<GetId>(p) : nullptr;
  }();
  unsigned long long id = 0;
  return get && get(nullptr, &id) == CUDA_SUCCESS ? id + 1 : 0;
}

// Lets KERNEL use up to the whole SM's shared memory.  The limit belongs to the context (a second context of
// the device, or the one behind cudaDeviceReset, starts without it): one driver call per kernel and context,
// and one more whenever more than 64 contexts share a slot.
template <auto KERNEL>
inline cudaError_t allow_smem() {
  static std::atomic<uint64_t> done[64];
  const uint64_t ctx = context_number();
  std::atomic<uint64_t>& slot = done[ctx % 64];
  if (ctx && slot.load(std::memory_order_acquire) == ctx) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess) slot.store(ctx, std::memory_order_release);
  return e;
}

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_allow() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

}  // namespace vc
