// launch_util.cuh -- host helpers shared by the kernel translation units.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace mhd {

// Raise the dynamic shared-memory limit of kernel `Fn` to `bytes`, once per device.
template <auto Fn>
cudaError_t ensure_smem(int bytes) {
  static std::atomic<unsigned long long> done{0};
  static std::atomic<int> done_bytes[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if ((done.load() & bit) && done_bytes[dev & 63].load() >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(Fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  done_bytes[dev & 63].store(bytes);
  done.fetch_or(bit);
  return cudaSuccess;
}

// Programmatic dependent launch.  A kernel launched by launch_after may start once the blocks of the
// kernel before it on the stream have finished, without waiting for that kernel's completion to reach
// the front end; every kernel so launched first calls after_previous(), which waits until the kernels
// before it have completed and their writes are visible.  Nothing before that call reads or writes
// memory, so the order of all memory operations is that of plain launches.  A chain of small kernels is
// bound by its launches: one 32^3 right-hand side without allocation 92 -> 69 us, one 64^3 right-hand
// side 176 -> 154, a 32^3 step of a captured run 43.9 -> 41.8.  (Letting the next kernel start early,
// griddepcontrol.launch_dependents, held SM resources idle: 512^3 double-float step 34.5 -> 37.3 ms,
// 32^3 step 48.9 us.)
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace mhd
