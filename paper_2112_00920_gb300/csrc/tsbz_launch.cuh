// Launches of the kernels that a time step chains.  A step of few orbitals is six
// launches of 5 to 30 us, and with programmatic stream serialisation the next
// kernel is launched as the last CTAs of the one before it leave, instead of after
// its drain and flush.  step_enter() is the first statement of such a kernel: it waits
// until the kernel before it has completed and its writes are visible.
// Measured per step: 8 k-points at 16^3 92 -> 80 us (FP32) and 862 -> 847 us (FP64), 8^3 with
// 16 orbitals 162 -> 147 us, 10 x 12 x 14 161 -> 146 us.  Letting the next kernel be
// placed from the start of this one (griddepcontrol.launch_dependents) was slower
// than none of it (936 us, 171 us): its CTAs crowd the SMs that happen to be free.
#pragma once
#include <cuda_runtime.h>

__device__ __forceinline__ void step_enter() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// Dynamic shared memory above 48 KB, for a kernel whose need differs from cell to cell.
// The limit belongs to the kernel, not to a context or a thread, so every launch sets
// it to the same value, the most that a block can have: a limit set to what one cell needs
// was lowered by a context with a smaller cell between another thread's call and its
// launch, which was then refused.
template <auto kernel> inline void smem_limit(size_t bytes) {
  if (bytes <= 48 * 1024) return;
  static const int most = [] {
    cudaFuncAttributes a = {};
    cudaFuncGetAttributes(&a, kernel);
    return 227 * 1024 - (int)a.sharedSizeBytes;
  }();
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

template <typename... K, typename... A>
inline void step_launch(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, void* stream, A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)stream;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, (K)args...);
}
