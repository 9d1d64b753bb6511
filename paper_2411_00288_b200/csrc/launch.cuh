// Launching a kernel that may start while the one before it in the stream still runs.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace ssconv {

// SMs of the current device (148 where it cannot be asked: grids are sized by it, nothing else).
inline int device_sms() {
  static std::atomic<int> known[64];
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  sms = known[dev].load(std::memory_order_relaxed);
  if (sms == 0) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
    known[dev].store(sms, std::memory_order_relaxed);
  }
  return sms;
}

// Launch with programmatic stream serialisation, for kernels whose every thread calls grid_dependency_wait() before its
// first access to global memory (by plain loads: read-only ones could be moved above the wait, or find a line that was
// cached before it): the launch and the index arithmetic overlap the tail of the grid before.  Such a launch also takes the
// caller less time than a plain one (2.0 us against 2.5).
template <class... Params, class... Args>
inline cudaError_t launch_dependent_if(bool early, void (*kernel)(Params...), dim3 grid, dim3 threads, size_t smem,
                                       cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = threads;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <class... Params, class... Args>
inline cudaError_t launch_dependent_smem(void (*kernel)(Params...), dim3 grid, dim3 threads, size_t smem, cudaStream_t st,
                                         Args... args) {
  return launch_dependent_if(true, kernel, grid, threads, smem, st, args...);
}
template <class... Params, class... Args>
inline cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 threads, cudaStream_t st, Args... args) {
  return launch_dependent_smem(kernel, grid, threads, 0, st, args...);
}

// Kernels of one element or group per thread may be short, or stream through memory for many waves of blocks.  The short
// ones are launched early.  In the others each block would pay for the wait (a few hundred ns, also where nothing is waited
// for, which a wave of blocks with little to do cannot hide), and for plain loads instead of read-only ones: they have a form
// without either, and are launched plainly.  us, plain form / early form (with the wait, but launched plainly, in brackets):
//   choice from logits   1000 blocks of 256 threads 2.01 / 1.74, 2500 3.30 / 3.73, 4000 3.87 / 5.11, 9000 6.68 / (10.34)
//   by magnitude         1000 2.27 / 1.94, 3000 4.00 / 3.83, 4000 4.84 / 4.84, 9000 9.02 / (10.43)
//   bf16 -> e4m3         1000 2.57 / 2.25, 3000 4.02 / 3.80, 4000 4.91 / 5.01, 5000 5.86 / (6.46)
//   compress             300 3.17 / 2.77, 1000 5.01 / 4.24, 4000 19.4 / 17.5
//   AdamW                1000 4.11 / 3.88, 4000 10.6 / 10.1      soft mask 1000 4.08 / 3.79, 4000 10.1 / 9.7
//   mask gradient        1000 3.16 / 3.06, 4000 8.56 / 7.94
// bf16 -> e4m3 and the convolution that reads it, plain / early: 3136 blocks 30.7 / 29.1, 11109 32.9 / 35.7, 27094 80.9 / 86.6.
constexpr unsigned long long kEarlyBlocks = 4096, kEarlyBlocksLogits = 1184;
template <class... Params, class... Args>
inline cudaError_t launch_short(void (*early)(Params...), void (*plain)(Params...), unsigned long long most, dim3 grid,
                                dim3 threads, cudaStream_t st, Args... args) {
  const bool few = (unsigned long long)grid.x * grid.y * grid.z <= most;
  return launch_dependent_if(few, few ? early : plain, grid, threads, 0, st, args...);
}
// What the two forms of such a kernel differ in.
template <bool EARLY>
__device__ __forceinline__ void short_begin() {
  if (EARLY) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <bool EARLY>
__device__ __forceinline__ void short_wait() {
  if (EARLY) asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <bool EARLY, class T>
__device__ __forceinline__ T short_load(const T* p) {
  return EARLY ? *p : __ldg(p);
}

}  // namespace ssconv
