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

// The same for kernels of one element or group per thread, which may be short or stream through memory for many waves of
// blocks: those are launched plainly.  bf16 -> e4m3 and the convolution that reads it, us, plain / dependent: 802 blocks
// of 256 threads 9.7 / 9.3, 3136 23.7 / 23.2, 3986 21.3 / 20.5; 11109 32.9 / 35.7, 27094 80.9 / 86.6.
constexpr unsigned long long kMostDependentBlocks = 4096;
template <class... Params, class... Args>
inline cudaError_t launch_short(void (*kernel)(Params...), dim3 grid, dim3 threads, cudaStream_t st, Args... args) {
  const bool early = (unsigned long long)grid.x * grid.y * grid.z <= kMostDependentBlocks;
  return launch_dependent_if(early, kernel, grid, threads, 0, st, args...);
}

}  // namespace ssconv
