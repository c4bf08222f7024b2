// Host launch helpers: per-device caches of kernel properties, and launches
// that may overlap the tail of the kernel before them.
#pragma once

#include <atomic>
#include <cuda_runtime.h>

namespace bsrht {

// Value of f() for the current device, computed once per device and slot
// array (values >= 0; a failed f(), negative, is not kept).  Every writer
// stores the same value, so host threads may race.
struct DeviceCache {
  std::atomic<int> v[64];
  template <typename F>
  int get(F&& f) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return f();
    const int c = v[dev].load(std::memory_order_relaxed);
    if (c > 0) return c - 1;
    const int x = f();
    if (x >= 0) v[dev].store(x + 1, std::memory_order_relaxed);
    return x;
  }
};

// Launches kern on s.  overlap: programmatic dependent launch -- the grid may
// start once every CTA of the kernel before it on s has called
// launch_dependents() or ended; it must call wait_for_prior_grid() before it
// touches anything that kernel writes or reads.
template <typename... K, typename... A>
cudaError_t launch_kernel(bool overlap, void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<K>(args)...);
}

__device__ __forceinline__ void wait_for_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Whether launches on s may overlap: not while s is being captured (the
// captured graphs are updated in place for new pointers).
inline bool may_overlap(cudaStream_t s) {
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(s, &c) == cudaSuccess && c == cudaStreamCaptureStatusNone;
}

}  // namespace bsrht
