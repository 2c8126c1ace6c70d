// adi_chain.cuh -- consecutive kernels of a time loop that overlap their
// launches (programmatic dependent launch).
#pragma once

#include <cuda_runtime.h>

namespace adi {

// Programmatic dependent launch: a kernel launched with launch_chained() may
// start while the kernel before it is finishing; it touches nothing that
// kernel writes before chain_wait(), which returns once that kernel (and
// with it everything before it) has completed.
// chain_release() lets the next kernel's CTAs in as soon as every CTA of this
// one has called it; without it they come as this one's CTAs exit.  Only the
// one-pass steps release early: they have work to do before chain_wait().
// The sweeps, the reverse step and the models have next to none, and the
// waiting CTAs cost them shared memory that is L1 otherwise (us per step of
// the sweeps at tau = 2h, early release and none: 1024^2 17.4 and 14.3, 3001
// x 1501 72 and 64.0, 4096^2 151 and 136.5; graphs without overlap 15.4, 64.0
// and 136.8; a gradient at 1024^2, 100 steps, 4.83 and 4.27 ms).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch attribute of a kernel that may overlap the end of the one before it
// in the stream.  Every such kernel begins with chain_wait().
inline cudaLaunchAttribute chain_attribute(bool overlap = true) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  return at;
}

template <typename... P, typename... A>
cudaError_t launch_after(bool overlap, void (*kern)(P...), dim3 blocks, dim3 threads, size_t smem, cudaStream_t st,
                         const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = blocks;
  cfg.blockDim = threads;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1] = {chain_attribute(overlap)};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 blocks, dim3 threads, size_t smem, cudaStream_t st,
                           const A&... args) {
  return launch_after(true, kern, blocks, threads, smem, st, args...);
}

}  // namespace adi
