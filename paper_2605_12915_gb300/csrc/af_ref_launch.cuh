// af_ref_launch.cuh -- host side of the kernel-per-stage step (af_ref_kernels.cuh),
// and the launch helper shared with the fused step.
#pragma once

#include <cuda_runtime.h>

#include "af_ref_kernels.cuh"

namespace af {

// Launches `kern` so that it may be scheduled while the stream's previous kernel
// drains (programmatic dependent launch); the kernel itself waits for that
// kernel's results (pdl_wait) before it touches memory.  Saves the launch gap
// between steps: 8.35 -> 6.54 us per fused step at 64 x 64 cells, 18.6 -> 16.8 at
// 256^2.
// The attribute speaks of the kernel before, not of what else the stream may have been
// given in between (a wait for another stream's event, a copy), so it is used between
// kernels of this library only: a call's first kernel that reads or writes the caller's
// memory, and one that follows the library's own copies, is launched without it.
template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool dependent, void (*kern)(P...), dim3 grid, dim3 threads,
                                 size_t smem, cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = threads;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&c, kern, args...);
}
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, dim3 threads, size_t smem,
                                    cudaStream_t s, const A&... args) {
  return launch_kernel(true, kern, grid, threads, smem, s, args...);
}

template <typename T>
inline unsigned ref_blocks(const StepArgs<T>& a) {
  return (unsigned)(((size_t)a.nx * a.ny + REF_THREADS - 1) / REF_THREADS);
}

// centres and acoustic increments (`dependent`: of the first kernel)
template <typename T, bool COMP>
inline cudaError_t launch_ref_nodes(const StepArgs<T>& a, cudaStream_t s, bool dependent) {
  const unsigned b = ref_blocks(a);
  const cudaError_t e = launch_kernel(dependent, k_center<T, COMP>, dim3(b), REF_THREADS, 0, s,
                                      a, TopSpeed{});
  if (e != cudaSuccess) return e;
  return launch_dependent(k_acoustic<T>, dim3(b, 4), REF_THREADS, 0, s, a);
}

// the whole step
template <typename T, bool COMP>
inline cudaError_t launch_ref_step(const StepArgs<T>& a, cudaStream_t s, bool dependent = true) {
  const unsigned b = ref_blocks(a);
  cudaError_t e = launch_ref_nodes<T, COMP>(a, s, dependent);
  if (e != cudaSuccess) return e;
  e = launch_dependent(k_points<T, true>, dim3(b, 3), REF_THREADS, 0, s, a);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_average<T, COMP>, dim3(b), REF_THREADS, 0, s, a, node_flux_of(a));
}

// the intermediates that the adjoint linearises about: centres, increments,
// half-step points and the new points (of an adjoint step, which has just been given
// the caller's planes)
template <typename T, bool COMP>
inline cudaError_t launch_ref_intermediates(const StepArgs<T>& a, cudaStream_t s) {
  const cudaError_t e = launch_ref_nodes<T, COMP>(a, s, false);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_points<T, false>, dim3(ref_blocks(a), 3), REF_THREADS, 0, s, a);
}

}  // namespace af
