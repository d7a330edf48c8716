// af_tiles.cu -- the fused step on tiles smaller than 32 x 32 cells: the kernels of
// grids that give the chip fewer tiles than it has SMs, or whose last wave of
// 32 x 32 tiles would be nearly empty (STEP_GEOMS in af_launch.cuh).
#include "af_launch.cuh"

namespace af {

template <bool COMP>
cudaError_t launch_small_tiles(int geom, cudaStream_t s, const StepArgs<float>& a) {
  switch (geom) {
    case GEOM_8x4: return launch_step_tiles<8, 4, 256, 2, COMP>(s, a);
    case GEOM_8x8: return launch_step_tiles<8, 8, 512, 1, COMP>(s, a);
    case GEOM_16x8: return launch_step_tiles<16, 8, 512, 1, COMP>(s, a);
    case GEOM_16x16: return launch_step_tiles<16, 16, 512, 1, COMP>(s, a);
    case GEOM_32x16: return launch_step_tiles<32, 16, 512, 1, COMP>(s, a);
    case GEOM_32x24: return launch_step_tiles<32, 24, 512, 1, COMP>(s, a);
  }
  return cudaErrorNotSupported;
}

template <bool COMP>
cudaError_t launch_pipe_28(cudaStream_t s, const StepArgs<float>& a, int ctas,
                           const TileMaps* maps) {
  return launch_step_pipe<FUSED_TX, 28, FUSED_NT, AF_FUSED_MINB, COMP, false>(s, a, ctas, maps);
}

template cudaError_t launch_small_tiles<false>(int, cudaStream_t, const StepArgs<float>&);
template cudaError_t launch_small_tiles<true>(int, cudaStream_t, const StepArgs<float>&);
template cudaError_t launch_pipe_28<false>(cudaStream_t, const StepArgs<float>&, int,
                                           const TileMaps*);
template cudaError_t launch_pipe_28<true>(cudaStream_t, const StepArgs<float>&, int,
                                          const TileMaps*);

}  // namespace af
