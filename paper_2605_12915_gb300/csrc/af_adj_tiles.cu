// af_adj_tiles.cu -- the fused reverse sweep of the adjoint on one CTA per tile
// (ADJ_GEOMS in af_adjoint.cuh).
#include "af_adjoint.cuh"

namespace af {

template <bool COMP>
cudaError_t launch_adj_tiles_geom(int geom, cudaStream_t s, const StepArgs<float>& a,
                             const AdjView<float>& v) {
  switch (geom) {
    case ADJ_8x8: return launch_adj_tiles<8, 8, 256, 1, COMP>(s, a, v);
    case ADJ_16x8: return launch_adj_tiles<16, 8, 512, 1, COMP>(s, a, v);
    case ADJ_16x16: return launch_adj_tiles<16, 16, 512, 1, COMP>(s, a, v);
    case ADJ_32x8: return launch_adj_tiles<32, 8, 256, 2, COMP>(s, a, v);
    case ADJ_32x24: return launch_adj_tiles<32, 24, 512, 1, COMP>(s, a, v);
  }
  return cudaErrorNotSupported;
}

template cudaError_t launch_adj_tiles_geom<false>(int, cudaStream_t, const StepArgs<float>&,
                                             const AdjView<float>&);
template cudaError_t launch_adj_tiles_geom<true>(int, cudaStream_t, const StepArgs<float>&,
                                            const AdjView<float>&);

}  // namespace af
