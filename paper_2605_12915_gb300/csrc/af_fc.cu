// af_fc.cu -- launch of the foot-centred point update (af_fc.cuh), in a
// translation unit of its own so that the library's units compile in parallel.
#include "af_fc.cuh"

namespace af {

cudaError_t launch_fc_points(const StepArgs<double>& a, cudaStream_t s) {
  const size_t n = (size_t)a.nx * a.ny;
  const size_t nv = (8 * n + FC_THREADS - 1) / FC_THREADS, ne = (4 * n + FC_THREADS - 1) / FC_THREADS;
  k_points_fc<<<(unsigned)(nv + 2 * ne), FC_THREADS, 0, s>>>(a, (int)nv, (int)ne);
  return cudaGetLastError();
}

}  // namespace af
