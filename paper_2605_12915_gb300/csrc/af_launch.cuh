// af_launch.cuh -- host side of the fused step: launch configuration, the
// pipelined kernel's eligibility and tensor maps, and the batched launch.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "af_fused.cuh"
#include "af_ref_launch.cuh"

namespace af {

// Raises kernel KERN's dynamic shared-memory limit to `bytes` on the current
// device (the attribute belongs to the device: it is set once per device).
template <auto KERN>
inline cudaError_t allow_smem(size_t bytes) {
  constexpr int MAX_DEVICES = 64;
  static bool done[MAX_DEVICES] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < MAX_DEVICES && done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && dev >= 0 && dev < MAX_DEVICES) done[dev] = true;
  return e;
}

// The pipelined kernel's conditions on the grid (tiles of FUSED_TX x ty cells) and
// the input planes.
inline bool pipe_eligible(const StepArgs<float>& a, int ty = FUSED_TY) {
  if ((a.nx & 3) != 0 || a.nx < FUSED_TX + 8 || a.ny < ty + 6) return false;
  uintptr_t bits = 0;
  for (int q = 0; q < 4; ++q) bits |= (uintptr_t)a.in.avg[q] | (uintptr_t)a.in.lo[q];
  for (int f = 0; f < 3; ++f)
    for (int k = 0; k < 4; ++k) bits |= (uintptr_t)a.in.pt[f][k];
  return (bits & 15) == 0;
}

// Encodes the tensor maps of the 20 input planes in `a` (row-major nx x ny
// floats, staging box of tiles of FUSED_TX x ty cells); false if the driver lacks
// the encoder or rejects a map.
inline bool encode_tile_maps(const StepArgs<float>& a, TileMaps* out, int ty = FUSED_TY) {
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                             const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                             const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static Encode enc = nullptr;
  if (!enc) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      cudaGetLastError();
      return false;
    }
    enc = (Encode)fn;
  }
  using G = FusedGeom<FUSED_TX, FUSED_TY>;
  const cuuint64_t dims[2] = {(cuuint64_t)a.nx, (cuuint64_t)a.ny};
  const cuuint64_t strides[1] = {(cuuint64_t)a.nx * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)G::SW, (cuuint32_t)(ty + 6)}, unit[2] = {1, 1};
  for (int p = 0; p < 20; ++p) {
    float* base = p < 12 ? a.in.pt[p >> 2][p & 3] : p < 16 ? a.in.avg[p - 12] : a.in.lo[p - 16];
    if (enc(&out->m[p], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, unit,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return false;
  }
  return true;
}

// Whether one CTA per tile of ty rows can be launched: the tile rows are a grid's y
// dimension, which ends at 65535.  (Only grids of 2 to 16 columns and more than a
// million rows would choose a tile that does not fit; they get a taller one.)
inline bool tile_rows_fit(int ny, int ty) { return (ny + (int64_t)ty - 1) / ty <= 65535; }

// One CTA per tile of TX x TY cells.
template <int TX, int TY, int NT, int MINB, bool COMP>
inline cudaError_t launch_step_tiles(cudaStream_t s, const StepArgs<float>& a) {
  using G = FusedGeom<TX, TY>;
  constexpr auto kern = k_fused_step<TX, TY, NT, MINB, COMP>;
  const cudaError_t e = allow_smem<kern>(G::SMEM);
  if (e != cudaSuccess) return e;
  return launch_dependent(kern, dim3((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY), NT, G::SMEM, s,
                          a);
}

// Persistent pipelined CTAs over the tiles of TX x TY cells (tensor-copy staging
// when `maps` is given).
template <int TX, int TY, int NT, int MINB, bool COMP, bool INTER>
inline cudaError_t launch_step_pipe(cudaStream_t s, const StepArgs<float>& a, int ctas,
                                    const TileMaps* maps) {
  using G = FusedGeom<TX, TY>;
  constexpr auto kern = k_fused_step_pipe<TX, TY, NT, MINB, COMP, INTER>;
  const cudaError_t e = allow_smem<kern>(G::SMEM_PIPE);
  if (e != cudaSuccess) return e;
  static TileMaps none;
  const int ntiles = ((a.nx + TX - 1) / TX) * ((a.ny + TY - 1) / TY);
  // (INTER: the first kernel of an adjoint step)
  return launch_kernel(!INTER, kern, dim3(ntiles < ctas ? ntiles : ctas), NT, G::SMEM_PIPE, s, a,
                       maps ? *maps : none, maps ? 1 : 0);
}

// Tile geometries of a lone grid's step.  Results do not depend on the choice
// (every value a tile recomputes for its halo rounds the same way).
//
// A step is a sequence of dependent phases, and its time is (waves of one tile per
// SM) x (time of one tile): a tile of 32 x 32 cells takes 28 us however few of
// them a grid has, so a grid too small to give every SM one of those runs faster
// on smaller tiles although they recompute more halo.  `us` is the measured time
// of one wave (FP32_COMP, GB300); the geometry with the smallest sum is taken.
// Measured per step, 32 x 32 tiles -> chosen: 32^2 27.4 -> 5.1 us (8 x 4), 64^2 30.8 -> 6.4
// (8 x 8), 128^2 30.8 -> 7.1 (16 x 8), 192^2 30.9 -> 10.9 (16 x 16), 256^2 30.9 -> 16.5
// (32 x 16), 333 x 250 30.8 -> 21.6 (32 x 24), 448^2 57.7 -> 42 (32 x 24), 512^2 57.7 ->
// 48 (persistent, 28 rows: two full waves).
struct StepGeometry {
  int tx, ty;
  int pipe;      // persistent CTAs with the next tile's input staged asynchronously
  float us;      // time of one wave
  float fill;    // once per step (pipelined: the first tile's input)
};
enum { GEOM_8x4, GEOM_8x8, GEOM_16x8, GEOM_16x16, GEOM_32x16, GEOM_32x24, GEOM_32x32,
       GEOM_PIPE_32x28, GEOM_PIPE_32x32, N_STEP_GEOMS };
constexpr StepGeometry STEP_GEOMS[N_STEP_GEOMS] = {
    {8, 4, 0, 5.7f, 0.f},   {8, 8, 0, 6.4f, 0.f},   {16, 8, 0, 7.2f, 0.f},
    {16, 16, 0, 10.9f, 0.f}, {32, 16, 0, 16.5f, 0.f}, {32, 24, 0, 21.5f, 0.f},
    {FUSED_TX, FUSED_TY, 0, 28.2f, 0.f},
    {FUSED_TX, 28, 1, 22.f, 4.f}, {FUSED_TX, FUSED_TY, 1, 25.1f, 4.f}};

inline int choose_step_geometry(const StepArgs<float>& a, int sms) {
  int best = GEOM_32x32;
  float best_us = 1e30f;
  for (int g = 0; g < N_STEP_GEOMS; ++g) {
    const StepGeometry& q = STEP_GEOMS[g];
    if (q.pipe ? !pipe_eligible(a, q.ty) : !tile_rows_fit(a.ny, q.ty)) continue;
    const int64_t tiles = (int64_t)((a.nx + q.tx - 1) / q.tx) * ((a.ny + q.ty - 1) / q.ty);
    const float us = (float)((tiles + sms - 1) / sms) * q.us + q.fill;
    if (us < best_us) {
      best_us = us;
      best = g;
    }
  }
  // One CTA per 32 x 32 tile is for grids the persistent kernel does not take: where both
  // can run, one wave takes 27.9 us persistent and 29.0 so (384 x 384; 320 x 432 the same).
  if (best == GEOM_32x32 && pipe_eligible(a)) best = GEOM_PIPE_32x32;
  return best;
}

// The steps of the geometries smaller than 32 x 32 (af_tiles.cu).
template <bool COMP>
cudaError_t launch_small_tiles(int geom, cudaStream_t s, const StepArgs<float>& a);
template <bool COMP>
cudaError_t launch_pipe_28(cudaStream_t s, const StepArgs<float>& a, int ctas,
                           const TileMaps* maps);

// One step of the grid described by `a` with 32 x 32 tiles: the persistent
// pipelined kernel on `ctas` CTAs when `pipe` is set and the grid allows it
// (tensor-copy staging when `maps` is given), else one CTA per tile.  INTER
// (pipelined kernel only) also stores the intermediates the adjoint needs.
template <bool COMP, bool INTER = false>
inline cudaError_t launch_fused_step(cudaStream_t s, const StepArgs<float>& a, bool pipe,
                                     int ctas, const TileMaps* maps) {
  if (pipe && ctas > 0 && pipe_eligible(a))
    return launch_step_pipe<FUSED_TX, FUSED_TY, FUSED_NT, AF_FUSED_MINB, COMP, INTER>(s, a, ctas,
                                                                                      maps);
  if (INTER) return cudaErrorNotSupported;
  return launch_step_tiles<FUSED_TX, FUSED_TY, FUSED_NT, AF_FUSED_MINB, COMP>(s, a);
}

// Tile geometries available to the batched launch (the autotuner picks one): one
// CTA per tile of 32x32, 32x16 (or 24x16, two per SM) or 16x16 cells, or (pipe)
// persistent CTAs stepping through the 32x32 tiles with the next tile staged
// asynchronously.
struct BatchGeometry {
  int tx, ty, nt, minb, pipe;
};
constexpr int N_BATCH_GEOMS = 4, BATCH_24x16 = N_BATCH_GEOMS;
constexpr BatchGeometry BATCH_GEOMS[N_BATCH_GEOMS + 1] = {
    {32, 32, 512, 1, 0}, {32, 16, 512, 1, 0}, {16, 16, 512, 1, 0},
    {FUSED_TX, FUSED_TY, FUSED_NT, AF_FUSED_MINB, 1}, {24, 16, 256, 2, 0}};

// Whether geometry 1 stands for 24x16 tiles (two CTAs per SM) instead of 32x16 ones,
// given the ensemble's tile counts in both: the smaller of waves x measured time of
// a wave (26 and 17 us).  Eight grids of 64^2 and 128^2 (240 and 160 tiles) take
// 26.6 and 33.1 us a step, eight of 64^2 to 256^2 (624 and 448 tiles) 62.8 and 49.5.
inline bool batch_prefers_24x16(int64_t n24, int64_t n32, int sms) {
  return (float)((n24 + 2 * sms - 1) / (2 * sms)) * 26.f < (float)((n32 + sms - 1) / sms) * 17.f;
}

template <int TX, int TY, int NT, int MINB, bool COMP>
inline cudaError_t launch_batch_geom(bool dependent, cudaStream_t s, const StepArgs<float>* args,
                                     const int4* tiles, int ntiles) {
  using G = FusedGeom<TX, TY>;
  constexpr auto kern = k_fused_step_batch<TX, TY, NT, MINB, COMP>;
  const cudaError_t e = allow_smem<kern>(G::SMEM);
  if (e != cudaSuccess) return e;
  return launch_kernel(dependent, kern, dim3(ntiles), NT, G::SMEM, s, args, tiles);
}

// The persistent form: `ctas` CTAs over the tile table; maps (device, one
// TileMaps per grid) or null for cp.async staging only.
template <bool COMP>
inline cudaError_t launch_batch_pipe(bool dependent, cudaStream_t s, const StepArgs<float>* args,
                                     const int4* tiles, int ntiles, const TileMaps* maps,
                                     int ctas) {
  using G = FusedGeom<FUSED_TX, FUSED_TY>;
  constexpr auto kern = k_fused_step_batch_pipe<FUSED_TX, FUSED_TY, FUSED_NT, AF_FUSED_MINB, COMP>;
  const cudaError_t e = allow_smem<kern>(G::SMEM_PIPE);
  if (e != cudaSuccess) return e;
  return launch_kernel(dependent, kern, dim3(ntiles < ctas ? ntiles : ctas), FUSED_NT,
                       G::SMEM_PIPE, s, args, tiles, ntiles, maps);
}

// `dependent`: the kernel before on the stream is a step of the same batch
template <bool COMP>
inline cudaError_t launch_batch(int geom, bool dependent, cudaStream_t s,
                                const StepArgs<float>* args, const int4* tiles, int ntiles,
                                const TileMaps* maps, int ctas) {
  const bool d = dependent;
  switch (geom) {
    case 0: return launch_batch_geom<32, 32, 512, 1, COMP>(d, s, args, tiles, ntiles);
    case 1: return launch_batch_geom<32, 16, 512, 1, COMP>(d, s, args, tiles, ntiles);
    case 2: return launch_batch_geom<16, 16, 512, 1, COMP>(d, s, args, tiles, ntiles);
    case BATCH_24x16: return launch_batch_geom<24, 16, 256, 2, COMP>(d, s, args, tiles, ntiles);
    default: return launch_batch_pipe<COMP>(d, s, args, tiles, ntiles, maps, ctas);
  }
}

}  // namespace af
