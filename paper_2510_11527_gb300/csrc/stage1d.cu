// Instantiations of the fused 1D stage kernels (FP64 and FP32-mixed forms).
#include "launch.h"
#include "stage1d.cuh"

namespace af {

// Tile shape by mesh length: meshes with fewer 256-cell tiles than SMs are spread over
// the SMs in one-warp tiles (see Tile1D), the others keep the longer tile, whose halo
// costs 2 % of the work instead of 23 %.
constexpr int WARP_TILE_MAX_CELLS = 152 * 256;

template <int FLUX, class T, class PT>
static cudaError_t go1(const DevModel& m, const StageArgs2D<PT>& a, cudaStream_t s) {
  if (a.nx <= WARP_TILE_MAX_CELLS) {
    using L = Tile1DWarp;
    stage1d_warp_kernel<FLUX, T, PT><<<(a.nx + L::TX - 1) / L::TX, L::NT, 0, s>>>(m, a);
  } else {
    using L = Tile1DLong;
    stage1d_kernel<FLUX, T, PT><<<(a.nx + L::TX - 1) / L::TX, L::NT, 0, s>>>(m, a);
  }
  return cudaGetLastError();
}

// whole steps of a mesh of at most MARCH_MAX_CELLS cells: one cluster
template <int FLUX, class T, class PT>
static cudaError_t march1(const DevModel& m, const MarchArgs<PT>& M, cudaStream_t s) {
  const int tiles = (M.st[0].nx + Tile1DWarp::TX - 1) / Tile1DWarp::TX;
  const int warps = (tiles + MARCH_CTAS - 1) / MARCH_CTAS;
  if (warps > MARCH_WARPS) return cudaErrorInvalidValue;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = MARCH_CTAS;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(MARCH_CTAS);
  cfg.blockDim = dim3(32 * warps);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, march1d_kernel<FLUX, T, PT>, m, M);
}

template <class T, class PT>
static cudaError_t disp(int flux, const DevModel& m, const StageArgs2D<PT>& a, cudaStream_t s) {
  switch (flux) {
    case FLUX_ZERO: return go1<FLUX_ZERO, T, PT>(m, a, s);
    case FLUX_LINEAR: return go1<FLUX_LINEAR, T, PT>(m, a, s);
    case FLUX_BURGERS: return go1<FLUX_BURGERS, T, PT>(m, a, s);
    case FLUX_BL: return go1<FLUX_BL, T, PT>(m, a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <class T, class PT>
static cudaError_t disp_march(int flux, const DevModel& m, const MarchArgs<PT>& M, cudaStream_t s) {
  switch (flux) {
    case FLUX_ZERO: return march1<FLUX_ZERO, T, PT>(m, M, s);
    case FLUX_LINEAR: return march1<FLUX_LINEAR, T, PT>(m, M, s);
    case FLUX_BURGERS: return march1<FLUX_BURGERS, T, PT>(m, M, s);
    case FLUX_BL: return march1<FLUX_BL, T, PT>(m, M, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_stage1d_f64(int flux, const DevModel& m, const StageArgs2D<double>& a, cudaStream_t s) {
  return disp<double, double>(flux, m, a, s);
}
cudaError_t launch_stage1d_f32(int flux, const DevModel& m, const StageArgs2D<float>& a, cudaStream_t s) {
  return disp<float, float>(flux, m, a, s);
}
cudaError_t launch_march1d_f64(int flux, const DevModel& m, const MarchArgs<double>& M, cudaStream_t s) {
  return disp_march<double, double>(flux, m, M, s);
}
cudaError_t launch_march1d_f32(int flux, const DevModel& m, const MarchArgs<float>& M, cudaStream_t s) {
  return disp_march<float, float>(flux, m, M, s);
}

}  // namespace af
