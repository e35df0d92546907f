// Internal launch helpers shared by the translation units of libaf (not installed).
#pragma once
#include <cuda_runtime.h>

#include "reduce.cuh"
#include "stage2d.cuh"
#include "stage3d.cuh"

namespace af {

cudaError_t launch_stage2d_f64(int flux, bool blend, const DevModel& m, const StageArgs2D<double>& a,
                               cudaStream_t s);
cudaError_t launch_stage2d_f32(int flux, bool blend, const DevModel& m, const StageArgs2D<float>& a,
                               cudaStream_t s);
// Whole steps of a short 1D mesh in one launch of one cluster (march1d_kernel).
constexpr int WARP_TILE_1D = 26;   // cells of a one-warp 1D tile
constexpr int MARCH_CTAS = 8;    // portable cluster size
constexpr int MARCH_WARPS = 4;   // most warps per CTA: 8 x 4 x 26 = 832 cells
constexpr int MARCH_MAX_CELLS = MARCH_CTAS * MARCH_WARPS * WARP_TILE_1D;

template <class PT>
struct MarchArgs {
  int nstages;
  int nsteps;          // at most this many steps
  double dt_fixed;     // > 0: the step; else the CFL step of fin
  StageArgs2D<PT> st[5];
  DtFinal fin;
};

// bk: 0 no blend, 1 smoothness blend with the plain indicator, 2 with the external one
cudaError_t launch_stream2d_f32(int flux, int bk, const DevModel& m, const StageArgs2D<float>& a, cudaStream_t s);
cudaError_t launch_stream2d_blend_f32(int flux, int bk, const DevModel& m, const StageArgs2D<float>& a,
                                      cudaStream_t s);
cudaError_t launch_stage2d_rect_f64(int flux, bool blend, const DevModel& m, const StageArgs2D<double>& a,
                                    cudaStream_t s);
cudaError_t launch_stage2d_rect_f32(int flux, bool blend, const DevModel& m, const StageArgs2D<float>& a,
                                    cudaStream_t s);
cudaError_t launch_stage3d_f64(int flux, const DevModel& m, const StageArgs3D<double>& a, cudaStream_t s);
cudaError_t launch_stage3d_f32(int flux, const DevModel& m, const StageArgs3D<float>& a, cudaStream_t s);
// the marching 3D stage (march3d.cuh; FP64: the zero flux)
cudaError_t launch_march3d_f64(const DevModel& m, const StageArgs3D<double>& a, cudaStream_t s);
cudaError_t launch_march3d_f32(int flux, const DevModel& m, const StageArgs3D<float>& a, cudaStream_t s);
cudaError_t launch_rate3d(int flux, const DevModel& m, const int* n, const double* ub, const double* inv_h, double kmax,
                          unsigned long long* rate_bits, const DtFinal& fin, int blocks, cudaStream_t s);
cudaError_t launch_stage1d_f64(int flux, const DevModel& m, const StageArgs2D<double>& a, cudaStream_t s);
cudaError_t launch_stage1d_f32(int flux, const DevModel& m, const StageArgs2D<float>& a, cudaStream_t s);
cudaError_t launch_march1d_f64(int flux, const DevModel& m, const MarchArgs<double>& M, cudaStream_t s);
cudaError_t launch_march1d_f32(int flux, const DevModel& m, const MarchArgs<float>& M, cudaStream_t s);

}  // namespace af
