// Instantiations of the z-marching 3D stage, FP64 form (the zero flux).
#include "march3d.cuh"

namespace af {
cudaError_t launch_march3d_f64(const DevModel& m, const StageArgs3D<double>& a, cudaStream_t s) {
  return march3d_diff<FLUX_ZERO, double>(m, a, s);
}
}  // namespace af
