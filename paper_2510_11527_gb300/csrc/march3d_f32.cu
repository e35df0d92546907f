// Instantiations of the z-marching 3D stage, FP32-mixed form.
#include "march3d.cuh"

namespace af {
cudaError_t launch_march3d_f32(int flux, const DevModel& m, const StageArgs3D<float>& a, cudaStream_t s) {
  switch (flux) {
    case FLUX_ZERO: return march3d_diff<FLUX_ZERO, float>(m, a, s);
    case FLUX_LINEAR: return march3d_diff<FLUX_LINEAR, float>(m, a, s);
    case FLUX_BURGERS: return march3d_diff<FLUX_BURGERS, float>(m, a, s);
    default: return cudaErrorInvalidValue;
  }
}
}  // namespace af
