// Instantiations of the z-marching 3D stage, FP32-mixed form.
#include "march3d.cuh"

namespace af {
cudaError_t launch_march3d_f32(int flux, const DevModel& m, const StageArgs3D<float>& a, cudaStream_t s) {
  return march3d_flux<float>(flux, m, a, s);
}
}  // namespace af
