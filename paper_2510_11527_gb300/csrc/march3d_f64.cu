// Instantiations of the z-marching 3D stage, FP64 form.
#include "march3d.cuh"

namespace af {
cudaError_t launch_march3d_f64(int flux, const DevModel& m, const StageArgs3D<double>& a, cudaStream_t s) {
  return march3d_flux<double>(flux, m, a, s);
}
}  // namespace af
