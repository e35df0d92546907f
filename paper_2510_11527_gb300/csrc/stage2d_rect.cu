// Instantiations of the fused 2D stage kernel on rectangles with outflow ends (padded
// layout, reflected ghost loads, masked stores), FP64 form.
#include "stage2d_launch.cuh"

namespace af {

cudaError_t launch_stage2d_rect_f64(int flux, bool blend, const DevModel& m, const StageArgs2D<double>& a,
                                    cudaStream_t s) {
  return stage2d_dispatch<double, true>(flux, blend, m, a, s);
}

}  // namespace af
