// The column-marching 2D stage kernel with the smoothness blend (FP32-mixed form,
// periodic meshes; compiled with -fmad=false like stream2d_f32.cu, for the same
// reason), and the pass that forms the plain indicator for it.
#include <algorithm>

#include "launch.h"
#include "stream2d.cuh"

namespace af {

// The plain indicator (see blend_s_tile, same values) of one mesh, marching: a warp owns 28
// columns (lanes 2 .. 29; the others supply the halo) and S rows, averages of neighbouring
// columns come by shuffles and of the rows before from registers, so each average is
// converted and each s~ formed once (1.14 times) and no index is wrapped per value. What
// bounds it is instruction issue, then HBM (16 bytes per cell). In 32 x 8 tiles it took 188
// us at 4096^2; with the CFL rate's smaller cost the blended Buckley-Leverett step there
// went from 4.44 to 3.94 ms.
__global__ void __launch_bounds__(128) blend_s_march_kernel(const double* __restrict__ ub, int nx, int ny, double umid,
                                                            int S, int bands, float* __restrict__ s1,
                                                            float* __restrict__ s2) {
  const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int band = w % bands, rs = (w / bands) * S;
  if (rs >= ny) return;   // whole warp
  const int re = min(rs + S, ny);
  const int giu = band * STREAM_BAND - 2 + lane, gi = wrapi(giu, nx);
  const bool out = lane >= 2 && lane < 2 + STREAM_BAND && giu < nx;
  const float sixth = 1.0f / 6.0f;
  auto stl = [](float a, float b, float c) {
    return __fdividef(fabsf(a - 2.0f * b + c), fabsf(a) + 2.0f * fabsf(b) + fabsf(c) + 1e-13f);
  };
  int gj = wrapi(rs - 2, ny);
  auto row = [&](int j) { return to_stencil_nb<float>(__ldg(ub + (size_t)j * nx + gi), umid); };
  auto up = [&](int j) { return j + 1 == ny ? 0 : j + 1; };
  // rows r-1 and r-2 of the averages, s~_2 of rows r-2 and r-3
  float u2 = row(gj);
  gj = up(gj);
  float u1 = row(gj), t2 = 0.0f, t3 = 0.0f;
  gj = up(gj);
  float next = row(gj);
  for (int r = rs; r < re + 2; ++r) {
    const float u = next;
    gj = up(gj);
    if (r + 1 < re + 2) next = row(gj);
    const float t1 = stl(u2, u1, u);   // s~_2 of row r-1
    if (r < re) {
      const float x = stl(shup(u), u, shdn(u));
      const float v = (shup(x) + 4.0f * x + shdn(x)) * sixth;
      if (out) s1[(size_t)r * nx + giu] = v;
    }
    if (r - 2 >= rs && out) s2[(size_t)(r - 2) * nx + giu] = (t3 + 4.0f * t2 + t1) * sixth;
    t3 = t2;
    t2 = t1;
    u2 = u1;
    u1 = u;
  }
}

// the diffusion kind: compiled in for the cubic potential (Buckley-Leverett), else the
// model's runtime kind
template <int FLUX, int BK>
static cudaError_t stream2d_blend_dispatch(const DevModel& m, const StageArgs2D<float>& a, cudaStream_t s) {
  if (m.diff_kind == AF_DIFF_CUBIC) return stream2d_go<FLUX, DK_CUBIC, BK>(m, a, s);
  return stream2d_go<FLUX, DK_GENERIC, BK>(m, a, s);
}

template <int BK>
static cudaError_t stream2d_blend_flux(int flux, const DevModel& m, const StageArgs2D<float>& a, cudaStream_t s) {
  switch (flux) {
    case FLUX_ZERO: return stream2d_blend_dispatch<FLUX_ZERO, BK>(m, a, s);
    case FLUX_LINEAR: return stream2d_blend_dispatch<FLUX_LINEAR, BK>(m, a, s);
    case FLUX_BURGERS: return stream2d_blend_dispatch<FLUX_BURGERS, BK>(m, a, s);
    case FLUX_BL: return stream2d_blend_dispatch<FLUX_BL, BK>(m, a, s);
    default: return cudaErrorInvalidValue;
  }
}

// bk 1: the plain indicator, formed first into a.sb[0], a.sb[1] (two FP32 arrays of
// nx * ny); bk 2: the external indicator a.s_ext (one FP64 value per cell)
cudaError_t launch_stream2d_blend_f32(int flux, int bk, const DevModel& m, const StageArgs2D<float>& a,
                                      cudaStream_t s) {
  if (bk == 1) {
    if (!a.sb[0] || !a.sb[1]) return cudaErrorInvalidValue;
    // strips of 8 to 64 rows, about two waves of 64 warps per SM
    const int bands = (a.nx + STREAM_BAND - 1) / STREAM_BAND;
    const int S = (int)std::min(64LL, std::max(8LL, (long long)bands * a.ny / (152 * 128)));
    const long long blocks = ((long long)bands * ((a.ny + S - 1) / S) + 3) / 4;
    if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    blend_s_march_kernel<<<(unsigned)blocks, 128, 0, s>>>(a.ub, a.nx, a.ny, m.umid, S, bands,
                                                          const_cast<float*>(a.sb[0]), const_cast<float*>(a.sb[1]));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return stream2d_blend_flux<1>(flux, m, a, s);
  }
  if (bk == 2) {
    if (!a.s_ext) return cudaErrorInvalidValue;
    return stream2d_blend_flux<2>(flux, m, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace af
