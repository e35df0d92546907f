// Launchers of the fused 2D stage kernels (internal). The FP32-mixed form of a periodic
// mesh runs the column-marching kernel (stream2d.cuh), with or without the blend. The
// others run one CTA per 32 x 8 tile of the mesh, or of the padded layout of a
// rectangle with ends (RECT): the FP64 form and the blended FP32 rectangle
// stage2d_kernel, the FP32 rectangle without the blend the compilation for 48 warps per
// SM. The translation units instantiate the periodic (RECT = false) and the rectangle
// (RECT = true) launchers separately, so they compile in parallel and the periodic
// kernels are unaffected by the rectangle's code.
#pragma once
#include <type_traits>

#include "launch.h"

namespace af {

template <int FLUX, class T, bool BLEND, bool RECT, int TX, int TY, int NT>
static auto stage2d_kernel_for() {
  if constexpr (std::is_same_v<T, float> && !BLEND && TX == 32) return stage2d_kernel_f32occ<FLUX, RECT, TY>;
  else return stage2d_kernel<FLUX, T, T, BLEND, RECT, TX, TY, NT>;
}

// Work of a mesh's busiest SM with TX x TY tiles of halo H, in warps of box positions:
// tiles dealt to 152 SMs, each worth its box (what the FP64 unit of an SM spends on a
// tile; on a short mesh also the length of a CTA's phases).
inline long long tile_cost(int nx, int ny, int TX, int TY, int H) {
  const long long tiles = (long long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY);
  return (tiles + 151) / 152 * (((TX + 2 * H) * (TY + 2 * H) + 31) / 32);
}

template <int FLUX, class T, bool BLEND, bool RECT, int TX, int TY, int NT = TX * TY>
static cudaError_t stage2d_tiles(const DevModel& m, const StageArgs2D<T>& a, cudaStream_t s) {
  using L = Tile2D<FLUX, T, BLEND, TX, TY, NT>;
  static bool attr = false;
  auto k = stage2d_kernel_for<FLUX, T, BLEND, RECT, TX, TY, NT>();
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const long long tiles = (long long)((a.nx + TX - 1) / TX) * ((a.ny + TY - 1) / TY);
  if (tiles > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
  k<<<(unsigned)tiles, L::NT, L::SMEM, s>>>(m, a);
  return cudaGetLastError();
}

// Tile shape by mesh: 32 x 8 on large meshes (its halo box is 1.7 times the tile), 12 x 8
// (2 times) where the larger one leaves SMs without work, with two threads per cell so
// that a phase over the box is one pass: a stage of a short mesh lasts as long as one
// CTA's chain of phases. Porous medium FP64, one stage at 32 x 8 / 12 x 8 with 96 threads
// / with 192: 40^2 26.8 / 20.6 / 16.5 us, 100^2 31.8 / 25.6 / 20.5 us, 200^2 40.3 / 30.8 /
// 28.2 us, 300^2 53.4 / 53.9 / 59.5 us, 600^2 155 / 167 / 186 us (8 x 8 and 8 x 4 tiles
// were no faster on the short ones). The smaller tile's phases are less evenly filled, so
// it has to be worth a sixth less (200 x 215 FP64, Burgers, 24 against 28: 57 / 56 us).
//
// The FP32 rectangle without the blend is bound by instruction issue, so on larger meshes
// the box's share counts: 32 x 12 tiles (1.5 times the tile) with 384 threads, where they
// are worth a tenth less. Example 6.9, one step at 32 x 8 / 32 x 12: 385 x 301 57.6 / 63.7
// us, 512^2 94.4 / 94.3, 768^2 151.9 / 149.7, 1536^2 518 / 495, 2048^2 898 / 849 us (one
// stage there: 32 x 8 294, 32 x 12 279, 32 x 16 287, 16 x 16 304, 64 x 8 297, 32 x 24 304).
template <int FLUX, class T, bool BLEND, bool RECT>
static cudaError_t stage2d_go(const DevModel& m, const StageArgs2D<T>& a, cudaStream_t s) {
  if constexpr (std::is_same_v<T, float> && !RECT) {
    return launch_stream2d_f32(FLUX, BLEND ? (a.blend_external ? 2 : 1) : 0, m, a, s);
  } else {
    constexpr int H = BLEND ? 3 : 2;
    const long long c32 = tile_cost(a.nx, a.ny, 32, 8, H);
    if (6 * tile_cost(a.nx, a.ny, 12, 8, H) < 5 * c32) return stage2d_tiles<FLUX, T, BLEND, RECT, 12, 8, 192>(m, a, s);
    if constexpr (std::is_same_v<T, float> && !BLEND) {
      if (10 * tile_cost(a.nx, a.ny, 32, 12, H) < 9 * c32) return stage2d_tiles<FLUX, T, BLEND, RECT, 32, 12>(m, a, s);
    }
    return stage2d_tiles<FLUX, T, BLEND, RECT, 32, 8>(m, a, s);
  }
}

template <class T, bool RECT>
static cudaError_t stage2d_dispatch(int flux, bool blend, const DevModel& m, const StageArgs2D<T>& a,
                                    cudaStream_t s) {
  switch (flux) {
    case FLUX_ZERO: return blend ? stage2d_go<FLUX_ZERO, T, true, RECT>(m, a, s) : stage2d_go<FLUX_ZERO, T, false, RECT>(m, a, s);
    case FLUX_LINEAR:
      return blend ? stage2d_go<FLUX_LINEAR, T, true, RECT>(m, a, s) : stage2d_go<FLUX_LINEAR, T, false, RECT>(m, a, s);
    case FLUX_BURGERS:
      return blend ? stage2d_go<FLUX_BURGERS, T, true, RECT>(m, a, s) : stage2d_go<FLUX_BURGERS, T, false, RECT>(m, a, s);
    case FLUX_BL: return blend ? stage2d_go<FLUX_BL, T, true, RECT>(m, a, s) : stage2d_go<FLUX_BL, T, false, RECT>(m, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace af
