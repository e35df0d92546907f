// Tiling of the z-marching 3D stage (march3d.cuh) and the rule that chooses it over the
// four kernels of stage3d.cu (host code).
#pragma once
#include "af.h"

namespace af {

constexpr int M3_BAND = 28;   // output columns per tile

// Rows per CTA, the larger and the smaller choice. The CTA's registers are the SM's: 16
// rows at 128, 12 at 168 and 8 at 255 registers per thread; more rows cost fewer halo rows
// per output row, fewer registers spill (porous medium 80^3 FP64 at 8 / 12 rows: 2.85 / 2.67
// ms per SSP-RK(5,4) step). The smaller one is for meshes that leave SMs without a tile.
constexpr int m3_rows(int flux, bool fp64) { return fp64 ? 12 : (flux == AF_FLUX_ZERO ? 16 : 12); }
constexpr int M3_ROWS_SMALL = 8;

// Layers per strip and the cost of a launch with TY rows per CTA: the number of strips
// with the fewest steps over all waves of CTAs (one CTA per SM), in microseconds of an
// FP64 stage of the porous medium: a row of a step takes 3.0 us at 12 rows per CTA and 3.4
// us at 8 (fewer warps), a strip's warm-up and drain cost it about 1.2 steps, a CTA's halo
// rows about 0.8 rows (measured 128^3 2161 us, 80^3 425, 64^3 333, 33^3 102, 20^3 42).
struct M3Plan {
  int bands, rows, S;
  double cost;
};
inline M3Plan m3_plan(const int* n, int TY) {
  M3Plan p;
  p.bands = (n[0] + M3_BAND - 1) / M3_BAND;
  p.rows = (n[1] + TY - 5) / (TY - 4);
  p.S = n[2];
  const long long tiles = (long long)p.bands * p.rows;
  double best = -1.0;
  // one number of strips per height (the next one lowers it): about 2 sqrt(n[2]) of them, as
  // every stage's launch asks (1216 strips one by one took 5 us of host time per call)
  for (int s = 1, L; s <= n[2] && s <= 152 * 8; s = L > 1 ? (n[2] + L - 2) / (L - 1) : n[2] + 1) {
    L = (n[2] + s - 1) / s;
    const long long waves = (tiles * ((n[2] + L - 1) / L) + 151) / 152;
    if (best < 0.0 || waves * (L + 1.2) < best) {
      best = waves * (L + 1.2);
      p.S = L;
    }
  }
  p.cost = best * (TY - 4 + 0.8) * (TY > M3_ROWS_SMALL ? 3.0 : 3.4);
  return p;
}

// Whether a mesh's stage without the blend marches. FP32-mixed always does (128^3 zero /
// Burgers flux: 1922 -> 534 / 2101 -> 824 us per step; 20^3: 165 -> 42 us). FP64 is bound
// by the FP64 unit, and a marching tile repeats work in its halo: with a flux (six LLF
// fluxes per cell instead of three, only 8 rows per CTA for lack of registers) the four
// kernels were faster from 40^3 on (128^3: 13.2 against 15.9 ms per step), and the march has
// no such form; without one (porous medium) it depends on how well the mesh fills tiles of 28
// columns: a stage takes about 55 us + 1.13 ns per cell in four kernels and 4 us + m3_plan's
// cost here (33^3: 97 / 106 us; 40 x 45 x 26: 104 / 100; 21 x 102 x 61: 215 / 178; 128^3:
// 2377 / 2161; 20^3: 80 / 42); it marches where that predicts at least 3 % less.
inline bool march3d_takes(int flux, bool fp64, const int* n) {
  if (!fp64) return true;
  if (flux != AF_FLUX_ZERO) return false;
  const double a = m3_plan(n, m3_rows(flux, true)).cost, b = m3_plan(n, M3_ROWS_SMALL).cost;
  return 4.0 + (a < b ? a : b) < 0.97 * (55.0 + 1.13e-3 * n[0] * (double)n[1] * n[2]);
}

}  // namespace af
