// Fused 1D stage kernel of the compact fourth-order doubly conservative active flux
// method (arXiv 2510.11527, Sections 2 and 5.1; Appendix A for the diffusion form
// without double conservation). Same structure as the 2D kernel: each CTA owns TX cells
// (cell average ub_i and the point value P_i = u_{i+1/2}) and stages a +-3 cell halo
// in shared memory.
//   centre          u_i = (6 ub_i - u_{i-1/2} - u_{i+1/2}) / 4
//   point residual  5-point line [P_{i-1}, c_i, P_i, c_{i+1}, P_{i+1}]
//   DC potential    a^_i = (-a(P_{i-1}) + 8 a(c_i) - a(P_i)) / 6   (Proposition 2.1)
//   low order       LLF with interval wave speed, states u^{L,+-} with factor 2
//   limiter         theta^c (2 states; factor 6, or 2 without a diffusion term) and
//                   theta^d (4 states; factor 6)
// Without double conservation (Appendix A) the face flux is f(P_i) - kappa(P_i) D_c(u),
// D_c(u) = (P_{i-1} - 8 c_i + 8 c_{i+1} - P_{i+1}) / (6 dx), the point value takes
// 4/dx^2 sum_{m,n} b_mn kappa(z_m) z_n on its line, and the limiter blends the total
// face flux with F^L - (a(ub_{i+1}) - a(ub_i))/dx by Theta with factor 2.
// A bounded interval (Dirichlet / outflow ends) reads ghost cells and points from the
// boundary rule, updates the extra left end point u_{-1/2} in its first tile, and holds
// Dirichlet end points at the boundary values.
#pragma once
#include <cooperative_groups.h>

#include "launch.h"

namespace af {

// A tile of TX cells with a +-3 cell halo, worked on by NT threads. Two shapes: 256 cells
// by 256 threads for long meshes, and 26 cells by one warp (halo included, one box
// position per lane) for meshes that would otherwise leave most SMs idle: GB300's FP64
// unit passes 2 lanes per clock and SM, so a short mesh is bound by the FP64 rate of the
// few SMs it runs on. Launched steps of Example 6.5's problem, FP64, 256-cell tiles /
// one-warp tiles: 200 cells 57 / 43 us, 10,000 61 / 43 us, 38,000 66 / 49 us (when the
// scalars were stored by a switch, which cost both); beyond 152 x 256 cells the long tile,
// whose halo costs 2 % of the work instead of 23 %.
template <int TX_, int NT_>
struct Tile1D {
  static constexpr int TX = TX_, NT = NT_, H = 3, BX = TX + 2 * H;
  static_assert(NT == TX || NT >= BX, "one thread per cell, or per box position");
};
using Tile1DLong = Tile1D<256, 256>;
using Tile1DWarp = Tile1D<WARP_TILE_1D, 32>;

// barrier among the threads of one tile
template <int NT>
__device__ __forceinline__ void tile_sync() {
  if constexpr (NT == 32) __syncwarp();
  else __syncthreads();
}

// Cell average ub_i and point value u_{j+1/2} at any index: stored values inside, the
// boundary rule outside (periodic image; Dirichlet value; even reflection about the
// end point for outflow). Indices far beyond an end (never read by an owned output)
// are clamped to the first H ghosts so that every load stays inside the arrays.
template <class PT>
__device__ __forceinline__ double cell1d(const StageArgs2D<PT>& A, int i, int H) {
  const int n = A.nx;
  if (A.bc == AF_BC_PERIODIC) return A.ub[wrapi(i, n)];
  if (i >= 0 && i < n) return A.ub[i];
  if (A.bc == AF_BC_DIRICHLET) return i < 0 ? A.bc_left : A.bc_right;
  i = i < -H ? -H : (i >= n + H ? n + H - 1 : i);
  return A.ub[i < 0 ? -1 - i : 2 * n - 1 - i];
}
template <class PT>
__device__ __forceinline__ PT point1d(const StageArgs2D<PT>& A, int j, int H) {
  const int n = A.nx;
  if (A.bc == AF_BC_PERIODIC) return A.V[wrapi(j, n)];
  if (j >= -1 && j <= n - 1) return A.V[j + 1];
  if (A.bc == AF_BC_DIRICHLET) return PT(j < -1 ? A.bc_left : A.bc_right);
  j = j < -H - 1 ? -H - 1 : (j >= n + H ? n + H - 1 : j);
  return A.V[(j < -1 ? -2 - j : 2 * (n - 1) - j) + 1];
}

// 4 sum_{m,n} b_mn k_m z_n of Appendix A, B = [0 0; 0 M] - [M 0; 0 0] written out row
// by row (each row sums to zero)
template <class T>
__device__ __forceinline__ T nodc_d2(const T z[5], const T k[5]) {
  const T r0 = T(-1.0 / 8) * z[0] + T(1.0 / 6) * z[1] - T(1.0 / 24) * z[2];
  const T r1 = T(1.0 / 6) * z[0] + T(0.5) * z[1] - T(5.0 / 6) * z[2] + T(1.0 / 6) * z[3];
  const T r2 = T(-1.0 / 8) * (z[0] + z[4]) + T(0.5) * (z[1] + z[3]) - T(0.75) * z[2];
  const T r3 = T(1.0 / 6) * z[1] - T(5.0 / 6) * z[2] + T(0.5) * z[3] + T(1.0 / 6) * z[4];
  const T r4 = T(-1.0 / 24) * z[2] + T(1.0 / 6) * z[3] - T(1.0 / 8) * z[4];
  return T(4) * ((k[0] * r0 + k[1] * r1) + (k[2] * r2 + (k[3] * r3 + k[4] * r4)));
}

// double -> exact widening of a stencil value (FP32 on the integer pipe)
__device__ __forceinline__ double d_of(double v) { return v; }
__device__ __forceinline__ double d_of(float v) { return f2d_exact(v); }

// The launch's scalars, formed once per tile: GB300 runs FP64 arithmetic, FP64 compares
// and double <-> float conversions on its FP64 unit at 1/64 of the FP32 rate, so
// per-thread copies would cost each cell as much as its own FP64 work. Value k of output o
// comes from lane k; of a mesh's values (C_UMIN on) output 0's copy is read.
template <class T>
struct Scal1D {
  T t[2][32];
  double d[2][4];   // C_MU, C_NU unrounded
};
enum : int { C_TAU = 0, C_MU, C_NU, C_M2, C_N2, C_K6, C_Q6, C_CA, C_CF, C_UMIN = 16, C_UMAX, C_IH, C_I6H, C_I3H2,
             C_G, C_I4HH, C_I2H };

// shared memory of one tile
template <class T, int BX>
struct Shared1D {
  T U[BX], P[BX], C[BX];
  // aP / aC hold kappa instead of a without double conservation (no DC potential)
  T fP[BX], aP[BX], fC[BX], aC[BX], dP[BX], dC[BX], fU[BX], aU[BX];
  T FH[BX], AH[BX], FL[BX], ULp[BX], ULm[BX], Flim[BX], Alim[BX];
  T S[BX], TC[BX], TD[BX];
  Scal1D<T> sc;
};

// One tile of cells i0 .. i0 + TX - 1 (tid: the thread's index in the tile): one or two
// limited forward-Euler evaluations with step tcoef * dtv, their combination and store.
template <int FLUX, class T, class PT, class L>
__device__ __forceinline__ void stage1d_tile(const DevModel& m, const StageArgs2D<PT>& A, double dtv, int i0, int tid,
                                             Shared1D<T, L::BX>& sm) {
  constexpr int TX = L::TX, NT = L::NT, H = L::H, BX = L::BX;
  // flux direction of the model functions: the 1D Buckley-Leverett flux is the gravity
  // form f1 (1 - g (1-u)^2), which the model keeps as direction 1 (Example 6.6)
  constexpr int XD = FLUX == FLUX_BL ? 1 : 0;
  T *sU = sm.U, *sP = sm.P, *sC = sm.C, *fP = sm.fP, *aP = sm.aP, *fC = sm.fC, *aC = sm.aC, *dP = sm.dP, *dC = sm.dC,
    *fU = sm.fU, *aU = sm.aU, *sFH = sm.FH, *sAH = sm.AH, *sFL = sm.FL, *sULp = sm.ULp, *sULm = sm.ULm,
    *sFlim = sm.Flim, *sAlim = sm.Alim, *sS = sm.S, *sTC = sm.TC, *sTD = sm.TD;
  Scal1D<T>& sc = sm.sc;
  const int nx = A.nx;
  // formed at once by the lanes of warp o (output o) and the upper lanes of warp 0 (the
  // mesh's values): GB300's FP64 unit takes as long for a warp instruction with one
  // active lane as with 32. Lane l evaluates fl(fl(fl(x y1) y2) y3) with the factors of
  // its value's formula (a factor 1 is exact, so each value is rounded as its formula
  // is; the divided line scales come from the host) and stores it at its own index (a
  // switch over the lanes' destinations ran its 17 cases one after the other, in the chain
  // that every stage of a short mesh starts with: 200 cells FP64 35.0 -> 33.0 us per step
  // on its own, 5000 43.2 -> 37.1).
  for (int o = tid >> 5; o < A.nout; o += NT / 32) {
    const int l = tid & 31;
    const double ih = A.inv_h1, tau = A.tcoef[o] * dtv;
    double x = tau, y1 = 1.0, y2 = 1.0, y3 = 1.0;
    if (l < 16) {
      // 0: tau; 1: mu; 2: nu; 3: 2 mu; 4: 2 nu; 5: (2 or 2 P) mu; 6: 6 nu; 7, 8: cA, cF
      if (l >= 1 && l <= 6) y1 = ih;
      if (l == 2 || l == 4 || l == 6) y2 = ih;
      if (l == 3) y2 = 2.0;
      if (l == 5) y2 = A.nodc ? 2.0 : double(2 * m.lim_parts);
      if (l == 4) y3 = 2.0;
      if (l == 6) y3 = 6.0;
      if (l == 7) x = A.cA[o];
      if (l == 8) x = A.cF[o];
    } else {
      // 16, 17: u_min, u_max; 18: 1/h; 19: 1/(6h); 20: (1/h/h)/3; 21: gamma; 22: (4/h)/h;
      // 23: 2/h
      x = l == 16   ? m.umin
          : l == 17 ? m.umax
          : l == 21 ? A.gamma
          : l == 22 ? 4.0
          : l == 23 ? 2.0
          : l == 19 ? A.i6h[0]
          : l == 20 ? A.i3h2[0]
                    : ih;
      y1 = (l == 22 || l == 23) ? ih : 1.0;
      y2 = l == 22 ? ih : 1.0;
    }
    const double d = ((x * y1) * y2) * y3;
    sc.t[o][l] = T(d);
    if (l < 4) sc.d[o][l] = d;
  }
  tile_sync<NT>();
  const T umin = sc.t[0][C_UMIN], umax = sc.t[0][C_UMAX];
  const bool blend = A.blend != 0;
  const bool ext = A.blend == 2;
  const bool nodc = A.nodc != 0;
  const bool bounded = A.bc != AF_BC_PERIODIC;
  const int poff = bounded ? 1 : 0;   // point u_{j+1/2} is stored at index j + poff

  for (int k = tid; k < BX; k += NT) {
    // rounded toward the nearer bound, as the 2D stages round the averages (integer ops)
    sU[k] = to_stencil_nb<T>(cell1d(A, i0 - H + k, H), m.umid);
    sP[k] = T(point1d(A, i0 - H + k, H));
  }
  tile_sync<NT>();
  for (int b = tid; b < BX; b += NT) {
    const T u = sU[b];
    fU[b] = flux<FLUX, T>(m, XD, u);
    aU[b] = apot<T>(m, u);
    const T p = sP[b];
    fP[b] = flux<FLUX, T>(m, XD, p);
    if constexpr (FLUX != FLUX_BURGERS) dP[b] = dflux_abs<FLUX, T>(m, XD, p);
    aP[b] = nodc ? kappa_fn<T>(m, p) : apot<T>(m, p);
    if (b >= 1) {
      const T c = (T(6) * u - sP[b - 1] - p) * T(0.25);
      sC[b] = c;
      fC[b] = flux<FLUX, T>(m, XD, c);
      if constexpr (FLUX != FLUX_BURGERS) dC[b] = dflux_abs<FLUX, T>(m, XD, c);
      aC[b] = nodc ? kappa_fn<T>(m, c) : apot<T>(m, c);
    }
    if (blend && !ext && b >= 1 && b < BX - 1) {
      const T um = sU[b - 1], up = sU[b + 1];
      sTC[b] = tabs(um - T(2) * u + up) / (tabs(um) + T(2) * tabs(u) + tabs(up) + T(1e-13));
    }
  }
  tile_sync<NT>();
  const T ih = sc.t[0][C_IH], i6h = sc.t[0][C_I6H], i3h2 = sc.t[0][C_I3H2];
  // points updated by this thread: its own u_{i+1/2} and, in the first tile of a bounded
  // interval, thread 0 also the left end point u_{-1/2} (held at the boundary value
  // when the end is Dirichlet)
  // (a one-warp tile gives it to a lane without a cell of its own instead)
  constexpr bool SPARE = NT > TX;
  const bool extra = bounded && i0 == 0 && tid == (SPARE ? TX : 0);
  const int nq = SPARE ? (tid < TX || extra ? 1 : 0) : (extra ? 2 : 1);
  const int bq[2] = {SPARE && tid >= TX ? H - 1 : H + tid, H - 1};
  // high-order point residual
  T rH[2] = {T(0), T(0)};
  for (int q = 0; q < nq; ++q) {
    const int b = bq[q];
    // max |f'| over the line; for Burgers |2p| max |z| (the same value: rounding is
    // monotone), which spares two FP64 multiplies per cell
    T alpha;
    if constexpr (FLUX == FLUX_BURGERS)
      alpha = tabs(T(2) * par<T>(m.fp, m.fpf, 0)) *
              tmax(tmax(tmax(tabs(sP[b - 1]), tabs(sC[b])), tmax(tabs(sC[b + 1]), tabs(sP[b + 1]))), tabs(sP[b]));
    else
      alpha = tmax(tmax(tmax(dP[b - 1], dC[b]), tmax(dC[b + 1], dP[b + 1])), dP[b]);
    if (!nodc) {
      rH[q] = line_res<T>(sP[b - 1], sC[b], sP[b], sC[b + 1], sP[b + 1], fP[b - 1], fC[b], fC[b + 1], fP[b + 1],
                          alpha, aP[b - 1], aC[b], aP[b], aC[b + 1], aP[b + 1], i6h, i3h2);
    } else {
      const T z[5] = {sP[b - 1], sC[b], sP[b], sC[b + 1], sP[b + 1]};
      const T k[5] = {aP[b - 1], aC[b], aP[b], aC[b + 1], aP[b + 1]};
      rH[q] = line_res<T>(z[0], z[1], z[2], z[3], z[4], fP[b - 1], fC[b], fC[b + 1], fP[b + 1], alpha, T(0), T(0),
                          T(0), T(0), T(0), i6h, i3h2) +
              nodc_d2<T>(z, k) * (T(3) * i3h2);
    }
  }
  for (int b = H - 2 + tid; b <= H + TX; b += NT) {
    const T ul = sU[b], ur = sU[b + 1];
    // LLF flux (f_l + f_r - alpha (u_r - u_l)) / 2: one multiply-add and one multiply
    const T fl = T(0.5) * ((fU[b] + fU[b + 1]) - alpha_interval<FLUX, T>(m, XD, ul, ur) * (ur - ul));
    if (!nodc) {
      if (b >= H - 1 && b < H + TX) sFH[b] = fP[b];
      if (b >= H - 1) sAH[b] = (T(8) * aC[b] - aP[b - 1] - aP[b]) * T(1.0 / 6.0);
      sFL[b] = fl;
    } else {
      // total face fluxes: f(P) - kappa(P) D_c(u) and F^L - (a(ub_{i+1}) - a(ub_i)) / dx
      if (b >= H - 1 && b < H + TX)
        sFH[b] = fP[b] - aP[b] * (((sP[b - 1] - sP[b + 1]) + T(8) * (sC[b + 1] - sC[b])) * i6h);
      sFL[b] = fl - (aU[b + 1] - aU[b]) * ih;
    }
  }
  if (blend) {
    for (int b = H - 1 + tid; b <= H + TX; b += NT) {
      sS[b] = ext ? T(A.s_ext[wrapi(i0 - H + b, nx)]) : (sTC[b - 1] + T(4) * sTC[b] + sTC[b + 1]) * T(1.0 / 6.0);
    }
  }
  tile_sync<NT>();
  T rP[2] = {rH[0], rH[1]};
  if (blend) {
    const T g = sc.t[0][C_G];
    for (int b = H - 1 + tid; b <= H + TX; b += NT) {
      sTD[b] = exp(-g * sS[b]);
      if (b < H + TX) sTC[b] = exp(-g * (T(0.5) * (sS[b] + sS[b + 1])));
    }
    tile_sync<NT>();
    for (int b = H - 1 + tid; b <= H + TX; b += NT) {
      if (b < H + TX) sFH[b] = sTC[b] * sFH[b] + (T(1) - sTC[b]) * sFL[b];
      sAH[b] = sTD[b] * sAH[b] + (T(1) - sTD[b]) * aU[b];
    }
    for (int q = 0; q < nq; ++q) {
      const int b = bq[q];
      const T zm = sU[b], z0 = sP[b], zp = sU[b + 1];
      const T Fr = T(0.5) * (fP[b] + fU[b + 1]) - T(0.5) * alpha_interval<FLUX, T>(m, XD, z0, zp) * (zp - z0);
      const T Fl = T(0.5) * (fU[b] + fP[b]) - T(0.5) * alpha_interval<FLUX, T>(m, XD, zm, z0) * (z0 - zm);
      const T RL = (aU[b + 1] - T(2) * aP[b] + aU[b]) * sc.t[0][C_I4HH] - (Fr - Fl) * sc.t[0][C_I2H];
      rP[q] = sTC[b] * rH[q] + (T(1) - sTC[b]) * RL;
    }
    tile_sync<NT>();
  }
  const int gi = i0 + tid;
  const bool own = tid < TX && gi < nx;
  T* Flim = A.limiter ? sFlim : sFH;
  T* Alim = A.limiter ? sAlim : sAH;
  for (int o = 0; o < A.nout; ++o) {
    const double mu = sc.d[o][C_MU], nu = sc.d[o][C_NU];
    const bool comb = !is_zero_bits(A.cA[o]);
    if (A.limiter) {
      const T m2 = sc.t[o][C_M2], n2 = sc.t[o][C_N2];
      for (int b = H - 2 + tid; b <= H + TX + 1; b += NT) {
        const T u = sU[b], f = fU[b], a = aU[b];
        if (!nodc) {
          if (b <= H + TX) sULp[b] = u - m2 * (sFL[b] - f) + n2 * (aU[b + 1] - a);
          if (b >= H - 1) sULm[b] = u - m2 * (f - sFL[b - 1]) - n2 * (a - aU[b - 1]);
        } else {
          // sFL already holds the total low-order face flux (diffusion included)
          if (b <= H + TX) sULp[b] = u - m2 * (sFL[b] - f);
          if (b >= H - 1) sULm[b] = u - m2 * (f - sFL[b - 1]);
        }
      }
      tile_sync<NT>();
      // face factor 2 * parts (6 with diffusion, 2 without); the total face flux of the
      // form without double conservation takes factor 2 (the average is the mean of
      // u^{L,+} and u^{L,-}, one face correction each)
      const T k6 = sc.t[o][C_K6], q6 = sc.t[o][C_Q6];
      for (int b = H - 1 + tid; b <= H + TX; b += NT) {
        if (b < H + TX) {
          const T fh = sFH[b], fl = sFL[b], dF = fh - fl;
          const T zp = sULp[b], zm = sULm[b + 1];
          const T t = tmin(theta_fn<T>(zp, zp - k6 * dF, umin, umax), theta_fn<T>(zm, zm + k6 * dF, umin, umax));
          sFlim[b] = is_one(t) ? fh : fl + t * dF;
        }
        if (!nodc) {
          const T ah = sAH[b], al = aU[b], d = q6 * (ah - al);
          const T t = tmin(tmin(theta_fn<T>(sULp[b - 1], sULp[b - 1] + d, umin, umax),
                                theta_fn<T>(sULp[b], sULp[b] - d, umin, umax)),
                           tmin(theta_fn<T>(sULm[b], sULm[b] - d, umin, umax),
                                theta_fn<T>(sULm[b + 1], sULm[b + 1] + d, umin, umax)));
          sAlim[b] = is_one(t) ? ah : al + t * (ah - al);
        }
      }
      tile_sync<NT>();
    }
    if (own) {
      const int b = H + tid;
      const size_t g = (size_t)gi;
      double ubfe = A.ub[g] - mu * (d_of(Flim[b]) - d_of(Flim[b - 1]));
      if (!nodc) ubfe += nu * ((d_of(Alim[b + 1]) - 2.0 * d_of(Alim[b])) + d_of(Alim[b - 1]));
      double ubo = comb ? rk_comb(A.cA[o], A.Aub[o][g], A.cF[o], ubfe) : rk_scale(A.cF[o], ubfe);
      if (A.limiter && A.sg[o]) ubo = safeguard<double>(ubo, m.umin, m.umax, A.tol, A.stats, true);
      A.Oub[o][g] = ubo;
    }
    for (int q = 0; q < nq; ++q) {
      const int gj = q == 0 && tid < TX ? gi : -1;   // point index j of u_{j+1/2}
      if (gj >= nx) continue;
      const size_t g = (size_t)(gj + poff);
      PT po;
      if (A.bc == AF_BC_DIRICHLET && (gj == -1 || gj == nx - 1)) {
        po = PT(gj == -1 ? A.bc_left : A.bc_right);
      } else {
        T p = sP[bq[q]] + sc.t[o][C_TAU] * rP[q];
        if (A.limiter) p = tmin(tmax(p, umin), umax);
        po = comb ? PT(rk_comb(sc.t[o][C_CA], T(A.AV[o][g]), sc.t[o][C_CF], p)) : PT(rk_scale(sc.t[o][C_CF], p));
        if (A.limiter && A.sg[o]) po = safeguard<PT>(po, PT(umin), PT(umax), A.tol, A.stats);
      }
      A.OV[o][g] = po;
    }
    if (o + 1 < A.nout) tile_sync<NT>();
  }
}

// One CTA per 256-cell tile (4 CTAs per SM: 64 registers).
template <int FLUX, class T, class PT>
__global__ void __launch_bounds__(256, 4) stage1d_kernel(const DevModel m, const StageArgs2D<PT> A) {
  using L = Tile1DLong;
  __shared__ Shared1D<T, L::BX> sm;
  const double dtv = *A.dt;
  if (is_zero_bits(dtv)) return;   // uniform over the grid
  stage1d_tile<FLUX, T, PT, L>(m, A, dtv, blockIdx.x * L::TX, threadIdx.x, sm);
}

// One warp per 26-cell tile, CTAs of one warp so that a short mesh spreads over the SMs.
template <int FLUX, class T, class PT>
__global__ void __launch_bounds__(32) stage1d_warp_kernel(const DevModel m, const StageArgs2D<PT> A) {
  using L = Tile1DWarp;
  __shared__ Shared1D<T, L::BX> sm;
  const double dtv = *A.dt;
  if (is_zero_bits(dtv)) return;   // uniform over the grid
  stage1d_tile<FLUX, T, PT, L>(m, A, dtv, blockIdx.x * L::TX, threadIdx.x, sm);
}

// Whole steps of a short mesh in one launch.
//
// A short mesh is bound by latency: as 5 launches per step (rate, step size, 3 stages) a
// 200-cell FP64 run took 59 us per step, launch gaps and one SM's FP64 unit. Here one
// cluster of 8 CTAs takes up to `nsteps` whole steps: warp w of CTA r works on tile
// r + 8 w (26 cells), every stage ends in a cluster barrier (hardware, no spinning), the
// CFL maximum is exchanged through distributed shared memory, and each CTA forms the same
// step from it: 28 us per step, now the chain of ~1300 instructions of one tile per stage.
// Up to 832 cells a step costs the same; launched stages of one-warp tiles take 37 us.
template <int FLUX, class T, class PT>
__global__ void __launch_bounds__(32 * MARCH_WARPS) march1d_kernel(const DevModel m,
                                                                   const __grid_constant__ MarchArgs<PT> M) {
  using L = Tile1DWarp;
  __shared__ Shared1D<T, L::BX> sm[MARCH_WARPS];
  __shared__ unsigned long long wbits[MARCH_WARPS];
  __shared__ unsigned wflags[MARCH_WARPS];
  __shared__ unsigned long long cbits[MARCH_CTAS];   // written by every CTA of the cluster
  __shared__ unsigned cflags[MARCH_CTAS];
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int warps = blockDim.x >> 5;
  const StageArgs2D<PT>& A0 = M.st[0];
  const int nx = A0.nx, tile = rank + MARCH_CTAS * warp, i0 = tile * L::TX;
  const bool has = i0 < nx;   // whole warp
  double t = M.fin.t_acc ? *M.fin.t_acc : 0.0, dt = 0.0, steps = 0.0;
  cl.sync();   // every CTA has started: its shared memory may be written
  for (int n = 0; n < M.nsteps; ++n) {
    if (M.dt_fixed > 0.0) {
      dt = M.dt_fixed;
    } else {
      // the rate of this warp's cells (see dt_rate_maxu_kernel and dt_rate_kernel)
      unsigned long long bits = 0ull;
      unsigned flags = 0u;
      const int i = i0 + lane;
      if (has && lane < L::TX && i < nx) {
        const double* ub = A0.ub;
        const double u = ub[i], ih = M.fin.inv_h1, kd = M.fin.kmax * ih * ih;
        auto rate = [&](double v) {
          double d;
          if constexpr (FLUX == FLUX_BL) d = bl_eval<double>(m, v).d[1];
          else d = alpha_interval<FLUX, double>(m, 0, v, v);
          return rate_bits_of(d * ih + kd);
        };
        bits = rate(u);
        if (A0.bc == AF_BC_DIRICHLET && (i == 0 || i == nx - 1)) {   // the end faces' ghosts (nx >= 4)
          const unsigned long long e = rate(i == 0 ? A0.bc_left : A0.bc_right);
          bits = e > bits ? e : bits;
        }
        if constexpr (FLUX == FLUX_BL) {
          double un = ub[i + 1 == nx ? 0 : i + 1];
          if (A0.bc != AF_BC_PERIODIC && i + 1 == nx) un = A0.bc == AF_BC_DIRICHLET ? A0.bc_right : u;
          flags = crit_flags<FLUX>(m, 0, u, un);
          if (A0.bc == AF_BC_DIRICHLET && i == 0) flags |= crit_flags<FLUX>(m, 0, A0.bc_left, u);
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, bits, o);
        bits = v > bits ? v : bits;
      }
      flags = __reduce_or_sync(0xffffffffu, flags);
      if (lane == 0) {
        wbits[warp] = bits;
        wflags[warp] = flags;
      }
      __syncthreads();
      if (threadIdx.x < MARCH_CTAS) {
        for (int w = 0; w < warps; ++w) {
          bits = wbits[w] > bits ? wbits[w] : bits;
          flags |= wflags[w];
        }
        // lane r stores this CTA's maximum into CTA r
        cl.map_shared_rank(cbits, threadIdx.x)[rank] = bits;
        cl.map_shared_rank(cflags, threadIdx.x)[rank] = flags;
      }
      cl.sync();
      bits = 0ull;
      flags = 0u;
      for (int r = 0; r < MARCH_CTAS; ++r) {
        bits = cbits[r] > bits ? cbits[r] : bits;
        flags |= cflags[r];
      }
      dt = cfl_step(m, M.fin, bits, flags, t);
      if (is_zero_bits(dt)) break;   // the end time is reached (uniform over the cluster)
      if (dt > 0.0) steps += 1.0;
    }
    t += dt;
    for (int k = 0; k < M.nstages; ++k) {
      if (has) stage1d_tile<FLUX, T, PT, L>(m, M.st[k], dt, i0, lane, sm[warp]);
      __syncwarp();
      cl.sync();   // the stage's stores are visible to the cluster; also ends the reads of cbits
    }
  }
  if (rank == 0 && threadIdx.x == 0) {
    *M.fin.dt_out = dt;
    if (M.fin.t_acc) *M.fin.t_acc = t;
    if (M.fin.t_acc && M.fin.t_end > 0.0) *M.fin.count += steps;
  }
}

}  // namespace af
