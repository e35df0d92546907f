// 3D stage without the blend, marching along z: the limited forward-Euler evaluation and
// Shu-Osher combination of Section 5.2 with d = 3 (arXiv 2510.11527; periodic meshes) in
// one launch per output and without scratch arrays.
//
// A CTA owns a tile of 28 columns by TY - 4 rows and a strip of layers. Its TY warps are
// the rows y0 - 2 .. y0 + TY - 3 of the tile, lane L the column x0 - 2 + L, so every
// thread holds one column of cells (lanes 2 .. 29 of rows 2 .. TY - 3 produce outputs, the
// others supply the +-2 halo; a halo row forms only what its neighbours read). The CTA
// marches up its strip one layer of cells per step. Neighbours along x are reached by
// shuffles, along y through shared memory (one barrier per step), along z through
// registers. At step r layer r arrives; its centres, cell potentials, face fluxes,
// x- and y-limiters and the x- and y-lines of its points are formed; the z-lines finish the
// points of layer r - 1, the z-limiter works on cell r - 1 and the averages of layer r - 2
// are finished.
//
// FP64 form (zero flux): a cell's 27 half-spaced locations enter its centre and its three
// potentials only through 8 sums (the centre; the pairs of x-, y- and z-faces; the fours of
// xy-, xz- and yz-edges; the 8 corners), each built from sums along one axis after another:
// 19 additions and 8 operations per direction instead of 27 weighted terms per direction.
//
// FP32-mixed form: stencils and limiters in FP32; the averages are updated from the widened
// face values in FP64 (differences, products with mu and nu, sums). That costs: with the
// increment as FP32 pairs, which hold 46 bits of it and lose them for states near FP32's
// smallest normals, a step of the porous medium at 128^3 took 503 instead of 531 us and one of
// Burgers' equation with constant diffusion 742 instead of 824 us.
//
// Measured (porous medium; against the four kernels with 19 scratch arrays, which the blend
// and, where they are faster, FP64 meshes still take: march3d_takes): FP32-mixed 128^3
// SSP-RK3 step 1.90 -> 0.53 ms, FP64 80^3 SSP-RK(5,4) step 3.36 -> 2.55 ms. FP64 is bound by
// the FP64 unit (77 % of its cycles busy), FP32-mixed by instruction issue (about 900
// instructions per layer and full row) and the waits of one CTA's 16 warps on each other at
// the barrier; DRAM moves 58 bytes per cell and stage. With two barriers per step the FP32
// step took 0.66 ms.
#pragma once
#include "launch.h"
#include "march3d_plan.h"
#include "stencil.cuh"

namespace af {

// the launch's scalars
template <class T>
struct M3Scal {
  double mu[3], nu[3];
  T mu6[3], nu6[3], kc[3], kd[3];     // 6 mu, 6 nu, (18 or 6) mu, 18 nu
  T taut, umin, umax, cAt, cFt;
  T mid;                              // -30 sum_l 1 / (3 h_l^2)
};

// lanes of one warp: lane l = 3 kind + dir forms fl(fl(fl(tau / h) [/ h]) factor); lanes
// 18 .. 22 round tau, u_min, u_max, cA, cF
template <class T>
__device__ __forceinline__ void m3_scalars(const DevModel& m, const StageArgs3D<T>& A, int o, double dtv,
                                           M3Scal<T>& sc) {
  const int l = threadIdx.x & 31, kind = l / 3, dir = l % 3;
  const double tau = A.tcoef[o] * dtv, ih = A.inv_h[dir];
  if (l == 23) sc.mid = T(-30.0 * (A.i3h2[0] + A.i3h2[1] + A.i3h2[2]));
  double x = tau, y1 = ih, y2 = 1.0, y3 = 1.0;
  if (l < 18) {
    if (kind == 1 || kind == 3 || kind == 5) y2 = ih;
    y3 = kind < 2 ? 1.0 : (kind < 4 ? 6.0 : (kind == 4 ? double(6 * m.lim_parts) : 18.0));
  } else {
    y1 = 1.0;
    x = l == 18 ? tau : (l == 19 ? m.umin : (l == 20 ? m.umax : (l == 21 ? A.cA[o] : A.cF[o])));
  }
  const double d = ((x * y1) * y2) * y3;
  const T t = T(d);
  if (l < 18) {
    switch (kind) {
      case 0: sc.mu[dir] = d; break;
      case 1: sc.nu[dir] = d; break;
      case 2: sc.mu6[dir] = t; break;
      case 3: sc.nu6[dir] = t; break;
      case 4: sc.kc[dir] = t; break;
      default: sc.kd[dir] = t; break;
    }
  } else {
    switch (l) {
      case 18: sc.taut = t; break;
      case 19: sc.umin = t; break;
      case 20: sc.umax = t; break;
      case 21: sc.cAt = t; break;
      case 22: sc.cFt = t; break;
      default: break;
    }
  }
}

// exact widening of a stencil value, the FP32 one with integer operations (f2d_exact) but
// with the test for subnormal values made once for three of them
__device__ __forceinline__ double m3_wide(float f) {   // zero or normal
  const unsigned u = __float_as_uint(f), mag = u & 0x7FFFFFFFu;
  return __hiloint2double((int)(mag == 0u ? u : (u & 0x80000000u) | ((mag >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ void m3_wide3(const double (&x)[3], double (&y)[3]) {
  for (int k = 0; k < 3; ++k) y[k] = x[k];
}
__device__ __forceinline__ void m3_wide3(const float (&x)[3], double (&y)[3]) {
  unsigned t = 0xFFFFFFFFu;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    y[k] = m3_wide(x[k]);
    t = min(t, (__float_as_uint(x[k]) & 0x7FFFFFFFu) - 1u);
  }
  if (t < 0x007FFFFFu) {
#pragma unroll
    for (int k = 0; k < 3; ++k) y[k] = f2d_exact(x[k]);
  }
}

// increment of a cell average, in FP64 whatever the stencil type: the two cells of a face
// take its value with the same rounding
template <class T>
struct Incr {
  double v;
  __device__ __forceinline__ void zero() { v = 0.0; }
  // - mu (f0 - fm)
  __device__ __forceinline__ void conv(const M3Scal<T>& k, int l, T f0, T fm) {
    const T x[3] = {f0, fm, T(0)};
    double y[3];
    m3_wide3(x, y);
    v = __fma_rn(-k.mu[l], y[0] - y[1], v);
  }
  // nu (ap - 2 a0 + am)
  __device__ __forceinline__ void diff(const M3Scal<T>& k, int l, T ap, T a0, T am) {
    const T x[3] = {ap, a0, am};
    double y[3];
    m3_wide3(x, y);
    v = __fma_rn(k.nu[l], __fma_rn(-2.0, y[1], y[0] + y[2]), v);
  }
};

// What a layer leaves for the one above it: sums over its upper plane of z-faces. The FP64
// form adds the 27 locations by kind (see the top of this file): the z-face, the pairs of
// xz- and yz-edges and the four corners of z and a. The FP32 form keeps
// the order of the weighted 27-term sums, whose rounding shows in FP32: their first nine
// (three) terms, and the plane's nine values of a.
template <class T> struct M3Level;
template <> struct M3Level<double> {
  double z[4], a[4];
  __device__ __forceinline__ void clear() {
    for (int k = 0; k < 4; ++k) z[k] = a[k] = 0.0;
  }
};
template <> struct M3Level<float> {
  float cz, ax, ay, fx, fy, a[9];
  __device__ __forceinline__ void clear() {
    cz = ax = ay = fx = fy = 0.0f;
    for (int k = 0; k < 9; ++k) a[k] = 0.0f;
  }
};
// Simpson weight of location 3 (my + 1) + mx + 1 of a plane
constexpr __device__ float m3_w(int q) { return (q % 3 == 1 ? 4.0f : 1.0f) * (q / 3 == 1 ? 4.0f : 1.0f); }

// f_l(z) = c z with c = p0 z (Burgers) or the constant velocity (linear), so that it can
// enter a multiply-add unrounded
template <int FLUX, class T>
__device__ __forceinline__ T m3_c(const DevModel& m, int l, T z) {
  if constexpr (FLUX == FLUX_BURGERS) return par<T>(m.fp, m.fpf, 0) * z;
  else return par<T>(m.fp, m.fpf, l);
}
// f_l(z) - x and x - f_l(z)
template <int FLUX, class T>
__device__ __forceinline__ T m3_fminus(const DevModel& m, int l, T z, T x) { return sfma(m3_c<FLUX, T>(m, l, z), z, -x); }
template <int FLUX, class T>
__device__ __forceinline__ T m3_minusf(const DevModel& m, int l, T x, T z) { return sfma(-m3_c<FLUX, T>(m, l, z), z, x); }

// 5-point line residual of a point along l, added to that of the axes before (l > 0). The
// FP64 form of pure diffusion leaves out the middle point, whose term -30 a sum_l
// 1/(3 h_l^2) is added once (m3_middle).
template <int FLUX, class T>
__device__ __forceinline__ T m3_line(const DevModel& m, const StageArgs3D<T>& A, int l, T z0, T z1, T z2, T z3, T z4,
                                     T a0, T a1, T a2, T a3, T a4, T acc) {
  if constexpr (FLUX == FLUX_ZERO) {
    if constexpr (sizeof(T) == 8) {
      const T d = sfma(T(16), a1 + a3, -(a0 + a4));
      return l == 0 ? d * A.i3h2T[l] : sfma(d, A.i3h2T[l], acc);
    } else {
      const T r = sfma(T(-30), a2, sfma(T(16), a1 + a3, -(a0 + a4))) * A.i3h2T[l];
      return l == 0 ? r : acc + r;
    }
  } else {
    T alpha;
    if constexpr (FLUX == FLUX_BURGERS)
      alpha = tabs(T(2) * par<T>(m.fp, m.fpf, 0)) * fmx(fmx(fmx(tabs(z0), tabs(z1)), fmx(tabs(z3), tabs(z4))), tabs(z2));
    else
      alpha = tabs(par<T>(m.fp, m.fpf, l));
    const T f04 = m3_fminus<FLUX, T>(m, l, z0, flux<FLUX, T>(m, l, z4));
    const T f31 = m3_fminus<FLUX, T>(m, l, z3, flux<FLUX, T>(m, l, z1));
    const T cf = sfma(T(8), f31, f04);
    const T dz = sfma(T(6), z2, sfma(T(-4), z1 + z3, z0 + z4));
    const T da = sfma(T(-30), a2, sfma(T(16), a1 + a3, -(a0 + a4)));
    const T r = sfma(da, A.i3h2T[l], -(sfma(alpha, dz, cf) * A.i6hT[l]));
    return l == 0 ? r : acc + r;
  }
}
// the middle point's share of the three lines where m3_line leaves it out
template <int FLUX, class T>
__device__ __forceinline__ T m3_middle(const M3Scal<T>& k, T a, T acc) {
  if constexpr (FLUX == FLUX_ZERO && sizeof(T) == 8) return sfma(k.mid, a, acc);
  else return acc;
}

// LLF flux between two averages
template <int FLUX, class T>
__device__ __forceinline__ T m3_llf(const DevModel& m, int l, T ul, T ur) {
  const T al = alpha_interval_pre<FLUX, T>(m, l, ul, ur, T(0), T(0));
  const T f = sfma(m3_c<FLUX, T>(m, l, ul), ul, flux<FLUX, T>(m, l, ur));
  return T(0.5) * f - T(0.5) * al * (ur - ul);
}

// Monolithic limiter of one direction at a cell: its averages before, at and after (um,
// u, up), their potentials, the high-order flux of its upper face and its high-order
// potential -> limited flux and potential. Theta is evaluated only when a high-order state
// leaves the bounds.
template <int FLUX, class T>
__device__ __forceinline__ void m3_limit(const DevModel& m, const M3Scal<T>& k, bool lim, int l, T um, T u, T up, T am,
                                         T a, T ap, T FH, T AH, T& Fl, T& Al) {
  Fl = FH;
  Al = AH;
  if (!lim) return;
  const T dA = AH - a, e = k.kd[l] * dA, dp = ap - a, dm = a - am, n6 = k.nu6[l];
  T zp = u, zm = up, p0 = um, q0 = u;
  T dF = T(0), FL = T(0);
  if constexpr (FLUX != FLUX_ZERO) {
    const T m6 = k.mu6[l];
    FL = m3_llf<FLUX, T>(m, l, u, up);
    const T FLm = m3_llf<FLUX, T>(m, l, um, u);
    zp = sfma(-m6, m3_minusf<FLUX, T>(m, l, FL, u), u);
    zm = sfma(-m6, m3_fminus<FLUX, T>(m, l, up, FL), up);
    p0 = sfma(-m6, m3_minusf<FLUX, T>(m, l, FLm, um), um);
    q0 = sfma(-m6, m3_fminus<FLUX, T>(m, l, u, FLm), u);
    dF = FH - FL;
  }
  zp = sfma(n6, dp, zp);
  zm = sfma(-n6, dp, zm);
  p0 = sfma(n6, dm, p0);
  q0 = sfma(-n6, dm, q0);
  const T h0 = p0 + e, h1 = zp - e, h2 = q0 - e, h3 = zm + e;
  T gp = zp, gm = zm;
  if constexpr (FLUX != FLUX_ZERO) {
    const T g = k.kc[l] * dF;
    gp = zp - g;
    gm = zm + g;
  }
  bool out;
  if constexpr (sizeof(T) == 8) {
    out = !(inb(h0, k.umin, k.umax) & inb(h1, k.umin, k.umax) & inb(h2, k.umin, k.umax) & inb(h3, k.umin, k.umax));
  } else {
    T lo = fmn(fmn(h0, h1), fmn(h2, h3)), hi = fmx(fmx(h0, h1), fmx(h2, h3));
    if constexpr (FLUX != FLUX_ZERO) {
      lo = fmn(lo, fmn(gp, gm));
      hi = fmx(hi, fmx(gp, gm));
    }
    out = tlt(lo, k.umin) | tlt(k.umax, hi);
  }
  if (out) {
    const T td = tmin(tmin(theta_fn<T>(p0, h0, k.umin, k.umax), theta_fn<T>(zp, h1, k.umin, k.umax)),
                      tmin(theta_fn<T>(q0, h2, k.umin, k.umax), theta_fn<T>(zm, h3, k.umin, k.umax)));
    Al = is_one(td) ? AH : sfma(td, dA, a);
    if constexpr (FLUX != FLUX_ZERO) {
      const T tc = tmin(theta_fn<T>(zp, gp, k.umin, k.umax), theta_fn<T>(zm, gm, k.umin, k.umax));
      Fl = is_one(tc) ? FH : sfma(tc, dF, FL);
    }
  }
}

// Shared memory: a layer's values by kind (read in its own step and in the next one, so
// three layers are kept) and, one step later, its centres' potentials and its y-limiter's
// results (two steps). With that one barrier per step is enough: a slot is written again
// only after a barrier that every reader of its last contents has passed.
template <int FLUX, class T, int TY>
struct M3Shared {
  static constexpr int NA = 7 + 1 + (FLUX == FLUX_ZERO ? 4 : 7);   // a of kinds 1 .. 7, U, z
  static constexpr int NB = FLUX == FLUX_ZERO ? 2 : 4;             // a(C), A_y limited [, C, F_y limited]
  T a[3][NA][TY][32];
  T b[2][NB][TY][32];
  M3Scal<T> sc;
  // slot of z of kind s
  static constexpr __device__ int zslot(int s) {
    return FLUX == FLUX_ZERO ? 8 + (s == 2 ? 0 : (s == 3 ? 1 : (s == 6 ? 2 : 3))) : 7 + s;
  }
};

template <int FLUX, int DIFF, class T, int TY>
__global__ void __launch_bounds__(32 * TY, 1)
    march3d_kernel(const DevModel m, const __grid_constant__ StageArgs3D<T> A, int o, int S, int bands, int rows) {
  using SH = M3Shared<FLUX, T, TY>;
  constexpr bool CONV = FLUX != FLUX_ZERO;
  static_assert(sizeof(T) == 4 || !CONV, "FP64 meshes with a flux take the four kernels (march3d_takes)");
  extern __shared__ __align__(16) unsigned char m3_raw[];
  SH& sh = *reinterpret_cast<SH*>(m3_raw);
  const double dtv = *A.dt;
  if (is_zero_bits(dtv)) return;   // uniform over the grid
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  if (row == 0) m3_scalars<T>(m, A, o, dtv, sh.sc);
  __syncthreads();
  const M3Scal<T>& k = sh.sc;
  const int n0 = A.n[0], n1 = A.n[1], n2 = A.n[2];
  const int bx = blockIdx.x % bands, by = (blockIdx.x / bands) % rows, bz = blockIdx.x / (bands * rows);
  const int xi = bx * M3_BAND - 2 + lane, yi = by * (TY - 4) - 2 + row;
  const int zs = bz * S, ze = min(zs + S, n2);
  const bool mid = row >= 1 && row < TY - 1;      // forms centres and the y-limiter
  const bool full = row >= 2 && row < TY - 2;     // forms everything
  const bool out = full && lane >= 2 && lane < 2 + M3_BAND && xi < n0 && yi < n1;
  // the FP64 ends of a step's averages, all at its end, would queue at the FP64 unit: half
  // of a scheduler's warps form theirs at its start (FP32-mixed porous medium 128^3, step
  // 570 -> 556 us; with a flux, fewer rows and more work between them, it cost registers)
  const bool early = sizeof(T) == 4 && !CONV && ((row >> 2) & 1);
  const bool lim = A.limiter != 0, comb = !is_zero_bits(A.cA[o]), sg = lim && A.sg[o];
  const unsigned plane = (unsigned)n0 * n1;
  const unsigned qxy = (unsigned)wrapi(yi, n1) * n0 + wrapi(xi, n0);
  const int rm = row > 0 ? row - 1 : 0, rp = row < TY - 1 ? row + 1 : row;   // rows read by `mid` rows only

  // layer values: kinds 0 (centre) .. 7 of layers r, r - 1, r - 2 (z of r - 2 only with a flux)
  T z[8], a[8], z1[8], a1[8], z2[8], a2[8], res1[8];
  T U = T(0), U1 = T(0), U2 = T(0), aU1 = T(0), aU2 = T(0);
  M3Level<T> lv;
  lv.clear();
  T AHz1 = T(0), FHz1 = T(0), Az2 = T(0), Az3 = T(0), Fz2 = T(0), Fz3 = T(0);
  Incr<T> inc1, inc2;   // x and y parts of layers r - 1, r - 2
  inc1.zero();
  inc2.zero();
#pragma unroll
  for (int s = 0; s < 8; ++s) z[s] = a[s] = z1[s] = a1[s] = z2[s] = a2[s] = res1[s] = T(0);

  int gz = wrapi(zs - 2, n2);
  unsigned q = (unsigned)gz * plane + qxy, q1 = 0, q2 = 0;
  double un = A.ub[q];
  T pn[8];
#pragma unroll
  for (int s = 1; s < 8; ++s) pn[s] = A.pt[s][q];

  T Ay1 = T(0), Fy1 = T(0);   // y-limiter of layer r - 1
  int ca = 0, pa = 0;           // slots of layers r and r - 1
#pragma unroll 1
  for (int r = zs - 2; r <= ze + 1; ++r) {
    const int par = r & 1;
    U = to_stencil<T>(un);
    const double uc = un;
    // of the last layer only the averages are read (in FP32 the test costs more than it saves)
    const bool pts = sizeof(T) == 4 || r <= ze;
#pragma unroll
    for (int s = 1; s < 8; ++s) {
      z[s] = pn[s];
      if (pts) a[s] = apot_k<DIFF, T>(m, z[s]);
    }
    const unsigned qc = q;
    // next layer
    gz = gz + 1 == n2 ? 0 : gz + 1;
    q = (unsigned)gz * plane + qxy;
    if (r < ze + 1) {
      un = A.ub[q];
#pragma unroll
      for (int s = 1; s < 8; ++s) pn[s] = A.pt[s][q];
    }
    // combination inputs of this step's outputs: points of layer r - 1, average of r - 2
    const bool outp = out && r - 1 >= zs && r - 1 < ze, outu = out && r - 2 >= zs && r - 2 < ze;
    T Ap[8];
    double ubj = 0.0, Aub = 0.0;
    if (outp && comb) {
#pragma unroll
      for (int s = 1; s < 8; ++s) Ap[s] = A.Apt[o][s][q1];
    }
    if (outu) {
      if constexpr (sizeof(T) == 8) ubj = A.ub[q2];
      if (comb) Aub = A.Aub[o][q2];
    }
    pa = ca;
    ca = ca == 2 ? 0 : ca + 1;
#pragma unroll
    for (int s = 1; s < 8; ++s) sh.a[ca][s - 1][row][lane] = a[s];
    sh.a[ca][7][row][lane] = U;
    if (mid) {   // layer r - 1
      sh.b[par][0][row][lane] = a1[0];
      sh.b[par][1][row][lane] = Ay1;
      if constexpr (CONV) {
        sh.b[par][2][row][lane] = z1[0];
        sh.b[par][3][row][lane] = Fy1;
      }
    }
    if constexpr (CONV) {
#pragma unroll
      for (int s = 1; s < 8; ++s) sh.a[ca][SH::zslot(s)][row][lane] = z[s];
    } else {
      sh.a[ca][SH::zslot(2)][row][lane] = z[2];
      sh.a[ca][SH::zslot(3)][row][lane] = z[3];
      sh.a[ca][SH::zslot(6)][row][lane] = z[6];
      sh.a[ca][SH::zslot(7)][row][lane] = z[7];
    }
    __syncthreads();
    const T aU = apot_k<DIFF, T>(m, U);
    // ---- z-limiter of cell r - 1, averages of layer r - 2
    T Fz1 = T(0), Az1 = T(0);
    auto finish = [&]() {
      m3_limit<FLUX, T>(m, k, lim, 2, U2, U1, U, aU2, aU1, aU, FHz1, AHz1, Fz1, Az1);
      if (outu) {
        Incr<T> w = inc2;
        if constexpr (CONV) w.conv(k, 2, Fz2, Fz3);
        w.diff(k, 2, Az1, Az2, Az3);
        const double v = sizeof(T) == 8 ? ubj + w.v : w.v;
        double ubo = comb ? rk_comb(A.cA[o], Aub, A.cF[o], v) : rk_scale(A.cF[o], v);
        if (sg) ubo = safeguard<double>(ubo, m.umin, m.umax, A.tol, A.stats, true);
        A.Oub[o][q2] = ubo;
      }
    };
    if (full && early) finish();
    const bool xy = r >= zs && r < ze;   // x- and y-directions of layer r are needed
    T AHx = T(0), AHz = T(0), FHx = T(0), FHz = T(0), Fy = T(0), Ay = T(0);
    T am2, am3, am6, am7, zm2, zm3, zm6, zm7;   // row below
    const T a1x = shup(a[1]), a3x = shup(a[3]), a5x = shup(a[5]), a7x = shup(a[7]);   // column before
    if (mid && pts) {
      am2 = sh.a[ca][1][rm][lane];
      am3 = sh.a[ca][2][rm][lane];
      am6 = sh.a[ca][5][rm][lane];
      am7 = sh.a[ca][6][rm][lane];
      zm2 = sh.a[ca][SH::zslot(2)][rm][lane];
      zm3 = sh.a[ca][SH::zslot(3)][rm][lane];
      zm6 = sh.a[ca][SH::zslot(6)][rm][lane];
      zm7 = sh.a[ca][SH::zslot(7)][rm][lane];
      T AHy = T(0), FHy = T(0);
      if constexpr (sizeof(T) == 4) {
        // the layer's plane of centres (kinds 0 .. 3) and its upper plane of z-faces (4 .. 7)
        // as 3 x 3 locations around the cell, index 3 (my + 1) + mx + 1
        const T z1x = shup(z[1]), z3x = shup(z[3]), z5x = shup(z[5]), z7x = shup(z[7]);
        const T zc[9] = {shup(zm3), zm2, zm3, z1x, T(0), z[1], z3x, z[2], z[3]};
        const T zu[9] = {shup(zm7), zm6, zm7, z5x, z[4], z[5], z7x, z[6], z[7]};
        T acc = lv.cz;
#pragma unroll
        for (int q9 = 0; q9 < 9; ++q9)
          if (q9 != 4) acc = sfma(m3_w(q9) * T(4), zc[q9], acc);
        T up = T(0);
#pragma unroll
        for (int q9 = 0; q9 < 9; ++q9) {
          acc = sfma(m3_w(q9), zu[q9], acc);
          up = sfma(m3_w(q9), zu[q9], up);
        }
        lv.cz = up;
        z[0] = sfma(T(216), U, -acc) * T(1.0 / 64.0);
        a[0] = apot_k<DIFF, T>(m, z[0]);
        const T ac[9] = {shup(am3), am2, am3, a1x, a[0], a[1], a3x, a[2], a[3]};
        const T au[9] = {shup(am7), am6, am7, a5x, a[4], a[5], a7x, a[6], a[7]};
        // s + w (-lo + 8 mid - hi) / 6
        auto hat = [](T w, T lo, T md, T hi, T s) {
          return sfma(w, (sfma(T(8), md, -lo) - hi) * T(1.0 / 6.0), s);
        };
        T sx = lv.ax, sy = lv.ay, sz = T(0), ux = T(0), uy = T(0);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const T w = e == 1 ? T(4) : T(1);
          sx = hat(w * T(4), ac[3 * e], ac[3 * e + 1], ac[3 * e + 2], sx);
          sy = hat(w * T(4), ac[e], ac[3 + e], ac[6 + e], sy);
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const T w = e == 1 ? T(4) : T(1);
          sx = hat(w, au[3 * e], au[3 * e + 1], au[3 * e + 2], sx);
          sy = hat(w, au[e], au[3 + e], au[6 + e], sy);
          ux = hat(w, au[3 * e], au[3 * e + 1], au[3 * e + 2], ux);
          uy = hat(w, au[e], au[3 + e], au[6 + e], uy);
        }
#pragma unroll
        for (int q9 = 0; q9 < 9; ++q9) {
          sz = hat(m3_w(q9), lv.a[q9], ac[q9], au[q9], sz);
          lv.a[q9] = au[q9];
        }
        lv.ax = ux;
        lv.ay = uy;
        AHx = sx * T(1.0 / 36.0);
        AHy = sy * T(1.0 / 36.0);
        AHz = sz * T(1.0 / 36.0);
        if constexpr (CONV) {
          // Simpson averages of f_l over the upper faces
          const T r36 = T(1.0 / 36.0);
          const T fx1 = lv.fx, fy1 = lv.fy;
          T fx = T(0), fy = T(0), fz = T(0);
          // lower-plane terms of the next layer's x- and y-faces: mx (my) = +1
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const T w = e == 1 ? T(4) : T(1);
            fx = sfma(w, flux<FLUX, T>(m, 0, zu[3 * e + 2]), fx);
            fy = sfma(w, flux<FLUX, T>(m, 1, zu[6 + e]), fy);
          }
          lv.fx = fx;
          lv.fy = fy;
          fx = fx1;
          fy = fy1;
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const T w = e == 1 ? T(16) : T(4);
            fx = sfma(w, flux<FLUX, T>(m, 0, zc[3 * e + 2]), fx);
            fy = sfma(w, flux<FLUX, T>(m, 1, zc[6 + e]), fy);
          }
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const T w = e == 1 ? T(4) : T(1);
            fx = sfma(w, flux<FLUX, T>(m, 0, zu[3 * e + 2]), fx);
            fy = sfma(w, flux<FLUX, T>(m, 1, zu[6 + e]), fy);
          }
#pragma unroll
          for (int q9 = 0; q9 < 9; ++q9) fz = sfma(m3_w(q9), flux<FLUX, T>(m, 2, zu[q9]), fz);
          FHx = fx * r36;
          FHy = fy * r36;
          FHz = fz * r36;
        }
      } else {
        // sums over the cell's locations, axis by axis: of z for the centre ...
        const T y3 = zm3 + z[3], y7 = zm7 + z[7];
        const T e1 = shup(z[1]) + z[1], e2 = zm2 + z[2], e3 = shup(y3) + y3;
        const T e5 = shup(z[5]) + z[5], e6 = zm6 + z[6], e7 = shup(y7) + y7;
        const T fsum = e1 + e2 + (lv.z[0] + z[4]), esum = e3 + (lv.z[1] + e5) + (lv.z[2] + e6);
        const bool whole = r > zs - 2;   // the first layer only leaves its upper plane
        if (whole) {
          z[0] = sfma(T(216), U, -sfma(T(16), fsum, sfma(T(4), esum, lv.z[3] + e7))) * T(1.0 / 64.0);
          a[0] = apot_k<DIFF, T>(m, z[0]);
        }
        lv.z[0] = z[4];
        lv.z[1] = e5;
        lv.z[2] = e6;
        lv.z[3] = e7;
        // ... and of a for the potentials
        const T v3 = am3 + a[3], v7 = am7 + a[7];
        const T b1 = a1x + a[1], b2 = am2 + a[2], b3 = shup(v3) + v3;
        const T b5 = a5x + a[5], b6 = am6 + a[6], b7 = shup(v7) + v7;
        const T Fz = lv.a[0] + a[4], Exz = lv.a[1] + b5, Eyz = lv.a[2] + b6, V = lv.a[3] + b7;
        lv.a[0] = a[4];
        lv.a[1] = b5;
        lv.a[2] = b6;
        lv.a[3] = b7;
        if (whole) {
          const T r216 = T(1.0 / 216.0);
          AHx = sfma(T(8), sfma(T(16), a[0], sfma(T(4), b2 + Fz, Eyz)), -sfma(T(16), b1, sfma(T(4), b3 + Exz, V))) * r216;
          AHy = sfma(T(8), sfma(T(16), a[0], sfma(T(4), b1 + Fz, Exz)), -sfma(T(16), b2, sfma(T(4), b3 + Eyz, V))) * r216;
          AHz = sfma(T(8), sfma(T(16), a[0], sfma(T(4), b1 + b2, b3)), -sfma(T(16), Fz, sfma(T(4), Exz + Eyz, V))) * r216;
        }
      }
      if (xy) {
        const T um = sh.a[ca][7][rm][lane], up = sh.a[ca][7][rp][lane];
        m3_limit<FLUX, T>(m, k, lim, 1, um, U, up, apot_k<DIFF, T>(m, um), aU, apot_k<DIFF, T>(m, up), FHy, AHy, Fy, Ay);
      }
    }
    if (full) {
      T res[8];
      Incr<T> inc;
      inc.zero();
      if constexpr (sizeof(T) == 4) inc.v = uc;   // the average itself, its terms added in turn
      if (xy) {
        // ---- averages: x part of layer r
        {
          const T um = shup(U), up = shdn(U);
          T Fx, Ax;
          m3_limit<FLUX, T>(m, k, lim, 0, um, U, up, apot_k<DIFF, T>(m, um), aU, apot_k<DIFF, T>(m, up), FHx, AHx, Fx, Ax);
          if constexpr (CONV) inc.conv(k, 0, Fx, shup(Fx));
          inc.diff(k, 0, shdn(Ax), Ax, shup(Ax));
        }
        // ---- points: x-lines, kinds t and t + 1
#pragma unroll
        for (int t = 0; t < 8; t += 2) {
          const T A1m = t == 0 ? a1x : (t == 2 ? a3x : (t == 4 ? a5x : a7x)), A1p = shdn(a[t + 1]), A0p = shdn(a[t]);
          T Z1m = T(0), Z1p = T(0), Z0p = T(0), Z0m = T(0);
          if constexpr (CONV) {
            Z1m = shup(z[t + 1]);
            Z1p = shdn(z[t + 1]);
            Z0p = shdn(z[t]);
          }
          res[t + 1] = m3_line<FLUX, T>(m, A, 0, Z1m, z[t], z[t + 1], Z0p, Z1p, A1m, a[t], a[t + 1], A0p, A1p, T(0));
          if (t > 0) {
            const T A0m = shup(a[t]);
            if constexpr (CONV) Z0m = shup(z[t]);
            res[t] = m3_line<FLUX, T>(m, A, 0, Z0m, Z1m, z[t], z[t + 1], Z0p, A0m, A1m, a[t], a[t + 1], A0p, T(0));
          }
        }
      }
      // ---- layer r - 1: y part of its averages, y- and z-lines; its points are finished
      if (r - 1 >= zs && r - 1 < ze) {
        if constexpr (CONV) inc1.conv(k, 1, Fy1, sh.b[par][3][rm][lane]);
        inc1.diff(k, 1, sh.b[par][1][rp][lane], Ay1, sh.b[par][1][rm][lane]);
        // y-lines, kinds t and t + 2
#pragma unroll
        for (int tt = 0; tt < 4; ++tt) {
          const int t = (tt & 1) + 4 * (tt >> 1);
          auto ya = [&](int s, int rr) { return s == 0 ? sh.b[par][0][rr][lane] : sh.a[pa][s - 1][rr][lane]; };
          auto yz = [&](int s, int rr) {
            if constexpr (CONV) return s == 0 ? sh.b[par][2][rr][lane] : sh.a[pa][SH::zslot(s == 0 ? 1 : s)][rr][lane];
            else return T(0);
          };
          const T A1m = ya(t + 2, rm), A1p = ya(t + 2, rp), A0p = ya(t, rp);
          const T Z1m = yz(t + 2, rm), Z1p = yz(t + 2, rp), Z0p = yz(t, rp);
          res1[t + 2] = m3_line<FLUX, T>(m, A, 1, Z1m, z1[t], z1[t + 2], Z0p, Z1p, A1m, a1[t], a1[t + 2], A0p, A1p,
                                         res1[t + 2]);
          if (t > 0)
            res1[t] = m3_line<FLUX, T>(m, A, 1, yz(t, rm), Z1m, z1[t], z1[t + 2], Z0p, ya(t, rm), A1m, a1[t],
                                       a1[t + 2], A0p, res1[t]);
        }
        T po[8];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const T l1 = m3_line<FLUX, T>(m, A, 2, z2[t + 4], z1[t], z1[t + 4], z[t], z[t + 4], a2[t + 4], a1[t],
                                        a1[t + 4], a[t], a[t + 4], res1[t + 4]);
          po[t + 4] = rk_fma(k.taut, m3_middle<FLUX, T>(k, a1[t + 4], l1), z1[t + 4]);
          if (t > 0) {
            const T l0 = m3_line<FLUX, T>(m, A, 2, z2[t], z2[t + 4], z1[t], z1[t + 4], z[t], a2[t], a2[t + 4], a1[t],
                                          a1[t + 4], a[t], res1[t]);
            po[t] = rk_fma(k.taut, m3_middle<FLUX, T>(k, a1[t], l0), z1[t]);
          }
        }
        if (outp) {
          T lo = k.umax, hi = k.umin;
#pragma unroll
          for (int s = 1; s < 8; ++s) {
            if (lim) po[s] = tmin(tmax(po[s], k.umin), k.umax);
            po[s] = comb ? rk_comb(k.cAt, Ap[s], k.cFt, po[s]) : rk_scale(k.cFt, po[s]);
            if constexpr (sizeof(T) == 4) {
              lo = fmn(lo, po[s]);
              hi = fmx(hi, po[s]);
            }
          }
          // post-stage safeguard: in FP32 one test for the seven values
          if (sg && (sizeof(T) == 8 || lo < k.umin || hi > k.umax)) {
#pragma unroll
            for (int s = 1; s < 8; ++s) po[s] = safeguard<T>(po[s], k.umin, k.umax, A.tol, A.stats);
          }
#pragma unroll
          for (int s = 1; s < 8; ++s) A.Opt[o][s][q1] = po[s];
        }
      }
      if (!early) finish();
      Fz3 = Fz2;
      Fz2 = Fz1;
      Az3 = Az2;
      Az2 = Az1;
      inc2 = inc1;
      inc1 = inc;
      AHz1 = AHz;
      FHz1 = FHz;
#pragma unroll
      for (int s = 1; s < 8; ++s) res1[s] = xy ? res[s] : T(0);
#pragma unroll
      for (int s = 1; s < 8; ++s) {
        a2[s] = a1[s];
        a1[s] = a[s];
        z2[s] = z1[s];
        z1[s] = z[s];
      }
    }
    a1[0] = a[0];
    z1[0] = z[0];
    Ay1 = Ay;
    Fy1 = Fy;
    U2 = U1;
    U1 = U;
    aU2 = aU1;
    aU1 = aU;
    q2 = q1;
    q1 = qc;
  }
}

// ---- launch (host)

template <int FLUX, int DIFF, class T, int TY>
static cudaError_t march3d_rows(const DevModel& m, const StageArgs3D<T>& a, const M3Plan& p, cudaStream_t s) {
  const long long blocks = (long long)p.bands * p.rows * ((a.n[2] + p.S - 1) / p.S);
  if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
  auto kern = march3d_kernel<FLUX, DIFF, T, TY>;
  const int smem = (int)sizeof(M3Shared<FLUX, T, TY>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  for (int o = 0; o < a.nout; ++o) {
    kern<<<(unsigned)blocks, 32 * TY, smem, s>>>(m, a, o, p.S, p.bands, p.rows);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int FLUX, int DIFF, class T>
static cudaError_t march3d_go(const DevModel& m, const StageArgs3D<T>& a, cudaStream_t s) {
  constexpr int TY = m3_rows(FLUX, sizeof(T) == 8);
  const M3Plan p = m3_plan(a.n, TY);
  if constexpr (TY > M3_ROWS_SMALL) {
    const M3Plan q = m3_plan(a.n, M3_ROWS_SMALL);
    if (q.cost < p.cost) return march3d_rows<FLUX, DIFF, T, M3_ROWS_SMALL>(m, a, q, s);
  }
  return march3d_rows<FLUX, DIFF, T, TY>(m, a, p, s);
}

template <int FLUX, class T>
static cudaError_t march3d_diff(const DevModel& m, const StageArgs3D<T>& a, cudaStream_t s) {
  if (m.diff_kind == AF_DIFF_CONST) return march3d_go<FLUX, DK_CONST, T>(m, a, s);
  if (m.diff_kind == AF_DIFF_PME && m.pme_e == 2) return march3d_go<FLUX, DK_PME2, T>(m, a, s);
  return march3d_go<FLUX, DK_GENERIC, T>(m, a, s);
}

}  // namespace af
