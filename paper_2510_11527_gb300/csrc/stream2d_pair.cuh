// Column-marching 2D stage of pure diffusion (zero flux), two columns per lane: the march of
// stream2d.cuh without the blend (same quantities, same order, same roundings) with the FP32
// stencil arithmetic in packed pairs.
//
// The one-column march is bound by instruction issue (about 560 instructions per lane and
// row). Blackwell adds, multiplies and fuses two FP32 values per instruction, so a lane
// that holds two neighbouring columns forms both columns' stencils at the issue cost of one
// (the multiply-add rate is the same; only issue slots are saved), a neighbour value costs
// one shuffle per two columns, and the halo is 4 of 64 columns instead of 4 of 32. The
// price is registers: 12 warps per SM at 163 instead of 16 at 128. With a flux the form
// needs 231 registers, 8 warps per SM hide too little (46 % of the issue slots used), and
// degenerate Burgers at 2048^2 ran at the one-column kernel's speed (both 0.44 ms per step),
// so only the zero flux takes it: porous medium 2048^2 0.38 -> 0.30 ms, 4096^2 1.23 -> 0.87
// ms per step at each one's best strips.
//
// A packed operation rounds each half as the scalar one does. Where the scalar code
// negates an operand the packed one uses the mirrored form -(a b - c) = (-a) b + c with
// coefficients negated once (rounding to nearest is symmetric), so results differ at most
// in the sign of a zero. The convection terms, exact zeros, are not formed (of an unlimited
// state that has overflowed FP32 they make some infinities NaN).
#pragma once
#include "stream2d.cuh"

namespace af {

constexpr int PAIR_BAND = 60;   // output columns per warp
constexpr int PAIR_WPB = 4;     // warps per block

struct F2 {
  float x, y;
};
__device__ __forceinline__ float2 raw2(F2 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ F2 f2(float2 a) { return F2{a.x, a.y}; }
__device__ __forceinline__ F2 dup(float a) { return F2{a, a}; }
// Packed arithmetic. A product is formed as fma(a, b, Z) with a zero Z that the compiler
// cannot see (PairScal::zero): it fuses a packed product and a following packed sum into one
// rounding otherwise, whatever the contraction flag and the rounding modifiers say.
__device__ __forceinline__ unsigned long long bits2(F2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ F2 of_bits2(unsigned long long r) {
  F2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(bits2(a)), "l"(bits2(b)));
  return of_bits2(r);
}
__device__ __forceinline__ F2 sfma(F2 a, F2 b, F2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(bits2(a)), "l"(bits2(b)), "l"(bits2(c)));
  return of_bits2(r);
}
// a - b (one rounding: the product with -1 is exact)
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return sfma(b, dup(-1.0f), a); }
__device__ __forceinline__ F2 mul(F2 a, F2 b, F2 Z) { return sfma(a, b, Z); }
__device__ __forceinline__ F2 fmx(F2 a, F2 b) { return F2{fmaxf(a.x, b.x), fmaxf(a.y, b.y)}; }
__device__ __forceinline__ F2 fmn(F2 a, F2 b) { return F2{fminf(a.x, b.x), fminf(a.y, b.y)}; }
__device__ __forceinline__ F2 tabs(F2 a) { return F2{fabsf(a.x), fabsf(a.y)}; }
// the columns before / after
__device__ __forceinline__ F2 xm(F2 a) { return F2{shup(a.y), a.x}; }
__device__ __forceinline__ F2 xp(F2 a) { return F2{a.y, shdn(a.x)}; }

// per-warp constants of one launch (a value used by packed arithmetic twice)
struct PairScal {
  F2 n4_1, nn4_1, n4_2, nn4_2;                 // 4 nu_l, -4 nu_l
  F2 q1, q2, n1, n2;                           // 12 nu_l, nu_l
  F2 ni3h21, ni3h22;                           // -1 / (3 h_l^2)
  F2 taut, cAt, cFt;
  float umin, umax, zero;
  double cA, cF, umid;
};

// values of one input row that later steps read (see RowSlot)
struct PairSlot {
  F2 V, X, Y, U;
  F2 aV, aX, aY, aC, aU;
  F2 Vm, aVm;
  F2 AH2;
  F2 rV, rX, rY;
  F2 ULp2, ULm2, Alim2;
  F2 tD2lo, tD1;
};

struct PairIn {
  double ub0, ub1;
  F2 V, X, Y;
};

template <int DIFF>
__device__ __forceinline__ F2 apot2(const DevModel& m, F2 u, F2 Z) {
  if constexpr (DIFF == DK_NONE) {
    return dup(0.0f);
  } else if constexpr (DIFF == DK_CONST) {
    return mul(dup(m.dpf[0]), u, Z);
  } else if constexpr (DIFF == DK_PWL) {
    return mul(dup(m.dpf[0]), fmn(u - dup(m.dpf[1]), dup(0.0f)), Z) +
           mul(dup(m.dpf[2]), fmx(u - dup(m.dpf[3]), dup(0.0f)), Z);
  } else if constexpr (DIFF == DK_PME2) {
    return mul(u, u, Z);
  } else if constexpr (DIFF == DK_CUBIC) {
    return mul(mul(mul(dup(m.dpf[2]), u, Z) + dup(m.dpf[1]), u, Z) + dup(m.dpf[0]), u, Z);
  } else {
    return F2{apot<float>(m, u.x), apot<float>(m, u.y)};
  }
}

// diffusion part of line_res_s: (-da) (-1/(3h^2))
__device__ __forceinline__ F2 line2(F2 a0, F2 a1, F2 a2, F2 a3, F2 a4, F2 ni3h2, F2 Z) {
  return mul(sfma(dup(30.0f), a2, sfma(dup(-16.0f), a1 + a3, a0 + a4)), ni3h2, Z);
}

// cell_pot: (8 a - 4 b + 32 ac - sv) / 36
__device__ __forceinline__ F2 cell_pot2(F2 sv, F2 a, F2 b, F2 ac, F2 Z) {
  return mul(sfma(dup(-32.0f), ac, sfma(dup(-8.0f), a, sfma(dup(4.0f), b, sv))), dup(-(float)(1.0 / 36.0)), Z);
}

// s + err = a - b exactly (two_sum with b negated)
__device__ __forceinline__ void two_diff2(F2 a, F2 b, F2& s, F2& err) {
  const F2 r = a - b, bb = r - a;
  err = (a - (r - bb)) - (b + bb);
  s = r;
}
__device__ __forceinline__ void two_sum2(F2 a, F2 b, F2& s, F2& err) {
  const F2 r = a + b, bb = r - a;
  err = (a - (r - bb)) + (b - bb);
  s = r;
}

struct PairCtx {
  int nx, ny, g0, g1, rs, re;
  bool out0, out1;   // this lane's columns produce outputs
  bool vec;          // even mesh width: the columns are one aligned pair in memory
  bool comb;
};

template <int DIFF>
__device__ __forceinline__ void pair_step(const DevModel& m, const StageArgs2D<float>& A, const PairScal& k,
                                          const PairCtx& c, F2 Z, int r, const PairIn& in, PairSlot& p2, PairSlot& p1,
                                          PairSlot& cur) {
  const bool lim = A.limiter != 0;

  // ---- combination inputs of the cells finalised in this step (row r - 2)
  const int j = r - 2;
  const bool outr = j >= c.rs && j < c.re && c.out0;
  double ub0 = 0.0, ub1 = 0.0, Au0 = 0.0, Au1 = 0.0;
  F2 AV = dup(0.0f), AX = AV, AY = AV;
  if (outr) {
    const size_t go = (size_t)j * c.nx + c.g0;
    if (c.vec) {
      const double2 u = __ldg(reinterpret_cast<const double2*>(A.ub + go));
      ub0 = u.x;
      ub1 = u.y;
      if (c.comb) {
        const double2 a = *reinterpret_cast<const double2*>(A.Aub[0] + go);
        Au0 = a.x;
        Au1 = a.y;
        AV = f2(__ldg(reinterpret_cast<const float2*>(A.AV[0] + go)));
        AX = f2(__ldg(reinterpret_cast<const float2*>(A.AX[0] + go)));
        AY = f2(__ldg(reinterpret_cast<const float2*>(A.AY[0] + go)));
      }
    } else {
      const size_t g1 = (size_t)j * c.nx + c.g1;
      ub0 = __ldg(A.ub + go);
      ub1 = __ldg(A.ub + g1);
      if (c.comb) {
        Au0 = A.Aub[0][go];
        Au1 = A.Aub[0][g1];
        AV = F2{__ldg(A.AV[0] + go), __ldg(A.AV[0] + g1)};
        AX = F2{__ldg(A.AX[0] + go), __ldg(A.AX[0] + g1)};
        AY = F2{__ldg(A.AY[0] + go), __ldg(A.AY[0] + g1)};
      }
    }
  }

  // ---- row r: points, centre, pointwise functions
  cur.U = F2{to_stencil_nb<float>(in.ub0, k.umid), to_stencil_nb<float>(in.ub1, k.umid)};
  cur.V = in.V;
  cur.X = in.X;
  cur.Y = in.Y;
  cur.Vm = xm(cur.V);
  const F2 C = mul(sfma(dup(-36.0f), cur.U,
                        sfma(dup(4.0f), (xm(cur.X) + cur.X) + (p1.Y + cur.Y), (p1.Vm + p1.V) + (cur.Vm + cur.V))),
                   dup(-0.0625f), Z);
  cur.aV = apot2<DIFF>(m, cur.V, Z);
  cur.aX = apot2<DIFF>(m, cur.X, Z);
  cur.aY = apot2<DIFF>(m, cur.Y, Z);
  cur.aC = apot2<DIFF>(m, C, Z);
  cur.aU = apot2<DIFF>(m, cur.U, Z);

  // ---- cell potentials of row r
  cur.aVm = xm(cur.aV);
  const F2 aXm = xm(cur.aX);
  F2 AH1;
  {
    const F2 sv = (p1.aVm + p1.aV) + (cur.aVm + cur.aV), sx = aXm + cur.aX, sy = p1.aY + cur.aY;
    cur.AH2 = cell_pot2(sv, sx, sy, cur.aC, Z);
    AH1 = cell_pot2(sv, sy, sx, cur.aC, Z);
  }

  // ---- point residuals: x-lines of row r
  {
    const F2 aYp = xp(cur.aY);
    cur.rV = line2(cur.aVm, cur.aY, cur.aV, aYp, xp(cur.aV), k.ni3h21, Z);
    cur.rX = line2(aXm, cur.aC, cur.aX, xp(cur.aC), xp(cur.aX), k.ni3h21, Z);
    cur.rY = line2(xm(cur.aY), cur.aVm, cur.aY, cur.aV, aYp, k.ni3h21, Z);
  }
  // y-lines of row r-1, added to its x-lines
  p1.rV = p1.rV + line2(p2.aV, p1.aX, p1.aV, cur.aX, cur.aV, k.ni3h22, Z);
  p1.rX = p1.rX + line2(p2.aX, p2.aV, p1.aX, p1.aV, cur.aX, k.ni3h22, Z);
  p1.rY = p1.rY + line2(p2.aY, p1.aC, p1.aY, cur.aC, cur.aY, k.ni3h22, Z);

  // ---- limiter: x-direction of row r, y-direction of row r-1 (the low-order states; the
  // face limiters' high-order states are the low-order ones)
  F2 Alim1 = AH1;
  p1.Alim2 = p1.AH2;
  if (lim) {
    const F2 ULp1 = sfma(k.n4_1, xp(cur.aU) - cur.aU, cur.U), ULm1 = sfma(k.nn4_1, cur.aU - xm(cur.aU), cur.U);
    const F2 dU2 = cur.aU - p1.aU;
    p1.ULp2 = sfma(k.n4_2, dU2, p1.U);
    cur.ULm2 = sfma(k.nn4_2, dU2, cur.U);
    // the neighbours' states are the ones they form themselves
    const F2 ULm1p = xp(ULm1), ULp1m = xm(ULp1);
    const F2 dA1 = AH1 - cur.aU, e1 = mul(k.q1, dA1, Z);
    const F2 dA2 = p1.AH2 - p1.aU, e2 = mul(k.q2, dA2, Z);
    const F2 zl[8] = {ULp1m, ULp1, ULm1, ULm1p, p2.ULp2, p1.ULp2, p1.ULm2, cur.ULm2};
    const F2 zh[8] = {ULp1m + e1, ULp1 - e1, ULm1 - e1, ULm1p + e1, p2.ULp2 + e2, p1.ULp2 - e2, p1.ULm2 - e2, cur.ULm2 + e2};
    float lo = fminf(zh[0].x, zh[0].y), hi = fmaxf(zh[0].x, zh[0].y);
#pragma unroll
    for (int q = 1; q < 8; ++q) {
      lo = min3(lo, zh[q].x, zh[q].y);
      hi = max3(hi, zh[q].x, zh[q].y);
    }
    if ((lo < k.umin) | (k.umax < hi)) {
      auto one = [&](auto&& get, float AH, float dA, float aU, int q) {
        auto th = [&](int i) { return theta_fn<float>(get(zl[i]), get(zh[i]), k.umin, k.umax); };
        const float td = tmin(tmin(th(q), th(q + 1)), tmin(th(q + 2), th(q + 3)));
        return is_one(td) ? AH : sfma(td, dA, aU);
      };
      auto gx = [](F2 v) { return v.x; };
      auto gy = [](F2 v) { return v.y; };
      Alim1 = F2{one(gx, AH1.x, dA1.x, cur.aU.x, 0), one(gy, AH1.y, dA1.y, cur.aU.y, 0)};
      p1.Alim2 = F2{one(gx, p1.AH2.x, dA2.x, p1.aU.x, 4), one(gy, p1.AH2.y, dA2.y, p1.aU.y, 4)};
    }
  }
  // update terms (see stream_step)
  cur.tD1 = mul(k.n1, xp(Alim1) - Alim1, Z);
  p1.tD2lo = mul(k.n2, p1.Alim2 - p2.Alim2, Z);

  // ---- finalise the cells of row j = r - 2
  const F2 tD1m = xm(p2.tD1);
  if (outr) {
    F2 hs, ls, e;
    two_diff2(p2.tD1, tD1m, hs, ls);
    two_sum2(hs, p1.tD2lo, hs, e);
    ls = ls + e;
    two_diff2(hs, p2.tD2lo, hs, e);
    ls = ls + e;
    const double fe0 = ub0 + (f2d_exact(hs.x) + f2d_exact(ls.x));
    const double fe1 = ub1 + (f2d_exact(hs.y) + f2d_exact(ls.y));
    F2 v = sfma(k.taut, p2.rV, p2.V), x = sfma(k.taut, p2.rX, p2.X), y = sfma(k.taut, p2.rY, p2.Y);
    if (lim) {
      const F2 lo2 = dup(k.umin), hi2 = dup(k.umax);
      v = fmn(fmx(v, lo2), hi2);
      x = fmn(fmx(x, lo2), hi2);
      y = fmn(fmx(y, lo2), hi2);
    }
    double o0, o1;
    if (c.comb) {
      o0 = rk_comb(k.cA, Au0, k.cF, fe0);
      o1 = rk_comb(k.cA, Au1, k.cF, fe1);
      v = sfma(k.cAt, AV, mul(k.cFt, v, Z));
      x = sfma(k.cAt, AX, mul(k.cFt, x, Z));
      y = sfma(k.cAt, AY, mul(k.cFt, y, Z));
    } else {
      o0 = rk_scale(k.cF, fe0);
      o1 = rk_scale(k.cF, fe1);
      v = mul(k.cFt, v, Z);
      x = mul(k.cFt, x, Z);
      y = mul(k.cFt, y, Z);
    }
    // post-stage safeguard: one test for the eight values, the clamp path only if needed
    if (lim && A.sg[0]) {
      const F2 l3 = fmn(fmn(v, x), y), h3 = fmx(fmx(v, x), y);
      if (tlt(o0, m.umin) | tlt(m.umax, o0) | tlt(o1, m.umin) | tlt(m.umax, o1) | (fminf(l3.x, l3.y) < k.umin) |
          (fmaxf(h3.x, h3.y) > k.umax)) {
        o0 = safeguard<double>(o0, m.umin, m.umax, A.tol, A.stats, true);
        v.x = safeguard<float>(v.x, k.umin, k.umax, A.tol, A.stats);
        x.x = safeguard<float>(x.x, k.umin, k.umax, A.tol, A.stats);
        y.x = safeguard<float>(y.x, k.umin, k.umax, A.tol, A.stats);
        if (c.out1) {
          o1 = safeguard<double>(o1, m.umin, m.umax, A.tol, A.stats, true);
          v.y = safeguard<float>(v.y, k.umin, k.umax, A.tol, A.stats);
          x.y = safeguard<float>(x.y, k.umin, k.umax, A.tol, A.stats);
          y.y = safeguard<float>(y.y, k.umin, k.umax, A.tol, A.stats);
        }
      }
    }
    const size_t g = (size_t)j * c.nx + c.g0;
    if (c.vec) {
      *reinterpret_cast<double2*>(A.Oub[0] + g) = make_double2(o0, o1);
      *reinterpret_cast<float2*>(A.OV[0] + g) = raw2(v);
      *reinterpret_cast<float2*>(A.OX[0] + g) = raw2(x);
      *reinterpret_cast<float2*>(A.OY[0] + g) = raw2(y);
    } else {
      A.Oub[0][g] = o0;
      A.OV[0][g] = v.x;
      A.OX[0][g] = x.x;
      A.OY[0][g] = y.x;
      if (c.out1) {
        A.Oub[0][g + 1] = o1;
        A.OV[0][g + 1] = v.y;
        A.OX[0][g + 1] = x.y;
        A.OY[0][g + 1] = y.y;
      }
    }
  }
}

// One warp's march over its band of 60 columns and strip of S rows (all 32 lanes).
template <int DIFF>
__device__ __forceinline__ void pair_run(const DevModel& m, const StageArgs2D<float>& A, int S, int band, int strip) {
  const double dtv = *A.dt;
  if (is_zero_bits(dtv)) return;   // uniform over the mesh
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int nx = A.nx, ny = A.ny;
  const int rs = strip * S;
  if (rs >= ny) return;   // whole warp
  __shared__ PairScal skw[PAIR_WPB];
  {
    // the lanes form one scalar each at once (see stream_run): lane l rounds
    // fl(fl(fl(x y1) y2) y3) to FP32
    const double tau = A.tcoef[0] * dtv;
    const double ih = (lane & 1) ? A.inv_h2 : A.inv_h1;
    double x = tau, y1 = ih, y2 = 1.0, y3 = 1.0;
    if (lane < 6) {
      const int kind = lane >> 1;   // 4 nu, 12 nu, nu
      y2 = ih;
      y3 = kind == 0 ? 4.0 : (kind == 1 ? 12.0 : 1.0);
    } else {
      // 12 .. 17: tau, u_min, u_max, cA, cF, 0 tau
      x = lane == 13 ? m.umin : (lane == 14 ? m.umax : (lane == 15 ? A.cA[0] : (lane == 16 ? A.cF[0] : tau)));
      y1 = lane == 17 ? 0.0 : 1.0;
    }
    const float v = (float)(((x * y1) * y2) * y3);
    auto at = [&](int l) { return __shfl_sync(0xffffffffu, v, l); };
    PairScal k;
    k.n4_1 = dup(at(0));
    k.n4_2 = dup(at(1));
    k.nn4_1 = dup(-at(0));
    k.nn4_2 = dup(-at(1));
    k.q1 = dup(at(2));
    k.q2 = dup(at(3));
    k.n1 = dup(at(4));
    k.n2 = dup(at(5));
    k.taut = dup(at(12));
    k.umin = at(13);
    k.umax = at(14);
    k.cAt = dup(at(15));
    k.cFt = dup(at(16));
    k.zero = at(17);
    k.ni3h21 = dup(-A.i3h2f[0]);
    k.ni3h22 = dup(-A.i3h2f[1]);
    k.cA = A.cA[0];
    k.cF = A.cF[0];
    k.umid = m.umid;
    __syncwarp();   // the slot's previous contents have been read
    if (lane == 0) skw[wib] = k;
  }
  __syncwarp();
  const PairScal& k = skw[wib];
  const int giu = band * PAIR_BAND - 2 + 2 * lane;
  PairCtx c;
  c.nx = nx;
  c.ny = ny;
  c.g0 = wrapi(giu, nx);
  c.g1 = wrapi(giu + 1, nx);
  c.rs = rs;
  c.re = min(rs + S, ny);
  c.out0 = lane >= 1 && lane < 1 + PAIR_BAND / 2 && giu < nx;
  c.out1 = c.out0 && giu + 1 < nx;
  c.vec = (nx & 1) == 0;
  c.comb = !is_zero_bits(A.cA[0]);

  auto load = [&](int gj) {
    PairIn in;
    const size_t g = (size_t)gj * nx + c.g0;
    if (c.vec) {
      const double2 u = __ldg(reinterpret_cast<const double2*>(A.ub + g));
      in.ub0 = u.x;
      in.ub1 = u.y;
      in.V = f2(__ldg(reinterpret_cast<const float2*>(A.V + g)));
      in.X = f2(__ldg(reinterpret_cast<const float2*>(A.X + g)));
      in.Y = f2(__ldg(reinterpret_cast<const float2*>(A.Y + g)));
    } else {
      const size_t h = (size_t)gj * nx + c.g1;
      in.ub0 = __ldg(A.ub + g);
      in.ub1 = __ldg(A.ub + h);
      in.V = F2{__ldg(A.V + g), __ldg(A.V + h)};
      in.X = F2{__ldg(A.X + g), __ldg(A.X + h)};
      in.Y = F2{__ldg(A.Y + g), __ldg(A.Y + h)};
    }
    return in;
  };
  const F2 Z = dup(k.zero);
  PairSlot s0, s1, s2;
  // rows rs-3 .. rs-1 feed the first steps; their slots start as the wrapped row rs-3 so
  // that the warm-up steps read finite values (their results are never stored)
  int gj = wrapi(rs - 3, ny);
  {
    const PairIn a = load(gj);
    s0 = PairSlot{};
    s0.U = F2{to_stencil_nb<float>(a.ub0, k.umid), to_stencil_nb<float>(a.ub1, k.umid)};
    s0.V = a.V;
    s0.X = a.X;
    s0.Y = a.Y;
    s1 = s0;
    s2 = s0;
  }
  gj = gj + 1 == ny ? 0 : gj + 1;
  PairIn in = load(gj);
  auto next_row = [&]() {
    gj = gj + 1 == ny ? 0 : gj + 1;
    return load(gj);
  };
  const int r1 = c.re + 1;   // steps rs - 2 .. re + 1
#pragma unroll 1
  for (int r = rs - 2; r <= r1; ++r) {
    const PairIn nin = next_row();
    pair_step<DIFF>(m, A, k, c, Z, r, in, s1, s2, s0);
    const PairSlot t = s1;
    s1 = s2;
    s2 = s0;
    s0 = t;
    in = nin;
  }
}

// 3 CTAs per SM (168 registers per thread)
template <int DIFF>
__global__ void __launch_bounds__(32 * PAIR_WPB, 3)
    pair2d_kernel(const DevModel m, const StageArgs2D<float> A, int S, int bands) {
  const int w = blockIdx.x * PAIR_WPB + (threadIdx.x >> 5);
  pair_run<DIFF>(m, A, S, w % bands, w / bands);
}

// ---- launch (host)

static StripPlan pair_plan(int nx, int ny) {
  const int bands = (nx + PAIR_BAND - 1) / PAIR_BAND;
  return strip_plan(MARCH_PAIR, [=](int S) { return (long long)bands * ((ny + S - 1) / S); });
}

// one launch per output of the stage
template <int DIFF>
static cudaError_t pair2d_go(const DevModel& m, const StageArgs2D<float>& a, int S, cudaStream_t s) {
  const int bands = (a.nx + PAIR_BAND - 1) / PAIR_BAND;
  const long long warps = (long long)bands * ((a.ny + S - 1) / S);
  const long long blocks = (warps + PAIR_WPB - 1) / PAIR_WPB;
  if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
  for (int o = 0; o < a.nout; ++o) {
    pair2d_kernel<DIFF><<<(unsigned)blocks, 32 * PAIR_WPB, 0, s>>>(m, one_output(a, o), S, bands);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace af
