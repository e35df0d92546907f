// Small device functions shared by the marching stage kernels (2D column marching, 3D
// plane marching): compile-time diffusion kinds, explicit multiply-adds, warp shuffles by
// one lane and the 5-point line residual.
#pragma once
#include "af_model.cuh"

namespace af {

// max / min for values that are never NaN in a valid state: one FMNMX in FP32 (tmax /
// tmin keep the select semantics of the tile kernel); FP64 keeps the integer compare
__device__ __forceinline__ float fmx(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ float fmn(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double fmx(double a, double b) { return tmax(a, b); }
__device__ __forceinline__ double fmn(double a, double b) { return tmin(a, b); }

// largest / smallest of three (one instruction in FP32) and of five
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max5(float a, float b, float c, float d, float e) { return max3(max3(a, b, c), d, e); }

// Diffusion kinds compiled into the column-marching kernel (DK_GENERIC takes the
// model's runtime kind).
enum : int { DK_GENERIC = -1, DK_NONE = 0, DK_CONST = 1, DK_PWL = 2, DK_PME2 = 3, DK_CUBIC = 4 };

template <int DIFF, class T>
__device__ __forceinline__ T apot_k(const DevModel& m, T u) {
  if constexpr (DIFF == DK_NONE) {
    return T(0);
  } else if constexpr (DIFF == DK_CONST) {
    return par<T>(m.dp, m.dpf, 0) * u;
  } else if constexpr (DIFF == DK_PWL) {
    // both branches always: a zero coefficient contributes a signed zero, which does not
    // change the sum
    return par<T>(m.dp, m.dpf, 0) * fmn(u - par<T>(m.dp, m.dpf, 1), T(0)) +
           par<T>(m.dp, m.dpf, 2) * fmx(u - par<T>(m.dp, m.dpf, 3), T(0));
  } else if constexpr (DIFF == DK_PME2) {
    return u * u;
  } else if constexpr (DIFF == DK_CUBIC) {
    return ((par<T>(m.dp, m.dpf, 2) * u + par<T>(m.dp, m.dpf, 1)) * u + par<T>(m.dp, m.dpf, 0)) * u;
  } else {
    return apot<T>(m, u);
  }
}

// a * b + c with one rounding, written out (the translation unit of this kernel is
// compiled without contraction)
__device__ __forceinline__ float sfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double sfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// line residual of stage_tile's line_res with its multiply-adds fused explicitly
template <class T>
__device__ __forceinline__ T line_res_s(T z0, T z1, T z2, T z3, T z4, T f0, T f1, T f3, T f4, T alpha, T a0, T a1,
                                        T a2, T a3, T a4, T i6h, T i3h2) {
  const T cf = sfma(T(8), f3 - f1, f0 - f4);
  const T dz = sfma(T(6), z2, sfma(T(-4), z1 + z3, z0 + z4));
  const T da = sfma(T(-30), a2, sfma(T(16), a1 + a3, -(a0 + a4)));
  return sfma(da, i3h2, -(sfma(alpha, dz, cf) * i6h));
}

template <class T>
__device__ __forceinline__ T shup(T v) { return __shfl_up_sync(0xffffffffu, v, 1); }
template <class T>
__device__ __forceinline__ T shdn(T v) { return __shfl_down_sync(0xffffffffu, v, 1); }

}  // namespace af
