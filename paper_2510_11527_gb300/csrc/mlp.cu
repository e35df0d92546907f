// Learned smoothness indicator for the blend of Section 5.1.3 / 5.2 of arXiv
// 2510.11527: a 21 -> 32 -> 32 -> 1 network maps a normalised patch of cell averages and
// point values around a cell to s >= 0, which replaces the smoothness indicator s in
// theta^{c,s} = exp(-gamma s_face), theta^{d,s} = exp(-gamma s). The MPP limiter and the
// projection still run after it, so bounds and conservation do not depend on it.
//
// Kernels:
//   indicator (fused inference): gather + normalise the patch, two bf16 tensor-core
//     layers (mma.sync m16n8k16, FP32 accumulate, layer-1 accumulators reused as layer-2
//     A fragments), FP32 output layer, softplus; one warp per 16 cells.
//   features: training data (the same patch in FP32) and the plain indicator's label.
//   train: FP32 forward (same bf16 rounding points as the tensor-core path) and backward
//     of tiles of 32 samples, gradients summed per CTA.
//   adam: sum over the CTAs, Adam update of the FP32 master weights and refresh of their
//     bf16 copies.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "af.h"
#include "batch2d.cuh"
#include "ctx.h"

namespace {

constexpr int NIN = 21, NH = 32;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH;
constexpr int OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH, NPARAM = OFF_B3 + 1;   // 1793
static_assert(NPARAM == AF_MLP_NPARAM, "parameter count");

// periodic index for offsets of a few cells (one compare each way; the modulo only on
// meshes smaller than the offset)
__device__ __forceinline__ int wrapm(int i, int n) {
  if (i < 0) {
    i += n;
    if (i < 0) {
      i %= n;
      if (i < 0) i += n;
    }
  } else if (i >= n) {
    i -= n;
    if (i >= n) i %= n;
  }
  return i;
}

// FP32 copies of state values without the FP64 unit (truncating, as the stage kernels)
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(double x) { return af::to_stencil<float>(x); }

// normalised patch from values in FP32: (v_k - v_4) / (max_k |v_k| + 1e-13), v_4 being
// the cell's own average
__device__ __forceinline__ void normalise(const float v[NIN], float f[NIN]) {
  float sc = 0.0f;
#pragma unroll
  for (int k = 0; k < NIN; ++k) sc = fmaxf(sc, fabsf(v[k]));
  const float r = 1.0f / (sc + 1e-13f), m = v[4];
#pragma unroll
  for (int k = 0; k < NIN; ++k) f[k] = (v[k] - m) * r;
}

__device__ __forceinline__ float softplusf(float z) { return z > 20.0f ? z : log1pf(expf(z)); }

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&p);
}

// Tensor-core network on 16 rows held (bf16, [16][40]) in shared memory; returns the
// output pre-activation z (s = softplus(z)) of rows g and g + 8 in all four lanes of
// quad g.
struct NetFrags {
  uint32_t b1[2][4][2], b2[2][4][2];
  float bias1[4][2], bias2[4][2], w3[4][2], b3;
};

__device__ __forceinline__ void load_frags(NetFrags& F, const __nv_bfloat16* w1q, const __nv_bfloat16* w2q,
                                           const float* params, int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int kb = 0; kb < 2; ++kb)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const int n = 8 * nt + g, k0 = 16 * kb + 2 * t;
      F.b1[kb][nt][0] = *reinterpret_cast<const uint32_t*>(w1q + n * 32 + k0);
      F.b1[kb][nt][1] = *reinterpret_cast<const uint32_t*>(w1q + n * 32 + k0 + 8);
      F.b2[kb][nt][0] = *reinterpret_cast<const uint32_t*>(w2q + n * 32 + k0);
      F.b2[kb][nt][1] = *reinterpret_cast<const uint32_t*>(w2q + n * 32 + k0 + 8);
    }
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int col = 8 * nt + 2 * t + e;
      F.bias1[nt][e] = params[OFF_B1 + col];
      F.bias2[nt][e] = params[OFF_B2 + col];
      F.w3[nt][e] = params[OFF_W3 + col];
    }
  F.b3 = params[OFF_B3];
}

__device__ __forceinline__ void net_rows(const NetFrags& F, const __nv_bfloat16 (*sx)[40], int lane, float* s0,
                                         float* s8) {
  const int g = lane >> 2, t = lane & 3;
  float c1[4][4];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) c1[nt][0] = c1[nt][1] = c1[nt][2] = c1[nt][3] = 0.0f;
#pragma unroll
  for (int kb = 0; kb < 2; ++kb) {
    uint32_t a[4];
    a[0] = *reinterpret_cast<const uint32_t*>(&sx[g][16 * kb + 2 * t]);
    a[1] = *reinterpret_cast<const uint32_t*>(&sx[g + 8][16 * kb + 2 * t]);
    a[2] = *reinterpret_cast<const uint32_t*>(&sx[g][16 * kb + 2 * t + 8]);
    a[3] = *reinterpret_cast<const uint32_t*>(&sx[g + 8][16 * kb + 2 * t + 8]);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) mma16816(c1[nt], a, F.b1[kb][nt]);
  }
  // bias + ReLU, rounded to bf16: the layer-1 accumulator tiles 2kb, 2kb+1 are exactly
  // the A fragment of layer-2 k-block kb
  uint32_t a2[2][4];
#pragma unroll
  for (int kb = 0; kb < 2; ++kb) {
    const int n0 = 2 * kb, n1 = 2 * kb + 1;
    a2[kb][0] = pack_bf16(fmaxf(c1[n0][0] + F.bias1[n0][0], 0.f), fmaxf(c1[n0][1] + F.bias1[n0][1], 0.f));
    a2[kb][1] = pack_bf16(fmaxf(c1[n0][2] + F.bias1[n0][0], 0.f), fmaxf(c1[n0][3] + F.bias1[n0][1], 0.f));
    a2[kb][2] = pack_bf16(fmaxf(c1[n1][0] + F.bias1[n1][0], 0.f), fmaxf(c1[n1][1] + F.bias1[n1][1], 0.f));
    a2[kb][3] = pack_bf16(fmaxf(c1[n1][2] + F.bias1[n1][0], 0.f), fmaxf(c1[n1][3] + F.bias1[n1][1], 0.f));
  }
  float c2[4][4];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) c2[nt][0] = c2[nt][1] = c2[nt][2] = c2[nt][3] = 0.0f;
#pragma unroll
  for (int kb = 0; kb < 2; ++kb)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) mma16816(c2[nt], a2[kb], F.b2[kb][nt]);
  float r0 = 0.f, r8 = 0.f;
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      r0 += F.w3[nt][e] * fmaxf(c2[nt][e] + F.bias2[nt][e], 0.f);
      r8 += F.w3[nt][e] * fmaxf(c2[nt][2 + e] + F.bias2[nt][e], 0.f);
    }
  r0 += __shfl_xor_sync(0xffffffffu, r0, 1);
  r0 += __shfl_xor_sync(0xffffffffu, r0, 2);
  r8 += __shfl_xor_sync(0xffffffffu, r8, 1);
  r8 += __shfl_xor_sync(0xffffffffu, r8, 2);
  (void)t;
  *s0 = r0 + F.b3;
  *s8 = r8 + F.b3;
}

// Fused inference on a state, s (double) per cell. Each CTA takes 32 x 8 tiles of
// cells: the tile's cell averages with a +-2 halo and its point values with a -1 halo
// are staged in shared memory (coalesced row loads, converted to FP32 once), every lane
// builds the patch of one cell from there, and each warp runs the network on its 32
// patches as two 16-row blocks.
// Resident CTAs per SM the indicator kernel is compiled for (3: 85 registers, the
// weight fragments partly spilled; 2: 122 registers, no spill).
#ifndef AF_INDICATOR_MIN_CTAS
#define AF_INDICATOR_MIN_CTAS 3
#endif

// The values of a 32 x 8 tile's patches in FP32: cell averages with a +-2 halo, points
// with a -1 halo.
struct PatchTile {
  static constexpr int UX = 36, UY = 12, PX = 33, PY = 9;
  float U[UY][UX], V[PY][PX], X[PY][PX], Y[PY][PX];
};

// stages the tile at (i0, j0) of a periodic mesh, by all 256 threads (no barrier); the
// averages also as stored into dU [UY][UX] if given
template <class PT>
__device__ __forceinline__ void load_patch_tile(PatchTile& S, const double* __restrict__ ub,
                                                const PT* __restrict__ V, const PT* __restrict__ X,
                                                const PT* __restrict__ Y, int nx, int ny, int i0, int j0,
                                                double* dU = nullptr) {
  constexpr int UX = PatchTile::UX, UY = PatchTile::UY, PX = PatchTile::PX, PY = PatchTile::PY;
  for (int k = threadIdx.x; k < UX * UY; k += 256) {
    const int bx = k % UX, by = k / UX;
    const double u = ub[(size_t)wrapm(j0 - 2 + by, ny) * nx + wrapm(i0 - 2 + bx, nx)];
    S.U[by][bx] = af::to_stencil<float>(u);
    if (dU) dU[k] = u;
  }
  for (int k = threadIdx.x; k < PX * PY; k += 256) {
    const int bx = k % PX, by = k / PX;
    const size_t g = (size_t)wrapm(j0 - 1 + by, ny) * nx + wrapm(i0 - 1 + bx, nx);
    S.V[by][bx] = to_f32(V[g]);
    S.X[by][bx] = to_f32(X[g]);
    S.Y[by][bx] = to_f32(Y[g]);
  }
}

// normalised patch of the tile's cell (tx, ty)
__device__ __forceinline__ void patch_of(const PatchTile& S, int tx, int ty, float f[NIN]) {
  constexpr int kPatchA[13] = {-1, 0, 1, -1, 0, 1, -1, 0, 1, -2, 2, 0, 0};
  constexpr int kPatchB[13] = {-1, -1, -1, 0, 0, 0, 1, 1, 1, 0, 0, -2, 2};
  float v[NIN];
#pragma unroll
  for (int k = 0; k < 13; ++k) v[k] = S.U[ty + 2 + kPatchB[k]][tx + 2 + kPatchA[k]];
  v[13] = S.V[ty][tx];
  v[14] = S.V[ty][tx + 1];
  v[15] = S.V[ty + 1][tx];
  v[16] = S.V[ty + 1][tx + 1];
  v[17] = S.X[ty + 1][tx];
  v[18] = S.X[ty + 1][tx + 1];
  v[19] = S.Y[ty][tx + 1];
  v[20] = S.Y[ty + 1][tx + 1];
  normalise(v, f);
}

// One 32 x 8 tile (cells i0 .. i0 + 31, j0 .. j0 + 7) of a periodic mesh: the patches
// are gathered into shared memory, each warp runs the network on its row of 32 cells
// and writes s. Called by all 256 threads of the CTA, which it leaves synchronised.
template <class PT>
__device__ __forceinline__ void indicator_tile(const NetFrags& F, const double* __restrict__ ub,
                                               const PT* __restrict__ V, const PT* __restrict__ X,
                                               const PT* __restrict__ Y, int nx, int ny, int i0, int j0,
                                               double* __restrict__ out) {
  __shared__ PatchTile S;
  __shared__ __align__(16) __nv_bfloat16 sx[8][32][40];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  {
    load_patch_tile<PT>(S, ub, V, X, Y, nx, ny, i0, j0);
    __syncthreads();
    {
      // cell (i0 + lane, j0 + warp)
      float f[NIN];
      patch_of(S, lane, warp, f);
#pragma unroll
      for (int k = 0; k < 32; k += 2)
        *reinterpret_cast<uint32_t*>(&sx[warp][lane][k]) =
            pack_bf16(k < NIN ? f[k] : 0.f, k + 1 < NIN ? f[k + 1] : 0.f);
    }
    __syncwarp();
    const int j = j0 + warp;
    float z[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) net_rows(F, sx[warp] + 16 * h, lane, &z[h][0], &z[h][1]);
    {
      // the four lanes of a quad share the four pre-activations (rows g, g + 8 of both
      // 16-row blocks): each applies the output activation to one of them
      const int t = lane & 3, h = t >> 1, w = t & 1;
      const float s = softplusf(z[h][w]);
      const int i = i0 + 16 * h + (lane >> 2) + 8 * w;
      if (j < ny && i < nx) out[(size_t)j * nx + i] = af::f2d_exact(s);
    }
    __syncthreads();
  }
}

template <class PT>
__global__ void __launch_bounds__(256, AF_INDICATOR_MIN_CTAS) indicator_kernel(const double* __restrict__ ub, const PT* __restrict__ V,
                                                           const PT* __restrict__ X, const PT* __restrict__ Y, int nx,
                                                           int ny, const __nv_bfloat16* __restrict__ w1q,
                                                           const __nv_bfloat16* __restrict__ w2q,
                                                           const float* __restrict__ params, double* __restrict__ out) {
  NetFrags F;
  load_frags(F, w1q, w2q, params, threadIdx.x & 31);
  const int tiles_x = (nx + 31) / 32, tiles = tiles_x * ((ny + 7) / 8);
  for (int t = blockIdx.x; t < tiles; t += gridDim.x)
    indicator_tile<PT>(F, ub, V, X, Y, nx, ny, (t % tiles_x) * 32, (t / tiles_x) * 8, out);
}

// The same over every instance of a batch (state buffer `in` of each, s into its
// indicator array): the 32 x 8 tiles of instance k are numbered from inst[k].ind_begin
// on, so a tile's instance is found by bisection.
template <class PT>
__global__ void __launch_bounds__(256, AF_INDICATOR_MIN_CTAS)
    indicator_batch_kernel(const af::BatchInst* __restrict__ inst, int n, int total, int in,
                           const __nv_bfloat16* __restrict__ w1q, const __nv_bfloat16* __restrict__ w2q,
                           const float* __restrict__ params) {
  NetFrags F;
  load_frags(F, w1q, w2q, params, threadIdx.x & 31);
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    int lo = 0, hi = n - 1;   // the last instance whose first tile is <= w
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (inst[mid].ind_begin <= w) lo = mid;
      else hi = mid - 1;
    }
    const af::BatchInst& I = inst[lo];
    const int t = w - I.ind_begin, tiles_x = (I.nx + 31) / 32;
    indicator_tile<PT>(F, I.ub[in], (const PT*)I.pv[in], (const PT*)I.px[in], (const PT*)I.py[in], I.nx, I.ny,
                       (t % tiles_x) * 32, (t / tiles_x) * 8, I.s);
  }
}

// network on given FP32 feature rows (n x 21) -> out (n)
__global__ void __launch_bounds__(256) infer_rows_kernel(const float* __restrict__ feat, long long n,
                                                         const __nv_bfloat16* __restrict__ w1q,
                                                         const __nv_bfloat16* __restrict__ w2q,
                                                         const float* __restrict__ params, float* __restrict__ out) {
  __shared__ __align__(16) __nv_bfloat16 sx[8][16][40];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  NetFrags F;
  load_frags(F, w1q, w2q, params, lane);
  for (long long base = ((long long)blockIdx.x * 8 + warp) * 16; base < n; base += (long long)gridDim.x * 128) {
    if (lane < 16) {
      const long long row = base + lane;
#pragma unroll
      for (int k = 0; k < 32; k += 2) {
        const float lo = (row < n && k < NIN) ? feat[row * NIN + k] : 0.f;
        const float hi = (row < n && k + 1 < NIN) ? feat[row * NIN + k + 1] : 0.f;
        *reinterpret_cast<uint32_t*>(&sx[warp][lane][k]) = pack_bf16(lo, hi);
      }
    }
    __syncwarp();
    float z0, z8;
    net_rows(F, sx[warp], lane, &z0, &z8);
    // lanes t = 0, 1 of each quad apply the output activation to rows g, g + 8
    const int t = lane & 3;
    if (t < 2) {
      const long long row = base + (lane >> 2) + 8 * t;
      const float s = softplusf(t ? z8 : z0);
      if (row < n) out[row] = s;
    }
    __syncwarp();
  }
}

// Training data: FP32 patch and the plain indicator max(s_1, s_2) (FP64) per cell, on
// 32 x 8 tiles staged as the fused inference stages them. What bounds it is GB300's FP64
// unit (the label's divisions): each s~ is formed once per location, 2.3 per cell instead
// of the 6 of a cell by itself, and the patches, 21 floats per cell, leave through shared
// memory so that a warp's 32 rows are one contiguous store.
template <class PT>
__global__ void __launch_bounds__(256) features_kernel(const double* __restrict__ ub, const PT* __restrict__ V,
                                                       const PT* __restrict__ X, const PT* __restrict__ Y, int nx,
                                                       int ny, float* __restrict__ feat, float* __restrict__ label) {
  __shared__ PatchTile S;
  __shared__ double dU[PatchTile::UY][PatchTile::UX];
  __shared__ double st1[8][34], st2[10][32];   // s~_1 on columns -1 .. 32, s~_2 on rows -1 .. 8
  __shared__ float rows[8][32 * NIN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles_x = (nx + 31) / 32, tiles = tiles_x * ((ny + 7) / 8);
  for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int i0 = (t % tiles_x) * 32, j0 = (t / tiles_x) * 8;
    load_patch_tile<PT>(S, ub, V, X, Y, nx, ny, i0, j0, label ? &dU[0][0] : nullptr);
    __syncthreads();
    if (label) {
      auto st = [](double um, double uc, double up) {
        return fabs(um - 2.0 * uc + up) / (fabs(um) + 2.0 * fabs(uc) + fabs(up) + 1e-13);
      };
      for (int k = tid; k < 8 * 34 + 10 * 32; k += 256) {
        if (k < 8 * 34) {
          const int x = k % 34, y = k / 34;
          st1[y][x] = st(dU[y + 2][x], dU[y + 2][x + 1], dU[y + 2][x + 2]);
        } else {
          const int x = (k - 8 * 34) % 32, y = (k - 8 * 34) / 32;
          st2[y][x] = st(dU[y][x + 2], dU[y + 1][x + 2], dU[y + 2][x + 2]);
        }
      }
    }
    float f[NIN];
    patch_of(S, lane, warp, f);
#pragma unroll
    for (int k = 0; k < NIN; ++k) rows[warp][lane * NIN + k] = f[k];
    __syncthreads();
    const int j = j0 + warp, w = min(32, nx - i0);
    if (j < ny) {
      const size_t c = (size_t)j * nx + i0;
      for (int k = lane; k < w * NIN; k += 32) feat[c * NIN + k] = rows[warp][k];
      if (label && lane < w) {
        const double s1 = st1[warp][lane] + 4.0 * st1[warp][lane + 1] + st1[warp][lane + 2];
        const double s2 = st2[warp][lane] + 4.0 * st2[warp + 1][lane] + st2[warp + 2][lane];
        label[c + lane] = (float)(fmax(s1, s2) * (1.0 / 6.0));
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// programmatic dependent launch (sm_90 and later): let the next launch of the stream start,
// and wait for the completion of the one before
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Load, after grid_dependency_wait, of what an earlier launch may still have been writing
// when this one started. Such memory changes while the kernel runs, so its pointers are not
// __restrict__ and it is not read through the read-only path: volatile keeps the load
// behind the wait, and a relaxed load at device scope sees what the wait made visible.
__device__ __forceinline__ float load_written(const float* p) {
  float v;
  asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Forward + backward of a minibatch in FP32 with the tensor-core path's rounding points
// (bf16 inputs and weights of the two hidden layers): the gradient of the batch-mean loss
// summed over the samples of each CTA into its row of `partial` (TRAIN_ROW floats: the
// parameters' gradient, then the loss), which adam_kernel / grad_kernel add up in a fixed
// order, so a step is deterministic. Sample k of the batch is k itself when seed == 0,
// else a splitmix64 draw over [0, nsamples).
//
// The work is a few thousand multiply-adds per sample: what bounds it is the length of one
// thread's chain and how many SMs take part. One sample per thread with its 1793 shared
// atomics took 0.5 ms per step of 4096 samples (16 CTAs); here a CTA takes tiles of 32
// samples, lane = sample, and each of its 8 warps forms 4 of the 32 units of every layer
// (weights as one broadcast 16-byte read per input), so 4096 samples are 128 CTAs and a
// warp's chain is an eighth of the network's. The weight gradients are products of two
// [unit][sample] arrays in shared memory, 4 + 3 entries per thread, kept in registers over
// the CTA's tiles. Sums over a layer's inputs run in the order of the single-sample form.
//
// A step is two short dependent launches (this one and adam_kernel), each launched while
// the one before still runs (programmatic dependent launch): the loads that do not depend
// on it -- the first tile's sample indices, features and targets -- are made before
// griddepcontrol.wait, which returns when the launch before has completed and its writes
// are visible.
constexpr int TRAIN_TILE = 32;            // samples per tile (one per lane)
constexpr int TRAIN_LD = TRAIN_TILE + 4;  // row stride: 16-byte aligned, 8 rows on distinct banks
constexpr int TRAIN_MAX_CTAS = 152 * 2;   // rows of the partial sums
constexpr int TRAIN_ROW = NPARAM + 7;     // 1800 floats per row: gradient, loss at NPARAM

__global__ void __launch_bounds__(256, 2) train_kernel(const float* __restrict__ feat, const float* __restrict__ label,
                                                    long long nsamples, int batch, unsigned long long seed, int step,
                                                    const float* params, float* partial) {
  __shared__ __align__(16) float W1T[NIN][NH], W2T[NH][NH], W2[NH][NH];   // [input][unit], [input][unit], [unit][input]
  __shared__ float b1[NH], b2[NH], w3[NH];
  __shared__ __align__(16) float xT[NIN][TRAIN_LD], h1T[NH][TRAIN_LD], h2T[NH][TRAIN_LD];
  __shared__ __align__(16) float d1T[NH][TRAIN_LD], d2T[NH][TRAIN_LD], d3[TRAIN_LD];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  launch_dependents();
  const int tiles = (batch - 1) / TRAIN_TILE + 1;
  // a tile's targets (one per lane) and this warp's four sample rows (one input per lane)
  float target = 0.f, rows[4];
  bool live = false;
  auto fetch = [&](int tile) {
    const long long k = (long long)tile * TRAIN_TILE + lane;
    live = k < batch;
    long long idx = 0;
    if (live)
      idx = seed == 0 ? k
                      : (long long)(splitmix64(seed ^ ((unsigned long long)step << 32) ^ (unsigned long long)k) %
                                    (unsigned long long)nsamples);
    target = live ? label[idx] : 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int sl = 4 * warp + r;
      const long long row = __shfl_sync(0xffffffffu, idx, sl);
      rows[r] = lane < NIN && k - lane + sl < batch ? bfr(feat[row * NIN + lane]) : 0.f;
    }
  };
  if (blockIdx.x < tiles) fetch(blockIdx.x);
  grid_dependency_wait();
  for (int k = tid; k < NH * NIN; k += 256) W1T[k % NIN][k / NIN] = bfr(load_written(params + OFF_W1 + k));
  for (int k = tid; k < NH * NH; k += 256) {
    const float w = bfr(load_written(params + OFF_W2 + k));
    W2[k / NH][k % NH] = w;
    W2T[k % NH][k / NH] = w;
  }
  if (tid < NH) {
    b1[tid] = load_written(params + OFF_B1 + tid);
    b2[tid] = load_written(params + OFF_B2 + tid);
    w3[tid] = load_written(params + OFF_W3 + tid);
  }
  const float b3 = load_written(params + OFF_B3);
  // this thread's gradient entries: W2 (unit go, inputs gq + 8 k), W1 (unit go, inputs
  // gq + 8 k < 21) and one entry of b1, b2, w3 or b3
  const int go = tid >> 3, gq = tid & 7;
  float gw2[4] = {0.f, 0.f, 0.f, 0.f}, gw1[3] = {0.f, 0.f, 0.f}, gb = 0.f, lossv = 0.f;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (tile != (int)blockIdx.x) fetch(tile);
    __syncthreads();   // the previous tile's arrays have been read (and the weights written)
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (lane < NIN) xT[lane][4 * warp + r] = rows[r];
    __syncthreads();
    const int u0 = 4 * warp;   // this warp's units of each layer
    float z1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < NIN; ++q) {
      const float4 w = *reinterpret_cast<const float4*>(&W1T[q][u0]);
      const float x = xT[q][lane];
      z1[0] = fmaf(w.x, x, z1[0]);
      z1[1] = fmaf(w.y, x, z1[1]);
      z1[2] = fmaf(w.z, x, z1[2]);
      z1[3] = fmaf(w.w, x, z1[3]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      z1[e] += b1[u0 + e];
      h1T[u0 + e][lane] = bfr(fmaxf(z1[e], 0.f));
    }
    __syncthreads();
    float z2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < NH; ++q) {
      const float4 w = *reinterpret_cast<const float4*>(&W2T[q][u0]);
      const float h = h1T[q][lane];
      z2[0] = fmaf(w.x, h, z2[0]);
      z2[1] = fmaf(w.y, h, z2[1]);
      z2[2] = fmaf(w.z, h, z2[2]);
      z2[3] = fmaf(w.w, h, z2[3]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      z2[e] += b2[u0 + e];
      h2T[u0 + e][lane] = fmaxf(z2[e], 0.f);
    }
    __syncthreads();
    // output layer and its gradient, formed by every warp for its lanes' samples
    float z3 = 0.f;
#pragma unroll
    for (int o = 0; o < NH; ++o) z3 = fmaf(w3[o], h2T[o][lane], z3);
    z3 += b3;
    const float r = softplusf(z3) - target;
    const float dz3 = live ? 2.f / (float)batch * r / (1.f + expf(-z3)) : 0.f;
    if (warp == 0) {
      d3[lane] = dz3;
      if (live) lossv += r * r / (float)batch;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) d2T[u0 + e][lane] = z2[e] > 0.f ? dz3 * w3[u0 + e] : 0.f;
    __syncthreads();
    float dh[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int o = 0; o < NH; ++o) {
      const float4 w = *reinterpret_cast<const float4*>(&W2[o][u0]);
      const float d = d2T[o][lane];
      dh[0] = fmaf(d, w.x, dh[0]);
      dh[1] = fmaf(d, w.y, dh[1]);
      dh[2] = fmaf(d, w.z, dh[2]);
      dh[3] = fmaf(d, w.w, dh[3]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) d1T[u0 + e][lane] = z1[e] > 0.f ? dh[e] : 0.f;
    __syncthreads();
    // gradient entries of this tile
#pragma unroll
    for (int s = 0; s < TRAIN_TILE; s += 4) {
      const float4 a2 = *reinterpret_cast<const float4*>(&d2T[go][s]);
      const float4 a1 = *reinterpret_cast<const float4*>(&d1T[go][s]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 h = *reinterpret_cast<const float4*>(&h1T[gq + 8 * e][s]);
        gw2[e] = fmaf(a2.w, h.w, fmaf(a2.z, h.z, fmaf(a2.y, h.y, fmaf(a2.x, h.x, gw2[e]))));
      }
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        if (gq + 8 * e < NIN) {
          const float4 x = *reinterpret_cast<const float4*>(&xT[gq + 8 * e][s]);
          gw1[e] = fmaf(a1.w, x.w, fmaf(a1.z, x.z, fmaf(a1.y, x.y, fmaf(a1.x, x.x, gw1[e]))));
        }
      }
    }
    if (warp < 4) {
      // b1, b2, w3 (unit = lane), b3 (lane 0 of warp 3)
      const float* a = warp == 0 ? d1T[lane] : (warp == 1 ? d2T[lane] : (warp == 2 ? h2T[lane] : d3));
      float acc = 0.f;
      if (warp < 2 || (warp == 3 && lane == 0)) {
        for (int s = 0; s < TRAIN_TILE; ++s) acc += a[s];
      } else if (warp == 2) {
        for (int s = 0; s < TRAIN_TILE; ++s) acc = fmaf(d3[s], a[s], acc);
      }
      gb += acc;
    }
  }
  float* row = partial + (size_t)blockIdx.x * TRAIN_ROW;
#pragma unroll
  for (int e = 0; e < 4; ++e) row[OFF_W2 + go * NH + gq + 8 * e] = gw2[e];
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (gq + 8 * e < NIN) row[OFF_W1 + go * NIN + gq + 8 * e] = gw1[e];
  if (warp == 0) {
    row[OFF_B1 + lane] = gb;
    for (int o = 16; o > 0; o >>= 1) lossv += __shfl_xor_sync(0xffffffffu, lossv, o);
    if (lane == 0) row[NPARAM] = lossv;
  } else if (warp == 1) {
    row[OFF_B2 + lane] = gb;
  } else if (warp == 2) {
    row[OFF_W3 + lane] = gb;
  } else if (warp == 3 && lane == 0) {
    row[OFF_B3] = gb;
  }
}

// sum over the CTAs' rows of column q = 32 blockIdx + lane (the gradient entries, then the
// loss at NPARAM) in a fixed order: warp w takes rows w, w + 8, ..., then the warps in
// order; valid in warp 0
__device__ __forceinline__ float column_sum(const float* partial, int rows) {
  __shared__ float sm[8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x * 32 + lane;
  float acc = 0.f;
  if (q <= NPARAM) {
#pragma unroll 16
    for (int r = warp; r < rows; r += 8) acc += load_written(partial + (size_t)r * TRAIN_ROW + q);
  }
  sm[warp][lane] = acc;
  __syncthreads();
  float g = 0.f;
  for (int w = 0; w < 8; ++w) g += sm[w][lane];
  return g;
}
constexpr int COLUMN_CTAS = (NPARAM + 1 + 31) / 32;

// Adam on the FP32 master weights with the gradient summed over the CTAs' rows; refreshes
// the bf16 copies
__global__ void __launch_bounds__(256) adam_kernel(float* p, float* m, float* v, const float* partial, int rows,
                                                   float lr, float c1, float c2, __nv_bfloat16* w1q,
                                                   __nv_bfloat16* w2q, float* loss) {
  launch_dependents();
  grid_dependency_wait();
  const float g = column_sum(partial, rows);
  const int q = blockIdx.x * 32 + (int)threadIdx.x;
  if (threadIdx.x >= 32 || q > NPARAM) return;
  if (q == NPARAM) {
    *loss = g;
    return;
  }
  const float mq = 0.9f * load_written(m + q) + 0.1f * g, vq = 0.999f * load_written(v + q) + 0.001f * g * g;
  m[q] = mq;
  v[q] = vq;
  const float w = load_written(p + q) - lr * (mq / c1) / (sqrtf(vq / c2) + 1e-8f);
  p[q] = w;
  if (q < OFF_B1) w1q[(q / NIN) * 32 + q % NIN] = __float2bfloat16_rn(w);
  else if (q >= OFF_W2 && q < OFF_B2) w2q[q - OFF_W2] = __float2bfloat16_rn(w);
}

// the summed gradient (and the loss at NPARAM) alone
__global__ void __launch_bounds__(256) grad_kernel(const float* partial, int rows, float* grad) {
  const float g = column_sum(partial, rows);
  const int q = blockIdx.x * 32 + (int)threadIdx.x;
  if (threadIdx.x < 32 && q <= NPARAM) grad[q] = g;
}

__global__ void quantize_kernel(const float* __restrict__ p, __nv_bfloat16* w1q, __nv_bfloat16* w2q) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < 32 * 32) {
    const int n = q / 32, k = q % 32;
    w1q[q] = __float2bfloat16_rn(k < NIN ? p[OFF_W1 + n * NIN + k] : 0.f);
    w2q[q] = __float2bfloat16_rn(p[OFF_W2 + q]);
  }
}

}  // namespace

struct af_mlp {
  unsigned char* block = nullptr;
  float* params = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;      // summed gradient, then the loss
  float* loss = nullptr;
  float* partial = nullptr;   // TRAIN_MAX_CTAS rows of partial sums
  __nv_bfloat16* w1q = nullptr;
  __nv_bfloat16* w2q = nullptr;
  int t = 0;
  cudaStream_t stream = nullptr;
};

namespace af {
cudaError_t mlp_indicator_launch(const af_ctx* c, const af_mlp* net, int buf, double* out) {
  if (c->dim != 2) return cudaErrorInvalidValue;
  const long long tiles = (long long)((c->nx + 31) / 32) * ((c->ny + 7) / 8);
  const int grid = (int)std::min<long long>(tiles, 152LL * AF_INDICATOR_MIN_CTAS);
  if (c->prec == AF_PREC_FP64)
    indicator_kernel<double><<<grid, 256, 0, c->stream>>>(c->ub[buf], (const double*)c->pv[buf],
                                                          (const double*)c->px[buf], (const double*)c->py[buf],
                                                          c->nx, c->ny, net->w1q, net->w2q, net->params, out);
  else
    indicator_kernel<float><<<grid, 256, 0, c->stream>>>(c->ub[buf], (const float*)c->pv[buf],
                                                         (const float*)c->px[buf], (const float*)c->py[buf], c->nx,
                                                         c->ny, net->w1q, net->w2q, net->params, out);
  return cudaGetLastError();
}

cudaError_t mlp_indicator_batch_launch(const af_mlp* net, const BatchInst* inst, int n, int total, int in, int prec,
                                       cudaStream_t s) {
  if (total < 1 || n < 1) return cudaErrorInvalidValue;
  const int grid = (int)std::min<long long>(total, 152LL * AF_INDICATOR_MIN_CTAS);
  if (prec == AF_PREC_FP64)
    indicator_batch_kernel<double><<<grid, 256, 0, s>>>(inst, n, total, in, net->w1q, net->w2q, net->params);
  else
    indicator_batch_kernel<float><<<grid, 256, 0, s>>>(inst, n, total, in, net->w1q, net->w2q, net->params);
  return cudaGetLastError();
}
}  // namespace af

namespace {
// launch that may start while the launch before it in the stream runs (its kernel waits)
template <class... P, class... A>
cudaError_t launch_early(void (*kern)(P...), int grid, A... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(256);
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// CTAs (rows of partial sums) of a minibatch
int train_rows(int batch) { return std::min((batch - 1) / TRAIN_TILE + 1, TRAIN_MAX_CTAS); }
}  // namespace

extern "C" {

af_status af_mlp_create(af_mlp** out) {
  if (!out) return AF_E_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return AF_E_UNSUPPORTED;
  af_mlp* net = new (std::nothrow) af_mlp;
  if (!net) return AF_E_OOM;
  const size_t bytes = (10240 + TRAIN_MAX_CTAS * TRAIN_ROW) * sizeof(float) + 2 * 32 * 32 * sizeof(__nv_bfloat16) + 256;
  if (cudaMalloc(&net->block, bytes) != cudaSuccess) {
    cudaGetLastError();
    delete net;
    return AF_E_OOM;
  }
  cudaMemset(net->block, 0, bytes);
  float* f = (float*)net->block;
  net->params = f;
  net->m = f + 2048;
  net->v = f + 4096;
  net->grad = f + 6144;
  net->loss = f + 8192;
  net->partial = f + 10240;
  net->w1q = (__nv_bfloat16*)(net->partial + TRAIN_MAX_CTAS * TRAIN_ROW);
  net->w2q = net->w1q + 32 * 32;
  *out = net;
  return AF_OK;
}

af_status af_mlp_destroy(af_mlp* net) {
  if (!net) return AF_E_ARG;
  cudaDeviceSynchronize();
  cudaFree(net->block);
  delete net;
  return AF_OK;
}

af_status af_mlp_set_params(af_mlp* net, const float* host, int n) {
  if (!net || !host || n != NPARAM) return AF_E_ARG;
  if (cudaMemcpy(net->params, host, NPARAM * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return AF_E_CUDA;
  cudaMemset(net->m, 0, NPARAM * sizeof(float));
  cudaMemset(net->v, 0, NPARAM * sizeof(float));
  net->t = 0;
  quantize_kernel<<<4, 256>>>(net->params, net->w1q, net->w2q);
  return cudaDeviceSynchronize() == cudaSuccess ? AF_OK : AF_E_CUDA;
}

af_status af_mlp_get_params(const af_mlp* net, float* host) {
  if (!net || !host) return AF_E_ARG;
  return cudaMemcpy(host, net->params, NPARAM * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? AF_OK
                                                                                                      : AF_E_CUDA;
}

af_status af_mlp_features(af_ctx* c, float* feat_dev, float* label_dev) {
  if (!c || !feat_dev || c->dim != 2 || c->bounds_pending) return AF_E_ARG;
  const long long tiles = (long long)((c->nx + 31) / 32) * ((c->ny + 7) / 8);
  const int grid = (int)std::min<long long>(tiles, 152 * 4);
  if (c->prec == AF_PREC_FP64)
    features_kernel<double><<<grid, 256, 0, c->stream>>>(c->ub[0], (const double*)c->pv[0], (const double*)c->px[0],
                                                         (const double*)c->py[0], c->nx, c->ny, feat_dev, label_dev);
  else
    features_kernel<float><<<grid, 256, 0, c->stream>>>(c->ub[0], (const float*)c->pv[0], (const float*)c->px[0],
                                                        (const float*)c->py[0], c->nx, c->ny, feat_dev, label_dev);
  if (cudaGetLastError() != cudaSuccess) return AF_E_CUDA;
  return cudaStreamSynchronize(c->stream) == cudaSuccess ? AF_OK : AF_E_CUDA;
}

af_status af_mlp_infer(const af_mlp* net, const float* feat_dev, long long n, float* out_dev) {
  if (!net || !feat_dev || !out_dev || n < 1) return AF_E_ARG;
  const int grid = (int)std::min<long long>((n + 127) / 128, 152 * 16);
  infer_rows_kernel<<<grid, 256>>>(feat_dev, n, net->w1q, net->w2q, net->params, out_dev);
  if (cudaGetLastError() != cudaSuccess) return AF_E_CUDA;
  return cudaDeviceSynchronize() == cudaSuccess ? AF_OK : AF_E_CUDA;
}

af_status af_mlp_indicator(const af_mlp* net, af_ctx* c, double* s_dev) {
  if (!net || !c || !s_dev || c->dim != 2 || c->bounds_pending) return AF_E_ARG;
  if (af::mlp_indicator_launch(c, net, 0, s_dev) != cudaSuccess) return AF_E_CUDA;
  return cudaStreamSynchronize(c->stream) == cudaSuccess ? AF_OK : AF_E_CUDA;
}

af_status af_mlp_grad(af_mlp* net, const float* feat_dev, const float* label_dev, int nsamples, float* grad_host,
                      float* loss_host) {
  if (!net || !feat_dev || !label_dev || nsamples < 1) return AF_E_ARG;
  const int rows = train_rows(nsamples);
  train_kernel<<<rows, 256>>>(feat_dev, label_dev, nsamples, nsamples, 0ull, 0, net->params, net->partial);
  grad_kernel<<<COLUMN_CTAS, 256>>>(net->partial, rows, net->grad);
  if (cudaGetLastError() != cudaSuccess) return AF_E_CUDA;
  if (grad_host && cudaMemcpy(grad_host, net->grad, NPARAM * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return AF_E_CUDA;
  if (loss_host && cudaMemcpy(loss_host, net->grad + NPARAM, sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return AF_E_CUDA;
  return AF_OK;
}

af_status af_mlp_train(af_mlp* net, const float* feat_dev, const float* label_dev, long long nsamples, int batch,
                       int steps, float lr, unsigned long long seed, float* loss_host) {
  if (!net || !feat_dev || !label_dev || nsamples < 1 || batch < 1 || steps < 0 || !(lr > 0.f)) return AF_E_ARG;
  if (seed == 0 && batch > nsamples) return AF_E_ARG;   // seed 0: rows 0..batch-1 in order
  float last = 0.f;
  const int rows = train_rows(batch);
  for (int s = 0; s < steps; ++s) {
    // (the first launch waits for the stream as usual: the rows may just have been written)
    if (s == 0)
      train_kernel<<<rows, 256>>>(feat_dev, label_dev, nsamples, batch, seed, s, net->params, net->partial);
    else if (launch_early(train_kernel, rows, feat_dev, label_dev, nsamples, batch, seed, s, net->params,
                          net->partial) != cudaSuccess)
      return AF_E_CUDA;
    net->t += 1;
    const float c1 = 1.f - powf(0.9f, (float)net->t), c2 = 1.f - powf(0.999f, (float)net->t);
    if (launch_early(adam_kernel, COLUMN_CTAS, net->params, net->m, net->v, net->partial, rows, lr, c1, c2, net->w1q,
                     net->w2q, net->loss) != cudaSuccess)
      return AF_E_CUDA;
    if (cudaGetLastError() != cudaSuccess) return AF_E_CUDA;
    if (s == steps - 1 && loss_host) {
      if (cudaMemcpy(&last, net->loss, sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return AF_E_CUDA;
      *loss_host = last;
    }
  }
  return cudaDeviceSynchronize() == cudaSuccess ? AF_OK : AF_E_CUDA;
}

af_status af_set_mlp(af_ctx* c, const af_mlp* net) {
  if (!c) return AF_E_ARG;
  if (net && (c->dim != 2 || c->opts.blend != AF_BLEND_EXTERNAL)) return AF_E_ARG;
  c->mlp = net;
  return AF_OK;
}

}  // extern "C"
