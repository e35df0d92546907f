// Global reductions of the active flux driver: the CFL time step (eq.
// multid_av_pp_dt of arXiv 2510.11527 with the interval wave speed of Section 5.2),
// the total mass and the min/max over all DoFs. Every reduction is deterministic:
// max/min are order independent, and sums are formed per block in a fixed tree order
// and then summed by one block in block order.
#pragma once
#include "af_model.cuh"

namespace af {

constexpr int RED_THREADS = 256;
constexpr int RED_MAX_BLOCKS = 1024;   // partial-result slots per reduction

// The CFL rate max over faces of alpha_face / h + kappa_max / h^2, with alpha_face =
// max |f_l'| over the interval spanned by the two cell averages. Its maximum over all
// faces equals the maximum over cells of |f_l'(u)| / h + kappa_max / h^2 (every cell
// average is an end point of faces in both directions, and rounding is monotone),
// together with |f_l'(c)| / h + kappa_max / h^2 for each interior extremum c of f_l'
// that lies strictly inside some face interval. The kernel reduces the first term into
// rate_bits[0] (non-negative doubles order like their bit patterns) and flags the
// extrema met (bit 8 l + k) in rate_bits[1]; dt_finish adds their terms.
// A bounded 1D interval (bc != AF_BC_PERIODIC) has no wrap-around face; its two end
// faces join the end cells to their ghosts: the Dirichlet values gl / gr are then face
// end points too, while an outflow ghost repeats the end cell (nothing new). A 2D
// rectangle with outflow ends arrives in its padded layout (nx, ny = padded sizes): row
// and column 0 are skipped, and its last column / row has no face beyond.
template <int FLUX>
__device__ __forceinline__ unsigned crit_flags(const DevModel& m, int dir, double a, double b) {
  unsigned f = 0u;
  if constexpr (FLUX == FLUX_BL) {
    const double lo = tmin(a, b), hi = tmax(a, b);
    for (int k = 0; k < m.ncrit[dir]; ++k)
      if (tlt(lo, m.crit[dir][k]) && tlt(m.crit[dir][k], hi)) f |= 1u << k;
  }
  return f;
}

// bits of a rate (never negative), ordered as the rate, a NaN of either sign above all. The
// sign is cleared in the high word: a mask of all 64 bits is compiled as the FP64 unit's
// absolute value, which leaves a NaN's sign as it was.
__device__ __forceinline__ unsigned long long rate_bits_of(double r) {
  return ((unsigned long long)(unsigned)(__double2hiint(r) & 0x7FFFFFFF) << 32) | (unsigned)__double2loint(r);
}

// rate over the flagged extrema (see dt_rate_kernel)
__device__ __forceinline__ double crit_rate(const DevModel& m, int dim, double inv_h1, double inv_h2, double kmax,
                                            unsigned long long flags, double rate) {
  const double kd1 = kmax * inv_h1 * inv_h1, kd2 = kmax * inv_h2 * inv_h2;
  for (int d = 0; d < dim; ++d)
    for (int k = 0; k < m.ncrit[d]; ++k)
      if ((flags >> (8 * d + k)) & 1ull)
        rate = tmax(rate, d == 0 ? m.critv[0][k] * inv_h1 + kd1 : m.critv[1][k] * inv_h2 + kd2);
  return rate;
}

// How a CFL rate becomes the step: where the step goes (dt_out), the simulated time it
// advances (t_acc, optional), the end time it is clipped to (t_end > 0) and the count of
// positive steps; crit_dim directions of interior extrema (0 in 3D: there are none).
struct DtFinal {
  int crit_dim;
  double inv_h1, inv_h2, cfl, cfl_diff, kmax, inv_hmin2, t_end;
  double* dt_out;
  double* t_acc;
  double* count;
};

// dt = 1 / max(rate / C, kappa_max / (h_min^2 Cd)); with t_end > 0 clipped to the time
// left after t (0 once less than t_end * 1e-14 is left)
__device__ __forceinline__ double cfl_step(const DevModel& m, const DtFinal& f, unsigned long long rate_bits,
                                           unsigned long long flags, double t) {
  const double rate =
      crit_rate(m, f.crit_dim, f.inv_h1, f.inv_h2, f.kmax, flags, __longlong_as_double((long long)rate_bits));
  double r = rate / f.cfl;
  if (f.cfl_diff > 0.0 && f.kmax > 0.0) r = fmax(r, f.kmax * f.inv_hmin2 / f.cfl_diff);
  double dt = r > 0.0 ? 1.0 / r : 0.0;
  if (f.t_acc && f.t_end > 0.0) {
    const double left = f.t_end - t;
    dt = left > f.t_end * 1e-14 ? fmin(dt, left) : 0.0;
  }
  return dt;
}

// The end of a rate kernel, by thread 0 of each block after its atomics on acc[0] (rate
// bits) and acc[1] (extremum flags): the block that arrives last (ticket acc[2]) forms
// the step, advances the time and resets the accumulators for the next reduction. One
// launch instead of two: the single-thread launch that did this by itself cost 3 us and a
// gap of its own per step.
__device__ __forceinline__ void dt_finish(unsigned long long* acc, const DevModel& m, const DtFinal& f) {
  __threadfence();
  if (atomicAdd(acc + 2, 1ull) != (unsigned long long)gridDim.x - 1ull) return;
  __threadfence();
  const unsigned long long bits = __ldcg(acc), flags = __ldcg(acc + 1);
  const double dt = cfl_step(m, f, bits, flags, f.t_acc ? *f.t_acc : 0.0);
  if (f.t_acc && f.t_end > 0.0 && dt > 0.0) *f.count += 1.0;
  *f.dt_out = dt;
  if (f.t_acc) *f.t_acc += dt;
  acc[0] = acc[1] = acc[2] = 0ull;
}

// The same rate for a flux whose |f_l'| is a nondecreasing function of |u| (Burgers) or a
// constant (linear, zero): rounding is monotone, so the largest rate is the rate at the
// largest |u|. A maximum of the magnitude bits (integer units only) per block, the rate
// formed once per block.
template <int FLUX>
__global__ void __launch_bounds__(RED_THREADS) dt_rate_maxu_kernel(const DevModel m, int dim, int nx, int ny,
                                                                    double inv_h1, double inv_h2, double kmax,
                                                                    const double* __restrict__ ub,
                                                                    unsigned long long* rate_bits, int bc, double gl,
                                                                    double gr, const DtFinal fin) {
  const size_t n = (size_t)nx * ny;
  const double kd1 = kmax * inv_h1 * inv_h1, kd2 = kmax * inv_h2 * inv_h2;
  const bool rect = dim == 2 && bc != AF_BC_PERIODIC;
  unsigned long long mb = 0ull;
  if constexpr (FLUX == FLUX_BURGERS) {
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
      if (rect) {
        const int i = (int)(k % nx), j = (int)(k / nx);
        if (i == 0 || j == 0) continue;
      }
      const unsigned long long b = (unsigned long long)__double_as_longlong(ub[k]) & 0x7FFFFFFFFFFFFFFFull;
      mb = b > mb ? b : mb;
    }
    if (dim == 1 && bc == AF_BC_DIRICHLET && blockIdx.x == 0 && threadIdx.x == 0) {
      const unsigned long long bl = (unsigned long long)__double_as_longlong(gl) & 0x7FFFFFFFFFFFFFFFull;
      const unsigned long long br = (unsigned long long)__double_as_longlong(gr) & 0x7FFFFFFFFFFFFFFFull;
      mb = bl > mb ? bl : mb;
      mb = br > mb ? br : mb;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = v > mb ? v : mb;
  }
  __shared__ unsigned long long smb[RED_THREADS / 32];
  if ((threadIdx.x & 31) == 0) smb[threadIdx.x >> 5] = mb;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < RED_THREADS / 32; ++w) mb = smb[w] > mb ? smb[w] : mb;
    const double u = __longlong_as_double((long long)mb);
    const double a1 = alpha_interval<FLUX, double>(m, 0, u, u), a2 = alpha_interval<FLUX, double>(m, 1, u, u);
    double b = a1 * inv_h1 + kd1;
    if (dim == 2) b = tmax(b, a2 * inv_h2 + kd2);
    atomicMax(rate_bits, (unsigned long long)__double_as_longlong(b));
    dt_finish(rate_bits, m, fin);
  }
}

template <int FLUX>
__global__ void __launch_bounds__(RED_THREADS) dt_rate_kernel(const DevModel m, int dim, int nx, int ny,
                                                               double inv_h1, double inv_h2, double kmax,
                                                               const double* __restrict__ ub,
                                                               unsigned long long* rate_bits, int bc, double gl,
                                                               double gr, const DtFinal fin) {
  static_assert(FLUX == FLUX_BL, "the other fluxes take dt_rate_maxu_kernel");
  unsigned long long best = 0ull;   // magnitude bits of the largest rate
  unsigned flags = 0u;
  const double kd1 = kmax * inv_h1 * inv_h1, kd2 = kmax * inv_h2 * inv_h2;
  const bool rect = dim == 2 && bc != AF_BC_PERIODIC;
  // The cell's rate max_l |f_l'(u)| / h_l + kappa_max / h_l^2 (1D: the gravity form,
  // whose extrema tables sit in slot 0), in FP64 and as an FP32 estimate (within a few
  // ulps). The FP64 one costs a division on GB300's slow FP64 unit, so it is formed only
  // for the cells whose estimate is within 2^-12 of the block's largest estimate: the
  // cell with the largest FP64 rate is always among them, so the maximum is the same.
  // (Finding each cell's coordinates by 64-bit divisions, and estimating every cell twice,
  // had cost most of the kernel: 0.28 ms per step at 4096^2.) An estimate that overflows or
  // is NaN (a NaN average, an average too large for FP32) compares as larger than all
  // others: estimates are reduced by their magnitude bits, the threshold of such a block is
  // NaN and all of its cells are looked at in FP64.
  auto rate64 = [&](double u) {
    const BLVals<double> r = bl_eval<double>(m, u);
    double b = r.d[dim == 1 ? 1 : 0] * inv_h1 + kd1;
    if (dim == 2) b = tmax(b, r.d[1] * inv_h2 + kd2);
    return rate_bits_of(b);
  };
  const float ih1f = (float)inv_h1, ih2f = (float)inv_h2, kd1f = (float)kd1, kd2f = (float)kd2;
  auto rate32 = [&](double u) {
    const BLVals<float> r = bl_eval<float>(m, to_stencil<float>(u));
    float b = r.d[dim == 1 ? 1 : 0] * ih1f + kd1f;
    if (dim == 2) b = fmaxf(b, r.d[1] * ih2f + kd2f);
    return b;
  };
  auto mag32 = [](float v) { return __float_as_uint(v) & 0x7FFFFFFFu; };   // ordered as |v|, NaN above all
  // cells in segments of up to RATE_SEG columns of a row, so that a thread's cells need no
  // division to find their coordinates
  constexpr int RATE_SEG = 4 * RED_THREADS;
  const int spr = (nx + RATE_SEG - 1) / RATE_SEG;   // segments per row
  const long long nseg = (long long)spr * ny;
  auto cells = [&](auto&& f) {
    for (long long sg = blockIdx.x; sg < nseg; sg += gridDim.x) {
      const int j = (int)(sg / spr), b = (int)(sg - (long long)j * spr) * RATE_SEG;
      if (rect && j == 0) continue;
      const int e = min(b + RATE_SEG, nx);
      for (int i = b + (int)threadIdx.x; i < e; i += RED_THREADS)
        if (!(rect && i == 0)) f(i, j, (size_t)j * nx + i);
    }
  };
  auto bits_of = [](double u) { return (unsigned long long)__double_as_longlong(u); };
  unsigned m32 = 0u;   // magnitude bits of the largest estimate
  {
    unsigned long long last = 0ull;   // bits of the last u evaluated
    bool any = false;
    cells([&](int i, int j, size_t k) {
      const double u = ub[k];
      if (!any || bits_of(u) != last) {
        m32 = max(m32, mag32(rate32(u)));
        last = bits_of(u);
        any = true;
      }
      // an extremum lies strictly inside a face's interval only if its ends differ
      double un = ub[(size_t)j * nx + (i + 1 == nx ? 0 : i + 1)];
      if (dim == 1 && bc != AF_BC_PERIODIC && i + 1 == nx) un = bc == AF_BC_DIRICHLET ? gr : u;
      if (rect && i + 1 == nx) un = u;
      if (bits_of(un) != bits_of(u)) flags |= crit_flags<FLUX>(m, 0, u, un);
      if (dim == 1 && bc == AF_BC_DIRICHLET && k == 0) flags |= crit_flags<FLUX>(m, 0, gl, u);
      if (dim == 2) {
        const double ut = (rect && j + 1 == ny) ? u : ub[(size_t)(j + 1 == ny ? 0 : j + 1) * nx + i];
        if (bits_of(ut) != bits_of(u)) flags |= crit_flags<FLUX>(m, 1, u, ut) << 8;
      }
    });
  }
  {
    const float mine = __uint_as_float(m32);   // the largest estimate among this thread's cells
    __shared__ unsigned s32[RED_THREADS / 32];
    m32 = __reduce_max_sync(0xffffffffu, m32);
    if ((threadIdx.x & 31) == 0) s32[threadIdx.x >> 5] = m32;
    __syncthreads();
    for (int w = 0; w < RED_THREADS / 32; ++w) m32 = max(m32, s32[w]);
    const float top = __uint_as_float(m32), thr = top - top * (1.0f / 4096.0f);
    if (!(mine < thr)) {   // only threads with a candidate look at their cells again (NaN: all)
      unsigned long long last = 0ull;
      bool any = false;
      cells([&](int, int, size_t k) {
        const double u = ub[k];
        if (any && bits_of(u) == last) return;
        if (rate32(u) < thr) return;
        last = bits_of(u);
        any = true;
        best = max(best, rate64(u));
      });
    }
  }
  if (dim == 1 && bc == AF_BC_DIRICHLET && blockIdx.x == 0 && threadIdx.x == 0) {
    const double gv[2] = {gl, gr};
    for (int s = 0; s < 2; ++s) best = max(best, rate_bits_of(bl_eval<double>(m, gv[s]).d[1] * inv_h1 + kd1));
  }
  for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
  flags = __reduce_or_sync(0xffffffffu, flags);
  __shared__ unsigned long long sm[RED_THREADS / 32];
  __shared__ unsigned sf[RED_THREADS / 32];
  if ((threadIdx.x & 31) == 0) {
    sm[threadIdx.x >> 5] = best;
    sf[threadIdx.x >> 5] = flags;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long b = sm[0];
    unsigned f = sf[0];
    for (int w = 1; w < RED_THREADS / 32; ++w) {
      b = max(b, sm[w]);
      f |= sf[w];
    }
    atomicMax(rate_bits, b);
    if (f) atomicOr(rate_bits + 1, (unsigned long long)f);
    dt_finish(rate_bits, m, fin);
  }
}

// *dt = v and, when t_acc is given, *t_acc += v
static __global__ void set_dt_kernel(double* dt, double* t_acc, double v) {
  *dt = v;
  if (t_acc) *t_acc += v;
}

// ---- deterministic sum / min / max ------------------------------------------------------
// op 0: sum of x; op 1: min; op 2: max. Each block reduces a contiguous chunk.
__device__ __forceinline__ double red_op(int op, double a, double b) {
  return op == 0 ? a + b : (op == 1 ? fmin(a, b) : fmax(a, b));
}

template <class S>
__global__ void __launch_bounds__(RED_THREADS) partial_kernel(const S* __restrict__ x, size_t n, int op,
                                                              double init, double* partial) {
  const size_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const size_t beg = blockIdx.x * chunk, end = beg + chunk < n ? beg + chunk : n;
  double acc = init;
  for (size_t k = beg + threadIdx.x; k < end; k += RED_THREADS) acc = red_op(op, acc, (double)x[k]);
  __shared__ double sm[RED_THREADS];
  sm[threadIdx.x] = acc;
  __syncthreads();
  for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sm[threadIdx.x] = red_op(op, sm[threadIdx.x], sm[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sm[0];
}

// the same over the entries of a row-major array with rows of width w whose column is
// >= ilo and row >= jlo (the DoFs of a padded 2D rectangle)
template <class S>
__global__ void __launch_bounds__(RED_THREADS) partial_masked_kernel(const S* __restrict__ x, size_t n, int w,
                                                                     int ilo, int jlo, int op, double init,
                                                                     double* partial) {
  const size_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const size_t beg = blockIdx.x * chunk, end = beg + chunk < n ? beg + chunk : n;
  double acc = init;
  for (size_t k = beg + threadIdx.x; k < end; k += RED_THREADS)
    if ((int)(k % w) >= ilo && (int)(k / w) >= jlo) acc = red_op(op, acc, (double)x[k]);
  __shared__ double sm[RED_THREADS];
  sm[threadIdx.x] = acc;
  __syncthreads();
  for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sm[threadIdx.x] = red_op(op, sm[threadIdx.x], sm[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sm[0];
}

// combine nparts partials into *out (op as above; combined with the existing *out when
// accumulate != 0). One block of RED_THREADS: thread t folds partials t, t + RED_THREADS,
// ... in order, then a fixed tree; the result depends only on nparts and the partials.
static __global__ void __launch_bounds__(RED_THREADS) finalize_kernel(const double* partial, int nparts, int op,
                                                                      double* out, int accumulate) {
  __shared__ double sm[RED_THREADS];
  const int t = threadIdx.x;
  // partial[0] is neutral for min/max over a set that contains it
  double acc = op == 0 ? 0.0 : partial[0];
  for (int k = t; k < nparts; k += RED_THREADS) acc = red_op(op, acc, partial[k]);
  sm[t] = acc;
  __syncthreads();
  for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
    if (t < s) sm[t] = red_op(op, sm[t], sm[t + s]);
    __syncthreads();
  }
  if (t == 0) *out = accumulate ? red_op(op, *out, sm[0]) : sm[0];
}

}  // namespace af
