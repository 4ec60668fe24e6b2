// stage_fp64.cuh -- FP64 kernels of one Runge-Kutta stage of the IB-WENO/TENO method
// (arXiv:1905.00182, Sec. 2).  Included twice: once with IBFSA_STRICT = 1 and --fmad=false
// (every operation rounded separately, in the order the formulas are written below, quotients
// rounded as divisions, spreading summed in marker order), once with IBFSA_STRICT = 0 (fused
// multiply-add, reciprocals, atomic spreading).
//
// Per stage:  pad (ghosts + primitives + split speeds)  ->  IB interpolation and penalty force
//   (Eq. 7-8)  ->  convective flux differences x, y, z  ->  viscous fluxes and their divergence
//   (Eq. 2-5)  ->  IB spreading (Eq. 9)  ->  finish (sponge, IB source, RK combination).
// The fast form interpolates and spreads in one kernel between the convective and the viscous terms
// (unless the caller waits for the forces) and takes the viscous divergence in finish.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fp_bits.cuh"
#include "ibfsa_internal.h"
#include "launch.cuh"
#include "marker.cuh"
#include "mesh.cuh"

#ifndef IBFSA_STRICT
#error "define IBFSA_STRICT to 0 or 1"
#endif

namespace ibfsa {
namespace IBFSA_MODE_NS {

constexpr bool STRICT = IBFSA_STRICT != 0;
constexpr int THREADS = 256;

// ------------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------------
// x / d given inv_d = 1/d correctly rounded.  Strict: the correctly rounded quotient without the
// divider, by Markstein's theorem: from a q within an ulp of x/d, RN(q + inv_d RN(x - d q)) is
// x/d correctly rounded (the remainder is exact, its product a correction far below an ulp).  One
// such step brings x inv_d within an ulp of x/d, the second rounds it: 5 FP64 operations against
// ~9.  The divider outside the exponents where nothing over- or underflows on the way.
__device__ __forceinline__ double divide(double x, double d, double inv_d) {
  if constexpr (STRICT) {
    const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    const unsigned ed = ((unsigned)__double2hiint(d) >> 20) & 0x7ffu;
    if (ex - 600u < 900u && ed - 723u < 600u) {
      double q = x * inv_d;
      q = __fma_rn(__fma_rn(-d, q, x), inv_d, q);
      return __fma_rn(__fma_rn(-d, q, x), inv_d, q);
    }
    return x == 0.0 && ed - 723u < 600u ? x * inv_d : x / d;
  } else {
    return x * inv_d;
  }
}

// x / 6 in the same way; the rounded sixth is within a quarter of an ulp (2^-54 relative), so the
// product is already within an ulp and one step rounds it: 3 operations
__device__ __forceinline__ double divide6(double x) {
  const double r = 1.0 / 6.0;
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  if (ex - 600u < 900u) {
    const double q = x * r;
    return __fma_rn(__fma_rn(-6.0, q, x), r, q);
  }
  return x == 0.0 ? x * r : x / 6.0;
}

// ghost rule of one direction: interior index, or -1 for a free-stream ghost
__device__ __forceinline__ int map_index(int i, int n, int rlo, int rhi) {
  if (i < 0) {
    if (rlo == IBFSA_BC_ZERO_GRAD || rlo == IBFSA_BC_CHARACTERISTIC) return 0;
    if (rlo == IBFSA_BC_PERIODIC) return n + i;
    return -1;
  }
  if (i >= n) {
    if (rhi == IBFSA_BC_ZERO_GRAD || rhi == IBFSA_BC_CHARACTERISTIC) return n - 1;
    if (rhi == IBFSA_BC_PERIODIC) return i - n;
    return -1;
  }
  return i;
}

// the boundary cell of a characteristic face along a (its normal term comes from k_char_faces)
__device__ __forceinline__ bool char_cell(const Plan &p, int a, int i) {
  return (i == 0 && p.bc[a][0] == IBFSA_BC_CHARACTERISTIC) ||
         (i == p.n[a] - 1 && p.bc[a][1] == IBFSA_BC_CHARACTERISTIC);
}

__device__ __forceinline__ long long pad_index(const Plan &p, int i, int j, int k) {
  return ((long long)(k + p.g[2]) * p.P[1] + (j + p.g[1])) * (long long)p.P[0] + (i + p.g[0]);
}

__device__ __forceinline__ long long int_index(const Plan &p, int i, int j, int k) {
  return ((long long)k * p.n[1] + j) * (long long)p.n[0] + i;
}

__device__ __forceinline__ double load_alpha(const Plan &p, int a) {
  return __longlong_as_double((long long)p.alpha_bits[a]);
}

// first of the four support nodes of position x along direction a, and their weights
__device__ __forceinline__ int support(const Plan &p, int a, double x, double w[4]) {
  double s = divide(x - p.lo[a], p.h[a], p.inv_h[a]) - 0.5;
  int j0 = (int)floor(s) - 1;
#pragma unroll
  for (int r = 0; r < 4; r++) w[r] = marker::peskin(s - (double)(j0 + r));
  return j0;
}

// ------------------------------------------------------------------------------------------
// fifth-order reconstruction at face i+1/2 from (f_{i-2}, ..., f_{i+2})
// ------------------------------------------------------------------------------------------
struct Cands {
  double q0, q1, q2, b0, b1, b2;
};

__device__ __forceinline__ Cands candidates(double a, double b, double c, double d, double e) {
  Cands r;
  // third-order candidates on {i-2..i}, {i-1..i+1}, {i..i+2}
  if constexpr (STRICT) {
    r.q0 = (2.0 * a - 7.0 * b + 11.0 * c) / 6.0;
    r.q1 = (-b + 5.0 * c + 2.0 * d) / 6.0;
    r.q2 = (2.0 * c + 5.0 * d - e) / 6.0;
  } else {
    const double s6 = 1.0 / 6.0;
    r.q0 = (2.0 * a - 7.0 * b + 11.0 * c) * s6;
    r.q1 = (-b + 5.0 * c + 2.0 * d) * s6;
    r.q2 = (2.0 * c + 5.0 * d - e) * s6;
  }
  // Jiang-Shu smoothness indicators
  double t;
  t = a - 2.0 * b + c;       r.b0 = 13.0 / 12.0 * t * t;
  t = a - 4.0 * b + 3.0 * c; r.b0 += 0.25 * t * t;
  t = b - 2.0 * c + d;       r.b1 = 13.0 / 12.0 * t * t;
  t = b - d;                 r.b1 += 0.25 * t * t;
  t = c - 2.0 * d + e;       r.b2 = 13.0 / 12.0 * t * t;
  t = 3.0 * c - 4.0 * d + e; r.b2 += 0.25 * t * t;
  return r;
}

// WENO5-JS: alpha_k = d_k / (1e-6 + beta_k)^2, omega = alpha / sum alpha, d = (0.1, 0.6, 0.3)
__device__ __forceinline__ double weno5js(double a, double b, double c, double d, double e) {
  Cands k = candidates(a, b, c, d, e);
  const double eps = 1e-6;
  if constexpr (STRICT) {
    double al0 = 0.1 / ((eps + k.b0) * (eps + k.b0));
    double al1 = 0.6 / ((eps + k.b1) * (eps + k.b1));
    double al2 = 0.3 / ((eps + k.b2) * (eps + k.b2));
    double s = al0 + al1 + al2;
    return (al0 / s) * k.q0 + (al1 / s) * k.q1 + (al2 / s) * k.q2;
  } else {
    // common denominator: alpha_k proportional to d_k prod_{j != k} (eps + beta_j)^2
    double s0 = (eps + k.b0) * (eps + k.b0);
    double s1 = (eps + k.b1) * (eps + k.b1);
    double s2 = (eps + k.b2) * (eps + k.b2);
    double al0 = 0.1 * (s1 * s2), al1 = 0.6 * (s0 * s2), al2 = 0.3 * (s0 * s1);
    return (al0 * k.q0 + al1 * k.q1 + al2 * k.q2) / (al0 + al1 + al2);
  }
}

// TENO5: gamma_k = (1 + tau5/(beta_k + 1e-40))^6, tau5 = |beta_0 - beta_2|; stencil k kept when
// gamma_k / sum gamma >= 1e-5; omega = normalised linear weights of the kept stencils
__device__ __forceinline__ int teno_keep(const Cands &k) {
  const double eps = 1e-40, CT = 1e-5;
  double tau5 = fabs(k.b0 - k.b2);
  double g0, g1, g2;
  int mask;
  if constexpr (STRICT) {
    double x, x2;
    x = 1.0 + tau5 / (k.b0 + eps); x2 = x * x; g0 = x2 * x2 * x2;
    x = 1.0 + tau5 / (k.b1 + eps); x2 = x * x; g1 = x2 * x2 * x2;
    x = 1.0 + tau5 / (k.b2 + eps); x2 = x * x; g2 = x2 * x2 * x2;
    double s = g0 + g1 + g2;
    mask = ((g0 / s) >= CT ? 1 : 0) | ((g1 / s) >= CT ? 2 : 0) | ((g2 / s) >= CT ? 4 : 0);
  } else {
    double e0 = k.b0 + eps, e1 = k.b1 + eps, e2 = k.b2 + eps;
    double r = tau5 / (e0 * e1 * e2);
    double x, x2;
    x = 1.0 + r * (e1 * e2); x2 = x * x; g0 = x2 * x2 * x2;
    x = 1.0 + r * (e0 * e2); x2 = x * x; g1 = x2 * x2 * x2;
    x = 1.0 + r * (e0 * e1); x2 = x * x; g2 = x2 * x2 * x2;
    double th = CT * (g0 + g1 + g2);
    mask = (g0 >= th ? 1 : 0) | (g1 >= th ? 2 : 0) | (g2 >= th ? 4 : 0);
  }
  return mask;
}

__device__ __forceinline__ double teno5(const Plan &p, double a, double b, double c, double d,
                                        double e) {
  const Cands k = candidates(a, b, c, d, e);
  const double *w = p.teno_w[teno_keep(k)];
  return w[0] * k.q0 + w[1] * k.q1 + w[2] * k.q2;
}

// TENO5 keeps every stencil when tau5 <= 4 (min beta + eps) -- each gamma_k lies in [1, 5^6], so
// chi_k >= 1/(3 5^6) = 2.1e-5 > C_T -- and its weights are then the linear ones.  Only this
// sufficient test is taken in FP32 (the FP64 pipe is the bound), from the stencil's four FP64
// first differences d: t0 = d1 - d0, u0 = 3 d1 - d0, t1 = d2 - d1, u1 = d1 + d2, t2 = d3 - d2,
// u2 = d3 - 3 d2, indicators times 4, kt_k = (13/3) t_k^2 plus u_k^2.  Each indicator is a
// positive definite form of its two differences, so its relative error stays a few 1e-7 (where t
// or u cancels, the other term dominates) -- far inside the test's factor-2 margin in chi_k: a
// stencil the test keeps is one TENO5 keeps; where the test fails (or anything is not finite),
// the FP64 TENO5 decides.  Reversing the stencil swaps the outer indicators and leaves the test.
// Fast form: differences below FP32's range flush to zero and pass; their stencils vary by less
// than 1e-17 of the flux, whatever TENO5 would cut.  Strict form: its indicators carry the
// rounding of a - 4b + 3c and the like, up to 1e-15 |f| in their square roots, so the test passes
// only where the smallest is at least (2e-13 c)^2 (c the stencil's middle value; an indicator is
// at least 0.98 of its squared differences, so values much larger than c imply a larger one) and
// well inside FP32's range.
__device__ __forceinline__ bool all_kept(float d0, float d1, float d2, float d3, float kt0,
                                         float kt1, float kt2, double c) {
  const float u0 = fmaf(3.f, d1, -d0), u1 = d1 + d2, u2 = fmaf(-3.f, d2, d3);
  const float b0 = fmaf(u0, u0, kt0), b1 = fmaf(u1, u1, kt1), b2 = fmaf(u2, u2, kt2);
  const float m = fminf(b0, fminf(b1, b2));
  if constexpr (STRICT)
    return fabsf(b0 - b2) <= 4.f * m &&
           m >= fmaxf(1e-35f, 4e-26f * low_precision(c) * low_precision(c));
  else
    return fabsf(b0 - b2) <= fmaf(4.f, m, 1.6e-29f);
}

// Strict form, constant stencil (quiescent fluid): every difference and the first two indicators
// are exactly zero; the third carries the rounding of 3c, r = (3c - 4c) + c, beta2 = r^2 / 4.
// r = 0: all stencils kept (7).  |r| > 1e-18: tau5 / (0 + 1e-40) > 2000, so the third stencil's
// weight, at most 64 of 2 (2000)^6, is cut and the others' are near a half (3).  Otherwise, or if
// the stencil is not constant: -1.
__device__ __forceinline__ int constant_mask(double d0, double d1, double d2, double d3, double c) {
  const unsigned long long any =
      (unsigned long long)(__double_as_longlong(d0) | __double_as_longlong(d1) |
                           __double_as_longlong(d2) | __double_as_longlong(d3));
  if (any << 1) return -1;
  const double r = 3.0 * c - 4.0 * c + c;
  return r == 0.0 ? 7 : fabs(r) > 1e-18 ? 3 : -1;
}

// Reconstruction at K consecutive faces of one line from one side's split fluxes f[0 .. K+3]
// (in increasing cell index): face j from f[j .. j+4], upwind to downwind (REV: downwind to
// upwind).  What neighbouring faces share is taken once: first differences, second differences
// and their squares.  Of the 12 FP64 operations a TENO5 face took by itself (four differences,
// four conversions, four fused multiply-adds) 4 + (K + 3)/K remain; WENO5-JS goes from 62 to 38.
// strict: every value the oracle computes is computed by the same roundings, once instead of for
// each face that uses it, and TENO5's weights are looked up without its divisions where the
// sufficient test above proves that it keeps every stencil.  Returns the faces (bit j) whose
// stencil neither passes that test nor is constant: the caller replaces their h by teno5.
template <int SCHEME, bool REV, int K>
__device__ __forceinline__ unsigned faces_of_line(const Plan &p, const double (&f)[K + 4],
                                                  double (&h)[K]) {
  unsigned fail = 0;
  if constexpr (SCHEME == IBFSA_TENO5) {
    double d[K + 3];
    float s[K + 3], kt[K + 2];
#pragma unroll
    for (int j = 0; j < K + 3; j++) {
      d[j] = f[j + 1] - f[j];
      s[j] = low_precision(d[j]);
    }
#pragma unroll
    for (int j = 0; j < K + 2; j++) {
      const float t = s[j + 1] - s[j];
      kt[j] = (13.f / 3.f) * t * t;
    }
#pragma unroll
    for (int j = 0; j < K; j++) {
      const double a = f[REV ? j + 4 : j], b = f[REV ? j + 3 : j + 1], c = f[j + 2];
      const double dd = f[REV ? j + 1 : j + 3], e = f[REV ? j : j + 4];
      const bool keep = all_kept(s[j], s[j + 1], s[j + 2], s[j + 3], kt[j], kt[j + 1], kt[j + 2], c);
      if constexpr (STRICT) {
        int mask = 7;
        if (!keep) {
          mask = constant_mask(d[j], d[j + 1], d[j + 2], d[j + 3], c);
          if (mask < 0) fail |= 1u << j;
        }
        const double *w = p.teno_w[mask & 7];
        const double q0 = divide6(2.0 * a - 7.0 * b + 11.0 * c);
        const double q1 = divide6(-b + 5.0 * c + 2.0 * dd);
        const double q2 = divide6(2.0 * c + 5.0 * dd - e);
        h[j] = w[0] * q0 + w[1] * q1 + w[2] * q2;
      } else {
        if (!keep) fail |= 1u << j;
        // the linear combination (2a - 13b + 47c + 27d - 3e)/60 as c plus its differences: four
        // fused multiply-adds, and a constant stencil gives c exactly
        const double sg = REV ? -1.0 : 1.0;
        const double e1 = d[REV ? j + 3 : j], e2 = d[REV ? j + 2 : j + 1];
        const double e3 = d[REV ? j + 1 : j + 2], e4 = d[REV ? j : j + 3];
        h[j] = fma(sg * -3.0 / 60.0, e4,
                   fma(sg * 24.0 / 60.0, e3, fma(sg * 11.0 / 60.0, e2, fma(sg * -2.0 / 60.0, e1, c))));
      }
    }
  } else if constexpr (STRICT) {
    // kt[j] of the triple f[j], f[j+1], f[j+2], its second difference rounded in the order the
    // stencil's direction gives
    double kt[K + 2];
#pragma unroll
    for (int j = 0; j < K + 2; j++) {
      const double t = REV ? f[j + 2] - 2.0 * f[j + 1] + f[j] : f[j] - 2.0 * f[j + 1] + f[j + 2];
      kt[j] = 13.0 / 12.0 * t * t;
    }
#pragma unroll
    for (int j = 0; j < K; j++) {
      const double a = f[REV ? j + 4 : j], b = f[REV ? j + 3 : j + 1], c = f[j + 2];
      const double d = f[REV ? j + 1 : j + 3], e = f[REV ? j : j + 4];
      const double eps = 1e-6;
      double t;
      t = a - 4.0 * b + 3.0 * c;
      const double b0 = kt[REV ? j + 2 : j] + 0.25 * t * t;
      t = b - d;
      const double b1 = kt[j + 1] + 0.25 * t * t;
      t = 3.0 * c - 4.0 * d + e;
      const double b2 = kt[REV ? j : j + 2] + 0.25 * t * t;
      const double al0 = 0.1 / ((eps + b0) * (eps + b0));
      const double al1 = 0.6 / ((eps + b1) * (eps + b1));
      const double al2 = 0.3 / ((eps + b2) * (eps + b2));
      const double s = al0 + al1 + al2;
      h[j] = (al0 / s) * divide6(2.0 * a - 7.0 * b + 11.0 * c) +
             (al1 / s) * divide6(-b + 5.0 * c + 2.0 * d) + (al2 / s) * divide6(2.0 * c + 5.0 * d - e);
    }
  } else {
    // S_k = 4 (eps + beta_k), weights d_k / S_k^2 over their common denominator, the
    // reconstruction as c plus a weighted mean of the candidates' differences from c
    double d[K + 3], kt[K + 2];
#pragma unroll
    for (int j = 0; j < K + 3; j++) d[j] = f[j + 1] - f[j];
#pragma unroll
    for (int j = 0; j < K + 2; j++) {
      const double t = d[j + 1] - d[j];
      kt[j] = fma(13.0 / 3.0 * t, t, 4e-6);
    }
#pragma unroll
    for (int j = 0; j < K; j++) {
      const double sg = REV ? -1.0 : 1.0;
      const double e1 = sg * d[REV ? j + 3 : j], e2 = sg * d[REV ? j + 2 : j + 1];
      const double e3 = sg * d[REV ? j + 1 : j + 2], e4 = sg * d[REV ? j : j + 3];
      const double u0 = fma(3.0, e2, -e1), u1 = e2 + e3, u2 = fma(-3.0, e3, e4);
      double s0 = fma(u0, u0, kt[REV ? j + 2 : j]), s1 = fma(u1, u1, kt[j + 1]);
      double s2 = fma(u2, u2, kt[REV ? j : j + 2]);
      s0 *= s0;
      s1 *= s1;
      s2 *= s2;
      const double p0 = s1 * s2, p1 = s0 * s2, p2 = s0 * s1;  // weights p0 : 6 p1 : 3 p2
      const double x3 = 12.0 * e3;
      const double n0 = fma(5.0, e2, -2.0 * e1), n1 = fma(6.0, e2, x3), n2 = fma(-3.0, e4, x3);
      const double num = fma(p2, n2, fma(p1, n1, p0 * n0));  // 6 (candidate - c), weighted
      const double den = fma(18.0, p2, fma(36.0, p1, 6.0 * p0));
      h[j] = f[j + 2] + num / den;
    }
  }
  return fail;
}

template <int SCHEME>
__device__ __forceinline__ double recon(const Plan &p, double a, double b, double c, double d,
                                        double e) {
  if constexpr (SCHEME == IBFSA_TENO5 && !STRICT) {
    const double f[5] = {a, b, c, d, e};
    double h[1];
    return faces_of_line<IBFSA_TENO5, false, 1>(p, f, h) ? teno5(p, a, b, c, d, e) : h[0];
  } else if constexpr (SCHEME == IBFSA_TENO5) {
    return teno5(p, a, b, c, d, e);
  } else {
    return weno5js(a, b, c, d, e);
  }
}

// ------------------------------------------------------------------------------------------
// pad: ghost fill by index mapping, primitives on the padded grid, split speeds
// ------------------------------------------------------------------------------------------
template <int DIM>
__global__ void __launch_bounds__(THREADS) k_pad(Plan p, const double *__restrict__ Q) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double wmax[3] = {0.0, 0.0, 0.0};
  double c2 = 0.0, ua[3] = {0.0, 0.0, 0.0};  // fast form: c^2 and |u_a| of an interior cell
  bool have = false;
  if (t < p.NP) {
    int ix = (int)(t % p.P[0]);
    long long r = t / p.P[0];
    int iy = (int)(r % p.P[1]);
    int iz = (int)(r / p.P[1]);
    int I[3] = {ix - p.g[0], iy - p.g[1], iz - p.g[2]};
    bool free_ghost = false, interior = true;
    int S[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
      if (a < DIM) {
        S[a] = map_index(I[a], p.n[a], p.bc[a][0], p.bc[a][1]);
        if (S[a] < 0) free_ghost = true;
        if (I[a] < 0 || I[a] >= p.n[a]) interior = false;
      } else {
        S[a] = 0;
      }
    }
    double q[NV];
    if (free_ghost) {
#pragma unroll
      for (int c = 0; c < NV; c++) q[c] = p.qinf[c];
    } else {
      long long o = int_index(p, S[0], S[1], S[2]);
#pragma unroll
      for (int c = 0; c < NV; c++) q[c] = Q[c * p.N + o];
    }
#pragma unroll
    for (int c = 0; c < NV; c++) p.Qp[c * p.NP + t] = q[c];
    double rho = q[0];
    double ke = 0.0, u[DIM];
    // one reciprocal of rho (strict: the quotients rounded as divisions, see divide)
    const double inv_rho = 1.0 / rho;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      u[a] = divide(q[1 + a], rho, inv_rho);
      ke += q[1 + a] * u[a];
      p.Wp[a * p.NP + t] = u[a];
    }
    double pr = p.gm1 * (q[NV - 1] - 0.5 * ke);
    p.Wp[DIM * p.NP + t] = pr;
    if (interior) {
      if constexpr (STRICT) {
        const double c = sqrt(divide(p.gamma * pr, rho, inv_rho));
#pragma unroll
        for (int a = 0; a < DIM; a++) wmax[a] = fabs(u[a]) + c;
      } else {
        c2 = p.gamma * pr * inv_rho;
#pragma unroll
        for (int a = 0; a < DIM; a++) ua[a] = fabs(u[a]);
        have = true;
      }
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if constexpr (!STRICT) {
    // The block's maxima in FP32 first: the FP64 sound speed is taken only where |u| + c in
    // FP32 lies within 2e-6 of the block's FP32 maximum (their relative errors, and that of
    // the threshold, stay below 3e-7, so the cell of the exact maximum is among them); the
    // other cells give 0 -- the same FP64 maxima for a fraction of the square roots.  A value
    // beyond FP32's range gives NaN there, and its cell takes the FP64 speed.  Sound speeds below
    // 1.1e-19 give 0, less than 1.1e-7 of maxima of 1e-12 and more; in a block of smaller speeds
    // every cell takes the FP64 speed.
    __shared__ float red32[3][THREADS / 32];
    const float c32 = have ? sqrtf(low_precision(c2)) : 0.f;
    float ua32[3];
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      ua32[a] = low_precision(ua[a]);
      float v = have ? ua32[a] + c32 : 0.f;
      for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (lane == 0) red32[a][wid] = v;
    }
    __syncthreads();
    float m32[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < DIM; a++)
      for (int w = 0; w < THREADS / 32; w++) m32[a] = fmaxf(m32[a], red32[a][w]);
    bool near = false;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const float far = m32[a] < 1e-12f ? 0.f : m32[a] * (1.f - 2e-6f);
      near |= have && !(ua32[a] + c32 < far);  // NaN counts as near
    }
    if (near) {
      const double c = sqrt(c2);
#pragma unroll
      for (int a = 0; a < DIM; a++) wmax[a] = ua[a] + c;
    }
  }
  // block max of the (non-negative) speeds on their bits (the order of non-negative doubles is
  // that of their bit patterns; a NaN's pattern exceeds every finite one), then one atomic per
  // block
  __shared__ unsigned long long red[3][THREADS / 32];
#pragma unroll
  for (int a = 0; a < DIM; a++) {
    unsigned long long v = (unsigned long long)__double_as_longlong(wmax[a]);
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
      v = w > v ? w : v;
    }
    if (lane == 0) red[a][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < DIM) {
    unsigned long long b = 0;
    for (int w = 0; w < THREADS / 32; w++) b = red[threadIdx.x][w] > b ? red[threadIdx.x][w] : b;
    const double v = __longlong_as_double((long long)b);
    if (!(v <= 1e300)) atomicOr(p.status, IBFSA_STATUS_NONFINITE);
    else atomicMax(&p.alpha_bits[threadIdx.x], b);
  }
}

// ------------------------------------------------------------------------------------------
// convective term along direction A
// ------------------------------------------------------------------------------------------
// ------------------------------------------------------------------------------------------
// characteristic-wise option: eigenvectors of the Euler flux Jacobian along A at the Roe
// average of the face's two cells (sqrt(rho)-weighted velocity and total enthalpy).  Right
// eigenvectors are the columns of R, left ones the rows of Lv, in the order u-c, entropy,
// shears (transverse directions in increasing order), u+c.  Written operation by operation in
// the order of the formulas, so that the strict form is reproducible.
// ------------------------------------------------------------------------------------------
template <int DIM, int A>
__device__ __forceinline__ void roe_eigen(const Plan &p, const double *Ql, const double *Qr,
                                          double R[DIM + 2][DIM + 2],
                                          double Lv[DIM + 2][DIM + 2]) {
  constexpr int NV = DIM + 2;
  const double gm1 = p.gm1;
  double sl = sqrt(Ql[0]), sr = sqrt(Qr[0]);
  double u[DIM], kel = 0.0, ker = 0.0;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    double ul = Ql[1 + b] / Ql[0], ur = Qr[1 + b] / Qr[0];
    u[b] = (sl * ul + sr * ur) / (sl + sr);
    kel = kel + Ql[1 + b] * ul;
    ker = ker + Qr[1 + b] * ur;
  }
  double pl = gm1 * (Ql[NV - 1] - 0.5 * kel);
  double pr = gm1 * (Qr[NV - 1] - 0.5 * ker);
  double Hl = (Ql[NV - 1] + pl) / Ql[0], Hr = (Qr[NV - 1] + pr) / Qr[0];
  double H = (sl * Hl + sr * Hr) / (sl + sr);
  double q2 = 0.0;
#pragma unroll
  for (int b = 0; b < DIM; b++) q2 = q2 + u[b] * u[b];
  double c2 = gm1 * (H - 0.5 * q2);
  double c = sqrt(c2);
  double b1 = gm1 / c2, b2 = 0.5 * q2 * b1;
  double ua = u[A];
#pragma unroll
  for (int i = 0; i < NV; i++)
#pragma unroll
    for (int j = 0; j < NV; j++) {
      R[i][j] = 0.0;
      Lv[i][j] = 0.0;
    }
  constexpr int km = 0, ke = 1, kp = NV - 1;
  R[0][km] = 1.0;
  R[0][ke] = 1.0;
  R[0][kp] = 1.0;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    R[1 + b][km] = u[b] - (b == A ? c : 0.0);
    R[1 + b][ke] = u[b];
    R[1 + b][kp] = u[b] + (b == A ? c : 0.0);
  }
  R[NV - 1][km] = H - ua * c;
  R[NV - 1][ke] = 0.5 * q2;
  R[NV - 1][kp] = H + ua * c;
  Lv[km][0] = 0.5 * (b2 + ua / c);
  Lv[kp][0] = 0.5 * (b2 - ua / c);
  Lv[ke][0] = 1.0 - b2;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    Lv[km][1 + b] = 0.5 * (-b1 * u[b] - (b == A ? 1.0 / c : 0.0));
    Lv[kp][1 + b] = 0.5 * (-b1 * u[b] + (b == A ? 1.0 / c : 0.0));
    Lv[ke][1 + b] = b1 * u[b];
  }
  Lv[km][NV - 1] = 0.5 * b1;
  Lv[kp][NV - 1] = 0.5 * b1;
  Lv[ke][NV - 1] = -b1;
  int t = 0;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    if (b == A) continue;
    R[1 + b][2 + t] = 1.0;
    R[NV - 1][2 + t] = u[b];
    Lv[2 + t][0] = -u[b];
    Lv[2 + t][1 + b] = 1.0;
    t++;
  }
}

template <int A>
struct ConvTile {
  // A == 0: 4 lines (y/z) of 63 cells; otherwise 32 lines (consecutive x) of 15 cells
  static constexpr int ROWS = A == 0 ? 4 : 32;
  static constexpr int SEG = A == 0 ? 63 : 15;
  static constexpr int LEN = SEG + 6;          // cells staged per line
  static constexpr int FACES = SEG + 1;        // faces per line
  static constexpr int PASSES = (ROWS * FACES + THREADS - 1) / THREADS;
};

template <int DIM, int A>
__host__ __device__ constexpr size_t conv_smem_bytes() {
  return sizeof(double) * 2 * (DIM + 2) * ConvTile<A>::ROWS * ConvTile<A>::LEN;
}

// characteristic-wise: split fluxes of a tile of lines staged in shared memory, one face per
// thread per pass, conservative difference into L
template <int DIM, int A, int SCHEME>
__global__ void __launch_bounds__(THREADS) k_conv_char(Plan p, int first) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  using T = ConvTile<A>;
  extern __shared__ double sm[];
  double *sfp = sm;                              // [NV][ROWS][LEN]
  double *sfm = sm + NV * T::ROWS * T::LEN;      // [NV][ROWS][LEN]
  const double alpha = load_alpha(p, A);

  // tile origin
  int seg0, line0, other;
  if constexpr (A == 0) {
    seg0 = blockIdx.x * T::SEG;
    line0 = blockIdx.y * T::ROWS;   // y of the first line
    other = blockIdx.z;             // z
  } else {
    const unsigned nseg = (p.n[A] + T::SEG - 1) / T::SEG;
    // blocks start in the order of x, y: the line tiles slowest, so that the short last ones, which
    // take less time, come after all full ones (33^3, a step: 2.13 -> 1.95 ms)
    const unsigned id = blockIdx.y * gridDim.x + blockIdx.x, rest = id / nseg;
    seg0 = (int)(id % nseg) * T::SEG;
    line0 = (int)(rest / gridDim.y) * T::ROWS;  // x of the first line
    other = (int)(rest % gridDim.y);            // z for A = 1, y for A = 2
  }
  auto cell_of = [&](int row, int l, int I[3]) -> bool {
    // row-th line of the tile, position l along A (tile-relative, may be negative)
    if constexpr (A == 0) {
      int y = line0 + row;
      if (y >= p.n[1]) return false;
      I[0] = seg0 + l;
      I[1] = y;
      I[2] = other;
    } else {
      int x = line0 + row;
      if (x >= p.n[0]) return false;
      I[0] = x;
      I[A] = seg0 + l;
      I[A == 1 ? 2 : 1] = other;
    }
    return true;
  };

  // 1. split fluxes f+- = (F_A(Q) +- alpha Q)/2 of the staged cells
  for (int e = threadIdx.x; e < T::ROWS * T::LEN; e += THREADS) {
    int row, l;
    if constexpr (A == 0) { row = e / T::LEN; l = e % T::LEN; }
    else { row = e % T::ROWS; l = e / T::ROWS; }
    int I[3];
    bool ok = cell_of(row, l - 3, I);
    if (ok && I[A] > p.n[A] + 2) ok = false;
    if (ok) {
      long long s = pad_index(p, I[0], I[1], I[2]);
      double ua = p.Wp[A * p.NP + s];
      double pr = p.Wp[DIM * p.NP + s];
#pragma unroll
      for (int c = 0; c < NV; c++) {
        double q = p.Qp[c * p.NP + s];
        double F;
        if (c == 0) F = p.Qp[(1 + A) * p.NP + s];
        else if (c == NV - 1) F = (q + pr) * ua;
        else {
          F = q * ua;
          if (c - 1 == A) F += pr;
        }
        sfp[(c * T::ROWS + row) * T::LEN + l] = 0.5 * (F + alpha * q);
        sfm[(c * T::ROWS + row) * T::LEN + l] = 0.5 * (F - alpha * q);
      }
    } else {
#pragma unroll
      for (int c = 0; c < NV; c++) {
        sfp[(c * T::ROWS + row) * T::LEN + l] = 0.0;
        sfm[(c * T::ROWS + row) * T::LEN + l] = 0.0;
      }
    }
  }
  __syncthreads();

  // 2. faces m+1/2 for m = seg0-1 .. seg0+SEG-1 (tile-relative face index fi = m - seg0 + 1)
  double Fh[T::PASSES][NV];
#pragma unroll
  for (int ps = 0; ps < T::PASSES; ps++) {
    int e = threadIdx.x + ps * THREADS;
    if (e < T::ROWS * T::FACES) {
      int row, fi;
      if constexpr (A == 0) { row = e / T::FACES; fi = e % T::FACES; }
      else { row = e % T::ROWS; fi = e / T::ROWS; }
      // staged index of cell m is (m - seg0) + 3 = fi + 2
      int b = fi + 2;
      // characteristic fields of the stencil at the Roe average of cells m and m+1 (only
      // the faces -1/2 .. n-1/2 are used)
      int I[3];
      bool ok = cell_of(row, fi - 1, I) && I[A] <= p.n[A] - 1;
      if (ok) {
        long long sl = pad_index(p, I[0], I[1], I[2]);
        I[A] += 1;
        long long sr = pad_index(p, I[0], I[1], I[2]);
        double Ql[NV], Qr[NV];
#pragma unroll
        for (int c = 0; c < NV; c++) {
          Ql[c] = p.Qp[c * p.NP + sl];
          Qr[c] = p.Qp[c * p.NP + sr];
        }
        double R[NV][NV], Lv[NV][NV];
        roe_eigen<DIM, A>(p, Ql, Qr, R, Lv);
        double hk[NV];
#pragma unroll
        for (int k = 0; k < NV; k++) {
          double vp[5], vm[5];
#pragma unroll
          for (int r = 0; r < 5; r++) {
            double sp = 0.0, sn = 0.0;
#pragma unroll
            for (int c = 0; c < NV; c++) {
              const double *fp = sfp + (c * T::ROWS + row) * T::LEN;
              const double *fm = sfm + (c * T::ROWS + row) * T::LEN;
              sp = sp + Lv[k][c] * fp[b - 2 + r];
              sn = sn + Lv[k][c] * fm[b + 3 - r];
            }
            vp[r] = sp;
            vm[r] = sn;
          }
          hk[k] = recon<SCHEME>(p, vp[0], vp[1], vp[2], vp[3], vp[4]) +
                  recon<SCHEME>(p, vm[0], vm[1], vm[2], vm[3], vm[4]);
        }
#pragma unroll
        for (int c = 0; c < NV; c++) {
          double acc = 0.0;
#pragma unroll
          for (int k = 0; k < NV; k++) acc = acc + R[c][k] * hk[k];
          Fh[ps][c] = acc;
        }
      } else {
#pragma unroll
        for (int c = 0; c < NV; c++) Fh[ps][c] = 0.0;
      }
    }
  }
  __syncthreads();
  constexpr int FST = A == 0 ? T::FACES : T::FACES + 1;  // odd stride when lanes walk rows
  double *sh = sm;  // reuse: face fluxes [NV][ROWS][FST]
#pragma unroll
  for (int ps = 0; ps < T::PASSES; ps++) {
    int e = threadIdx.x + ps * THREADS;
    if (e < T::ROWS * T::FACES) {
      int row, fi;
      if constexpr (A == 0) { row = e / T::FACES; fi = e % T::FACES; }
      else { row = e % T::ROWS; fi = e / T::ROWS; }
#pragma unroll
      for (int c = 0; c < NV; c++) sh[(c * T::ROWS + row) * FST + fi] = Fh[ps][c];
    }
  }
  __syncthreads();

  // 3. L = L - (Fhat_{m+1/2} - Fhat_{m-1/2}) / h
  for (int e = threadIdx.x; e < T::ROWS * T::SEG; e += THREADS) {
    int row, l;
    if constexpr (A == 0) { row = e / T::SEG; l = e % T::SEG; }
    else { row = e % T::ROWS; l = e / T::ROWS; }
    int I[3];
    if (!cell_of(row, l, I) || I[A] >= p.n[A]) continue;
    long long o = int_index(p, I[0], I[1], I[2]);
#pragma unroll
    for (int c = 0; c < NV; c++) {
      const double *hh = sh + (c * T::ROWS + row) * FST;
      // dx/dxi at the cell (the spacing h on a uniform direction); the boundary cell of a
      // characteristic face takes its normal term from k_char_faces instead
      double d = char_cell(p, A, I[A]) ? 0.0
                 : p.mm[A] ? divide(hh[l + 1] - hh[l], p.mm[A][I[A] + NG], p.minv[A][I[A] + NG])
                           : divide(hh[l + 1] - hh[l], p.h[A], p.inv_h[A]);
      double prev = first ? 0.0 : p.L[c * p.N + o];
      p.L[c * p.N + o] = prev - d;
    }
  }
}


// Component-wise: a tile is 32 lines by up to 8 K faces of one component; a warp takes the 32 lines
// of K consecutive faces.  The lines are consecutive in x (A > 0) or the rows of a plane (A = 0).
// With JOIN they are segments of rows, numbered through y, z and then the segments, so that lanes
// are idle in the last tile only (100000 x 4: 4 lanes of 32 work without); a line's place is then
// looked up, ~2 us a pass.  The kernel is bound by the FP64 pipe (1.7 lanes per clock and SM, so a
// warp instruction costs its SM quarter ~75 cycles): what counts is FP64 operations, and that every
// SM quarter has several warps to issue them from.  Hence K faces per thread, whose differences are
// shared (faces_of_line), a block per component (the split fluxes of one take 27 KB; a small grid has
// five times the blocks), segments of equal length instead of a short last one, idle lanes only in
// whole warps, and a K chosen by the launcher (conv_tiles): 4 on large grids, less where tiles of 31
// cells would leave SMs idle.
// Against one face per thread on tiles of 63 (x) or 15 (y, z) cells with all components staged:
// TENO5 at 256^3 x 8.06 -> 3.53 ms, y and z 5.92 -> 3.48 ms (FP64 operations per cell of a pass,
// counted by ncu at 192^3 with K = 2: 121, before ~300 in x); WENO5-JS at 256^2 x 138 -> 70 us,
// y 92 -> 70 us; strict TENO5 at 61 x 53 x 47 x 620 -> 225 us (joined), y and z 961 -> 212 us.
template <int A, int K>
struct LineTile {
  static constexpr int R = 32;                      // lines
  static constexpr int FACES = (THREADS / 32) * K;  // faces per line
  static constexpr int LEN = FACES + 5;             // staged cells per line (odd)
  static constexpr int SL = A == 0 ? 1 : R, SR = A == 0 ? LEN : 1;      // staged strides
  static constexpr int HL = A == 0 ? 1 : R, HR = A == 0 ? FACES + 1 : 1;  // face strides
  static constexpr size_t BYTES = sizeof(double) * (2 * LEN * R + (FACES + 1) * R);
};

template <int DIM, int A, int SCHEME, int K, bool JOIN>
__global__ void __launch_bounds__(THREADS, 3) k_conv(Plan p, int first, int nseg) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  using T = LineTile<A, K>;
  // TENO5's weights depend on ratios of indicators only (its floors aside), so its fast form
  // reconstructs F +- alpha q and halves in the difference (a power of two: the same bits);
  // WENO5-JS's eps = 1e-6 is not scale-free
  constexpr bool FOLD = !STRICT && SCHEME == IBFSA_TENO5;
  extern __shared__ double sm[];
  double *sfp = sm;                   // f+ of the staged cells
  double *sfm = sm + T::LEN * T::R;   // f-
  double *sh = sfm + T::LEN * T::R;   // face fluxes
  const double alpha = load_alpha(p, A);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x % NV;                    // component
  const int segl = (p.n[A] + nseg - 1) / nseg;
  // first cell along A, cells of the tile (JOIN: of its longest line) and its lines; offsets of its
  // first staged and its first own cell
  int seg0 = 0, ncell = segl, nrow;
  long long pad0 = 0, int0 = 0;
  // JOIN: the same of every line
  __shared__ int line_seg0[JOIN ? T::R : 1], line_ncell[JOIN ? T::R : 1];
  __shared__ int line_pad0[JOIN ? T::R : 1], line_int0[JOIN ? T::R : 1];
  constexpr int LN = A == 0 ? 1 : 0;  // direction of the tile's lines
  const long long stp[3] = {1, p.P[0], (long long)p.P[0] * p.P[1]};
  const long long sti[3] = {1, p.n[0], (long long)p.n[0] * p.n[1]};
  if constexpr (JOIN) {
    static_assert(A == 0, "rows along x");
    const unsigned rows = (unsigned)(p.n[1] * p.n[2]), first_line = blockIdx.x / NV * T::R;
    nrow = (int)min((unsigned)T::R, rows * nseg - first_line);
    if (warp == 0) {
      const unsigned line = first_line + min(lane, nrow - 1), seg = line / rows;
      const unsigned row = line - seg * rows;
      const int z = (int)(row / p.n[1]), y = (int)row - z * p.n[1], x = (int)seg * segl;
      line_seg0[lane] = x;
      line_ncell[lane] = min(segl, p.n[0] - x);  // 0 or less: an empty last segment
      line_pad0[lane] = (int)(pad_index(p, x, y, z) - 3);
      line_int0[lane] = (int)int_index(p, x, y, z);
    }
    __syncthreads();
  } else {
    seg0 = (blockIdx.x / NV % nseg) * segl;
    const int line0 = blockIdx.x / (NV * nseg) * T::R;
    ncell = min(segl, p.n[A] - seg0);
    if (ncell <= 0) return;
    nrow = min(T::R, p.n[LN] - line0);
    int I[3] = {0, 0, 0};
    I[A] = seg0;
    I[LN] = line0;
    if (DIM > 2) I[3 - A - LN] = blockIdx.y;
    pad0 = pad_index(p, I[0], I[1], I[2]) - 3 * stp[A];
    int0 = int_index(p, I[0], I[1], I[2]);
  }
  const double *Qb = p.Qp + pad0, *Wb = p.Wp + pad0;
  double *Lb = p.L + int0;
  const int nface = ncell + 1, nst = ncell + 6;

  // the slots a warp's last faces read beyond the staged cells hold zeros
  for (int l = nst - 1 + warp; l < T::LEN; l += THREADS / 32) {
    sfm[lane * T::SR + l * T::SL] = 0.0;
    if (l >= nst) sfp[lane * T::SR + l * T::SL] = 0.0;
  }
  // 1. split fluxes f+- = (F_A(Q) +- alpha Q)/2 of the staged cells, consecutive threads along x
  constexpr int NS = (T::LEN * T::R + THREADS - 1) / THREADS;
#pragma unroll
  for (int i = 0; i < NS; i++) {
    const int e = threadIdx.x + i * THREADS;
    const int l = A == 0 ? e % nst : e / T::R, row = A == 0 ? e / nst : e % T::R;
    if (l >= nst || row >= nrow) continue;
    if (JOIN && l >= line_ncell[row] + 6) continue;
    const int go = JOIN ? line_pad0[row] + l : (int)(row * stp[LN] + l * stp[A]);
    const double q = Qb[c * p.NP + go];
    double F;
    if (c == 0) {
      F = Qb[(1 + A) * p.NP + go];
    } else {
      const double ua = Wb[A * p.NP + go], pr = Wb[DIM * p.NP + go];
      if (c == NV - 1) {
        F = (q + pr) * ua;
      } else {
        F = q * ua;
        if (c - 1 == A) F += pr;
      }
    }
    // f+ of staged cell l at l, f- at l - 1 (that of cell 0, which no face reads, lands on a
    // slot that no face reads: the last one of the line before, or of f+)
    const int so = row * T::SR + l * T::SL;
    sfp[so] = FOLD ? fma(alpha, q, F) : 0.5 * (F + alpha * q);
    sfm[so - T::SL] = FOLD ? fma(-alpha, q, F) : 0.5 * (F - alpha * q);
  }
  __syncthreads();
  // 2. faces m+1/2, m = seg0 - 1 + fi: f+ of staged cells fi .. fi+4, f- of fi+1 .. fi+5
  const int fi0 = warp * K;  // this warp's first face
  if (fi0 < nface) {
    const int line = min(lane, nrow - 1), at = line * T::SR + fi0 * T::SL;
    double f[K + 4], h[K], g[K];
#pragma unroll
    for (int j = 0; j < K + 4; j++) f[j] = sfp[at + j * T::SL];
    unsigned fail = faces_of_line<SCHEME, false, K>(p, f, h);
#pragma unroll
    for (int j = 0; j < K + 4; j++) f[j] = sfm[at + j * T::SL];
    fail |= faces_of_line<SCHEME, true, K>(p, f, g) << K;
    if constexpr (SCHEME == IBFSA_TENO5) {
      // slots that hold a face
      const int faces = (JOIN ? line_ncell[line] + 1 : nface) - fi0;
      const unsigned some = (1u << max(0, min(K, faces))) - 1;
      fail &= some | some << K;
      // full TENO5 where the sufficient test failed: each lane walks its own failed stencils
      // (re-read from shared memory), one copy of the code
#pragma unroll 1
      while (fail) {
        const int j = __ffs(fail) - 1;
        fail &= fail - 1;
        const double *v = j < K ? sfp + at + j * T::SL : sfm + at + (j - K + 4) * T::SL;
        const int st = j < K ? T::SL : -T::SL;
        const double t = teno5(p, v[0], v[st], v[2 * st], v[3 * st], v[4 * st]);
#pragma unroll
        for (int i = 0; i < K; i++) {
          if (j == i) h[i] = t;
          if (j == K + i) g[i] = t;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < K; j++) sh[lane * T::HR + (fi0 + j) * T::HL] = h[j] + g[j];
  }
  __syncthreads();
  // 3. L = L - (Fhat_{m+1/2} - Fhat_{m-1/2}) / (dx/dxi); the boundary cell of a characteristic
  // face takes its normal term from k_char_faces instead.  A = 0: a warp walks the rows.
  constexpr int NW = THREADS / 32;
#pragma unroll
  for (int i = 0; i < (A == 0 ? T::R / NW : (T::FACES + NW - 1) / NW); i++) {
    const int row = A == 0 ? warp + i * NW : lane, l = A == 0 ? lane : warp + i * NW;
    if (l >= ncell || row >= nrow) continue;
    if (JOIN && l >= line_ncell[row]) continue;
    const double *hh = sh + row * T::HR + l * T::HL;
    const double dh = hh[T::HL] - hh[0];
    const int ia = (JOIN ? line_seg0[row] : seg0) + l;
    constexpr double half = FOLD ? 0.5 : 1.0;
    const bool str = p.mm[A] != nullptr;
    const double inv = half * (str ? p.minv[A][ia + NG] : p.inv_h[A]);
    double *Lc = Lb + c * p.N + (JOIN ? line_int0[row] + l : row * sti[LN] + l * sti[A]);
    const double prev = first ? 0.0 : *Lc;
    if (char_cell(p, A, ia)) *Lc = prev;
    else if (STRICT) *Lc = prev - divide(dh, str ? p.mm[A][ia + NG] : p.h[A], inv);
    else *Lc = fma(-dh, inv, prev);
  }
}

// ------------------------------------------------------------------------------------------
// characteristic non-reflecting faces (Sec. 2, after Thompson): at the boundary cell the normal
// convective term is dF_a/dx_a in characteristic form, from fourth-order one-sided derivatives
// of the primitives with the entering waves' amplitudes set to zero
// ------------------------------------------------------------------------------------------
// fourth-order one-sided derivative into the domain (s = +1 from the low face, -1 from the high
// face) of the padded field phi at padded offset o, stride st along the direction;
// (-25 f0 + 48 f1 - 36 f2 + 16 f3 - 3 f4)/12 on the differences f_k - f0
__device__ __forceinline__ double one_sided(const double *phi, long long o, long long st, int s,
                                            double h12, double inv_h12) {
  const double f0 = phi[o];
  double acc = 0.0;
  acc = acc + 48.0 * (phi[o + s * st] - f0);
  acc = acc + -36.0 * (phi[o + 2 * s * st] - f0);
  acc = acc + 16.0 * (phi[o + 3 * s * st] - f0);
  acc = acc + -3.0 * (phi[o + 4 * s * st] - f0);
  return divide((double)s * acc, h12, inv_h12);
}

// the normal convective term (dF_a/dx_a)_char of the cell I on the face (a, side), in the order the
// formulas are written (the strict form reproduces a sequential evaluation)
template <int DIM>
__device__ __forceinline__ void char_term(const Plan &p, int a, int side, const int I[3],
                                          double D[DIM + 2]) {
  constexpr int NV = DIM + 2;
  const int s = side == 0 ? 1 : -1;
  const long long o = pad_index(p, I[0], I[1], I[2]);
  const long long st = a == 0 ? 1 : a == 1 ? (long long)p.P[0] : (long long)p.P[0] * p.P[1];
  const double h12 = p.mm[a] ? 12.0 * p.mm[a][I[a] + NG] : p.h12[a];
  const double ih12 = p.mm[a] ? p.minv12[a][I[a] + NG] : p.inv_h12[a];
  const double r = p.Qp[o], pr = p.Wp[DIM * p.NP + o];
  const double c = sqrt(p.gamma * pr / r);
  const double ua = p.Wp[a * p.NP + o];
  const double rx = one_sided(p.Qp, o, st, s, h12, ih12);
  const double px = one_sided(p.Wp + DIM * p.NP, o, st, s, h12, ih12);
  const double uxa = one_sided(p.Wp + a * p.NP, o, st, s, h12, ih12);
  const double lam1 = ua - c, lam2 = ua, lam5 = ua + c;
  // a speed points into the domain when it has the sign of s
  const double L1 = (lam1 * (double)s > 0.0) ? 0.0 : lam1 * (px - r * c * uxa);
  const double L2 = (lam2 * (double)s > 0.0) ? 0.0 : lam2 * (c * c * rx - px);
  const double L5 = (lam5 * (double)s > 0.0) ? 0.0 : lam5 * (px + r * c * uxa);
  double dv[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    if (b == a) continue;
    double utx = one_sided(p.Wp + b * p.NP, o, st, s, h12, ih12);
    dv[b] = (lam2 * (double)s > 0.0) ? 0.0 : lam2 * utx;
  }
  const double d1 = (L2 + 0.5 * (L5 + L1)) / (c * c);
  const double d2 = 0.5 * (L5 + L1);
  dv[a] = (L5 - L1) / (2.0 * r * c);
  double ke = 0.0, work = 0.0;
  D[0] = d1;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    double ub = p.Wp[b * p.NP + o];
    D[1 + b] = ub * d1 + r * dv[b];
    ke = ke + ub * ub;
    work = work + ub * dv[b];
  }
  D[NV - 1] = 0.5 * ke * d1 + d2 / p.gm1 + r * work;
}

// All characteristic faces in one launch, one thread per cell: the cell of a corner or an edge
// belongs to the thread of its first face, which takes its faces' terms in order (direction by
// direction, low face first).
template <int DIM>
__global__ void __launch_bounds__(128) k_char_faces(Plan p) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int I[3], face = -1;
#pragma unroll
  for (int a = 0; a < DIM; a++)
#pragma unroll
    for (int side = 0; side < 2; side++) {
      if (face >= 0 || p.bc[a][side] != IBFSA_BC_CHARACTERISTIC) continue;
      const int b1 = (a + 1) % 3, b2 = (a + 2) % 3;
      const long long cells = (long long)p.n[b1] * p.n[b2];
      if (t < cells) {
        face = 2 * a + side;
        I[a] = side == 0 ? 0 : p.n[a] - 1;
        I[b1] = (int)(t % p.n[b1]);
        I[b2] = (int)(t / p.n[b1]);
      }
      t -= cells;
    }
  if (face < 0) return;
  for (int a = 0; a < face / 2; a++)
    if (char_cell(p, a, I[a])) return;  // another thread's cell
  const long long oi = int_index(p, I[0], I[1], I[2]);
  double L[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) L[c] = p.L[c * p.N + oi];
  for (int f = face; f < 2 * DIM; f++) {
    const int a = f / 2, side = f % 2;
    if (p.bc[a][side] != IBFSA_BC_CHARACTERISTIC || I[a] != (side == 0 ? 0 : p.n[a] - 1)) continue;
    double D[NV];
    char_term<DIM>(p, a, side, I, D);
#pragma unroll
    for (int c = 0; c < NV; c++) L[c] = L[c] - D[c];
  }
#pragma unroll
  for (int c = 0; c < NV; c++) p.L[c * p.N + oi] = L[c];
}

// ------------------------------------------------------------------------------------------
// viscous term (Eq. 2, 5): gradients of u by 4th-order central differences on the box
// [-2, n+2), tau_ij = du_i/dx_j + du_j/dx_i - 2/3 delta_ij div u, b_j = u_i tau_ij, then
// (1/Re) sum_a D4_a [0, tau_{.a}, b_a]
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ double d4(double fm2, double fm1, double fp1, double fp2, double h12,
                                     double inv_h12) {
  return divide(8.0 * (fp1 - fm1) - (fp2 - fm2), h12, inv_h12);
}

// 12 dx/dxi at node i of direction a and its reciprocal, rounded as 12 h is on a uniform one
__device__ __forceinline__ double metric12(const Plan &p, int a, int i, double *inv) {
  *inv = p.mm[a] ? p.minv12[a][i + NG] : p.inv_h12[a];
  return STRICT && p.mm[a] ? 12.0 * p.mm[a][i + NG] : p.h12[a];
}

// Bound by the FP64 pipe (as k_conv).  The strict form takes every gradient by itself; the fast
// form scales a pair of cross gradients as it adds them and stores the symmetric tau once (a <= ci):
// 51 operations a cell in 3D instead of 59, 1.98 -> 1.76 ms at 256^3.
template <int DIM>
__global__ void __launch_bounds__(THREADS) k_visc_flux(Plan p) {
  begin_kernel();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.NB) return;
  int bx = (int)(t % p.B[0]);
  long long r = t / p.B[0];
  int by = (int)(r % p.B[1]);
  int bz = (int)(r / p.B[1]);
  int I[3] = {bx - 2, DIM > 1 ? by - 2 : by, DIM > 2 ? bz - 2 : bz};
  long long s = pad_index(p, I[0], I[1], I[2]);
  long long stride[3] = {1, p.P[0], (long long)p.P[0] * p.P[1]};
  if constexpr (!STRICT) {
    double inv[DIM], tau[DIM][DIM], div = 0.0;
    // 12 h du_ci/dx_a
    auto diff = [&](int ci, int a) {
      const double *u = p.Wp + ci * p.NP + s;
      const long long st = stride[a];
      return 8.0 * (u[st] - u[-st]) - (u[2 * st] - u[-2 * st]);
    };
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      inv[a] = p.mm[a] ? p.minv12[a][I[a] + NG] : p.inv_h12[a];
      tau[a][a] = diff(a, a) * inv[a];
      div = a ? div + tau[a][a] : tau[a][a];
    }
    const double third = 2.0 / 3.0 * div;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      tau[a][a] = 2.0 * tau[a][a] - third;
      p.V[(long long)(a * (DIM + 1) + a) * p.NB + t] = tau[a][a];
#pragma unroll
      for (int ci = a + 1; ci < DIM; ci++) {
        tau[a][ci] = tau[ci][a] = diff(ci, a) * inv[a] + diff(a, ci) * inv[ci];
        p.V[(long long)(a * (DIM + 1) + ci) * p.NB + t] = tau[a][ci];
      }
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      double b = p.Wp[s] * tau[a][0];
#pragma unroll
      for (int ci = 1; ci < DIM; ci++) b += p.Wp[ci * p.NP + s] * tau[a][ci];
      p.V[(long long)(a * (DIM + 1) + DIM) * p.NB + t] = b;
    }
    return;
  }
  double g[DIM][DIM];
#pragma unroll
  for (int ci = 0; ci < DIM; ci++) {
    const double *u = p.Wp + ci * p.NP + s;
#pragma unroll
    for (int dj = 0; dj < DIM; dj++) {
      long long st = stride[dj];
      double inv;
      const double h12 = metric12(p, dj, I[dj], &inv);
      g[ci][dj] = d4(u[-2 * st], u[-st], u[st], u[2 * st], h12, inv);
    }
  }
  double div = 0.0;
#pragma unroll
  for (int a = 0; a < DIM; a++) div += g[a][a];
#pragma unroll
  for (int a = 0; a < DIM; a++) {
    double b = 0.0;
#pragma unroll
    for (int ci = 0; ci < DIM; ci++) {
      double tau = g[ci][a] + g[a][ci];
      if (ci == a) tau -= 2.0 / 3.0 * div;
      p.V[(long long)(a * (DIM + 1) + ci) * p.NB + t] = tau;
      b += p.Wp[ci * p.NP + s] * tau;
    }
    p.V[(long long)(a * (DIM + 1) + DIM) * p.NB + t] = b;
  }
}

// strict form: the divergence by itself, operation by operation (the fast form's is in k_finish)
template <int DIM>
__global__ void __launch_bounds__(THREADS) k_visc_div(Plan p) {
  begin_kernel();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.N) return;
  int i = (int)(t % p.n[0]);
  long long r = t / p.n[0];
  int j = (int)(r % p.n[1]);
  int k = (int)(r / p.n[1]);
  long long b = ((long long)(DIM > 2 ? k + 2 : k) * p.B[1] + (DIM > 1 ? j + 2 : j)) * p.B[0] + (i + 2);
  long long stride[3] = {1, p.B[0], (long long)p.B[0] * p.B[1]};
#pragma unroll
  for (int fc = 0; fc <= DIM; fc++) {
    double sum = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const double *F = p.V + (long long)(a * (DIM + 1) + fc) * p.NB + b;
      long long st = stride[a];
      double inv;
      const double h12 = metric12(p, a, a == 0 ? i : a == 1 ? j : k, &inv);
      sum += d4(F[-2 * st], F[-st], F[st], F[2 * st], h12, inv);
    }
    long long o = (long long)(fc + 1) * p.N + t;
    p.L[o] = p.L[o] + divide(sum, p.Re, p.inv_Re);
  }
}

// ------------------------------------------------------------------------------------------
// immersed boundary (Eq. 7-9)
// ------------------------------------------------------------------------------------------
// the four-point supports of point k of X [dim][nm] in every direction (Eq. 10-11)
template <int DIM>
__device__ __forceinline__ bool marker_support(const Plan &p, const double *X, int nm, int k,
                                               int j0[3], double w[3][4]) {
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    if (a < DIM) {
      if (p.mx[a]) {
        double s, hl;
        j0[a] = mesh::support_stretched(p, a, X[a * nm + k], &s, &hl);
#pragma unroll
        for (int r = 0; r < 4; r++) w[a][r] = marker::peskin(s - (double)(j0[a] + r));
      } else {
        j0[a] = support(p, a, X[a * nm + k], w[a]);
      }
      if (j0[a] < 0 || j0[a] + 3 > p.n[a] - 1) ok = false;
    } else {
      j0[a] = 0;
      w[a][0] = 1.0; w[a][1] = 0.0; w[a][2] = 0.0; w[a][3] = 0.0;
    }
  }
  return ok;
}

// ---- strict form: supports of STRICT_MARKERS markers per block, one weight per thread -------
constexpr int STRICT_MARKERS = 8;
template <int DIM>
constexpr int strict_support_cells = DIM > 2 ? 64 : 16;

// Supports of markers k0 .. k0 + STRICT_MARKERS - 1 into shared memory: weights, first cells,
// whether the support leaves the grid, the product of the local spacings (shp may be NULL); every
// thread of the block (at least 96) calls it.
template <int DIM>
__device__ __forceinline__ void strict_supports(const Plan &p, int k0,
                                                double (*sw)[3][4], int (*sj)[3], int *sbad,
                                                double *shp) {
  __shared__ double shl[STRICT_MARKERS][3];
  const int tid = threadIdx.x, m = tid / 12, a = tid % 12 / 4, q = tid % 4, k = k0 + m;
  if (tid < STRICT_MARKERS) sbad[tid] = 0;
  __syncthreads();
  if (m < STRICT_MARKERS && k < p.nm) {
    if (a < DIM) {
      const double x = p.X[(long long)a * p.max_markers + k];
      double sx = 0.0, hl = p.h[a];
      int j;
      if (p.mx[a]) {
        j = mesh::support_stretched(p, a, x, &sx, &hl);
      } else {
        sx = divide(x - p.lo[a], p.h[a], p.inv_h[a]) - 0.5;
        j = (int)floor(sx) - 1;
      }
      sw[m][a][q] = marker::peskin(sx - (double)(j + q));
      if (q == 0) {
        sj[m][a] = j;
        shl[m][a] = hl;
        if (j < 0 || j > p.n[a] - 4) sbad[m] = 1;
      }
    } else {
      sw[m][a][q] = q == 0 ? 1.0 : 0.0;
      if (q == 0) {
        sj[m][a] = 0;
        shl[m][a] = 1.0;
      }
    }
  }
  __syncthreads();
  if (shp && tid < STRICT_MARKERS) {
    double hp = 1.0;
#pragma unroll
    for (int b = 0; b < DIM; b++) hp *= shl[tid][b];
    shp[tid] = hp;
  }
}

// strict form: U_ib = sum_j u_j prod lambda (Eq. 8), F = alpha xi + beta (U_ib - U) (Eq. 7), and the
// RK update of xi (xi' = U_ib - U) when the stage is advanced
template <int DIM>
__global__ void k_ib_interp(Plan p, const double *__restrict__ xis, const double *xin,
                            double *xio, double A, double Bc, double dt, int advance) {
  begin_kernel();
  const int nm = p.nm, M = p.max_markers;
  // strict: the weights of SM markers one per thread, the products u (w w w) of their support
  // cells one per thread, then one thread per marker and component adds them up in the order of
  // the formula (z, y, x)
  constexpr int S = strict_support_cells<DIM>, SM = STRICT_MARKERS;
  __shared__ double sw[SM][3][4], sv[SM][DIM][S + 1];
  __shared__ int sj[SM][3], sbad[SM];
  const int k0 = blockIdx.x * SM, tid = threadIdx.x;
  strict_supports<DIM>(p, k0, sw, sj, sbad, nullptr);
  for (int e = tid; e < SM * S; e += blockDim.x) {
    const int m = e / S, r = e % S, r0 = r & 3, r1 = (r >> 2) & 3, r2 = r >> 4;
    if (k0 + m >= nm || sbad[m]) continue;
    const double wt = sw[m][0][r0] * sw[m][1][r1] * sw[m][2][r2];
    const long long o = pad_index(p, sj[m][0] + r0, sj[m][1] + r1, sj[m][2] + r2);
#pragma unroll
    for (int a = 0; a < DIM; a++) sv[m][a][r] = p.Wp[a * p.NP + o] * wt;
  }
  __syncthreads();
  for (int e = tid; e < SM * DIM; e += blockDim.x) {
    const int m = e / DIM, a = e % DIM, k = k0 + m;
    if (k >= nm) continue;
    if (sbad[m]) {
      if (a == 0) atomicOr(p.status, IBFSA_STATUS_BOUNDS);
      p.F[a * M + k] = 0.0;
      if (advance) xio[a * M + k] = xin[a * M + k];
      continue;
    }
    double acc = 0.0;
#pragma unroll 8
    for (int r = 0; r < S; r++) acc += sv[m][a][r];
    double slip = acc - p.U[a * M + k];
    p.F[a * M + k] = p.alpha_pen * xis[a * M + k] + p.beta_pen * slip;
    if (advance) xio[a * M + k] = A * xin[a * M + k] + Bc * (xis[a * M + k] + dt * slip);
  }
}

// Strict spreading: every cell sums its contributions in marker order, f_j = f_j - F_k w dS_k /
// prod h (Eq. 9).  First a table of the markers' supports (weights, first cells, spacings) in the
// padded state's storage, which the stage has finished with; then one thread per cell, a block
// per tile of 256 cells, gathers: the block picks the markers whose support reaches its tile, in
// marker order (a ballot per 256 markers), and each cell takes those that cover it.  The table's
// bounding box lets the blocks away from the body write their zeros at once.  One block walking
// the markers one after the other (each waiting for the weights and the read-modify-write of its
// cells) took 12 us per marker: 400 markers 4720 us, table and gather 74 us.
struct SpreadTable {
  double *w;     // [12][n] weights (direction, offset)
  double *hp;    // [n] product of the local spacings
  double *ihp;   // [n] its reciprocal
  int *j0;       // [3][n] first support cells (INT_MIN / 2: no support)
  int *box;      // [6]: smallest first cell, minus the largest, per direction
  static constexpr int DOUBLES = 16;  // per marker: 12 + 2, and three ints
};

template <int DIM>
__global__ void __launch_bounds__(128) k_spread_table(Plan p, SpreadTable t, int first, int n) {
  begin_kernel();
  __shared__ double sw[STRICT_MARKERS][3][4], shp[STRICT_MARKERS];
  __shared__ int sj[STRICT_MARKERS][3], sbad[STRICT_MARKERS];
  const int i0 = blockIdx.x * STRICT_MARKERS, tid = threadIdx.x;
  strict_supports<DIM>(p, first + i0, sw, sj, sbad, shp);
  const int m = tid / 12, e = tid % 12, i = i0 + m;
  __syncthreads();
  if (m >= STRICT_MARKERS || i >= n) return;
  t.w[(long long)e * n + i] = sw[m][e / 4][e % 4];
  if (e == 0) {
    t.hp[i] = shp[m];
    t.ihp[i] = 1.0 / shp[m];
  }
  if (e < 3) {
    const int j = sbad[m] ? -(1 << 30) : sj[m][e];
    t.j0[(long long)e * n + i] = j;
    if (!sbad[m]) {
      atomicMin(&t.box[e], j);
      atomicMin(&t.box[3 + e], -j);
    }
  }
}

template <int DIM>
struct SpreadTile {
  static constexpr int X = DIM > 2 ? 8 : 16, Y = DIM > 2 ? 8 : 16, Z = DIM > 2 ? 4 : 1;
};

template <int DIM>
__global__ void __launch_bounds__(THREADS) k_spread_gather(Plan p, SpreadTable t, int first, int n) {
  begin_kernel();
  using T = SpreadTile<DIM>;
  static_assert(T::X * T::Y * T::Z == THREADS, "one thread per cell");
  __shared__ int list[THREADS], cnt[THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ext[3] = {T::X, T::Y, T::Z};
  const unsigned gx = (p.n[0] + T::X - 1) / T::X, gy = (p.n[1] + T::Y - 1) / T::Y;
  const int b[3] = {(int)(blockIdx.x % gx) * T::X, (int)(blockIdx.x / gx % gy) * T::Y,
                    (int)(blockIdx.x / (gx * gy)) * T::Z};
  const int I[3] = {b[0] + tid % T::X, b[1] + tid / T::X % T::Y, b[2] + tid / (T::X * T::Y)};
  const bool own = I[0] < p.n[0] && I[1] < p.n[1] && I[2] < p.n[2];
  const long long o = own ? int_index(p, I[0], I[1], I[2]) : 0;
  double f[DIM];
#pragma unroll
  for (int a = 0; a < DIM; a++) f[a] = first > 0 && own ? p.f[a * p.N + o] : 0.0;
  bool near = true;  // the tile meets the supports' bounding box
#pragma unroll
  for (int a = 0; a < DIM; a++) near &= b[a] + ext[a] > t.box[a] && b[a] <= -t.box[3 + a] + 3;
  for (int base = 0; near && base < n; base += THREADS) {  // uniform over the block
    const int i = base + tid;
    bool hit = i < n;
    if (hit) {
#pragma unroll
      for (int a = 0; a < DIM; a++) {
        const int j = t.j0[(long long)a * n + i];
        hit &= j + 3 >= b[a] && j < b[a] + ext[a];
      }
    }
    const unsigned votes = __ballot_sync(0xffffffffu, hit);
    if (lane == 0) cnt[warp] = __popc(votes);
    __syncthreads();
    int at = 0, total = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; w++) {
      if (w < warp) at += cnt[w];
      total += cnt[w];
    }
    if (hit) list[at + __popc(votes & ((1u << lane) - 1))] = i;
    __syncthreads();
    for (int q = 0; q < total; q++) {
      const int m = list[q];
      const int d0 = I[0] - t.j0[m], d1 = I[1] - t.j0[n + m];
      const int d2 = DIM > 2 ? I[2] - t.j0[2 * (long long)n + m] : 0;
      if ((unsigned)d0 > 3u || (unsigned)d1 > 3u || (unsigned)d2 > 3u) continue;
      const double wt = t.w[(long long)d0 * n + m] * t.w[(long long)(4 + d1) * n + m] *
                        t.w[(long long)(8 + d2) * n + m];
      const double dS = p.dS[first + m], hp = t.hp[m], ihp = t.ihp[m];
#pragma unroll
      for (int a = 0; a < DIM; a++)
        f[a] -= divide(p.F[(long long)a * p.max_markers + first + m] * wt * dS, hp, ihp);
    }
    __syncthreads();
  }
  if (own)
#pragma unroll
    for (int a = 0; a < DIM; a++) p.f[a * p.N + o] = f[a];
}

// the strict spreading of all markers, as many at a time as the padded state's storage holds
template <int DIM>
cudaError_t spread_strict(const Plan &p, cudaStream_t st) {
  using T = SpreadTile<DIM>;
  const long long room = (DIM + 2) * p.NP - 8;  // doubles; the box takes the last ones
  const int most = (int)(room / SpreadTable::DOUBLES < p.nm ? room / SpreadTable::DOUBLES : p.nm);
  const unsigned tiles = (unsigned)((p.n[0] + T::X - 1) / T::X) *
                         ((p.n[1] + T::Y - 1) / T::Y) * ((p.n[2] + T::Z - 1) / T::Z);
  for (int first = 0; first < p.nm; first += most) {
    const int n = p.nm - first < most ? p.nm - first : most;
    SpreadTable t;
    t.w = p.Qp;
    t.hp = t.w + 12LL * n;
    t.ihp = t.hp + n;
    t.j0 = reinterpret_cast<int *>(t.ihp + n);
    t.box = reinterpret_cast<int *>(p.Qp + room);
    cudaError_t e = cudaMemsetAsync(t.box, 0x7f, 6 * sizeof(int), st);
    if (e != cudaSuccess) return e;
    launch(k_spread_table<DIM>, (n + STRICT_MARKERS - 1) / STRICT_MARKERS, 128, 0, st, p, t, first,
           n);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch(k_spread_gather<DIM>, tiles, THREADS, 0, st, p, t, first, n);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Fast form: markers, a group of G lanes each (marker.cuh): interpolation and penalty force, and the
// spreading with atomics straight into L: momentum += f, energy += f.u
template <int DIM, int G, int PART>
__global__ void __launch_bounds__(128) k_markers(Plan p, const double *__restrict__ xis,
                                                 const double *xin, double *xio, double A,
                                                 double Bc, double dt, int advance) {
  begin_kernel();
  constexpr int C = marker::Support<DIM, G>::C;
  const int r = threadIdx.x % G, M = p.max_markers;
  const unsigned km = blockIdx.x * (blockDim.x / G) + threadIdx.x / G, nm = (unsigned)p.nm;
  const int k = (int)min(km, nm - 1);
  const auto t = marker::support<DIM, G>(p, p.X, M, k, r);
  const long long s = pad_index(p, t.c0[0], t.c0[1], t.c0[2]);
  double F[DIM];
  if constexpr (PART & marker::INTERP) {
    double acc[DIM];
#pragma unroll
    for (int a = 0; a < DIM; a++) acc[a] = 0.0;
    if (t.ok) {
#pragma unroll
      for (int a = 0; a < DIM; a++)
#pragma unroll
        for (int r0 = 0; r0 < C; r0++) acc[a] = fma(p.Wp[a * p.NP + s + r0], t.w0[r0], acc[a]);
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) acc[a] = marker::group_sum<G>(acc[a] * t.wr);
    double mine = 0.0;
    if (km < nm) {
      if (t.ok) mine = marker::force<DIM>(p, k, r, acc, xis, xin, xio, A, Bc, dt, advance);
      else marker::off_grid<DIM>(p, k, r, xin, xio, advance);
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) F[a] = __shfl_sync(0xffffffffu, mine, a, G);
  }
  if constexpr (!(PART & marker::SPREAD)) return;
  if (km >= nm || !t.ok) return;
  const long long o = int_index(p, t.c0[0], t.c0[1], t.c0[2]);
  const double sc = t.wr * (p.dS[k] * t.ihp);
  double f[DIM];
#pragma unroll
  for (int a = 0; a < DIM; a++) f[a] = -(PART & marker::INTERP ? F[a] : p.F[a * M + k]) * sc;
#pragma unroll
  for (int r0 = 0; r0 < C; r0++) {
    double pw = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const double fa = f[a] * t.w0[r0];
      atomicAdd(&p.L[(1 + a) * p.N + o + r0], fa);
      pw += fa * p.Wp[a * p.NP + s + r0];
    }
    atomicAdd(&p.L[(DIM + 1) * p.N + o + r0], pw);
  }
}

// ------------------------------------------------------------------------------------------
// finish: sponge, strict-mode IB source, then RHS out or RK combination a Qn + b (Qs + dt L)
// ------------------------------------------------------------------------------------------
// VISC (fast form): the divergence of the viscous fluxes as well.  With the metric and 1/Re in one
// factor per direction, multiplied in as the sum adds up (on uniform directions by the host), it
// takes 48 FP64 operations a cell in 3D instead of 64, and the sum stays in registers instead of
// passing through L: divergence and finish 3.08 -> 2.22 ms at 256^3, 16 -> 12 us at 256^2.
struct ViscScale {
  double c[3];  // 1 / (12 h Re); of a stretched direction 1 / Re
};

template <int DIM, bool VISC>
__global__ void __launch_bounds__(THREADS) k_finish(Plan p, const double *__restrict__ Qs,
                                                    const double *Qn, double *out, double A,
                                                    double Bc, double dt, int advance,
                                                    ViscScale vs) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.N) return;
  int I[3];
  I[0] = (int)(t % p.n[0]);
  long long r = t / p.n[0];
  I[1] = (int)(r % p.n[1]);
  I[2] = (int)(r / p.n[1]);
  double Lc[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) Lc[c] = p.L[c * p.N + t];
  if constexpr (VISC) {
    const long long b =
        ((long long)(DIM > 2 ? I[2] + 2 : I[2]) * p.B[1] + (I[1] + 2)) * p.B[0] + (I[0] + 2);
    const long long stride[3] = {1, p.B[0], (long long)p.B[0] * p.B[1]};
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const double scale = p.mm[a] ? p.minv12[a][I[a] + NG] * vs.c[a] : vs.c[a];
      const long long st = stride[a];
#pragma unroll
      for (int fc = 0; fc <= DIM; fc++) {
        const int lo = fc < a ? fc : a, hi = fc < a ? a : fc;  // tau is stored once
        const double *F = p.V + (long long)(lo * (DIM + 1) + hi) * p.NB + b;
        Lc[fc + 1] += scale * (8.0 * (F[st] - F[-st]) - (F[2 * st] - F[-2 * st]));
      }
    }
  }
  if (p.sponge_cells > 0) {
    int S = p.sponge_cells;
    int nmin = 1 << 30;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      int e = I[a] < p.n[a] - 1 - I[a] ? I[a] : p.n[a] - 1 - I[a];
      if (e < nmin) nmin = e;
    }
    if (nmin < S) {
      double rr = (double)(S - nmin) / (double)S;
      double sig = p.sponge_sigma * rr * rr * rr;
#pragma unroll
      for (int c = 0; c < NV; c++) Lc[c] = Lc[c] - sig * (Qs[c * p.N + t] - p.qinf[c]);
    }
  }
  if (p.src_on) {  // periodic Gaussian pressure source (Sec. 3.6, Eq. 16), energy equation
    const double LN2 = 0.693147180559945309417;
    double r2 = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      double x = mesh::node(p, a, I[a]);
      r2 = r2 + (x - p.src_xc[a]) * (x - p.src_xc[a]);
    }
    Lc[NV - 1] = Lc[NV - 1] + exp(-(p.src_b * LN2) * r2) * p.src_scale;
  }
  if constexpr (STRICT) {
    if (p.nm > 0) {
      long long s = pad_index(p, I[0], I[1], I[2]);
      double pw = 0.0;
#pragma unroll
      for (int a = 0; a < DIM; a++) {
        double fa = p.f[a * p.N + t];
        Lc[1 + a] = Lc[1 + a] + fa;
        pw += fa * p.Wp[a * p.NP + s];
      }
      Lc[NV - 1] = Lc[NV - 1] + pw;
    }
  }
  if (!advance) {
#pragma unroll
    for (int c = 0; c < NV; c++) out[c * p.N + t] = Lc[c];
  } else {
    bool bad = false;
#pragma unroll
    for (int c = 0; c < NV; c++) {
      double v = A * Qn[c * p.N + t] + Bc * (Qs[c * p.N + t] + dt * Lc[c]);
      out[c * p.N + t] = v;
      bad |= !isfinite(v);
    }
    if (bad) atomicOr(p.status, IBFSA_STATUS_NONFINITE);
  }
}

// ------------------------------------------------------------------------------------------
// probes: dp = sum_j p_j prod lambda - p_inf
// ------------------------------------------------------------------------------------------
template <int DIM>
__global__ void k_probe(Plan p, int np, const double *__restrict__ xp, double *__restrict__ out) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= np) return;
  int j0[3];
  double w[3][4];
  if (!marker_support<DIM>(p, xp, np, k, j0, w)) {
    atomicOr(p.status, IBFSA_STATUS_BOUNDS);
    out[k] = 0.0;
    return;
  }
  constexpr int C2 = DIM > 2 ? 4 : 1;
  const double *pr = p.Wp + DIM * p.NP;
  double acc = 0.0;
  for (int r2 = 0; r2 < C2; r2++)
    for (int r1 = 0; r1 < 4; r1++)
#pragma unroll
      for (int r0 = 0; r0 < 4; r0++)
        acc += pr[pad_index(p, j0[0] + r0, j0[1] + r1, j0[2] + r2)] *
               (w[0][r0] * w[1][r1] * w[2][r2]);
  out[k] = acc - p.p_inf;
}

// ------------------------------------------------------------------------------------------
// host-side orchestration of one stage
// ------------------------------------------------------------------------------------------
inline unsigned blocks_for(long long n, int threads) {
  return (unsigned)((n + threads - 1) / threads);
}

// One block keeps an SM's FP64 pipe busy.  With few blocks one at a time per SM is faster (more than
// half of its shared memory asked for): the next one starts where a block ends, instead of two or
// three that take long (TENO5's full evaluation) on one SM beside SMs that are done.  TENO5, a step
// one at a time up to 5 blocks per SM / as many as fit: 33^3 1.95 / 2.96 ms, 56^3 5.4 / 5.9, 64^3
// 7.8 / 8.4, 64 x 48 x 40 4.09 / 3.91; with more blocks 100^3 29.3 / 28.6, 1021 x 771 7.9 / 7.7.
template <int DIM, int A, int SCHEME>
cudaError_t launch_conv_char(const Plan &p, int first, cudaStream_t st) {
  using T = ConvTile<A>;
  constexpr size_t need = conv_smem_bytes<DIM, A>(), alone = need > 116 * 1024 ? need : 116 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_conv_char<DIM, A, SCHEME>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)alone);
  if (e != cudaSuccess) return e;
  dim3 grid;
  if (A == 0) {
    grid = dim3((p.n[0] + T::SEG - 1) / T::SEG, (p.n[1] + T::ROWS - 1) / T::ROWS, p.n[2]);
  } else {
    int nseg = (p.n[A] + T::SEG - 1) / T::SEG;
    int nx = (p.n[0] + T::ROWS - 1) / T::ROWS;
    grid = dim3(nseg * nx, A == 1 ? p.n[2] : p.n[1]);
  }
  const size_t smem = (long long)grid.x * grid.y * grid.z <= 5 * 152 ? alone : need;
  launch(k_conv_char<DIM, A, SCHEME>, grid, THREADS, smem, st, p, first);
  return cudaGetLastError();
}

// The tiles of a pass of k_conv.  Faces per thread: the K whose tiles give the smallest (tiles of the
// busiest SM) x (FP64 operations of a tile), the tiles of a line being as equal as they can be.  A
// face costs ~2 (4 + (K + 3)/K) + 1 operations, a staged cell ~3.  Measured, TENO5: 256^3, a y pass
// 3.47 / 3.82 / 4.91 ms with K = 4 / 2 / 1; WENO5-JS at 256^2, where 31-cell tiles give 1.9 blocks
// per SM, 70 / 73 / 80 us; TENO5 at 383 x 257, x pass 59 / 50 / 54 us.
// Joined rows along x where that saves an eighth of more than two tiles per SM, the whole step
// without / with: WENO5-JS, 100000 x 4 7.59 / 2.67 ms, strict 19.7 / 6.46, 300 x 33 x 33 3.74 / 3.07,
// strict 9.59 / 7.78; one tile per SM or less, 16 x 16 96 / 104 us, 65 x 65 108 / 111.
struct ConvTiles {
  int K, nseg;
  bool join;
  long long tiles;  // of one component
};

template <int DIM, int A>
inline ConvTiles conv_tiles(const Plan &p) {
  const int n = p.n[A];
  ConvTiles best{};
  double cost = -1.0;
  for (int K = 4; K >= 1; K /= 2) {
    const int most = 8 * K - 1, ns = (n + most - 1) / most, seg = (n + ns - 1) / ns;
    const long long across = A == 0 ? (long long)((p.n[1] + 31) / 32) * p.n[2]
                                    : (long long)((p.n[0] + 31) / 32) * p.n[A == 1 ? 2 : 1];
    const long long joined = ((long long)p.n[1] * p.n[2] * ns + 31) / 32;
    const bool join = A == 0 && (DIM + 2) * across * ns > 2 * 152 && 8 * joined <= 7 * across * ns;
    const long long tiles = join ? joined : across * ns;
    const double tile = (seg + 1) * (9.0 + 2.0 * (K + 3) / K) + 3.0 * (seg + 6) + 2.0 * seg;
    const double c = (double)(((DIM + 2) * tiles + 151) / 152) * tile;
    if (cost < 0.0 || c < cost) {
      cost = c;
      best = {K, ns, join, tiles};
    }
  }
  return best;
}

template <int DIM, int A, int SCHEME, int K, bool JOIN>
cudaError_t launch_conv_k(const Plan &p, int first, const ConvTiles &t, cudaStream_t st) {
  constexpr size_t smem = LineTile<A, K>::BYTES;
  static_assert(smem <= 47 * 1024, "with the lines' places within the default shared memory");
  static_assert(LineTile<A, K>::FACES <= 32, "the update walks a line of cells with one warp");
  const int planes = JOIN ? 1 : p.n[A == 2 ? 1 : 2];
  dim3 grid((unsigned)((DIM + 2) * (t.tiles / planes)), planes);
  launch(k_conv<DIM, A, SCHEME, K, JOIN>, grid, THREADS, smem, st, p, first, t.nseg);
  return cudaGetLastError();
}

template <int DIM, int A, int SCHEME, int K>
cudaError_t launch_conv_k(const Plan &p, int first, const ConvTiles &t, cudaStream_t st) {
  if constexpr (A == 0)
    if (t.join) return launch_conv_k<DIM, A, SCHEME, K, true>(p, first, t, st);
  return launch_conv_k<DIM, A, SCHEME, K, false>(p, first, t, st);
}

template <int DIM, int A, int SCHEME>
cudaError_t launch_conv(const Plan &p, int first, cudaStream_t st) {
  if (p.charwise) return launch_conv_char<DIM, A, SCHEME>(p, first, st);
  const ConvTiles t = conv_tiles<DIM, A>(p);
  switch (t.K) {
    case 4: return launch_conv_k<DIM, A, SCHEME, 4>(p, first, t, st);
    case 2: return launch_conv_k<DIM, A, SCHEME, 2>(p, first, t, st);
    default: return launch_conv_k<DIM, A, SCHEME, 1>(p, first, t, st);
  }
}

template <int DIM, int SCHEME>
cudaError_t run_stage(const Plan &p, const StageArgs &s, cudaStream_t st) {
  cudaError_t e;
  Prof *pr = s.prof;
  e = cudaMemsetAsync(p.alpha_bits, 0, 3 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  prof_begin(pr, st);
  launch(k_pad<DIM>, blocks_for(p.NP, THREADS), THREADS, 0, st, p, s.Qs);
  prof_end(pr, K_PAD, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  int advance = s.stage >= 0;
  // Markers.  Strict: interpolation now, spreading after the viscous term.  Fast: both in one launch
  // after the convective term, unless someone waits for the forces (the coupled step, which is 2D).
  using Interp = std::integral_constant<int, marker::INTERP>;
  using Spread = std::integral_constant<int, marker::SPREAD>;
  using Both = std::integral_constant<int, marker::BOTH>;
  auto markers = [&](auto part) -> cudaError_t {
    if (p.nm <= 0) return cudaSuccess;
    cudaError_t es = cudaSuccess;
    prof_begin(pr, st);
    if constexpr (!STRICT) {
      marker::with_group<DIM>(p.nm, [&](auto g) {
        launch(k_markers<DIM, g(), part()>, blocks_for((long long)p.nm * g(), 128), 128, 0, st, p,
               s.xis, s.xin, s.xio, s.a, s.b, s.dt, advance);
      });
    } else if constexpr (part() == marker::INTERP) {
      launch(k_ib_interp<DIM>, (p.nm + STRICT_MARKERS - 1) / STRICT_MARKERS, 128, 0, st, p, s.xis,
             s.xin, s.xio, s.a, s.b, s.dt, advance);
    } else {
      es = spread_strict<DIM>(p, st);
    }
    prof_end(pr, part() == marker::INTERP ? K_INTERP : K_SPREAD, st);
    return es != cudaSuccess ? es : cudaGetLastError();
  };
  if (DIM > 2 && s.forces) return cudaErrorNotSupported;
  if constexpr (STRICT || DIM == 2) {
    if ((STRICT || s.forces) && (e = markers(Interp())) != cudaSuccess) return e;
    if (s.forces && (e = cudaEventRecord(s.forces, st)) != cudaSuccess) return e;
  }
  prof_begin(pr, st);
  e = launch_conv<DIM, 0, SCHEME>(p, 1, st);
  prof_end(pr, K_CONV_X, st);
  if (e != cudaSuccess) return e;
  prof_begin(pr, st);
  e = launch_conv<DIM, 1, SCHEME>(p, 0, st);
  prof_end(pr, K_CONV_Y, st);
  if (e != cudaSuccess) return e;
  if constexpr (DIM == 3) {
    prof_begin(pr, st);
    e = launch_conv<DIM, 2, SCHEME>(p, 0, st);
    prof_end(pr, K_CONV_Z, st);
    if (e != cudaSuccess) return e;
  }
  if (const long long cells = char_cells(p)) {
    prof_begin(pr, st);
    launch(k_char_faces<DIM>, blocks_for(cells, 128), 128, 0, st, p);
    prof_end(pr, K_CONV_X, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // strict: the viscous divergence into L, then the spreading; fast: the spreading, then the
  // divergence as part of finish
  if constexpr (!STRICT) {
    if constexpr (DIM == 2) e = s.forces ? markers(Spread()) : markers(Both());
    else e = markers(Both());
    if (e != cudaSuccess) return e;
  }
  const bool viscous = p.Re > 0.0;
  if (viscous) {
    prof_begin(pr, st);
    launch(k_visc_flux<DIM>, blocks_for(p.NB, THREADS), THREADS, 0, st, p);
    prof_end(pr, K_VISC_FLUX, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if constexpr (STRICT) {
    if (viscous) {
      prof_begin(pr, st);
      launch(k_visc_div<DIM>, blocks_for(p.N, THREADS), THREADS, 0, st, p);
      prof_end(pr, K_VISC_DIV, st);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = markers(Spread())) != cudaSuccess) return e;
  }
  double *out = advance ? s.Qo : s.Lout;
  prof_begin(pr, st);
  Plan q = p;
  q.src_scale = s.src_scale;
  ViscScale vs{};
  for (int a = 0; a < DIM; a++) vs.c[a] = p.mm[a] ? p.inv_Re : p.inv_h12[a] * p.inv_Re;
  const unsigned blocks = blocks_for(p.N, THREADS);
  if (!STRICT && viscous)
    launch(k_finish<DIM, !STRICT>, blocks, THREADS, 0, st, q, s.Qs, s.Qn, out, s.a, s.b, s.dt,
           advance, vs);
  else
    launch(k_finish<DIM, false>, blocks, THREADS, 0, st, q, s.Qs, s.Qn, out, s.a, s.b, s.dt,
           advance, vs);
  prof_end(pr, K_FINISH, st);
  return cudaGetLastError();
}

inline cudaError_t stage_impl(const Plan &p, const StageArgs &s, cudaStream_t st) {
  if (p.dim == 2)
    return p.scheme == IBFSA_TENO5 ? run_stage<2, IBFSA_TENO5>(p, s, st)
                                   : run_stage<2, IBFSA_WENO5JS>(p, s, st);
  return p.scheme == IBFSA_TENO5 ? run_stage<3, IBFSA_TENO5>(p, s, st)
                                 : run_stage<3, IBFSA_WENO5JS>(p, s, st);
}

inline cudaError_t wavespeed_impl(const Plan &p, const double *Q, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(p.alpha_bits, 0, 3 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  if (p.dim == 2) launch(k_pad<2>, blocks_for(p.NP, THREADS), THREADS, 0, st, p, Q);
  else launch(k_pad<3>, blocks_for(p.NP, THREADS), THREADS, 0, st, p, Q);
  return cudaGetLastError();
}

inline cudaError_t probe_impl(const Plan &p, const double *Q, int np, const double *xp,
                              double *out, cudaStream_t st, Prof *pr) {
  prof_begin(pr, st);
  cudaError_t e = wavespeed_impl(p, Q, st);  // pad + primitives of the current state
  prof_end(pr, K_PAD, st);
  if (e != cudaSuccess) return e;
  prof_begin(pr, st);
  if (p.dim == 2) k_probe<2><<<blocks_for(np, 128), 128, 0, st>>>(p, np, xp, out);
  else k_probe<3><<<blocks_for(np, 128), 128, 0, st>>>(p, np, xp, out);
  prof_end(pr, K_PROBE, st);
  return cudaGetLastError();
}

}  // namespace IBFSA_MODE_NS
}  // namespace ibfsa
