// stage_fp32.cu -- the perturbation form of one Runge-Kutta stage (arXiv:1905.00182, Sec. 2):
// the stencil arithmetic in FP32 on q' = Q - q_inf and on primitive perturbations, expanded so
// that no O(1) free-stream term ever cancels, while the RK state and its combination, the IB
// markers (Eq. 7-9) and the probes stay FP64.
//
// Perturbation algebra (u = u_inf + u', m_inf = rho_inf u_inf, H_inf = E_inf + p_inf):
//   u'_a = (m'_a - rho' u_inf_a) / rho
//   p'   = (gamma - 1) (E' - (m' . u + m_inf . u') / 2)
//   F'_d = [m'_d,  m'_i u_d + m_inf_i u'_d + p' delta_id,  (E' + p') u_d + H_inf u'_d]
// The split f+-' = (F'_d +- alpha_d q')/2 differs from f+- by a constant, and both candidate
// polynomials and smoothness indicators are invariant under constant shifts, so the
// reconstructed flux differences are those of the full fluxes.  Gradients of u equal those of
// u', and b_j = (u_inf + u')_i tau_ij.
//
// Stage values inside a step are FP32 increments over the FP64 state: with a_s + b_s = 1,
//   Q^(s+1) - Qn = b_s (Q^(s) - Qn + dt L(Q^(s))),
// so d1 = dt L(Qn), d2 = (d1 + dt L(Q1))/4 and the step ends with Qn += 2/3 (d2 + dt L(Q2)),
// added in FP64 -- the only FP64 arithmetic of the bulk.  qn32 = (float)(Qn - q_inf) is
// refreshed from the FP64 state at the end of every step, so stencil inputs never drift.
//
// TENO5 in FP32: eps = 1e-40 is below the FP32 normal range, so eps = 1e-30 is used, and the
// cut-off is evaluated on gamma_k / gamma_max = ((1 + r_k)/(1 + r_max))^6 (r = tau5/(beta + eps)),
// which keeps every quantity in [0, 1] without changing the decision gamma_k >= C_T sum gamma.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fp_bits.cuh"
#include "ibfsa_internal.h"
#include "launch.cuh"
#include "marker.cuh"
#include "mesh.cuh"
#include "mlp_tile.cuh"
#include "tma.cuh"

namespace ibfsa {
namespace fp32_ns {

constexpr int THREADS = 256;

struct Free {
  float rho, p, H, gamma, gm1;
  float u[3], m[3];
};

__device__ __forceinline__ Free free_stream(const Plan &p) {
  Free f;
  f.rho = p.rho_inf32;
  f.p = p.p_inf32;
  f.H = p.H_inf32;
  f.gamma = p.gamma32;
  f.gm1 = p.gm1_32;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    f.u[a] = p.u_inf32[a];
    f.m[a] = p.m_inf32[a];
  }
  return f;
}

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

// the boundary cell of a characteristic face along a (its normal term comes from k_char_faces32)
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

// four-point supports of point k of X [dim][stride] (Eq. 10-11; FP64, as the IB and the probes)
template <int DIM>
__device__ __forceinline__ bool point_support(const Plan &p, const double *X, int stride, int k,
                                              int j0[3], double w[3][4]) {
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    if (a < DIM) {
      double s, hl;
      if (p.mx[a]) {
        j0[a] = mesh::support_stretched(p, a, X[a * stride + k], &s, &hl);
      } else {
        s = (X[a * stride + k] - p.lo[a]) * p.inv_h[a] - 0.5;
        j0[a] = (int)floor(s) - 1;
      }
#pragma unroll
      for (int r = 0; r < 4; r++) w[a][r] = marker::peskin(s - (double)(j0[a] + r));
      if (j0[a] < 0 || j0[a] + 3 > p.n[a] - 1) ok = false;
    } else {
      j0[a] = 0;
      w[a][0] = 1.0; w[a][1] = 0.0; w[a][2] = 0.0; w[a][3] = 0.0;
    }
  }
  return ok;
}

// ------------------------------------------------------------------------------------------
// FP32 reconstructions at face i+1/2 from (f_{i-2}, ..., f_{i+2})
// ------------------------------------------------------------------------------------------
struct Cands {
  float q0, q1, q2, b0, b1, b2;
};

__device__ __forceinline__ Cands candidates(float a, float b, float c, float d, float e) {
  Cands r;
  const float s6 = 1.f / 6.f;
  r.q0 = (2.f * a - 7.f * b + 11.f * c) * s6;
  r.q1 = (-b + 5.f * c + 2.f * d) * s6;
  r.q2 = (2.f * c + 5.f * d - e) * s6;
  const float k13 = 13.f / 12.f;
  float t, u;
  t = a - 2.f * b + c; u = a - 4.f * b + 3.f * c; r.b0 = k13 * t * t + 0.25f * u * u;
  t = b - 2.f * c + d; u = b - d;                 r.b1 = k13 * t * t + 0.25f * u * u;
  t = c - 2.f * d + e; u = 3.f * c - 4.f * d + e; r.b2 = k13 * t * t + 0.25f * u * u;
  return r;
}

__device__ __forceinline__ float weno5js(float a, float b, float c, float d, float e) {
  Cands k = candidates(a, b, c, d, e);
  const float eps = 1e-6f;
  float s0 = (eps + k.b0) * (eps + k.b0);
  float s1 = (eps + k.b1) * (eps + k.b1);
  float s2 = (eps + k.b2) * (eps + k.b2);
  float al0 = 0.1f * (s1 * s2), al1 = 0.6f * (s0 * s2), al2 = 0.3f * (s0 * s1);
  return __fdividef(al0 * k.q0 + al1 * k.q1 + al2 * k.q2, al0 + al1 + al2);
}

__device__ __forceinline__ int teno_mask(const Cands &k) {
  const float eps = 1e-30f, CT = 1e-5f;
  float tau = fabsf(k.b0 - k.b2);
  float r0 = __fdividef(tau, k.b0 + eps);
  float r1 = __fdividef(tau, k.b1 + eps);
  float r2 = __fdividef(tau, k.b2 + eps);
  float inv = __fdividef(1.f, 1.f + fmaxf(r0, fmaxf(r1, r2)));
  float t, t2, g0, g1, g2;
  t = (1.f + r0) * inv; t2 = t * t; g0 = t2 * t2 * t2;
  t = (1.f + r1) * inv; t2 = t * t; g1 = t2 * t2 * t2;
  t = (1.f + r2) * inv; t2 = t * t; g2 = t2 * t2 * t2;
  float th = CT * (g0 + g1 + g2);
  return (g0 >= th ? 1 : 0) | (g1 >= th ? 2 : 0) | (g2 >= th ? 4 : 0);
}

// E: factor of the indicators' floor, for stencils scaled by its square root
template <int E = 1>
__device__ __forceinline__ float teno5(const Plan &tw, float a, float b, float c, float d,
                                       float e) {
  Cands k = candidates(a, b, c, d, e);
  const float eps = E * 1e-30f, CT = 1e-5f;
  float tau = fabsf(k.b0 - k.b2);
  float r0 = __fdividef(tau, k.b0 + eps);
  float r1 = __fdividef(tau, k.b1 + eps);
  float r2 = __fdividef(tau, k.b2 + eps);
  float inv = __fdividef(1.f, 1.f + fmaxf(r0, fmaxf(r1, r2)));
  float t, t2, g0, g1, g2;
  t = (1.f + r0) * inv; t2 = t * t; g0 = t2 * t2 * t2;
  t = (1.f + r1) * inv; t2 = t * t; g1 = t2 * t2 * t2;
  t = (1.f + r2) * inv; t2 = t * t; g2 = t2 * t2 * t2;
  float th = CT * (g0 + g1 + g2);
  int mask = (g0 >= th ? 1 : 0) | (g1 >= th ? 2 : 0) | (g2 >= th ? 4 : 0);
  const float *w = tw.teno_w32[mask];
  return w[0] * k.q0 + w[1] * k.q1 + w[2] * k.q2;
}

// Smoothness indicators only (the candidates are not needed on the smooth path).
__device__ __forceinline__ void indicators(float a, float b, float c, float d, float e,
                                           float &b0, float &b1, float &b2) {
  const float k13 = 13.f / 12.f;
  float t, u;
  t = a - 2.f * b + c; u = a - 4.f * b + 3.f * c; b0 = k13 * t * t + 0.25f * u * u;
  t = b - 2.f * c + d; u = b - d;                 b1 = k13 * t * t + 0.25f * u * u;
  t = c - 2.f * d + e; u = 3.f * c - 4.f * d + e; b2 = k13 * t * t + 0.25f * u * u;
}

// TENO5 keeps every stencil when tau5 <= 4 (min beta + eps): then each gamma_k lies in
// [1, 5^6] and chi_k >= 1/(3 5^6) = 2.1e-5 > C_T = 1e-5.  The reconstruction is then the
// optimal linear combination (2a - 13b + 47c + 27d - 3e)/60, without divisions or powers.
__device__ __forceinline__ bool teno_all_kept(float b0, float b1, float b2) {
  return fabsf(b0 - b2) <= 4.f * (fminf(b0, fminf(b1, b2)) + 1e-30f);
}

__device__ __forceinline__ float linear5(float a, float b, float c, float d, float e) {
  return (2.f * a - 13.f * b + 47.f * c + 27.f * d - 3.f * e) * (1.f / 60.f);
}

__device__ __forceinline__ float teno5_fast(const Plan &tw, float a, float b, float c, float d,
                                            float e) {
  float b0, b1, b2;
  indicators(a, b, c, d, e, b0, b1, b2);
  if (teno_all_kept(b0, b1, b2)) return linear5(a, b, c, d, e);
  return teno5(tw, a, b, c, d, e);
}

// make_float2(v, v)
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

// K adjacent faces (2, or 1), both split fluxes each, on packed FP32x2 arithmetic.  The input is
// the interleaved face stencils z_k = (f+ at staged cell i+k, f- at staged cell i+k+1), k = 0..K+3,
// of the faces after staged cells i+2, i+3: the .x lanes are the f+ stencils upwind to downwind,
// the .y lanes the f- stencils downwind to upwind, so one load per k fetches both sides.  First
// differences, second differences and their squares are taken once for both faces (each face by
// itself: 26 packed operations, the pair: 41; the passes are bound by instruction issue).  Pairs for
// single faces: TENO5 at 512^3 x 2.27 -> 1.97 ms, y and z 2.36 -> 2.22 ms (1.78, 1.99 and 2.02 since
// k_conv32_x and the exchange of k_conv32_tma); WENO5-JS at 2048^2, single faces not packed, x 95 ->
// 67 us, y 101 -> 70 us (65 and 63 since).  With the f- stencil reversed, the packed indicator of
// z0 z1 z2 is (beta_0+, beta_2-) and that of z2 z3 z4 is (beta_2+, beta_0-) (the squares are
// symmetric under the reversal), so tau5 and the all-kept test are those of each side; the linear
// combination takes per-lane coefficient pairs.
//
// TENO5: the all-kept test is scale-invariant, so the indicators are taken times 4, (13/3) t^2 +
// u^2, of twice the split flux (STAGE_SCALE), with the floor 16e-30.  The linear (all-kept) result
// is computed without branches; only when some lane of the warp has a side that cuts a stencil does
// the whole warp enter the full TENO5 (a uniform branch, no divergence to reconverge): every lane of
// the warp must call it, and v0, v1 say which of its faces exist.
// WENO5-JS: weights d_k / (eps + beta_k)^2 over their common denominator, the reconstruction as
// the middle value plus a weighted mean of the candidates' differences from it.
template <int SCHEME, int K>
__device__ __forceinline__ void faces_pz(const Plan &tw, const float2 (&z)[K + 4], bool v0, bool v1,
                                         float (&h)[K]) {
  float2 d[K + 3], kt[K + 2];
#pragma unroll
  for (int j = 0; j < K + 3; j++) d[j] = __ffma2_rn(f2(-1.f), z[j], z[j + 1]);
#pragma unroll
  for (int j = 0; j < K + 2; j++) {
    const float2 t = __ffma2_rn(f2(-1.f), d[j], d[j + 1]);
    // WENO5-JS: eps with the indicator (four times that of half the split flux)
    if constexpr (SCHEME == IBFSA_TENO5) kt[j] = __fmul2_rn(__fmul2_rn(f2(13.f / 3.f), t), t);
    else kt[j] = __ffma2_rn(__fmul2_rn(f2(13.f / 3.f), t), t, f2(1e-6f));
  }
#pragma unroll
  for (int j = 0; j < K; j++) {
    const float2 u0 = __ffma2_rn(f2(-3.f), d[j + 1], d[j]);
    const float2 u1 = __fadd2_rn(d[j + 1], d[j + 2]);
    const float2 u2 = __ffma2_rn(f2(-3.f), d[j + 2], d[j + 3]);
    float2 b0 = __ffma2_rn(u0, u0, kt[j]), b1 = __ffma2_rn(u1, u1, kt[j + 1]);
    float2 b2 = __ffma2_rn(u2, u2, kt[j + 2]);
    if constexpr (SCHEME == IBFSA_TENO5) {
      const float2 tau = __ffma2_rn(f2(-1.f), b2, b0);
      const bool kx = fabsf(tau.x) <= fmaf(4.f, fminf(b0.x, fminf(b1.x, b2.x)), 6.4e-29f);
      const bool ky = fabsf(tau.y) <= fmaf(4.f, fminf(b0.y, fminf(b1.y, b2.y)), 6.4e-29f);
      float2 lin = __fmul2_rn(make_float2(2.f / 60.f, -3.f / 60.f), z[j]);
      lin = __ffma2_rn(make_float2(-13.f / 60.f, 27.f / 60.f), z[j + 1], lin);
      lin = __ffma2_rn(f2(47.f / 60.f), z[j + 2], lin);
      lin = __ffma2_rn(make_float2(27.f / 60.f, -13.f / 60.f), z[j + 3], lin);
      lin = __ffma2_rn(make_float2(-3.f / 60.f, 2.f / 60.f), z[j + 4], lin);
      h[j] = lin.x + lin.y;
      if (__any_sync(0xffffffffu, (j ? v1 : v0) && !(kx && ky))) {
        const float hx = kx ? lin.x : teno5<4>(tw, z[j].x, z[j + 1].x, z[j + 2].x, z[j + 3].x,
                                               z[j + 4].x);
        const float hy = ky ? lin.y : teno5<4>(tw, z[j + 4].y, z[j + 3].y, z[j + 2].y, z[j + 1].y,
                                               z[j].y);
        h[j] = hx + hy;
      }
    } else {
      b0 = __fmul2_rn(b0, b0);
      b1 = __fmul2_rn(b1, b1);
      b2 = __fmul2_rn(b2, b2);
      const float2 p0 = __fmul2_rn(b1, b2), p1 = __fmul2_rn(b0, b2), p2 = __fmul2_rn(b0, b1);
      const float2 n0 = __ffma2_rn(make_float2(5.f / 60.f, -12.f / 60.f), d[j + 1],
                                   __fmul2_rn(make_float2(-2.f / 60.f, 3.f / 60.f), d[j]));
      const float2 n1 = __ffma2_rn(make_float2(0.1f, -0.2f), d[j + 1],
                                   __fmul2_rn(make_float2(0.2f, -0.1f), d[j + 2]));
      const float2 n2 = __ffma2_rn(make_float2(12.f / 60.f, -5.f / 60.f), d[j + 2],
                                   __fmul2_rn(make_float2(-3.f / 60.f, 2.f / 60.f), d[j + 3]));
      const float2 num = __ffma2_rn(p2, n2, __ffma2_rn(p1, n1, __fmul2_rn(p0, n0)));
      const float2 d01 = __ffma2_rn(f2(0.6f), p1, __fmul2_rn(make_float2(0.1f, 0.3f), p0));
      const float2 den = __ffma2_rn(make_float2(0.3f, 0.1f), p2, d01);
      h[j] = (z[j + 2].x + __fdividef(num.x, den.x)) + (z[j + 2].y + __fdividef(num.y, den.y));
    }
  }
}

// TENO5 at one face of the interleaved stencils (faces_pz): (h+, h-) and whether each side keeps
// all three stencils (by the all-kept test or, where that fails, by the full cut-off).  Every lane
// of the warp must call it.
__device__ __forceinline__ float2 teno5_pz_sides(const Plan &tw, float2 z0, float2 z1, float2 z2,
                                                 float2 z3, float2 z4, bool &kx, bool &ky) {
  float2 t0 = __fadd2_rn(__ffma2_rn(f2(-2.f), z1, z0), z2);
  float2 t1 = __fadd2_rn(__ffma2_rn(f2(-2.f), z2, z1), z3);
  float2 t2 = __fadd2_rn(__ffma2_rn(f2(-2.f), z3, z2), z4);
  float2 u0 = __ffma2_rn(f2(3.f), z2, __ffma2_rn(f2(-4.f), z1, z0));
  float2 u1 = __ffma2_rn(f2(-1.f), z3, z1);
  float2 u2 = __ffma2_rn(f2(3.f), z2, __ffma2_rn(f2(-4.f), z3, z4));
  const float2 k13 = f2(13.f / 3.f);
  float2 b0 = __ffma2_rn(__fmul2_rn(k13, t0), t0, __fmul2_rn(u0, u0));
  float2 b1 = __ffma2_rn(__fmul2_rn(k13, t1), t1, __fmul2_rn(u1, u1));
  float2 b2 = __ffma2_rn(__fmul2_rn(k13, t2), t2, __fmul2_rn(u2, u2));
  float2 tau = __ffma2_rn(f2(-1.f), b2, b0);
  kx = fabsf(tau.x) <= fmaf(4.f, fminf(b0.x, fminf(b1.x, b2.x)), 1.6e-29f);
  ky = fabsf(tau.y) <= fmaf(4.f, fminf(b0.y, fminf(b1.y, b2.y)), 1.6e-29f);
  float2 lin = __fmul2_rn(make_float2(2.f / 60.f, -3.f / 60.f), z0);
  lin = __ffma2_rn(make_float2(-13.f / 60.f, 27.f / 60.f), z1, lin);
  lin = __ffma2_rn(f2(47.f / 60.f), z2, lin);
  lin = __ffma2_rn(make_float2(27.f / 60.f, -13.f / 60.f), z3, lin);
  lin = __ffma2_rn(make_float2(-3.f / 60.f, 2.f / 60.f), z4, lin);
  if (__any_sync(0xffffffffu, !(kx && ky))) {
    if (!kx) {
      const Cands k = candidates(z0.x, z1.x, z2.x, z3.x, z4.x);
      const int mask = teno_mask(k);
      const float *w = tw.teno_w32[mask];
      lin.x = w[0] * k.q0 + w[1] * k.q1 + w[2] * k.q2;
      kx = mask == 7;
    }
    if (!ky) {
      const Cands k = candidates(z4.y, z3.y, z2.y, z1.y, z0.y);
      const int mask = teno_mask(k);
      const float *w = tw.teno_w32[mask];
      lin.y = w[0] * k.q0 + w[1] * k.q1 + w[2] * k.q2;
      ky = mask == 7;
    }
  }
  return lin;
}

// The learned weights' face loop, in two phases.  First, unrolled as the component-wise pass,
// packed TENO5 at every face and the eligibility of each side (TENO5 keeping all three stencils
// and an amplitude above the floor), one bit per (pass, component, side).  Then a rolled loop
// over (pass, component) with one call site of the warp-wide network (unrolled, the network's
// code was copied 2 x NV x MAXP times and the kernel ran out of the instruction cache) visits
// only the faces where some lane of the warp is eligible: a side with an eligible lane runs the
// network for all 32 lanes' stencils of that side, and its eligible lanes take the delta-form
// reconstruction with the network's weights.  zat(ps, c, valid) gives the interleaved stencil
// z_0 (z_k ZS float2 further) of this thread's face slot ps, component c, and whether the slot
// holds a face (an empty slot points at a valid stencil, its results unused).  Every lane of the
// warp must call it; used / seen accumulate this lane's counts.
template <int MAXP, int NV, int ZS, typename ZAt>
__device__ __forceinline__ void learned_faces(const Plan &p, const unsigned char *img,
                                              float (&Fh)[MAXP][NV], unsigned &used,
                                              unsigned &seen, ZAt zat) {
  static_assert(2 * MAXP * NV <= 32, "one eligibility bit per (pass, component, side)");
  unsigned emask = 0;
#pragma unroll
  for (int ps = 0; ps < MAXP; ps++) {
    bool valid = false;
#pragma unroll
    for (int c = 0; c < NV; c++) {
      const float2 *z = zat(ps, c, valid);
      const float2 z0 = z[0], z1 = z[ZS], z2 = z[2 * ZS], z3 = z[3 * ZS], z4 = z[4 * ZS];
      bool kx, ky;
      const float2 h = teno5_pz_sides(p, z0, z1, z2, z3, z4, kx, ky);
      Fh[ps][c] = h.x + h.y;
      // amplitude max_j |v_j - v_2| of each side (the same set of values in either order)
      const float2 d0 = __ffma2_rn(f2(-1.f), z2, z0), d1 = __ffma2_rn(f2(-1.f), z2, z1);
      const float2 d3 = __ffma2_rn(f2(-1.f), z2, z3), d4 = __ffma2_rn(f2(-1.f), z2, z4);
      const float ax = fmaxf(fmaxf(fabsf(d0.x), fabsf(d1.x)), fmaxf(fabsf(d3.x), fabsf(d4.x)));
      const float ay = fmaxf(fmaxf(fabsf(d0.y), fabsf(d1.y)), fmaxf(fabsf(d3.y), fabsf(d4.y)));
      const bool ex = valid && kx && ax > p.mlp_floor, ey = valid && ky && ay > p.mlp_floor;
      const int j = 2 * (ps * NV + c);
      emask |= (ex ? 1u << j : 0u) | (ey ? 2u << j : 0u);
    }
    seen += valid ? 2 * NV : 0;
  }
  used += __popc(emask);
#pragma unroll 1
  for (int it = 0; it < MAXP * NV; it++) {
    const unsigned bits = (emask >> (2 * it)) & 3u;
    const unsigned bx = __ballot_sync(0xffffffffu, bits & 1u);
    const unsigned by = __ballot_sync(0xffffffffu, bits & 2u);
    if ((bx | by) == 0u) continue;  // warp-uniform
    const int ps = it / NV, c = it % NV;
    bool valid;
    const float2 *z = zat(ps, c, valid);
    // phase 1's TENO5 values again, where some lane keeps one of them (a side it is not
    // eligible on): warp-uniform
    float2 h = make_float2(0.f, 0.f);
    if (__any_sync(0xffffffffu, bits != 3u)) {
      bool kx, ky;
      h = teno5_pz_sides(p, z[0], z[ZS], z[2 * ZS], z[3 * ZS], z[4 * ZS], kx, ky);
    }
#pragma unroll 1
    for (int sd = 0; sd < 2; sd++) {
      if ((sd ? by : bx) == 0u) continue;  // warp-uniform
      // this side's stencil upwind to downwind, re-read from shared memory (nothing of it stays
      // live across the network): f+ = z_0..z_4 .x, f- = z_4..z_0 .y
      const volatile float *f = reinterpret_cast<const volatile float *>(z) + sd;
      const int o = sd ? 8 * ZS : 0, st = sd ? -2 * ZS : 2 * ZS;
      float v[5];
#pragma unroll
      for (int k = 0; k < 5; k++) v[k] = f[o + k * st];
      float amp = 0.f;
#pragma unroll
      for (int k = 0; k < 5; k++) amp = fmaxf(amp, fabsf(v[k] - v[2]));
      const float inv = amp > 1e-30f ? __fdividef(1.f, amp) : 0.f;
      float x[5];
#pragma unroll
      for (int k = 0; k < 5; k++) x[k] = (v[k] - v[2]) * inv;
      float w[3];
      mlp::warp_weights2(img, x, w);
      if ((bits >> sd) & 1u) {
#pragma unroll
        for (int k = 0; k < 5; k++) v[k] = f[o + k * st];
        // delta form: constant stencils are reproduced exactly whatever the weights
        const Cands q = candidates(v[0], v[1], v[2], v[3], v[4]);
        const float hs = v[2] + w[0] * (q.q0 - v[2]) + w[1] * (q.q1 - v[2]) + w[2] * (q.q2 - v[2]);
        if (sd) h.y = hs;
        else h.x = hs;
      }
    }
    Fh[ps][c] = h.x + h.y;
  }
}

template <int SCHEME>
__device__ __forceinline__ float recon(const Plan &tw, float a, float b, float c, float d,
                                       float e) {
  if constexpr (SCHEME == IBFSA_TENO5) return teno5_fast(tw, a, b, c, d, e);
  else return weno5js(a, b, c, d, e);
}

// ------------------------------------------------------------------------------------------
// pad: q' = Q - q_inf (subtracted in FP64, then rounded to FP32), primitive perturbations,
// split speeds of the stage input
// ------------------------------------------------------------------------------------------
template <int DIM>
__global__ void __launch_bounds__(THREADS) k_pad32(Plan p, const float *__restrict__ din) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;  // padded cells fit in 31 bits
  float wmax[3] = {0.f, 0.f, 0.f};
  if (t < (unsigned)p.NP) {
    Free fs = free_stream(p);
    const unsigned r = t / (unsigned)p.P[0], rz = r / (unsigned)p.P[1];
    const int ix = (int)(t - r * p.P[0]), iy = (int)(r - rz * p.P[1]), iz = (int)rz;
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
    float q[NV];
    if (free_ghost) {
#pragma unroll
      for (int c = 0; c < NV; c++) q[c] = 0.f;
    } else {
      long long o = int_index(p, S[0], S[1], S[2]);
#pragma unroll
      for (int c = 0; c < NV; c++) q[c] = p.qn32[c * p.N + o] + (din ? din[c * p.N + o] : 0.f);
    }
#pragma unroll
    for (int c = 0; c < NV; c++) p.Qp32[c * p.NP + t] = q[c];
    float rho = fs.rho + q[0];
    float inv_rho = 1.f / rho;
    float ke2 = 0.f;  // m'.u + m_inf.u'
    float u[DIM];
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      float up = (q[1 + a] - q[0] * fs.u[a]) * inv_rho;
      u[a] = fs.u[a] + up;
      ke2 += q[1 + a] * u[a] + fs.m[a] * up;
      p.Wp32[a * p.NP + t] = up;
    }
    float pp = fs.gm1 * (q[NV - 1] - 0.5f * ke2);
    p.Wp32[DIM * p.NP + t] = pp;
    if (interior) {
      float c = sqrtf(fs.gamma * (fs.p + pp) * inv_rho);
#pragma unroll
      for (int a = 0; a < DIM; a++) wmax[a] = fabsf(u[a]) + c;
    }
  }
  __shared__ float red[3][THREADS / 32];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int a = 0; a < DIM; a++) {
    float v = wmax[a];
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) red[a][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < DIM) {
    float v = 0.f;
    for (int w = 0; w < THREADS / 32; w++) v = fmaxf(v, red[threadIdx.x][w]);
    if (!(v <= 1e30f)) atomicOr(p.status, IBFSA_STATUS_NONFINITE);
    else atomicMax(&p.alpha_bits[threadIdx.x], (unsigned long long)__double_as_longlong((double)v));
  }
}

// ------------------------------------------------------------------------------------------
// convective term along A: split flux perturbations of a tile of line segments in shared
// memory, faces of the tile (only those that exist), conservative difference into L
// ------------------------------------------------------------------------------------------
template <int A>
struct Tile {
  // A == 0: 8 lines (y) of 63 cells; otherwise 32 lines (consecutive x) of 15 cells -- two
  // faces per thread either way
  static constexpr int ROWS = A == 0 ? 8 : 32;
  static constexpr int SEG = A == 0 ? 63 : 15;
  static constexpr int LEN = SEG + 6;
  static constexpr int FACES = SEG + 1;
};

template <int DIM, int A>
constexpr size_t conv_smem() {
  return sizeof(float) * 2 * (DIM + 2) * Tile<A>::ROWS * Tile<A>::LEN;  // >= face-flux area
}

// What the split fluxes f+-' = (F' +- alpha q') / 2 are staged as (a power of two: the same bits):
// the fixed component-wise schemes stage F' +- alpha q' itself for TENO5, which depends on ratios of
// indicators only (its floors take the square of the scale), and half of f+-' for WENO5-JS, whose
// indicators (eps is not scale-free) come out times four; every other form (-1) stages f+-'.
template <int SCHEME>
constexpr float STAGE_SCALE = SCHEME < 0 ? 0.5f : SCHEME == IBFSA_TENO5 ? 1.f : 0.25f;
// and what takes a flux difference back
template <int SCHEME>
constexpr float FLUX_SCALE = 0.5f / STAGE_SCALE<SCHEME>;

// split fluxes along A of one staged cell, from q', u'_A and p'; F' is the perturbation-expanded
// flux (no O(1) free-stream terms cancel)
template <int DIM, int A, int SCHEME = -1>
__device__ __forceinline__ void split_cell(const Free &fs, float alpha, const float q[DIM + 2],
                                           float up, float pp, float fpv[DIM + 2],
                                           float fmv[DIM + 2]) {
  constexpr int NV = DIM + 2;
  const float ua = fs.u[A] + up;
#pragma unroll
  for (int c = 0; c < NV; c++) {
    float F;
    if (c == 0) F = q[1 + A];
    else if (c == NV - 1) F = (q[c] + pp) * ua + fs.H * up;
    else {
      F = q[c] * ua + fs.m[c - 1] * up;
      if (c - 1 == A) F += pp;
    }
    const float aq = alpha * q[c];
    fpv[c] = STAGE_SCALE<SCHEME> * (F + aq);
    fmv[c] = STAGE_SCALE<SCHEME> * (F - aq);
  }
}

// Characteristic-wise option in the perturbation form: eigenvectors of the Euler flux Jacobian
// along A at the Roe average of the face's two cells, from their full primitive state
// (rho_inf + rho', u_inf + u', p_inf + p'), H = gamma p/((gamma - 1) rho) + |u|^2/2; right
// eigenvectors are the columns of R, left ones the rows of Lv, in the order u-c, entropy,
// shears, u+c.  The split-flux perturbations are projected on them: their constant free-stream
// part would pass through L and R unchanged and cancel in the face difference.
// Whether entry c of left eigenvector k is zero whatever the state: the shears (k = 2 .. NV-2, one
// per direction but A in increasing order) have entries for the density and their own momentum
// only.  (Right eigenvectors: the momentum rows have the same zeros, the density row all shears'.)
template <int DIM, int A>
__host__ __device__ constexpr bool shear_zero(int k, int c) {
  if (k < 2 || k > DIM || c == 0) return false;
  const int t = k - 2, b = t < A ? t : t + 1;  // the shear's direction
  return c != 1 + b;
}

template <int DIM, int A>
__device__ __forceinline__ void roe_eigen32(const Free &fs, const float wl[DIM + 2],
                                            const float wr[DIM + 2], float R[DIM + 2][DIM + 2],
                                            float Lv[DIM + 2][DIM + 2]) {
  // w = [rho', u'_0 .. u'_{DIM-1}, p']
  constexpr int NV = DIM + 2;
  const float rl = fs.rho + wl[0], rr = fs.rho + wr[0];
  const float sl = sqrtf(rl), sr = sqrtf(rr), inv = 1.f / (sl + sr);
  const float kap = fs.gamma / fs.gm1;
  float u[DIM], kl = 0.f, kr = 0.f;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    float ul = fs.u[b] + wl[1 + b], ur = fs.u[b] + wr[1 + b];
    u[b] = (sl * ul + sr * ur) * inv;
    kl += ul * ul;
    kr += ur * ur;
  }
  const float Hl = kap * (fs.p + wl[NV - 1]) / rl + 0.5f * kl;
  const float Hr = kap * (fs.p + wr[NV - 1]) / rr + 0.5f * kr;
  const float H = (sl * Hl + sr * Hr) * inv;
  float q2 = 0.f;
#pragma unroll
  for (int b = 0; b < DIM; b++) q2 += u[b] * u[b];
  const float c2 = fs.gm1 * (H - 0.5f * q2);
  const float c = sqrtf(c2), ic = 1.f / c;
  const float b1 = fs.gm1 / c2, b2 = 0.5f * q2 * b1;
  const float ua = u[A];
#pragma unroll
  for (int i = 0; i < NV; i++)
#pragma unroll
    for (int j = 0; j < NV; j++) {
      R[i][j] = 0.f;
      Lv[i][j] = 0.f;
    }
  constexpr int km = 0, ke = 1, kp = NV - 1;
  R[0][km] = 1.f;
  R[0][ke] = 1.f;
  R[0][kp] = 1.f;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    R[1 + b][km] = u[b] - (b == A ? c : 0.f);
    R[1 + b][ke] = u[b];
    R[1 + b][kp] = u[b] + (b == A ? c : 0.f);
  }
  R[NV - 1][km] = H - ua * c;
  R[NV - 1][ke] = 0.5f * q2;
  R[NV - 1][kp] = H + ua * c;
  Lv[km][0] = 0.5f * (b2 + ua * ic);
  Lv[kp][0] = 0.5f * (b2 - ua * ic);
  Lv[ke][0] = 1.f - b2;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    Lv[km][1 + b] = 0.5f * (-b1 * u[b] - (b == A ? ic : 0.f));
    Lv[kp][1 + b] = 0.5f * (-b1 * u[b] + (b == A ? ic : 0.f));
    Lv[ke][1 + b] = b1 * u[b];
  }
  Lv[km][NV - 1] = 0.5f * b1;
  Lv[kp][NV - 1] = 0.5f * b1;
  Lv[ke][NV - 1] = -b1;
  int t = 0;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    if (b == A) continue;
    R[1 + b][2 + t] = 1.f;
    R[NV - 1][2 + t] = u[b];
    Lv[2 + t][0] = -u[b];
    Lv[2 + t][1 + b] = 1.f;
    t++;
  }
}

// Tiles by plain loads: the learned weights and the characteristic-wise option in every direction,
// the fixed component-wise schemes along y and z where the x extent is not a multiple of 4.  Six
// blocks per SM (42 registers) for the fixed schemes, four (64) for the learned form's warp-wide
// network tiles.  The characteristic-wise option: four blocks for y and z, three for x (85
// registers; four there spill and are 6 % slower); with one (138 registers, and each stencil
// loaded and projected with the eigenvectors' zeros, field by field) a pass over 160 x 144 x 150
// took 432 / 559 / 543 us, now 213 / 191 / 181 us.  The x pass gives each warp one row of the tile.
constexpr int conv32_blocks(int a, int scheme, bool chr) {
  return scheme == IBFSA_MLP_TENO5 ? 4 : chr ? (a == 0 ? 3 : 4) : 6;
}

template <int DIM, int A, int SCHEME, bool CHAR = false>
__global__ void __launch_bounds__(THREADS, conv32_blocks(A, SCHEME, CHAR))
    k_conv32(Plan p, int first) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  using T = Tile<A>;
  static_assert(A != 0 || T::ROWS * 32 == THREADS, "x pass: one warp per row");
  // face fluxes are stored with an odd row stride when a warp walks the rows (A != 0), so the
  // 32 lanes hit 32 different banks
  constexpr int FST = A == 0 ? T::FACES : T::FACES + 1;
  extern __shared__ float smf[];
  // the component-wise forms stage the interleaved face stencils z_l = (f+ at l, f- at l+1),
  // [NV][ROWS][LEN] float2; the characteristic-wise option f+ and f- apart, [NV][ROWS][LEN]
  constexpr bool ZL = !CHAR;
  // faces of a thread: one row's adjacent pair (component-wise), or THREADS apart
  constexpr bool PAIR = !CHAR && SCHEME != IBFSA_MLP_TENO5;
  float *sfp = smf;
  float *sfm = smf + NV * T::ROWS * T::LEN;
  const float alpha = (float)__longlong_as_double((long long)p.alpha_bits[A]);
  Free fs = free_stream(p);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  int seg0, line0, other;
  if constexpr (A == 0) {
    seg0 = blockIdx.x * T::SEG;
    line0 = blockIdx.y * T::ROWS;
    other = blockIdx.z;
  } else {
    int nseg = (p.n[A] + T::SEG - 1) / T::SEG;
    seg0 = (blockIdx.x % nseg) * T::SEG;
    line0 = (blockIdx.x / nseg) * T::ROWS;
    other = blockIdx.y;
  }
  const int ncell = min(T::SEG, p.n[A] - seg0);   // cells of this tile along A
  const int nface = ncell + 1;
  const int nrow = A == 0 ? min(T::ROWS, p.n[1] - line0) : min(T::ROWS, p.n[0] - line0);
  // 32-bit offsets inside one component array: padded cell (row, l) and interior cell (row, l)
  const int PX = p.P[0], PXY = p.P[0] * p.P[1];
  const int NX = p.n[0], NXY = p.n[0] * p.n[1];
  int pbase, prs, pas, ibase, irs, ias;
  if constexpr (A == 0) {
    pbase = (other + p.g[2]) * PXY + (line0 + p.g[1]) * PX + (seg0 + p.g[0]);
    prs = PX; pas = 1;
    ibase = other * NXY + line0 * NX + seg0;
    irs = NX; ias = 1;
  } else {
    int y = A == 1 ? seg0 : other, z = A == 1 ? other : seg0;
    pbase = (z + p.g[2]) * PXY + (y + p.g[1]) * PX + (line0 + p.g[0]);
    prs = 1; pas = A == 1 ? PX : PXY;
    ibase = z * NXY + y * NX + line0;
    irs = 1; ias = A == 1 ? NX : NXY;
  }
  const float *Wa = p.Wp32 + (size_t)A * p.NP;
  const float *Wpr = p.Wp32 + (size_t)DIM * p.NP;

  if constexpr (SCHEME == IBFSA_MLP_TENO5) {
    mlp::stage_inference_image(reinterpret_cast<uint4 *>(smf + 2 * NV * T::ROWS * T::LEN),
                               reinterpret_cast<const uint4 *>(p.mlp_img), threadIdx.x, THREADS);
  }
  // 1. f+-' of the staged cells (seg0-3 .. seg0+ncell+2)
  constexpr int S1 = A == 0 ? (T::LEN + 31) / 32 : (T::ROWS * T::LEN + THREADS - 1) / THREADS;
#pragma unroll
  for (int k = 0; k < S1; k++) {
    int row, l;
    if constexpr (A == 0) {
      row = warp;
      l = lane + 32 * k;
      if (l >= T::LEN) break;
    } else {
      const int e = threadIdx.x + k * THREADS;
      if (e >= T::ROWS * T::LEN) break;
      row = e % T::ROWS;
      l = e / T::ROWS;
    }
    if (row >= nrow || l >= ncell + 6) continue;
    const int s = pbase + row * prs + (l - 3) * pas;
    float q[NV], fpv[NV], fmv[NV];
#pragma unroll
    for (int c = 0; c < NV; c++) q[c] = p.Qp32[(size_t)c * p.NP + s];
    split_cell<DIM, A, PAIR ? SCHEME : -1>(fs, alpha, q, Wa[s], Wpr[s], fpv, fmv);
    if constexpr (ZL) {
#pragma unroll
      for (int c = 0; c < NV; c++) {
        float2 *zr = reinterpret_cast<float2 *>(smf) + (c * T::ROWS + row) * T::LEN;
        zr[l].x = fpv[c];
        if (l > 0) zr[l - 1].y = fmv[c];
      }
    } else {
#pragma unroll
      for (int c = 0; c < NV; c++) {
        sfp[(c * T::ROWS + row) * T::LEN + l] = fpv[c];
        sfm[(c * T::ROWS + row) * T::LEN + l] = fmv[c];
      }
    }
  }
  __syncthreads();

  // 2. faces m+1/2, m = seg0-1 .. seg0+ncell-1 (tile face index fi = m - seg0 + 1)
  constexpr int MAXP = (T::ROWS * T::FACES + THREADS - 1) / THREADS;
  float Fh[MAXP][NV];
  // the thread's face slot ps (row >= nrow or fi >= nface: none).  Learned weights along x: the
  // tile's existing faces are numbered through its rows, so that a short last tile fills a few warps
  // (the network costs a warp the same for one face as for 32): at 128^3, where the third tile of a
  // row holds 2 of its 63 cells, the pass takes 870 us (1038 with the slots numbered through all 64
  // places of a row).
  const unsigned face_magic = 65536u / nface + 1;  // e / nface for e < 512, nface <= 64
  auto face_of = [&](int ps, int &row, int &fi) {
    const int e = threadIdx.x + ps * THREADS;
    if constexpr (PAIR) { row = lane; fi = 2 * warp + ps; }
    else if constexpr (A == 0 && SCHEME == IBFSA_MLP_TENO5) {
      row = (int)(e * face_magic >> 16);
      fi = e - row * nface;
    } else if constexpr (A == 0) { row = e / T::FACES; fi = e % T::FACES; }
    else { row = e % T::ROWS; fi = e / T::ROWS; }
  };
  if constexpr (SCHEME == IBFSA_MLP_TENO5) {
    unsigned char *img = reinterpret_cast<unsigned char *>(smf + 2 * NV * T::ROWS * T::LEN);
    unsigned used = 0, seen = 0;
    const float2 *Z = reinterpret_cast<const float2 *>(smf);
    learned_faces<MAXP, NV, 1>(p, img, Fh, used, seen, [&](int ps, int c, bool &valid) {
      int row, fi;
      face_of(ps, row, fi);
      valid = row < nrow && fi < nface;
      if (!valid) { row = 0; fi = 0; }  // in-bounds reads; results discarded
      return Z + (c * T::ROWS + row) * T::LEN + fi;
    });
    used = __reduce_add_sync(0xffffffffu, used);  // warp totals
    seen = __reduce_add_sync(0xffffffffu, seen);
    if ((threadIdx.x & 31) == 0 && seen) {
      atomicAdd(&p.mlp_counts[0], (unsigned long long)used);
      atomicAdd(&p.mlp_counts[1], (unsigned long long)seen);
    }
  } else if constexpr (CHAR) {
    // characteristic-wise: per face the Roe-averaged eigen-system of cells m and m+1 (staged
    // cells fi + 2 and fi + 3), the stencils of each characteristic field, back-projection
#pragma unroll 1
    for (int ps = 0; ps < MAXP; ps++) {
      int e = threadIdx.x + ps * THREADS;
      int row, fi;
      if constexpr (A == 0) { row = e / T::FACES; fi = e % T::FACES; }
      else { row = e % T::ROWS; fi = e / T::ROWS; }
#pragma unroll
      for (int c = 0; c < NV; c++) Fh[ps][c] = 0.f;
      if (e < T::ROWS * T::FACES && row < nrow && fi < nface) {
        const int b = fi + 2;
        const int sl = pbase + row * prs + (b - 3) * pas, sr = sl + pas;
        float wl[NV], wr[NV];
        wl[0] = p.Qp32[sl];
        wr[0] = p.Qp32[sr];
#pragma unroll
        for (int k = 0; k <= DIM; k++) {
          wl[1 + k] = p.Wp32[(size_t)k * p.NP + sl];
          wr[1 + k] = p.Wp32[(size_t)k * p.NP + sr];
        }
        float Rm[NV][NV], Lv[NV][NV];
        roe_eigen32<DIM, A>(fs, wl, wr, Rm, Lv);
        // one side after the other: its stencils of all components are loaded once (a load per
        // field and component made 250 of them per face), and the eigenvectors' structural zeros
        // (shear_zero) are skipped; each product sum in the order of the components
        float hk[NV];
#pragma unroll
        for (int k = 0; k < NV; k++) hk[k] = 0.f;
#pragma unroll 1
        for (int sd = 0; sd < 2; sd++) {
          const float *f0 = (sd ? sfm + b + 3 : sfp + b - 2) + row * T::LEN;
          const int st = sd ? -1 : 1;
          float f[NV][5];
#pragma unroll
          for (int c = 0; c < NV; c++)
#pragma unroll
            for (int r = 0; r < 5; r++) f[c][r] = f0[c * T::ROWS * T::LEN + r * st];
#pragma unroll
          for (int k = 0; k < NV; k++) {
            float v[5];
#pragma unroll
            for (int r = 0; r < 5; r++) {
              float acc = 0.f;
#pragma unroll
              for (int c = 0; c < NV; c++)
                if (!shear_zero<DIM, A>(k, c)) acc = fmaf(Lv[k][c], f[c][r], acc);
              v[r] = acc;
            }
            hk[k] += recon<SCHEME>(p, v[0], v[1], v[2], v[3], v[4]);
          }
        }
#pragma unroll
        for (int c = 0; c < NV; c++) {
          float acc = 0.f;
#pragma unroll
          for (int k = 0; k < NV; k++)
            if (!(c == 0 ? k > 1 && k < NV - 1 : c < NV - 1 && shear_zero<DIM, A>(k, c)))
              acc = fmaf(Rm[c][k], hk[k], acc);
          Fh[ps][c] = acc;
        }
      }
    }
  } else {
    // the thread's pair of adjacent faces fi, fi + 1 (face fi + 1/2 - 1 between staged cells fi + 2
    // and fi + 3: z_fi .. z_fi+4).  Every lane of the warp takes part (the slow path is warp-
    // uniform): lanes without a face evaluate a valid one and store nothing.
    static_assert(MAXP == 2, "two faces per thread");
    static_assert(!PAIR || A != 0, "the x pass is k_conv32_x");
    int row = lane, fi = 2 * warp;
    const bool v0 = row < nrow && fi < nface, v1 = row < nrow && fi + 1 < nface;
    if (!v0) fi = 0;
    if (row >= nrow) row = 0;
    const float2 *zr = reinterpret_cast<const float2 *>(smf) + row * T::LEN + fi;
#pragma unroll
    for (int c = 0; c < NV; c++) {
      float2 z[6];
#pragma unroll
      for (int j = 0; j < 6; j++) z[j] = zr[c * T::ROWS * T::LEN + j];
      float h[2];
      faces_pz<SCHEME, 2>(p, z, v0, v1, h);
      Fh[0][c] = h[0];
      Fh[1][c] = h[1];
    }
  }
  __syncthreads();
  float *sh = smf;
#pragma unroll
  for (int ps = 0; ps < MAXP; ps++) {
    int row, fi;
    face_of(ps, row, fi);
    if (row < nrow && fi < nface) {
#pragma unroll
      for (int c = 0; c < NV; c++) sh[(c * T::ROWS + row) * FST + fi] = Fh[ps][c];
    }
  }
  __syncthreads();

  // 3. L' = L' - (Fhat_{m+1/2} - Fhat_{m-1/2}) / (dx/dxi)
  constexpr int S3 = A == 0 ? (T::SEG + 31) / 32 : (T::ROWS * T::SEG + THREADS - 1) / THREADS;
#pragma unroll
  for (int k = 0; k < S3; k++) {
    int row, l;
    if constexpr (A == 0) {
      row = warp;
      l = lane + 32 * k;
      if (l >= T::SEG) break;
    } else {
      const int e = threadIdx.x + k * THREADS;
      if (e >= T::ROWS * T::SEG) break;
      row = e % T::ROWS;
      l = e / T::ROWS;
    }
    if (row >= nrow || l >= ncell) continue;
    int o = ibase + row * irs + l * ias;
    // the boundary cell of a characteristic face takes its normal term from k_char_faces32
    const float inv_h = char_cell(p, A, seg0 + l)
                            ? 0.f : FLUX_SCALE<PAIR ? SCHEME : -1> * mesh::inv32(p, A, seg0 + l);
#pragma unroll
    for (int c = 0; c < NV; c++) {
      const float *hh = sh + (c * T::ROWS + row) * FST;
      float d = (hh[l + 1] - hh[l]) * inv_h;
      float *Lc = p.L32 + (size_t)c * p.N;
      Lc[o] = (first ? 0.f : Lc[o]) - d;
    }
  }
}

// ------------------------------------------------------------------------------------------
// x pass of the fixed component-wise schemes (the first pass: L' is written)
// ------------------------------------------------------------------------------------------
// LPR lanes per row of up to 2 LPR cells, two adjacent faces per lane; the rows of a block are
// numbered through y and z.  After the staged split fluxes everything stays in the row's lanes:
// the right face of a lane's second cell is its neighbour's first face (a shuffle), and that of a
// full row's last cell is taken by the row's first NV lanes, one component each.  The last six
// staged cells of all rows are staged together by a few warps.  One barrier, no face fluxes in
// shared memory.
// Against tiles of 63 cells whose face fluxes went through shared memory: TENO5 at 512^3 1.97 ->
// 1.78 ms (eight rows of 64 instead of nine of 63, two barriers and 30 shared-memory accesses per
// lane fewer); WENO5-JS at 2048^2 66.5 -> 64.8 us.  Five blocks per SM for TENO5 (1.81 ms with six,
// which spill), six for WENO5-JS (69 us with five).
template <int DIM, int LPR>
struct RowTile {
  static constexpr int NV = DIM + 2, CELLS = 2 * LPR, PITCH = CELLS + 6, RW = 32 / LPR;
  static constexpr int ROWS = RW * THREADS / 32;
  static constexpr size_t BYTES = sizeof(float2) * NV * ROWS * PITCH;
};

template <int DIM, int SCHEME, int LPR>
__global__ void __launch_bounds__(THREADS, SCHEME == IBFSA_TENO5 ? 5 : 6)
    k_conv32_x(Plan p, int seg, int nseg) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  using T = RowTile<DIM, LPR>;
  extern __shared__ __align__(16) float2 sz[];   // [NV][ROWS][PITCH]: z_l = (f+ at l, f- at l+1)
  constexpr int SC = T::ROWS * T::PITCH;
  const float alpha = (float)__longlong_as_double((long long)p.alpha_bits[0]);
  const int lane = threadIdx.x & 31, sl = lane % LPR, row = (threadIdx.x >> 5) * T::RW + lane / LPR;
  const int seg0 = (int)(blockIdx.x % nseg) * seg, row0 = (int)(blockIdx.x / nseg) * T::ROWS;
  const int ncell = min(seg, p.n[0] - seg0), nface = ncell + 1, nrows = p.n[1] * p.n[2];
  if (ncell <= 0) return;
  const bool own = row0 + row < nrows;
  // padded offset of staged cell 0 (cell seg0 - 3) of row r of the tile (rows past the end: the last)
  auto padded = [&](int r) {
    const int R = min(row0 + r, nrows - 1), z = R / p.n[1], y = R - z * p.n[1];
    return ((z + p.g[2]) * p.P[1] + y + p.g[1]) * p.P[0] + seg0 + p.g[0] - 3;
  };
  const Free fs = free_stream(p);
  const float *Wa = p.Wp32, *Wpr = p.Wp32 + (size_t)DIM * p.NP;
  auto stage = [&](int r, int l, int s) {
    float q[NV], fp[NV], fm[NV];
#pragma unroll
    for (int c = 0; c < NV; c++) q[c] = p.Qp32[(size_t)c * p.NP + s];
    split_cell<DIM, 0, SCHEME>(fs, alpha, q, Wa[s], Wpr[s], fp, fm);
    float2 *z = sz + r * T::PITCH + l;
#pragma unroll
    for (int c = 0; c < NV; c++) {
      z[c * SC].x = fp[c];
      if (l > 0) z[c * SC - 1].y = fm[c];
    }
  };
  const int pb = padded(row);
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const int l = sl + k * LPR;
    if (l < ncell + 6) stage(row, l, pb + l);
  }
  if (ncell + 6 > T::CELLS && threadIdx.x < 6 * T::ROWS) {
    const int r = threadIdx.x / 6, l = T::CELLS + threadIdx.x % 6;
    if (l < ncell + 6) stage(r, l, padded(r) + l);
  }
  __syncthreads();
  const int fi = min(2 * sl, (nface - 1) & ~1);  // lanes past the last face repeat its pair
  const bool v0 = own && 2 * sl < nface, v1 = own && 2 * sl + 1 < nface;
  const float4 *z4 = reinterpret_cast<const float4 *>(sz + row * T::PITCH + fi);
  float h0[NV], h1[NV], hn[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) {
    float2 z[6];
#pragma unroll
    for (int j = 0; j < 3; j++) {
      const float4 v = z4[c * (SC / 2) + j];
      z[2 * j] = make_float2(v.x, v.y);
      z[2 * j + 1] = make_float2(v.z, v.w);
    }
    float h[2];
    faces_pz<SCHEME, 2>(p, z, v0, v1, h);
    h0[c] = h[0];
    h1[c] = h[1];
    hn[c] = __shfl_down_sync(0xffffffffu, h[0], 1, LPR);
  }
  if (ncell == T::CELLS) {  // the last face of a full row
    float2 z[5];
    const float2 *zl = sz + min(sl, NV - 1) * SC + row * T::PITCH + T::CELLS;
#pragma unroll
    for (int j = 0; j < 5; j++) z[j] = zl[j];
    float h[1];
    faces_pz<SCHEME, 1>(p, z, own && sl < NV, false, h);
#pragma unroll
    for (int c = 0; c < NV; c++) {
      const float v = __shfl_sync(0xffffffffu, h[0], c, LPR);
      if (sl == LPR - 1) hn[c] = v;
    }
  }
  // L' = 0 - (Fhat_{m+1/2} - Fhat_{m-1/2}) / (dx/dxi) of cells 2 sl, 2 sl + 1; the boundary cell of
  // a characteristic face takes its normal term from k_char_faces32
  const int l = 2 * sl, i = seg0 + l;
  if (!own || l >= ncell) return;
  const bool two = l + 1 < ncell;
  const float inv0 = char_cell(p, 0, i) ? 0.f : FLUX_SCALE<SCHEME> * mesh::inv32(p, 0, i);
  const float inv1 =
      !two || char_cell(p, 0, i + 1) ? 0.f : FLUX_SCALE<SCHEME> * mesh::inv32(p, 0, i + 1);
  float *L = p.L32 + (size_t)(row0 + row) * p.n[0] + i;
  const bool pair = two && !(p.n[0] & 1);  // 8-byte stores: rows and segments start at even cells
#pragma unroll
  for (int c = 0; c < NV; c++) {
    const float d0 = 0.f - (h1[c] - h0[c]) * inv0, d1 = 0.f - (hn[c] - h1[c]) * inv1;
    float *Lc = L + (size_t)c * p.N;
    if (pair) *reinterpret_cast<float2 *>(Lc) = make_float2(d0, d1);
    else {
      Lc[0] = d0;
      if (two) Lc[1] = d1;
    }
  }
}

// y and z passes of the fixed schemes with tensor copies (x extent a multiple of 4, so every
// stride of the copied tensors is a multiple of 16 bytes).  A tile is 32 consecutive x-lines by
// the staged cells along A; a warp covers the 32 lines of one position along A, so there is no
// index division and every shared-memory access of a warp falls in 32 banks.
//   shared memory: [ q' (NV) | u'_A | p' ] staged cells, [NV][LEN][32], reused for the block's
//   L' [NV][SEG][32] once the split fluxes are built; f+ at staged cells 0..LEN-2 and f- at
//   1..LEN-1 (the only ones the faces read), [NV][LEN-1][32] each, reused for the face fluxes;
//   one barrier.  44 KB in 3D: five blocks per SM.
// One thread issues the copies: the staged inputs (three copies) at entry, the block's L' after
// the split fluxes (its latency hides behind the reconstruction); L' is updated in shared
// memory and written back with a tensor store.  Waits are bounded: on expiry the block reports
// IBFSA_STATUS_TIMEOUT and ends.
template <int DIM, int A>
struct TmaTile {
  using T = Tile<A>;
  static constexpr int NV = DIM + 2, R = T::ROWS, LEN = T::LEN, SEG = T::SEG;
  static constexpr int IN = (NV + 2) * LEN * R;     // floats of the staged inputs
  static constexpr int LT = NV * SEG * R;           // floats of the L' tile
  static constexpr int SF = NV * (LEN - 1) * R;     // floats of f+ (and of f-)
  static constexpr size_t BYTES = sizeof(float) * (IN + 2 * SF) + 16;
  static_assert(LT <= IN, "the L' tile reuses the staged inputs");
  static_assert(R == 32, "one warp spans the x-lines of a tile");
};

// Wait (bounded) for phase `parity` of the block's barrier; every thread of the block calls it.
// On expiry the block reports IBFSA_STATUS_TIMEOUT, thread 0 waits once more (bounded) for
// copies still in flight, and the function returns false: the caller then returns.
__device__ __forceinline__ bool block_wait_or_report(const Plan &p, uint64_t *bar,
                                                     uint32_t parity) {
  if (__syncthreads_or(!tma::mbar_wait(bar, parity))) {
    if (threadIdx.x == 0) {
      atomicOr(p.status, IBFSA_STATUS_TIMEOUT);
      tma::mbar_wait(bar, parity);
    }
    return false;
  }
  return true;
}

template <int DIM, int A, int SCHEME>
__global__ void __launch_bounds__(THREADS, SCHEME == IBFSA_MLP_TENO5 ? 4 : 5)
    k_conv32_tma(Plan p, const __grid_constant__ CUtensorMap tq,
                 const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tl) {
  begin_kernel();
  using TT = TmaTile<DIM, A>;
  using T = Tile<A>;
  constexpr int NV = TT::NV, R = TT::R, LEN = TT::LEN, SEG = TT::SEG;
  constexpr int FST = T::FACES + 1;
  // faces of a thread: an adjacent pair (fixed schemes), or NW apart (learned weights)
  constexpr bool PAIR = SCHEME != IBFSA_MLP_TENO5;
  extern __shared__ __align__(128) float smf[];
  float *in = smf;                         // [NV + 2][LEN][R], then L' [NV][SEG][R]
  float *sfp = smf + TT::IN;               // [NV][LEN - 1][R]: f+ at staged cells 0..LEN-2
  float *sfm = sfp + TT::SF;               // [NV][LEN - 1][R]: f- at staged cells 1..LEN-1
  uint64_t *bar = reinterpret_cast<uint64_t *>(sfm + TT::SF);
  // the learned weights' parameter image follows the barrier (16-byte aligned)
  unsigned char *img = reinterpret_cast<unsigned char *>(bar) + 16;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = THREADS / 32;
  static_assert((sizeof(float) * (TT::IN + 2 * TT::SF) + 16) % 16 == 0, "image alignment");

  const int nseg = (p.n[A] + SEG - 1) / SEG;
  const int seg0 = (blockIdx.x % nseg) * SEG;
  const int line0 = (blockIdx.x / nseg) * R;
  const int other = blockIdx.y;
  const int ncell = min(SEG, p.n[A] - seg0);
  const int nface = ncell + 1;
  const bool row_ok = lane < min(R, p.n[0] - line0);
  const int yi = A == 1 ? seg0 : other, zi = A == 1 ? other : seg0;  // first owned cell

  if (threadIdx.x == 0) tma::mbar_init(bar, 1);
  if constexpr (SCHEME == IBFSA_MLP_TENO5)
    mlp::stage_inference_image(reinterpret_cast<uint4 *>(img),
                               reinterpret_cast<const uint4 *>(p.mlp_img), threadIdx.x, THREADS);
  __syncthreads();
  if (threadIdx.x == 0) {
    tma::mbar_expect_tx(bar, (uint32_t)(sizeof(float) * TT::IN));
    const int px = line0 + p.g[0];
    const int py = (A == 1 ? yi - 3 : yi) + p.g[1], pz = (A == 2 ? zi - 3 : zi) + p.g[2];
    tma::load_4d(in, &tq, px, py, pz, 0, bar);
    tma::load_4d(in + NV * LEN * R, &tw, px, py, pz, A, bar);
    tma::load_4d(in + (NV + 1) * LEN * R, &tw, px, py, pz, DIM, bar);
  }
  if (!block_wait_or_report(p, bar, 0)) return;

  // 1. f+-' of the staged cells l = 0 .. ncell+5 (cells seg0-3 .. seg0+ncell+2)
  const float alpha = (float)__longlong_as_double((long long)p.alpha_bits[A]);
  {
    Free fs = free_stream(p);
#pragma unroll
    for (int k = 0; k < (LEN + NW - 1) / NW; k++) {
      const int l = warp + k * NW;
      if (l >= ncell + 6) break;
      float q[NV], fpv[NV], fmv[NV];
#pragma unroll
      for (int c = 0; c < NV; c++) q[c] = in[(c * LEN + l) * R + lane];
      split_cell<DIM, A, PAIR ? SCHEME : -1>(fs, alpha, q, in[(NV * LEN + l) * R + lane],
                                             in[((NV + 1) * LEN + l) * R + lane], fpv, fmv);
      // interleaved face stencils z_l = (f+ at l, f- at l+1), [NV][LEN-1][R] float2
      float2 *Z = reinterpret_cast<float2 *>(sfp);
#pragma unroll
      for (int c = 0; c < NV; c++) {
        if (l < LEN - 1) Z[(c * (LEN - 1) + l) * R + lane].x = fpv[c];
        if (l > 0) Z[(c * (LEN - 1) + l - 1) * R + lane].y = fmv[c];
      }
    }
  }
  __syncthreads();
  // the staged inputs are consumed: the block's L' comes into their place
  if (threadIdx.x == 0) {
    tma::mbar_expect_tx(bar, (uint32_t)(sizeof(float) * TT::LT));
    tma::load_4d(in, &tl, line0, yi, zi, 0, bar);
  }

  // 2. faces fi = warp, warp + NW (face m+1/2 with m = seg0-1+fi): f+ at staged cells
  //    fi .. fi+4, f- at fi+1 .. fi+5
  constexpr int MAXP = (T::FACES + NW - 1) / NW;
  float Fh[MAXP][NV];
  if constexpr (SCHEME == IBFSA_MLP_TENO5) {
    const float2 *Z = reinterpret_cast<const float2 *>(sfp);
    unsigned used = 0, seen = 0;
    learned_faces<MAXP, NV, R>(p, img, Fh, used, seen, [&](int ps, int c, bool &valid) {
      int fi = warp + ps * NW;
      valid = fi < nface && row_ok;
      if (fi >= nface) fi = 0;  // in-bounds reads; results discarded
      return Z + (c * (LEN - 1) + fi) * R + lane;
    });
    used = __reduce_add_sync(0xffffffffu, used);  // warp totals
    seen = __reduce_add_sync(0xffffffffu, seen);
    if (lane == 0 && seen) {
      atomicAdd(&p.mlp_counts[0], (unsigned long long)used);
      atomicAdd(&p.mlp_counts[1], (unsigned long long)seen);
    }
  } else {
    static_assert(MAXP == 2, "two faces per thread");
    const int fi = 2 * warp;  // the same for the whole warp
    if (fi < nface) {
#pragma unroll
      for (int c = 0; c < NV; c++) {
        const float2 *zc = reinterpret_cast<const float2 *>(sfp) + (c * (LEN - 1) + fi) * R + lane;
        float2 z[6];
#pragma unroll
        for (int j = 0; j < 6; j++) z[j] = zc[j * R];
        float h[2];
        faces_pz<SCHEME, 2>(p, z, row_ok, row_ok && fi + 1 < nface, h);
        Fh[0][c] = h[0];
        Fh[1][c] = h[1];
      }
    }
  }
  __syncthreads();
  // 3. L' = L' - (Fhat_{m+1/2} - Fhat_{m-1/2}) / (dx/dxi) on the copied tile, then stored back
  auto inverse = [&](int l) {
    return char_cell(p, A, seg0 + l) ? 0.f
                                     : FLUX_SCALE<PAIR ? SCHEME : -1> * mesh::inv32(p, A, seg0 + l);
  };
  if constexpr (PAIR) {
    // a warp owns faces 2 warp, 2 warp + 1 and the cells right of them; only the second cell's
    // right face, the next warp's first, goes through shared memory (all of them before: with the
    // staged fluxes' factor of a half left out, 2.22 -> 2.00 ms at 512^3)
    float *sx = sfp;  // [NW][NV][R]
    if (2 * warp < nface) {
#pragma unroll
      for (int c = 0; c < NV; c++) sx[(warp * NV + c) * R + lane] = Fh[0][c];
    }
    __syncthreads();
    if (!block_wait_or_report(p, bar, 1)) return;
    const int l = 2 * warp;
    if (row_ok && l < ncell) {
      const float i0 = inverse(l);
#pragma unroll
      for (int c = 0; c < NV; c++) in[(c * SEG + l) * R + lane] -= (Fh[1][c] - Fh[0][c]) * i0;
      if (l + 1 < ncell) {
        const float i1 = inverse(l + 1);
#pragma unroll
        for (int c = 0; c < NV; c++)
          in[(c * SEG + l + 1) * R + lane] -= (sx[((warp + 1) * NV + c) * R + lane] - Fh[1][c]) * i1;
      }
    }
  } else {
    float *sh = sfp;  // face fluxes [NV][R][FST]
#pragma unroll
    for (int ps = 0; ps < MAXP; ps++) {
      const int fi = warp + ps * NW;
      if (fi < nface) {
#pragma unroll
        for (int c = 0; c < NV; c++) sh[(c * R + lane) * FST + fi] = Fh[ps][c];
      }
    }
    __syncthreads();
    if (!block_wait_or_report(p, bar, 1)) return;
    if (row_ok) {
      for (int l = warp; l < ncell; l += NW) {
        const float inv_h = inverse(l);
#pragma unroll
        for (int c = 0; c < NV; c++) {
          const float *hh = sh + (c * R + lane) * FST;
          in[(c * SEG + l) * R + lane] -= (hh[l + 1] - hh[l]) * inv_h;
        }
      }
    }
  }
  tma::fence_async_shared();
  __syncthreads();
  if (threadIdx.x == 0) tma::store_4d(&tl, line0, yi, zi, 0, in);
}

// ------------------------------------------------------------------------------------------
// characteristic non-reflecting faces (Sec. 2, after Thompson) on the perturbations: the
// one-sided derivatives of rho', u', p' are those of rho, u, p; the wave speeds and the map
// back to the conservative variables use the full state
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float one_sided32(const float *phi, long long o, long long st, int s,
                                             float inv12) {
  const float f0 = phi[o];
  float acc = 48.f * (phi[o + s * st] - f0);
  acc = fmaf(-36.f, phi[o + 2 * s * st] - f0, acc);
  acc = fmaf(16.f, phi[o + 3 * s * st] - f0, acc);
  acc = fmaf(-3.f, phi[o + 4 * s * st] - f0, acc);
  return (float)s * acc * inv12;
}

// the normal convective term D of the cell I on the face (a, side)
template <int DIM>
__device__ __forceinline__ void char_term32(const Plan &p, const Free &fs, int a, int side,
                                            const int I[3], float D[DIM + 2]) {
  constexpr int NV = DIM + 2;
  const int s = side == 0 ? 1 : -1;
  const long long o = pad_index(p, I[0], I[1], I[2]);
  const long long st = a == 0 ? 1 : a == 1 ? (long long)p.P[0] : (long long)p.P[0] * p.P[1];
  const float inv12 = mesh::inv12_32(p, a, I[a]);
  const float r = fs.rho + p.Qp32[o], pr = fs.p + p.Wp32[DIM * p.NP + o];
  const float c = sqrtf(fs.gamma * pr / r);
  const float ua = fs.u[a] + p.Wp32[a * p.NP + o];
  const float rx = one_sided32(p.Qp32, o, st, s, inv12);
  const float px = one_sided32(p.Wp32 + DIM * p.NP, o, st, s, inv12);
  const float uxa = one_sided32(p.Wp32 + a * p.NP, o, st, s, inv12);
  const float lam1 = ua - c, lam2 = ua, lam5 = ua + c, rc = r * c;
  const float L1 = (lam1 * (float)s > 0.f) ? 0.f : lam1 * (px - rc * uxa);
  const float L2 = (lam2 * (float)s > 0.f) ? 0.f : lam2 * (c * c * rx - px);
  const float L5 = (lam5 * (float)s > 0.f) ? 0.f : lam5 * (px + rc * uxa);
  float dv[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    if (b == a) continue;
    float utx = one_sided32(p.Wp32 + b * p.NP, o, st, s, inv12);
    dv[b] = (lam2 * (float)s > 0.f) ? 0.f : lam2 * utx;
  }
  const float d1 = (L2 + 0.5f * (L5 + L1)) / (c * c);
  const float d2 = 0.5f * (L5 + L1);
  dv[a] = (L5 - L1) / (2.f * rc);
  float ke = 0.f, work = 0.f;
  D[0] = d1;
#pragma unroll
  for (int b = 0; b < DIM; b++) {
    float ub = fs.u[b] + p.Wp32[b * p.NP + o];
    D[1 + b] = ub * d1 + r * dv[b];
    ke += ub * ub;
    work += ub * dv[b];
  }
  D[NV - 1] = 0.5f * ke * d1 + d2 / fs.gm1 + r * work;
}

// All characteristic faces in one launch, one thread per cell: the cell of a corner or an edge
// belongs to the thread of its first face, which takes its faces' terms in order (direction by
// direction, low face first), as one launch per face did: 9.6 us each for a thousand cells, all of
// it latency; with one launch the 1021 x 771 wake's six steps went from 2543 to 2143 us.
template <int DIM>
__global__ void __launch_bounds__(128) k_char_faces32(Plan p) {
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
  const Free fs = free_stream(p);
  const long long oi = int_index(p, I[0], I[1], I[2]);
  float L[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) L[c] = p.L32[c * p.N + oi];
  for (int f = face; f < 2 * DIM; f++) {
    const int a = f / 2, side = f % 2;
    if (p.bc[a][side] != IBFSA_BC_CHARACTERISTIC || I[a] != (side == 0 ? 0 : p.n[a] - 1)) continue;
    float D[NV];
    char_term32<DIM>(p, fs, a, side, I, D);
#pragma unroll
    for (int c = 0; c < NV; c++) L[c] -= D[c];
  }
#pragma unroll
  for (int c = 0; c < NV; c++) p.L32[c * p.N + oi] = L[c];
}

// ------------------------------------------------------------------------------------------
// viscous term on the velocity perturbations
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float d4f(float fm2, float fm1, float fp1, float fp2, float inv_h12) {
  return (8.f * (fp1 - fm1) - (fp2 - fm2)) * inv_h12;
}

// ------------------------------------------------------------------------------------------
// immersed boundary in FP64 from the FP64 stage state
// ------------------------------------------------------------------------------------------
// FP64 value of component c of the stage state at interior cell o: Qn + increment
__device__ __forceinline__ double stage_q(const Plan &p, const double *__restrict__ Qn,
                                          const float *__restrict__ din, int c, long long o) {
  double v = Qn[c * p.N + o];
  return din ? v + (double)din[c * p.N + o] : v;
}

// Markers, a group of G lanes each (marker.cuh).  Interpolation (Eq. 8) and penalty force (Eq. 7) in
// FP64, and the spreading (Eq. 9) into the FP32 right-hand side: the kernel weights and the
// marker's force are FP64; the per-cell force, the fluid velocity of the power term f.u and the
// atomic additions are FP32, the precision of the right-hand side they enter.
template <int DIM, int G, int PART>
__global__ void __launch_bounds__(128) k_markers32(Plan p, const double *__restrict__ Qn,
                                                   const float *__restrict__ din,
                                                   const double *__restrict__ xis,
                                                   const double *xin, double *xio, double A,
                                                   double Bc, double dt, int advance) {
  begin_kernel();
  constexpr int C = marker::Support<DIM, G>::C;
  const int r = threadIdx.x % G, M = p.max_markers;
  const unsigned km = blockIdx.x * (blockDim.x / G) + threadIdx.x / G, nm = (unsigned)p.nm;
  const int k = (int)min(km, nm - 1);
  const auto t = marker::support<DIM, G>(p, p.X, M, k, r);
  const long long o = int_index(p, t.c0[0], t.c0[1], t.c0[2]);
  double F[DIM];
  if constexpr (PART & marker::INTERP) {
    double acc[DIM];
#pragma unroll
    for (int a = 0; a < DIM; a++) acc[a] = 0.0;
    if (t.ok) {
#pragma unroll
      for (int r0 = 0; r0 < C; r0++) {
        const double wi = t.w0[r0] * (1.0 / stage_q(p, Qn, din, 0, o + r0));
#pragma unroll
        for (int a = 0; a < DIM; a++)
          acc[a] = fma(stage_q(p, Qn, din, 1 + a, o + r0), wi, acc[a]);
      }
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
  if (km >= nm || !t.ok) return;  // the interpolation reports markers off the grid
  const double sc = p.dS[k] * t.ihp;
  float f[DIM];
#pragma unroll
  for (int a = 0; a < DIM; a++)
    f[a] = (float)(-(PART & marker::INTERP ? F[a] : p.F[a * M + k]) * sc);
  const Free fs = free_stream(p);
#pragma unroll
  for (int r0 = 0; r0 < C; r0++) {
    const float wt = (float)(t.w0[r0] * t.wr);
    const float d0 = p.qn32[o + r0] + (din ? din[o + r0] : 0.f);
    const float inv_rho = 1.f / (fs.rho + d0);
    float pw = 0.f;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const long long at = (1 + a) * p.N + o + r0;
      const float da = p.qn32[at] + (din ? din[at] : 0.f);
      const float fa = f[a] * wt;
      atomicAdd(&p.L32[at], fa);
      pw += fa * ((fs.m[a] + da) * inv_rho);
    }
    atomicAdd(&p.L32[(DIM + 1) * p.N + o + r0], pw);
  }
}

// ------------------------------------------------------------------------------------------
// finish: sponge on the FP32 right-hand side, then
//   mode 0: L out (FP64 copy);  mode 1: dout = b (din + dt L);
//   mode 2: Qn += b (din + dt L) in FP64 and qn32 = (float)(Qn - q_inf)
// ------------------------------------------------------------------------------------------
// periodic Gaussian pressure source (Sec. 3.6, Eq. 16) of cell (i, j, k): energy-equation term
template <bool STRETCHED = true>
__device__ __forceinline__ float pressure_source32(const Plan &p, int dim, int i, int j, int k) {
  const int I[3] = {i, j, k};
  float r2 = 0.f;
  for (int a = 0; a < dim; a++) {
    double x = STRETCHED ? mesh::node(p, a, I[a]) : p.lo[a] + ((double)I[a] + 0.5) * p.h[a];
    float dx = (float)(x - p.src_xc[a]);
    r2 += dx * dx;
  }
  return expf(-(float)(p.src_b * 0.693147180559945309417) * r2) * (float)p.src_scale;
}

// The end of a stage at one cell: sponge and pressure source on the right-hand side Lc of cell
// (i, j, k), offset t, stage increment Dc, then the right-hand side out (mode 0) or the RK update
template <int DIM, bool STRETCHED>
__device__ __forceinline__ void finish_cell(const Plan &p, float (&Lc)[DIM + 2],
                                            const float (&Dc)[DIM + 2], int i, int j, int k,
                                            long long t, float *__restrict__ dout, double *Qn,
                                            double *__restrict__ Lout, float Bc, float dt,
                                            int mode) {
  constexpr int NV = DIM + 2;
  if (p.sponge_cells > 0) {
    const int I[3] = {i, j, k};
    int S = p.sponge_cells, nmin = 1 << 30;
#pragma unroll
    for (int a = 0; a < DIM; a++) nmin = min(nmin, min(I[a], p.n[a] - 1 - I[a]));
    if (nmin < S) {
      float rr = (float)(S - nmin) / (float)S;
      float sig = (float)p.sponge_sigma * rr * rr * rr;
#pragma unroll
      for (int c = 0; c < NV; c++) Lc[c] -= sig * (p.qn32[c * p.N + t] + Dc[c]);
    }
  }
  if (p.src_on) Lc[NV - 1] += pressure_source32<STRETCHED>(p, DIM, i, j, k);
  if (mode == 0) {
#pragma unroll
    for (int c = 0; c < NV; c++) Lout[c * p.N + t] = widen(Lc[c]);
    return;
  }
  bool bad = false;
  float inc[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) {
    inc[c] = Bc * (Dc[c] + dt * Lc[c]);
    bad |= !isfinite(inc[c]);
  }
  if (mode == 1) {
#pragma unroll
    for (int c = 0; c < NV; c++) dout[c * p.N + t] = inc[c];
  } else {
    // The compiler has to take every store for one to Qn, so loads come one after the other unless
    // they stand before the first store: last stage at 2048^2 126 -> 104 us (152 with conversion
    // instructions).  In 3D, where the march has no registers for all five, two at a time: the pass
    // at 512^3, mean of the stages, 3.77 ms with conversion instructions, 3.55 without, 3.25 so
    // (4.8 with all five ahead).
    constexpr bool AHEAD = DIM == 2;
    double q[NV];
#pragma unroll
    for (int c = 0; c < NV; c++)
      if (AHEAD) q[c] = Qn[c * p.N + t];
#pragma unroll
    for (int c = 0; c < NV; c++) {
      if (!AHEAD && c % 2 == 0) {
        q[c] = Qn[c * p.N + t];
        if (c + 1 < NV) q[c + 1] = Qn[(c + 1) * p.N + t];
      }
      q[c] += widen(inc[c]);
      Qn[c * p.N + t] = q[c];
      p.qn32[c * p.N + t] = narrow(q[c] - p.qinf[c]);
    }
  }
  if (bad) atomicOr(p.status, IBFSA_STATUS_NONFINITE);
}

// inviscid: one thread per cell
template <int DIM>
__global__ void __launch_bounds__(THREADS) k_finish32(Plan p, const float *__restrict__ din,
                                                      float *__restrict__ dout, double *Qn,
                                                      double *__restrict__ Lout, float Bc,
                                                      float dt, int mode) {
  begin_kernel();
  constexpr int NV = DIM + 2;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;  // cells fit in 31 bits
  if (t >= (unsigned)p.N) return;
  float Lc[NV], Dc[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) {
    Lc[c] = p.L32[c * p.N + t];
    Dc[c] = din ? din[c * p.N + t] : 0.f;
  }
  const unsigned r = t / (unsigned)p.n[0], k = r / (unsigned)p.n[1];
  finish_cell<DIM, true>(p, Lc, Dc, (int)(t - r * p.n[0]), (int)(r - k * p.n[1]), (int)k, t, dout,
                         Qn, Lout, Bc, dt, mode);
}

// 2D viscous term + finish.  A block of 256 threads owns 64 x 16 cells: the velocity perturbations
// with a halo of four in shared memory, from them the viscous fluxes at the block's cells and at the
// two halo points per side that the divergence needs, in shared memory, then the divergence, sponge
// and RK update.  The right-hand side and the stage increment are loaded while the fluxes are
// evaluated.  Before, a kernel wrote the six flux arrays and the finish pass read them (48 B of
// 136 per cell and stage) and both found their cell by 64-bit divisions:
// together 132 -> 85 us per stage at 2048^2 and 244 -> 157 us at 4096 x 2048 (event times); 69 and
// 125 us with the update of finish_cell as it is now, of which the last stage takes half.
namespace v2 {
constexpr int TX = 64, TY = 16, PER = TX * TY / THREADS;  // cells of a block, per thread
constexpr int SX = TX + 8, SY = TY + 8;                   // staged points
constexpr int FX = TX + 4, FY = TY + 4;                   // points of F_v,x and F_v,y
constexpr size_t SMEM = sizeof(float) * (2 * SX * SY + 3 * FX * TY + 3 * TX * FY);
}  // namespace v2

template <bool STRETCHED>
__global__ void __launch_bounds__(THREADS, 4) k_visc_finish32(Plan p, const float *__restrict__ din,
                                                           float *__restrict__ dout, double *Qn,
                                                           double *__restrict__ Lout, float Bc,
                                                           float dt, int mode) {
  begin_kernel();
  using namespace v2;
  extern __shared__ float smm[];
  float *su = smm, *sv = su + SX * SY;            // [SY][SX]
  float *fx = sv + SX * SY, *fy = fx + 3 * FX * TY;  // [3][TY][FX], [3][FY][TX]
  const int tx = threadIdx.x % TX, tq = threadIdx.x / TX;
  constexpr int RS = THREADS / TX;                // rows tq, tq + RS, ...
  const int tiles_x = (p.n[0] + TX - 1) / TX;
  const int x0 = (int)(blockIdx.x % tiles_x) * TX, y0 = (int)(blockIdx.x / tiles_x) * TY;
  const int X = x0 + tx;
  const Free fs = free_stream(p);
  const float *W0 = p.Wp32, *W1 = p.Wp32 + p.NP;
#pragma unroll
  for (int e = threadIdx.x; e < SX * SY; e += THREADS) {
    const int sx = e % SX, sy = e / SX;
    const int gx = min(x0 - 4 + sx, p.n[0] + 3), gy = min(y0 - 4 + sy, p.n[1] + 3);
    const int o = (gy + p.g[1]) * p.P[0] + gx + p.g[0];
    su[e] = W0[o];
    sv[e] = W1[o];
  }
  float L[PER][4], D[PER][4];
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int Y = y0 + tq + k * RS;
    if (X < p.n[0] && Y < p.n[1]) {
      const int t = Y * p.n[0] + X;
#pragma unroll
      for (int c = 0; c < 4; c++) {
        L[k][c] = p.L32[c * p.N + t];
        D[k][c] = din ? din[c * p.N + t] : 0.f;
      }
    }
  }
  __syncthreads();
  // 1/(12 dx/dxi) of node i along a; indices of staged points beyond the box (their results are
  // never used) are clamped into it
  auto ihat = [&](int a, int i) -> float {
    if constexpr (STRETCHED)
      return p.minv12_32[a] ? p.minv12_32[a][mesh::clamp_node(p, a, i) + NG] : p.inv_h12_32[a];
    else
      return p.inv_h12_32[a];
  };
  // viscous fluxes at tile position (px, py), -2 .. TX+1 and -2 .. TY+1: [tau_0a, tau_1a, b_a]
  auto flux = [&](int px, int py, bool wx, bool wy) {
    const float ihx = ihat(0, x0 + px), ihy = ihat(1, y0 + py);
    const int e = (py + 4) * SX + px + 4;
    const float *m[2] = {su + e, sv + e};
    float g[2][2];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      g[i][0] = d4f(m[i][-2], m[i][-1], m[i][1], m[i][2], ihx);
      g[i][1] = d4f(m[i][-2 * SX], m[i][-SX], m[i][SX], m[i][2 * SX], ihy);
    }
    const float div = g[0][0] + g[1][1];
#pragma unroll
    for (int a = 0; a < 2; a++) {
      if (a == 0 ? !wx : !wy) continue;
      float *F = a == 0 ? fx + py * FX + px + 2 : fy + (py + 2) * TX + px;
      const int st = a == 0 ? FX * TY : TX * FY;
      float b = 0.f;
#pragma unroll
      for (int i = 0; i < 2; i++) {
        float tau = g[i][a] + g[a][i];
        if (i == a) tau -= (2.f / 3.f) * div;
        F[i * st] = tau;
        b += (fs.u[i] + m[i][0]) * tau;
      }
      F[2 * st] = b;
    }
  };
#pragma unroll
  for (int k = 0; k < PER; k++) flux(tx, tq + k * RS, true, true);
  flux(tx, tq < 2 ? tq - 2 : TY + tq - 2, false, true);  // y halo: four rows of TX points
  if (threadIdx.x < 4 * TY) {                               // x halo: four columns of TY points
    const int h = threadIdx.x % 4;
    flux(h < 2 ? h - 2 : TX + h - 2, threadIdx.x / 4, true, false);
  }
  __syncthreads();
  const float ihx = ihat(0, X);
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int py = tq + k * RS, Y = y0 + py;
    if (X >= p.n[0] || Y >= p.n[1]) continue;
    const float ihy = ihat(1, Y);
    float Lc[4], Dc[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      Lc[c] = L[k][c];
      Dc[c] = D[k][c];
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const float *Fx = fx + (c * TY + py) * FX + tx + 2, *Fy = fy + (c * FY + py + 2) * TX + tx;
      float sum = 0.f;
      sum += d4f(Fx[-2], Fx[-1], Fx[1], Fx[2], ihx);
      sum += d4f(Fy[-2 * TX], Fy[-TX], Fy[TX], Fy[2 * TX], ihy);
      Lc[c + 1] += sum * p.inv_Re32;
    }
    finish_cell<2, STRETCHED>(p, Lc, Dc, X, Y, 0, (long long)Y * p.n[0] + X, dout, Qn, Lout, Bc, dt,
                              mode);
  }
}

// 3D viscous term + finish, marching along z.  A 32 x 8 block of threads owns 32 x 8 columns
// and walks a z-chunk of zc planes (chosen by march_chunk): velocity perturbations of five planes
// (x, y halo 4) sit in a shared-memory ring, refilled from registers loaded one plane ahead; at each
// plane c the 9 gradients
// are evaluated at the block's cells and at the x/y halo points the x/y divergence needs,
// giving F_v,x and F_v,y (shared memory, divergence taken at once) and F_v,z, whose
// z-differences are accumulated per thread into the cells c-2 .. c+2 of its column; cell c-2
// is then complete: L += (1/Re) sum_a D4_a F_v,a, sponge, RK update.
#ifndef VM_MIN_BLOCKS
#define VM_MIN_BLOCKS 4
#endif
namespace vm {
constexpr int TX = 32, TY = 8;                 // block columns
constexpr int VT = TX * TY;                    // threads (one column each)
constexpr int SX = TX + 8, SY = TY + 8;        // staged plane (halo 4)
constexpr int PX = TX + 4, PY = TY + 4;        // flux points (halo 2)
constexpr size_t SMEM = sizeof(float) * (5 * 3 * SX * SY + 4 * PX * TY + 4 * TX * PY);
}  // namespace vm

// STRETCHED: some direction has a non-uniform mesh (per-point metrics); otherwise the uniform
// 1/(12 h) constants, with no per-point lookups
template <bool STRETCHED>
__global__ void __launch_bounds__(vm::VT, VM_MIN_BLOCKS) k_visc_march32(Plan p, const float *__restrict__ din,
                                                          float *__restrict__ dout, double *Qn,
                                                          double *__restrict__ Lout, float Bc,
                                                          float dt, int mode, int zc) {
  begin_kernel();
  using namespace vm;
  extern __shared__ float smm[];
  float *ring = smm;                              // [5][3][SY][SX]
  float *fx = smm + 5 * 3 * SX * SY;              // F_v,x at [TY][PX], 4 components
  float *fy = fx + 4 * PX * TY;                   // F_v,y at [PY][TX], 4 components
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, zs = blockIdx.z * zc;
  const int ze = min(zs + zc, p.n[2]);
  const int X = x0 + tx, Y = y0 + ty;
  const bool own = X < p.n[0] && Y < p.n[1];
  Free fs = free_stream(p);
  const float ih[3] = {p.inv_h12_32[0], p.inv_h12_32[1], p.inv_h12_32[2]};
  const int PLANE = 3 * SX * SY;

  // plane z (ghost range -4 .. n+3) is read into registers one iteration before it enters
  // ring slot z mod 5, so its global-memory latency hides behind the gradients of a plane.
  // Per thread, the staged points it loads and their padded offsets within a plane are fixed:
  // computed once.
  constexpr int PER = (SX * SY + VT - 1) / VT;
  const int PXY = p.P[0] * p.P[1];
  const float *W0 = p.Wp32, *W1 = p.Wp32 + p.NP, *W2 = p.Wp32 + 2 * p.NP;
  int foff[PER];
#pragma unroll
  for (int j = 0; j < PER; j++) {
    int e = threadIdx.x + j * VT;
    int sx = e % SX, sy = e / SX;
    int gx = min(x0 - 4 + sx, p.n[0] + 3), gy = min(y0 - 4 + sy, p.n[1] + 3);
    foff[j] = (gy + p.g[1]) * p.P[0] + (gx + p.g[0]);
  }
  float R[PER][3];
  auto fetch = [&](int z) {
    const int zo = (z + p.g[2]) * PXY;
#pragma unroll
    for (int j = 0; j < PER; j++) {
      if (threadIdx.x + j * VT < SX * SY) {
        const int o = zo + foff[j];
        R[j][0] = W0[o];
        R[j][1] = W1[o];
        R[j][2] = W2[o];
      }
    }
  };
  auto put = [&](int slot) {
    float *dst = ring + slot * PLANE + threadIdx.x;
#pragma unroll
    for (int j = 0; j < PER; j++) {
      if (threadIdx.x + j * VT < SX * SY) {
#pragma unroll
        for (int c = 0; c < 3; c++) dst[c * SX * SY + j * VT] = R[j][c];
      }
    }
  };
  // 1/(12 dx/dxi) of node i along a (the plan's 1/(12 h) on a uniform direction); indices of
  // staged points beyond the box (their results are never used) are clamped into it
  auto ihat = [&](int a, int i) -> float {
    if constexpr (STRETCHED)
      return p.minv12_32[a] ? p.minv12_32[a][mesh::clamp_node(p, a, i) + NG] : ih[a];
    else
      return ih[a];
  };
  // gradients g[i][j] = du_i/dx_j at staged position (sx, sy) = offset e of plane c (ihx, ihy,
  // ihz: the metrics there)
  auto grads = [&](const float *const pl[5], int e, float ihx, float ihy, float ihz,
                   float g[3][3], float u[3]) {
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const float *m = pl[2] + i * SX * SY + e;
      u[i] = m[0];
      g[i][0] = d4f(m[-2], m[-1], m[1], m[2], ihx);
      g[i][1] = d4f(m[-2 * SX], m[-SX], m[SX], m[2 * SX], ihy);
      g[i][2] = d4f(pl[0][i * SX * SY + e], pl[1][i * SX * SY + e], pl[3][i * SX * SY + e],
                    pl[4][i * SX * SY + e], ihz);
    }
  };
  // viscous flux of direction a: [tau_0a, tau_1a, tau_2a, b_a]
  auto vflux = [&](int a, const float g[3][3], const float u[3], float f[4]) {
    float div = g[0][0] + g[1][1] + g[2][2];
    float b = 0.f;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      float tau = g[i][a] + g[a][i];
      if (i == a) tau -= (2.f / 3.f) * div;
      f[i] = tau;
      b += (fs.u[i] + u[i]) * tau;
    }
    f[3] = b;
  };

  // divergence of the viscous flux of this column's cells c-2 .. c+2, accumulated as the
  // fluxes arrive: F_v,z of plane c enters the z-differences of cells c-2, c-1, c+1, c+2
  // (weights -1, 8, -8, 1 over 12 dx/dxi of that cell), the x/y divergence of plane c enters
  // cell c
  float acc[5][4];
#pragma unroll
  for (int o = 0; o < 5; o++)
#pragma unroll
    for (int k = 0; k < 4; k++) acc[o][k] = 0.f;
  const float ihx_own = ihat(0, X), ihy_own = ihat(1, Y);
  // the halo point this thread evaluates each plane (threads below 4 TY + 4 TX): F_v,x at x
  // offsets -2, -1, TX, TX+1 of a row, or F_v,y at y offsets -2, -1, TY, TY+1 of a column; its
  // staged offset, its metrics and where its flux goes, fixed for the whole march
  const int hkind = threadIdx.x < 4 * TY ? 1 : (threadIdx.x < 4 * TY + 4 * TX ? 2 : 0);
  int he = 0, hout = 0;
  float hihx = ih[0], hihy = ih[1];
  if (hkind == 1) {
    int r = threadIdx.x / 4, h = threadIdx.x % 4, px = h < 2 ? h : TX + h;  // 0,1,TX+2,TX+3
    he = (r + 4) * SX + px + 2;
    hout = r * PX + px;
    hihx = ihat(0, x0 - 4 + px + 2);
    hihy = ihat(1, y0 + r);
  } else if (hkind == 2) {
    int e2 = threadIdx.x - 4 * TY, col = e2 % TX, h = e2 / TX, py = h < 2 ? h : TY + h;
    he = (py + 2) * SX + col + 4;
    hout = py * TX + col;
    hihx = ihat(0, x0 + col);
    hihy = ihat(1, y0 - 4 + py + 2);
  }
  const int eown = (ty + 4) * SX + tx + 4;
  // inputs of the cell finished next (L, stage increment), loaded one plane ahead
  const int NXY = p.n[0] * p.n[1];
  const int town = Y * p.n[0] + X;  // interior offset within a plane (own columns)
  float Lnext[5], Dnext[5];
  auto fetch_cell = [&](int d) {
    if (own && d >= zs && d < ze) {
      const long long t = (long long)d * NXY + town;
#pragma unroll
      for (int cc = 0; cc < 5; cc++) {
        Lnext[cc] = p.L32[cc * p.N + t];
        Dnext[cc] = din ? din[cc * p.N + t] : 0.f;
      }
    }
  };

  // ring slot of plane z: (z + 8) mod 5, advanced incrementally
  int slot = (zs - 4 + 8) % 5;
  for (int z = zs - 4; z <= zs; z++) {
    fetch(z);
    put(slot);
    slot = slot == 4 ? 0 : slot + 1;
  }
  fetch(zs + 1);
  // slot now belongs to plane zs + 1; planes c - 2 .. c + 2 for c = zs - 2 start at slot of
  // plane zs - 4
  int s0 = (zs - 4 + 8) % 5;
  __syncthreads();
  for (int c = zs - 2; c < ze + 2; c++) {
    // ring slots of planes c-2 .. c+2, once per plane
    const float *pl[5];
#pragma unroll
    for (int o = 0; o < 5; o++) {
      int so = s0 + o;
      pl[o] = ring + (so >= 5 ? so - 5 : so) * PLANE;
    }
    // own cell: all three fluxes; halo points: F_v,x (x offsets -2,-1,32,33) or F_v,y
    const float ihz = ihat(2, c);
    {
      float g[3][3], u[3], f[4];
      grads(pl, eown, ihx_own, ihy_own, ihz, g, u);
      vflux(0, g, u, f);
#pragma unroll
      for (int k = 0; k < 4; k++) fx[(k * TY + ty) * PX + tx + 2] = f[k];
      vflux(1, g, u, f);
#pragma unroll
      for (int k = 0; k < 4; k++) fy[(k * PY + ty + 2) * TX + tx] = f[k];
      vflux(2, g, u, f);
      const float zm2 = ihat(2, c - 2), zm1 = 8.f * ihat(2, c - 1);
      const float zp1 = 8.f * ihat(2, c + 1), zp2 = ihat(2, c + 2);
#pragma unroll
      for (int k = 0; k < 4; k++) {
        acc[0][k] -= zm2 * f[k];
        acc[1][k] += zm1 * f[k];
        acc[3][k] -= zp1 * f[k];
        acc[4][k] += zp2 * f[k];
      }
    }
    static_assert(4 * TY + 4 * TX <= VT, "one halo point per thread at most");
    if (hkind) {
      float g[3][3], u[3], f[4];
      grads(pl, he, hihx, hihy, ihz, g, u);
      if (hkind == 1) {  // x-halo point
        vflux(0, g, u, f);
#pragma unroll
        for (int k = 0; k < 4; k++) fx[k * TY * PX + hout] = f[k];
      } else {           // y-halo point
        vflux(1, g, u, f);
#pragma unroll
        for (int k = 0; k < 4; k++) fy[k * PY * TX + hout] = f[k];
      }
    }
    __syncthreads();
    // x/y divergence at this column's cell of plane c
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const float *Fx = fx + (k * TY + ty) * PX + tx + 2;
      const float *Fy = fy + (k * PY + ty + 2) * TX + tx;
      acc[2][k] += d4f(Fx[-2], Fx[-1], Fx[1], Fx[2], ihx_own) +
                   d4f(Fy[-2 * TX], Fy[-TX], Fy[TX], Fy[2 * TX], ihy_own);
    }
    // plane d = c - 2 is complete: viscous term, sponge, RK update
    int d = c - 2;
    if (own && d >= zs && d < ze) {
      const long long t = (long long)d * NXY + town;
      float Lc[5];
#pragma unroll
      for (int cc = 0; cc < 5; cc++) Lc[cc] = Lnext[cc];
#pragma unroll
      for (int k = 0; k < 4; k++) Lc[k + 1] += acc[0][k] * p.inv_Re32;
      finish_cell<3, STRETCHED>(p, Lc, Dnext, X, Y, d, t, dout, Qn, Lout, Bc, dt, mode);
    }
    // plane c + 3 (needed from the next iteration on) replaces plane c - 2, whose gradients
    // were all taken before the barrier above; plane c + 4 starts loading
#pragma unroll
    for (int o = 0; o < 4; o++)
#pragma unroll
      for (int k = 0; k < 4; k++) acc[o][k] = acc[o + 1][k];
#pragma unroll
    for (int k = 0; k < 4; k++) acc[4][k] = 0.f;
    if (c + 1 < ze + 2) {
      put(s0);  // plane c + 3 takes the slot of plane c - 2
      if (c + 2 < ze + 2) fetch(c + 4);
      fetch_cell(c - 1);
    }
    s0 = s0 == 4 ? 0 : s0 + 1;
    __syncthreads();
  }
}

// the rounded state of a new FP64 state, bound by the FP64 pipe (hence narrow): once per state set,
// 512^3 and two steps 69.1 -> 68.4 ms, 4096 x 2048 and two coupled steps 2.86 -> 2.83
template <int DIM>
__global__ void __launch_bounds__(THREADS) k_refresh32(Plan p, const double *__restrict__ Q) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.N) return;
#pragma unroll
  for (int c = 0; c < DIM + 2; c++) p.qn32[c * p.N + t] = narrow(Q[c * p.N + t] - p.qinf[c]);
}

template <int DIM>
__global__ void k_probe64(Plan p, const double *__restrict__ Q, int np,
                          const double *__restrict__ xp, double *__restrict__ out) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= np) return;
  int j0[3];
  double w[3][4];
  if (!point_support<DIM>(p, xp, np, k, j0, w)) {
    atomicOr(p.status, IBFSA_STATUS_BOUNDS);
    out[k] = 0.0;
    return;
  }
  constexpr int C2 = DIM > 2 ? 4 : 1;
  double acc = 0.0;
  for (int r2 = 0; r2 < C2; r2++)
    for (int r1 = 0; r1 < 4; r1++)
      for (int r0 = 0; r0 < 4; r0++) {
        long long o = int_index(p, j0[0] + r0, j0[1] + r1, j0[2] + r2);
        double rho = Q[o], ke = 0.0;
        for (int a = 0; a < DIM; a++) {
          double m = Q[(1 + a) * p.N + o];
          ke += m * (m / rho);
        }
        double pr = p.gm1 * (Q[(DIM + 1) * p.N + o] - 0.5 * ke);
        acc += pr * (w[0][r0] * w[1][r1] * w[2][r2]);
      }
  out[k] = acc - p.p_inf;
}

// ------------------------------------------------------------------------------------------
inline unsigned blocks_for(long long n, int threads) {
  return (unsigned)((n + threads - 1) / threads);
}

// Tensor maps of the y/z tile copies: q' and the primitives over the padded box, L' over the
// interior, each as a rank-4 tensor (x, y, z, component) with boxes of 32 x-lines by the staged
// (or owned) cells along A.
template <int DIM, int A>
cudaError_t conv_tensor_maps(const Plan &p, CUtensorMap *tq, CUtensorMap *tw, CUtensorMap *tl) {
  using T = Tile<A>;
  const uint64_t P0 = p.P[0], P1 = p.P[1], P2 = p.P[2], n0 = p.n[0], n1 = p.n[1], n2 = p.n[2];
  const uint64_t ps[3] = {4 * P0, 4 * P0 * P1, 4 * (uint64_t)p.NP};
  const uint64_t is[3] = {4 * n0, 4 * n0 * n1, 4 * (uint64_t)p.N};
  const uint64_t dq[4] = {P0, P1, P2, (uint64_t)DIM + 2}, dw[4] = {P0, P1, P2, (uint64_t)DIM + 1};
  const uint64_t dl[4] = {n0, n1, n2, (uint64_t)DIM + 2};
  const uint32_t ly = A == 1 ? T::LEN : 1, lz = A == 2 ? T::LEN : 1;
  const uint32_t sy = A == 1 ? T::SEG : 1, sz = A == 2 ? T::SEG : 1;
  const uint32_t bq[4] = {T::ROWS, ly, lz, DIM + 2}, bw[4] = {T::ROWS, ly, lz, 1};
  const uint32_t bl[4] = {T::ROWS, sy, sz, DIM + 2};
  cudaError_t e;
  if ((e = tma::encode_f32_4d(tq, p.Qp32, dq, ps, bq)) != cudaSuccess) return e;
  if ((e = tma::encode_f32_4d(tw, p.Wp32, dw, ps, bw)) != cudaSuccess) return e;
  return tma::encode_f32_4d(tl, p.L32, dl, is, bl);
}

template <int DIM, int SCHEME, int LPR>
cudaError_t launch_conv_x(const Plan &p, int nseg, cudaStream_t st) {
  using T = RowTile<DIM, LPR>;
  int seg = (p.n[0] + nseg - 1) / nseg;  // equal segments, starting at even cells
  seg += seg & 1;
  const long long rows = (long long)p.n[1] * p.n[2];
  const long long blocks = (rows + T::ROWS - 1) / T::ROWS * nseg;
  static_assert(T::BYTES <= 48 * 1024, "within the default dynamic shared memory");
  launch(k_conv32_x<DIM, SCHEME, LPR>, (unsigned)blocks, THREADS, T::BYTES, st, p, seg, nseg);
  return cudaGetLastError();
}

template <int DIM, int A, int SCHEME>
cudaError_t launch_conv(const Plan &p, int first, cudaStream_t st) {
  using T = Tile<A>;
  cudaError_t e;
  if constexpr (SCHEME != IBFSA_MLP_TENO5) {
    if (p.charwise) {  // the characteristic-wise option: generic tiles for every direction
      constexpr size_t smem = conv_smem<DIM, A>();
      e = cudaFuncSetAttribute(k_conv32<DIM, A, SCHEME, true>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      dim3 grid;
      if (A == 0) {
        grid = dim3((p.n[0] + T::SEG - 1) / T::SEG, (p.n[1] + T::ROWS - 1) / T::ROWS, p.n[2]);
      } else {
        int nseg = (p.n[A] + T::SEG - 1) / T::SEG;
        grid = dim3(nseg * ((p.n[0] + T::ROWS - 1) / T::ROWS), A == 1 ? p.n[2] : p.n[1]);
      }
      launch(k_conv32<DIM, A, SCHEME, true>, grid, THREADS, smem, st, p, first);
      return cudaGetLastError();
    }
  }
  if constexpr (A == 0 && SCHEME != IBFSA_MLP_TENO5) {
    // rows of 64 cells per warp, or of 32 (two rows per warp) where that leaves fewer empty slots
    // (their halo of six cells costs ~5 % more)
    const int n = p.n[0], wide = (n + 63) / 64, narrow = (n + 31) / 32;
    return 64 * wide > 34 * narrow ? launch_conv_x<DIM, SCHEME, 16>(p, narrow, st)
                                   : launch_conv_x<DIM, SCHEME, 32>(p, wide, st);
  }
  if constexpr (A != 0) {
    if (p.n[0] % 4 == 0 && !first) {
      using TT = TmaTile<DIM, A>;
      constexpr size_t smem =
          TT::BYTES + (SCHEME == IBFSA_MLP_TENO5 ? (size_t)mlp::PACKED_BYTES : 0);
      e = cudaFuncSetAttribute(k_conv32_tma<DIM, A, SCHEME>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      CUtensorMap tq, tw, tl;
      if ((e = conv_tensor_maps<DIM, A>(p, &tq, &tw, &tl)) != cudaSuccess) return e;
      int nseg = (p.n[A] + T::SEG - 1) / T::SEG;
      int nx = (p.n[0] + T::ROWS - 1) / T::ROWS;
      dim3 grid(nseg * nx, A == 1 ? p.n[2] : p.n[1]);
      launch(k_conv32_tma<DIM, A, SCHEME>, grid, THREADS, smem, st, p, tq, tw, tl);
      return cudaGetLastError();
    }
  }
  if constexpr (A != 0 || SCHEME == IBFSA_MLP_TENO5) {
    constexpr size_t smem =
        conv_smem<DIM, A>() + (SCHEME == IBFSA_MLP_TENO5 ? (size_t)mlp::PACKED_BYTES : 0);
    e = cudaFuncSetAttribute(k_conv32<DIM, A, SCHEME>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid;
    if (A == 0) {
      grid = dim3((p.n[0] + T::SEG - 1) / T::SEG, (p.n[1] + T::ROWS - 1) / T::ROWS, p.n[2]);
    } else {
      int nseg = (p.n[A] + T::SEG - 1) / T::SEG;
      int nx = (p.n[0] + T::ROWS - 1) / T::ROWS;
      grid = dim3(nseg * nx, A == 1 ? p.n[2] : p.n[1]);
    }
    launch(k_conv32<DIM, A, SCHEME>, grid, THREADS, smem, st, p, first);
    return cudaGetLastError();
  }
}

// z-chunk of k_visc_march32.  A block's time is its planes (zc plus ~7 of start-up: the ring's
// first planes and the two flux planes on each side), whatever its neighbours on the SM do (the
// pass is bound by latency per plane), so the chunk that minimises (waves of 152 SMs x 4 blocks)
// x (zc + 7) is taken: long chunks where the columns alone fill the chip, short ones where they
// do not.  Against a fixed chunk of 64: 99 x 77 x 85 (80 blocks, now 600) 160 -> 45 us, 128^3
// 176 -> 86 us, 512^3 (chunk 128) 3.80 -> 3.76 ms (the whole pass since: 42, 79 us and
// 3.25 ms).
inline int march_chunk(const int n[3]) {
  const long long cols =
      (long long)((n[0] + vm::TX - 1) / vm::TX) * ((n[1] + vm::TY - 1) / vm::TY);
  const long long slots = 152 * VM_MIN_BLOCKS;
  int best = 128;
  long long cost = -1;
  for (int zc = 128; zc >= 4; zc--) {
    const long long blocks = cols * ((n[2] + zc - 1) / zc);
    const long long c = (blocks + slots - 1) / slots * (zc + 7);
    if (cost < 0 || c < cost) {
      cost = c;
      best = zc;
    }
  }
  return best;
}

template <int DIM, int SCHEME>
cudaError_t run_stage(const Plan &p, const StageArgs &s, cudaStream_t st) {
  cudaError_t e;
  Prof *pr = s.prof;
  e = cudaMemsetAsync(p.alpha_bits, 0, 3 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  // stage increments: none at the step start, d1 after stage 1, d2 after stage 2
  const float *din = s.stage == 1 ? p.d1 : s.stage == 2 ? p.d2 : nullptr;
  float *dout = s.stage == 0 ? p.d1 : s.stage == 1 ? p.d2 : nullptr;
  const double *Qn = s.Qn;
  prof_begin(pr, st);
  launch(k_pad32<DIM>, blocks_for(p.NP, THREADS), THREADS, 0, st, p, din);
  prof_end(pr, K_PAD, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  int advance = s.stage >= 0;
  auto markers = [&](auto part, int cls) -> cudaError_t {
    if (p.nm <= 0) return cudaSuccess;
    prof_begin(pr, st);
    marker::with_group<DIM>(p.nm, [&](auto g) {
      launch(k_markers32<DIM, g(), part()>, blocks_for((long long)p.nm * g(), 128), 128, 0, st, p,
             Qn, din, s.xis, s.xin, s.xio, s.a, s.b, s.dt, advance);
    });
    prof_end(pr, cls, st);
    return cudaGetLastError();
  };
  // interpolation and spreading in one launch after the convective term, unless someone waits for
  // the forces (the coupled step, which is 2D)
  using Interp = std::integral_constant<int, marker::INTERP>;
  using Spread = std::integral_constant<int, marker::SPREAD>;
  using Both = std::integral_constant<int, marker::BOTH>;
  if constexpr (DIM == 2) {
    if (s.forces && (e = markers(Interp(), K_INTERP)) != cudaSuccess) return e;
    if (s.forces && (e = cudaEventRecord(s.forces, st)) != cudaSuccess) return e;
  } else if (s.forces) {
    return cudaErrorNotSupported;
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
    launch(k_char_faces32<DIM>, blocks_for(cells, 128), 128, 0, st, p);
    prof_end(pr, K_CONV_X, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if constexpr (DIM == 2) e = s.forces ? markers(Spread(), K_SPREAD) : markers(Both(), K_SPREAD);
  else e = markers(Both(), K_SPREAD);
  if (e != cudaSuccess) return e;
  int mode = !advance ? 0 : (s.stage < 2 ? 1 : 2);
  Plan q = p;
  q.src_scale = s.src_scale;
  prof_begin(pr, st);
  if (p.Re > 0.0 && DIM == 3) {
    using namespace vm;
    const bool stretched = p.minv12_32[0] || p.minv12_32[1] || p.minv12_32[2];
    auto kern = stretched ? k_visc_march32<true> : k_visc_march32<false>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
    if (e != cudaSuccess) return e;
    const int zc = march_chunk(p.n);
    dim3 grid((p.n[0] + TX - 1) / TX, (p.n[1] + TY - 1) / TY, (p.n[2] + zc - 1) / zc);
    launch(kern, grid, VT, SMEM, st, q, din, dout, const_cast<double *>(Qn), s.Lout, (float)s.b,
           (float)s.dt, mode, zc);
  } else if (p.Re > 0.0) {
    using namespace v2;
    const bool stretched = p.minv12_32[0] || p.minv12_32[1];
    auto kern = stretched ? k_visc_finish32<true> : k_visc_finish32<false>;
    static_assert(SMEM <= 48 * 1024, "within the default dynamic shared memory");
    const unsigned tiles = (unsigned)((p.n[0] + TX - 1) / TX) * ((p.n[1] + TY - 1) / TY);
    launch(kern, tiles, THREADS, SMEM, st, q, din, dout, const_cast<double *>(Qn), s.Lout,
           (float)s.b, (float)s.dt, mode);
  } else {
    launch(k_finish32<DIM>, blocks_for(p.N, THREADS), THREADS, 0, st, q, din, dout,
           const_cast<double *>(Qn), s.Lout, (float)s.b, (float)s.dt, mode);
  }
  prof_end(pr, K_FINISH, st);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// training stencils of the learned weights from the current state
// ------------------------------------------------------------------------------------------
struct Coef9 {
  float c[9];  // face value of the 9-point upwind-biased reconstruction from cells i-4 .. i+4
};

__device__ __forceinline__ unsigned long long splitmix(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

template <int DIM>
__global__ void k_mlp_sample(Plan p, int n_max, unsigned long long seed, int attempts, Coef9 cf,
                             float *__restrict__ S, float *__restrict__ T, int *count) {
  constexpr int NV = DIM + 2;
  long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  Free fs = free_stream(p);
  for (int att = 0; att < attempts; att++) {
    unsigned long long r = splitmix(seed ^ splitmix((unsigned long long)tid * attempts + att));
    int A = (int)(r % DIM);
    int c = (int)((r >> 8) % NV);
    int sign = (int)((r >> 16) & 1);
    unsigned long long r2 = splitmix(r);
    int I[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
      unsigned span = a == A ? (unsigned)(p.n[a] - 1) : (unsigned)p.n[a];
      I[a] = a < DIM ? (int)((r2 >> (20 * a)) % (span ? span : 1u)) : 0;
    }
    if (p.n[A] < 2) continue;
    const float alpha = (float)__longlong_as_double((long long)p.alpha_bits[A]);
    float f[10];
#pragma unroll
    for (int o = 0; o < 10; o++) {
      int J[3] = {I[0], I[1], I[2]};
      J[A] += o - 4;
      long long sidx = ((long long)(J[2] + p.g[2]) * p.P[1] + (J[1] + p.g[1])) * p.P[0] + (J[0] + p.g[0]);
      float up = p.Wp32[A * p.NP + sidx];
      float pp = p.Wp32[DIM * p.NP + sidx];
      float ua = fs.u[A] + up;
      float q = p.Qp32[c * p.NP + sidx];
      float F;
      if (c == 0) F = p.Qp32[(1 + A) * p.NP + sidx];
      else if (c == NV - 1) F = (q + pp) * ua + fs.H * up;
      else {
        F = q * ua + fs.m[c - 1] * up;
        if (c - 1 == A) F += pp;
      }
      f[o] = 0.5f * (sign == 0 ? F + alpha * q : F - alpha * q);
    }
    float v[5];
    if (sign == 0) { v[0] = f[2]; v[1] = f[3]; v[2] = f[4]; v[3] = f[5]; v[4] = f[6]; }
    else { v[0] = f[7]; v[1] = f[6]; v[2] = f[5]; v[3] = f[4]; v[4] = f[3]; }
    Cands k = candidates(v[0], v[1], v[2], v[3], v[4]);
    float amp = 0.f;
#pragma unroll
    for (int j = 0; j < 5; j++) amp = fmaxf(amp, fabsf(v[j] - v[2]));
    if (teno_mask(k) != 7 || !(amp > p.mlp_floor)) continue;
    // upwind side of the face: cells i-4 .. i+4 for the right-going flux, the mirror image
    // (cells i+5 .. i-3) for the left-going one
    float tgt = 0.f;
#pragma unroll
    for (int o = 0; o < 9; o++) tgt += cf.c[o] * (sign == 0 ? f[o] : f[9 - o]);
    int idx = atomicAdd(count, 1);
    if (idx >= n_max) return;
#pragma unroll
    for (int j = 0; j < 5; j++) S[(size_t)idx * 5 + j] = v[j];
    T[idx] = tgt;
  }
}

}  // namespace fp32_ns

// coefficients c_o (o = -4..4) with sum_o c_o avg_o(h) = h(0) for polynomials h of degree <= 8,
// avg_o = mean over [o-1, o] (the cell left of the face is o = 0): the flux-reconstruction target
// of the ninth-order upwind-biased scheme
static void upwind9(float out[9]) {
  constexpr int K = 9;
  double M[K][K + 1];
  for (int pw = 0; pw < K; pw++) {
    for (int j = 0; j < K; j++) {
      double o = j - 4;
      M[pw][j] = (pow(o, pw + 1) - pow(o - 1.0, pw + 1)) / (pw + 1);
    }
    M[pw][K] = pw == 0 ? 1.0 : 0.0;
  }
  for (int col = 0; col < K; col++) {
    int piv = col;
    for (int r = col + 1; r < K; r++)
      if (fabs(M[r][col]) > fabs(M[piv][col])) piv = r;
    for (int k = 0; k <= K; k++) {
      double tmp = M[col][k];
      M[col][k] = M[piv][k];
      M[piv][k] = tmp;
    }
    for (int r = 0; r < K; r++) {
      if (r == col) continue;
      double fct = M[r][col] / M[col][col];
      for (int k = col; k <= K; k++) M[r][k] -= fct * M[col][k];
    }
  }
  for (int j = 0; j < K; j++) out[j] = (float)(M[j][K] / M[j][j]);
}

cudaError_t fp32_mlp_sample(const Plan &p, const double *Q, int n_max, unsigned long long seed,
                            int attempts, float *stencils, float *targets, int *count,
                            cudaStream_t st) {
  using namespace fp32_ns;
  cudaError_t e = fp32_wavespeed(p, Q, st);  // qn32, padded perturbation and split speeds
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(count, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  Coef9 cf;
  upwind9(cf.c);
  int threads = 256, blocks = 152 * 8;
  if (p.dim == 2)
    k_mlp_sample<2><<<blocks, threads, 0, st>>>(p, n_max, seed, attempts, cf, stencils, targets,
                                               count);
  else
    k_mlp_sample<3><<<blocks, threads, 0, st>>>(p, n_max, seed, attempts, cf, stencils, targets,
                                               count);
  return cudaGetLastError();
}

// Self-test of the bounded wait: one block announces bytes on its barrier and issues no copy,
// so the phase never completes; the block must give up after the poll limit, report
// IBFSA_STATUS_TIMEOUT through the same path as the convective kernels, and end (nothing is in
// flight when it exits).
__global__ void __launch_bounds__(fp32_ns::THREADS) k_wait_selftest(Plan p) {
  __shared__ __align__(8) uint64_t bar[1];
  if (threadIdx.x == 0) tma::mbar_init(bar, 1);
  __syncthreads();
  if (threadIdx.x == 0) tma::mbar_expect_tx(bar, 16);  // no copy will deliver these bytes
  if (!fp32_ns::block_wait_or_report(p, bar, 0)) return;
  if (threadIdx.x == 0) atomicOr(p.status, IBFSA_STATUS_NONFINITE);  // unreachable
}

cudaError_t wait_selftest(const Plan &p, cudaStream_t st) {
  k_wait_selftest<<<1, fp32_ns::THREADS, 0, st>>>(p);
  return cudaGetLastError();
}

// Force the fluid exerts on the body and the power it delivers, from the Lagrangian penalty
// forces of the last evaluated stage (Eq. 7): sum_k F_k dS_k and sum_k (F_k . U_k) dS_k, in
// FP64, summed by one block in a fixed order (reproducible).
__global__ void k_body_force(Plan p, const double *__restrict__ U, double *__restrict__ out) {
  __shared__ double red[4][256];
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const int M = p.max_markers;
  for (int k = threadIdx.x; k < p.nm; k += blockDim.x) {
    double pw = 0.0;
    for (int a = 0; a < p.dim; a++) {
      double fa = p.F[a * M + k] * p.dS[k];
      acc[a] += fa;
      pw += fa * U[a * M + k];
    }
    acc[3] += pw;
  }
  for (int c = 0; c < 4; c++) red[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o)
      for (int c = 0; c < 4; c++) red[c][threadIdx.x] += red[c][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x < 4) out[threadIdx.x] = red[threadIdx.x][0];
}

cudaError_t body_force(const Plan &p, const double *U, double *out, cudaStream_t st) {
  k_body_force<<<1, 256, 0, st>>>(p, U, out);
  return cudaGetLastError();
}

cudaError_t fp32_stage(const Plan &p, const StageArgs &s, cudaStream_t st) {
  using namespace fp32_ns;
  if (p.dim == 2) {
    if (p.scheme == IBFSA_MLP_TENO5) return run_stage<2, IBFSA_MLP_TENO5>(p, s, st);
    return p.scheme == IBFSA_TENO5 ? run_stage<2, IBFSA_TENO5>(p, s, st)
                                   : run_stage<2, IBFSA_WENO5JS>(p, s, st);
  }
  if (p.scheme == IBFSA_MLP_TENO5) return run_stage<3, IBFSA_MLP_TENO5>(p, s, st);
  return p.scheme == IBFSA_TENO5 ? run_stage<3, IBFSA_TENO5>(p, s, st)
                                 : run_stage<3, IBFSA_WENO5JS>(p, s, st);
}

cudaError_t fp32_refresh(const Plan &p, const double *Q, cudaStream_t st) {
  using namespace fp32_ns;
  if (p.dim == 2) k_refresh32<2><<<blocks_for(p.N, THREADS), THREADS, 0, st>>>(p, Q);
  else k_refresh32<3><<<blocks_for(p.N, THREADS), THREADS, 0, st>>>(p, Q);
  return cudaGetLastError();
}

cudaError_t fp32_wavespeed(const Plan &p, const double *Q, cudaStream_t st) {
  using namespace fp32_ns;
  cudaError_t e = fp32_refresh(p, Q, st);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(p.alpha_bits, 0, 3 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  if (p.dim == 2) launch(k_pad32<2>, blocks_for(p.NP, THREADS), THREADS, 0, st, p, nullptr);
  else launch(k_pad32<3>, blocks_for(p.NP, THREADS), THREADS, 0, st, p, nullptr);
  return cudaGetLastError();
}

cudaError_t fp32_probe(const Plan &p, const double *Q, int np, const double *xp, double *out,
                       cudaStream_t st, Prof *pr) {
  using namespace fp32_ns;
  prof_begin(pr, st);
  if (p.dim == 2) k_probe64<2><<<blocks_for(np, 128), 128, 0, st>>>(p, Q, np, xp, out);
  else k_probe64<3><<<blocks_for(np, 128), 128, 0, st>>>(p, Q, np, xp, out);
  prof_end(pr, K_PROBE, st);
  return cudaGetLastError();
}

}  // namespace ibfsa
