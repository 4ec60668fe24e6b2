// marker.cuh -- the four-point support of a Lagrangian marker (Eq. 10-11) shared by a group of
// lanes, for the immersed-boundary kernels whose sums need no fixed order (FP32 form, fast FP64).
//
// A group of 16 lanes owns one marker, lane r in 3D the row of four support cells along x at (y, z)
// offsets (r & 3, r >> 2), in 2D the cell (r & 3, r >> 2); many 2D markers take 4 lanes each, lane r
// the row at y offset r.  What bounds these kernels is the FP64 pipe (1.7 lanes per clock and
// SM): a warp instruction costs ~75 cycles whatever its active lanes, so the 4 DIM kernel weights
// are evaluated one per lane and exchanged, each row is summed by its lane, and only the rows' sums
// are reduced by shuffles.  Few lanes per marker are fewer instructions in all, many a shorter chain:
// 16 lanes in 2D while every quarter of an SM gets at most two warps.
// Interpolation and spreading together (event times, ~4 us a launch), against one thread per marker
// for the interpolation (a chain of 64 divisions in 3D) and, in FP64, the weights of a marker
// evaluated by each of its 64 threads for the spreading: FP32 form, 20000 markers in 3D 196 -> 98 us,
// 1500 82 -> 18; FP64, 5000 in 3D 212 -> 28; 2D, 1024 (FP32) 36 -> 12.
#pragma once

#include "ibfsa_internal.h"
#include "mesh.cuh"

#include <type_traits>

namespace ibfsa {
namespace marker {

// Peskin's four-point kernel, Eq. 11: one root per lane of a group
__device__ __forceinline__ double peskin4(double r) {
  const double a = fabs(r);
  if (a >= 2.0) return 0.0;
  const bool in = a < 1.0;
  const double rad = in ? 1.0 + 4.0 * a - 4.0 * a * a : -7.0 + 12.0 * a - 4.0 * a * a;
  return ((in ? 3.0 : 5.0) - 2.0 * a - (in ? -1.0 : 1.0) * sqrt(rad)) * 0.125;
}

// the same values with a branch, for threads that evaluate several weights (two roots in one thread's
// chain: 500 probes 32.8 us, 34.9 with peskin4)
__device__ __forceinline__ double peskin(double r) {
  const double a = fabs(r);
  if (a < 1.0) return (3.0 - 2.0 * a + sqrt(1.0 + 4.0 * a - 4.0 * a * a)) * 0.125;
  if (a < 2.0) return (5.0 - 2.0 * a - sqrt(-7.0 + 12.0 * a - 4.0 * a * a)) * 0.125;
  return 0.0;
}

// first support node and position in node units of coordinate x along a; the local spacing
__device__ __forceinline__ int first_node(const Plan &p, int a, double x, double *s, double *hl) {
  if (p.mx[a]) {
    *s = 0.0;
    *hl = 1.0;
    return mesh::support_stretched(p, a, x, s, hl);
  }
  *s = (x - p.lo[a]) * p.inv_h[a] - 0.5;
  *hl = p.h[a];
  return (int)floor(*s) - 1;
}

// G: lanes per marker
template <int DIM, int G>
struct Support {
  static constexpr int C = (DIM > 2 ? 64 : 16) / G;  // support cells per lane: 4 along x, or 1
  int j0[3];      // first support cell per direction
  int c0[3];      // this lane's first cell
  double w0[C];   // weights along x of this lane's cells
  double wr;      // product of this lane's weights along y (and z)
  double ihp;     // 1 / product of the local spacings (h^d of the delta)
  bool ok;        // the support lies inside the grid (where the spacing is constant)
};

// The support of marker k of X [DIM][stride]; r: lane within the group of G.  Every lane of the
// warp calls it (a group without a marker passes a valid k and discards the result).
template <int DIM, int G>
__device__ __forceinline__ Support<DIM, G> support(const Plan &p, const double *X, int stride,
                                                   int k, int r) {
  static_assert(DIM > 2 ? G == 16 : (G == 4 || G == 16), "");
  constexpr unsigned ALL = 0xffffffffu;
  Support<DIM, G> t;
  double s, hl;
  if constexpr (DIM > 2) {
    const int a = r < 12 ? r >> 2 : 2;  // lane 4a + q evaluates weight q along a
    const int j = first_node(p, a, X[a * stride + k], &s, &hl);
    const double w = peskin4(s - (double)(j + (r & 3)));
    const int bad = j < 0 || j > p.n[a] - 4;
#pragma unroll
    for (int b = 0; b < 3; b++) t.j0[b] = __shfl_sync(ALL, j, 4 * b, G);
#pragma unroll
    for (int q = 0; q < 4; q++) t.w0[q] = __shfl_sync(ALL, w, q, G);
    t.wr = __shfl_sync(ALL, w, 4 + (r & 3), G) * __shfl_sync(ALL, w, 8 + (r >> 2), G);
    t.ok = !(__shfl_sync(ALL, bad, 0, G) | __shfl_sync(ALL, bad, 4, G) |
             __shfl_sync(ALL, bad, 8, G));
    t.ihp = p.inv_h[0] * p.inv_h[1] * p.inv_h[2];
    if (p.mx[0] || p.mx[1] || p.mx[2]) {  // uniform over the grid
      t.ihp = 1.0 / (__shfl_sync(ALL, hl, 0, G) * __shfl_sync(ALL, hl, 4, G) *
                     __shfl_sync(ALL, hl, 8, G));
    }
  } else if constexpr (G == 16) {
    const int a = (r >> 2) & 1;  // lane 4a + q evaluates weight q along a
    const int j = first_node(p, a, X[a * stride + k], &s, &hl);
    const double w = peskin4(s - (double)(j + (r & 3)));
    const int bad = j < 0 || j > p.n[a] - 4;
    t.j0[0] = __shfl_sync(ALL, j, 0, G);
    t.j0[1] = __shfl_sync(ALL, j, 4, G);
    t.j0[2] = 0;
    t.w0[0] = __shfl_sync(ALL, w, r & 3, G);
    t.wr = __shfl_sync(ALL, w, 4 + (r >> 2), G);
    t.ok = !(__shfl_sync(ALL, bad, 0, G) | __shfl_sync(ALL, bad, 4, G));
    t.ihp = p.inv_h[0] * p.inv_h[1];
    if (p.mx[0] || p.mx[1])
      t.ihp = 1.0 / (__shfl_sync(ALL, hl, 0, G) * __shfl_sync(ALL, hl, 4, G));
  } else {
    double s1, h1;
    const int j = first_node(p, 0, X[k], &s, &hl), i = first_node(p, 1, X[stride + k], &s1, &h1);
    const double w = peskin4(s - (double)(j + r));
    t.wr = peskin4(s1 - (double)(i + r));
#pragma unroll
    for (int q = 0; q < 4; q++) t.w0[q] = __shfl_sync(ALL, w, q, G);
    t.j0[0] = j;
    t.j0[1] = i;
    t.j0[2] = 0;
    t.ok = !(j < 0 || j > p.n[0] - 4 || i < 0 || i > p.n[1] - 4);
    t.ihp = p.mx[0] || p.mx[1] ? 1.0 / (hl * h1) : p.inv_h[0] * p.inv_h[1];
  }
  constexpr bool CELL = Support<DIM, G>::C == 1;
  t.c0[0] = t.j0[0] + (CELL ? r & 3 : 0);
  t.c0[1] = t.j0[1] + (CELL ? r >> 2 : r & 3);
  t.c0[2] = t.j0[2] + (DIM > 2 ? r >> 2 : 0);
  return t;
}

// sum over the group's lanes (every lane gets it)
template <int G>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Penalty force and the RK update of the integral (Eq. 7) of marker k from its interpolated
// velocity: lane a of the group handles component a and returns the force's component.
template <int DIM>
__device__ __forceinline__ double force(const Plan &p, int k, int r, const double (&u)[DIM],
                                        const double *xis, const double *xin, double *xio, double A,
                                        double Bc, double dt, int advance) {
  if (r >= DIM) return 0.0;
  const int at = r * p.max_markers + k;
  const double slip = (r == 0 ? u[0] : r == 1 ? u[1] : u[DIM - 1]) - p.U[at];
  const double xi = xis[at];
  const double F = p.alpha_pen * xi + p.beta_pen * slip;
  p.F[at] = F;
  if (advance) xio[at] = A * xin[at] + Bc * (xi + dt * slip);
  return F;
}

// a marker whose support leaves the grid: no force, its integral kept, the status raised
template <int DIM>
__device__ __forceinline__ void off_grid(const Plan &p, int k, int r, const double *xin,
                                         double *xio, int advance) {
  if (r == 0) atomicOr(p.status, IBFSA_STATUS_BOUNDS);
  if (r >= DIM) return;
  const int at = r * p.max_markers + k;
  p.F[at] = 0.0;
  if (advance) xio[at] = xin[at];
}

// What a launch of the marker kernels does: spreading right after the interpolation, in the same
// lanes, wherever nothing needs the forces sooner -- a marker's spreading takes its own force only,
// and evaluating the support again and launching again cost about as much as the spreading itself.
// Event times, two launches / one: FP32 2D, 1024 markers (with 16 lanes each) 25 / 12 us; 3D, 1500
// markers 27 / 18, 20000 markers 134 / 97 us; FP64, 2D 400 markers 17 / 8 us, 3D 5000 40 / 27 us.
enum Part { INTERP = 1, SPREAD = 2, BOTH = 3 };

// calls f(G) with the lanes per marker for nm markers, an integral_constant
template <int DIM, typename F>
inline void with_group(int nm, F f) {
  if constexpr (DIM == 2) {
    // with 16 lanes (two markers a warp) more than two warps for each quarter of an SM
    if (nm > 2 * 4 * 152 * 2) return f(std::integral_constant<int, 4>());
  }
  f(std::integral_constant<int, 16>());
}

}  // namespace marker
}  // namespace ibfsa
