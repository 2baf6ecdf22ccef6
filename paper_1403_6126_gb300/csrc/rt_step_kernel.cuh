// What the step kernels share (Jiang, Stone & Davis 2014, arXiv:1403.6126, secs.
// 3-4): boundary mapping, alpha, face constants, the index checks of the debug
// build, and the tile geometry of the kernels that pass slopes and fluxes
// through shared memory (rt_step_quad.cuh, rt_step_pair.cuh).
#pragma once

#include <math.h>

#include "rt_internal.h"

namespace rtg {

namespace stepk {

constexpr int kHalo = 2;

// Index checking.  A debug build defines RT_BOUNDS_CHECK: every shared- and
// global-memory index of the float step's per-tile code then passes through
// RT_IDX(i, n), or RT_AT for pointers, or is one that did (a staged cell, the own
// cell), and an index outside [0, n) adds one to the step's failure
// count (the same word as a failed temperature solve, so rt_sync reports
// it) and is replaced by 0, which turns an out-of-bounds access into a
// reported error instead of a fault.  In the product build RT_IDX(i, n) is
// i and costs nothing.
__device__ __forceinline__ long long checked_index(long long i, long long n, int *status) {
  if (i >= 0 && i < n) return i;
  atomicAdd(status, 1);
  return 0;
}
// RT_AT(p, base, n): the same for a pointer that walks through the n elements at
// base; it is replaced by base.
template <class T>
__device__ __forceinline__ T *checked_pointer(T *p, T *base, long long n, int *status) {
  return base + checked_index(p - base, n, status);
}
#ifdef RT_BOUNDS_CHECK
#define RT_IDX(i, n) (::rtg::stepk::checked_index((i), (n), a.status))
#define RT_AT(p, base, n) (::rtg::stepk::checked_pointer((p), (base), (n), a.status))
#else
#define RT_IDX(i, n) (i)
#define RT_AT(p, base, n) (p)
#endif
constexpr double kPi = 3.14159265358979323846;

enum { BC_PERIODIC = 0, BC_VACUUM = 1, BC_COPY = 2, BC_INFLOW = 3 };

__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ float alpha_of(float dl, float st) {
  float s = 10.0f * dl * st;
  float tau = s * s;
  if (tau < 1e-12f) return 1.0f;
  return sqrtf(-expm1f(-tau) / tau);
}
__device__ __forceinline__ double alpha_of(double dl, double st) {
  double s = 10.0 * dl * st;
  double tau = s * s;
  if (tau < 1e-12) return 1.0;
  return sqrt(-expm1(-tau) / tau);
}

// Tile geometry shared by host and device.  A tile of T[0] x T[1] x T[2]
// cells (one thread each) is staged with a two-cell halo on every active
// axis; only the cross-shaped part of the padded box is read (the stencil
// moves along one axis at a time), so only the tile cells and the four
// halo layers of each axis are staged ("cross" cells).  Slopes are kept for
// the tile plus one extension layer per axis, face fluxes for the T[d]+1
// faces per axis.
struct Geo {
  int T[3] = {1, 1, 1}, B[3] = {1, 1, 1}, P[3] = {1, 1, 1};   // tile, padded box, cells per layer
  int ncell = 1, nbox = 1, ncross = 1, next = 0, nlow = 0;
  int RX = 1, RXF = 1;          // row lengths of the x slope / flux arrays
  int sl_off[4] = {0, 0, 0, 0}, fx_off[4] = {0, 0, 0, 0};  // slope / flux array offsets per axis
  bool quad = false;            // the layout of the quad kernel (16-byte entries)
  __host__ __device__ constexpr void init(int dim, int tx, int ty, int tz, bool q = false) {
    quad = q;
    T[0] = tx; T[1] = ty; T[2] = tz;
    ncell = tx * ty * tz;
    nbox = 1;
    ncross = ncell;
    next = 0;
    nlow = 0;
    // Threads are ordered x, then z, then y, so a warp holds 32/tx rows of
    // x at consecutive z.  Rows of the x arrays are padded to a length
    // congruent to tx mod 32, which puts those rows on disjoint banks.
    RX = tx >= 32 ? tx + 2 : tx + 32;
    RXF = tx >= 32 ? tx + 1 : tx + 32;
    // The quad kernel's 16-byte entries take eight lanes per shared-memory
    // wavefront.  Its x-halo, x-extension and lowest-x-face work items run
    // along y, so there the box row and the rows of the x arrays (y
    // innermost) have odd lengths: eight items consecutive in y then fall on
    // eight different bank groups.  Tile rows along x are conflict free
    // with any row length.
    if (quad) {
      RX = (tx + 2) | 1;
      RXF = (tx + 1) | 1;
    }
    sl_off[0] = fx_off[0] = 0;
    for (int d = 0; d < 3; ++d) {
      bool act = d < dim;
      B[d] = act ? T[d] + 2 * kHalo : 1;
      if (quad && d == 0 && dim >= 2) B[0] |= 1;
      nbox *= B[d];
      P[d] = ncell / T[d];
      ncross += act ? 2 * kHalo * P[d] : 0;
      next += act ? 2 * P[d] : 0;
      nlow += act ? P[d] : 0;
      sl_off[d + 1] = sl_off[d] + (act ? sl_size(d) : 0);
      fx_off[d + 1] = fx_off[d] + (act ? fx_size(d) : 0);
    }
  }
  // Slope of the cell at local (lx, ly, lz) along axis d, l_d in [-1, T_d].
  __host__ __device__ constexpr int sl_idx(int d, int lx, int ly, int lz) const {
    return d == 0 ? (lx + 1) + RX * (quad ? ly + T[1] * lz : lz + T[2] * ly)
           : d == 1 ? lx + T[0] * (lz + T[2] * (ly + 1))
                    : lx + T[0] * ((lz + 1) + (T[2] + 2) * ly);
  }
  __host__ __device__ constexpr int sl_size(int d) const {
    return d == 0 ? RX * T[2] * T[1] : d == 1 ? T[0] * T[2] * (T[1] + 2) : T[0] * (T[2] + 2) * T[1];
  }
  __host__ __device__ constexpr int sl_step(int d) const { return d == 0 ? 1 : d == 1 ? T[0] * T[2] : T[0]; }
  // Flux of face f along d (between local f-1 and f) in the row of (lx, ly, lz).
  __host__ __device__ constexpr int fx_idx(int d, int f, int lx, int ly, int lz) const {
    return d == 0   ? f + RXF * (quad ? ly + T[1] * lz : lz + T[2] * ly)
           : d == 1 ? lx + T[0] * (lz + T[2] * f)
                    : lx + T[0] * (f + (T[2] + 1) * ly);
  }
  __host__ __device__ constexpr int fx_size(int d) const {
    return d == 0 ? RXF * T[2] * T[1] : d == 1 ? T[0] * T[2] * (T[1] + 1) : T[0] * (T[2] + 1) * T[1];
  }
  __host__ __device__ constexpr int fx_step(int d) const { return d == 0 ? 1 : d == 1 ? T[0] * T[2] : T[0]; }
};

// The same geometry for a compile-time shape, as constants, for device
// code (runtime-indexed member arrays would put the struct in memory).
template <int DIM, int TX, int TY, int TZ, bool Q = false>
struct GeoT {
  __host__ __device__ static constexpr Geo g() {
    Geo x;
    x.init(DIM, TX, TY, TZ, Q);
    return x;
  }
  static constexpr int ncell = g().ncell, nbox = g().nbox, ncross = g().ncross, next = g().next, nlow = g().nlow;
  static constexpr int B0 = g().B[0], B1 = g().B[1];
  static constexpr int P0 = g().P[0], P1 = g().P[1], P2 = g().P[2];
  static constexpr int SL0 = g().sl_off[0], SL1 = g().sl_off[1], SL2 = g().sl_off[2], SL3 = g().sl_off[3];
  static constexpr int FX0 = g().fx_off[0], FX1 = g().fx_off[1], FX2 = g().fx_off[2], FX3 = g().fx_off[3];
  static constexpr int RX = g().RX, RXF = g().RXF;
  __host__ __device__ static constexpr int T(int d) { return d == 0 ? TX : d == 1 ? TY : TZ; }
  __host__ __device__ static constexpr int P(int d) { return d == 0 ? P0 : d == 1 ? P1 : P2; }
  __host__ __device__ static constexpr int bstride(int d) { return d == 0 ? 1 : d == 1 ? B0 : B0 * B1; }
  __host__ __device__ static constexpr int sl_off(int d) { return d == 0 ? SL0 : d == 1 ? SL1 : SL2; }
  __host__ __device__ static constexpr int fx_off(int d) { return d == 0 ? FX0 : d == 1 ? FX1 : FX2; }
  __host__ __device__ static constexpr int sl_idx(int d, int lx, int ly, int lz) {
    return d == 0 ? (lx + 1) + RX * (Q ? ly + TY * lz : lz + TZ * ly)
           : d == 1 ? lx + TX * (lz + TZ * (ly + 1))
                    : lx + TX * ((lz + 1) + (TZ + 2) * ly);
  }
  __host__ __device__ static constexpr int sl_step(int d) { return d == 0 ? 1 : d == 1 ? TX * TZ : TX; }
  __host__ __device__ static constexpr int fx_idx(int d, int f, int lx, int ly, int lz) {
    return d == 0   ? f + RXF * (Q ? ly + TY * lz : lz + TZ * ly)
           : d == 1 ? lx + TX * (lz + TZ * f)
                    : lx + TX * (f + (TZ + 1) * ly);
  }
  __host__ __device__ static constexpr int fx_step(int d) { return d == 0 ? 1 : d == 1 ? TX * TZ : TX; }
};

// What a tile of M angles took in shared memory when the double kernel kept every
// right-hand side there (20 table entries per angle, one value per cell and
// angle, the staging arrays).  The shapes a context of RT_FP64 may choose are
// still those this holds to 227 KB (rt_set_tile refuses the others).
__host__ __device__ inline size_t smem_bytes(int dim, int M, bool has_v, int tx, int ty, int tz, size_t rs) {
  Geo g;
  g.init(dim, tx, ty, tz);
  size_t q = has_v ? 2 : 1;
  size_t reals = 20 * (size_t)M + (size_t)M * g.ncell + q * g.nbox + q * g.sl_off[3] + g.fx_off[3];
  return reals * rs + 16;
}

// Maps coordinate g along an axis of n cells onto the grid: the periodic
// image, or the nearest cell for the other boundary kinds.
__device__ __forceinline__ int map_in(int g, int n, int kind_lo, int kind_hi) {
  if (g < 0) return kind_lo == BC_PERIODIC ? ((g % n) + n) % n : 0;
  if (g >= n) return kind_hi == BC_PERIODIC ? g % n : n - 1;
  return g;
}

// alpha, 1 - |v_face| dt/dx and the left-state weight of the face between
// cells gl and gu (grid coordinates, both inside the grid) along axis d.
template <typename Real, bool VEL>
__device__ __forceinline__ void face_consts(const StepArgs<Real> &a, int d, const int gl[3], const int gu[3], Real *al,
                                            Real *hv, Real *wl) {
  const long long N = a.N;
  const long long cl = gl[0] + (long long)a.n[0] * (gl[1] + (long long)a.n[1] * gl[2]);
  const long long cu = gu[0] + (long long)a.n[0] * (gu[1] + (long long)a.n[1] * gu[2]);
  *al = Real(0.5) * (alpha_of(a.dx[d], a.sa[RT_IDX(cl, N)] + a.ss[RT_IDX(cl, N)]) +
                     alpha_of(a.dx[d], a.sa[RT_IDX(cu, N)] + a.ss[RT_IDX(cu, N)]));
  const Real vf = VEL ? Real(0.5) * (a.v[d * N + RT_IDX(cl, N)] + a.v[d * N + RT_IDX(cu, N)]) : Real(0);
  *hv = Real(1) - (vf < Real(0) ? -vf : vf) * a.dtdx[d];
  *wl = vf > Real(0) ? Real(1) : (vf < Real(0) ? Real(0) : Real(0.5));
}

// Staged cross cells per thread of a tile shape.
__host__ __device__ constexpr int slots_for(int dim, int tx, int ty, int tz) {
  Geo g;
  g.init(dim, tx, ty, tz);
  return (g.ncross + g.ncell - 1) / g.ncell;
}

}  // namespace stepk

}  // namespace rtg
