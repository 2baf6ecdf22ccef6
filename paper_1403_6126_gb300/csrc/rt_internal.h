// Internal declarations shared by the host runtime and the device kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rtg {

constexpr int kMaxAngles = 256;
constexpr int kMomComps = 10;  // E, Fx, Fy, Fz, Pxx, Pyy, Pzz, Pxy, Pxz, Pyz

// Everything one fused step launch needs.  Real is the intensity and
// transport type (double for the FP64 path, float for the mixed path);
// temperature and the gas energy source are always double.
template <typename Real>
struct StepArgs {
  int dim;            // active axes
  int n[3];           // cells per axis (1 on inactive axes)
  int M;              // angles
  long long N;        // cells
  int bc[3][2];       // boundary kinds per axis / side
  Real C, invC, P;    // Crat, 1/Crat, Prat
  Real dt;            // time step
  Real dtdx[3];       // dt / dx_d
  Real dx[3];         // cell sizes
  double dt_d, kv_per_rho;  // dt and R/(gamma-1) in double
  int hold_T, estimate_v;
  int newton_max_it;  // Newton on T: iteration cap and stopping tolerance
  double newton_rtol;
  Real wnorm;         // 1 - 1 / (sum of the weights as the float table holds them)
  float msum[10][2];  // the float table's normalised quadrature sums (table_moment_sums)
  const Real *ang;    // [M][4]: n_x, n_y, n_z, W
  const Real *inflow; // [3][2][M]
  int sym;            // float quad layout: angles stored as opposite pairs (pair_order)
  // Intensities.  Double: angle-major [M][N].  Float: quad-interleaved,
  // ceil(M/4) planes of float4 ([q][c] holds angles 4q .. 4q+3 of cell c,
  // angles past M zero).
  const Real *I_in;
  Real *I_out;
  const Real *rho, *sa, *ss;  // [N]
  // alpha of each cell for the cell side of each axis [N] (one array where the
  // sides are equal), for the double kernel and the 3-D pair kernel of a context;
  // the others form it from sa and ss.
  const Real *alpha[3];
  const Real *v;      // [3][N]
  const double *T_in; // [N]
  double *T_out;      // [N]
  const double *mom_in;  // [10][N] moments of I_in
  double *mom_out;       // [10][N] moments of I_out
  // Float quad layout: each cell's smallest intensity over its angles, of
  // I_in (read) and of I_out (written); null: formed from I_in in the kernel
  // and not written.
  const float *cen_in;
  float *cen_out;
  double *dEgas;      // [N]
  double *dMom;       // [3][N]
  int *status;        // [0]: cells whose T Newton failed
  // bf16 storage (RT_BF16, float kernels only): the stored value of angle m
  // in cell c (angle-major [M][N]) is delta = I / J - 1 with J = E / (4 pi)
  // of the cell's stored moments; I_in / I_out are unused then and Q is a
  // float [M][N] scratch for the right-hand sides Q_m.  Null otherwise.
  const unsigned short *I16_in;
  unsigned short *I16_out;
  float *Q;
  // The launch covers tile layers [outer_begin, outer_begin + outer_count)
  // along the outermost active axis (z in 3-D, y in 2-D, x in 1-D;
  // outer_count = 0: every layer).  Tiles are independent within a step, so
  // a grid stepped in slabs gives bitwise the whole-grid result.
  int outer_begin, outer_count;
};

// The float kernels take their angle sums over the weights of the float
// table ang4 ([M][4], W in slot 3) divided by their sum S (1 + O(1e-8) after
// rounding each weight), so that the weights they use sum to exactly 1.
// weight_norm returns 1 - 1/S, S summed in double (exact for comparable
// weights) and the result rounded to float once.
inline double weight_sum(const float *ang4, int M) {
  double s = 0.0;
  for (int m = 0; m < M; ++m) s += (double)ang4[4 * m + 3];
  return s;
}
inline float weight_norm(const float *ang4, int M) { return (float)(1.0 - 1.0 / weight_sum(ang4, M)); }

// The quadrature sums of a float angle table ang4 ([M][4]: n_x, n_y, n_z,
// W) that the float kernels' moments are taken against, over the normalised
// weights W / S (see weight_norm): sum W (1), sum W n_i (x, y, z), sum W n_i
// n_j (xx, yy, zz, xy, xz, yz), each summed in double and split into a float
// pair (hi, lo).
inline void table_moment_sums(const float *ang4, int M, float out[10][2]) {
  double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int m = 0; m < M; ++m) {
    const double x = ang4[4 * m], y = ang4[4 * m + 1], z = ang4[4 * m + 2], W = ang4[4 * m + 3];
    s[0] += W;
    s[1] += W * x; s[2] += W * y; s[3] += W * z;
    s[4] += W * x * x; s[5] += W * y * y; s[6] += W * z * z;
    s[7] += W * x * y; s[8] += W * x * z; s[9] += W * y * z;
  }
  for (int k = 0; k < 10; ++k) {
    const double v = s[k] / s[0];
    out[k][0] = (float)v;
    out[k][1] = (float)(v - (double)out[k][0]);
  }
}

// Where alpha of each cell goes: one array per distinct cell side, null for
// the others.
template <typename Real>
struct CellAlpha {
  Real *out[3];
  Real dx[3];
};

struct TileShape {
  int tx, ty, tz;
};

// Launch the fused step; returns the CUDA error of the launch.
template <typename Real>
cudaError_t launch_step(const StepArgs<Real> &a, int dim, bool has_v, TileShape tile, cudaStream_t s);

// The default tile of an n[0] x n[1] x n[2] grid on sms SMs: the first compiled
// shape that fits shared memory for (dim, M, has_v), or in 1-D and 2-D the
// smallest further one (down to 64 cells; 128 in 2-D float, 32 in 1-D double) that
// still has no more tiles than there are SMs.  Such a grid runs as one CTA per SM, so a
// step lasts as long as one tile and the smaller tile is the shorter one;
// past one CTA per SM its larger halo costs more than it spreads
// (us per step with the first shape and with the chosen one: float 1-D 512 x 8
// angles 12.6 and 8.8, 4096 x 48 24.9 and 16.7, 2-D 64 x 48 x 24 16.0 and 14.3,
// 128^2 x 24 16.3 and 14.6; double 512 x 8 38 and 16.5, 128^2 x 24 126 and 115;
// the other way, 256 x 128 x 80 in double, 16 x 16 377, 16 x 8 600).  3-D
// keeps its first shape, the fastest from 24^3 up.  False if no shape fits.
template <typename Real>
bool choose_tile(int dim, int M, bool has_v, const int *n, int sms, TileShape *out);

// Whether a tile shape can be launched: thread count within the kernel's
// launch bound, shared memory within the opt-in limit, and enough staging
// slots for its halo.
template <typename Real>
bool tile_ok(int dim, int M, bool has_v, TileShape t);

// The compiled shapes that can run (dim, M, has_v), preferred first; out
// holds up to 8.  Returns their count.
template <typename Real>
int tile_candidates(int dim, int M, bool has_v, TileShape *out);

// The bf16-storage step (RT_BF16): one compiled tile per dimension (16x8x4,
// 32x16, 512); choose_tile_b16 gives it, or false when its shared memory
// does not fit M angles.
cudaError_t launch_b16(const StepArgs<float> &a, int dim, bool vel, TileShape t, cudaStream_t s);
bool choose_tile_b16(int dim, int M, TileShape *out);

// The float step on the quad-interleaved layout (RT_FP32).  host_ang [M][4]
// and host_inflow [6][M] are the float tables the device holds: for M <= 80
// they travel as a launch-parameter table, larger sets read the device
// tables a.ang / a.inflow into shared memory.
cudaError_t launch_step_quad(const StepArgs<float> &a, const float *host_ang, const float *host_inflow, int dim,
                             bool vel, TileShape t, cudaStream_t s);

// Opposite pairs (rt_step_sym.cuh): whether the angles of a float table ang4
// ([M][4]: n_x, n_y, n_z, W) are pairs (n, -n) of one weight, exactly as the
// floats stand (those of every level-symmetric set are), whole quads of them
// and at most 80 angles.  Then order[i] is the index of the angle stored i-th.
bool pair_order(const float *ang4, int M, int *order);

// The float step on opposite pairs: host_ang, host_inflow and the intensities
// in stored order.
cudaError_t launch_step_sym(const StepArgs<float> &a, const float *host_ang, const float *host_inflow, int dim,
                            bool vel, TileShape t, cudaStream_t s);

// Where each of the caller's angles is stored (identity unless the set is
// stored as opposite pairs).
struct AngleMap {
  unsigned char slot[kMaxAngles];
};

// Elementwise helpers (all stream-ordered).
template <typename Real>
cudaError_t launch_convert_in(const double *src, Real *dst, long long n, cudaStream_t s);
// Isotropic equilibrium T^4/(4 pi): angle-major [M][N] (double), or the
// quad-interleaved float layout with zero padding (quad = true).
template <typename Real>
cudaError_t launch_isotropic(const double *T, Real *I, int M, long long N, bool quad, cudaStream_t s);
// E, F, P (double [10][N]) of an intensity field (angle-major, or the quad
// layout when quad is set), times wscale (float intensities only).
template <typename Real>
cudaError_t launch_moments(const Real *I, const Real *ang, int M, long long N, bool quad, double wscale, double *mom,
                           cudaStream_t s);
// Each cell's smallest intensity over its M angles (quad layout) into cen [N].
cudaError_t launch_centers(const float *I, int M, long long N, float *cen, cudaStream_t s);
// Eddington tensor f = P / E (6 components, [6][N]) from stored moments
// [10][N]; 0 where E = 0.
cudaError_t launch_eddington(const double *mom, double *f, long long N, cudaStream_t s);
// Elements [off, off + n) of an angle-major double field (element i is angle
// i / N of cell i % N) into / out of the quad-interleaved float layout.
cudaError_t launch_quad_in(const double *src, float *dst, long long off, long long n, long long N, const AngleMap &map,
                           cudaStream_t s);
cudaError_t launch_quad_out(const float *src, double *dst, long long off, long long n, long long N, const AngleMap &map,
                            cudaStream_t s);
// Up to three arrays of doubles (n = 0: none) in one launch.
struct FieldsOut {
  const double *src[3];
  double *dst[3];
  long long n[3];
};
cudaError_t launch_fields_out(const FieldsOut &f, cudaStream_t s);
// Every angle of the quad layout to the caller's [M][N] doubles (order.slot: the
// caller's index of each stored angle).
cudaError_t launch_intensity_out(const float *src, double *dst, int M, long long N, const AngleMap &order,
                                 cudaStream_t s);
// Quad-layout intensities in another order of their angles (a multiple of four, at
// most 80): angle m of dst is angle from.slot[m] of src.
cudaError_t launch_reorder(const float *src, float *dst, int M, long long N, const AngleMap &from, cudaStream_t s);

// bf16 storage: encode a float intensity array [M][N] as deviations from
// the mean intensity of each cell (E [N] its energy density), and decode
// elements [off, off + n) of a stored array to doubles.
cudaError_t launch_encode_b16(const float *I, const double *E, unsigned short *out, int M, long long N, cudaStream_t s);
cudaError_t launch_decode_b16(const unsigned short *in, const double *E, double *out, long long off, long long n,
                              long long N, cudaStream_t s);

// Scans n doubles: ORs bit 0 into *flag for a non-finite value or one below
// `lo` (or equal to it when strict), and ORs `nzbit` for a nonzero value.
cudaError_t launch_check(const double *x, long long n, double lo, int strict, int nzbit, int *flag, cudaStream_t s);
// The gas fields in doubles on the device: rho, T, sigma_a, sigma_s [N], v [3][N].
struct FieldSrc {
  const double *rho, *T, *v, *sa, *ss;
};
// Scan of the gas fields over cells [c0, c0 + n) into *flag (bit 0: a
// value out of range, bit 1: some v != 0); with convert also the copy into
// the context's arrays (rho, sigma_a, sigma_s, v in Real; T in double) and
// alpha of those cells.
template <typename Real>
cudaError_t launch_fields_in(const FieldSrc &src, long long N, long long c0, long long n, bool convert, Real *rho,
                             Real *sa, Real *ss, Real *v, double *T, const CellAlpha<Real> &al, int *flag,
                             cudaStream_t s);
// Scan of all N cells and a copy of them in stage (rho, T, v, sigma_a, sigma_s), in
// one pass over the caller's device arrays.
cudaError_t launch_fields_stage(const FieldSrc &src, long long N, double *stage, int *flag, cudaStream_t s);
// alpha of N cells from their opacities.
template <typename Real>
cudaError_t launch_alpha(const Real *sa, const Real *ss, long long N, const CellAlpha<Real> &al, cudaStream_t s);

}  // namespace rtg
