// Fused radiation-transfer step with double intensities (Jiang, Stone & Davis
// 2014, arXiv:1403.6126, secs. 3-4), angle-major storage.
//
// One CTA owns a tile of cells (one thread per cell in the implicit steps).
// The transport walks lines of up to eight cells, one angle at a time, with
// the van Leer differences, slopes and the last flux in registers (the line
// geometry of rt_step_sym.cuh): several angles' lines per round of two CTA
// barriers, so that a small tile gives every thread a line.  After a round
// each cell's thread forms the right-hand sides Q_m (kept in the output
// array) and every angle sum of the implicit steps; then it solves its cell:
// the T^4 energy equation of Step 4 (sec. 4.3) reduced to a scalar quartic, the
// 2x2 system of Step 5 (sec. 4.4), then I^{n+1}, the moments E_r, F_r, P_r
// (sec. 3) and the gas sources.
//
// What bounds it: the FP64 pipe (about two multiply-adds per cycle and SM) on
// grids that fill the GPU, and the latency of its chains on small ones.  So
// double operations are counted: one difference per cell and axis (a line
// shares it between two slopes), a three-operation reciprocal, sign tests on
// the bit pattern (a double compare takes the same pipe), the beta-weighted
// sums of Step 5 as combinations of power sums of n.v, and, without velocity
// terms, no per-angle work for sums that are the weights' own.
//
// Measured against the kernel it replaced (slopes and fluxes through shared
// memory, one angle per three barriers, IEEE divisions throughout): 512-cell
// slab of 8 angles 72 -> 40 us per step, 256 x 128 x 80 shadow problem 577 -> 377
// us, 40^3 x 24 moving box 1008 -> 689 us.  Since then, with smaller tiles on small
// grids, alpha formed with the fields, no solves that vanish without velocity and
// the groups below: slab 11.4, shadow problem 371.
//
// Reduction used (both implicit steps are linear in I for fixed T):
//   Step 4 row m:  d_m I_m = r_m + e_m theta - kappa S,   theta = T^4/(4 pi)
//     d_m = 1 + dt C sa - dt sa vn_m,  e_m = dt sa (C + 3 vn_m),
//     kappa = dt sa / C,  S = sum_l g_l I_l,  g_l = W_l (v.v + vn_l^2),
//     vn_m = n_m . v~ ;
//   Step 5 (unknowns x = W I): a_m x_m + sum_l (b_l + c_m) x_l = r'_m with
//     r'_m = I4_m (+ Delta F_m when sigma_s > sigma_a),
//     I4_m = Q_m + (e_m/d_m) theta - kappa S / d_m,
//     Q_m  = r_m / d_m (+ Delta F_m when sigma_s > sigma_a).
// The sums are kept as moments of vn: sum W vn^k f over the angles, k = 0 .. 3,
// with f = 1/d (T_k), r/d (U_k), 1/a' (P_k), 1/(a' d) (D_k), Q/a' (K_k), where
// 1/a_m = W_m / a'_m.
#pragma once

#include "rt_step_sym.cuh"

namespace rtg {

namespace stepk {

// Table of one angle: n (0-2), W (3), W n_i (4-6), W n_i n_j (7-12: xx, yy, zz,
// xy, xz, yz), per axis C mu dt/2dx and mu dt/dx (13-18).
constexpr int kTabD = 19;

// Groups of threads per tile: each takes every GR-th round of angles of all the
// tile's cells, and the groups add their sums up.  An FP64 instruction holds a
// scheduler for 64 cycles whether one lane of the warp is active or all
// (measured: 65 to 77 cycles per multiply-add at 1 to 32 lanes, one warp per
// scheduler), so a small grid gains by more and shorter warps alone: the 1-D tile
// of 32 cells runs four groups, a warp per scheduler, on lines of two cells.  us
// per step on 64-cell tiles of one group and here: 512 cells x 8 angles 24.7 and
// 16.5, 512 x 32 68 and 31, 4096 x 48 99 and 43 (one launch at a time; 11.4 in a
// graph for the first).
template <int DIM, int TX, int TY, int TZ>
constexpr int kGroupsD = DIM == 1 && TX == 32 ? 4 : 1;

template <int DIM, bool VEL, int TX, int TY, int TZ>
struct DoubleGeo {
  static constexpr int GR = kGroupsD<DIM, TX, TY, TZ>;
  using G = SymGeo<DIM, TX, TY, TZ, (GR > 1 ? 2 : 8)>;
  static constexpr int ROUND = G::NT / G::LINES < 8 ? G::NT / G::LINES : 8;   // angles per round
  static constexpr int SUMS = 21;   // partial sums of a group and cell
  static_assert(GR == 1 || G::NT == 32, "a group is a warp");
  __host__ static size_t smem_bytes(int M) {
    return sizeof(double) * (kTabD * (size_t)M + GR * ROUND * ((VEL ? 2 : 1) * G::NBOX + G::NF) +
                             (VEL ? 3 * G::NBOX : 0) + (GR > 1 ? GR * SUMS * G::NT : 0)) +
           sizeof(double2) * G::NC + sizeof(PackedLine) * G::LINES;
  }
};

// 1/x by one step of the cubically convergent hyperpower iteration r (1 + e + e^2),
// e = 1 - x r (M. Altman, Pacific J. Math. 10 (1960) 1107), from the hardware's
// approximation: its relative error is below 2^-19 where x is a normal number
// below 2^1022 in magnitude, so e^3 is below 2^-57 and the result within one unit
// in the last place (1.0 / x is within half of one).  Beyond that range,
// NaN for zero, subnormal and infinite x, 0 from 2^1022 on.
__device__ __forceinline__ double rcp_seed(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rcp_cubic(double x) {
  const double r = rcp_seed(x);
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// Whether rcp_cubic(x) is 1/x: |x| at least 2^-1022 and below 2^1022 (in integers,
// off the FP64 pipe).
__device__ __forceinline__ bool rcp_range(double x) {
  return (unsigned)(__double2hiint(x) & 0x7ff00000) - 0x00100000u < 0x7fc00000u;
}

// 1/x and n/x of every x.
__device__ __forceinline__ double rcp_any(double x) { return rcp_range(x) ? rcp_cubic(x) : 1.0 / x; }
__device__ __forceinline__ double div_any(double n, double x) { return rcp_range(x) ? n * rcp_cubic(x) : n / x; }

// Half van Leer slope from the one-sided differences (see vl_half2).  Their product
// is tested on its bit pattern, off the FP64 pipe: positive up to infinity, which
// a NaN is not.  Where it is, |dl + dr| is at least 2^-537.
__device__ __forceinline__ double vl_diff(double dl, double dr) {
  const double pr = dl * dr;
  const double h = pr * rcp_cubic(dl + dr);
  return (unsigned long long)__double_as_longlong(pr) - 1 < 0x7ff0000000000000ull ? h : 0.0;
}

template <int DIM, bool VEL, int TX, int TY, int TZ>
__device__ __forceinline__ void process_tile_d(const StepArgs<double> &a, int thread, int tbx, int tby, int tbz,
                                               unsigned char *smem_raw) {
  using DG = DoubleGeo<DIM, VEL, TX, TY, TZ>;
  using G = typename DG::G;
  constexpr int NT = G::NT, ROUND = DG::ROUND, SLOTS = G::SLOTS, NBOX = G::NBOX, GR = DG::GR;
  const int tid = GR > 1 ? thread % NT : thread, group = GR > 1 ? thread / NT : 0;
  const int M = a.M;
  const long long N = a.N;
  const int org[3] = {tbx * TX, tby * TY, tbz * TZ};

  double2 *s_fc = reinterpret_cast<double2 *>(smem_raw);        // face constants [NC]
  double *s_tab = reinterpret_cast<double *>(s_fc + G::NC);     // [M][kTabD]
  double *s_all = s_tab + kTabD * M;                            // per group: I~, Delta F, IV
  constexpr int PART = ROUND * ((VEL ? 2 : 1) * NBOX + G::NF);
  double *s_It = s_all + group * PART;                          // I~ [ROUND][NBOX]
  double *s_F = s_It + ROUND * NBOX;                            // Delta F per axis [ROUND][NF]
  double *s_IV = s_F + ROUND * G::NF;                           // IV [ROUND][NBOX] (VEL)
  double *s_w = s_all + GR * PART;                              // w = 3 J v [3][NBOX] (VEL)
  double *s_sum = s_w + (VEL ? 3 * NBOX : 0);                   // [GR][SUMS][NT] (GR > 1)
  PackedLine *s_line = reinterpret_cast<PackedLine *>(s_sum + (GR > 1 ? GR * DG::SUMS * NT : 0));   // [LINES]
  const double C = a.C, invC = a.invC, dt = a.dt;

  // One entry per thread and turn: as products of three factors they cost the warp
  // two operations for every NT entries.
  for (int k = thread; k < kTabD * M; k += NT * GR) {
    const int m = k / kTabD, e = k - kTabD * m;
    // n_i; W; W n_i; W n_i n_j; (C/2) n_d (dt/dx), n_d (dt/dx)
    const int i = e < 3 ? e : e < 4 ? 3 : e < 7 ? e - 4 : e < 10 ? e - 7 : e < 13 ? (e == 12 ? 1 : 0) : (e - 13) >> 1;
    const int j = e < 10 ? e - 7 : e == 10 ? 1 : 2;
    const double *n = a.ang + 4 * m, ni = n[i], dtdx = i == 0 ? a.dtdx[0] : i == 1 ? a.dtdx[1] : a.dtdx[2];
    const double x = e < 4 ? 1.0 : e < 13 ? n[3] : e & 1 ? 0.5 * C : 1.0;
    s_tab[k] = x * ni * (e < 7 ? 1.0 : e < 13 ? n[j] : dtdx);
  }

  // ---- staged cells of this thread (see process_tile_sym) ----------------------
  int sl_box[SLOTS], sl_g[SLOTS];
  auto used = [&](int s) { return (s + 1) * NT <= G::NCROSS || tid + s * NT < G::NCROSS; };
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    sl_box[s] = sl_g[s] = 0;
    if (!used(s)) continue;
    int l[3];
    const int box = G::staged(tid + s * NT, l);
    int g[3], code = 0;
    for (int d = 0; d < 3; ++d) {
      g[d] = d < DIM ? org[d] + l[d] : 0;
      if (d < DIM && (g[d] < 0 || g[d] >= a.n[d])) {
        if (code == 0) code = 1 + 2 * d + (g[d] >= a.n[d] ? 1 : 0);
        g[d] = map_in(g[d], a.n[d], a.bc[d][0], a.bc[d][1]);
      }
    }
    if (code) {
      const int axis = (code - 1) >> 1, side = (code - 1) & 1;
      const int kind = a.bc[axis][side];
      code = (kind == BC_VACUUM || kind == BC_INFLOW) ? (1 | (kind == BC_INFLOW ? 2 : 0) | (axis << 2) | (side << 4)) : 0;
    }
    sl_box[s] = box | (code << 16);
    sl_g[s] = (int)(g[0] + (long long)a.n[0] * (g[1] + (long long)a.n[1] * g[2]));
    if (VEL && group == 0) {
      const double w3 = (3.0 / (4.0 * kPi)) * a.mom_in[sl_g[s]];
      for (int d = 0; d < 3; ++d) s_w[d * NBOX + box] = w3 * a.v[d * N + sl_g[s]];
    }
  }
  double pf[ROUND][SLOTS];   // the next round's angles of each staged cell
  auto fetch = [&](int m0) {
#pragma unroll
    for (int k = 0; k < ROUND; ++k)
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (m0 + k < M && used(s)) pf[k][s] = a.I_in[(long long)(m0 + k) * N + sl_g[s]];
  };
  fetch(group * ROUND);

  // ---- alpha and v of the cells -1 .. T of every axis: face constants -----------
  // alpha of each cell (per axis where the cell sides differ), kept in the I~
  // arrays meanwhile
  double *c_al = s_all, *c_v = s_all;
  const bool same_dx = (DIM < 2 || a.dx[1] == a.dx[0]) && (DIM < 3 || a.dx[2] == a.dx[0]);
  for (int pass = 0; pass < (same_dx ? 1 : DIM); ++pass) {
    if (pass) __syncthreads();
    for (int k = thread; k < G::INNER; k += NT * GR) {
      int l[3], g[3];
      const int box = G::staged(G::inner(k), l);
      for (int d = 0; d < 3; ++d) {
        g[d] = d < DIM ? org[d] + l[d] : 0;
        if (d < DIM && (g[d] < 0 || g[d] >= a.n[d])) g[d] = map_in(g[d], a.n[d], a.bc[d][0], a.bc[d][1]);
      }
      const long long cc = g[0] + (long long)a.n[0] * (g[1] + (long long)a.n[1] * g[2]);
      c_al[box] = (pass == 0 ? a.alpha[0] : pass == 1 ? a.alpha[1] : a.alpha[2])[cc];
    }
    __syncthreads();
    if (thread < G::LINES) {
      Line ln{};
      const int d = G::line(tid, ln), L = d == 0 ? G::LX : d == 1 ? G::LY : G::LZ;
      if (pass == 0) s_line[tid].pack(ln);
      if (same_dx || d == pass) {
        const int np = d == 0 ? G::NPX : d == 1 ? G::NPY : G::NPZ;
        double2 *fc = s_fc + (d == 0 ? tid : d == 1 ? G::CY + tid - G::NPX : G::CZ + tid - G::NPX - G::NPY);
        double al = c_al[ln.lo + ln.slo];
        for (int f = 0; f <= L; ++f) {
          const double al1 = c_al[f < L ? ln.core + f * ln.sc : ln.hi];
          fc[f * np].x = 0.5 * (al + al1);
          al = al1;
        }
      }
    }
  }
  if (VEL) {
    // g = +-(1 - |v_face| dt/dx), positive (and alpha negative) when the cell
    // below the face is the upwind one, infinite at a face of zero velocity
#pragma unroll 1
    for (int d = 0; d < DIM; ++d) {
      __syncthreads();
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
        if (group == 0 && used(s)) c_v[sl_box[s] & 0xffff] = a.v[d * N + sl_g[s]];
      __syncthreads();
      const int first = d == 0 ? 0 : d == 1 ? G::NPX : G::NPX + G::NPY, np = d == 0 ? G::NPX : d == 1 ? G::NPY : G::NPZ;
      if (thread < np) {
        Line ln{};
        G::line(first + tid, ln);
        double2 *fc = s_fc + (d == 0 ? 0 : d == 1 ? G::CY : G::CZ) + tid;
        const int L = d == 0 ? G::LX : d == 1 ? G::LY : G::LZ;
        double v = c_v[ln.lo + ln.slo];
        for (int f = 0; f <= L; ++f) {
          const double v1 = c_v[f < L ? ln.core + f * ln.sc : ln.hi], vf = 0.5 * (v + v1);
          const double h = 1.0 - fabs(vf) * (d == 0 ? a.dtdx[0] : d == 1 ? a.dtdx[1] : a.dtdx[2]);
          fc[f * np].y = vf > 0.0 ? h : vf < 0.0 ? -h : __hiloint2double(0x7ff00000, 0);
          if (vf > 0.0) fc[f * np].x = -fc[f * np].x;
          v = v1;
        }
      }
    }
  }
  __syncthreads();

  // ---- the own cell ---------------------------------------------------------------
  const int lx = tid % TX, ly = (tid / TX) % TY, lz = tid / (TX * TY);
  const int gx = org[0] + lx, gy = org[1] + ly, gz = org[2] + lz;
  const bool valid = gx < a.n[0] && gy < a.n[1] && gz < a.n[2];
  const long long c = valid ? gx + (long long)a.n[0] * (gy + (long long)a.n[1] * gz) : 0;
  double rho = 1, sa = 0, ss = 0, vt[3] = {0, 0, 0}, vin[3] = {0, 0, 0}, T0 = 1;
  if (valid) {
    rho = a.rho[c];
    sa = a.sa[c];
    ss = a.ss[c];
    T0 = a.T_in[c];
    if (VEL) {
      for (int d = 0; d < 3; ++d) vt[d] = vin[d] = a.v[d * N + c];
      if (a.estimate_v) {
        // Step 3 (sec. 4.5): per axis, backward-Euler momentum exchange with
        // E, F, P_dd held at their step-n values
        const double E = a.mom_in[c];
        const double h = 0.5 * dt * (sa + ss);
        for (int d = 0; d < 3; ++d) {
          const double Fd = a.mom_in[(1 + d) * N + c], Pdd = a.mom_in[(4 + d) * N + c];
          const double num = rho * vin[d] + h * (C * rho * vin[d] + a.P * Fd);
          const double den = rho + h * (C * rho + a.P * (E + Pdd) * invC);
          vt[d] = div_any(num, den);
        }
      }
    }
  }
  const bool scat = ss > sa;
  const double A0 = 1.0 + dt * C * sa, A1 = dt * sa, a0 = 1.0 + dt * C * ss, a1 = dt * ss;
  const double rd0 = VEL ? 0.0 : rcp_any(A0), ra0 = VEL ? 0.0 : rcp_any(a0);

  // ---- transport, Q_m and the angle sums: ROUND angles per two barriers -------------
  double Tk[4] = {0, 0, 0, 0}, Pk[4] = {0, 0, 0, 0}, Dk[4] = {0, 0, 0, 0};
  double Uk[3] = {0, 0, 0}, Kk[3] = {0, 0, 0}, pre[3] = {0, 0, 0}, Ws = 0;
  const int kq = tid / G::LINES, line = tid % G::LINES;
  const int axis = line < G::NPX ? 0 : DIM == 2 || line < G::NPX + G::NPY ? 1 : 2;
#pragma unroll 1
  for (int mr = 0; mr < M; mr += GR * ROUND) {
    const int m0 = mr + group * ROUND;   // the group's angles of this round
    double I0[ROUND];   // the own cell's I^n (slot 0 is the own cell)
#pragma unroll
    for (int k = 0; k < ROUND; ++k) {
      const int m = m0 + k;
      I0[k] = pf[k][0];
      if (m >= M) break;
      const double *t = s_tab + kTabD * m;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        if (!used(s)) continue;
        const int box = sl_box[s] & 0xffff, code = sl_box[s] >> 16;
        double I = pf[k][s];
        if (code) {
          // beyond a vacuum or inflow face, the rays that come in
          const int ax = (code >> 2) & 3, side = (code >> 4) & 1;
          const double mu = t[ax];
          if (side ? (mu < 0.0) : (mu > 0.0)) I = (code & 2) ? a.inflow[(ax * 2 + side) * M + m] : 0.0;
        }
        if (VEL) {
          const double iv = t[0] * s_w[box] + t[1] * s_w[NBOX + box] + t[2] * s_w[2 * NBOX + box];
          s_IV[k * NBOX + box] = iv;
          I -= iv * invC;
        }
        s_It[k * NBOX + box] = I;
      }
    }
    fetch(m0 + GR * ROUND);
    __syncthreads();
    if (kq < ROUND && m0 + kq < M) {
      const double *t = s_tab + kTabD * (m0 + kq);
      const double hc = t[13 + 2 * axis], mud = t[14 + 2 * axis], hca = fabs(hc);
      const Line at = s_line[line].unpack();
      auto walk = [&](auto length, auto lines, auto step, double *F, const double2 *fc) {
        constexpr int L = decltype(length)::value, NP = decltype(lines)::value, SF = decltype(step)::value;
        const double *It = s_It + kq * NBOX, *IV = VEL ? s_IV + kq * NBOX : s_It;
        int p = at.lo + at.slo;
        double Ls = It[p], q = It[at.core], d = q - Ls, sL = vl_diff(Ls - It[at.lo], d), fl = 0.0;
        double vL = 0, v = 0, dv = 0, sLv = 0;
        if (VEL) {
          vL = IV[p];
          v = IV[at.core];
          dv = v - vL;
          sLv = vl_diff(vL - IV[at.lo], dv);
        }
        p = at.core;
#pragma unroll
        for (int f = 0; f <= L; ++f) {
          p = f + 1 < L ? p + at.sc : f + 1 == L ? at.hi : p + at.shi;
          const double qn = It[p];
          const double2 k = fc[f * NP];
          const double e = qn - q;
          const double sR = vl_diff(d, e);
          const double ha = hca * fabs(k.x);             // alpha C |mu| dt / 2dx
          const double hl = 1.0 - 2.0 * ha;              // 1 - nu
          const double S = Ls + hl * sL, R = q - hl * sR;
          double g = (hc + ha) * S + (hc - ha) * R;
          if (VEL) {
            // IV at the face: the upwind cell's state (sec. 4.2), or the mean
            // of both at a face of zero velocity
            const double vn = IV[p], ev = vn - v, sRv = vl_diff(dv, ev);
            const bool below = __double2hiint(k.x) < 0, zero = __double2hiint(k.y) == 0x7ff00000;
            double iv;
            if (zero)
              iv = 0.5 * ((vL + sLv) + (v - sRv));
            else
              iv = k.y * (below ? sLv : sRv) + (below ? vL : v);
            g += mud * iv;
            vL = v;
            v = vn;
            dv = ev;
            sLv = sRv;
          }
          if (f > 0) F[(f - 1) * SF] = fl - g;
          fl = g;
          Ls = q;
          q = qn;
          d = e;
          sL = sR;
        }
      };
      double *F = s_F + kq * G::NF;
      if (axis == 0)
        walk(IntTag<G::LX>{}, IntTag<G::NPX>{}, IntTag<G::SX>{}, F + line, s_fc + line);
      else if constexpr (DIM >= 2) {
        if (axis == 1)
          walk(IntTag<G::LY>{}, IntTag<G::NPY>{}, IntTag<G::SY>{}, F + G::FY + line - G::NPX, s_fc + G::CY + line - G::NPX);
        else if constexpr (DIM == 3)
          walk(IntTag<G::LZ>{}, IntTag<G::NPZ>{}, IntTag<G::SZ>{}, F + G::FZ + line - G::NPX - G::NPY,
               s_fc + G::CZ + line - G::NPX - G::NPY);
      }
    }
    __syncthreads();
    if (!valid) continue;
#pragma unroll
    for (int k = 0; k < ROUND; ++k) {
      const int m = m0 + k;
      if (m >= M) break;
      const double *t = s_tab + kTabD * m, *F = s_F + k * G::NF;
      double dF = F[G::part_x(lx, ly, lz)];
      if (DIM >= 2) dF += F[G::part_y(lx, ly, lz)];
      if (DIM == 3) dF += F[G::part_z(lx, ly, lz)];
      const double full = I0[k] + dF, r = scat ? I0[k] : full, W = t[3];
      double Q;
      if (VEL) {
        const double vn = t[0] * vt[0] + t[1] * vt[1] + t[2] * vt[2];
        const double rd = rcp_any(A0 - A1 * vn), ra = rcp_any(a0 - a1 * vn);
        const double u = r * rd;
        Q = scat ? u + dF : u;
        const double z = Q * ra, pd = ra * rd, y1 = W * vn, y2 = y1 * vn, y3 = y2 * vn;
        Tk[0] += W * rd; Tk[1] += y1 * rd; Tk[2] += y2 * rd; Tk[3] += y3 * rd;
        Pk[0] += W * ra; Pk[1] += y1 * ra; Pk[2] += y2 * ra; Pk[3] += y3 * ra;
        Dk[0] += W * pd; Dk[1] += y1 * pd; Dk[2] += y2 * pd; Dk[3] += y3 * pd;
        Uk[0] += W * u; Uk[1] += y1 * u; Uk[2] += y2 * u;
        Kk[0] += W * z; Kk[1] += y1 * z; Kk[2] += y2 * z;
      } else {
        const double u = r * rd0;
        Q = scat ? u + dF : u;
        Ws += W;
        Uk[0] += W * u;
        Kk[0] += W * Q;
      }
      for (int i = 0; i < 3; ++i) pre[i] += t[4 + i] * full;   // sum W n (I^n + Delta F)
      a.I_out[(long long)m * N + c] = Q;
    }
  }
  // Adds up n sums of the groups (in their order) and hands the totals to every thread.
  auto total = [&](auto count, double *const (&x)[decltype(count)::value]) {
    constexpr int n = decltype(count)::value;
    static_assert(n <= DG::SUMS, "room for a group's sums");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < n; ++i) s_sum[(group * n + i) * NT + tid] = *x[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < n; ++i) {
      double t = s_sum[i * NT + tid];
#pragma unroll
      for (int g = 1; g < GR; ++g) t += s_sum[(g * n + i) * NT + tid];
      *x[i] = t;
    }
  };
  if constexpr (GR == 1) {
    if (!valid) return;
  } else if constexpr (VEL) {
    total(IntTag<21>{}, {&Tk[0], &Tk[1], &Tk[2], &Tk[3], &Pk[0], &Pk[1], &Pk[2], &Pk[3], &Dk[0], &Dk[1], &Dk[2],
                         &Dk[3], &Uk[0], &Uk[1], &Uk[2], &Kk[0], &Kk[1], &Kk[2], &pre[0], &pre[1], &pre[2]});
  } else {
    total(IntTag<6>{}, {&Ws, &Uk[0], &Kk[0], &pre[0], &pre[1], &pre[2]});
  }
  if (!VEL) {
    Tk[0] = Ws * rd0;
    Pk[0] = Ws * ra0;
    Dk[0] = Ws * (rd0 * ra0);
    Kk[0] *= ra0;
  }

  // ---- Step 4 solve: S, J, v.H affine in theta; scalar quartic in T ---------
  // Without velocity terms vn = 0, only the sums without vn remain, and S, H and s2 vanish.
  double v2 = 0, kap = 0, S0 = 0, S1 = 0, J0 = Uk[0], H0 = 0, H1 = 0, omJ1 = Tk[0];
  if (VEL) {
    v2 = vt[0] * vt[0] + vt[1] * vt[1] + vt[2] * vt[2];
    kap = A1 * invC;
    const double Gr = v2 * Uk[0] + Uk[2], G1 = v2 * Tk[0] + Tk[2];
    const double Ve = A1 * (C * Tk[1] + 3.0 * Tk[2]);
    const double Ge = A1 * (C * G1 + 3.0 * (v2 * Tk[1] + Tk[3]));
    const double Wq = Tk[0] - 4.0 * A1 * Tk[1];     // sum W (d - e) / d
    const double den = 1.0 + kap * G1;
    S0 = div_any(Gr, den);
    S1 = div_any(Ge, den);
    J0 = Uk[0] - kap * S0 * Tk[0];
    H0 = Uk[1] - kap * S0 * Tk[1];
    H1 = Ve - kap * S1 * Tk[1];
    omJ1 = Wq + kap * S1 * Tk[0];   // 1 - dJ/dtheta, cancellation-free
  }
  const double kv = rho * a.kv_per_rho;
  double T1 = T0;
  if (!a.hold_T && (GR == 1 || valid)) {
    const double beta = a.P * C * (VEL ? 1.0 - v2 * invC * invC : 1.0) * sa;
    const double kin0 = VEL ? 8.0 * kPi * a.P * sa * (H0 - S0 * invC) : 0.0;
    const double kin1 = VEL ? 2.0 * a.P * sa * (H1 - S1 * invC) : 0.0;
    const double c0 = dt * (kin0 - 4.0 * kPi * beta * J0) - kv * T0;
    const double c4 = dt * (kin1 + beta * omJ1);
    // the FP64 reference's iteration and stopping rule (with its default
    // options): Newton from T^n until |dT| <= newton_rtol T, then one more
    // step, at most newton_max_it steps
    const double rtol = a.newton_rtol;
    const int max_it = a.newton_max_it;
    double T = T0;
    int extra = -1, it;
    for (it = 0; it < max_it; ++it) {
      const double T3 = T * T * T;
      const double f = c4 * T3 * T + kv * T + c0;
      const double fp = 4.0 * c4 * T3 + kv;
      double Tn = T - div_any(f, fp);
      if (!(Tn > 0)) Tn = 0.5 * T;
      const double dT = Tn - T;
      T = Tn;
      if (extra == 0) break;
      if (extra < 0 && fabs(dT) <= rtol * T) extra = 0;
    }
    if (it >= max_it && group == 0) atomicAdd(a.status, 1);
    T1 = T;
  }
  const double T1sq = T1 * T1, th = T1sq * T1sq * (1.0 / (4.0 * kPi));
  double kS = 0, s1, s2 = 0, cq = 0;
  if (VEL) {
    kS = kap * (S0 + th * S1);

    // ---- Step 5 solve: (1+B1) s1 + Bc s2 = Br,  A1 s1 + (1+Ac) s2 = Ar -------
    // b_m = bq0 + bq1 vn + bq2 vn^2, c_m = cq vn; e_m / d_m = A1 (C + 3 vn) / d_m
    const double bq0 = -a1 * C - a1 * v2 * invC, bq1 = 2.0 * a1, bq2 = -a1 * invC;
    cq = -3.0 * a1;
    const double Bd = bq0 * Dk[0] + bq1 * Dk[1] + bq2 * Dk[2], Bdv = bq0 * Dk[1] + bq1 * Dk[2] + bq2 * Dk[3];
    const double Ap = A1 * (C * Dk[0] + 3.0 * Dk[1]), Bp = A1 * (C * Bd + 3.0 * Bdv);
    const double BQ = bq0 * Kk[0] + bq1 * Kk[1] + bq2 * Kk[2];
    const double Ar = Kk[0] + th * Ap - kS * Dk[0];
    const double Br = BQ + th * Bp - kS * Bd;
    // 1 + sum W b / a', formed without cancellation
    const double m11 = (1.0 - a1 * v2 * invC) * Pk[0] + a1 * Pk[1] - a1 * invC * Pk[2];
    const double m12 = cq * (bq0 * Pk[1] + bq1 * Pk[2] + bq2 * Pk[3]);
    const double m21 = Pk[0], m22 = 1.0 + cq * Pk[1];
    const double det = m11 * m22 - m12 * m21;
    s1 = div_any(Br * m22 - m12 * Ar, det);
    s2 = div_any(m11 * Ar - m21 * Br, det);
  } else {
    // (1 + B1) s1 = Br alone, with b_m = -a1 C
    s1 = div_any(-a1 * C * (Kk[0] + th * (A1 * C * Dk[0])), Pk[0]);
  }

  // ---- I^{n+1} over Q_m, quadrature (sec. 3) ------------------------------------
  // I = (Q + (y0 + y1 vn) / d - s1 - cq s2 vn) / a'
  const double y0 = A1 * C * th - kS, y1 = 3.0 * A1 * th, z1 = cq * s2;
  const double k0 = (y0 * rd0 - s1) * ra0;   // without velocity: I = Q / a' + k0
  double mom[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  // the group's next angle, its right-hand sides read two angles ahead
  auto after = [](int m) { return GR == 1 || (m + 1) % ROUND ? m + 1 : m + 1 + (GR - 1) * ROUND; };
  const int first = group * ROUND;
  auto read = [&](int m) { return (GR == 1 || valid) && m < M ? a.I_out[(long long)m * N + c] : 0.0; };
  double Qn = read(first), Qnn = read(after(first));
#pragma unroll 2
  for (int m = first; m < M; m = after(m)) {
    const double Q = Qn;
    Qn = Qnn;
    Qnn = read(after(after(m)));
    const double *t = s_tab + kTabD * m;
    double I1;
    if (VEL) {
      const double vn = t[0] * vt[0] + t[1] * vt[1] + t[2] * vt[2];
      const double rd = rcp_any(A0 - A1 * vn), ra = rcp_any(a0 - a1 * vn);
      I1 = (Q + rd * (y0 + y1 * vn) - s1 - z1 * vn) * ra;
    } else {
      I1 = Q * ra0 + k0;
    }
    if (GR == 1 || valid) a.I_out[(long long)m * N + c] = I1;
#pragma unroll
    for (int i = 0; i < 10; ++i) mom[i] += t[3 + i] * I1;   // W, W n_i, W n_i n_j
  }
  if constexpr (GR == 1) {
    for (int i = 0; i < 10; ++i) a.mom_out[(long long)i * N + c] = 4.0 * kPi * mom[i];
  } else {
    // group 0 adds up E, F and goes on to the sources, the others two of P each
    static_assert(GR == 4, "four groups");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 10; ++i) s_sum[(group * 10 + i) * NT + tid] = mom[i];
    __syncthreads();
    auto moment = [&](int i) {
      double t = s_sum[i * NT + tid];
#pragma unroll
      for (int g = 1; g < GR; ++g) t += s_sum[(g * 10 + i) * NT + tid];
      if (valid) a.mom_out[(long long)i * N + c] = 4.0 * kPi * t;
      return t;
    };
    if (group > 0) {
      moment(2 + 2 * group);
      moment(3 + 2 * group);
      return;
    }
    for (int i = 0; i < 4; ++i) mom[i] = moment(i);
    if (!valid) return;
  }

  // ---- gas sources (sec. 4.3: Delta E_T, eqs. momentumchange, kinetichange)
  const double kmom = -4.0 * kPi * a.P * invC;
  double dEK = 0, work[3];   // 2 rho times the work on each component
  for (int i = 0; i < 3; ++i) {
    const double dmom = kmom * (mom[1 + i] - pre[i]);
    a.dMom[i * N + c] = dmom;
    const double m0 = rho * vin[i];
    work[i] = (m0 + dmom) * (m0 + dmom) - m0 * m0;
  }
  const double rho2 = 2.0 * rho;
  if (rcp_range(rho2)) {   // one test for the three of them
    const double r = rcp_cubic(rho2);
    for (int i = 0; i < 3; ++i) dEK += work[i] * r;
  } else {
    for (int i = 0; i < 3; ++i) dEK += work[i] / rho2;
  }
  a.T_out[c] = T1;
  a.dEgas[c] = kv * (T1 - T0) + dEK;
}

template <int DIM, bool VEL, int TX, int TY, int TZ>
__global__ void __launch_bounds__(TX * TY * TZ * kGroupsD<DIM, TX, TY, TZ>) step_kernel_d(const StepArgs<double> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int o = a.outer_begin;
  process_tile_d<DIM, VEL, TX, TY, TZ>(a, threadIdx.x, blockIdx.x + (DIM == 1 ? o : 0), blockIdx.y + (DIM == 2 ? o : 0),
                                       blockIdx.z + (DIM == 3 ? o : 0), smem_raw);
}

template <int DIM, bool VEL, int TX, int TY, int TZ>
cudaError_t launch_shape_d(const StepArgs<double> &a, cudaStream_t s) {
  const size_t sm = DoubleGeo<DIM, VEL, TX, TY, TZ>::smem_bytes(a.M);
  auto kern = step_kernel_d<DIM, VEL, TX, TY, TZ>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid((a.n[0] + TX - 1) / TX, (a.n[1] + TY - 1) / TY, (a.n[2] + TZ - 1) / TZ);
  if (a.outer_count > 0) (DIM == 3 ? grid.z : DIM == 2 ? grid.y : grid.x) = a.outer_count;
  kern<<<grid, TX * TY * TZ * kGroupsD<DIM, TX, TY, TZ>, sm, s>>>(a);
  return cudaGetLastError();
}

}  // namespace stepk

}  // namespace rtg
