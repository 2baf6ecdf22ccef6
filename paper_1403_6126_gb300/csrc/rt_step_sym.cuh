// Fused radiation-transfer step with float intensities for angle sets made
// of opposite pairs (Jiang, Stone & Davis 2014, arXiv:1403.6126, secs. 3-4).
//
// Every level-symmetric set (sec. 3) holds with each angle n its opposite -n
// at the same weight.  A context whose set does keeps its intensities pair by
// pair (pair_order): the quad-interleaved layout of rt_step_quad.cuh with (n,
// n', -n, -n') in a float4.  It takes this kernel; other sets take the quad
// kernel.  Same method, deviation arithmetic and per-cell solves as there; what
// differs:
//
//  * The velocity term.  IV_m = 3 (n_m.v) J changes sign with n, and so does
//    its van Leer slope, so the face term mu IV is the same for n and -n:
//    staged, sloped and upwinded once per pair.
//  * One |mu| per axis and pair: 1 - nu and the two upwind weights of a face
//    (c1 = C mu dt/2dx + alpha C |mu| dt/2dx on the state below, c2 = the
//    difference on the state above) are formed once, and -n takes them
//    swapped and negated.
//  * The transport runs along lines.  A thread takes a line of up to eight
//    cells of the tile along one axis for one quad and walks it with the van
//    Leer differences, slopes and the last flux in registers: each is formed
//    once per line (plus its two extension cells), and only I^n, IV and Delta F
//    per axis pass through shared memory: 24 128-bit accesses per cell and quad
//    instead of 57 (by the wavefronts counted), and two CTA barriers per round of ROUND quads
//    instead of three per quad.
//  * I^n comes in by asynchronous copies, a round of quads ahead, in a second
//    buffer; I~ = I - IV/C is formed as a walk reads a cell.
//  * Q_m and the sums that depend on the intensity are taken as soon as a
//    round's Delta F is there, with I^n from shared memory: Delta F never goes
//    to global memory and I^n is read once.  The sums that depend on the
//    velocity and the opacities alone have a loop of their own.
//  * The angle sums take the even and odd parts of a pair: sums of W vn^k
//    f(vn) need f(vn) +- f(-vn) only, and the quadrature of sec. 3 has one
//    term per pair.
//
// What bounds it: issue and latency together.  At 96^3 cells x 80 angles (8x8x4
// tile, two CTAs of 256 threads at 125 registers) it issues 173 thread
// instructions per cell-angle (the quad kernel 197) at 57 % of the issue rate
// (48 %), FMA pipe 42 %, 97 shared-memory wavefronts per warp and quad (227),
// DRAM 0.80 GB for 0.57 GB of intensities: 0.545 ms against 0.726 ms without the
// profiler; 128^3 x 80: 1.27 against 1.72 ms.  Measured and not kept (96^3): 128-thread CTAs, three
// per SM, with the long x and y lines in one phase and the short z lines in
// the next (0.77: 12 warps); one pair per thread, two threads per cell, 64
// registers (0.76: 32 warps, but twice the instructions without the packed
// arithmetic of two pairs); three CTAs at 80 registers (0.77: spills); a
// separate source loop over Delta F in global memory (0.58).
//
// Sums run in the stored order of the angles and no arithmetic depends on
// the tile shape, so results are bitwise the same for every tile shape, in a
// batch, and in the allocation-free step (which reads and writes the
// caller's angle order: GATHER).
#pragma once

#include "rt_step_quad.cuh"

namespace rtg {

namespace stepk {

constexpr int kSymMaxAngles = 80;
constexpr int kSymQuads = kSymMaxAngles / 4;

// Table entries per quad: pairs of floats, (value at n, value at n'), ready as
// operands of the packed arithmetic.
enum {
  kSymN = 0,     // n_x, n_y, n_z
  kSymW = 3,     // W
  kSymWn = 4,    // W n_i
  kSymWnn = 7,   // W n_i n_j: xx, yy, zz, xy, xz, yz
  kSymHc = 13,   // per axis: C mu dt/2dx (13, 15, 17), mu dt/dx (14, 16, 18)
  kSymTab = 20   // (the last is padding)
};

// The table in the launch parameters, the inflow intensities per face and
// angle in stored order, and (GATHER) the caller's index of each stored angle.
struct SymTable {
  float4 e[kSymQuads][kSymTab / 2];   // two entries each
  float inflow[6][kSymMaxAngles];
  unsigned char slot[kSymMaxAngles];
  unsigned char pairs[kSymQuads];   // (GATHER) both halves of the quad lie on 8-byte words of the caller's layout
};

// Entries of one quad from its four angles q16 = (n_x, n_y, n_z, W) of n, n',
// -n, -n'.
__host__ __device__ inline void sym_tab_quad(float2 *out, const float *q16, float C, const float dtdx[3]) {
  const float hC = 0.5f * C;
  for (int l = 0; l < 2; ++l) {
    const float *n = q16 + 4 * l;
    const float W = n[3];
    float v[kSymTab];
    for (int d = 0; d < 3; ++d) {
      v[kSymN + d] = n[d];
      v[kSymHc + 2 * d] = hC * n[d] * dtdx[d];
      v[kSymHc + 2 * d + 1] = n[d] * dtdx[d];
      v[kSymWn + d] = W * n[d];
      v[kSymWnn + d] = W * n[d] * n[d];
    }
    v[kSymW] = W;
    v[kSymWnn + 3] = W * n[0] * n[1];
    v[kSymWnn + 4] = W * n[0] * n[2];
    v[kSymWnn + 5] = W * n[1] * n[2];
    v[kSymTab - 1] = 0.0f;
    for (int j = 0; j < kSymTab; ++j) (l == 0 ? out[j].x : out[j].y) = v[j];
  }
}

// Host side: ang [M][4] and inflow [6][M] (or NULL) in stored order; order
// (or NULL) the caller's index of each stored angle.
inline void fill_symtable(SymTable *t, const float *ang, int M, float C, const float dtdx[3], const float *inflow,
                          const int *order) {
  for (int q = 0; q < M / 4; ++q) sym_tab_quad(reinterpret_cast<float2 *>(t->e[q]), ang + 16 * q, C, dtdx);
  for (int f = 0; f < 6; ++f)
    for (int m = 0; m < kSymMaxAngles; ++m) t->inflow[f][m] = (inflow && m < M) ? inflow[f * M + m] : 0.0f;
  for (int m = 0; m < kSymMaxAngles; ++m) t->slot[m] = (unsigned char)((order && m < M) ? order[m] : m);
  for (int q = 0; q < kSymQuads; ++q) {
    const unsigned char *m = t->slot + 4 * q;
    t->pairs[q] = m[0] % 2 == 0 && m[1] == m[0] + 1 && m[2] % 2 == 0 && m[3] == m[2] + 1;
  }
}

// Where a line's staged cells lie in shared memory (index, step).
struct Line {
  int lo, slo;      // cells -2, -1
  int core, sc;     // cells 0 .. L - 1
  int hi, shi;      // cells L, L + 1
};

// The same in 16-bit fields.
struct PackedLine {
  unsigned lo_slo, core_sc, hi_shi;
  __device__ __forceinline__ void pack(const Line &l) {
    lo_slo = l.lo | l.slo << 16;
    core_sc = l.core | l.sc << 16;
    hi_shi = l.hi | l.shi << 16;
  }
  __device__ __forceinline__ Line unpack() const {
    Line l;
    l.lo = lo_slo & 0xffff; l.slo = lo_slo >> 16;
    l.core = core_sc & 0xffff; l.sc = core_sc >> 16;
    l.hi = hi_shi & 0xffff; l.shi = hi_shi >> 16;
    return l;
  }
};

// Geometry of a tile of NT cells.  Staged cells: the tile with its x halo in
// rows of odd length (core), then the y halo [z][4][x] and the z halo
// [4][y][x].  Lines of an axis: L? cells each, NP? of them; their Delta F is
// kept as [position][line], x and y with one line of padding (threads that
// read a row along x then fall on different banks), their face constants as
// [face][line].
//
// Lines of eight cells, or of four in a 3-D tile of 128 cells: its lines along y
// and z are that short already, and the eight-cell ones along x kept the other
// threads waiting (8x4x4, us per step: 96 x 80 x 72 x 24 angles 211 -> 162,
// 75 x 50 x 61 x 48 without velocity 134 -> 99, 128^3 x 80 2066 -> 1363; the larger tiles, with
// a line for every thread, lose by it: 8x8x4 1261 -> 1381).
template <int DIM, int TX, int TY, int TZ>
constexpr int kLineMax = DIM == 3 && TX * TY * TZ == 128 ? 4 : 8;

template <int DIM, int TX, int TY, int TZ, int LMAX = kLineMax<DIM, TX, TY, TZ>>
struct SymGeo {
  static constexpr int NT = TX * TY * TZ;
  static constexpr int LX = TX < LMAX ? TX : LMAX, LY = TY < LMAX ? TY : LMAX, LZ = TZ;
  static constexpr int NPX = NT / LX, NPY = DIM >= 2 ? NT / LY : 0, NPZ = DIM >= 3 ? NT / LZ : 0;
  static constexpr int LINES = NPX + NPY + NPZ;         // lines of one quad
  static constexpr int ROUND = NT / LINES < 4 ? NT / LINES : 4;   // quads per round: a line per thread at most
  static_assert(ROUND >= 1, "a thread for every line of a quad");
  static constexpr int RX = (TX + 2 * kHalo) | 1;
  static constexpr int CORE = RX * TY * TZ, YH = DIM >= 2 ? 2 * kHalo * TX * TZ : 0;
  static constexpr int NBOX = CORE + YH + (DIM >= 3 ? 2 * kHalo * TX * TY : 0);
  static constexpr int NCROSS = NT + 2 * kHalo * (TY * TZ + (DIM >= 2 ? TX * TZ : 0) + (DIM >= 3 ? TX * TY : 0));
  static constexpr int SX = NPX + 1, SY = NPY + 1, SZ = NPZ;   // Delta F: steps along the line
  static constexpr int FY = LX * SX, FZ = FY + LY * SY, NF = FZ + (DIM >= 3 ? LZ * SZ : 0);
  // face constants: face f of line p of an axis at C? + f NP? + p
  static constexpr int CY = (LX + 1) * NPX, CZ = CY + (LY + 1) * NPY, NC = CZ + (LZ + 1) * NPZ;
  static constexpr int SLOTS = (NCROSS + NT - 1) / NT;   // staged cells per thread

  // Staged cell k (0 .. NCROSS - 1: the tile, x halo, y halo, z halo): its
  // place in the tile (-2 .. T + 1) and, returned, in shared memory.  The x
  // halo runs over its four layers fastest: the two cells of a side share a
  // 32-byte sector of the intensity array.
  __host__ __device__ static constexpr int staged(int k, int l[3]) {
    if (k < NT) {
      l[0] = k % TX; l[1] = (k / TX) % TY; l[2] = k / (TX * TY);
      return l[0] + kHalo + RX * (l[1] + TY * l[2]);
    }
    k -= NT;
    if (k < 2 * HX) {
      const int r = k / (2 * kHalo);
      l[0] = outside(k % (2 * kHalo), TX); l[1] = r % TY; l[2] = r / TY;
      return l[0] + kHalo + RX * r;
    }
    k -= 2 * HX;
    if (k < YH) {
      l[0] = k % TX; l[1] = outside((k / TX) % (2 * kHalo), TY); l[2] = k / (2 * kHalo * TX);
      return CORE + k;
    }
    k -= YH;
    l[0] = k % TX; l[1] = (k / TX) % TY; l[2] = outside(k / (TX * TY), TZ);
    return CORE + YH + k;
  }
  __host__ __device__ static constexpr int outside(int h, int T) { return h < kHalo ? h - kHalo : T + h - kHalo; }

  // Of the staged cells, the tile's and the inner halo layers (-1 and T): item k
  // (0 .. INNER - 1) is staged cell inner(k).
  static constexpr int HX = 2 * TY * TZ, HY = DIM >= 2 ? 2 * TX * TZ : 0, HZ = DIM >= 3 ? 2 * TX * TY : 0;
  static constexpr int INNER = NT + HX + HY + HZ;
  __host__ __device__ static constexpr int inner(int k) {
    if (k < NT) return k;
    k -= NT;
    if (k < HX) return NT + 2 * kHalo * (k >> 1) + 1 + (k & 1);
    k -= HX;
    if (k < HY) return NT + 2 * HX + 2 * kHalo * TX * (k / (2 * TX)) + TX + k % (2 * TX);
    k -= HY;
    return NT + 2 * HX + 2 * HY + TX * TY + k;
  }

  // Place in the tile of position pos of line p along axis d.
  __host__ __device__ static constexpr void line_cell(int d, int p, int pos, int l[3]) {
    if (d == 0) {
      const int r = p % (TY * TZ);
      l[0] = (p / (TY * TZ)) * LX + pos; l[1] = r % TY; l[2] = r / TY;
    } else if (d == 1) {
      l[0] = p % TX; l[1] = (p / (TX * TZ)) * LY + pos; l[2] = (p / TX) % TZ;
    } else {
      l[0] = p % TX; l[1] = (p / TX) % TY; l[2] = (p / (TX * TY)) * LZ + pos;
    }
  }

  // Line e of a quad (x lines, then y, then z); returns its axis.
  __host__ __device__ static constexpr int line(int e, Line &ln) {
    if (e < NPX) {
      const int r = e % (TY * TZ), seg = e / (TY * TZ);
      ln.core = RX * r + kHalo + seg * LX;
      ln.sc = ln.slo = ln.shi = 1;
      ln.lo = ln.core - kHalo;
      ln.hi = ln.core + LX;
      return 0;
    }
    if (DIM == 2 || e < NPX + NPY) {
      const int p = e - NPX;
      const int x = p % TX, z = (p / TX) % TZ, seg = p / (TX * TZ);
      const int yh = CORE + x + TX * 2 * kHalo * z;
      // a long column is several lines, whose inner ends lie in the core
      const bool first = seg == 0, last = (seg + 1) * LY == TY;
      ln.core = x + kHalo + RX * (seg * LY + TY * z);
      ln.sc = RX;
      ln.lo = first ? yh : ln.core - kHalo * RX;
      ln.slo = first ? TX : RX;
      ln.hi = last ? yh + kHalo * TX : ln.core + LY * RX;
      ln.shi = last ? TX : RX;
      return 1;
    }
    const int p = e - NPX - NPY;
    ln.core = p % TX + kHalo + RX * (p / TX);
    ln.sc = RX * TY;
    ln.lo = CORE + YH + p;
    ln.slo = ln.shi = TX * TY;
    ln.hi = ln.lo + kHalo * TX * TY;
    return 2;
  }
  // Where the parts of Delta F of the tile's cell at (x, y, z) lie.
  __host__ __device__ static constexpr int part_x(int x, int y, int z) {
    return (x % LX) * SX + y + TY * (z + TZ * (x / LX));
  }
  __host__ __device__ static constexpr int part_y(int x, int y, int z) {
    return FY + (y % LY) * SY + x + TX * (z + TZ * (y / LY));
  }
  __host__ __device__ static constexpr int part_z(int x, int y, int z) { return FZ + z * SZ + x + TX * y; }
};

template <int DIM, bool VEL, int TX, int TY, int TZ>
__host__ __device__ constexpr size_t smem_bytes_sym_t(bool tab_param) {
  using G = SymGeo<DIM, TX, TY, TZ>;
  return (tab_param ? 0 : kSymQuads * kSymTab * sizeof(float2)) +
         G::ROUND * ((2 * G::NBOX + G::NF) * sizeof(float4) + (VEL ? G::NBOX * sizeof(float2) : 0)) + G::NC * sizeof(float2) +
         (VEL ? 3 * G::NBOX * sizeof(float) : 0) + G::LINES * sizeof(PackedLine);
}

// With GATHER also room for I^{n+1} of the tile.
template <int DIM, bool VEL, int TX, int TY, int TZ>
__host__ __device__ constexpr size_t smem_bytes_gather_t(int M) {
  const size_t step = smem_bytes_sym_t<DIM, VEL, TX, TY, TZ>(true), out = (size_t)M * TX * TY * TZ * sizeof(float);
  return step > out ? step : out;
}

// Asynchronous copy of BYTES bytes from global to shared memory (16: past L1;
// 4, 8: through it, as the other words of a sector belong to later copies).
template <int BYTES>
__device__ __forceinline__ void copy_async(void *smem, const void *gmem) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem);
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(dst), "l"(gmem), "n"(BYTES) : "memory");
}

// Half van Leer slope from the one-sided differences (see vl_half2).
__device__ __forceinline__ f2 vl_diff(f2 dl, f2 dr) {
  const f2 pr = p_mul(dl, dr);
  const f2 h = p_mul(pr, p_rcp(p_add(dl, dr)));
  return make_float2(pr.x > 0.0f ? h.x : 0.0f, pr.y > 0.0f ? h.y : 0.0f);
}

// The state of a walk along a line: the cell below the next face (It, slope;
// the pair n, n' in p, the opposite pair in n), the cell above it, the
// difference across the face, and the flux of the last face (n: negated).
template <bool VEL, bool GEN>
struct Walk {
  f2 Lp, Ln, sLp, sLn, qp, qn, dp, dn, fp, fn;
  f2 vL, v, dv, sLv;   // the same of IV

  // Cells -2, -1, 0.
  __device__ __forceinline__ void start(float4 a, float4 b, float4 c, f2 va, f2 vb, f2 vc) {
    Lp = lo2(b); Ln = hi2(b);
    qp = lo2(c); qn = hi2(c);
    dp = p_sub(qp, Lp); dn = p_sub(qn, Ln);
    sLp = vl_diff(p_sub(Lp, lo2(a)), dp);
    sLn = vl_diff(p_sub(Ln, hi2(a)), dn);
    if (VEL) {
      vL = vb;
      v = vc;
      dv = p_sub(v, vL);
      sLv = vl_diff(p_sub(vL, va), dv);
    }
  }

  // The next face, with the cell after the one above it (x, vx); hc = C mu
  // dt/2dx, hca its magnitude and mud = mu dt/dx of (n, n'); k: the face's constants (alpha,
  // negative when the cell below is the upwind one; g = +-(1 - |v_face| dt/dx),
  // positive when it is, infinite at a face of exactly zero velocity, which
  // takes the mean of both sides' states; GEN: there may be such faces).
  // Returns flux below minus flux above of the cell passed.
  __device__ __forceinline__ float4 face(float4 x, f2 vx, f2 hc, f2 hca, f2 mud, float2 k) {
    const f2 ep = p_sub(lo2(x), qp), en = p_sub(hi2(x), qn);
    const f2 sRp = vl_diff(dp, ep), sRn = vl_diff(dn, en);
    const float al = fabsf(k.x);
    const f2 ha = make_float2(hca.x * al, hca.y * al);               // alpha C |mu| dt / 2dx
    const f2 hl = p_fma(ha, dup(-2.0f), dup(1.0f)), nhl = make_float2(-hl.x, -hl.y);   // 1 - nu
    const f2 c1 = p_add(hc, ha), c2 = p_sub(hc, ha);
    const f2 Sp = p_fma(hl, sLp, Lp), Rp = p_fma(nhl, sRp, qp);
    const f2 Sn = p_fma(hl, sLn, Ln), Rn = p_fma(nhl, sRn, qn);
    f2 gp, gn;
    if (VEL) {
      const f2 ev = p_sub(vx, v);
      const f2 sRv = vl_diff(dv, ev);
      const bool below = __float_as_int(k.x) < 0;
      const f2 qu = make_float2(below ? vL.x : v.x, below ? vL.y : v.y);
      const f2 su = make_float2(below ? sLv.x : sRv.x, below ? sLv.y : sRv.y);
      f2 iv = make_float2(fmaf(k.y, su.x, qu.x), fmaf(k.y, su.y, qu.y));
      if (GEN) {   // a face of zero velocity (h = 1): the mean of both states
        const f2 mean = p_mul(dup(0.5f), p_add(p_add(vL, sLv), p_sub(v, sRv)));
        const bool zero = k.y > 1e30f;
        iv = make_float2(zero ? mean.x : iv.x, zero ? mean.y : iv.y);
      }
      // mu IV is the same for n and -n
      const f2 m = p_mul(mud, iv);
      gp = p_fma(c1, Sp, p_fma(c2, Rp, m));
      gn = p_fma(c2, Sn, p_fma(c1, Rn, make_float2(-m.x, -m.y)));
      vL = v;
      v = vx;
      dv = ev;
      sLv = sRv;
    } else {
      gp = p_fma(c1, Sp, p_mul(c2, Rp));
      gn = p_fma(c2, Sn, p_mul(c1, Rn));
    }
    const float4 out = mk4(p_sub(fp, gp), p_sub(gn, fn));
    fp = gp; fn = gn;
    Lp = qp; Ln = qn;
    sLp = sRp; sLn = sRn;
    dp = ep; dn = en;
    qp = lo2(x); qn = hi2(x);
    return out;
  }
};

template <int V>
struct IntTag {
  static constexpr int value = V;
};

// n.v~ of the pairs (n, n'), and 1 / (b + s vn): scalar multiply-adds, whose
// operands need not be doubled into register pairs.
__device__ __forceinline__ f2 vn_of(const float vt[3], f2 nx, f2 ny, f2 nz) {
  return make_float2(fmaf(nz.x, vt[2], fmaf(nx.x, vt[0], ny.x * vt[1])), fmaf(nz.y, vt[2], fmaf(nx.y, vt[0], ny.y * vt[1])));
}
__device__ __forceinline__ f2 rcp_of(float b, float s, f2 vn) {
  return make_float2(fast_rcp(fmaf(s, vn.x, b)), fast_rcp(fmaf(s, vn.y, b)));
}

// One tile of one problem.  tab: a SymTable in the launch parameters
// (TAB_PARAM), or NULL and the table is built in shared memory from a.ang and
// a.inflow (stored order).
template <int DIM, bool VEL, int TX, int TY, int TZ, bool TAB_PARAM, bool GATHER>
__device__ __forceinline__ void process_tile_sym(const StepArgs<float> &a, const SymTable *tab, int tid, int tbx,
                                                 int tby, int tbz, unsigned char *smem_raw) {
  using G = SymGeo<DIM, TX, TY, TZ>;
  static_assert(DIM >= 2 && (TAB_PARAM || !GATHER), "pairs: 2-D and 3-D");
  constexpr int NT = G::NT, ROUND = G::ROUND, SLOTS = G::SLOTS, NBOX = G::NBOX;
  static_assert(4 * ROUND * (NBOX + G::NF) >= 6 * NBOX, "set-up scratch fits the second buffer and Delta F");
  const int NQ = a.M / 4;
  const long long N = a.N;
  const int org[3] = {tbx * TX, tby * TY, tbz * TZ};

  __syncthreads();   // the previous tile of a persistent CTA is done with shared memory
  f2 *s_tab = reinterpret_cast<f2 *>(smem_raw);   // [NQ][kSymTab] (shared table only)
  float4 *s_I = reinterpret_cast<float4 *>(s_tab + (TAB_PARAM ? 0 : kSymQuads * kSymTab));   // I^n [2][ROUND][NBOX]
  float4 *s_F = s_I + 2 * ROUND * NBOX;                        // Delta F per axis [ROUND][NF]
  f2 *s_IV = reinterpret_cast<f2 *>(s_F + ROUND * G::NF);      // IV [ROUND][NBOX] (VEL)
  float2 *s_fc = s_IV + (VEL ? ROUND * NBOX : 0);              // face constants [NC]
  float *s_w = reinterpret_cast<float *>(s_fc + G::NC);        // w = 3 J v [3][NBOX] (VEL)
  // the lines, read again each round: their addresses would fill the registers
  PackedLine *s_line = reinterpret_cast<PackedLine *>(s_w + (VEL ? 3 * NBOX : 0));   // [LINES]
  auto tabv = [&](int q, int j) -> f2 {
    float4 x;
    if constexpr (TAB_PARAM)
      x = tab->e[q][j >> 1];
    else
      x = reinterpret_cast<const float4 *>(s_tab)[RT_IDX(kSymTab / 2 * q + (j >> 1), kSymQuads * kSymTab / 2)];
    return j & 1 ? hi2(x) : lo2(x);
  };
  auto inflow = [&](int face, int m) -> float {
    if constexpr (TAB_PARAM)
      return tab->inflow[face][m];
    else
      return a.inflow[RT_IDX(face * a.M + m, 6 * a.M)];
  };
  // a cell's quad q: of I^n in whatever order (its smallest value is all that is
  // asked of it), of I_out in stored order (GATHER: until the last write)
  auto load4 = [&](const float *I, int q, long long cell) -> float4 {
    return reinterpret_cast<const float4 *>(I)[RT_IDX((long long)q * N + cell, NQ * N)];
  };
  auto store4 = [&](float *I, int q, long long cell, float4 x) {
    reinterpret_cast<float4 *>(I)[RT_IDX((long long)q * N + cell, NQ * N)] = x;
  };

  if constexpr (!TAB_PARAM) {
    for (int q = tid; q < NQ; q += NT) {
      float q16[8];
      for (int i = 0; i < 8; ++i) q16[i] = a.ang[RT_IDX(16 * q + i, 4 * a.M)];
      sym_tab_quad(s_tab + RT_IDX(kSymTab * q, kSymQuads * kSymTab - kSymTab + 1), q16, a.C, a.dtdx);
    }
  }

  // ---- the own cell: what the implicit steps need of it in the transport loop --------
  const int lx = tid % TX, ly = (tid / TX) % TY, lz = tid / (TX * TY);
  const int gx = org[0] + lx, gy = org[1] + ly, gz = org[2] + lz;
  const bool valid = gx < a.n[0] && gy < a.n[1] && gz < a.n[2];
  const long long c = valid ? RT_IDX(gx + (long long)a.n[0] * (gy + (long long)a.n[1] * gz), N) : 0;
  float vt[3] = {0, 0, 0}, R = 0, A0 = 1, A1 = 0, a0 = 1, a1 = 0, rd0 = 0, ra0 = 0, scat = 0;
  if (valid) {
    CellIn ci;
    ci.template load<VEL>(a, c);
    for (int d = 0; d < 3; ++d) vt[d] = ci.vt[d];
    A0 = ci.A0; A1 = ci.A1; a0 = ci.a0; a1 = ci.a1;
    rd0 = ci.rd0; ra0 = ci.ra0;
    scat = ci.to_scat ? 1.0f : 0.0f;
    // the center: written by the step that produced I^n, or formed here
    if (a.cen_in) {
      R = a.cen_in[c];
    } else {
      float4 q = load4(a.I_in, 0, c);
      R = fminf(fminf(q.x, q.y), fminf(q.z, q.w));
#pragma unroll 6
      for (int j = 1; j < NQ; ++j) {
        q = load4(a.I_in, j, c);
        R = fminf(R, fminf(fminf(q.x, q.y), fminf(q.z, q.w)));
      }
    }
  }

  // ---- staged cells of this thread: the tile's, then the halo ----------------------
  // sl_box: place in shared memory, and from bit 16 on how the cell lies beyond
  // a vacuum or inflow face (0: it does not): bit 0 set, 1 inflow, 2-3 axis, 4
  // upper side.  alpha per axis and v go to scratch past the first buffer.
  int sl_box[SLOTS], sl_g[SLOTS];
  auto full = [](int s) { return (s + 1) * NT <= G::NCROSS; };
  auto used = [&](int s) { return full(s) || tid + s * NT < G::NCROSS; };
  float *c_al = reinterpret_cast<float *>(s_I + ROUND * NBOX), *c_v = c_al + 3 * NBOX;   // [3][NBOX] each
  const bool same_dx = (DIM < 2 || a.dx[1] == a.dx[0]) && (DIM < 3 || a.dx[2] == a.dx[0]);
  bool special = false;
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    sl_box[s] = sl_g[s] = 0;
    if (!used(s)) continue;
    int l[3];
    const int box = (int)RT_IDX(G::staged(tid + s * NT, l), NBOX);
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
    special |= code != 0;
    sl_box[s] = box | (code << 16);
    sl_g[s] = (int)RT_IDX(g[0] + (long long)a.n[0] * (g[1] + (long long)a.n[1] * g[2]), N);
  }
  // asynchronous copies of round j0's quads of this thread's cells into buffer b
  auto fetch = [&](int j0, int b) {
#pragma unroll
    for (int k = 0; k < ROUND; ++k) {
      if (j0 + k >= NQ) break;
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        if (!used(s)) continue;
        float4 *dst = s_I + RT_IDX((b * ROUND + k) * NBOX + (sl_box[s] & 0xffff), 2 * ROUND * NBOX);
        if constexpr (GATHER) {
          // a cell's place in a plane is a 32-bit byte offset (fewer than 2^28 cells)
          const unsigned at = 16u * (unsigned)sl_g[s];
          float *d = reinterpret_cast<float *>(dst);
          const unsigned char *m = tab->slot + 4 * (j0 + k);
          auto from = [&](int h) {
            return reinterpret_cast<const char *>(a.I_in) + 16 * (long long)(m[h] >> 2) * N + 4 * (m[h] & 3);
          };
          if (tab->pairs[j0 + k]) {
            copy_async<8>(d, RT_AT(from(0) + at, reinterpret_cast<const char *>(a.I_in), 16 * NQ * N - 7));
            copy_async<8>(d + 2, RT_AT(from(2) + at, reinterpret_cast<const char *>(a.I_in), 16 * NQ * N - 7));
          } else {
#pragma unroll
            for (int h = 0; h < 4; ++h)
              copy_async<4>(d + h, RT_AT(from(h) + at, reinterpret_cast<const char *>(a.I_in), 16 * NQ * N - 3));
          }
        } else {
          copy_async<16>(dst, reinterpret_cast<const float4 *>(a.I_in) + RT_IDX((long long)(j0 + k) * N + sl_g[s], NQ * N));
        }
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  fetch(0, 0);
  {
    // every load before the first store to shared memory: one latency
    // (in 3-D alpha comes with the context's fields: gas loop of 96 x 80 x 72 x 24
    // angles 264 -> 257 us; in 2-D, where a grid is a wave of CTAs that all wait for
    // their loads, forming it here is faster, 866 against 900 us for 20 steps of
    // 256^2 x 80: sa and ss are then in L1 when the cell's own fields are read)
    constexpr bool KEPT = DIM == 3 && !GATHER;
    float st[SLOTS], al[SLOTS][3], v[SLOTS][3];
    double E[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      if (!used(s)) continue;
      const long long cc = sl_g[s];
      if constexpr (!KEPT) {
        st[s] = a.sa[cc] + a.ss[cc];
      } else {
        al[s][0] = a.alpha[0][cc];
        if (!same_dx) {
          al[s][1] = a.alpha[1][cc];
          if (DIM == 3) al[s][2] = a.alpha[2][cc];
        }
      }
      if (VEL) {
        E[s] = a.mom_in[cc];
#pragma unroll
        for (int d = 0; d < 3; ++d) v[s][d] = a.v[d * N + cc];
      }
    }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      if (!used(s)) continue;
      const int box = sl_box[s] & 0xffff;
      c_al[RT_IDX(box, NBOX)] = KEPT ? al[s][0] : alpha_of(a.dx[0], st[s]);
      if (!same_dx) {   // cells of unequal sides: one alpha per axis
        c_al[RT_IDX(NBOX + box, 3 * NBOX)] = KEPT ? al[s][1] : alpha_of(a.dx[1], st[s]);
        if (DIM == 3) c_al[RT_IDX(2 * NBOX + box, 3 * NBOX)] = KEPT ? al[s][2] : alpha_of(a.dx[2], st[s]);
      }
      if (VEL) {
        const float w3 = float(3.0 / (4.0 * kPi)) * d2f_rn(E[s]);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (d < DIM) c_v[RT_IDX(d * NBOX + box, 3 * NBOX)] = v[s][d];
          s_w[RT_IDX(d * NBOX + box, 3 * NBOX)] = w3 * v[s][d];
        }
      }
    }
  }
  __syncthreads();

  // ---- lines and their face constants (see Walk::face): alpha is the mean of the two
  // cells', the face velocity the mean of theirs -------------------------------------
  if (tid < G::LINES) {
    Line ln{};
    const int d = G::line(tid, ln), L = d == 0 ? G::LX : d == 1 ? G::LY : G::LZ;
    s_line[RT_IDX(tid, G::LINES)].pack(ln);
    const int np = d == 0 ? G::NPX : d == 1 ? G::NPY : G::NPZ;
    float2 *fc = s_fc + (d == 0 ? tid : d == 1 ? G::CY + tid - G::NPX : G::CZ + tid - G::NPX - G::NPY);
    const float *l_al = c_al + (same_dx ? 0 : d * NBOX), *l_v = c_v + d * NBOX;
    const float dtdx = d == 0 ? a.dtdx[0] : d == 1 ? a.dtdx[1] : a.dtdx[2];
    int at = (int)RT_IDX(ln.lo + ln.slo, NBOX);   // the cell below the face
    float al = l_al[at], v = VEL ? l_v[at] : 0.0f;
    for (int f = 0; f <= L; ++f) {
      at = (int)RT_IDX(f < L ? ln.core + f * ln.sc : ln.hi, NBOX);
      const float al1 = l_al[at];
      float2 k = make_float2(0.5f * (al + al1), 0.0f);
      if (VEL) {
        const float v1 = l_v[at], vf = 0.5f * (v + v1);
        const float h = 1.0f - fabsf(vf) * dtdx;
        if (vf > 0.0f) k = make_float2(-k.x, h);
        else k.y = vf < 0.0f ? -h : __int_as_float(0x7f800000);
        special |= vf == 0.0f;
        v = v1;
      }
      *RT_AT(fc + f * np, s_fc, G::NC) = k;
      al = al1;
    }
  }
  // A tile with no staged cell beyond a vacuum or inflow face and no face of
  // exactly zero velocity skips those two cases (one vote per tile; the warp
  // vote lets the compiler see a warp-uniform choice).
  const bool general = __any_sync(0xffffffffu, __syncthreads_or(special) != 0);

  // ---- transport: Delta F_m of every quad, ROUND quads per two barriers -------------
  // This thread's line: of the quad in place kq.  The quads of a round hand
  // their lines out rotated, so that the long lines of one share a scheduler
  // with the short lines of the next.
  const int kq = tid / G::LINES;
  const int line = ROUND % 2 == 0 && (kq & 1) ? (tid + G::LINES / 2) % G::LINES : tid % G::LINES;
  const int axis = line < G::NPX ? 0 : DIM == 2 || line < G::NPX + G::NPY ? 1 : 2;
  // Sums over the pairs (p: n, n'; m: -n, -n') with e = f(vn) + f(-vn), o =
  // f(vn) - f(-vn): sum W vn^k f = sum of W vn^k (e for even k, o for odd k).
  // T_k: f = rd; A_k: f = ra; D_k: f = ra rd; U_k: f = rd rr; K_k: f = ra Q; pre =
  // sum W n (I^n + Delta F - R).  The beta-weighted sums of Step 5 (beta = bt0 +
  // bt1 vn + bt2 vn^2) are combinations of these.
  f2 U0 = dup(0.0f), U1 = dup(0.0f), U2 = dup(0.0f), K0 = dup(0.0f), K1 = dup(0.0f), K2 = dup(0.0f);
  f2 pre0 = dup(0.0f), pre1 = dup(0.0f), pre2 = dup(0.0f);
  int b = 0;
#pragma unroll 1
  for (int j0 = 0; j0 < NQ; j0 += ROUND, b ^= 1) {
    // the round's copies are this thread's own: complete before it patches
    // them and before the barrier publishes them
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (VEL || general) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s) {
        if (!used(s)) continue;
        const int box = sl_box[s] & 0xffff, code = sl_box[s] >> 16;
        f2 w0, w1, w2;
        if (VEL) {
          w0 = dup(s_w[RT_IDX(box, 3 * NBOX)]);
          w1 = dup(s_w[RT_IDX(NBOX + box, 3 * NBOX)]);
          w2 = dup(s_w[RT_IDX(2 * NBOX + box, 3 * NBOX)]);
        }
#pragma unroll
        for (int k = 0; k < ROUND; ++k) {
          const int j = j0 + k;
          if (j >= NQ) break;
          if (VEL)
            s_IV[RT_IDX(k * NBOX + box, ROUND * NBOX)] = p_fma(tabv(j, kSymN + 2), w2, p_fma(tabv(j, kSymN), w0, p_mul(tabv(j, kSymN + 1), w1)));
          if (general && code) {
            // beyond a vacuum or inflow face, the rays that come in: n with mu >
            // 0 through a lower face, mu < 0 through an upper one
            const int ax = (code >> 2) & 3, side = (code >> 4) & 1, face = ax * 2 + side;
            const f2 mu = tabv(j, kSymN + ax);
            const bool infl = (code & 2) != 0;
            float4 *x = s_I + RT_IDX((b * ROUND + k) * NBOX + box, 2 * ROUND * NBOX);
            if (side ? (mu.x < 0.0f) : (mu.x > 0.0f)) x->x = infl ? inflow(face, 4 * j) : 0.0f;
            if (side ? (mu.y < 0.0f) : (mu.y > 0.0f)) x->y = infl ? inflow(face, 4 * j + 1) : 0.0f;
            if (side ? (mu.x > 0.0f) : (mu.x < 0.0f)) x->z = infl ? inflow(face, 4 * j + 2) : 0.0f;
            if (side ? (mu.y > 0.0f) : (mu.y < 0.0f)) x->w = infl ? inflow(face, 4 * j + 3) : 0.0f;
          }
        }
      }
    }
    __syncthreads();
    if (j0 + ROUND < NQ) fetch(j0 + ROUND, b ^ 1);   // its last readers passed the barrier before
    if (kq < ROUND && j0 + kq < NQ) {
      const float4 *In = s_I + (b * ROUND + kq) * NBOX;
      const f2 *IV = s_IV + (VEL ? kq * NBOX : 0);
      float4 *F = s_F + kq * G::NF;
      const f2 hc = tabv(j0 + kq, kSymHc + 2 * axis), mud = tabv(j0 + kq, kSymHc + 2 * axis + 1);
      const f2 hca = make_float2(fabsf(hc.x), fabsf(hc.y));
      const Line at = s_line[RT_IDX(line, G::LINES)].unpack();
      // a walk of L cells; np lines of its kind, F's step sf
      auto walk = [&](auto length, auto gen, auto lines, auto step, float4 *Fl, const float2 *fc) {
        constexpr int L = decltype(length)::value, NP = decltype(lines)::value, SF = decltype(step)::value;
        auto cell = [&](const float4 *x, const f2 *v, f2 *iv) {   // I~ = I - IV/C, IV
          *iv = VEL ? *v : dup(0.0f);
          return VEL ? mk4(p_fma(*iv, dup(-a.invC), lo2(*x)), p_fma(*iv, dup(a.invC), hi2(*x))) : *x;
        };
        Walk<VEL, decltype(gen)::value> w;
        f2 va, vb, vc;
        const float4 ca = cell(In + RT_IDX(at.lo, NBOX), IV + RT_IDX(at.lo, NBOX), &va);
        const float4 cb = cell(In + RT_IDX(at.lo + at.slo, NBOX), IV + RT_IDX(at.lo + at.slo, NBOX), &vb);
        const float4 *x = In + RT_IDX(at.core, NBOX);
        const f2 *v = IV + RT_IDX(at.core, NBOX);
        w.start(ca, cb, cell(x, v, &vc), va, vb, vc);
        w.fp = w.fn = dup(0.0f);
#pragma unroll
        for (int f = 0; f <= L; ++f) {
          // the cell after the one above the face
          if (f + 1 < L) {
            x += at.sc;
            v += at.sc;
          } else if (f + 1 == L) {
            x = In + at.hi;
            v = IV + at.hi;
          } else {
            x += at.shi;
            v += at.shi;
          }
          x = RT_AT(x, In, NBOX);
          if (VEL) v = RT_AT(v, IV, NBOX);
          f2 iv;
          const float4 xt = cell(x, v, &iv);
          const float4 dF = w.face(xt, iv, hc, hca, mud, *RT_AT(fc + f * NP, static_cast<const float2 *>(s_fc), G::NC));
          if (f > 0) *RT_AT(Fl + (f - 1) * SF, F, G::NF) = dF;
        }
      };
      // one copy of the code per kind of line and for tiles with the two
      // special cases: x and y lines, and shorter ones
      auto walk_any = [&](auto gen) {
        const bool y = axis == 1;
        float4 *Fl = F + (y ? G::FY + line - G::NPX : line);
        const float2 *fc = s_fc + (y ? G::CY + line - G::NPX : line);
        if (DIM == 3 && axis == 2) {
          if constexpr (DIM == 3)
            walk(IntTag<G::LZ>{}, gen, IntTag<G::NPZ>{}, IntTag<G::SZ>{}, F + G::FZ + line - G::NPX - G::NPY,
                 s_fc + G::CZ + line - G::NPX - G::NPY);
        } else if (G::LX == G::LY || !y) {
          walk(IntTag<G::LX>{}, gen, IntTag<G::NPX>{}, IntTag<G::SX>{}, Fl, fc);
        } else {
          walk(IntTag<G::LY>{}, gen, IntTag<G::NPY>{}, IntTag<G::SY>{}, Fl, fc);
        }
      };
      if (general)
        walk_any(BoolTag<true>{});
      else
        walk_any(BoolTag<false>{});
    }
    __syncthreads();
    if (!valid) continue;
    // ---- Q_m of the round and the sums of the intensity ------------------------------
    const f2 sc = dup(scat), nsc = dup(1.0f - scat), Rv = dup(R);
#pragma unroll
    for (int k = 0; k < ROUND; ++k) {
      const int j = j0 + k;
      if (j >= NQ) break;
      const float4 *F = s_F + k * G::NF;
      const float4 i4 = s_I[RT_IDX((b * ROUND + k) * NBOX + lx + kHalo + G::RX * (ly + TY * lz), 2 * ROUND * NBOX)];
      const float4 fx = F[RT_IDX(G::part_x(lx, ly, lz), G::NF)], fy = F[RT_IDX(G::part_y(lx, ly, lz), G::NF)];
      f2 dFp = p_add(lo2(fx), lo2(fy)), dFm = p_add(hi2(fx), hi2(fy));
      if (DIM == 3) {
        const float4 fz = F[RT_IDX(G::part_z(lx, ly, lz), G::NF)];
        dFp = p_add(dFp, lo2(fz));
        dFm = p_add(dFm, hi2(fz));
      }
      const f2 W = tabv(j, kSymW);
      f2 rdp = dup(rd0), rdm = dup(rd0), rap = dup(ra0), ram = dup(ra0), vn = dup(0.0f);
      if (VEL) {
        vn = vn_of(vt, tabv(j, kSymN), tabv(j, kSymN + 1), tabv(j, kSymN + 2));
        rdp = rcp_of(A0, -A1, vn);
        rdm = rcp_of(A0, A1, vn);
        rap = rcp_of(a0, -a1, vn);
        ram = rcp_of(a0, a1, vn);
      }
      const f2 gp = p_sub(lo2(i4), Rv), gm = p_sub(hi2(i4), Rv);
      const f2 up = p_mul(rdp, p_fma(nsc, dFp, gp)), um = p_mul(rdm, p_fma(nsc, dFm, gm));   // rd rr
      const f2 Qp = p_fma(sc, dFp, up), Qm = p_fma(sc, dFm, um);
      store4(a.I_out, j, c, mk4(Qp, Qm));
      const f2 zp = p_mul(rap, Qp), zm = p_mul(ram, Qm);
      const f2 ue = p_add(up, um), ze = p_add(zp, zm);
      U0 = p_fma(W, ue, U0);
      K0 = p_fma(W, ze, K0);
      if (VEL) {
        const f2 y1 = p_mul(W, vn), y2 = p_mul(y1, vn);
        U1 = p_fma(y1, p_sub(up, um), U1);
        U2 = p_fma(y2, ue, U2);
        K1 = p_fma(y1, p_sub(zp, zm), K1);
        K2 = p_fma(y2, ze, K2);
      }
      const f2 go = p_sub(p_add(gp, dFp), p_add(gm, dFm));   // (I^n + Delta F) of n minus of -n
      pre0 = p_fma(tabv(j, kSymWn), go, pre0);
      pre1 = p_fma(tabv(j, kSymWn + 1), go, pre1);
      pre2 = p_fma(tabv(j, kSymWn + 2), go, pre2);
    }
  }
  // GATHER: I^{n+1} of the tile, in the caller's order of the angles, over the
  // staging arrays: the writes to global memory are whole float4s
  float4 *s_out = reinterpret_cast<float4 *>(smem_raw);   // [NQ][NT]
  if constexpr (GATHER) __syncthreads();
  if (!valid) return;

  // ---- sums that do not depend on the intensity, per-cell solves ----------------------
  const float wn = a.wnorm;
  auto hsum = [wn](f2 x) {
    const float t = x.x + x.y;
    return fmaf(-t, wn, t);
  };
  CellSums s;
  s.U0 = hsum(U0); s.U1 = hsum(U1); s.U2 = hsum(U2);
  const float q0 = hsum(K0), q1 = hsum(K1), q2 = hsum(K2);
  CellIn ci{};
  ci.template reload<VEL>(a, c, vt, R);   // the cell's fields again: cheaper than registers through the rounds
  float4 Qa = load4(a.I_out, 0, c), Qb = load4(a.I_out, NQ > 1 ? 1 : 0, c);   // the final loop's first two quads
  f2 T0p = dup(0.0f), T1p = dup(0.0f), T2p = dup(0.0f), T3p = dup(0.0f);
  f2 P0 = dup(0.0f), P1 = dup(0.0f), P2 = dup(0.0f), P3 = dup(0.0f);
  f2 D0 = dup(0.0f), D1 = dup(0.0f), D2 = dup(0.0f), D3 = dup(0.0f);
#pragma unroll 2
  for (int j = 0; j < NQ; ++j) {
    const f2 W = tabv(j, kSymW);
    f2 rdp = dup(rd0), rdm = dup(rd0), rap = dup(ra0), ram = dup(ra0), vn = dup(0.0f);
    if (VEL) {
      vn = vn_of(vt, tabv(j, kSymN), tabv(j, kSymN + 1), tabv(j, kSymN + 2));
      rdp = rcp_of(A0, -A1, vn);
      rdm = rcp_of(A0, A1, vn);
      rap = rcp_of(a0, -a1, vn);
      ram = rcp_of(a0, a1, vn);
    }
    const f2 pp = p_mul(rap, rdp), pm = p_mul(ram, rdm);
    const f2 te = p_add(rdp, rdm), ae = p_add(rap, ram), de = p_add(pp, pm);
    T0p = p_fma(W, te, T0p);
    P0 = p_fma(W, ae, P0);
    D0 = p_fma(W, de, D0);
    if (VEL) {
      const f2 y1 = p_mul(W, vn), y2 = p_mul(y1, vn), y3 = p_mul(y2, vn);
      const f2 to = p_sub(rdp, rdm), ao = p_sub(rap, ram), od = p_sub(pp, pm);
      T1p = p_fma(y1, to, T1p);
      T2p = p_fma(y2, te, T2p);
      T3p = p_fma(y3, to, T3p);
      P1 = p_fma(y1, ao, P1);
      P2 = p_fma(y2, ae, P2);
      P3 = p_fma(y3, ao, P3);
      D1 = p_fma(y1, od, D1);
      D2 = p_fma(y2, de, D2);
      D3 = p_fma(y3, od, D3);
    }
  }
  {
    s.T0 = hsum(T0p); s.T1 = hsum(T1p); s.T2 = hsum(T2p); s.T3 = hsum(T3p);
    const float k0 = hsum(P0), k1 = hsum(P1), k2 = hsum(P2), k3 = hsum(P3);
    const float d0 = hsum(D0), d1 = hsum(D1), d2 = hsum(D2), d3 = hsum(D3);
    const float b0 = ci.bt0, b1 = ci.bt1, b2 = ci.bt2;
    s.As1 = k0; s.Va = k1; s.Ad = d0; s.Adv = d1; s.AQ = q0;
    s.Bs = fmaf(b2, k2, fmaf(b1, k1, b0 * k0));
    s.Bv = fmaf(b2, k3, fmaf(b1, k2, b0 * k1));
    s.Bd = fmaf(b2, d2, fmaf(b1, d1, b0 * d0));
    s.Bdv = fmaf(b2, d3, fmaf(b1, d2, b0 * d1));
    s.BQ = fmaf(b2, q2, fmaf(b1, q1, b0 * q0));
  }
  const CellSolve x = solve_cell(a, ci, s);

  // ---- I^{n+1} over Q_m, quadrature (sec. 3) -----------------------------------------
  f2 mE = dup(0.0f), mF[3], mP[6];
  for (int i = 0; i < 3; ++i) mF[i] = dup(0.0f);
  for (int i = 0; i < 6; ++i) mP[i] = dup(0.0f);
  float cnext = __int_as_float(0x7f800000);   // the center of I^{n+1}: its smallest angle
  {
    const f2 Rv = dup(R), e2 = dup(x.e2);
#pragma unroll 2
    for (int j = 0; j < NQ; ++j) {
      const float4 cur = Qa;
      Qa = Qb;
      if (j + 2 < NQ) Qb = load4(a.I_out, j + 2, c);   // two quads ahead
      f2 rdp = dup(rd0), rdm = dup(rd0), rap = dup(ra0), ram = dup(ra0);
      f2 yp = dup(x.D0), ym = dup(x.D0), ep = dup(x.E0), em = dup(x.E0);
      if (VEL) {
        const f2 vn = vn_of(vt, tabv(j, kSymN), tabv(j, kSymN + 1), tabv(j, kSymN + 2));
        rdp = rcp_of(A0, -A1, vn);
        rdm = rcp_of(A0, A1, vn);
        rap = rcp_of(a0, -a1, vn);
        ram = rcp_of(a0, a1, vn);
        yp = make_float2(fmaf(x.D1, vn.x, x.D0), fmaf(x.D1, vn.y, x.D0));
        ym = make_float2(fmaf(-x.D1, vn.x, x.D0), fmaf(-x.D1, vn.y, x.D0));
        ep = make_float2(fmaf(x.E1, vn.x, x.E0), fmaf(x.E1, vn.y, x.E0));
        em = make_float2(fmaf(-x.E1, vn.x, x.E0), fmaf(-x.E1, vn.y, x.E0));
      }
      const f2 zp = p_add(p_fma(rdp, yp, lo2(cur)), ep), zm = p_add(p_fma(rdm, ym, hi2(cur)), em);
      const f2 Ip = p_add(Rv, p_fma(rap, zp, e2)), Im = p_add(Rv, p_fma(ram, zm, e2));
      if constexpr (GATHER) {
        float *out = reinterpret_cast<float *>(s_out + tid);
        auto put = [&](int h, float x) {
          const int m = tab->slot[4 * j + h];
          out[RT_IDX((m >> 2) * 4 * NT + (m & 3), 4 * (NQ * NT - tid))] = x;
        };
        put(0, Ip.x);
        put(1, Ip.y);
        put(2, Im.x);
        put(3, Im.y);
      } else {
        store4(a.I_out, j, c, mk4(Ip, Im));
      }
      cnext = fminf(cnext, fminf(fminf(Ip.x, Ip.y), fminf(Im.x, Im.y)));
      const f2 dp = p_sub(Ip, Rv), dm = p_sub(Im, Rv);   // the stored values' deviations (exact)
      const f2 ev = p_add(dp, dm), od = p_sub(dp, dm);
      mE = p_fma(tabv(j, kSymW), ev, mE);
#pragma unroll
      for (int i = 0; i < 3; ++i) mF[i] = p_fma(tabv(j, kSymWn + i), od, mF[i]);
#pragma unroll
      for (int i = 0; i < 6; ++i) mP[i] = p_fma(tabv(j, kSymWnn + i), ev, mP[i]);
    }
  }
  if constexpr (GATHER)
    for (int j = 0; j < NQ; ++j) store4(a.I_out, j, c, s_out[RT_IDX(j * NT + tid, NQ * NT)]);
  store_cell(a, ci, x, c, mE, mF, mP, pre0, pre1, pre2, cnext);
}

template <int DIM, bool VEL, int TX, int TY, int TZ>
__global__ void __launch_bounds__(TX * TY * TZ, kQMinBlocks<TX * TY * TZ>)
    step_kernel_sym(const StepArgs<float> a, const __grid_constant__ SymTable tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int o = a.outer_begin;
  process_tile_sym<DIM, VEL, TX, TY, TZ, true, false>(a, &tab, threadIdx.x, blockIdx.x, blockIdx.y + (DIM == 2 ? o : 0),
                                                      blockIdx.z + (DIM == 3 ? o : 0), smem_raw);
}

template <int DIM, bool VEL, int TX, int TY, int TZ>
cudaError_t launch_shape_sym(const StepArgs<float> &a, const SymTable &tab, cudaStream_t s) {
  constexpr size_t sm = smem_bytes_sym_t<DIM, VEL, TX, TY, TZ>(true);
  static_assert(sm <= 227 * 1024, "tile exceeds the shared memory of a CTA");
  auto kern = step_kernel_sym<DIM, VEL, TX, TY, TZ>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid((a.n[0] + TX - 1) / TX, (a.n[1] + TY - 1) / TY, (a.n[2] + TZ - 1) / TZ);
  if (a.outer_count > 0) (DIM == 3 ? grid.z : grid.y) = a.outer_count;
  kern<<<grid, TX * TY * TZ, sm, s>>>(a, tab);
  return cudaGetLastError();
}

}  // namespace stepk

}  // namespace rtg
