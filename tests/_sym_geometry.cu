// Host-side check of the tile geometry (SymGeo in rt_step_sym.cuh) of the pair
// and the double kernel, for every compiled tile shape.  Built and run by
// tests/test_sym_geometry.py; prints OK when every check holds.
//  - the staged cells are the cross-shaped halo, each once, at places of
//    shared memory of their own;
//  - every position -2 .. L + 1 of every line reads the place of the staged
//    cell that line_cell names, one step along the line's axis apart;
//  - the lines of an axis cover each cell once, and its part of Delta F lies
//    where the thread that adds the parts up looks for it;
//  - face constants have places of their own in [0, NC);
//  - the inner staged cells (inner) are the tile and its first halo layers.
#include <cstdio>
#include <map>
#include <vector>

#include "rt_step_sym.cuh"

using namespace rtg::stepk;

static int failures = 0;
#define CHECK(c)                                                                                        \
  do {                                                                                                  \
    if (!(c)) {                                                                                         \
      std::printf("failed: %s (line %d, shape %d:%dx%dx%d)\n", #c, __LINE__, DIM, TX, TY, TZ); \
      ++failures;                                                                                       \
    }                                                                                                   \
  } while (0)

template <int DIM, int TX, int TY, int TZ, int LMAX = 8>
void check() {
  using G = SymGeo<DIM, TX, TY, TZ, LMAX>;
  auto key = [](const int l[3]) { return (l[0] + 100) + 1000 * ((l[1] + 100) + 1000 * (l[2] + 100)); };
  const int T[3] = {TX, TY, TZ};
  std::map<int, int> place;
  std::vector<int> box(G::NBOX, 0);
  for (int k = 0; k < G::NCROSS; ++k) {
    int l[3];
    const int b = G::staged(k, l);
    CHECK(b >= 0 && b < G::NBOX && box[b]++ == 0);
    int out = 0;
    for (int d = 0; d < 3; ++d) {
      if (l[d] < 0 || l[d] >= T[d]) ++out;
      CHECK(l[d] >= -kHalo && l[d] < T[d] + kHalo && (d < DIM || l[d] == 0));
    }
    CHECK(out <= 1 && (out == 0) == (k < G::NT));
    CHECK(place.count(key(l)) == 0);
    place[key(l)] = b;
  }
  int inner = 0;
  std::vector<int> seen(G::NCROSS, 0);
  for (int k = 0; k < G::INNER; ++k) {
    int l[3];
    const int at = G::inner(k);
    CHECK(at >= 0 && at < G::NCROSS && seen[at]++ == 0);
    G::staged(at, l);
    bool in = true;
    for (int d = 0; d < 3; ++d) in = in && l[d] >= -1 && l[d] <= T[d];
    inner += in;
  }
  CHECK(inner == G::INNER);
  std::vector<int> F(G::NF, 0), C(G::NC, 0);
  const int np[3] = {G::NPX, G::NPY, G::NPZ}, len[3] = {G::LX, G::LY, G::LZ}, off[3] = {0, G::CY, G::CZ};
  int e = 0;
  for (int d = 0; d < DIM; ++d)
    for (int p = 0; p < np[d]; ++p, ++e) {
      Line ln{};
      CHECK(G::line(e, ln) == d);
      for (int pos = -kHalo; pos < len[d] + kHalo; ++pos) {
        int l[3];
        G::line_cell(d, p, pos, l);
        const int at = pos < 0 ? ln.lo + (pos + kHalo) * ln.slo
                       : pos < len[d] ? ln.core + pos * ln.sc : ln.hi + (pos - len[d]) * ln.shi;
        CHECK(place.count(key(l)) == 1 && place[key(l)] == at);
        if (pos >= 0 && pos < len[d]) {
          const int base[3] = {0, G::FY, G::FZ}, step[3] = {G::SX, G::SY, G::SZ};
          const int f = base[d] + pos * step[d] + p;
          const int want = d == 0 ? G::part_x(l[0], l[1], l[2])
                           : d == 1 ? G::part_y(l[0], l[1], l[2]) : G::part_z(l[0], l[1], l[2]);
          CHECK(f == want && f >= 0 && f < G::NF && F[f]++ == 0);
        }
      }
      for (int f = 0; f <= len[d]; ++f) {
        const int c = off[d] + f * np[d] + p;
        CHECK(c < G::NC && C[c]++ == 0);
      }
    }
  CHECK(e == G::LINES);
  int covered = 0;
  for (int x : F) covered += x;
  CHECK(covered == DIM * G::NT);
}

int main() {
  check<3, 8, 8, 4>();
  check<3, 16, 8, 4>();
  check<3, 8, 4, 4>();
  check<3, 4, 4, 4>();
  check<2, 32, 16, 1>();
  check<2, 16, 16, 1>();
  check<2, 16, 8, 1>();
  check<2, 8, 8, 1>();
  check<2, 8, 4, 1>();
  check<1, 256, 1, 1>();
  check<1, 128, 1, 1>();
  check<1, 64, 1, 1>();
  check<1, 32, 1, 1>();
  check<1, 32, 1, 1, 2>();
  check<3, 8, 4, 4, 4>();
  if (failures == 0) std::printf("OK\n");
  return failures == 0 ? 0 : 1;
}
