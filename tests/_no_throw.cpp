// rt_set_inflow, rt_save_state and rt_load_state with every operator new failing: they
// have no host memory to ask for, and no C++ exception may leave a C entry point.
// Built and run on a GPU by tests/test_gpu_no_throw.py; prints OK.
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "rt.h"

static bool fail_new = false;
static int failed = 0;

void *operator new(std::size_t n) {
  if (fail_new) {
    ++failed;
    throw std::bad_alloc();
  }
  if (void *p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }

template <class Call>
static int guarded(const char *name, Call call) {
  fail_new = true;
  int status = 100;
  try {
    status = call();
  } catch (...) {
  }
  fail_new = false;
  if (status != RT_OK) std::printf("%s: %s\n", name, status == 100 ? "threw" : rt_last_error());
  return status == RT_OK ? 0 : 1;
}

int main() {
  rt_grid g{};
  g.dim = 2;
  for (int d = 0; d < 3; ++d) {
    g.n[d] = d < 2 ? 6 : 1;
    g.hi[d] = 1.0;
  }
  g.bc[0][0] = RT_BC_INFLOW;
  g.bc[0][1] = RT_BC_VACUUM;
  double n[3 * 24], w[24];
  rt_angles ang{};
  if (rt_angle_set(RT_ANGLES_LEVEL_SYMMETRIC, 4, 24, &ang.m, n, w) != RT_OK) return 2;
  ang.n = n;
  ang.w = w;
  rt_options o;
  rt_options_default(&o);
  int bad = 0;
  for (int precision : {RT_FP64, RT_FP32}) {
    o.precision = precision;
    rt_ctx *c = nullptr;
    if (rt_create(&g, &ang, 10.0, 1.0, &o, &c) != RT_OK) return 2;
    std::vector<double> one(36, 1.0), v(108, 0.0), in(24, 0.5);
    if (rt_set_material(c, one.data(), one.data(), v.data(), one.data(), one.data()) != RT_OK) return 2;
    std::vector<unsigned char> state(rt_state_bytes(c));
    bad += guarded("rt_set_inflow", [&] { return rt_set_inflow(c, 0, 0, in.data()); });
    bad += guarded("rt_save_state", [&] { return rt_save_state(c, state.data(), state.size()); });
    bad += guarded("rt_load_state", [&] { return rt_load_state(c, state.data(), state.size()); });
    rt_destroy(c);
  }
  if (bad == 0) std::printf("OK\n");
  return bad;
}
