// Reciprocal and quotient of the double kernel (rt_step_double.cuh) against CUDA's
// correctly rounded division.  Built and run on a GPU by
// tests/test_gpu_reciprocal.py; prints OK when every check holds.
//  - over every exponent of the valid range, random mantissas and those next to
//    a power of two, both signs: the first approximation is good to 2^-19, and
//    rcp_cubic within one unit in the last place of 1/x, so at most one step from
//    the rounded 1.0 / x;
//  - rcp_range is that range and no more; beyond it rcp_any and div_any are the
//    division itself.
#include <cstdio>
#include <vector>

#include "rt_step_double.cuh"

using namespace rtg::stepk;

__device__ unsigned long long mantissa(int k) {
  constexpr unsigned long long kAll = (1ull << 52) - 1;
  if (k < 8) return k;               // 1 and the next ones
  if (k < 16) return kAll - (k - 8);   // below 2
  if (k < 24) return (1ull << 51) + k - 20;   // around 1.5
  unsigned long long h = k * 0x9e3779b97f4a7c15ull;
  h = (h ^ (h >> 30)) * 0xbf58476d1ce4e5b9ull;
  h = (h ^ (h >> 27)) * 0x94d049bb133111ebull;
  return (h ^ (h >> 31)) & kAll;
}

// blockIdx.x: the exponent field 0 .. 2047; bad: counts per check.
__global__ void check(int mantissas, unsigned long long *bad) {
  const int field = blockIdx.x;
  const bool valid = field >= 1 && field <= 2044;
  for (int k = threadIdx.x; k < 2 * mantissas; k += blockDim.x) {
    const unsigned long long u = ((unsigned long long)(k & 1) << 63) | ((unsigned long long)field << 52) | mantissa(k >> 1);
    const double x = __longlong_as_double((long long)u), q = 1.0 / x, n = 1.0 + 1e-3 * (k & 1023), nx = n / x;
    auto same = [](double a, double b) {
      return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
    };
    if (rcp_range(x) != valid) atomicAdd(bad, 1ull);
    if (valid) {
      const long long d = __double_as_longlong(rcp_cubic(x)) - __double_as_longlong(q);
      if (!(fabs(fma(-x, rcp_seed(x), 1.0)) < 0x1p-19)) atomicAdd(bad + 1, 1ull);
      if (d < -1 || d > 1) atomicAdd(bad + 2, 1ull);
      if (!same(rcp_any(x), rcp_cubic(x))) atomicAdd(bad + 3, 1ull);
      // n (1/x): two more roundings, of a result that may overflow or be subnormal
      if (fabs(nx) > 0x1p-1021 && fabs(nx) < 0x1p1023 && !(fabs(div_any(n, x) - nx) <= 0x1p-51 * fabs(nx))) atomicAdd(bad + 4, 1ull);
    } else {
      if (!same(rcp_any(x), q)) atomicAdd(bad + 5, 1ull);
      if (!same(div_any(n, x), nx) || !same(div_any(0.0, x), 0.0 / x)) atomicAdd(bad + 6, 1ull);
    }
  }
}

int main() {
  constexpr int kChecks = 7;
  unsigned long long *d = nullptr, bad[kChecks] = {};
  if (cudaMalloc(&d, sizeof bad) != cudaSuccess || cudaMemset(d, 0, sizeof bad) != cudaSuccess) return 2;
  check<<<2048, 256>>>(20000, d);
  if (cudaMemcpy(bad, d, sizeof bad, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  cudaFree(d);
  bool ok = true;
  for (int i = 0; i < kChecks; ++i) {
    if (bad[i]) std::printf("check %d: %llu failures\n", i, bad[i]);
    ok = ok && bad[i] == 0;
  }
  if (ok) std::printf("OK\n");
  return ok ? 0 : 1;
}
