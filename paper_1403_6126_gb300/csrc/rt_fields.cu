// The gas fields of a context: scan, conversion, and alpha of each cell.
//
// alpha is a function of the opacity and the cell side alone.  Formed in the step
// it costs an expm1, a square root and a division for every staged cell of every
// tile, up to twice per cell with the halo; written once here it costs 4 or 8 bytes
// per cell (512-cell double slab 24.6 -> 21.9 us per step, 48 x 40 x 36 x 24 double step with
// its host link 1639 -> 1577).  Compiled without implicit contraction, as the
// step kernels are: rt_step_noalloc, which has no place to keep alpha, forms
// the same bits in its kernel.
#include <math.h>

#include "rt_aux.cuh"
#include "rt_step_kernel.cuh"

namespace rtg {

namespace {

template <typename Real>
__device__ __forceinline__ void store_alpha(const CellAlpha<Real> &al, long long i, Real st) {
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (al.out[k]) al.out[k][i] = stepk::alpha_of(al.dx[k], st);
}

// Gas fields in doubles (N each; v three times N), cells [c0, c0 + n): bit 0 of *flag for a value out of
// range (rho, T > 0; sigma >= 0; all finite), bit 1 for a nonzero velocity;
// with kConvert also the context's arrays (Real, T in double) and alpha (sec. 4.1)
// of each cell for every distinct cell side dx; with kStage also a copy of
// the fields in stage, so that the caller's arrays are free once it is done.
enum FieldsMode { kScan, kConvert, kStage };

template <typename Real, int MODE>
__global__ void fields_in_kernel(const FieldSrc src, long long N, long long c0, long long n,
                                 Real *__restrict__ rho, Real *__restrict__ sa, Real *__restrict__ ss,
                                 Real *__restrict__ v, double *__restrict__ T, CellAlpha<Real> al, double *__restrict__ stage, int *flag) {
  int bits = 0;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
    const long long i = c0 + k;
    const double r = src.rho[i], t = src.T[i], vx = src.v[i], vy = src.v[N + i], vz = src.v[2 * N + i], a = src.sa[i],
                 s = src.ss[i];
    const unsigned long long ux = bits_of(vx), uy = bits_of(vy), uz = bits_of(vz);
    if (!(positive_bits(bits_of(r)) && positive_bits(bits_of(t)) && nonneg_bits(bits_of(a)) &&
          nonneg_bits(bits_of(s)) && finite_bits(ux) && finite_bits(uy) && finite_bits(uz)))
      bits |= 1;
    if (((ux | uy | uz) & kAbsMask) != 0) bits |= 2;
    if (MODE == kStage) {
      stage[i] = r;
      stage[N + i] = t;
      stage[2 * N + i] = vx;
      stage[3 * N + i] = vy;
      stage[4 * N + i] = vz;
      stage[5 * N + i] = a;
      stage[6 * N + i] = s;
    }
    if (MODE == kConvert) {
      rho[i] = (Real)r;
      sa[i] = (Real)a;
      ss[i] = (Real)s;
      v[i] = (Real)vx;
      v[N + i] = (Real)vy;
      v[2 * N + i] = (Real)vz;
      T[i] = t;
      store_alpha(al, i, (Real)a + (Real)s);
    }
  }
  const int bad = __syncthreads_or(bits & 1), nonzero = __syncthreads_or(bits & 2);
  if (threadIdx.x == 0 && (bad || nonzero)) atomicOr(flag, (bad ? 1 : 0) | (nonzero ? 2 : 0));
}

template <typename Real>
__global__ void alpha_kernel(const Real *__restrict__ sa, const Real *__restrict__ ss, long long N, CellAlpha<Real> al) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
    store_alpha(al, i, sa[i] + ss[i]);
}

}  // namespace

template <typename Real>
cudaError_t launch_fields_in(const FieldSrc &src, long long N, long long c0, long long n, bool convert, Real *rho,
                             Real *sa, Real *ss, Real *v, double *T, const CellAlpha<Real> &al, int *flag, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (convert)
    fields_in_kernel<Real, kConvert><<<grid_for(n, 256), 256, 0, s>>>(src, N, c0, n, rho, sa, ss, v, T, al, nullptr, flag);
  else
    fields_in_kernel<Real, kScan><<<grid_for(n, 256), 256, 0, s>>>(src, N, c0, n, rho, sa, ss, v, T, al, nullptr, flag);
  return cudaGetLastError();
}


template cudaError_t launch_fields_in<float>(const FieldSrc &, long long, long long, long long, bool, float *, float *,
                                             float *, float *, double *, const CellAlpha<float> &, int *,
                                             cudaStream_t);
template cudaError_t launch_fields_in<double>(const FieldSrc &, long long, long long, long long, bool, double *,
                                              double *, double *, double *, double *, const CellAlpha<double> &,
                                              int *, cudaStream_t);

cudaError_t launch_fields_stage(const FieldSrc &src, long long N, double *stage, int *flag, cudaStream_t s) {
  fields_in_kernel<double, kStage>
      <<<grid_for(N, 256), 256, 0, s>>>(src, N, 0, N, nullptr, nullptr, nullptr, nullptr, nullptr, {}, stage, flag);
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_alpha(const Real *sa, const Real *ss, long long N, const CellAlpha<Real> &al, cudaStream_t s) {
  alpha_kernel<Real><<<grid_for(N, 256), 256, 0, s>>>(sa, ss, N, al);
  return cudaGetLastError();
}

template cudaError_t launch_alpha<float>(const float *, const float *, long long, const CellAlpha<float> &, cudaStream_t);
template cudaError_t launch_alpha<double>(const double *, const double *, long long, const CellAlpha<double> &,
                                          cudaStream_t);

}  // namespace rtg
