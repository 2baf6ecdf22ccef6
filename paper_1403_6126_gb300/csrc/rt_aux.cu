// Elementwise device helpers of the runtime: precision conversion, the
// isotropic equilibrium intensity, the sec. 3 quadrature of a given field,
// and input scans.  All grid-stride, sized as a multiple of the SM count.
#include <cuda_bf16.h>
#include <algorithm>
#include <math.h>

#include "rt_aux.cuh"

namespace rtg {

namespace {

constexpr double kPi = 3.14159265358979323846;

template <typename Real>
__global__ void convert_in_kernel(const double *__restrict__ src, Real *__restrict__ dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = (Real)src[i];
}

template <typename Real>
__global__ void isotropic_kernel(const double *__restrict__ T, Real *__restrict__ I, int M, long long N) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    double t = T[c];
    Real b = (Real)(t * t * t * t / (4.0 * kPi));
    for (int m = 0; m < M; ++m) I[(long long)m * N + c] = b;
  }
}

// The same in the quad-interleaved float layout: one float4 per cell and
// quad, angles past M zero.
__global__ void isotropic_quad_kernel(const double *__restrict__ T, float4 *__restrict__ I, int M, long long N) {
  const int NQ = (M + 3) / 4;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    const double t = T[c];
    const float b = (float)(t * t * t * t / (4.0 * kPi));
    for (int q = 0; q < NQ; ++q) {
      const int m = 4 * q;
      I[(long long)q * N + c] = make_float4(b, m + 1 < M ? b : 0.0f, m + 2 < M ? b : 0.0f, m + 3 < M ? b : 0.0f);
    }
  }
}

// Angle-major doubles, elements [off, off + n) (element i: angle i / N of
// cell i % N), into the quad layout (angle m of cell c at float (s/4) 4N + 4c
// + s%4, s = map.slot[m]), and back.
__global__ void quad_in_kernel(const double *__restrict__ src, float *__restrict__ dst, long long off, long long n,
                               long long N, const AngleMap map) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long g = off + i, m = g / N, c = g - m * N, k = map.slot[m];
    dst[(k >> 2) * 4 * N + 4 * c + (k & 3)] = (float)src[i];
  }
}

__global__ void quad_out_kernel(const float *__restrict__ src, double *__restrict__ dst, long long off, long long n,
                                long long N, const AngleMap map) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long g = off + i, m = g / N, c = g - m * N, k = map.slot[m];
    dst[i] = (double)src[(k >> 2) * 4 * N + 4 * c + (k & 3)];
  }
}

// Exact conversion by moving the fields of the bit pattern: the hardware's float to
// double conversion runs at the FP64 rate.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) return (double)x;   // zero, subnormal, infinite, NaN
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// Every angle of every cell to the caller's [M][N], blockIdx.y = stored quad.
// Bound by memory: one float4 read and four coalesced doubles written per cell
// and quad.  Eight steps of 128^3 x 80 with their read-out 10.98 ms, where an element at a
// time into the staging buffer and a copy from there made it 11.70.
__global__ void intensity_out_kernel(const float4 *__restrict__ I, double *__restrict__ dst, int M, long long N,
                                     const AngleMap order) {
  const int q = blockIdx.y, left = M - 4 * q;
  const float4 *src = I + q * N;
  double *out[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) out[h] = dst + (h < left ? order.slot[4 * q + h] : 0) * N;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    const float4 x = __ldcs(src + c);
    __stcs(out[0] + c, widen(x.x));
    if (left > 1) __stcs(out[1] + c, widen(x.y));
    if (left > 2) __stcs(out[2] + c, widen(x.z));
    if (left > 3) __stcs(out[3] + c, widen(x.w));
  }
}

// Three arrays of doubles to the caller's, blockIdx.y = which.
__global__ void fields_out_kernel(const FieldsOut f) {
  const double *src = blockIdx.y == 0 ? f.src[0] : blockIdx.y == 1 ? f.src[1] : f.src[2];
  double *dst = blockIdx.y == 0 ? f.dst[0] : blockIdx.y == 1 ? f.dst[1] : f.dst[2];
  const long long n = blockIdx.y == 0 ? f.n[0] : blockIdx.y == 1 ? f.n[1] : f.n[2];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

// Quad-interleaved intensities of one order of the angles into another: angle m of
// the result is angle from.slot[m] of src (a multiple of four angles).  Bound by
// memory: float4s in and out, each cell's words exchanged in shared memory
// ([M/4][threads], a thread's own column).
__global__ void reorder_kernel(const float4 *__restrict__ src, float4 *__restrict__ dst, int M, long long N,
                               const AngleMap from) {
  extern __shared__ float4 s_q[];
  const int NT = blockDim.x, tid = threadIdx.x, NQ = M / 4;
  const float *s = reinterpret_cast<const float *>(s_q);
  for (long long c = blockIdx.x * (long long)NT + tid; c < N; c += (long long)gridDim.x * NT) {
#pragma unroll 4
    for (int q = 0; q < NQ; ++q) s_q[q * NT + tid] = src[q * N + c];
    for (int q = 0; q < NQ; ++q) {
      float v[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int k = from.slot[4 * q + h];
        v[h] = s[4 * ((k >> 2) * NT + tid) + (k & 3)];
      }
      dst[q * N + c] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// bf16 storage: delta = I / J - 1 with J = E / (4 pi) of the cell (the same
// arithmetic as the step kernel's b16_* helpers in rt_step_pair.cuh).
constexpr float kInv4PiF = float(1.0 / (4.0 * 3.14159265358979323846));

__global__ void encode_b16_kernel(const float *__restrict__ I, const double *__restrict__ E,
                                  unsigned short *__restrict__ out, int M, long long N) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    const float J = (float)E[c] * kInv4PiF;
    const float rJ = J > 1e-30f ? 1.0f / J : 0.0f;
    for (int m = 0; m < M; ++m) {
      const long long i = (long long)m * N + c;
      out[i] = __bfloat16_as_ushort(__float2bfloat16_rn(fmaf(I[i], rJ, -1.0f)));
    }
  }
}

__global__ void decode_b16_kernel(const unsigned short *__restrict__ in, const double *__restrict__ E,
                                  double *__restrict__ out, long long off, long long n, long long N) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long g = off + i;
    const float J = (float)E[g % N] * kInv4PiF;
    out[i] = (double)fmaf(J, __bfloat162float(__ushort_as_bfloat16(in[g])), J);
  }
}

// E = 4 pi sum W I, F = 4 pi sum W n I, P = 4 pi sum W n n I, accumulated
// in double whatever the storage type.
template <typename Real>
__global__ void moments_kernel(const Real *__restrict__ I, const Real *__restrict__ ang, int M, long long N,
                               double *__restrict__ mom) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int m = 0; m < M; ++m) {
      double nx = ang[4 * m], ny = ang[4 * m + 1], nz = ang[4 * m + 2];
      double wi = (double)ang[4 * m + 3] * (double)I[(long long)m * N + c];
      s[0] += wi;
      s[1] += nx * wi; s[2] += ny * wi; s[3] += nz * wi;
      s[4] += nx * nx * wi; s[5] += ny * ny * wi; s[6] += nz * nz * wi;
      s[7] += nx * ny * wi; s[8] += nx * nz * wi; s[9] += ny * nz * wi;
    }
    for (int q = 0; q < 10; ++q) mom[(long long)q * N + c] = 4.0 * kPi * s[q];
  }
}

// Float intensities (angle-major, or the quad layout when QUAD): products
// in float and each of the ten sums compensated (Kahan), read out as the
// double hi - lo times wscale (1 / sum W for the quad layout's kernels,
// whose sums are over the normalised weights; 1 otherwise).  In double this kernel would run at the FP64 rate (~20 FP64
// operations per cell-angle: milliseconds for a 128^3 x 80 field).
template <bool QUAD>
__global__ void moments_kernel_f(const float *__restrict__ I, const float *__restrict__ ang, int M, long long N,
                                 double wscale, double *__restrict__ mom) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    float hi[10], lo[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) hi[q] = lo[q] = 0.0f;
    for (int m = 0; m < M; ++m) {
      const float nx = ang[4 * m], ny = ang[4 * m + 1], nz = ang[4 * m + 2];
      const float Im = QUAD ? I[(long long)(m >> 2) * 4 * N + 4 * c + (m & 3)] : I[(long long)m * N + c];
      const float wi = ang[4 * m + 3] * Im;
      const float wx = nx * wi, wy = ny * wi, wz = nz * wi;
      const float term[10] = {wi, wx, wy, wz, nx * wx, ny * wy, nz * wz, ny * wx, nz * wx, nz * wy};
#pragma unroll
      for (int q = 0; q < 10; ++q) {
        const float y = term[q] - lo[q];
        const float s = hi[q] + y;
        lo[q] = (s - hi[q]) - y;
        hi[q] = s;
      }
    }
#pragma unroll
    for (int q = 0; q < 10; ++q) mom[(long long)q * N + c] = 4.0 * kPi * wscale * ((double)hi[q] - (double)lo[q]);
  }
}

// The smallest intensity of each cell over its M angles (quad layout,
// padding angles excluded): the center the float step's deviations are
// taken from.
__global__ void centers_kernel(const float4 *__restrict__ I, int M, long long N, float *__restrict__ cen) {
  const int NQ = (M + 3) / 4;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    float mn = I[c].x;
    for (int j = 0; j < NQ; ++j) {
      const float4 q = I[(long long)j * N + c];
      const int left = M - 4 * j;
      mn = fminf(mn, q.x);
      if (left > 1) mn = fminf(mn, q.y);
      if (left > 2) mn = fminf(mn, q.z);
      if (left > 3) mn = fminf(mn, q.w);
    }
    cen[c] = mn;
  }
}

// f = P / E of each cell (sec. 2: f = K/J), one double reciprocal per cell.
__global__ void eddington_kernel(const double *__restrict__ mom, double *__restrict__ f, long long N) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
    const double E = mom[c];
    const double rE = E != 0.0 ? 1.0 / E : 0.0;
#pragma unroll
    for (int q = 0; q < 6; ++q) f[(long long)q * N + c] = mom[(long long)(4 + q) * N + c] * rE;
  }
}

__global__ void check_kernel(const double *__restrict__ x, long long n, double lo, int strict, int nzbit, int *flag) {
  int bits = 0;
  const bool zero_lo = lo == 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = x[i];
    const unsigned long long u = bits_of(v);
    const bool ok = zero_lo ? (strict ? positive_bits(u) : nonneg_bits(u))
                            : (finite_bits(u) && (strict ? v > lo : v >= lo));
    if (!ok) bits |= 1;
    if ((u & kAbsMask) != 0) bits |= nzbit;
  }
  // one atomic per block: an atomic per thread on the one flag word would
  // serialize (nearly every thread sets the nonzero bit of a velocity field)
  const int bad = __syncthreads_or(bits & 1), nonzero = __syncthreads_or(bits & nzbit);
  if (threadIdx.x == 0 && (bad || nonzero)) atomicOr(flag, (bad ? 1 : 0) | (nonzero ? nzbit : 0));
}

}  // namespace

template <typename Real>
cudaError_t launch_convert_in(const double *src, Real *dst, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  convert_in_kernel<Real><<<grid_for(n, 256), 256, 0, s>>>(src, dst, n);
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_isotropic(const double *T, Real *I, int M, long long N, bool quad, cudaStream_t s) {
  if constexpr (sizeof(Real) == 4) {
    if (quad) {
      isotropic_quad_kernel<<<grid_for(N, 256), 256, 0, s>>>(T, reinterpret_cast<float4 *>(I), M, N);
      return cudaGetLastError();
    }
  }
  isotropic_kernel<Real><<<grid_for(N, 256), 256, 0, s>>>(T, I, M, N);
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_moments(const Real *I, const Real *ang, int M, long long N, bool quad, double wscale, double *mom,
                           cudaStream_t s) {
  if constexpr (sizeof(Real) == 4) {
    if (quad)
      moments_kernel_f<true><<<grid_for(N, 256), 256, 0, s>>>(I, ang, M, N, wscale, mom);
    else
      moments_kernel_f<false><<<grid_for(N, 256), 256, 0, s>>>(I, ang, M, N, wscale, mom);
  } else {
    moments_kernel<Real><<<grid_for(N, 256), 256, 0, s>>>(I, ang, M, N, mom);
  }
  return cudaGetLastError();
}

cudaError_t launch_centers(const float *I, int M, long long N, float *cen, cudaStream_t s) {
  centers_kernel<<<grid_for(N, 256), 256, 0, s>>>(reinterpret_cast<const float4 *>(I), M, N, cen);
  return cudaGetLastError();
}

cudaError_t launch_eddington(const double *mom, double *f, long long N, cudaStream_t s) {
  eddington_kernel<<<grid_for(N, 256), 256, 0, s>>>(mom, f, N);
  return cudaGetLastError();
}

cudaError_t launch_quad_in(const double *src, float *dst, long long off, long long n, long long N, const AngleMap &map,
                           cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  quad_in_kernel<<<grid_for(n, 256), 256, 0, s>>>(src, dst, off, n, N, map);
  return cudaGetLastError();
}

cudaError_t launch_quad_out(const float *src, double *dst, long long off, long long n, long long N, const AngleMap &map,
                            cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  quad_out_kernel<<<grid_for(n, 256), 256, 0, s>>>(src, dst, off, n, N, map);
  return cudaGetLastError();
}

cudaError_t launch_intensity_out(const float *src, double *dst, int M, long long N, const AngleMap &order,
                                 cudaStream_t s) {
  const dim3 grid(grid_for(N, 256), (M + 3) / 4);
  intensity_out_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<const float4 *>(src), dst, M, N, order);
  return cudaGetLastError();
}

cudaError_t launch_fields_out(const FieldsOut &f, cudaStream_t s) {
  const long long n = std::max(f.n[0], std::max(f.n[1], f.n[2]));
  if (n <= 0) return cudaSuccess;
  fields_out_kernel<<<dim3(grid_for(n, 256), 3), 256, 0, s>>>(f);
  return cudaGetLastError();
}

cudaError_t launch_reorder(const float *src, float *dst, int M, long long N, const AngleMap &from, cudaStream_t s) {
  constexpr int NT = 128;
  reorder_kernel<<<grid_for(N, NT), NT, (M / 4) * NT * sizeof(float4), s>>>(
      reinterpret_cast<const float4 *>(src), reinterpret_cast<float4 *>(dst), M, N, from);
  return cudaGetLastError();
}

cudaError_t launch_check(const double *x, long long n, double lo, int strict, int nzbit, int *flag, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  check_kernel<<<grid_for(n, 256), 256, 0, s>>>(x, n, lo, strict, nzbit, flag);
  return cudaGetLastError();
}

cudaError_t launch_encode_b16(const float *I, const double *E, unsigned short *out, int M, long long N, cudaStream_t s) {
  encode_b16_kernel<<<grid_for(N, 256), 256, 0, s>>>(I, E, out, M, N);
  return cudaGetLastError();
}

cudaError_t launch_decode_b16(const unsigned short *in, const double *E, double *out, long long off, long long n,
                              long long N, cudaStream_t s) {
  decode_b16_kernel<<<grid_for(n, 256), 256, 0, s>>>(in, E, out, off, n, N);
  return cudaGetLastError();
}

template cudaError_t launch_convert_in<float>(const double *, float *, long long, cudaStream_t);
template cudaError_t launch_convert_in<double>(const double *, double *, long long, cudaStream_t);
template cudaError_t launch_isotropic<float>(const double *, float *, int, long long, bool, cudaStream_t);
template cudaError_t launch_isotropic<double>(const double *, double *, int, long long, bool, cudaStream_t);
template cudaError_t launch_moments<float>(const float *, const float *, int, long long, bool, double, double *,
                                           cudaStream_t);
template cudaError_t launch_moments<double>(const double *, const double *, int, long long, bool, double, double *,
                                            cudaStream_t);

}  // namespace rtg
