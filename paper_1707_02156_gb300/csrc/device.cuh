// Small device helpers shared by the kernels of the library.
#pragma once
#include <cuda_runtime.h>

namespace bie {

// The hardware estimate of 1/sqrt(v), denormals taken as zero.  rsqrtf() wraps the same estimate in a test and
// two multiplications that rescale denormal arguments, which squared distances never are: with them the FP32
// pair kernel spent an eighth of its FMA-pipe slots on the wrapping (192 drops: 42.8 -> 36.4 ms without).
__device__ __forceinline__ float rsqrt_est(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

template <typename R>
__device__ inline R rsqrt_(R v);
// FP64 powers of 1/sqrt(v) from the FP32 hardware estimate y of 1/sqrt(v): with e = 1 - v y^2 (about 2^-22,
// formed by one fused multiply-add since y^2 is exact),
//   v^(-k/2) = y^k (1 - e)^(-k/2) = y^k (1 + (k/2) e + (k/2)(k/2 + 1)/2 e^2 + O(e^3)),
// so the truncated series leaves a relative error of order e^3 (2^-64), below FP64 rounding.  The FP64 pipe is
// the bound of every kernel that calls these, and conversions and comparisons of doubles run on it too:
// the estimate's argument and result pass through the integer pipe (rebased exponent, mantissa cut to
// 23 bits), and the test for the FP32 exponent range looks at the high word.  Five FP64 operations for
// 1/sqrt(v), seven for v^(-5/2).  Outside 2^-99 <= v < 2^99 (negative, infinite and NaN arguments
// included) the estimate is unusable and est returns false.
__device__ __forceinline__ bool rsqrt_est64(double v, double& y, double& e) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  if (hi - (924u << 20) >= (198u << 20)) return false;
  const unsigned f = __float_as_uint(rsqrt_est(__uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29))));
  y = __hiloint2double((int)((f >> 3) + (896u << 20)), (int)(f << 29));
  e = fma(-v, y * y, 1.0);
  return true;
}
template <>
__device__ inline double rsqrt_<double>(double v) {
  double y, e;
  if (!rsqrt_est64(v, y, e)) return 1.0 / sqrt(v);
  return fma(y, e * fma(0.375, e, 0.5), y);
}
template <>
__device__ inline float rsqrt_<float>(float v) {
  return rsqrt_est(v);
}

// v^(-5/2)
template <typename R>
__device__ inline R rsqrt5_(R v);
template <>
__device__ inline double rsqrt5_<double>(double v) {
  double y, e;
  if (!rsqrt_est64(v, y, e)) {
    const double r = 1.0 / sqrt(v), r2 = r * r;
    return r2 * r2 * r;
  }
  const double y2 = y * y, y5 = y2 * y2 * y;
  return fma(y5, e * fma(4.375, e, 2.5), y5);
}
template <>
__device__ inline float rsqrt5_<float>(float v) {
  const float r = rsqrt_est(v), r2 = r * r;
  return r2 * r2 * r;
}

// Block-wide sum of three values; the result is valid in thread 0.  sh holds 3 * 32 entries.
template <typename R>
__device__ inline void block_sum3(R& a, R& b, R& c, R* sh) {
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    sh[w * 3] = a;
    sh[w * 3 + 1] = b;
    sh[w * 3 + 2] = c;
  }
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    a = l < nw ? sh[l * 3] : (R)0;
    b = l < nw ? sh[l * 3 + 1] : (R)0;
    c = l < nw ? sh[l * 3 + 2] : (R)0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
      c += __shfl_down_sync(0xffffffffu, c, o);
    }
  }
}

// The point of the records r [7][N] nearest to x0, scanned by one warp, its lanes striding over the points (the first
// nearest point wins ties, as in a sequential scan); every lane gets its index and squared distance.
__device__ inline long long warp_nearest(const double* __restrict__ r, long long N, double x0, double x1, double x2,
                                         double& d2) {
  double best = 1e300;
  long long bi = N;
  for (long long s = threadIdx.x & 31; s < N; s += 32) {
    const double d0 = x0 - r[s], d1 = x1 - r[N + s], dz = x2 - r[2 * N + s];
    const double d = d0 * d0 + d1 * d1 + dz * dz;
    if (d < best) {
      best = d;
      bi = s;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {  // smallest distance, then smallest index
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const long long oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob < best || (ob == best && oi < bi)) {
      best = ob;
      bi = oi;
    }
  }
  d2 = best;
  return bi < N ? bi : 0;
}

// Degree n of the packed index r = n(n+1)+m (0 <= r < (p+1)^2).
__device__ inline int degree_of(int r) {
  int n = (int)sqrtf((float)r);
  while (n * n > r) --n;
  while ((n + 1) * (n + 1) <= r) ++n;
  return n;
}

}  // namespace bie
