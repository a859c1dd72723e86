// Butterflies, Fourier-symbol quotients and the regularised-delta kernels used by the IBDL kernels.
#pragma once

#include "ibdl_internal.cuh"

namespace ibdl {

template <typename T, bool INV>
__device__ __forceinline__ void dft2(cplx<T>* u) {
  const cplx<T> t = u[0];
  u[0] = cadd(t, u[1]);
  u[1] = csub(t, u[1]);
}

// multiply by −i (forward) or +i (inverse)
template <typename T, bool INV>
__device__ __forceinline__ cplx<T> rot90(cplx<T> a) {
  return INV ? mk(-a.y, a.x) : mk(a.y, -a.x);
}

template <typename T, bool INV>
__device__ __forceinline__ void dft4(cplx<T>& a0, cplx<T>& a1, cplx<T>& a2, cplx<T>& a3) {
  const cplx<T> t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3);
  const cplx<T> t3 = rot90<T, INV>(csub(a1, a3));
  a0 = cadd(t0, t2);
  a1 = cadd(t1, t3);
  a2 = csub(t0, t2);
  a3 = csub(t1, t3);
}

// 8-point DFT as two 4-point DFTs: X_{2k} = DFT4(u_r + u_{r+4}), X_{2k+1} = DFT4((u_r − u_{r+4}) ω₈^r)
template <typename T, bool INV>
__device__ __forceinline__ void dft8(cplx<T>* u) {
  const T c = T(0.70710678118654752440);
  cplx<T> a0 = cadd(u[0], u[4]), a1 = cadd(u[1], u[5]), a2 = cadd(u[2], u[6]), a3 = cadd(u[3], u[7]);
  cplx<T> b0 = csub(u[0], u[4]), b1 = csub(u[1], u[5]), b2 = csub(u[2], u[6]), b3 = csub(u[3], u[7]);
  b1 = INV ? mk((b1.x - b1.y) * c, (b1.x + b1.y) * c) : mk((b1.x + b1.y) * c, (b1.y - b1.x) * c);
  b2 = rot90<T, INV>(b2);
  b3 = INV ? mk(-(b3.x + b3.y) * c, (b3.x - b3.y) * c) : mk((b3.y - b3.x) * c, -(b3.x + b3.y) * c);
  dft4<T, INV>(a0, a1, a2, a3);
  dft4<T, INV>(b0, b1, b2, b3);
  u[0] = a0;
  u[1] = b0;
  u[2] = a1;
  u[3] = b1;
  u[4] = a2;
  u[5] = b2;
  u[6] = a3;
  u[7] = b3;
}

// whether a sum of squares is zero; in FP64 by its bits, which keeps the comparison off the FP64 pipe
__device__ __forceinline__ bool sym_zero(float a) { return a == 0.0f; }
__device__ __forceinline__ bool sym_zero(double a) { return __double_as_longlong(a) == 0; }

// a/b of a Fourier symbol: the hardware reciprocal estimate in 2-D FP32 (within 2 ulp, well inside the
// FP32 application's rounding), a corrected quotient in float-float, IEEE division in FP64
__device__ __forceinline__ float sym_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double sym_div(double a, double b) { return a / b; }

// The 3-D row kernels' buffers are padded with one element after every eight, which keeps the
// radix-8 stride-8 writes of the first stages free of bank conflicts for 8- and 16-byte elements.
__device__ __forceinline__ int pidx(int x) { return x + (x >> 3); }
__host__ __device__ constexpr size_t padded(size_t x) { return x + (x >> 3); }

// ------------------------------------------------------------------------------------------
// One-dimensional 4-point kernels φ of δ_h (Sec. 2.2.2) and their derivatives, FP64.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ double phi_cos(double r) {
  return fabs(r) < 2.0 ? 0.25 * (1.0 + cospi(0.5 * r)) : 0.0;
}
__device__ __forceinline__ double dphi_cos(double r) {
  return fabs(r) < 2.0 ? -0.125 * 3.14159265358979323846 * sinpi(0.5 * r) : 0.0;
}
// Peskin: (3 − 2a + √(1 + 4a − 4a²))/8 on a ≤ 1, (5 − 2a − √(−7 + 12a − 4a²))/8 on 1 < a < 2
__device__ __forceinline__ double phi_sqrt(double r) {
  const double a = fabs(r);
  if (a <= 1.0) return (3.0 - 2.0 * a + sqrt(1.0 + 4.0 * a - 4.0 * a * a)) * 0.125;
  if (a < 2.0) return (5.0 - 2.0 * a - sqrt(-7.0 + 12.0 * a - 4.0 * a * a)) * 0.125;
  return 0.0;
}
__device__ __forceinline__ double dphi_sqrt(double r) {
  const double a = fabs(r);
  double d = 0.0;
  if (a <= 1.0)
    d = (-2.0 + (2.0 - 4.0 * a) / sqrt(1.0 + 4.0 * a - 4.0 * a * a)) * 0.125;
  else if (a < 2.0)
    d = (-2.0 - (6.0 - 4.0 * a) / sqrt(-7.0 + 12.0 * a - 4.0 * a * a)) * 0.125;
  return r < 0.0 ? -d : d;
}
// second derivatives (even in r); at the joins |r| = 1 (√ form) and |r| = 2 the inner piece's value
__device__ __forceinline__ double ddphi_cos(double r) {
  const double c = 3.14159265358979323846 * 3.14159265358979323846 / 16.0;
  return fabs(r) < 2.0 ? -c * cospi(0.5 * r) : 0.0;
}
__device__ __forceinline__ double ddphi_sqrt(double r) {
  const double a = fabs(r);
  if (a <= 1.0) {
    const double q = 1.0 + 4.0 * a - 4.0 * a * a, sq = sqrt(q);
    return (-4.0 / sq - (2.0 - 4.0 * a) * (4.0 - 8.0 * a) / (2.0 * q * sq)) * 0.125;
  }
  if (a < 2.0) {
    const double q = -7.0 + 12.0 * a - 4.0 * a * a, sq = sqrt(q);
    return (4.0 / sq + (6.0 - 4.0 * a) * (12.0 - 8.0 * a) / (2.0 * q * sq)) * 0.125;
  }
  return 0.0;
}

}  // namespace ibdl
