// common.cuh -- types and small device helpers shared by the library's kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fde {

// Interleaved complex type of a real type.
template <typename T> struct cx;
template <> struct cx<float> { using t = float2; };
template <> struct cx<double> { using t = double2; };
template <typename T> using cplx = typename cx<T>::t;

template <typename T> __host__ __device__ __forceinline__ cplx<T> mk(T re, T im) {
  cplx<T> z; z.x = re; z.y = im; return z;
}
template <typename C> __host__ __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
  C z; z.x = a.x * b.x - a.y * b.y; z.y = a.x * b.y + a.y * b.x; return z;
}
// conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cmulc(C a, C b) {
  C z; z.x = a.x * b.x + a.y * b.y; z.y = a.x * b.y - a.y * b.x; return z;
}
template <typename C, typename T> __host__ __device__ __forceinline__ C cscale(C a, T s) { a.x *= s; a.y *= s; return a; }
// multiply by sign * i
template <typename C> __host__ __device__ __forceinline__ C cmuli(C a, int sign) {
  C z; if (sign > 0) { z.x = -a.y; z.y = a.x; } else { z.x = a.y; z.y = -a.x; } return z;
}
template <typename C> __host__ __device__ __forceinline__ C cconj(C a) { a.y = -a.y; return a; }

// FP32 complex values as packed pairs: one issue slot for both parts (the FP32 pipe takes two
// cycles for it, so the gain is the slot, which the transforms need for their loads and indices).
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }

// b + s a and m + sign i s d (sign i d without s) for real s, one rounding a part in FP32 and FP64.
template <typename C, typename T> __device__ __forceinline__ C caxpy(C a, T s, C b) { return cadd(b, cscale(a, s)); }
__device__ __forceinline__ float2 caxpy(float2 a, float s, float2 b) { return __ffma2_rn(a, make_float2(s, s), b); }
__device__ __forceinline__ double2 caxpy(double2 a, double s, double2 b) {
  return make_double2(fma(a.x, s, b.x), fma(a.y, s, b.y));
}
// b - s a
template <typename C, typename T> __device__ __forceinline__ C caxmy(C a, T s, C b) { return csub(b, cscale(a, s)); }
__device__ __forceinline__ float2 caxmy(float2 a, float s, float2 b) { return caxpy(a, -s, b); }
__device__ __forceinline__ double2 caxmy(double2 a, double s, double2 b) { return caxpy(a, -s, b); }
template <typename C, typename T> __device__ __forceinline__ C caddi(C m, C d, T s, int sign) {
  return cadd(m, cmuli(cscale(d, s), sign));
}
__device__ __forceinline__ float2 caddi(float2 m, float2 d, float s, int sign) {
  const float t = sign > 0 ? s : -s;
  return make_float2(fmaf(-t, d.y, m.x), fmaf(t, d.x, m.y));
}
__device__ __forceinline__ double2 caddi(double2 m, double2 d, double s, int sign) {
  const double t = sign > 0 ? s : -s;
  return make_double2(fma(-t, d.y, m.x), fma(t, d.x, m.y));
}
template <typename C> __device__ __forceinline__ C caddi(C m, C d, int sign) { return cadd(m, cmuli(d, sign)); }
__device__ __forceinline__ float2 caddi(float2 m, float2 d, int sign) {
  return sign > 0 ? make_float2(m.x - d.y, m.y + d.x) : make_float2(m.x + d.y, m.y - d.x);
}

// Device status word bits (checked by the host after synchronising calls).
enum : unsigned { ST_NONFINITE = 1u, ST_CHOLESKY = 2u, ST_NOCONV = 4u, ST_TIMEOUT = 8u, ST_TMEM_HELD = 16u };

// Largest supported 1D transform length (one line held by one warp in shared memory).
constexpr int kMaxLine = 320;
// Largest (x, y) plane side transformed inside one CTA.
constexpr int kMaxPlane = 160;
constexpr int kMaxStages = 8;

// One 1D transform length: its radix factorisation and twiddle table
// tw[m] = exp(-2 pi i m / n), m in [0, n).
template <typename T> struct LinePlan {
  int n;
  int nstages;
  int radix[kMaxStages];
  const cplx<T>* tw;
};

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

}  // namespace fde
