// fft3.cuh -- full-grid 3D transforms on two-step plans (fft2.cuh): FP32 and FP64 grids, and FP64
// grids in double-float arithmetic (dd.cuh); included by one translation unit per type.
//
// One axis per pass, in place.  A CTA takes the lines that fill 128 bytes of a grid row (256 for
// 16-byte values); each of its threads reads one butterfly's inputs from global memory, the two
// steps exchange through shared memory once, and the outputs go straight back to global memory.
// The strided axes run lanes over neighbouring lines, the contiguous one over neighbouring
// elements of a line.
#pragma once

#include "dd.cuh"
#include "fft2.cuh"
#include "kernels.h"
#include "prof.h"

namespace fde {

namespace {

template <typename C> __host__ __device__ constexpr int ax_lines() { return 16; }
template <typename C, int R1, int R2> __host__ __device__ constexpr int ax_threads() {
  return round_up(ax_lines<C>() * (R1 > R2 ? R1 : R2), 32);
}
// Lines and threads of a CTA of the contiguous axis: one round of items.  (256 threads for the 120
// items of eight double-float lines held 8 of 15 warps a CTA at its barrier: 70 us for 180-point lines
// of 72 x 72 x 180.)
template <typename C> __host__ __device__ constexpr int ctg_lines() { return sizeof(C) == 8 ? 16 : 8; }
template <typename C, int R1, int R2> __host__ __device__ constexpr int ctg_threads() {
  return round_up(ctg_lines<C>() * (R1 > R2 ? R1 : R2), 32);
}

// Global forms of the grid a pass reads and writes.
struct AsIs {};  // values of the transform's own type
struct AsF64 {}; // FP64 values of a double-float transform: split on reading, joined on writing
struct AsHigh {};  // FP32: the high parts (a normalised double-float rounded to FP32)
template <typename C> __device__ __forceinline__ C ax_get(const void* p, int i, AsIs) {
  return reinterpret_cast<const C*>(p)[i];
}
// The kernels transform forward (a sign known when they are compiled folds every root into an
// immediate); the inverse is the forward transform between two conjugations.
template <typename C> __device__ __forceinline__ C ax_conj(C v, bool conj) {
  if (conj) v.y = -v.y;
  return v;
}
template <typename C> __device__ __forceinline__ ddc ax_get(const void* p, int i, AsF64) {
  const double2 x = reinterpret_cast<const double2*>(p)[i];
  ddc v;
  v.x = dd_from_double(x.x);
  v.y = dd_from_double(x.y);
  return v;
}
template <typename C> __device__ __forceinline__ void ax_put(void* p, int i, C v, AsIs) {
  reinterpret_cast<C*>(p)[i] = v;
}
template <typename C> __device__ __forceinline__ void ax_put(void* p, int i, ddc v, AsHigh) {
  reinterpret_cast<float2*>(p)[i] = make_float2(v.x.hi, v.y.hi);
}
template <typename C> __device__ __forceinline__ void ax_put(void* p, int i, ddc v, AsF64) {
  reinterpret_cast<double2*>(p)[i] = make_double2(dd_to_double(v.x), dd_to_double(v.y));
}

// Strided axis: element e of line l = (o, t) at (o N + e) stride + t, t < stride; on the side's plan
// (prime-factor indices where it has coprime factors: no twiddles).
template <typename T, typename Plan, typename IN, typename OUT>
__global__ void __launch_bounds__(ax_threads<cplx<T>, Plan::R1, Plan::R2>())
k_fft_strided(const void* data, void* out, int nlines, int stride, const cplx<T>* __restrict__ tw, bool conj) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2, N = Plan::N, L = ax_lines<C>(), NT = ax_threads<C, R1, R2>();
  __shared__ __align__(16) C X[N * L];
  const int c = threadIdx.x % L, i = threadIdx.x / L;
  const int l = blockIdx.x * L + c;
  const bool live = l < nlines;
  const int o = l / stride;
  const int base = o * N * stride + (l - o * stride);
  static_assert(NT / L >= (R1 > R2 ? R1 : R2), "one butterfly a thread");
  if (live && i < R2) {
    C v[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r)
      v[r] = ax_conj(ax_get<C>(data, base + Plan::wrap(Plan::in0(i) + r * R2) * stride, IN()), conj);
    dft_r<R1>(v, -1);
#pragma unroll
    for (int q = 0; q < R1; ++q) X[(q * R2 + i) * L + c] = v[q];
  }
  __syncthreads();
  if (live && i < R1) {
    C v[R2];
#pragma unroll
    for (int j = 0; j < R2; ++j) {
      v[j] = X[(i * R2 + j) * L + c];
      if (!Plan::kCoprime && j) v[j] = cmul(v[j], tw[j * i]);
    }
    dft_r<R2>(v, -1);
#pragma unroll
    for (int p = 0; p < R2; ++p) ax_put<C>(out, base + Plan::output(i, p) * stride, ax_conj(v[p], conj), OUT());
  }
}

// Contiguous axis: line l at l N.  The exchange pads each run of R2 values to an odd length, so
// that step 2's lanes (neighbouring q) lie on different banks.
template <typename T, int R1, int R2, typename IN, typename OUT>
__global__ void __launch_bounds__(ctg_threads<cplx<T>, R1, R2>())
k_fft_contig(void* __restrict__ data, int nlines, const cplx<T>* __restrict__ tw, bool conj) {
  using C = cplx<T>;
  constexpr int N = R1 * R2, L = ctg_lines<C>(), NT = ctg_threads<C, R1, R2>(), RP = R2 | 1, XP = R1 * RP | 1;
  __shared__ __align__(16) C X[L * XP];
  const int l0 = blockIdx.x * L;
  for (int w = threadIdx.x; w < L * R2; w += NT) {
    const int c = w / R2, j = w - c * R2;
    if (l0 + c < nlines) {
      const int base = (l0 + c) * N;
      C v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = ax_conj(ax_get<C>(data, base + j + r * R2, IN()), conj);
      dft_r<R1>(v, -1);
#pragma unroll
      for (int q = 0; q < R1; ++q) X[c * XP + q * RP + j] = v[q];
    }
  }
  __syncthreads();
  for (int w = threadIdx.x; w < L * R1; w += NT) {
    const int c = w / R1, q = w - c * R1;
    if (l0 + c < nlines) {
      const int base = (l0 + c) * N;
      C v[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) {
        v[j] = X[c * XP + q * RP + j];
        if (j) v[j] = cmul(v[j], tw[j * q]);
      }
      dft_r<R2>(v, -1);
#pragma unroll
      for (int p = 0; p < R2; ++p) ax_put<C>(data, base + q + R1 * p, ax_conj(v[p], conj), OUT());
    }
  }
}

// One pass over the lengths of LIST; false when n is none of them.
#define FDE_AXIS_LAUNCHERS(SIDES, LINES)                                                                          \
  template <typename T, typename IN, typename OUT>                                                               \
  bool strided_axis(int n, long long nlines, int stride, void* data, void* out, const cplx<T>* tw, int sign,     \
                    cudaStream_t st) {                                                                            \
    const unsigned blocks = (unsigned)ceil_div(nlines, ax_lines<cplx<T>>());                                      \
    switch (n) { SIDES(FDE_STRIDED_CASE) }                                                                        \
    return false;                                                                                                 \
  }                                                                                                               \
  template <typename T, typename IN, typename OUT>                                                               \
  bool contig_axis(int n, long long nlines, void* data, const cplx<T>* tw, int sign, cudaStream_t st) {          \
    const unsigned blocks = (unsigned)ceil_div(nlines, ctg_lines<cplx<T>>());                                     \
    switch (n) { LINES(FDE_CONTIG_CASE) }                                                                         \
    return false;                                                                                                 \
  }
#define FDE_STRIDED_CASE(N, R1, R2)                                                                               \
  case N:                                                                                                         \
    count_launches(1);                                                                                            \
    k_fft_strided<T, SidePlan<R1, R2>, IN, OUT><<<blocks, ax_threads<cplx<T>, R1, R2>(), 0, st>>>(               \
        data, out, (int)nlines, stride, tw, sign > 0);                                                            \
    return true;
#define FDE_CONTIG_CASE(N, R1, R2)                                                                                \
  case N:                                                                                                         \
    count_launches(1);                                                                                            \
    k_fft_contig<T, R1, R2, IN, OUT><<<blocks, ctg_threads<cplx<T>, R1, R2>(), 0, st>>>(data, (int)nlines, tw,   \
                                                                                        sign > 0);               \
    return true;

inline bool grid_ok(const GridDims& g) {
  return split_side_ok(g.n1) && split_side_ok(g.n2) && split_of(g.n3).a > 0 &&
         (long long)g.n1 * g.n2 * g.n3 < (1ll << 31);  // 32-bit element indices
}

}  // namespace

}  // namespace fde
