// hpsi2_p.cuh -- the plane pass and the plane density (hpsi2.cuh): launches for square planes of
// every two-step side, one kernel with runtime sides for the others.
#pragma once

#include "hpsi2.cuh"

namespace fde {

constexpr int kPlaneThreads2 = 256;  // planes with different sides

// Planes with different sides: the steps of every length as functions of their own, chosen by the
// sides when the kernel runs (two lengths to a kernel would be 576 kernels a precision).
template <typename T, int R1, int R2>
__device__ __noinline__ void any_y_inv(cplx<T>* P, const cplx<T>* X, const PlaneDims& D, int pitch, const cplx<T>* tw) {
  using Plan = SidePlan<R1, R2>;
  plane_y_inv_1<T, Plan>(P, X, D, pitch, kPlaneThreads2);
  __syncthreads();
  plane_y_inv_2<T, Plan>(P, D, pitch, kPlaneThreads2, tw);
}
template <typename T, int R1, int R2>
__device__ __noinline__ void any_y_fwd(cplx<T>* P, cplx<T>* X, const PlaneDims& D, int pitch, const cplx<T>* tw) {
  using Plan = SidePlan<R1, R2>;
  plane_y_fwd_2<T, Plan>(P, D, pitch, kPlaneThreads2, tw);
  __syncthreads();
  plane_y_fwd_1<T, Plan>(P, X, D, pitch, kPlaneThreads2);
}
template <typename T, int R1, int R2>
__device__ __noinline__ void any_x_all(cplx<T>* P, cplx<T>* X, const PlaneDims& D, int pitch, int n2, int lb,
                                       const cplx<T>* tw, const T* vp) {
  plane_x_all<T, SidePlan<R1, R2>>(P, X, D, pitch, n2, lb, tw, vp);
}
template <typename T, int R1, int R2>
__device__ __noinline__ void any_x_rho(const cplx<T>* P, cplx<T>* X, const PlaneDims& D, int pitch, int n2, int lb,
                                       const cplx<T>* tw, double weight, bool first, typename RhoAcc<T>::t* rho) {
  plane_x_rho<T, SidePlan<R1, R2>>(P, X, D, pitch, n2, lb, tw, weight, first, rho);
}
#define FDE_ANY(SIDE, CALL)      \
  switch (SIDE) {                \
    FDE_PLANE_SIDES(CALL)        \
  }
#define FDE_Y_INV(N, R1, R2) \
  case N: any_y_inv<T, R1, R2>(P, X, D, pitch, tw2); break;
#define FDE_Y_FWD(N, R1, R2) \
  case N: any_y_fwd<T, R1, R2>(P, X, D, pitch, tw2); break;
#define FDE_X_ALL(N, R1, R2) \
  case N: any_x_all<T, R1, R2>(P, X, D, pitch, n2, lb, tw1, vp); break;
#define FDE_X_RHO(N, R1, R2) \
  case N: any_x_rho<T, R1, R2>(P, X, D, pitch, n2, lb, tw1, weight[b], b == b0, rho); break;

template <typename T>
__global__ void __launch_bounds__(kPlaneThreads2, 2)
k_plane_pass_any(const __grid_constant__ HpsiBatch<T> B, int n1, int n2, int n3, const cplx<T>* __restrict__ tw1,
                 const cplx<T>* __restrict__ tw2, int psize, int lb) {
  using C = cplx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);
  C* X = P + psize;
  const int pitch = n2 | 1;
  const HpsiItem<T>& I = B.it[batch_item(B, blockIdx.x, true)];
  const SphereDev& sp = I.sp;
  const int local = blockIdx.x - I.pstart;
  const int b = local / n3, i3 = local - b * n3;
  C* S = I.scratch + ((size_t)b * n3 + i3) * sp.ldc;
  const T* vp = I.vplane + (size_t)i3 * n1 * n2;
  const PlaneDims D = plane_dims<T>(sp);
  plane_columns_in<T, false>(X, S, sp, D, 0, kPlaneThreads2);
  __syncthreads();
  FDE_ANY(n2, FDE_Y_INV)
  __syncthreads();
  FDE_ANY(n1, FDE_X_ALL)
  __syncthreads();
  FDE_ANY(n2, FDE_Y_FWD)
  __syncthreads();
  plane_columns_out<T, false>(X, S, sp, D, 0, kPlaneThreads2);
}

template <typename T>
__global__ void __launch_bounds__(kPlaneThreads2, 2)
k_plane_rho_any(const cplx<T>* __restrict__ scratch, SphereDev sp, int nb, const double* __restrict__ weight,
                typename RhoAcc<T>::t* __restrict__ part, int n1, int n2, int n3, const cplx<T>* __restrict__ tw1,
                const cplx<T>* __restrict__ tw2, int psize, int lb) {
  using C = cplx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);
  C* X = P + psize;
  const int pitch = n2 | 1;
  const int i3 = blockIdx.x, g = blockIdx.y;
  const int b0 = (int)((long long)nb * g / gridDim.y), b1 = (int)((long long)nb * (g + 1) / gridDim.y);
  const PlaneDims D = plane_dims<T>(sp);
  auto* rho = part + ((size_t)g * n3 + i3) * n1 * n2;
#pragma unroll 1
  for (int b = b0; b < b1; ++b) {
    plane_columns_in<T, false>(X, scratch + ((size_t)b * n3 + i3) * sp.ldc, sp, D, 0, kPlaneThreads2);
    __syncthreads();
    FDE_ANY(n2, FDE_Y_INV)
    __syncthreads();
    FDE_ANY(n1, FDE_X_RHO)
  }
}

// Threads and least resident CTAs of a square plane's kernel.  A CTA has threads for one row of items of
// the y steps (0.46 N rows hold columns at the cutoffs the grids are made for) and for whole batches
// of columns, so that few rounds run with a handful of threads: 72 x 72, 33 rows of 9 items and two
// batches of 36 columns, 352 threads.
struct PlaneShape {
  int nt, minb;
};
template <typename T> __host__ __device__ constexpr PlaneShape plane_shape(int n) {
  if (sizeof(T) == 8) return n == 72 ? PlaneShape{352, 2} : PlaneShape{n <= 24 ? 192 : 256, 2};
  if (n <= 24) return PlaneShape{192, 4};
  if (n == 72) return PlaneShape{352, 3};
  if (n <= 90) return PlaneShape{256, 4};
  if (n <= 96) return PlaneShape{288, 3};
  if (n <= 108) return PlaneShape{256, 3};
  return PlaneShape{n == 144 ? 384 : 320, 2};
}
__host__ __device__ constexpr int side_rmax(int n) {
  switch (n) {
#define FDE_CASE(N, R1, R2) \
  case N:                   \
    return R1;
    FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
  }
  return 1;
}
template <typename T> __host__ __device__ constexpr int plane_lb(int n1, int n2) {
  return plane_batch(n2, side_rmax(n1), n1 == n2 ? plane_shape<T>(n1).nt : kPlaneThreads2);
}

// Shared memory of the plane pass: P for the widest span of the launch, X for one batch of columns and
// for the column stage of `rows` rows.
template <typename T> constexpr size_t plane_smem2(int n1, int n2, int span1, int span2, int rows) {
  const size_t p = (size_t)span1 * (n2 | 1);
  const size_t x = std::max((size_t)n1 * plane_lb<T>(n1, n2), (size_t)rows * (span2 | 1));
  return (p + x) * sizeof(cplx<T>);
}
// Square sides whose widest spheres need the column stage in runs of rows (of the planes that a context
// takes: whole planes in shared memory).
template <typename T> constexpr bool plane_has_runs(int n) {
  return plane_smem2<T>(n, n, n, n, n) > kCtaSmemMax && (size_t)n * (n + 1) * sizeof(cplx<T>) <= kCtaSmemMax;
}
// Rows of the column stage at a time: all span1 where they fit, else the fewest even runs; 0 when even
// one row does not fit, or on planes of different sides.
template <typename T> static int plane_rows(const GridDims& g, int span1, int span2) {
  if (plane_smem2<T>(g.n1, g.n2, span1, span2, span1) <= kCtaSmemMax) return span1;
  if (g.n1 != g.n2 || !plane_has_runs<T>(g.n1)) return 0;
  if (plane_smem2<T>(g.n1, g.n2, span1, span2, 1) > kCtaSmemMax) return 0;
  const int most = (int)(kCtaSmemMax / sizeof(cplx<T>) - (size_t)span1 * (g.n2 | 1)) / (span2 | 1);
  return ceil_div(span1, ceil_div(span1, most));
}
// Bytes of a launch whose widest spans are span1 and span2.
template <typename T> static size_t plane_launch_smem(const GridDims& g, int span1, int span2) {
  const int rows = plane_rows<T>(g, span1, span2);
  return plane_smem2<T>(g.n1, g.n2, span1, span2, rows > 0 ? rows : span1);
}

template <typename T> bool two_step_grid(const GridDims& g, const SphereDev& sp) {
  if (!split_side_ok(g.n1) || !split_side_ok(g.n2) || split_of(g.n3).a == 0) return false;
  return plane_rows<T>(g, sp.span1, sp.span2) > 0;
}
template <typename T> int plane_group(const GridDims& g, const HpsiItemDesc<T>* items, int nitems, int most) {
  int s1 = 0, s2 = 0, n = 0;
  for (; n < std::min(nitems, most); ++n) {
    s1 = std::max(s1, items[n].sp.span1);
    s2 = std::max(s2, items[n].sp.span2);
    if (plane_rows<T>(g, s1, s2) == 0) break;
  }
  return n;
}

// A plane's kernel: one CTA an SM where the column stage comes in runs (P takes more than half of an SM's
// shared memory then).
template <typename T, int R1, int R2>
static cudaError_t plane_square(unsigned blocks, const HpsiBatch<T>& B, int n3, const FftPlans<T>& fp, size_t sm,
                                int psize, int rows, bool runs, cudaStream_t st) {
  constexpr PlaneShape S = plane_shape<T>(R1 * R2);
  using Plan = SidePlan<R1, R2>;
  if constexpr (plane_has_runs<T>(R1 * R2)) {
    if (runs)
      return launch_sized(k_plane_pass<T, Plan, Plan, S.nt, 1, true>, blocks, S.nt, sm, st, B, n3, fp.p1.tw, fp.p2.tw,
                          psize, rows);
  }
  return launch_sized(k_plane_pass<T, Plan, Plan, S.nt, S.minb, false>, blocks, S.nt, sm, st, B, n3, fp.p1.tw,
                      fp.p2.tw, psize, rows);
}

template <typename T>
cudaError_t launch_plane_pass(const GridDims& g, unsigned blocks, const HpsiBatch<T>& B, const FftPlans<T>& fp,
                              cudaStream_t st) {
  int s1 = 0, s2 = 0;
  for (int i = 0; i < B.n; ++i) {
    s1 = std::max(s1, B.it[i].sp.span1);
    s2 = std::max(s2, B.it[i].sp.span2);
  }
  const int lb = plane_lb<T>(g.n1, g.n2);
  const size_t sm = plane_launch_smem<T>(g, s1, s2);
  const int psize = s1 * (g.n2 | 1), rows = plane_rows<T>(g, s1, s2);
  if (rows == 0) return cudaErrorInvalidValue;
  if (g.n1 == g.n2) {
    switch (g.n1) {
#define FDE_CASE(N, R1, R2) \
  case N:                   \
    return plane_square<T, R1, R2>(blocks, B, g.n3, fp, sm, psize, rows, rows < s1, st);
      FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
    }
    return cudaErrorInvalidValue;
  }
  return launch_sized(k_plane_pass_any<T>, blocks, kPlaneThreads2, sm, st, B, g.n1, g.n2, g.n3, fp.p1.tw, fp.p2.tw,
                      psize, lb);
}

// rho_plane (+)= the groups' partial sums, in group order.
__device__ __forceinline__ double rho_value(double v) { return v; }
__device__ __forceinline__ double rho_value(float2 v) { return dd_to_double(dd(v.x, v.y)); }
template <typename A>
__global__ void k_rho_groups(const A* __restrict__ part, int groups, double* __restrict__ rho_plane, int accumulate,
                             long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double s = accumulate ? rho_plane[i] : 0.0;
    for (int g = 0; g < groups; ++g) s += rho_value(part[(size_t)g * n + i]);
    rho_plane[i] = s;
  }
}

template <typename T, int R1, int R2>
static cudaError_t rho_square(dim3 grid, const cplx<T>* scr, const SphereDev& sp, int nb, const double* weight,
                              typename RhoAcc<T>::t* part, int n3, const FftPlans<T>& fp, size_t sm, int psize,
                              int rows, cudaStream_t st) {
  constexpr PlaneShape S = plane_shape<T>(R1 * R2);
  using Plan = SidePlan<R1, R2>;
  if constexpr (plane_has_runs<T>(R1 * R2)) {
    if (rows < sp.span1)
      return launch_sized(k_plane_rho<T, Plan, Plan, S.nt, 1, true>, grid, S.nt, sm, st, scr, sp, nb, weight, part, n3,
                          fp.p1.tw, fp.p2.tw, psize, rows);
  }
  return launch_sized(k_plane_rho<T, Plan, Plan, S.nt, S.minb, false>, grid, S.nt, sm, st, scr, sp, nb, weight, part,
                      n3, fp.p1.tw, fp.p2.tw, psize, rows);
}

// Groups of bands of a plane density: enough CTAs for four on each of 152 SMs.
int plane_density_groups(int nb, int n3);

template <typename T>
cudaError_t launch_plane_density(const GridDims& g, const cplx<T>* scr, const SphereDev& sp, int nb,
                                 const double* weight, double* part_, double* rho_plane, int accumulate,
                                 const FftPlans<T>& fp, cudaStream_t st) {
  using A = typename RhoAcc<T>::t;
  static_assert(sizeof(A) == sizeof(double), "partial sums take the space of a double");
  A* part = reinterpret_cast<A*>(part_);
  const int groups = plane_density_groups(nb, g.n3);
  const int lb = plane_lb<T>(g.n1, g.n2);
  const size_t sm = plane_launch_smem<T>(g, sp.span1, sp.span2);
  const int psize = sp.span1 * (g.n2 | 1), rows = plane_rows<T>(g, sp.span1, sp.span2);
  const dim3 grid(g.n3, groups);
  if (rows == 0) return cudaErrorInvalidValue;
  cudaError_t e = cudaErrorInvalidValue;
  if (g.n1 == g.n2) {
    switch (g.n1) {
#define FDE_CASE(N, R1, R2)                                                                    \
  case N:                                                                                      \
    e = rho_square<T, R1, R2>(grid, scr, sp, nb, weight, part, g.n3, fp, sm, psize, rows, st); \
    break;
      FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
    }
  } else {
    e = launch_sized(k_plane_rho_any<T>, grid, kPlaneThreads2, sm, st, scr, sp, nb, weight, part, g.n1, g.n2, g.n3,
                     fp.p1.tw, fp.p2.tw, psize, lb);
  }
  if (e != cudaSuccess) return e;
  const long long n = (long long)g.n1 * g.n2 * g.n3;
  count_launches(1);
  k_rho_groups<A><<<(unsigned)std::min<long long>((n + 255) / 256, 4096), 256, 0, st>>>(part, groups, rho_plane,
                                                                                      accumulate, n);
  return cudaSuccess;
}

}  // namespace fde
