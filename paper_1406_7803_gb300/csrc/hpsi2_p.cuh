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
// Threads and least resident CTAs of a square plane's kernel, for every side by one rule.  A CTA has threads
// for whole batches of columns: m batches, ceil(N / m) R1 threads in warps.  Of the m with 160 to 384
// threads (up to 512 for a CTA that has an SM to itself) the one is taken that keeps most busy threads on
// an SM, each counted by the share of its CTA that is busy (idle threads wait at the barriers too), and of
// equal ones the smallest CTA.  An SM holds as many as 64 (FP64 96) registers a thread allow and the
// shared memory of a sphere that spans 0.46 N, the cutoff the grids are made for.
// Against 256 threads for most sides and a few set by hand (192 to 384), planes of 0.46 N spans that fill the
// GPU take 0.97 times as long in the geometric mean of the 24 sides (FP32 0.78 .. 1.06, FP64 0.89 .. 1.02).
// With 128 to 256 threads they would take 0.91 times as long in FP32, but H psi of few planes or wide
// spheres gets slower: 128 planes of 32 x 32, FP64, 39 us instead of 33; 64 bands of 72 x 72 x 96, spans of
// 70, 490 us instead of 378; 32 bands of 144 x 144 x 288 1543 us instead of 1457.
struct PlaneShape {
  int nt, minb;
};
template <typename T> constexpr PlaneShape plane_shape(int n) {
  const int r1 = side_rmax(n), span = (46 * n / 100) | 1, regs = sizeof(T) == 4 ? 64 : 96;
  PlaneShape best{0, 1};
  double most = 0;
  for (int m = 1; m <= n; ++m) {
    const int lb = (n + m - 1) / m, nt = round_up(lb * r1, 32);
    const int x = n * lb > span * span ? n * lb : span * span;
    const int fit = 233472 / ((span * (n | 1) + x) * (int)sizeof(cplx<T>) + 1024);  // by shared memory
    if (nt < 160 || nt > (fit > 1 ? 384 : 512)) continue;
    int cta = 65536 / (nt * regs);
    if (cta > fit) cta = fit;
    if (cta < 1) cta = 1;
    const double busy = (double)(n * r1) / (m * nt), score = cta * nt * busy * busy;
    if (score < most) continue;
    most = score;
    best = PlaneShape{nt, cta};
  }
  return best;
}
// Columns of a batch (the shape of each square side found when this is compiled: it is asked for with
// every launch).
template <typename T> constexpr int plane_lb(int n1, int n2) {
  if (n1 == n2) switch (n1) {
#define FDE_CASE(N, R1, R2)                                           \
  case N: {                                                           \
    constexpr int lb = plane_batch(N, R1, plane_shape<T>(N).nt);      \
    return lb;                                                        \
  }
      FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
    }
  return plane_batch(n2, side_rmax(n1), kPlaneThreads2);
}

// Shared memory of the plane pass: P for the widest span of the launch, X for one batch of columns and
// for the column stage of `rows` rows.
template <typename T> constexpr size_t plane_smem2(int n1, int n2, int span1, int span2, int rows, int lb) {
  const size_t p = (size_t)span1 * (n2 | 1);
  const size_t x = std::max((size_t)n1 * lb, (size_t)rows * (span2 | 1));
  return (p + x) * sizeof(cplx<T>);
}
// Square sides whose widest spheres need the column stage in runs of rows (of the planes that a context
// takes: whole planes in shared memory), and the threads of their kernel: a CTA has an SM to itself, so
// the most whose batches fit beside a whole plane.
template <typename T> constexpr bool plane_has_runs(int n) {
  return plane_smem2<T>(n, n, n, n, n, plane_lb<T>(n, n)) > kCtaSmemMax &&
         (size_t)n * (n + 1) * sizeof(cplx<T>) <= kCtaSmemMax;
}
template <typename T> constexpr int plane_runs_threads(int n) {
  const int r1 = side_rmax(n);
  int nt = 0;
  for (int m = 1; m <= n; ++m) {
    const int lb = (n + m - 1) / m;
    nt = round_up(lb * r1, 32);
    if (nt <= 512 && (nt <= 160 || plane_smem2<T>(n, n, n, n, 1, lb) <= kCtaSmemMax)) break;
  }
  return nt;
}
template <typename T> constexpr int plane_runs_lb(int n) {
  switch (n) {
#define FDE_CASE(N, R1, R2)                                           \
  case N: {                                                           \
    constexpr int lb = plane_batch(N, R1, plane_runs_threads<T>(N));  \
    return lb;                                                        \
  }
    FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
  }
  return 1;
}
// How a launch whose widest spans are span1 and span2 runs: rows of the column stage at a time -- all span1
// where they fit, else the fewest even runs of them; 0 when even one row does not fit, or on planes of
// different sides -- whether by the kernel with runs, and its shared memory.
struct PlaneFit {
  int rows;
  bool runs;
  size_t smem;
};
template <typename T> static PlaneFit plane_fit(const GridDims& g, int span1, int span2) {
  const size_t all = plane_smem2<T>(g.n1, g.n2, span1, span2, span1, plane_lb<T>(g.n1, g.n2));
  if (all <= kCtaSmemMax) return {span1, false, all};
  if (g.n1 != g.n2 || (size_t)g.n1 * (g.n1 + 1) * sizeof(cplx<T>) > kCtaSmemMax) return {0, false, all};
  const int lb = plane_runs_lb<T>(g.n1);
  if (plane_smem2<T>(g.n1, g.n2, span1, span2, 1, lb) > kCtaSmemMax) return {0, false, all};
  const int most = (int)(kCtaSmemMax / sizeof(cplx<T>) - (size_t)span1 * (g.n2 | 1)) / (span2 | 1);
  const int rows = ceil_div(span1, ceil_div(span1, most));
  return {rows, true, plane_smem2<T>(g.n1, g.n2, span1, span2, rows, lb)};
}

template <typename T> bool two_step_grid(const GridDims& g, const SphereDev& sp) {
  if (!split_side_ok(g.n1) || !split_side_ok(g.n2) || split_of(g.n3).a == 0) return false;
  return plane_fit<T>(g, sp.span1, sp.span2).rows > 0;
}
template <typename T> int plane_group(const GridDims& g, const HpsiItemDesc<T>* items, int nitems, int most) {
  int s1 = 0, s2 = 0, n = 0;
  for (; n < std::min(nitems, most); ++n) {
    s1 = std::max(s1, items[n].sp.span1);
    s2 = std::max(s2, items[n].sp.span2);
    if (plane_fit<T>(g, s1, s2).rows == 0) break;
  }
  return n;
}

template <typename T, int R1, int R2>
static cudaError_t plane_square(unsigned blocks, const HpsiBatch<T>& B, int n3, const FftPlans<T>& fp, int psize,
                                const PlaneFit& f, cudaStream_t st) {
  constexpr PlaneShape S = plane_shape<T>(R1 * R2);
  using Plan = SidePlan<R1, R2>;
  if constexpr (plane_has_runs<T>(R1 * R2)) {
    constexpr int NT = plane_runs_threads<T>(R1 * R2);
    if (f.runs)
      return launch_sized(k_plane_pass<T, Plan, Plan, NT, 1, true>, blocks, NT, f.smem, st, B, n3, fp.p1.tw, fp.p2.tw,
                          psize, f.rows);
  }
  return launch_sized(k_plane_pass<T, Plan, Plan, S.nt, S.minb, false>, blocks, S.nt, f.smem, st, B, n3, fp.p1.tw,
                      fp.p2.tw, psize, f.rows);
}

template <typename T>
cudaError_t launch_plane_pass(const GridDims& g, unsigned blocks, const HpsiBatch<T>& B, const FftPlans<T>& fp,
                              cudaStream_t st) {
  int s1 = 0, s2 = 0;
  for (int i = 0; i < B.n; ++i) {
    s1 = std::max(s1, B.it[i].sp.span1);
    s2 = std::max(s2, B.it[i].sp.span2);
  }
  const PlaneFit f = plane_fit<T>(g, s1, s2);
  const int psize = s1 * (g.n2 | 1);
  if (f.rows == 0) return cudaErrorInvalidValue;
  if (g.n1 == g.n2) {
    switch (g.n1) {
#define FDE_CASE(N, R1, R2) \
  case N:                   \
    return plane_square<T, R1, R2>(blocks, B, g.n3, fp, psize, f, st);
      FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
    }
    return cudaErrorInvalidValue;
  }
  return launch_sized(k_plane_pass_any<T>, blocks, kPlaneThreads2, f.smem, st, B, g.n1, g.n2, g.n3, fp.p1.tw, fp.p2.tw,
                      psize, plane_lb<T>(g.n1, g.n2));
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
                              typename RhoAcc<T>::t* part, int n3, const FftPlans<T>& fp, int psize,
                              const PlaneFit& f, cudaStream_t st) {
  constexpr PlaneShape S = plane_shape<T>(R1 * R2);
  using Plan = SidePlan<R1, R2>;
  if constexpr (plane_has_runs<T>(R1 * R2)) {
    constexpr int NT = plane_runs_threads<T>(R1 * R2);
    if (f.runs)
      return launch_sized(k_plane_rho<T, Plan, Plan, NT, 1, true>, grid, NT, f.smem, st, scr, sp, nb, weight, part, n3,
                          fp.p1.tw, fp.p2.tw, psize, f.rows);
  }
  return launch_sized(k_plane_rho<T, Plan, Plan, S.nt, S.minb, false>, grid, S.nt, f.smem, st, scr, sp, nb, weight,
                      part, n3, fp.p1.tw, fp.p2.tw, psize, f.rows);
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
  const PlaneFit f = plane_fit<T>(g, sp.span1, sp.span2);
  const int psize = sp.span1 * (g.n2 | 1);
  const dim3 grid(g.n3, groups);
  if (f.rows == 0) return cudaErrorInvalidValue;
  cudaError_t e = cudaErrorInvalidValue;
  if (g.n1 == g.n2) {
    switch (g.n1) {
#define FDE_CASE(N, R1, R2)                                                             \
  case N:                                                                               \
    e = rho_square<T, R1, R2>(grid, scr, sp, nb, weight, part, g.n3, fp, psize, f, st); \
    break;
      FDE_PLANE_SIDES(FDE_CASE)
#undef FDE_CASE
    }
  } else {
    e = launch_sized(k_plane_rho_any<T>, grid, kPlaneThreads2, f.smem, st, scr, sp, nb, weight, part, g.n1, g.n2, g.n3,
                     fp.p1.tw, fp.p2.tw, psize, plane_lb<T>(g.n1, g.n2));
  }
  if (e != cudaSuccess) return e;
  const long long n = (long long)g.n1 * g.n2 * g.n3;
  count_launches(1);
  k_rho_groups<A><<<(unsigned)std::min<long long>((n + 255) / 256, 4096), 256, 0, st>>>(part, groups, rho_plane,
                                                                                      accumulate, n);
  return cudaSuccess;
}

}  // namespace fde
