// linalg.cu -- dense complex algebra of the subspace eigensolver (Eq. KS solved by block
// Davidson): band-block inner products (Gram / subspace Hamiltonian / projector
// contractions), band-block rotations, FP64 Cholesky with triangular inverse, and the
// row-wise residual / preconditioner helpers.
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "dd.cuh"
#include "dense.h"
#include "kernels.h"
#include "prof.h"

namespace fde {

// ---- C = A^H B over a long K ------------------------------------------------------------
// 32 x 32 output tile per CTA (256 threads, 2 x 2 outputs each), K split over gridDim.z;
// each split writes its partial tile, a second kernel sums the splits in a fixed order.
constexpr int kGT = 32, kGK = 32;

template <typename T, typename Acc>
__global__ void __launch_bounds__(256)
k_gemm_hn_partial(const cplx<T>* __restrict__ A, int lda, const cplx<T>* __restrict__ B, int ldb, int m, int n,
                  int K, int kchunk, double2* __restrict__ part) {
  using C = cplx<T>;
  __shared__ C As[kGT][kGK + 1];
  __shared__ C Bs[kGT][kGK + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i0 = blockIdx.x * kGT, j0 = blockIdx.y * kGT;
  const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
  Acc re[2][2] = {{0, 0}, {0, 0}}, im[2][2] = {{0, 0}, {0, 0}};
  for (int k0 = kb; k0 < ke; k0 += kGK) {
    for (int idx = threadIdx.x; idx < kGT * kGK; idx += 256) {
      const int r = idx / kGK, kk = idx % kGK;
      const int g = k0 + kk;
      const bool ok = g < ke;
      As[r][kk] = (ok && i0 + r < m) ? A[(size_t)(i0 + r) * lda + g] : mk<T>(0, 0);
      Bs[r][kk] = (ok && j0 + r < n) ? B[(size_t)(j0 + r) * ldb + g] : mk<T>(0, 0);
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kGK; ++kk) {
      C a0 = As[ty][kk], a1 = As[ty + 16][kk];
      C b0 = Bs[tx][kk], b1 = Bs[tx + 16][kk];
      // conj(a) * b
      re[0][0] += (Acc)a0.x * b0.x + (Acc)a0.y * b0.y; im[0][0] += (Acc)a0.x * b0.y - (Acc)a0.y * b0.x;
      re[0][1] += (Acc)a0.x * b1.x + (Acc)a0.y * b1.y; im[0][1] += (Acc)a0.x * b1.y - (Acc)a0.y * b1.x;
      re[1][0] += (Acc)a1.x * b0.x + (Acc)a1.y * b0.y; im[1][0] += (Acc)a1.x * b0.y - (Acc)a1.y * b0.x;
      re[1][1] += (Acc)a1.x * b1.x + (Acc)a1.y * b1.y; im[1][1] += (Acc)a1.x * b1.y - (Acc)a1.y * b1.x;
    }
    __syncthreads();
  }
  double2* P = part + (size_t)blockIdx.z * m * n;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
      if (i < m && j < n) P[(size_t)i * n + j] = make_double2((double)re[a][b], (double)im[a][b]);
    }
}

// FP64: C = A^H B with every lane of every warp on an output of its own.  The FP64 pipe takes a warp
// instruction every 64 cycles of an SM quarter here (1/64 of the FP32 rate), so the product is bound
// by its 4 m n K fused multiply-adds and by nothing else -- provided no lane computes padding and
// every SM has work.  A 32 x 32 tile (the form before) spent 2.5 times the work on the 72 x 17 outputs
// of a projector contraction and 6 FP64 instructions a product where 4 do; with at most two K-splits
// of 900 plane waves it kept 8 CTAs busy.  Here a CTA takes 256 consecutive outputs of the flattened
// m x n (of a Gram matrix, A = B: of its upper triangle) and one of as many K-splits as fill the GPU;
// idle warps of the last CTA cost nothing.
// 72 x 17 over 43.7 k plane waves: 1742 -> 466 us (the adds alone: 360 us); 36 x 36 over 898: 831 -> 10 us.
constexpr int kFO = 256;      // outputs (threads) a CTA
constexpr int kFK = 8;        // complex K values staged at a time (one 128-byte run of a row)
constexpr int kFJ = 128;      // widest tile of C columns
constexpr int kFP = kFK + 1;  // shared-memory pitch
constexpr int kFRows = 260;   // staged rows of A and B together: at most 256 / w + 2 + w for w columns

// Output o of the flattened upper triangle of an n x n matrix: row i, column j >= i.
__device__ __forceinline__ void triangle_of(int o, int n, int* i, int* j) {
  int r = (int)(((2.f * n + 1.f) - sqrtf((2.f * n + 1.f) * (2.f * n + 1.f) - 8.f * o)) * 0.5f);
  r = max(0, min(r, n - 1));
  while (r > 0 && r * n - r * (r - 1) / 2 > o) --r;
  while (r + 1 < n && (r + 1) * n - (r + 1) * r / 2 <= o) ++r;
  *i = r;
  *j = r + o - (r * n - r * (r - 1) / 2);
}

__global__ void __launch_bounds__(kFO)
k_gemm_hn_f64(const double2* __restrict__ A, int lda, const double2* __restrict__ B, int ldb, int m, int n, int K,
              int kchunk, int jw, int gram, double2* __restrict__ part) {
  __shared__ double2 sh[kFRows * kFP];
  // columns [j0, j0 + w) of C and, flattened over them, outputs [o0, o1)
  const int j0 = blockIdx.y * jw, w = min(jw, n - j0);
  const int total = gram ? n * (n + 1) / 2 : m * w;
  const int o0 = blockIdx.x * kFO, o1 = min(total, o0 + kFO);
  if (o0 >= o1) return;
  const int o = min(o0 + (int)threadIdx.x, o1 - 1);
  const bool live = o0 + (int)threadIdx.x < o1;
  int i, j, ilo, ihi, jlo, jhi;
  if (gram) {
    int t;
    triangle_of(o, n, &i, &j);
    triangle_of(o0, n, &ilo, &t);
    triangle_of(o1 - 1, n, &ihi, &t);
    jlo = ilo;
    jhi = n - 1;
  } else {
    i = o / w;
    j = j0 + o - i * w;
    ilo = o0 / w;
    ihi = (o1 - 1) / w;
    jlo = j0;
    jhi = j0 + w - 1;
  }
  const int na = ihi - ilo + 1, rows = na + (jhi - jlo + 1);
  const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
  const double2* sa = sh + (i - ilo) * kFP;
  const double2* sb = sh + (na + j - jlo) * kFP;
  const bool warp_live = o0 + (int)(threadIdx.x & ~31u) < o1;
  double re = 0, im = 0;
  for (int k0 = kb; k0 < ke; k0 += kFK) {
    for (int idx = threadIdx.x; idx < rows * kFK; idx += kFO) {
      const int r = idx / kFK, kk = idx % kFK, g = k0 + kk;
      double2 v = make_double2(0, 0);
      if (g < ke) v = r < na ? A[(size_t)(ilo + r) * lda + g] : B[(size_t)(jlo + r - na) * ldb + g];
      sh[r * kFP + kk] = v;
    }
    __syncthreads();
    if (warp_live) {
#pragma unroll
      for (int kk = 0; kk < kFK; ++kk) {
        const double2 a = sa[kk], b = sb[kk];  // conj(a) b
        re = fma(a.x, b.x, re);
        im = fma(a.x, b.y, im);
        re = fma(a.y, b.y, re);
        im = fma(-a.y, b.x, im);
      }
    }
    __syncthreads();
  }
  if (live) {
    double2* P = part + (size_t)blockIdx.z * m * n;
    P[(size_t)i * n + j] = make_double2(re, im);
    if (gram && i != j) P[(size_t)j * n + i] = make_double2(re, -im);
  }
}

// Tiling of an FP64 product: columns a tile, outputs' CTAs, K-splits (a whole number of staged runs
// each) such that about four CTAs are resident on every one of 152 SMs.
struct F64Tiling {
  int jw, nj, no, ns, kchunk, gram;
};
static F64Tiling f64_tiling(int m, int n, int K, bool same) {
  F64Tiling t;
  t.gram = same && m == n && n <= 192;
  t.nj = t.gram ? 1 : ceil_div(n, kFJ);
  t.jw = t.gram ? n : ceil_div(n, t.nj);
  t.no = ceil_div(t.gram ? (long long)n * (n + 1) / 2 : (long long)m * t.jw, kFO);
  const int most = std::max(1, ceil_div(K, 2 * kFK));
  const int s = std::max(1, std::min(ceil_div(4 * 152, t.no * t.nj), most));
  t.kchunk = ceil_div(std::max(K, 1), s);
  t.kchunk = (t.kchunk + kFK - 1) / kFK * kFK;
  t.ns = std::max(1, ceil_div(K, t.kchunk));
  return t;
}

// Sum of the K-split partial tiles: a CTA owns 32 consecutive outputs (one per lane, so
// every split's row segment is one coalesced read); warp w sums the splits s = w, w + 16, ..., and
// the sixteen warp sums are added in warp order (fixed order: the result does not depend on
// scheduling).  FP64 partial tiles are summed in FP64.  The tensor-core kernel's are FP32 values, held
// in FP32 (half the traffic) and summed in double-float on the FP32 pipes: exact sums of FP32 values to
// 48 bits, where the FP64 pipe's conversions and additions of 456 splits of 72 x 64 outputs took 60 us.
constexpr int kRW = 16;  // warps
struct SumF64 {
  double re = 0, im = 0;
  __device__ __forceinline__ void add(double2 v) {
    re += v.x;
    im += v.y;
  }
  __device__ __forceinline__ double2 value() const { return make_double2(re, im); }
};
struct SumDd {
  dd re = dd(0), im = dd(0);
  __device__ __forceinline__ static void add1(dd& a, float v) {
    const dd s = dd_two_sum(a.hi, v);
    a = dd_fast_two_sum(s.hi, __fadd_rn(s.lo, a.lo));
  }
  __device__ __forceinline__ void add(float2 v) {
    add1(re, v.x);
    add1(im, v.y);
  }
  __device__ __forceinline__ double2 value() const { return make_double2(dd_to_double(re), dd_to_double(im)); }
};
template <typename P> struct PartSum { using t = SumF64; };
template <> struct PartSum<float2> { using t = SumDd; };

// The calling CTA's (kRW warps) sum of part[s][idx] over the splits, for each lane's idx (live: whether
// the lane has one); valid in warp 0 after the call's barriers.
template <typename P>
__device__ __forceinline__ double2 sum_parts(const P* __restrict__ part, int nsplit, size_t mn, size_t idx, bool live,
                                             double2 (*acc)[32]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  typename PartSum<P>::t t;
  if (live) {
#pragma unroll 8
    for (int s = w; s < nsplit; s += kRW) t.add(part[(size_t)s * mn + idx]);
  }
  acc[w][lane] = t.value();
  __syncthreads();
  double2 r = make_double2(0, 0);
  if (w == 0) {
    double2 h[kRW / 4];
#pragma unroll
    for (int q = 0; q < kRW / 4; ++q) {
      h[q] = acc[4 * q][lane];
#pragma unroll
      for (int k = 1; k < 4; ++k) h[q] = cadd(h[q], acc[4 * q + k][lane]);
    }
    r = cadd(cadd(h[0], h[1]), cadd(h[2], h[3]));
  }
  return r;
}
template <typename P>
__global__ void __launch_bounds__(32 * kRW)
k_gemm_hn_reduce(const P* __restrict__ part, int nsplit, int m, int n, double2* C, int ldc) {
  __shared__ double2 acc[kRW][32];
  const long long mn = (long long)m * n;
  const long long idx = (long long)blockIdx.x * 32 + (threadIdx.x & 31);
  const double2 t = sum_parts(part, nsplit, (size_t)mn, (size_t)idx, idx < mn, acc);
  if (threadIdx.x < 32 && idx < mn) {
    const int i = (int)(idx / n), j = (int)(idx % n);
    C[(size_t)i * ldc + j] = t;
  }
}

static int gemm_hn_splits(int m, int n, int K) {
  const int tiles = ceil_div(m, kGT) * ceil_div(n, kGT);
  int s = ceil_div(4 * 152, tiles);
  const int smax = ceil_div(K, 512);
  if (s > smax) s = smax;
  if (s < 1) s = 1;
  return s;
}

size_t gemm_hn_work(int m, int n, int K) {
  const int f64 = std::max(f64_tiling(m, n, K, false).ns, f64_tiling(m, n, K, true).ns);
  return (size_t)std::max(std::max(gemm_hn_splits(m, n, K), f64), gemm_hn_tc_splits(m, n, K)) * m * n;
}

// FDE_GEMM_PATH (0, 1 or 3) in the environment sets the initial path.
static int initial_gemm_path() {
  const char* e = getenv("FDE_GEMM_PATH");
  const int p = e ? atoi(e) : 3;
  return (p == 0 || p == 1) ? p : 3;
}
static int g_gemm_path = initial_gemm_path();
void set_gemm_hn_path(int path) { g_gemm_path = (path == 0 || path == 1) ? path : 3; }
int gemm_hn_path() { return g_gemm_path; }
// Set once a tensor-core kernel kept its tensor memory (its MMAs could not be confirmed
// complete): every later product of the process takes the CUDA-core path.
static bool g_tc_disabled = false;
void disable_tensor_cores() { g_tc_disabled = true; }
bool tensor_cores_disabled() { return g_tc_disabled; }

template <typename P>
static void hn_reduce(const P* part, int nsplit, int m, int n, double2* C, int ldc, cudaStream_t st) {
  count_launches(1);
  ProfScope prof_r("k_gemm_hn_reduce", st);
  k_gemm_hn_reduce<P><<<ceil_div((long long)m * n, 32), 32 * kRW, 0, st>>>(part, nsplit, m, n, C, ldc);
}

// The product's partial tiles into work; returns their number (0: m or n is empty).
static int hn_partial(const double2* A, int lda, const double2* B, int ldb, int m, int n, int K, double2* work,
                      cudaStream_t st) {
  // FP64 products stay on the CUDA cores (the part's FP64 tensor rate is no faster)
  const F64Tiling t = f64_tiling(m, n, K, A == B && lda == ldb);
  count_launches(1);
  ProfScope prof_("k_gemm_hn_partial", st);
  k_gemm_hn_f64<<<dim3(t.no, t.nj, t.ns), kFO, 0, st>>>(A, lda, B, ldb, m, n, K, t.kchunk, t.jw, t.gram, work);
  return t.ns;
}
static int hn_partial_f32(const float2* A, int lda, const float2* B, int ldb, int m, int n, int K, double2* work,
                          cudaStream_t st) {
  const int s = gemm_hn_splits(m, n, K);
  int kchunk = ceil_div(K, s);
  kchunk = ((kchunk + kGK - 1) / kGK) * kGK;
  const int ns = ceil_div(K, kchunk > 0 ? kchunk : 1);
  const dim3 grid(ceil_div(m, kGT), ceil_div(n, kGT), ns > 0 ? ns : 1);
  count_launches(1);
  ProfScope prof_("k_gemm_hn_partial", st);
  k_gemm_hn_partial<float, float><<<grid, 256, 0, st>>>(A, lda, B, ldb, m, n, K, kchunk, work);
  return (int)grid.z;
}
// FP32 products go to the tensor cores unless the path or a held tensor memory says otherwise.
static int hn_partial_tc(const float2* A, int lda, const float2* B, int ldb, int m, int n, int K, float2* work,
                         cudaStream_t st) {
  if (g_gemm_path == 0 || g_tc_disabled || K <= 0) return 0;
  return launch_gemm_hn_tc(A, lda, B, ldb, m, n, K, g_gemm_path, work, st);
}

template <>
void launch_gemm_hn<double>(const double2* A, int lda, const double2* B, int ldb, int m, int n, int K, double2* C,
                            int ldc, double2* work, cudaStream_t st) {
  if (m <= 0 || n <= 0) return;
  const int ns = hn_partial(A, lda, B, ldb, m, n, K, work, st);
  hn_reduce(work, ns, m, n, C, ldc, st);
}
template <>
void launch_gemm_hn<float>(const float2* A, int lda, const float2* B, int ldb, int m, int n, int K, double2* C, int ldc,
                           double2* work, cudaStream_t st) {
  if (m <= 0 || n <= 0) return;
  float2* work32 = reinterpret_cast<float2*>(work);
  if (const int ns = hn_partial_tc(A, lda, B, ldb, m, n, K, work32, st)) {
    hn_reduce(work32, ns, m, n, C, ldc, st);
    return;
  }
  const int ns = hn_partial_f32(A, lda, B, ldb, m, n, K, work, st);
  hn_reduce(work, ns, m, n, C, ldc, st);
}

// ---- Y = alpha * U^T-combination of rows of X + beta * Y -----------------------------------
// FP32: a CTA takes 64 plane waves g and 32 or 16 output rows j, each of its threads a JT x 4 block of
// complex sums, so that 16 JT fused multiply-adds stand against 2 + JT / 2 shared-memory reads.  The
// coefficients come in FP64 and are rounded on their bit patterns (the FP64 pipe converts at 1/64
// of the FP32 rate).  72 projectors into 64 bands of 43.7 k plane waves (1.6 GFLOP): 61 us with one plane
// wave and eight rows a thread, 54 us here.
constexpr int kRI = 16;  // input rows a staged tile
constexpr int kRG = 64;  // plane waves a CTA
template <int JT>
__global__ void __launch_bounds__(256, 3)
k_gemm_rot_f32(const float2* __restrict__ X, int ldx, const double2* __restrict__ U, int ldu, int m, int n, int K,
               float2* __restrict__ Y, int ldy, float alpha, float beta) {
  constexpr int JW = 16 * JT;
  __shared__ __align__(16) float2 Xs[kRI][kRG];
  __shared__ __align__(16) float2 Us[kRI][JW];
  const int tg = threadIdx.x & 15, tj = threadIdx.x >> 4;
  const int g0 = blockIdx.x * kRG, j0 = blockIdx.y * JW;
  float re[JT][4], im[JT][4];
#pragma unroll
  for (int a = 0; a < JT; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) re[a][b] = im[a][b] = 0.f;
  constexpr int XL = kRI * kRG / 256, UL = kRI * JW / 256;
  float2 xr[XL], ur[UL];
  const auto load = [&](int i0) {
#pragma unroll
    for (int t = 0; t < XL; ++t) {
      const int idx = threadIdx.x + 256 * t, ii = idx / kRG, gg = idx % kRG;
      xr[t] = (i0 + ii < m && g0 + gg < K) ? X[(size_t)(i0 + ii) * ldx + g0 + gg] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int t = 0; t < UL; ++t) {
      const int idx = threadIdx.x + 256 * t, ii = idx / JW, jj = idx % JW;
      ur[t] = make_float2(0.f, 0.f);
      if (i0 + ii < m && j0 + jj < n) {
        const double2 u = U[(size_t)(i0 + ii) * ldu + j0 + jj];
        ur[t] = make_float2(float_of_double_bits(u.x), float_of_double_bits(u.y));
      }
    }
  };
  load(0);
  for (int i0 = 0; i0 < m; i0 += kRI) {
#pragma unroll
    for (int t = 0; t < XL; ++t) (&Xs[0][0])[threadIdx.x + 256 * t] = xr[t];
#pragma unroll
    for (int t = 0; t < UL; ++t) (&Us[0][0])[threadIdx.x + 256 * t] = ur[t];
    __syncthreads();
    if (i0 + kRI < m) load(i0 + kRI);
    // the tile's own sums first: a small term then rounds against its tile's sum, not against the
    // dominant coefficient's plane wave in the total (an orbital's own row)
    float pr[JT][4], pi[JT][4];
#pragma unroll
    for (int a = 0; a < JT; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) pr[a][b] = pi[a][b] = 0.f;
#pragma unroll
    for (int ii = 0; ii < kRI; ++ii) {
      float2 x[4], u[JT];
      // thread tg owns plane waves 2 tg, 2 tg + 1, 32 + 2 tg, 33 + 2 tg (16-byte reads, every bank once)
      *reinterpret_cast<float4*>(&x[0]) = *reinterpret_cast<const float4*>(&Xs[ii][2 * tg]);
      *reinterpret_cast<float4*>(&x[2]) = *reinterpret_cast<const float4*>(&Xs[ii][32 + 2 * tg]);
      if constexpr (JT == 1) {
        u[0] = Us[ii][tj];
      } else {
#pragma unroll
        for (int a = 0; a < JT; a += 2)
          *reinterpret_cast<float4*>(&u[a]) = *reinterpret_cast<const float4*>(&Us[ii][tj * JT + a]);
      }
#pragma unroll
      for (int a = 0; a < JT; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          pr[a][b] = fmaf(u[a].x, x[b].x, pr[a][b]);
          pi[a][b] = fmaf(u[a].x, x[b].y, pi[a][b]);
          pr[a][b] = fmaf(-u[a].y, x[b].y, pr[a][b]);
          pi[a][b] = fmaf(u[a].y, x[b].x, pi[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < JT; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        re[a][b] += pr[a][b];
        im[a][b] += pi[a][b];
      }
    __syncthreads();
  }
  // every old value is on its way before the first is used: read, added to and written one by one (Y may
  // alias itself as far as the compiler knows) the sixteen of a thread took longer than the sums
  float2 old[JT][4];
  if (beta != 0.f) {
#pragma unroll
    for (int a = 0; a < JT; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int j = j0 + tj * JT + a, g = g0 + (b < 2 ? 2 * tg + b : 30 + 2 * tg + b);
        old[a][b] = (j < n && g < K) ? Y[(size_t)j * ldy + g] : make_float2(0.f, 0.f);
      }
  }
#pragma unroll
  for (int a = 0; a < JT; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = j0 + tj * JT + a, g = g0 + (b < 2 ? 2 * tg + b : 30 + 2 * tg + b);
      if (j >= n || g >= K) continue;
      float2 o = make_float2(alpha * re[a][b], alpha * im[a][b]);
      if (beta != 0.f) {
        o.x += beta * old[a][b].x;
        o.y += beta * old[a][b].y;
      }
      Y[(size_t)j * ldy + g] = o;
    }
}

// FP64: bound by the FP64 pipe's 4 m n K fused multiply-adds (see k_gemm_hn_f64), so a lane owns a
// plane wave and a warp the output rows w, w + 8, ... of the CTA's JW.  A warp runs the loop compiled
// for the rows it has: predicated-off FP64 instructions take the pipe like live ones (one loop for
// eight rows a warp ran 17 bands at a quarter of the rate), and padding to 32 rows nearly doubled
// their work before that.
// 72 projectors into 17 bands of 43.7 k plane waves: 1363 -> 372 us.
template <int Q, int JW>
__device__ __forceinline__ void rot_f64_tile(const double2 (*Xs)[32], const double2 (*Us)[JW], int mi, int lane, int w,
                                             int nw, double* re, double* im) {
  for (int ii = 0; ii < mi; ++ii) {
    const double2 x = Xs[ii][lane];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const double2 u = Us[ii][w + nw * q];
      re[q] = fma(u.x, x.x, re[q]);
      im[q] = fma(u.x, x.y, im[q]);
      re[q] = fma(-u.y, x.y, re[q]);
      im[q] = fma(u.y, x.x, im[q]);
    }
  }
}
template <int JW>
__global__ void __launch_bounds__(256)
k_gemm_rot_f64(const double2* __restrict__ X, int ldx, const double2* __restrict__ U, int ldu, int m, int n, int K,
               double2* __restrict__ Y, int ldy, double alpha, double beta) {
  constexpr int NW = JW < 8 ? JW : 8, Q = JW / NW;  // warps, rows a warp at most
  __shared__ double2 Xs[kRI][32];
  __shared__ double2 Us[kRI][JW];
  // neighbouring CTAs start their rows on other warps: an uneven n spreads over the SM's quarters
  const int lane = threadIdx.x & 31, w = (int)((threadIdx.x >> 5) + blockIdx.x) % NW;
  const int g0 = blockIdx.x * 32, j0 = blockIdx.y * JW;
  const int g = g0 + lane;
  const int rows = min(JW, n - j0), nq = rows > w ? (rows - w + NW - 1) / NW : 0;
  double re[Q], im[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) re[q] = im[q] = 0;
  for (int i0 = 0; i0 < m; i0 += kRI) {
    for (int idx = threadIdx.x; idx < kRI * 32; idx += 32 * NW) {
      const int ii = idx / 32, gg = idx % 32;
      Xs[ii][gg] = (i0 + ii < m && g0 + gg < K) ? X[(size_t)(i0 + ii) * ldx + g0 + gg] : make_double2(0, 0);
    }
    for (int idx = threadIdx.x; idx < kRI * JW; idx += 32 * NW) {
      const int ii = idx / JW, jj = idx % JW;
      Us[ii][jj] = (i0 + ii < m && j0 + jj < n) ? U[(size_t)(i0 + ii) * ldu + j0 + jj] : make_double2(0, 0);
    }
    __syncthreads();
    const int mi = min(kRI, m - i0);
    switch (nq) {
      case 1: rot_f64_tile<1, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 2: if constexpr (Q >= 2) rot_f64_tile<2, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 3: if constexpr (Q >= 3) rot_f64_tile<3, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 4: if constexpr (Q >= 4) rot_f64_tile<4, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 5: if constexpr (Q >= 5) rot_f64_tile<5, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 6: if constexpr (Q >= 6) rot_f64_tile<6, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 7: if constexpr (Q >= 7) rot_f64_tile<7, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
      case 8: if constexpr (Q >= 8) rot_f64_tile<8, JW>(Xs, Us, mi, lane, w, NW, re, im); break;
    }
    __syncthreads();
  }
  if (g >= K) return;
  double2 old[Q];
  if (beta != 0.0) {
#pragma unroll
    for (int q = 0; q < Q; ++q)
      old[q] = q < nq ? Y[(size_t)(j0 + w + NW * q) * ldy + g] : make_double2(0, 0);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if (q >= nq) continue;
    double2 o = make_double2(alpha * re[q], alpha * im[q]);
    if (beta != 0.0) {
      o.x = fma(beta, old[q].x, o.x);
      o.y = fma(beta, old[q].y, o.y);
    }
    Y[(size_t)(j0 + w + NW * q) * ldy + g] = o;
  }
}

static bool gemm_rot_tensor(const float2* X, int ldx, const double2* U, int ldu, int m, int n, int K, float2* Y, int ldy,
                            double alpha, double beta, cudaStream_t st) {
  if (g_gemm_path == 0 || g_tc_disabled || m <= 0) return false;
  return launch_gemm_rot_tc(X, ldx, U, ldu, m, n, K, Y, ldy, alpha, beta, g_gemm_path, st);
}

template <>
void launch_gemm_rot<float>(const float2* X, int ldx, const double2* U, int ldu, int m, int n, int K, float2* Y, int ldy,
                            double alpha, double beta, cudaStream_t st, bool tensor) {
  if (n <= 0 || K <= 0) return;
  if (tensor && gemm_rot_tensor(X, ldx, U, ldu, m, n, K, Y, ldy, alpha, beta, st)) return;
  count_launches(1);
  ProfScope prof_("k_gemm_rot", st);
  const unsigned gx = (unsigned)ceil_div(K, kRG);
  const float a = (float)alpha, b = (float)beta;
  // 32 rows a CTA (three of 80 registers a thread on an SM): 64 rows, four a thread, halve the reads of
  // X but leave one CTA fewer resident and ran at two fifths of the issue rate
  if (n <= 16) k_gemm_rot_f32<1><<<dim3(gx, 1), 256, 0, st>>>(X, ldx, U, ldu, m, n, K, Y, ldy, a, b);
  else k_gemm_rot_f32<2><<<dim3(gx, ceil_div(n, 32)), 256, 0, st>>>(X, ldx, U, ldu, m, n, K, Y, ldy, a, b);
}
template <>
void launch_gemm_rot<double>(const double2* X, int ldx, const double2* U, int ldu, int m, int n, int K, double2* Y,
                             int ldy, double alpha, double beta, cudaStream_t st, bool) {
  if (n <= 0 || K <= 0) return;
  count_launches(1);
  ProfScope prof_("k_gemm_rot", st);
  const int gx = ceil_div(K, 32);
  // rows a CTA: the most (each staged tile of X serves them all) that leave two CTAs for every SM
  const auto fills = [&](int jw) { return (long long)gx * ceil_div(n, jw) >= 2 * 152; };
  if (n > 16 && fills(64)) k_gemm_rot_f64<64><<<dim3(gx, ceil_div(n, 64)), 256, 0, st>>>(X, ldx, U, ldu, m, n, K, Y, ldy, alpha, beta);
  else if (n > 8 && fills(16)) k_gemm_rot_f64<16><<<dim3(gx, ceil_div(n, 16)), 256, 0, st>>>(X, ldx, U, ldu, m, n, K, Y, ldy, alpha, beta);
  else k_gemm_rot_f64<4><<<dim3(gx, ceil_div(n, 4)), 128, 0, st>>>(X, ldx, U, ldu, m, n, K, Y, ldy, alpha, beta);
}

// ---- Cholesky and triangular inverse (one CTA) -------------------------------------------
__global__ void __launch_bounds__(512)
k_cholesky_inv(const double2* __restrict__ S, int n, double2* __restrict__ L, double2* __restrict__ Li,
               unsigned* status, double rel_pivot) {
  __shared__ int fail;
  if (threadIdx.x == 0) fail = 0;
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int i = idx / n, j = idx % n;
    L[idx] = (j <= i) ? S[idx] : make_double2(0, 0);
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const double d = L[(size_t)j * n + j].x;
    if (!(d > rel_pivot * S[(size_t)j * n + j].x)) {
      if (threadIdx.x == 0) {
        fail = 1;
        atomicOr(status, ST_CHOLESKY);
        status[1] = (unsigned)j;
      }
      break;
    }
    const double sd = sqrt(d);
    const double inv = 1.0 / sd;
    __syncthreads();
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) {
      double2 v = L[(size_t)i * n + j];
      v.x *= inv;
      v.y *= inv;
      L[(size_t)i * n + j] = v;
    }
    if (threadIdx.x == 0) L[(size_t)j * n + j] = make_double2(sd, 0.0);
    __syncthreads();
    const int rem = n - j - 1;
    for (int idx = threadIdx.x; idx < rem * rem; idx += blockDim.x) {
      const int i = j + 1 + idx / rem, k = j + 1 + idx % rem;
      if (k <= i) {
        const double2 a = L[(size_t)i * n + j], b = L[(size_t)k * n + j];
        double2 v = L[(size_t)i * n + k];
        // v -= a * conj(b)
        v.x -= a.x * b.x + a.y * b.y;
        v.y -= a.y * b.x - a.x * b.y;
        L[(size_t)i * n + k] = v;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  if (fail) return;
  // Li = L^{-1}: column c by forward substitution, one warp per column (lanes share the
  // inner products).
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int c = threadIdx.x >> 5; c < n; c += nw) {
    for (int i = lane; i < c; i += 32) Li[(size_t)i * n + c] = make_double2(0, 0);
    for (int i = c; i < n; ++i) {
      double re = 0.0, im = 0.0;
      for (int k = c + lane; k < i; k += 32) {
        const double2 l = L[(size_t)i * n + k], x = Li[(size_t)k * n + c];
        re += l.x * x.x - l.y * x.y;
        im += l.x * x.y + l.y * x.x;
      }
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (lane == 0) {
        const double dd = L[(size_t)i * n + i].x;
        Li[(size_t)i * n + c] = make_double2(((i == c) ? 1.0 : 0.0) - re, -im);
        Li[(size_t)i * n + c].x /= dd;
        Li[(size_t)i * n + c].y /= dd;
      }
      __syncwarp();
    }
  }
}

// The cluster-distributed factorisation (dense.cu) when n fits it, else one CTA.
void launch_cholesky_inv(const double2* S, int n, double2* L, double2* Linv, unsigned* status, double rel_pivot,
                         cudaStream_t st) {
  if (launch_cholesky_cluster(S, n, L, Linv, status, rel_pivot, st)) return;
  count_launches(1);
  k_cholesky_inv<<<1, 512, 0, st>>>(S, n, L, Linv, status, rel_pivot);
}

// ---- per-atom projector coupling ------------------------------------------------------------
// <beta|psi> and its coupling in one pass over the partial tiles: the CTA sums the K-splits of one
// atom's np rows and 32 columns (as k_gemm_hn_reduce) and applies the atom's np x np block,
// Q[a np + i][b] = sum_j D[i][j] P[a np + j][b] -- the same block for every atom (Datom null) or its own
// (screened couplings of ultrasoft-like atoms, Datom [natoms][np][np]).  The coupling of Eq. KB
// (nonlocal part) is block diagonal and needs no dense product.
template <typename P>
__global__ void __launch_bounds__(32 * kRW)
k_gemm_hn_couple(const P* __restrict__ part, int nsplit, KbBlock D, const double* __restrict__ Datom, int natoms, int nb,
                 double2* __restrict__ Q) {
  __shared__ double2 acc[kRW][32], sum[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int a = blockIdx.y, b = blockIdx.x * 32 + lane, np = D.np;
  const size_t mn = (size_t)natoms * np * nb;
  for (int i = 0; i < np; ++i) {
    const double2 t = sum_parts(part, nsplit, mn, (size_t)(a * np + i) * nb + b, b < nb, acc);
    if (w == 0) sum[i][lane] = t;
    __syncthreads();
  }
  if (b >= nb) return;
  const double* d = Datom ? Datom + (size_t)a * np * np : nullptr;
  for (int i = w; i < np; i += kRW) {
    double re = 0, im = 0;
    for (int j = 0; j < np; ++j) {
      const double c = d ? d[i * np + j] : D.d[i * np + j];
      const double2 p = sum[j][lane];
      re += c * p.x;
      im += c * p.y;
    }
    Q[(size_t)(a * np + i) * nb + b] = make_double2(re, im);
  }
}

template <typename P>
static void hn_couple(const P* part, int ns, const KbBlock& D, const double* Datom, int natoms, int nb, double2* Q,
                      cudaStream_t st) {
  count_launches(1);
  ProfScope prof_("k_kb_couple", st);
  k_gemm_hn_couple<P><<<dim3(ceil_div(nb, 32), natoms), 32 * kRW, 0, st>>>(part, ns, D, Datom, natoms, nb, Q);
}

template <>
void launch_project_couple<double>(const double2* beta, const double2* psi, int ld, int K, const KbBlock& D,
                                   const double* Datom, int natoms, int nb, double2* Q, double2* work, cudaStream_t st) {
  if (natoms <= 0 || nb <= 0) return;
  const int ns = hn_partial(beta, ld, psi, ld, natoms * D.np, nb, K, work, st);
  hn_couple(work, ns, D, Datom, natoms, nb, Q, st);
}
template <>
void launch_project_couple<float>(const float2* beta, const float2* psi, int ld, int K, const KbBlock& D,
                                  const double* Datom, int natoms, int nb, double2* Q, double2* work, cudaStream_t st) {
  if (natoms <= 0 || nb <= 0) return;
  float2* work32 = reinterpret_cast<float2*>(work);
  if (const int ns = hn_partial_tc(beta, ld, psi, ld, natoms * D.np, nb, K, work32, st)) {
    hn_couple(work32, ns, D, Datom, natoms, nb, Q, st);
    return;
  }
  const int ns = hn_partial_f32(beta, ld, psi, ld, natoms * D.np, nb, K, work, st);
  hn_couple(work, ns, D, Datom, natoms, nb, Q, st);
}

__global__ void k_hermitize(double2* A, int n) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * n) return;
  const int i = idx / n, j = idx % n;
  if (j < i) return;
  const double2 a = A[(size_t)i * n + j], b = A[(size_t)j * n + i];
  const double2 h = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
  A[(size_t)i * n + j] = h;
  A[(size_t)j * n + i] = make_double2(h.x, -h.y);
  if (i == j) A[(size_t)i * n + i].y = 0.0;
}

void launch_hermitize(double2* A, int n, cudaStream_t st) {
  count_launches(1);
  k_hermitize<<<ceil_div((long long)n * n, 256), 256, 0, st>>>(A, n);
}

// ---- row-wise helpers ----------------------------------------------------------------------
template <typename T>
__global__ void k_residual(const cplx<T>* __restrict__ HX, const cplx<T>* __restrict__ X, const double* eps, int K,
                           int ld, cplx<T>* __restrict__ R, int ldr) {
  const int j = blockIdx.y;
  const T e = (T)eps[j];
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < K; g += gridDim.x * blockDim.x) {
    const cplx<T> h = HX[(size_t)j * ld + g], x = X[(size_t)j * ld + g];
    R[(size_t)j * ldr + g] = mk<T>(h.x - e * x.x, h.y - e * x.y);
  }
}

template <typename T>
void launch_residual(const cplx<T>* HX, const cplx<T>* X, const double* eps, int nb, int K, int ld, cplx<T>* R,
                     int ldr, cudaStream_t st) {
  if (nb <= 0) return;
  count_launches(1);
  k_residual<T><<<dim3(ceil_div(K, 256 * 4), nb), 256, 0, st>>>(HX, X, eps, K, ld, R, ldr);
}

// out[j] = sum_g weight[g] |X[j][g]|^2 (weight NULL: 1); one CTA per row, fixed order.
template <typename T>
__global__ void k_row_norms(const cplx<T>* __restrict__ X, int ld, int K, const T* __restrict__ weight,
                            double* out) {
  __shared__ double red[32];
  const int j = blockIdx.x;
  double acc = 0;
  for (int g = threadIdx.x; g < K; g += blockDim.x) {
    const cplx<T> x = X[(size_t)j * ld + g];
    const double m2 = (double)x.x * x.x + (double)x.y * x.y;
    acc += weight ? (double)weight[g] * m2 : m2;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    out[j] = t;
  }
}

template <typename T>
void launch_row_norms(const cplx<T>* X, int ld, int nb, int K, const T* weight, double* out, double*,
                      cudaStream_t st) {
  if (nb <= 0) return;
  count_launches(1);
  k_row_norms<T><<<nb, 512, 0, st>>>(X, ld, K, weight, out);
}

// Teter-Payne-Allan kinetic preconditioner: W = K(x) R with x = |k+G|^2/2 / T_band,
// K(x) = (27 + 18x + 12x^2 + 8x^3) / (27 + 18x + 12x^2 + 8x^3 + 16x^4).
template <typename T>
__global__ void k_tpa(const cplx<T>* __restrict__ R, int ldr, const T* __restrict__ kin, const double* tband, int K,
                      cplx<T>* __restrict__ W, int ldw) {
  const int j = blockIdx.y;
  const T tb = (T)fmax(tband[j], 1e-12);
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < K; g += gridDim.x * blockDim.x) {
    const T x = kin[g] / tb;
    const T p = (T)27 + x * ((T)18 + x * ((T)12 + x * (T)8));
    const T f = p / (p + (T)16 * x * x * x * x);
    const cplx<T> r = R[(size_t)j * ldr + g];
    W[(size_t)j * ldw + g] = mk<T>(f * r.x, f * r.y);
  }
}

template <typename T>
void launch_tpa(const cplx<T>* R, int ldr, const T* kin, const double* tband, int nb, int K, cplx<T>* W, int ldw,
                cudaStream_t st) {
  if (nb <= 0) return;
  count_launches(1);
  k_tpa<T><<<dim3(ceil_div(K, 256 * 4), nb), 256, 0, st>>>(R, ldr, kin, tband, K, W, ldw);
}

template <typename T>
__global__ void k_scale_rows(cplx<T>* X, int ld, int K, const double* s) {
  const int j = blockIdx.y;
  const T f = (T)s[j];
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < K; g += gridDim.x * blockDim.x) {
    cplx<T> x = X[(size_t)j * ld + g];
    x.x *= f;
    x.y *= f;
    X[(size_t)j * ld + g] = x;
  }
}

template <typename T>
void launch_scale_rows(cplx<T>* X, int ld, int nb, int K, const double* s, cudaStream_t st) {
  if (nb <= 0) return;
  count_launches(1);
  k_scale_rows<T><<<dim3(ceil_div(K, 256 * 4), nb), 256, 0, st>>>(X, ld, K, s);
}

template <typename Ta, typename Tb>
__global__ void k_convert_c(const cplx<Ta>* a, cplx<Tb>* b, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = mk<Tb>((Tb)a[i].x, (Tb)a[i].y);
}

template <typename Ta, typename Tb>
void launch_convert_c(const cplx<Ta>* a, cplx<Tb>* b, size_t n, cudaStream_t st) {
  if (!n) return;
  count_launches(1);
  k_convert_c<Ta, Tb><<<(int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, st>>>(a, b, n);
}

template <typename T>
__global__ void k_shape_init(cplx<T>* X, int ld, const T* kin, int K) {
  const int j = blockIdx.y;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < K; g += gridDim.x * blockDim.x) {
    cplx<T> x = X[(size_t)j * ld + g];
    const T f = (T)1 / ((T)1 + kin[g]);
    x.x *= f;
    x.y *= f;
    X[(size_t)j * ld + g] = x;
  }
}

template <typename T>
void launch_shape_init(cplx<T>* X, int ld, const T* kin, int nb, int K, cudaStream_t st) {
  if (nb <= 0) return;
  count_launches(1);
  k_shape_init<T><<<dim3(ceil_div(K, 256 * 4), nb), 256, 0, st>>>(X, ld, kin, K);
}

#define FDE_INST_T(T)                                                                                            \
  template void launch_residual<T>(const cplx<T>*, const cplx<T>*, const double*, int, int, int, cplx<T>*, int,  \
                                   cudaStream_t);                                                                \
  template void launch_row_norms<T>(const cplx<T>*, int, int, int, const T*, double*, double*, cudaStream_t);    \
  template void launch_tpa<T>(const cplx<T>*, int, const T*, const double*, int, int, cplx<T>*, int,             \
                              cudaStream_t);                                                                     \
  template void launch_scale_rows<T>(cplx<T>*, int, int, int, const double*, cudaStream_t);                      \
  template void launch_shape_init<T>(cplx<T>*, int, const T*, int, int, cudaStream_t);
FDE_INST_T(float)
FDE_INST_T(double)
template void launch_convert_c<double, float>(const double2*, float2*, size_t, cudaStream_t);
template void launch_convert_c<float, double>(const float2*, double2*, size_t, cudaStream_t);
template void launch_convert_c<double, double>(const double2*, double2*, size_t, cudaStream_t);

}  // namespace fde
