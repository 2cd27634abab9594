// hpsi2.cuh -- H psi and band-density kernels on two-step transforms (fft2.cuh), for grids whose
// three lengths have a two-step plan.  Same data flow as hpsi.cu, whose runtime-length kernels
// serve every other grid; each precision is instantiated by its own translation units.
#pragma once

#include "dd.cuh"
#include "fft2.cuh"
#include "kernels.h"
#include "prof.h"

#include <algorithm>

namespace fde {

// Launches a kernel whose shared memory is computed when it runs, and returns the launch's own status: a
// refused launch leaves no other trace, and the passes after it would run on the data of the one before.
// The dynamic shared memory a kernel may be launched with is a property of the kernel, shared by every
// thread that launches it, so it is always set to the most a CTA can have: set to the bytes of one
// launch, it could be lowered between another thread's setting and launch, which is then refused.
constexpr size_t kCtaSmemMax = 232448;  // 227 KB
template <typename... A, typename... B>
inline cudaError_t launch_sized(void (*kernel)(A...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                const B&... args) {
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCtaSmemMax);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  count_launches(1);
  return cudaLaunchKernelEx(&cfg, kernel, A(args)...);
}

// Every (subsystem, k) block of bands is an item; the kernels below run a batch of items in
// one launch (the batch travels as a kernel parameter), so subsystems of uneven size share
// the GPU instead of taking one small launch each.  The first z-block and the first plane
// block of each item are prefix offsets; a CTA finds its item by scanning the table.
template <typename T> struct HpsiItem {
  SphereDev sp;
  const cplx<T>* psi;
  cplx<T>* hpsi;
  const T* kin;
  const T* vplane;
  cplx<T>* scratch;  // [nb][n3][ldc]
  int ld, nb, zstart, pstart;
};
constexpr int kBatchMax = 24;
template <typename T> struct HpsiBatch {
  int n;
  HpsiItem<T> it[kBatchMax];
};

template <typename T>
__device__ __forceinline__ int batch_item(const HpsiBatch<T>& B, int blk, bool plane) {
  int i = 0;
  for (int j = 1; j < B.n; ++j)
    if ((plane ? B.it[j].pstart : B.it[j].zstart) <= blk) i = j;
  return i;
}

// Position of grid index i in a run of len consecutive (signed) indices that starts at grid index
// lo, modulo n; len or more when it is outside the run.
__device__ __forceinline__ int run_offset(int i, int lo, int n) {
  const int d = i - lo;
  return d < 0 ? d + n : d;
}

// ---- z passes ------------------------------------------------------------------------------------
// A CTA takes the z lines of neighbouring sphere columns, as many as fill 128 bytes of a scratch
// row, so both global sides of the pass are whole 128-byte lines and nothing but the exchange
// between the two steps goes through shared memory: step 1 reads the columns' runs of plane waves
// (neighbouring items on neighbouring G), step 2 writes one scratch row per 16 (FP32) lanes.
template <typename T> __host__ __device__ constexpr int z_cols() { return 128 / (int)sizeof(cplx<T>); }
// Exchange pitch of a line: odd, so that the lanes of one column index lie on different banks; with
// an odd second radix also congruent to it modulo 16, which keeps step 1's runs apart too.
__host__ __device__ constexpr int z_pitch(int n, int r2) {
  int p = n | 1;
  if (r2 & 1)
    while (p % 16 != r2 % 16) p += 2;
  return p;
}
template <typename T, int R1, int R2> __host__ __device__ constexpr int z_threads() {
  return round_up(z_cols<T>() * (R1 > R2 ? R1 : R2), 32);
}

template <typename T, int R1, int R2>
__global__ void __launch_bounds__(z_threads<T, R1, R2>())
k_zinv_cols(const __grid_constant__ HpsiBatch<T> B, const cplx<T>* __restrict__ tw) {
  using C = cplx<T>;
  constexpr int N = R1 * R2, ZC = z_cols<T>(), XP = z_pitch(N, R2), NT = z_threads<T, R1, R2>();
  __shared__ __align__(16) C X[ZC * XP];
  const HpsiItem<T>& I = B.it[batch_item(B, blockIdx.x, false)];
  const SphereDev& sp = I.sp;
  const int ntile = (sp.ncol + ZC - 1) / ZC;
  const int local = blockIdx.x - I.zstart;
  const int b = local / ntile, c0 = (local - b * ntile) * ZC;
  const C* src = I.psi + (size_t)b * I.ld;
  for (int w = threadIdx.x; w < ZC * R2; w += NT) {
    const int c = w / R2, j = w - c * R2;
    const int col = c0 + c;
    C v[R1];
    if (col < sp.ncol) {
      const int s = sp.col_start[col], len = sp.col_start[col + 1] - s;
      int lo = sp.col_m3lo[col] % N;
      lo += lo < 0 ? N : 0;
#pragma unroll
      for (int r = 0; r < R1; ++r) {
        const int d = run_offset(j + r * R2, lo, N);
        v[r] = d < len ? src[s + d] : mk<T>(0, 0);
      }
      dft_r<R1>(v, +1);
#pragma unroll
      for (int q = 0; q < R1; ++q) X[c * XP + q * R2 + j] = v[q];
    }
  }
  __syncthreads();
  C* dst = I.scratch + (size_t)b * N * sp.ldc + c0;
  for (int w = threadIdx.x; w < R1 * ZC; w += NT) {
    const int q = w / ZC, c = w - q * ZC;
    if (c0 + c < sp.ncol) {
      C v[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) {
        v[j] = X[c * XP + q * R2 + j];
        if (j) v[j] = twist(v[j], tw[j * q], +1);
      }
      dft_r<R2>(v, +1);
#pragma unroll
      for (int p = 0; p < R2; ++p) dst[(size_t)(q + R1 * p) * sp.ldc + c] = v[p];
    }
  }
}

template <typename T, int R1, int R2>
__global__ void __launch_bounds__(z_threads<T, R1, R2>())
k_zfwd_cols(const __grid_constant__ HpsiBatch<T> B, T inv_nr, const cplx<T>* __restrict__ tw) {
  using C = cplx<T>;
  constexpr int N = R1 * R2, ZC = z_cols<T>(), XP = z_pitch(N, R2), NT = z_threads<T, R1, R2>();
  __shared__ __align__(16) C X[ZC * XP];
  const HpsiItem<T>& I = B.it[batch_item(B, blockIdx.x, false)];
  const SphereDev& sp = I.sp;
  const int ntile = (sp.ncol + ZC - 1) / ZC;
  const int local = blockIdx.x - I.zstart;
  const int b = local / ntile, c0 = (local - b * ntile) * ZC;
  const C* src = I.scratch + (size_t)b * N * sp.ldc + c0;
  for (int w = threadIdx.x; w < R1 * ZC; w += NT) {
    const int q = w / ZC, c = w - q * ZC;
    if (c0 + c < sp.ncol) {
      C v[R2];
#pragma unroll
      for (int p = 0; p < R2; ++p) v[p] = src[(size_t)(q + R1 * p) * sp.ldc + c];
      dft_r<R2>(v, -1);
#pragma unroll
      for (int j = 0; j < R2; ++j) X[c * XP + q * R2 + j] = j ? twist(v[j], tw[j * q], -1) : v[j];
    }
  }
  __syncthreads();
  const C* ps = I.psi + (size_t)b * I.ld;
  C* hs = I.hpsi + (size_t)b * I.ld;
  for (int w = threadIdx.x; w < ZC * R2; w += NT) {
    const int c = w / R2, j = w - c * R2;
    const int col = c0 + c;
    if (col < sp.ncol) {
      const int s = sp.col_start[col], len = sp.col_start[col + 1] - s;
      int lo = sp.col_m3lo[col] % N;
      lo += lo < 0 ? N : 0;
      C v[R1];
#pragma unroll
      for (int q = 0; q < R1; ++q) v[q] = X[c * XP + q * R2 + j];
      dft_r<R1>(v, -1);
#pragma unroll
      for (int r = 0; r < R1; ++r) {
        const int d = run_offset(j + r * R2, lo, N);
        if (d < len) {
          const C x = ps[s + d];
          const T kk = I.kin[s + d];
          hs[s + d] = mk<T>(v[r].x * inv_nr + kk * x.x, v[r].y * inv_nr + kk * x.y);
        }
      }
    }
  }
}

// ---- plane pass ----------------------------------------------------------------------------------
// One CTA per (item, band, z-plane).  Shared memory holds the plane's data rows only -- the
// span of m1 the sphere covers, P[row][N2], odd pitch -- and X, which carries the sphere columns
// in and out and the exchange of the x transforms of LB columns at a time:
//   columns -> X (coalesced) ; y inverse, step 1 X -> P, step 2 within P ;
//   for each batch of LB columns: x inverse step 1 (rows of P -> X; rows outside the span are
//   zero and never stored), step 2, the product with the potential and the forward transform's
//   first step on the same registers (X in place: an item rewrites the slots it read), the
//   forward's second step (X -> rows of P; rows outside the span are never computed into
//   memory) ; y forward within P, then P -> X ; X -> columns (coalesced).
// Item (j, c) of a batch's last step reads the X slots that item (j, c) of the next batch's
// first step writes, and rewrites the P column it read: two barriers per batch.
// Lanes run over rows in the y steps and over columns in the x steps, so every access but the
// row ends is free of bank conflicts.
struct PlaneDims {
  int n1s, n2s;   // span of m1 (rows of P) and of m2
  int lo1, lo2;   // grid index of the first row and column
  int W;          // X pitch of the column stage (odd)
  unsigned inv;   // row_inv(n1s): w / n1s = w inv >> 20 for w < 2^20 / n1s
};
__device__ __forceinline__ unsigned row_inv(int n1s) { return (1u << 20) / (unsigned)n1s + 1u; }

// Offset of the span's first index from element 0 of item j: element r sits at d = wrap(base + R2 r) of
// the span, inside it when d < span.
template <typename Plan> __device__ __forceinline__ int span_base(int j, int lo) {
  const int b = Plan::in0(j) - lo;
  return b < 0 ? b + Plan::N : b;
}

// Inverse y transforms: step 1 takes the columns from X to the rows of P, step 2 runs within P.
template <typename T, typename Plan>
__device__ __forceinline__ void plane_y_inv_1(cplx<T>* P, const cplx<T>* X, const PlaneDims& D, int pitch, int nt) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2;
  for (int w = threadIdx.x; w < D.n1s * R2; w += nt) {
    const int j = (int)(((unsigned)w * D.inv) >> 20), r = w - j * D.n1s;
    const int base = span_base<Plan>(j, D.lo2);
    const C* x = X + r * D.W;
    C v[R1];
#pragma unroll
    for (int q = 0; q < R1; ++q) {
      const int d = Plan::wrap(base + q * R2);
      v[q] = d < D.n2s ? x[d] : mk<T>(0, 0);
    }
    dft_r<R1>(v, +1);
    C* o = P + r * pitch;
    const int oj = Plan::out(j);
#pragma unroll
    for (int q = 0; q < R1; ++q) o[Plan::wrap(Plan::out0(q) + oj)] = v[q];
  }
}
template <typename T, typename Plan>
__device__ __forceinline__ void plane_y_inv_2(cplx<T>* P, const PlaneDims& D, int pitch, int nt,
                                              const cplx<T>* __restrict__ tw) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2;
  for (int w = threadIdx.x; w < D.n1s * R1; w += nt) {
    const int q = (int)(((unsigned)w * D.inv) >> 20), r = w - q * D.n1s;
    C* o = P + r * pitch;
    C v[R2];
#pragma unroll
    for (int j = 0; j < R2; ++j) {
      v[j] = o[Plan::output(q, j)];
      if (!Plan::kCoprime && j) v[j] = twist(v[j], tw[j * q], +1);
    }
    dft_r<R2>(v, +1);
#pragma unroll
    for (int p = 0; p < R2; ++p) o[Plan::output(q, p)] = v[p];
  }
}

// Forward y transforms: the same steps backwards.
template <typename T, typename Plan>
__device__ __forceinline__ void plane_y_fwd_2(cplx<T>* P, const PlaneDims& D, int pitch, int nt,
                                              const cplx<T>* __restrict__ tw) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2;
  for (int w = threadIdx.x; w < D.n1s * R1; w += nt) {
    const int q = (int)(((unsigned)w * D.inv) >> 20), r = w - q * D.n1s;
    C* o = P + r * pitch;
    C v[R2];
#pragma unroll
    for (int p = 0; p < R2; ++p) v[p] = o[Plan::output(q, p)];
    dft_r<R2>(v, -1);
#pragma unroll
    for (int j = 0; j < R2; ++j) o[Plan::output(q, j)] = (!Plan::kCoprime && j) ? twist(v[j], tw[j * q], -1) : v[j];
  }
}
template <typename T, typename Plan>
__device__ __forceinline__ void plane_y_fwd_1(const cplx<T>* P, cplx<T>* X, const PlaneDims& D, int pitch, int nt) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2;
  for (int w = threadIdx.x; w < D.n1s * R2; w += nt) {
    const int j = (int)(((unsigned)w * D.inv) >> 20), r = w - j * D.n1s;
    const C* o = P + r * pitch;
    const int oj = Plan::out(j);
    C v[R1];
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = o[Plan::wrap(Plan::out0(q) + oj)];
    dft_r<R1>(v, -1);
    const int base = span_base<Plan>(j, D.lo2);
    C* x = X + r * D.W;
#pragma unroll
    for (int q = 0; q < R1; ++q) {
      const int d = Plan::wrap(base + q * R2);
      if (d < D.n2s) x[d] = v[q];
    }
  }
}

// The x steps of all columns, lb at a time (lb max(R1, R2) <= nt: one item a thread and step).  What a
// thread's item needs -- the rows of its step-1 inputs, the potential's rows of its outputs, its
// twiddles -- depends on the item alone, so it is found once and kept over the batches.
// Step 1: rows of P into X[slot][c], slot = j R1 + q.  Step 2, the potential and the forward's first step:
// X in place.  The forward's second step: X back into the rows of P.
template <typename T, typename Plan>
struct XItem {
  int row[Plan::R1];  // step 1: offset in P of the item's element r, or -1 outside the span
  __device__ __forceinline__ void rows(const PlaneDims& D, int j, int c, int pitch) {
    const int base = span_base<Plan>(j, D.lo1);
#pragma unroll
    for (int q = 0; q < Plan::R1; ++q) {
      const int d = Plan::wrap(base + q * Plan::R2);
      row[q] = d < D.n1s ? d * pitch + c : -1;
    }
  }
};
template <typename T, typename Plan>
__device__ __forceinline__ void plane_x_in(const cplx<T>* P, cplx<T>* X, const XItem<T, Plan>& I, int j, int c, int c0,
                                           int lb) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1;
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = I.row[q] >= 0 ? P[I.row[q] + c0] : mk<T>(0, 0);
  dft_r<R1>(v, +1);
#pragma unroll
  for (int q = 0; q < R1; ++q) X[(j * R1 + q) * lb + c] = v[q];
}
template <typename T, typename Plan>
__device__ __forceinline__ void plane_x_out(cplx<T>* P, const cplx<T>* X, const XItem<T, Plan>& I, int j, int c, int c0,
                                            int lb) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1;
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = X[(j * R1 + q) * lb + c];
  dft_r<R1>(v, -1);
#pragma unroll
  for (int q = 0; q < R1; ++q)
    if (I.row[q] >= 0) P[I.row[q] + c0] = v[q];
}
template <typename T, typename Plan>
__device__ __forceinline__ void plane_x_all(cplx<T>* P, cplx<T>* X, const PlaneDims& D, int pitch, int n2, int lb,
                                            const cplx<T>* __restrict__ tw, const T* __restrict__ vp) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2;
  const int tid = threadIdx.x, j = tid / lb, c = tid - j * lb;  // the same pair serves both item kinds
  const bool in1 = j < R2, in2 = j < R1;
  XItem<T, Plan> I;
  if (in1) I.rows(D, j, c, pitch);
  int vo[R2];
  C t[Plan::kCoprime ? 1 : R2];
#pragma unroll
  for (int p = 0; p < R2; ++p) {
    vo[p] = Plan::output(j, p) * n2 + c;
    if constexpr (!Plan::kCoprime)
      if (p && in2) t[p] = tw[p * j];
  }
#pragma unroll 1
  for (int c0 = 0; c0 < n2; c0 += lb) {
    const bool have = c < n2 - c0;
    if (in1 && have) plane_x_in<T, Plan>(P, X, I, j, c, c0, lb);
    __syncthreads();
    if (in2 && have) {
      C v[R2];
#pragma unroll
      for (int p = 0; p < R2; ++p) {
        v[p] = X[(p * R1 + j) * lb + c];
        if constexpr (!Plan::kCoprime)
          if (p) v[p] = twist(v[p], t[p], +1);
      }
      dft_r<R2>(v, +1);
#pragma unroll
      for (int p = 0; p < R2; ++p) {
        const T s = vp[vo[p] + c0];
        v[p].x *= s;
        v[p].y *= s;
      }
      dft_r<R2>(v, -1);
#pragma unroll
      for (int p = 0; p < R2; ++p) {
        if constexpr (!Plan::kCoprime)
          if (p) v[p] = cmul(v[p], t[p]);
        X[(p * R1 + j) * lb + c] = v[p];
      }
    }
    __syncthreads();
    if (in1 && have) plane_x_out<T, Plan>(P, X, I, j, c, c0, lb);
  }
}

template <typename T>
__device__ __forceinline__ PlaneDims plane_dims(const SphereDev& sp) {
  return PlaneDims{sp.span1, sp.span2, sp.lo1, sp.lo2, sp.span2 | 1, row_inv(sp.span1)};
}
// Sphere columns of one plane into X[row][m2 - lo2] (slots without a column are zero), and back; RUNS: the
// columns of D.n1s rows alone, whose first slot is p0.
template <typename T, bool RUNS>
__device__ __forceinline__ void plane_columns_in(cplx<T>* X, const cplx<T>* __restrict__ S, const SphereDev& sp,
                                                 const PlaneDims& D, int p0, int nt) {
  const int n = D.n1s * D.W;
  for (int i = threadIdx.x; i < n; i += nt) X[i] = mk<T>(0, 0);
  __syncthreads();
  for (int c = threadIdx.x; c < sp.ncol; c += nt) {
    const int i = RUNS ? sp.col_pos[c] - p0 : sp.col_pos[c];
    if (!RUNS || (i >= 0 && i < n)) X[i] = S[c];
  }
}
template <typename T, bool RUNS>
__device__ __forceinline__ void plane_columns_out(const cplx<T>* X, cplx<T>* __restrict__ S, const SphereDev& sp,
                                                  const PlaneDims& D, int p0, int nt) {
  const int n = D.n1s * D.W;
  for (int c = threadIdx.x; c < sp.ncol; c += nt) {
    const int i = RUNS ? sp.col_pos[c] - p0 : sp.col_pos[c];
    if (!RUNS || (i >= 0 && i < n)) S[c] = X[i];
  }
}

// Columns -> X -> y inverse transforms in P, and back.  RUNS: X holds the columns of `rows` rows at a
// time, for spheres so wide that those of all rows do not fit beside P.  The alternative is the
// runtime-length kernels.  H psi on n x n x 96, FP32, n = 144, 32 bands, spans of 114 / 128 / 142: 6.08 /
// 6.76 / 7.58 ms there, 0.84 / 1.00 / 1.34 ms in runs; FP64, n = 96, 16 bands, spans of 88 / 94: 5.42 / 5.82
// and 2.83 / 3.06 ms.
template <typename T, typename Plan, bool RUNS>
__device__ __forceinline__ void plane_in(cplx<T>* P, cplx<T>* X, const cplx<T>* __restrict__ S, const SphereDev& sp,
                                         const PlaneDims& D, int rows, int pitch, int nt,
                                         const cplx<T>* __restrict__ tw) {
  if constexpr (!RUNS) {
    plane_columns_in<T, false>(X, S, sp, D, 0, nt);
    __syncthreads();
    plane_y_inv_1<T, Plan>(P, X, D, pitch, nt);
  } else {
#pragma unroll 1
    for (int r0 = 0; r0 < D.n1s; r0 += rows) {
      PlaneDims R = D;
      R.n1s = min(rows, D.n1s - r0);
      R.inv = row_inv(R.n1s);
      if (r0) __syncthreads();  // the rows before have left X
      plane_columns_in<T, true>(X, S, sp, R, r0 * D.W, nt);
      __syncthreads();
      plane_y_inv_1<T, Plan>(P + r0 * pitch, X, R, pitch, nt);
    }
  }
  __syncthreads();
  plane_y_inv_2<T, Plan>(P, D, pitch, nt, tw);
}
template <typename T, typename Plan, bool RUNS>
__device__ __forceinline__ void plane_out(cplx<T>* P, cplx<T>* X, cplx<T>* __restrict__ S, const SphereDev& sp,
                                          const PlaneDims& D, int rows, int pitch, int nt,
                                          const cplx<T>* __restrict__ tw) {
  plane_y_fwd_2<T, Plan>(P, D, pitch, nt, tw);
  __syncthreads();
  if constexpr (!RUNS) {
    plane_y_fwd_1<T, Plan>(P, X, D, pitch, nt);
    __syncthreads();
    plane_columns_out<T, false>(X, S, sp, D, 0, nt);
  } else {
#pragma unroll 1
    for (int r0 = 0; r0 < D.n1s; r0 += rows) {
      PlaneDims R = D;
      R.n1s = min(rows, D.n1s - r0);
      R.inv = row_inv(R.n1s);
      if (r0) __syncthreads();
      plane_y_fwd_1<T, Plan>(P + r0 * pitch, X, R, pitch, nt);
      __syncthreads();
      plane_columns_out<T, true>(X, S, sp, R, r0 * D.W, nt);
    }
  }
}

// Columns a batch of the x transforms takes: as many as let about NT threads hold one butterfly
// each, spread evenly over the batches.
__host__ __device__ constexpr int plane_batch(int n2, int rmax, int nt) {
  int lb = nt / rmax;
  if (lb < 1) lb = 1;
  if (lb > n2) lb = n2;
  const int nb = (n2 + lb - 1) / lb;
  return (n2 + nb - 1) / nb;
}

template <typename T, typename PX, typename PY, int NT, int MINB, bool RUNS>
__global__ void __launch_bounds__(NT, MINB)
k_plane_pass(const __grid_constant__ HpsiBatch<T> B, int n3, const cplx<T>* __restrict__ tw1,
             const cplx<T>* __restrict__ tw2, int psize, int rows) {
  using C = cplx<T>;
  constexpr int PITCH = PY::N | 1, LB = plane_batch(PY::N, PX::R1, NT);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);
  C* X = P + psize;
  const HpsiItem<T>& I = B.it[batch_item(B, blockIdx.x, true)];
  const SphereDev& sp = I.sp;
  const int local = blockIdx.x - I.pstart;
  const int b = local / n3, i3 = local - b * n3;
  C* S = I.scratch + ((size_t)b * n3 + i3) * sp.ldc;
  const PlaneDims D = plane_dims<T>(sp);
  plane_in<T, PY, RUNS>(P, X, S, sp, D, rows, PITCH, NT, tw2);
  __syncthreads();
  plane_x_all<T, PX>(P, X, D, PITCH, PY::N, LB, tw1, I.vplane + (size_t)i3 * PX::N * PY::N);
  __syncthreads();
  plane_out<T, PY, RUNS>(P, X, S, sp, D, rows, PITCH, NT, tw2);
}

// ---- band densities --------------------------------------------------------------------------------
// rho(r) += w |u(r)|^2 over the bands of a group, one CTA per (plane, group of bands), into a plane
// of partial sums of its own (written for the group's first band, then read, added to and written
// back: 8 bytes a point that stay in L2).  FP64 orbitals accumulate in FP64.  FP32 orbitals
// accumulate in double-float on the FP32 pipes: the squares are exact products, so w |u|^2 and
// the running sum carry 48 bits of values known to 24, while the FP64 pipe (1/64 of the FP32 rate)
// would take longer over its five operations a point than the transforms take altogether.
template <typename T> struct RhoAcc { using t = double; };
template <> struct RhoAcc<float> { using t = float2; };
__device__ __forceinline__ double rho_term(double w, double2 u) { return w * (u.x * u.x + u.y * u.y); }
__device__ __forceinline__ float2 rho_term(dd w, float2 u) {
  const float p = __fmul_rn(u.x, u.x), e = __fmaf_rn(u.x, u.x, -p);
  const float q = __fmul_rn(u.y, u.y), f = __fmaf_rn(u.y, u.y, -q);
  const dd s = dd_two_sum(p, q);
  const dd v = w * dd_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(e, f)));
  return make_float2(v.hi, v.lo);
}
__device__ __forceinline__ double rho_add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 rho_add(float2 a, float2 b) {
  const dd s = dd(a.x, a.y) + dd(b.x, b.y);
  return make_float2(s.hi, s.lo);
}
__device__ __forceinline__ double rho_weight(double w, double) { return w; }
__device__ __forceinline__ dd rho_weight(double w, float) { return dd_from_double(w); }

template <typename T, typename Plan>
__device__ __forceinline__ void plane_x_rho(const cplx<T>* P, cplx<T>* X, const PlaneDims& D, int pitch, int n2, int lb,
                                            const cplx<T>* __restrict__ tw, double weight, bool first,
                                            typename RhoAcc<T>::t* rho) {
  using C = cplx<T>;
  constexpr int R1 = Plan::R1, R2 = Plan::R2;
  const auto wt = rho_weight(weight, T(0));
  const int tid = threadIdx.x, j = tid / lb, c = tid - j * lb;
  const bool in1 = j < R2, in2 = j < R1;
  XItem<T, Plan> I;
  if (in1) I.rows(D, j, c, pitch);
#pragma unroll 1
  for (int c0 = 0; c0 < n2; c0 += lb) {
    const bool have = c < n2 - c0;
    if (in1 && have) plane_x_in<T, Plan>(P, X, I, j, c, c0, lb);
    __syncthreads();
    if (in2 && have) {
      C v[R2];
#pragma unroll
      for (int p = 0; p < R2; ++p) {
        v[p] = X[(p * R1 + j) * lb + c];
        if constexpr (!Plan::kCoprime)
          if (p) v[p] = twist(v[p], tw[p * j], +1);
      }
      dft_r<R2>(v, +1);
#pragma unroll
      for (int p = 0; p < R2; ++p) {
        auto* o = rho + Plan::output(j, p) * n2 + c0 + c;
        const auto d = rho_term(wt, v[p]);
        *o = first ? d : rho_add(*o, d);
      }
    }
    __syncthreads();
  }
}

// Bands [nb g / groups, nb (g + 1) / groups) of group g.
template <typename T, typename PX, typename PY, int NT, int MINB, bool RUNS>
__global__ void __launch_bounds__(NT, MINB)
k_plane_rho(const cplx<T>* __restrict__ scratch, SphereDev sp, int nb, const double* __restrict__ weight,
            typename RhoAcc<T>::t* __restrict__ part, int n3, const cplx<T>* __restrict__ tw1,
            const cplx<T>* __restrict__ tw2, int psize, int rows) {
  using C = cplx<T>;
  constexpr int PITCH = PY::N | 1, LB = plane_batch(PY::N, PX::R1, NT);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);
  C* X = P + psize;
  const int i3 = blockIdx.x, g = blockIdx.y;
  const int b0 = (int)((long long)nb * g / gridDim.y), b1 = (int)((long long)nb * (g + 1) / gridDim.y);
  const PlaneDims D = plane_dims<T>(sp);
  auto* rho = part + ((size_t)g * n3 + i3) * PX::N * PY::N;
#pragma unroll 1
  for (int b = b0; b < b1; ++b) {
    plane_in<T, PY, RUNS>(P, X, scratch + ((size_t)b * n3 + i3) * sp.ldc, sp, D, rows, PITCH, NT, tw2);
    __syncthreads();
    plane_x_rho<T, PX>(P, X, D, PITCH, PY::N, LB, tw1, weight[b], b == b0, rho);
  }
}

}  // namespace fde
