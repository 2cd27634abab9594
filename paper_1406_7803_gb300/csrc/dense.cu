// dense.cu -- FP64 dense kernels of the Rayleigh-Ritz step (Eq. KS, block solver) spread over
// many SMs.  FP64 arithmetic on this part runs at a small fraction of the FP32 rate per SM, so
// the O(n^3) factorisations are distributed over a thread-block cluster of P CTAs that hold
// the matrix rows cyclically in shared memory (row i in CTA i % P) and synchronise with the
// hardware cluster barrier; the embarrassingly parallel phases run as ordinary launches.
//
//   k_cl_cholesky   S = L L^H (right-looking, one cluster barrier per column)
//   k_tri_inverse   L^{-1}, one CTA per column
//   k_cl_tridiag    Householder reduction A = Q T Q^H (2 cluster barriers per column)
//   k_tri_eigvals   eigenvalues of T by 128-point multisection on Sturm counts (CTA each)
//   k_tri_solve     inverse iteration, one thread per eigenvector
//   k_tri_orth      modified Gram-Schmidt inside clusters of close eigenvalues
//   k_wy_gram       inner products of the reflectors, block by block
//   k_backtransform v = H_0 ... H_{n-2} z, one CTA per eigenvector, 16 reflectors at a time
// At these sizes (n up to a few hundred) every kernel is bound by latency: a dependent FP64
// operation takes some 70 cycles and a division or square root ten of them, so each step keeps its
// chain of dependent operations short (sums as trees, reciprocals formed once and by one warp,
// no division inside a recurrence) and its barriers few.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "dense.h"
#include "prof.h"

namespace cg = cooperative_groups;

namespace fde {

constexpr int kClThreads = 256;
constexpr int kClWarps = kClThreads / 32;

__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct ClusterLayout {
  int P, rank, nloc, sh;  // CTAs (a power of two, 2^sh), own rank, rows held
  __device__ __forceinline__ int owner(int i) const { return i & (P - 1); }
  __device__ __forceinline__ int local(int i) const { return i >> sh; }
};

__device__ __forceinline__ ClusterLayout cluster_layout(int n) {
  ClusterLayout c;
  c.P = (int)cg::this_cluster().num_blocks();
  c.rank = (int)cg::this_cluster().block_rank();
  c.nloc = (n + c.P - 1) / c.P;
  c.sh = 31 - __clz(c.P);
  return c;
}

// ---- Cholesky --------------------------------------------------------------------------------
// Every CTA gathers the raw column j of the trailing matrix (its owners' rows, through the cluster's
// shared memory) with the reciprocal of its pivot, and updates its own rows
//   A[i][k] -= (A[i][j] / d_j) conj(A[k][j]),
// one cluster barrier a column; the columns are scaled by 1 / sqrt(d_j) at the end, all at once, so no
// square root and one reciprocal sit in the chain of a column.  Shared memory: rows [nloc][n],
// col [n], piv [n] (the least accepted pivots, then 1 / sqrt(d_j)).  Writes the transpose of L,
// which k_tri_inverse reads by columns.
__global__ void __launch_bounds__(kClThreads)
k_cl_cholesky(const double2* __restrict__ S, int n, double2* __restrict__ LT, unsigned* status, double rel_pivot) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem[];
  const ClusterLayout c = cluster_layout(n);
  double2* rows = reinterpret_cast<double2*>(smem);
  double2* col = rows + (size_t)c.nloc * n;
  double* piv = reinterpret_cast<double*>(col + n);
  __shared__ double s_inv;
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int idx = tid; idx < c.nloc * n; idx += kClThreads) {
    const int li = idx / n, j = idx - li * n, i = li * c.P + c.rank;
    rows[idx] = (i < n && j <= i) ? S[(size_t)i * n + j] : make_double2(0, 0);
  }
  for (int j = tid; j < n; j += kClThreads) piv[j] = rel_pivot * S[(size_t)j * n + j].x;
  if (tid == 0) s_bad = 0;
  cl.sync();
  bool failed = false;
  int bad = 0;
  for (int j = 0; j < n; ++j) {
    for (int k = j + tid; k < n; k += kClThreads) {
      const double2* rk = cl.map_shared_rank(rows, c.owner(k));
      const double2 x = rk[(size_t)c.local(k) * n + j];
      col[k] = x;
      if (k == j) {  // thread 0
        if (!(x.x > piv[j])) s_bad = 1;
        s_inv = 1.0 / x.x;
        piv[j] = x.x;
      }
    }
    __syncthreads();
    if (s_bad) {  // the same values in every CTA: a uniform exit
      failed = true;
      bad = j;
      break;
    }
    const double inv = s_inv;
    for (int li = warp; li < c.nloc; li += kClWarps) {
      const int i = li * c.P + c.rank;
      if (i <= j || i >= n) continue;
      const double2 a = col[i];
      const double ax = a.x * inv, ay = a.y * inv;
      double2* ri = rows + (size_t)li * n;
      for (int k = j + 1 + lane; k <= i; k += 32) {
        const double2 b = col[k];
        double2 v = ri[k];
        v.x = fma(-ax, b.x, v.x);
        v.y = fma(-ay, b.x, v.y);
        v.x = fma(-ay, b.y, v.x);
        v.y = fma(ax, b.y, v.y);
        ri[k] = v;
      }
    }
    cl.sync();
  }
  if (failed) {
    if (c.rank == 0 && tid == 0) {
      atomicOr(status, ST_CHOLESKY);
      status[1] = (unsigned)bad;
    }
  } else {
    for (int j = tid; j < n; j += kClThreads) piv[j] = 1.0 / sqrt(piv[j]);
    __syncthreads();
    for (int idx = tid; idx < c.nloc * n; idx += kClThreads) {
      const int li = idx / n, j = idx - li * n, i = li * c.P + c.rank;
      if (i >= n) continue;
      double2 v = make_double2(0, 0);
      if (j <= i) {
        const double p = piv[j];
        v = rows[idx];
        v = (j == i) ? make_double2(v.x * p, 0.0) : make_double2(v.x * p, v.y * p);
      }
      LT[(size_t)j * n + i] = v;
    }
  }
  cl.sync();  // no CTA leaves while others may still read its shared memory
}

// ---- triangular inverse ------------------------------------------------------------------------
// Li = L^{-1} (lower); column c of the inverse by forward substitution, right-looking: one CTA per
// column, a thread per row, the residual in registers.  Row i's value is final once columns c .. i - 1
// have been taken off it; its thread publishes x_i = r_i / L_ii (a stored reciprocal) and every later
// row takes L[k][i] x_i off its own.  Reads L by columns (LT, coalesced).
constexpr int kTiThreads = 128;
constexpr int kTiRows = 4;  // rows a thread: n up to 512
__global__ void __launch_bounds__(kTiThreads)
k_tri_inverse(const double2* __restrict__ LT, int n, double2* __restrict__ Li, const unsigned* status) {
  if (*status & ST_CHOLESKY) return;
  extern __shared__ double2 xs[];  // [n] solution; [n] doubles of reciprocals behind it
  double* rd = reinterpret_cast<double*>(xs + n);
  const int c = blockIdx.x, tid = threadIdx.x;
  for (int i = c + tid; i < n; i += kTiThreads) rd[i] = 1.0 / LT[(size_t)i * n + i].x;
  double2 r[kTiRows], l[kTiRows];
#pragma unroll
  for (int s = 0; s < kTiRows; ++s) {
    const int k = tid + kTiThreads * s;
    r[s] = make_double2(k == c ? 1.0 : 0.0, 0.0);
    l[s] = (k > c && k < n) ? LT[(size_t)c * n + k] : make_double2(0, 0);
  }
  __syncthreads();
  for (int i = c; i < n; ++i) {
    const int own = i % kTiThreads, os = i / kTiThreads;
    if (tid == own) {
      double2 v = make_double2(0, 0);
#pragma unroll
      for (int s = 0; s < kTiRows; ++s)
        if (s == os) v = r[s];
      const double p = rd[i];
      xs[i] = make_double2(v.x * p, v.y * p);
    }
    __syncthreads();
    const double2 x = xs[i];
#pragma unroll
    for (int s = 0; s < kTiRows; ++s) {
      const int k = tid + kTiThreads * s;
      const double2 a = l[s];
      if (i + 1 < n && k > i + 1 && k < n) l[s] = LT[(size_t)(i + 1) * n + k];  // ahead of its use
      if (k > i && k < n) {
        r[s].x = fma(-a.x, x.x, r[s].x);
        r[s].y = fma(-a.x, x.y, r[s].y);
        r[s].x = fma(a.y, x.y, r[s].x);
        r[s].y = fma(-a.y, x.x, r[s].y);
      }
    }
  }
  for (int i = tid; i < n; i += kTiThreads) Li[(size_t)i * n + c] = i < c ? make_double2(0, 0) : xs[i];
}

// ---- Householder tridiagonalisation ----------------------------------------------------------
// A (n x n Hermitian, full storage) -> d[n], e[n] (T = Q^H A Q real symmetric tridiagonal),
// tau[n] and the reflector vectors Vh[k][j] (j > k; Vh[k][k+1] = 1) with
// H_k = I - tau_k v_k v_k^H.  Every CTA gathers the whole column (and later the whole product p = tau
// A v) through the cluster's shared memory and forms its norm, the reflector and p^H v itself: a
// column takes two cluster barriers instead of four and no second gather of partial sums.
// Shared memory: rows [nloc][n], v [n], w [n], pown [nloc] (double2).  192 x 192: 3.0 ms before.
__device__ __forceinline__ void warp_sum_d2(double& a, double& b) {
  for (int o = 16; o > 0; o >>= 1) {
    const double x = __shfl_xor_sync(0xffffffffu, a, o), y = __shfl_xor_sync(0xffffffffu, b, o);
    a += x;
    b += y;
  }
}
constexpr int kTdWarps = 16;  // most warps a CTA of the reduction
__global__ void __launch_bounds__(32 * kTdWarps)
k_cl_tridiag(const double2* __restrict__ A, int n, double* __restrict__ d, double* __restrict__ e,
             double2* __restrict__ tau, double2* __restrict__ Vh) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem[];
  const ClusterLayout c = cluster_layout(n);
  double2* rows = reinterpret_cast<double2*>(smem);
  double2* v = rows + (size_t)c.nloc * n;
  double2* w = v + n;
  double2* pown = w + n;
  __shared__ double2 red[kTdWarps];
  __shared__ double2 s_tau, s_sc, s_al;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  for (int idx = tid; idx < c.nloc * n; idx += nt) {
    const int li = idx / n, j = idx - li * n, i = li * c.P + c.rank;
    rows[idx] = (i < n) ? A[(size_t)i * n + j] : make_double2(0, 0);
  }
  cl.sync();
  for (int k = 0; k < n - 1; ++k) {
    // column k below the diagonal, |x|^2 below the subdiagonal
    double acc = 0;
    for (int j = k + 1 + tid; j < n; j += nt) {
      const double2 x = cl.map_shared_rank(rows, c.owner(j))[(size_t)c.local(j) * n + k];
      v[j] = x;
      if (j > k + 1) acc = fma(x.x, x.x, fma(x.y, x.y, acc));
    }
    acc = warp_sum_d(acc);
    if (lane == 0) red[warp].x = acc;
    __syncthreads();
    if (warp == 0) {
      double xn2 = lane < nw ? red[lane].x : 0.0;
      for (int o = kTdWarps / 2; o > 0; o >>= 1) xn2 += __shfl_xor_sync(0xffffffffu, xn2, o);
      if (lane == 0) {
        const double2 alpha = v[k + 1];
        double2 t = make_double2(0, 0), sc = make_double2(0, 0);
        double beta = alpha.x;
        if (!(xn2 == 0.0 && alpha.y == 0.0)) {
          beta = -copysign(sqrt(fma(alpha.x, alpha.x, fma(alpha.y, alpha.y, xn2))), alpha.x);
          const double ib = 1.0 / beta, ar = alpha.x - beta, ai = alpha.y, id = 1.0 / fma(ar, ar, ai * ai);
          t = make_double2((beta - alpha.x) * ib, -alpha.y * ib);
          sc = make_double2(ar * id, -ai * id);
        }
        s_tau = t;
        s_sc = sc;
        if (c.rank == 0) {
          e[k] = beta;
          tau[k] = t;
        }
        if (c.rank == k % c.P) d[k] = rows[(size_t)(k / c.P) * n + k].x;
      }
    }
    __syncthreads();
    const double2 tk = s_tau, sc = s_sc;
    const bool skip = (tk.x == 0.0 && tk.y == 0.0);  // uniform over the cluster
    for (int j = k + 1 + tid; j < n; j += nt) {
      const double2 x = j == k + 1 ? make_double2(1.0, 0.0) : (skip ? make_double2(0.0, 0.0) : cmul(v[j], sc));
      v[j] = x;
      if (c.rank == 0) Vh[(size_t)k * n + j] = x;
    }
    __syncthreads();
    if (skip) {
      cl.sync();  // the next column's rows are read after this barrier as after the others'
      continue;
    }
    // p_i = tau (A22 v)_i for the own trailing rows (warp per row)
    for (int li = warp; li < c.nloc; li += nw) {
      const int i = li * c.P + c.rank;
      if (i <= k || i >= n) continue;
      const double2* ri = rows + (size_t)li * n;
      double sr = 0, si = 0;
      for (int j = k + 1 + lane; j < n; j += 32) {
        const double2 a = ri[j], x = v[j];
        sr = fma(a.x, x.x, sr);
        si = fma(a.x, x.y, si);
        sr = fma(-a.y, x.y, sr);
        si = fma(a.y, x.x, si);
      }
      warp_sum_d2(sr, si);
      if (lane == 0) pown[li] = cmul(tk, make_double2(sr, si));
    }
    cl.sync();
    // the whole p, p^H v, w = p + alpha v with alpha = -tau (p^H v) / 2
    double dr = 0, di = 0;
    for (int j = k + 1 + tid; j < n; j += nt) {
      const double2 p = cl.map_shared_rank(pown, c.owner(j))[c.local(j)], x = v[j];
      w[j] = p;
      dr = fma(p.x, x.x, fma(p.y, x.y, dr));
      di = fma(p.x, x.y, fma(-p.y, x.x, di));
    }
    warp_sum_d2(dr, di);
    if (lane == 0) red[warp] = make_double2(dr, di);
    __syncthreads();
    if (warp == 0) {
      double2 t = lane < nw ? red[lane] : make_double2(0, 0);
      for (int o = kTdWarps / 2; o > 0; o >>= 1) {
        const double x = __shfl_xor_sync(0xffffffffu, t.x, o), y = __shfl_xor_sync(0xffffffffu, t.y, o);
        t.x += x;
        t.y += y;
      }
      if (lane == 0) s_al = cmul(make_double2(-0.5 * tk.x, -0.5 * tk.y), t);
    }
    __syncthreads();
    const double2 al = s_al;
    for (int j = k + 1 + tid; j < n; j += nt) w[j] = cadd(w[j], cmul(al, v[j]));
    __syncthreads();
    // A22 -= v w^H + w v^H on the own rows
    for (int li = warp; li < c.nloc; li += nw) {
      const int i = li * c.P + c.rank;
      if (i <= k || i >= n) continue;
      const double2 vi = v[i], wi = w[i];
      double2* ri = rows + (size_t)li * n;
      for (int j = k + 1 + lane; j < n; j += 32) {
        const double2 vj = v[j], wj = w[j];
        double2 a = ri[j];
        a.x = fma(-vi.x, wj.x, a.x);
        a.y = fma(-vi.y, wj.x, a.y);
        a.x = fma(-vi.y, wj.y, a.x);
        a.y = fma(vi.x, wj.y, a.y);
        a.x = fma(-wi.x, vj.x, a.x);
        a.y = fma(-wi.y, vj.x, a.y);
        a.x = fma(-wi.y, vj.y, a.x);
        a.y = fma(wi.x, vj.y, a.y);
        ri[j] = a;
      }
    }
    cl.sync();
  }
  if (tid == 0 && c.rank == (n - 1) % c.P) d[n - 1] = rows[(size_t)((n - 1) / c.P) * n + (n - 1)].x;
  if (tid == 0 && c.rank == 0) {
    e[n - 1] = 0.0;
    tau[n - 1] = make_double2(0, 0);
  }
  cl.sync();
}

// ---- eigenvalues of T -------------------------------------------------------------------------
// Number of eigenvalues of the scaled T below x: sign changes of the leading principal minors
//   p_j = (d_j - x) p_{j-1} - e_{j-1}^2 p_{j-2},
// one fused multiply-add deep per row (the quotient form's division is some ten).  T is scaled to a norm
// between one and two, so a row grows the pair by less than 2^3; a vanishing minor counts as a change and
// becomes -2^-100 of its predecessor (a pivot far below the rounding of T, as the quotient form's
// least pivot is), so a row shrinks the pair by at most some 2^-106; it is rescaled by a power of two
// every four rows.
__device__ __forceinline__ int sturm_count_minors(const double* d, const double* e2, int n, double x) {
  const double least = -7.888609052210118e-31;  // -2^-100
  double p0 = 1.0, p1 = d[0] - x;
  if (p1 == 0.0) p1 = least;
  int cnt = p1 < 0.0;
  for (int j = 1; j < n; ++j) {
    double p2 = fma(d[j] - x, p1, -(e2[j - 1] * p0));
    if (p2 == 0.0) p2 = least * p1;
    cnt += (__double2hiint(p2) ^ __double2hiint(p1)) < 0;
    p0 = p1;
    p1 = p2;
    if ((j & 3) == 0) {
      const int ex = max(__double2hiint(p0) & 0x7fffffff, __double2hiint(p1) & 0x7fffffff) >> 20;
      const double s = __hiloint2double((2046 - ex) << 20, 0);  // 2^-(exponent of the larger)
      p0 *= s;
      p1 *= s;
    }
  }
  return cnt;
}

// The power of two that scales ||T|| (its largest row sum tn) into [1, 2).
__device__ __forceinline__ double tri_scale(double tn) {
  const int ex = (__double2hiint(tn) & 0x7fffffff) >> 20;
  return ex < 24 || ex > 2022 ? 1.0 : __hiloint2double((2046 - ex) << 20, 0);
}

// w[i] = i-th smallest eigenvalue of T; one CTA of 128 threads per i, 128 Sturm counts per step (the
// interval shrinks 129-fold, so eight steps where 32 points take eleven; the four warps sit on the
// SM's four quarters).  CTA 0 leaves ||T|| in *tnorm.  192 eigenvalues of n = 192 took 1.3 ms in
// quotient form, a warp each; the 64 that are asked for now, 0.2 ms.
constexpr int kEvThreads = 128;
__global__ void __launch_bounds__(kEvThreads)
k_tri_eigvals(const double* __restrict__ dg, const double* __restrict__ eg, int n, double* w, double* tnorm) {
  extern __shared__ double sde[];
  __shared__ double red[3][kEvThreads / 32], xs[kEvThreads];
  __shared__ int first;
  double* d = sde;
  double* e2 = sde + n;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, i = blockIdx.x;
  double tn = 0, lo = 1e300, hi = -1e300;
  for (int j = tid; j < n; j += kEvThreads) {
    const double dj = dg[j], r = (j < n - 1 ? fabs(eg[j]) : 0.0) + (j > 0 ? fabs(eg[j - 1]) : 0.0);
    d[j] = dj;
    tn = fmax(tn, fabs(dj) + r);
    lo = fmin(lo, dj - r);
    hi = fmax(hi, dj + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    red[0][wp] = tn;
    red[1][wp] = lo;
    red[2][wp] = hi;
  }
  __syncthreads();
  for (int q = 0; q < kEvThreads / 32; ++q) {
    tn = fmax(tn, red[0][q]);
    lo = fmin(lo, red[1][q]);
    hi = fmax(hi, red[2][q]);
  }
  tn = fmax(tn, 1e-300);
  if (i == 0 && tid == 0) *tnorm = tn;
  const double sc = tri_scale(tn);
  for (int j = tid; j < n; j += kEvThreads) {
    d[j] *= sc;
    const double ej = j < n - 1 ? eg[j] * sc : 0.0;
    e2[j] = ej * ej;
  }
  lo = (lo - 1e-12 * tn - 1e-300) * sc;
  hi = (hi + 1e-12 * tn + 1e-300) * sc;
  for (int it = 0; it < 64; ++it) {
    if (hi - lo <= 2.2e-16 * fmax(fabs(lo), fabs(hi)) + 1e-19) break;
    const double x = lo + (hi - lo) / (double)(kEvThreads + 1) * (double)(tid + 1);
    xs[tid] = x;
    if (tid == 0) first = kEvThreads;
    __syncthreads();
    if (sturm_count_minors(d, e2, n, x) > i) atomicMin(&first, tid);
    __syncthreads();
    const int f = first;
    const double nlo = f > 0 ? xs[f - 1] : lo, nhi = f < kEvThreads ? xs[f] : hi;
    __syncthreads();
    if (!(nlo > lo || nhi < hi)) break;  // no representable progress
    lo = nlo;
    hi = nhi;
  }
  if (tid == 0) w[i] = 0.5 * (lo + hi) / sc;
}

// ---- eigenvectors of T by inverse iteration -----------------------------------------------
__device__ __forceinline__ double start_value_s(int i, int j) {
  unsigned h = (unsigned)(i * 2654435761u) ^ (unsigned)(j * 40503u + 0x9e3779b9u);
  h ^= h >> 15;
  h *= 2246822519u;
  h ^= h >> 13;
  return 0.5 + (double)(h & 0xffff) / 65536.0;
}

// 1 / a for 2^-53 <= |a| < 2^100 by two Newton steps from the FP32 reciprocal.
__device__ __forceinline__ double recip_newton(double a) {
  double r = (double)__frcp_rn((float)a);
  r = fma(r, fma(-a, r, 1.0), r);
  return fma(r, fma(-a, r, 1.0), r);
}

// Inverse iteration for vectors i < nvec: `iters` solves of (T - w_i I) z_new = z with the
// partially pivoted LU of the scaled T - w_i I, normalised at the end (one solve grows a vector by at
// most some 2^53 n); starts from the current Z and the factors an earlier call left in work (fresh = 0),
// or from a fixed pseudo-random vector, factorising first (fresh = 1).  Z[i][n] (row per vector);
// work: 5 n nvec doubles.  A CTA is one warp with VPC vectors, a thread each, all recurrences in
// shared memory: the factorisation's chain is a reciprocal and two operations a row, a solve's two
// and three (pivots kept as reciprocals; a pivot below 2^-52 ||T|| is set to it).
__global__ void __launch_bounds__(32)
k_tri_solve(const double* __restrict__ dg, const double* __restrict__ eg, int n, const double* w, int nvec, int fresh,
            int iters, double* __restrict__ Z, double* __restrict__ work, const double* __restrict__ tnorm, int vpc) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x, i0 = blockIdx.x * vpc, nv = min(vpc, nvec - i0);
  const size_t blk = (size_t)n * vpc;
  double* ia = sm;             // reciprocal pivots          [n][vpc]
  double* u1 = sm + blk;       // first superdiagonal
  double* u2 = sm + 2 * blk;   // second superdiagonal (fill-in)
  double* ml = sm + 3 * blk;   // multipliers
  double* sw = sm + 4 * blk;   // 1 where rows j and j + 1 were interchanged
  double* z = sm + 5 * blk;
  double* sd = sm + 6 * blk;   // scaled d [n], e [n]
  double* se = sd + n;
  double* save = work + (size_t)blockIdx.x * 5 * blk;
  const double sc = tri_scale(*tnorm);
  for (int j = lane; j < n; j += 32) {
    sd[j] = dg[j] * sc;
    se[j] = j < n - 1 ? eg[j] * sc : 0.0;
  }
  if (fresh) {
    for (size_t k = lane; k < blk; k += 32) z[k] = start_value_s(i0 + (int)(k % vpc), (int)(k / vpc));
  } else {
    for (size_t k = lane; k < 5 * blk; k += 32) sm[k] = save[k];
    for (int k = lane; k < nv * n; k += 32) z[(size_t)(k % n) * vpc + k / n] = Z[(size_t)(i0 + k / n) * n + k % n];
  }
  __syncwarp();
  if (lane < nv) {
    const double tiny = 2.2e-16;
    if (fresh) {
      const double lam = w[i0 + lane] * sc;
      double a = sd[0] - lam, u = n > 1 ? se[0] : 0.0;
      for (int j = 0; j < n - 1; ++j) {
        const double sub = se[j], dn = sd[j + 1] - lam, en = se[j + 1];
        const bool keep = fabs(a) >= fabs(sub);
        double p = keep ? a : sub;
        if (fabs(p) < tiny) p = copysign(tiny, p);
        const double r = recip_newton(p), m = (keep ? sub : a) * r;
        const size_t k = (size_t)j * vpc + lane;
        ia[k] = r;
        u1[k] = keep ? u : dn;
        u2[k] = keep ? 0.0 : en;
        ml[k] = m;
        sw[k] = keep ? 0.0 : 1.0;
        a = keep ? fma(-m, u, dn) : fma(-m, dn, u);
        u = keep ? en : -m * en;
      }
      const size_t k = (size_t)(n - 1) * vpc + lane;
      if (fabs(a) < tiny) a = copysign(tiny, a);
      ia[k] = recip_newton(a);
      u1[k] = u2[k] = ml[k] = sw[k] = 0.0;
    }
    double nn = 0;
    for (int it = 0; it < iters; ++it) {
      // the row operations
      double t = z[lane];
      for (int j = 0; j < n - 1; ++j) {
        const size_t k = (size_t)j * vpc + lane;
        const double nx = z[k + vpc], m = ml[k];
        const bool swp = sw[k] != 0.0;
        z[k] = swp ? nx : t;
        t = swp ? fma(-m, nx, t) : fma(-m, t, nx);
      }
      z[(size_t)(n - 1) * vpc + lane] = t;
      // back substitution
      double b1 = 0.0, b2 = 0.0;
      nn = 0;
      for (int j = n - 1; j >= 0; --j) {
        const size_t k = (size_t)j * vpc + lane;
        const double x = fma(-u1[k], b1, fma(-u2[k], b2, z[k])) * ia[k];
        z[k] = x;
        b2 = b1;
        b1 = x;
        nn = fma(x, x, nn);
      }
    }
    const double inv = 1.0 / sqrt(fmax(nn, 1e-300));
    for (int j = 0; j < n; ++j) z[(size_t)j * vpc + lane] *= inv;
  }
  __syncwarp();
  if (fresh)
    for (size_t k = lane; k < 5 * blk; k += 32) save[k] = sm[k];
  for (int k = lane; k < nv * n; k += 32) Z[(size_t)(i0 + k / n) * n + k % n] = z[(size_t)(k % n) * vpc + k / n];
}

// Modified Gram-Schmidt inside each cluster of eigenvalues closer than gap_rel * ||T||
// (one CTA per cluster; CTAs beyond the number of clusters return).  Z[i][n].
__global__ void k_tri_orth(int n, const double* w, int nvec, double gap_rel, double* __restrict__ Z,
                           const double* __restrict__ tnorm) {
  __shared__ double red[32];
  __shared__ int s_lo, s_hi;
  if (threadIdx.x < 32) {
    // bounds of cluster blockIdx.x: its start and the next start
    const double gap = gap_rel * *tnorm;
    const int lane = threadIdx.x;
    int seen = 0, lo = -1, hi = -1;
    for (int q0 = 0; q0 < nvec && hi < 0; q0 += 32) {
      const int q = q0 + lane;
      const bool start = q < nvec && (q == 0 || w[q] - w[q - 1] > gap);
      unsigned m = __ballot_sync(0xffffffffu, start);
      while (m && hi < 0) {
        const int q1 = q0 + __ffs(m) - 1;
        if (seen == (int)blockIdx.x) lo = q1;
        if (seen == (int)blockIdx.x + 1) hi = q1;
        ++seen;
        m &= m - 1;
      }
    }
    if (lane == 0) {
      s_lo = lo < 0 ? 0 : lo;
      s_hi = lo < 0 ? 0 : (hi < 0 ? nvec : hi);
    }
  }
  __syncthreads();
  const int lo = s_lo, hi = s_hi;
  if (hi - lo < 2) return;  // a single vector is already normalised
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = lo; q < hi; ++q) {
    double* zq = Z + (size_t)q * n;
    double acc = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) acc += zq[j] * zq[j];
    acc = warp_sum_d(acc);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    double t = 0;
    for (int k = 0; k < nw; ++k) t += red[k];
    const double inv = 1.0 / sqrt(fmax(t, 1e-300));
    for (int j = threadIdx.x; j < n; j += blockDim.x) zq[j] *= inv;
    __syncthreads();
    for (int r = q + 1 + warp; r < hi; r += nw) {
      double* zr = Z + (size_t)r * n;
      double s = 0;
      for (int j = lane; j < n; j += 32) s += zq[j] * zr[j];
      s = warp_sum_d(s);
      for (int j = lane; j < n; j += 32) zr[j] -= s * zq[j];
    }
    __syncthreads();
  }
}

// ---- back-transformation ---------------------------------------------------------------------------
// The reflectors are applied 16 at a time.  With s_k = v_k^H z for the whole block at once, the
// coefficient of H_k inside it is f_k = tau_k (s_k - sum_{l > k} (v_k^H v_l) f_l), so a block takes one
// pass over z for its 16 inner products, 16 short steps on one warp and one pass to subtract
// sum f_k v_k, instead of 16 dependent pairs of passes.
constexpr int kWy = 16;
// G[blk][a][b] = v_{k0 + a}^H v_{k0 + b}, a < b (a warp each).
__global__ void k_wy_gram(const double2* __restrict__ Vh, int n, int nref, double2* __restrict__ G) {
  const int lane = threadIdx.x & 31;
  const int id = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int blk = id / (kWy * kWy), a = id / kWy % kWy, b = id % kWy, k0 = blk * kWy;
  if (a >= b || k0 + b >= nref) return;
  const double2 *va = Vh + (size_t)(k0 + a) * n, *vb = Vh + (size_t)(k0 + b) * n;
  double sr = 0, si = 0;
  for (int j = k0 + b + 1 + lane; j < n; j += 32) {
    const double2 x = va[j], y = vb[j];
    sr = fma(x.x, y.x, fma(x.y, y.y, sr));
    si = fma(x.x, y.y, fma(-x.y, y.x, si));
  }
  warp_sum_d2(sr, si);
  if (lane == 0) G[(size_t)blk * kWy * kWy + a * kWy + b] = make_double2(sr, si);
}

// V[:, i] = H_0 H_1 ... H_{n-2} z_i (column i of the row-major n x n V; one CTA per vector);
// columns nvec..n-1 of V are zeroed.
constexpr int kBtThreads = 256;
__global__ void __launch_bounds__(kBtThreads)
k_backtransform(const double2* __restrict__ Vh, const double2* __restrict__ tau, const double2* __restrict__ G, int n,
                int nvec, const double* __restrict__ Z, double2* __restrict__ V) {
  extern __shared__ double2 zs[];  // [n]
  __shared__ double2 f[kWy];
  const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (i >= nvec) {
    for (int r = tid; r < n; r += kBtThreads) V[(size_t)r * n + i] = make_double2(0, 0);
    return;
  }
  for (int r = tid; r < n; r += kBtThreads) zs[r] = make_double2(Z[(size_t)i * n + r], 0.0);
  const int nref = n - 1;
  for (int blk = (nref - 1) / kWy; blk >= 0; --blk) {
    const int k0 = blk * kWy;
    __syncthreads();
    for (int a = warp; a < kWy; a += kBtThreads / 32) {
      double sr = 0, si = 0;
      if (k0 + a < nref) {
        const double2* v = Vh + (size_t)(k0 + a) * n;
        for (int j = k0 + a + 1 + lane; j < n; j += 32) {
          const double2 x = v[j], y = zs[j];
          sr = fma(x.x, y.x, fma(x.y, y.y, sr));
          si = fma(x.x, y.y, fma(-x.y, y.x, si));
        }
      }
      warp_sum_d2(sr, si);
      if (lane == 0) f[a] = make_double2(sr, si);
    }
    __syncthreads();
    if (warp == 0) {
      const int a = lane & (kWy - 1);
      double2 s = f[a];
      const double2 t = k0 + a < nref ? tau[k0 + a] : make_double2(0, 0);
      const double2* g = G + (size_t)blk * kWy * kWy + a * kWy;
      double2 out = make_double2(0, 0);
      for (int b = kWy - 1; b >= 0; --b) {
        const bool have = a < b && k0 + b < nref;
        const double2 c = have ? g[b] : make_double2(0, 0);  // v_a^H v_b
        double2 x = cmul(t, s);
        if (a == b) out = x;
        x.x = __shfl_sync(0xffffffffu, x.x, b);
        x.y = __shfl_sync(0xffffffffu, x.y, b);
        s.x = fma(-c.x, x.x, fma(c.y, x.y, s.x));
        s.y = fma(-c.x, x.y, fma(-c.y, x.x, s.y));
      }
      if (lane < kWy) f[a] = out;
    }
    __syncthreads();
    for (int j = k0 + 1 + tid; j < n; j += kBtThreads) {
      double2 y = zs[j];
      for (int a = 0; a < kWy; ++a) {
        if (j <= k0 + a || k0 + a >= nref) break;
        const double2 c = f[a], v = Vh[(size_t)(k0 + a) * n + j];
        y.x = fma(-c.x, v.x, fma(c.y, v.y, y.x));
        y.y = fma(-c.x, v.y, fma(-c.y, v.x, y.y));
      }
      zs[j] = y;
    }
  }
  __syncthreads();
  for (int r = tid; r < n; r += kBtThreads) V[(size_t)r * n + i] = zs[r];
}

// ---- host side -----------------------------------------------------------------------------
static int g_cluster_p = -1;  // CTAs per cluster (16, else 8; 0: clusters unusable)

static size_t tridiag_smem(int n, int P) {
  const int nloc = (n + P - 1) / P;
  return ((size_t)nloc * n + 2 * (size_t)n + nloc + 2) * sizeof(double2);
}
static size_t chol_smem(int n, int P) {
  const int nloc = (n + P - 1) / P;
  return ((size_t)nloc * n + n) * sizeof(double2) + (size_t)n * sizeof(double);
}

static int cluster_size() {
  if (g_cluster_p >= 0) return g_cluster_p;
  int dev = 0;
  cudaGetDevice(&dev);
  int cc = 0;
  cudaDeviceGetAttribute(&cc, cudaDevAttrComputeCapabilityMajor, dev);
  g_cluster_p = 0;
  if (cc < 9) return g_cluster_p;
  const size_t smax = 200 * 1024;
  for (int P : {16, 8}) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = smax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = P;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    bool ok = true;
    for (const void* f : {(const void*)k_cl_tridiag, (const void*)k_cl_cholesky}) {
      if (P > 8 && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ok = false;
      if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smax) != cudaSuccess) ok = false;
      int ncl = 0;
      if (ok && (cudaOccupancyMaxActiveClusters(&ncl, f, &cfg) != cudaSuccess || ncl < 1)) ok = false;
    }
    cudaGetLastError();
    if (ok) {
      g_cluster_p = P;
      break;
    }
  }
  return g_cluster_p;
}

int dense_cluster_max_n() {
  static int nmax = -1;
  if (nmax >= 0) return nmax;
  const int P = cluster_size();
  int n = 0;
  if (P > 0)
    while (tridiag_smem(n + 1, P) <= 200 * 1024 && chol_smem(n + 1, P) <= 200 * 1024) ++n;
  nmax = std::min(n, kTiThreads * kTiRows);
  return nmax;
}

static cudaLaunchConfig_t cluster_cfg(int P, int threads, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = P;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

bool launch_cholesky_cluster(const double2* S, int n, double2* L, double2* Li, unsigned* status, double rel_pivot,
                             cudaStream_t st) {
  if (n < 1 || n > dense_cluster_max_n()) return false;
  const int P = cluster_size();
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = cluster_cfg(P, kClThreads, chol_smem(n, P), st, at);
  count_launches(2);
  if (cudaLaunchKernelEx(&cfg, k_cl_cholesky, S, n, L, status, rel_pivot) != cudaSuccess) return false;
  k_tri_inverse<<<n, kTiThreads, (size_t)n * (sizeof(double2) + sizeof(double)), st>>>(L, n, Li, status);
  return true;
}

// Vectors a CTA of the inverse iteration takes: as many (up to 16) as its factors fit 200 KB.
static int tri_solve_vpc(int n) {
  int v = 16;
  while (v > 1 && ((size_t)6 * n * v + 2 * (size_t)n) * sizeof(double) > 200 * 1024) v /= 2;
  return v;
}
static size_t wy_doubles(int n) { return (size_t)2 * kWy * kWy * ((n + kWy - 1) / kWy); }

size_t heev_cluster_work_doubles(int n, int nvec) {
  // d, e | tau (2n) | Vh (2 n^2) | Z (nvec n) | factors (5 n nvec, rounded up to whole CTAs) | reflector
  // products | ||T||
  return (size_t)2 * n + 2 * (size_t)n + 2 * (size_t)n * n + (size_t)nvec * n + 5 * (size_t)n * (nvec + 16) +
         wy_doubles(n) + 64;
}

bool launch_heev_cluster(const double2* A, int n, int nvec, int nval, double* w, double2* V, double* work,
                         cudaStream_t st) {
  if (n < 2 || n > dense_cluster_max_n() || nvec < 1 || nvec > nval || nval > n) return false;
  const int P = cluster_size(), vpc = tri_solve_vpc(n);
  const size_t solve_smem = ((size_t)6 * n * vpc + 2 * (size_t)n) * sizeof(double);
  if (cudaFuncSetAttribute(k_tri_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
    return false;
  double* d = work;
  double* e = d + n;
  double2* tau = reinterpret_cast<double2*>(e + n);
  double2* Vh = tau + n;
  double2* G = Vh + (size_t)n * n;
  double* Z = reinterpret_cast<double*>(G) + wy_doubles(n);
  double* sw = Z + (size_t)nvec * n;
  double* tnorm = sw + 5 * (size_t)n * ((nvec + vpc - 1) / vpc) * vpc;
  cudaLaunchAttribute at[1];
  const int nloc = (n + P - 1) / P, warps = std::max(4, std::min(kTdWarps, nloc));
  cudaLaunchConfig_t cfg = cluster_cfg(P, 32 * warps, tridiag_smem(n, P), st, at);
  count_launches(1);
  if (cudaLaunchKernelEx(&cfg, k_cl_tridiag, A, n, d, e, tau, Vh) != cudaSuccess) return false;
  count_launches(7);
  k_tri_eigvals<<<nval, kEvThreads, 2 * n * sizeof(double), st>>>(d, e, n, w, tnorm);
  // Two rounds of (inverse iteration, Gram-Schmidt inside clusters of close eigenvalues).
  const double gap_rel = 1e-3;
  const int nc = (nvec + vpc - 1) / vpc, blocks = (n + kWy - 1) / kWy;
  k_tri_solve<<<nc, 32, solve_smem, st>>>(d, e, n, w, nvec, 1, 2, Z, sw, tnorm, vpc);
  k_tri_orth<<<nvec, 128, 0, st>>>(n, w, nvec, gap_rel, Z, tnorm);
  k_tri_solve<<<nc, 32, solve_smem, st>>>(d, e, n, w, nvec, 0, 1, Z, sw, tnorm, vpc);
  k_tri_orth<<<nvec, 128, 0, st>>>(n, w, nvec, gap_rel, Z, tnorm);
  k_wy_gram<<<(blocks * kWy * kWy + 3) / 4, 128, 0, st>>>(Vh, n, n - 1, G);
  k_backtransform<<<n, kBtThreads, (size_t)n * sizeof(double2), st>>>(Vh, tau, G, n, nvec, Z, V);
  return true;
}

}  // namespace fde
