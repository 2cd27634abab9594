// fft2.cuh -- two-step transforms: a line of N = R1 R2 points as R2 butterflies of radix R1 and R1
// butterflies of radix R2 with one exchange between them.
//
// Inverse (sign +1), input index n = j + R2 r, output index k = q + R1 p:
//   step 1, item j in [0, R2):  A[j][q] = sum_r x[j + R2 r] W_R1^{rq}
//   step 2, item q in [0, R1):  y[q + R1 p] = sum_j A[j][q] W_N^{jq} W_R2^{jp}
// The forward transform runs the same two steps backwards on the conjugate roots: item q takes
// the inputs q + R1 p, its radix-R2 outputs times W_N^{-jq} are B[j][q], and item j's radix-R1
// butterfly of B[j][.] gives the outputs j + R2 r.  So item q of the inverse ends with exactly
// the values item q of the forward starts with (a pointwise product fits between them in
// registers), and item j of the forward ends on the indices item j of the inverse began with.
//
// Each thread owns whole butterflies (up to 25 values in registers), so a line crosses shared
// memory once per direction instead of once per radix-8-or-9 stage (180 and 288 points took
// three stages, 96 and 144 too), a butterfly reads its inputs straight from global memory and
// writes its outputs straight back, and inputs outside the plane-wave sphere are never stored or
// loaded.  The composite radices are prime-factor (Good-Thomas) products where their factors
// are coprime -- no twiddles inside a butterfly -- and Cooley-Tukey for 8, 9, 16 and 25.
#pragma once

#include "fft.cuh"

namespace fde {

// ---- butterflies -------------------------------------------------------------------------------
// 8 points: 2 x 4.
template <typename C> __device__ __forceinline__ void dft8(C* v, int sign) {
  using T = decltype(v[0].x);
  constexpr T h = T(0.70710678118654752440);  // cos(pi/4)
  C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  dft4(e, sign);
  dft4(o, sign);
  const C p = caddi(o[1], o[1], sign);        // (1 + sign i) o_1
  const C q = caddi(o[3], o[3], -sign);       // (1 - sign i) o_3; W_8^3 o_3 = -h q
  v[0] = cadd(e[0], o[0]);
  v[4] = csub(e[0], o[0]);
  v[1] = caxpy(p, h, e[1]);
  v[5] = caxmy(p, h, e[1]);
  v[2] = caddi(e[2], o[2], sign);
  v[6] = caddi(e[2], o[2], -sign);
  v[3] = caxmy(q, h, e[3]);
  v[7] = caxpy(q, h, e[3]);
}

// A x A points with the inner roots exp(sign 2 pi i k / A^2), k = 0 .. (A - 1)^2, in wc / ws.
template <int A, typename C, typename T> __device__ __forceinline__ void dft_square(C* v, int sign, const T* wc, const T* ws) {
  C t[A][A];
#pragma unroll
  for (int n2 = 0; n2 < A; ++n2) {
    C u[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) u[n1] = v[n2 + A * n1];
    if constexpr (A == 3) dft3(u, sign);
    else if constexpr (A == 4) dft4(u, sign);
    else dft5(u, sign);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      const int e = n2 * k1;
      t[n2][k1] = e ? cmul(u[k1], mk<T>(wc[e], sign > 0 ? ws[e] : -ws[e])) : u[k1];
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    C u[A];
#pragma unroll
    for (int n2 = 0; n2 < A; ++n2) u[n2] = t[n2][k1];
    if constexpr (A == 3) dft3(u, sign);
    else if constexpr (A == 4) dft4(u, sign);
    else dft5(u, sign);
#pragma unroll
    for (int k2 = 0; k2 < A; ++k2) v[k1 + A * k2] = u[k2];
  }
}

template <typename C> __device__ __forceinline__ void dft9(C* v, int sign) {
  using T = decltype(v[0].x);
  constexpr T c[5] = {T(1), T(0.76604444311897803520), T(0.17364817766693034885), T(0), T(-0.93969262078590838405)};
  constexpr T s[5] = {T(0), T(0.64278760968653932632), T(0.98480775301220805936), T(0), T(0.34202014332566873304)};
  dft_square<3>(v, sign, c, s);
}
template <typename C> __device__ __forceinline__ void dft16(C* v, int sign) {
  using T = decltype(v[0].x);
  constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
  constexpr T c[10] = {T(1), T(c1), T(h), T(s1), T(0), T(0), T(-h), T(0), T(0), T(-c1)};
  constexpr T s[10] = {T(0), T(s1), T(h), T(c1), T(1), T(0), T(h), T(0), T(0), T(-s1)};
  dft_square<4>(v, sign, c, s);
}
template <typename C> __device__ __forceinline__ void dft25(C* v, int sign) {
  using T = decltype(v[0].x);
  constexpr T c[17] = {T(1), T(0.96858316112863106), T(0.87630668004386358), T(0.72896862742141154),
                       T(0.53582679497899666), T(0), T(0.06279051952931337), T(0), T(-0.42577929156507272),
                       T(-0.63742398974868975), T(0), T(0), T(-0.99211470131447788), T(0), T(0), T(0),
                       T(-0.63742398974868952)};
  constexpr T s[17] = {T(0), T(0.24868988716485479), T(0.48175367410171532), T(0.68454710592868862),
                       T(0.84432792550201508), T(0), T(0.99802672842827156), T(0), T(0.90482705246601958),
                       T(0.77051324277578925), T(0), T(0), T(0.12533323356430426), T(0), T(0), T(0),
                       T(-0.77051324277578936)};
  dft_square<5>(v, sign, c, s);
}

__host__ __device__ constexpr int crt_index(int a, int b, int ka, int kb) {
  for (int k = 0; k < a * b; ++k)
    if (k % a == ka && k % b == kb) return k;
  return 0;
}
template <int R, typename C> __device__ __forceinline__ void dft_r(C* v, int sign);
// A B points, A and B coprime: inputs n = (B n1 + A n2) mod AB, outputs k = (k mod A, k mod B).
template <int A, int B, typename C> __device__ __forceinline__ void dft_coprime(C* v, int sign) {
  constexpr int ea = crt_index(A, B, 1, 0), eb = crt_index(A, B, 0, 1);
  C t[B][A];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) t[n2][n1] = v[(B * n1 + A * n2) % (A * B)];
    dft_r<A>(t[n2], sign);
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    C u[B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) u[n2] = t[n2][k1];
    dft_r<B>(u, sign);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[(ea * k1 + eb * k2) % (A * B)] = u[k2];
  }
}
template <int R, typename C> __device__ __forceinline__ void dft_r(C* v, int sign) {
  if constexpr (R == 2) dft2(v, sign);
  else if constexpr (R == 3) dft3(v, sign);
  else if constexpr (R == 4) dft4(v, sign);
  else if constexpr (R == 5) dft5(v, sign);
  else if constexpr (R == 6) dft_coprime<2, 3>(v, sign);
  else if constexpr (R == 8) dft8(v, sign);
  else if constexpr (R == 9) dft9(v, sign);
  else if constexpr (R == 10) dft_coprime<2, 5>(v, sign);
  else if constexpr (R == 12) dft_coprime<4, 3>(v, sign);
  else if constexpr (R == 15) dft_coprime<3, 5>(v, sign);
  else if constexpr (R == 16) dft16(v, sign);
  else if constexpr (R == 18) dft_coprime<2, 9>(v, sign);
  else if constexpr (R == 20) dft_coprime<4, 5>(v, sign);
  else {
    static_assert(R == 25, "no butterfly of this radix");
    dft25(v, sign);
  }
}

// ---- lengths -----------------------------------------------------------------------------------
// Every length with a two-step plan, as X(N, A, B), N = A B, A <= B.  The sides serve the plane (at
// most 160 points) and the z lines, the long ones the z lines alone.  In groups, so that the
// double-float kernels (slow to compile) can be spread over translation units.
#define FDE_SPLIT_SIDES0(X) X(24, 4, 6) X(30, 5, 6) X(32, 4, 8) X(36, 6, 6) X(40, 5, 8) X(45, 5, 9) X(48, 6, 8)
#define FDE_SPLIT_SIDES1(X) X(50, 5, 10) X(54, 6, 9) X(60, 6, 10) X(64, 8, 8) X(72, 8, 9) X(75, 5, 15)
#define FDE_SPLIT_SIDES2(X) X(80, 8, 10) X(90, 9, 10) X(96, 8, 12) X(100, 10, 10) X(108, 9, 12) X(120, 10, 12)
#define FDE_SPLIT_SIDES3(X) X(128, 8, 16) X(135, 9, 15) X(144, 12, 12) X(150, 10, 15) X(160, 10, 16)
#define FDE_SPLIT_LONG0(X) X(162, 9, 18) X(180, 12, 15) X(192, 12, 16) X(200, 10, 20) X(216, 12, 18) X(225, 15, 15)
#define FDE_SPLIT_LONG1(X) \
  X(240, 15, 16) X(250, 10, 25) X(256, 16, 16) X(270, 15, 18) X(288, 16, 18) X(300, 15, 20) X(320, 16, 20)
#define FDE_SPLIT_SIDES(X) FDE_SPLIT_SIDES0(X) FDE_SPLIT_SIDES1(X) FDE_SPLIT_SIDES2(X) FDE_SPLIT_SIDES3(X)
#define FDE_SPLIT_LONG(X) FDE_SPLIT_LONG0(X) FDE_SPLIT_LONG1(X)
#define FDE_SPLIT_LINES(X) FDE_SPLIT_SIDES(X) FDE_SPLIT_LONG(X)

// (A, B) of a length: {0, 0} when it has no two-step plan.
struct Split {
  int a, b;
};
__host__ __device__ constexpr Split split_of(int n) {
  switch (n) {
#define FDE_CASE(N, A, B) \
  case N:                 \
    return Split{A, B};
    FDE_SPLIT_LINES(FDE_CASE)
#undef FDE_CASE
  }
  return Split{0, 0};
}
inline bool split_side_ok(int n) { return n <= 160 && split_of(n).a > 0; }

// Plan of a plane side N = R1 R2 (R1 >= R2).  Where N has coprime factors the two steps run on the
// prime-factor indices -- input n = (R2 r + R1 j) mod N, output k with k = q mod R1, k = p mod R2 -- and
// there are no twiddles between them: W_N^{nk} = W_R1^{rq} W_R2^{jp}.  That saves 14 % of the
// arithmetic of 72 = 9 x 8 and the loads of its 56 twiddles.  Other sides take the Cooley-Tukey
// indices n = j + R2 r, k = q + R1 p.
template <int R1_, int R2_> struct SidePlan {
  static constexpr int R1 = R1_, R2 = R2_, N = R1 * R2;
  static constexpr int gcd(int a, int b) { return b ? gcd(b, a % b) : a; }
  static constexpr bool kCoprime = gcd(R1, R2) == 1;
  // unit of q and of p in k (prime-factor form)
  static constexpr int E1 = kCoprime ? crt_index(R1, R2, 1 % R1, 0) : 0, E2 = kCoprime ? crt_index(R1, R2, 0, 1 % R2) : 0;
  // input index of element r of item j is in0(j) + R2 r, modulo N (each term below N)
  __host__ __device__ static constexpr int in0(int j) { return kCoprime ? R1 * j : j; }
  // output index of element p of item q is out0(q) + out(p), modulo N (each term below N)
  __host__ __device__ static constexpr int out0(int q) { return kCoprime ? q * E1 % N : q; }
  __host__ __device__ static constexpr int out(int p) { return kCoprime ? p * E2 % N : R1 * p; }
  __host__ __device__ static constexpr int wrap(int k) { return k >= N ? k - N : k; }
  __host__ __device__ static constexpr int output(int q, int p) {
    return kCoprime ? wrap(out0(q) + out(p)) : q + R1 * p;  // the latter never wraps
  }
};
// Sides as X(N, R1, R2), in the groups of FDE_SPLIT_SIDES.
#define FDE_PLANE_SIDES0(X) X(24, 8, 3) X(30, 6, 5) X(32, 8, 4) X(36, 9, 4) X(40, 8, 5) X(45, 9, 5) X(48, 16, 3)
#define FDE_PLANE_SIDES1(X) X(50, 10, 5) X(54, 9, 6) X(60, 12, 5) X(64, 8, 8) X(72, 9, 8) X(75, 15, 5)
#define FDE_PLANE_SIDES2(X) X(80, 16, 5) X(90, 10, 9) X(96, 12, 8) X(100, 10, 10) X(108, 12, 9) X(120, 15, 8)
#define FDE_PLANE_SIDES3(X) X(128, 16, 8) X(135, 15, 9) X(144, 16, 9) X(150, 15, 10) X(160, 16, 10)
#define FDE_PLANE_SIDES(X) FDE_PLANE_SIDES0(X) FDE_PLANE_SIDES1(X) FDE_PLANE_SIDES2(X) FDE_PLANE_SIDES3(X)

__host__ __device__ constexpr int round_up(int n, int m) { return (n + m - 1) / m * m; }

// x * W^e or x * conj(W^e) from the table tw[e] = exp(-2 pi i e / N).
template <typename C> __device__ __forceinline__ C twist(C x, C w, int sign) {
  if (sign > 0) w.y = -w.y;
  return cmul(x, w);
}

}  // namespace fde
