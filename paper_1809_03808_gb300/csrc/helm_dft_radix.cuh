// In-register R-point DFTs shared by the power-of-two and the mixed-radix
// transforms: y_q = sum_r v_r e^{SIGN 2 pi i r q / R}, natural order in and
// out, R in {2 .. 10, 16}.
#pragma once

#include "helm_kernels.cuh"

namespace helm {

// (SIGN i) a
template <typename C, int SIGN>
__device__ __forceinline__ C mul_si(C a) {
  C o;
  if (SIGN > 0) {
    o.x = -a.y;
    o.y = a.x;
  } else {
    o.x = a.y;
    o.y = -a.x;
  }
  return o;
}

// (cr + i ci) a for compile-time constants
template <typename C>
__device__ __forceinline__ C mul_c(C a, double cr, double ci) {
  using T = decltype(a.x);
  C o;
  o.x = a.x * (T)cr - a.y * (T)ci;
  o.y = a.x * (T)ci + a.y * (T)cr;
  return o;
}

// In-register R-point DFTs, natural order in and out:
// y_q = sum_r v_r e^{SIGN 2 pi i r q / R}.
template <typename C, int SIGN>
__device__ __forceinline__ void dft2(C* v) {
  const C a = v[0];
  v[0] = cadd(a, v[1]);
  v[1] = csub(a, v[1]);
}

template <typename C, int SIGN>
__device__ __forceinline__ void dft4s(C& v0, C& v1, C& v2, C& v3) {
  const C t0 = cadd(v0, v2), t1 = csub(v0, v2), t2 = cadd(v1, v3), t3 = mul_si<C, SIGN>(csub(v1, v3));
  v0 = cadd(t0, t2);
  v1 = cadd(t1, t3);
  v2 = csub(t0, t2);
  v3 = csub(t1, t3);
}

template <typename C, int SIGN>
__device__ __forceinline__ void dft4(C* v) {
  dft4s<C, SIGN>(v[0], v[1], v[2], v[3]);
}

constexpr double kH = 0.70710678118654752440;   // cos(pi/4)
constexpr double kC8 = 0.92387953251128675613;  // cos(pi/8)
constexpr double kS8 = 0.38268343236508977173;  // sin(pi/8)

template <typename C, int SIGN>
__device__ __forceinline__ void dft8(C* v) {
  // even and odd halves: E_q in v[2q], O_q in v[2q+1]
  dft4s<C, SIGN>(v[0], v[2], v[4], v[6]);
  dft4s<C, SIGN>(v[1], v[3], v[5], v[7]);
  const double s = SIGN;
  const C o1 = mul_c(v[3], kH, s * kH);     // W8^1 O_1
  const C o2 = mul_si<C, SIGN>(v[5]);       // W8^2 O_2
  const C o3 = mul_c(v[7], -kH, s * kH);    // W8^3 O_3
  const C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1);
  v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2);
  v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3);
  v[7] = csub(e3, o3);
}

template <typename C, int SIGN>
__device__ __forceinline__ void dft16(C* v) {
  // r = b + 4a: DFT4 over a for each b (results Z_b[q1] at v[b + 4 q1])
#pragma unroll
  for (int b = 0; b < 4; ++b) dft4s<C, SIGN>(v[b], v[b + 4], v[b + 8], v[b + 12]);
  // twiddles W16^{b q1}
  const double s = SIGN;
  v[5] = mul_c(v[5], kC8, s * kS8);     // b1 q1 = 1
  v[9] = mul_c(v[9], kH, s * kH);       // b1 q2 = 2
  v[13] = mul_c(v[13], kS8, s * kC8);   // b1 q3 = 3
  v[6] = mul_c(v[6], kH, s * kH);       // b2 q1 = 2
  v[10] = mul_si<C, SIGN>(v[10]);       // b2 q2 = 4
  v[14] = mul_c(v[14], -kH, s * kH);    // b2 q3 = 6
  v[7] = mul_c(v[7], kS8, s * kC8);     // b3 q1 = 3
  v[11] = mul_c(v[11], -kH, s * kH);    // b3 q2 = 6
  v[15] = mul_c(v[15], -kC8, -s * kS8); // b3 q3 = 9
  // DFT4 over b for each q1: y[q1 + 4 q2] lands at v[4 q1 + q2]
#pragma unroll
  for (int q1 = 0; q1 < 4; ++q1) dft4s<C, SIGN>(v[4 * q1], v[4 * q1 + 1], v[4 * q1 + 2], v[4 * q1 + 3]);
  C y[16];
#pragma unroll
  for (int q1 = 0; q1 < 4; ++q1)
#pragma unroll
    for (int q2 = 0; q2 < 4; ++q2) y[q1 + 4 * q2] = v[4 * q1 + q2];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = y[i];
}

// cos(2 pi k / R) and sin(2 pi k / R), 1 <= k <= (R - 1) / 2, R odd; folded
// at compile time in the unrolled loops below.
template <int R>
__host__ __device__ constexpr double root_cos(int k) {
  if (R == 3) return -0.5000000000000000000000;
  if (R == 5) return k == 1 ? 0.3090169943749474241023 : -0.8090169943749474241023;
  if (R == 7) return k == 1 ? 0.6234898018587335305250 : k == 2 ? -0.2225209339563144042889 : -0.9009688679024191262361;
  if (R == 9) return k == 1 ? 0.7660444431189780352024 : k == 2 ? 0.1736481776669303488517 : k == 3 ? -0.5000000000000000000000 : -0.9396926207859083840541;
  return 0.0;
}
template <int R>
__host__ __device__ constexpr double root_sin(int k) {
  if (R == 3) return 0.8660254037844386467637;
  if (R == 5) return k == 1 ? 0.9510565162951535721164 : 0.5877852522924731291687;
  if (R == 7) return k == 1 ? 0.7818314824680298087084 : k == 2 ? 0.9749279121818236070181 : 0.4338837391175581204758;
  if (R == 9) return k == 1 ? 0.6427876096865393263226 : k == 2 ? 0.9848077530122080593667 : k == 3 ? 0.8660254037844386467637 : 0.3420201433256687330441;
  return 0.0;
}

// Odd prime R (forward, SIGN = -1): with s_r = v_r + v_{R-r}, d_r = v_r -
// v_{R-r}, y_q = a_q - i b_q and y_{R-q} = a_q + i b_q, a_q = v_0 + sum_r
// cos(2 pi q r / R) s_r, b_q = sum_r sin(2 pi q r / R) d_r: half the products
// of the direct sum, real coefficients.
template <typename C, int R>
__device__ __forceinline__ void dft_odd(C* v) {
  using T = decltype(v[0].x);
  constexpr int H = (R - 1) / 2;
  C s[H + 1], d[H + 1];
#pragma unroll
  for (int r = 1; r <= H; ++r) {
    s[r] = cadd(v[r], v[R - r]);
    d[r] = csub(v[r], v[R - r]);
  }
  const C v0 = v[0];
#pragma unroll
  for (int r = 1; r <= H; ++r) v[0] = cadd(v[0], s[r]);
#pragma unroll
  for (int q = 1; q <= H; ++q) {
    C a = v0, b = mk<C>(0, 0);
#pragma unroll
    for (int r = 1; r <= H; ++r) {
      const int e = (q * r) % R;
      const T c = (T)root_cos<R>(e <= H ? e : R - e);
      const T sn = e <= H ? (T)root_sin<R>(e) : -(T)root_sin<R>(R - e);
      a.x = fma(c, s[r].x, a.x);
      a.y = fma(c, s[r].y, a.y);
      b.x = r == 1 ? sn * d[r].x : fma(sn, d[r].x, b.x);
      b.y = r == 1 ? sn * d[r].y : fma(sn, d[r].y, b.y);
    }
    v[q].x = a.x + b.y;
    v[q].y = a.y - b.x;
    v[R - q].x = a.x - b.y;
    v[R - q].y = a.y + b.x;
  }
}

template <typename C, int R>
__device__ __forceinline__ void dft_fwd(C* v);

// R = 9 as 3 x 3 with the twiddles e^{-2 pi i b q / 9}
template <typename C>
__device__ __forceinline__ void dft_nine(C* v) {
  C t[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
#pragma unroll
    for (int a = 0; a < 3; ++a) t[b][a] = v[b + 3 * a];
    dft_odd<C, 3>(t[b]);
  }
  t[1][1] = mul_c(t[1][1], root_cos<9>(1), -root_sin<9>(1));
  t[1][2] = mul_c(t[1][2], root_cos<9>(2), -root_sin<9>(2));
  t[2][1] = mul_c(t[2][1], root_cos<9>(2), -root_sin<9>(2));
  t[2][2] = mul_c(t[2][2], root_cos<9>(4), -root_sin<9>(4));
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    C w[3] = {t[0][q], t[1][q], t[2][q]};
    dft_odd<C, 3>(w);
#pragma unroll
    for (int p = 0; p < 3; ++p) v[q + 3 * p] = w[p];
  }
}

__host__ __device__ constexpr int inv_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if (a % m * x % m == 1) return x;
  return 1;
}

// R = A B with A and B coprime (Good's prime-factor index maps: no twiddles)
template <typename C, int A, int B>
__device__ __forceinline__ void dft_pfa(C* v) {
  constexpr int R = A * B;
  constexpr int EA = B * inv_mod(B, A), EB = A * inv_mod(A, B);
  C t[A][B];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    C w[A];
#pragma unroll
    for (int a = 0; a < A; ++a) w[a] = v[(B * a + A * b) % R];
    dft_fwd<C, A>(w);
#pragma unroll
    for (int a = 0; a < A; ++a) t[a][b] = w[a];
  }
#pragma unroll
  for (int a = 0; a < A; ++a) {
    dft_fwd<C, B>(t[a]);
#pragma unroll
    for (int b = 0; b < B; ++b) v[(EA * a + EB * b) % R] = t[a][b];
  }
}

// Forward R-point DFT, R in {2 .. 10}.
template <typename C, int R>
__device__ __forceinline__ void dft_fwd(C* v) {
  if constexpr (R == 2) dft2<C, -1>(v);
  else if constexpr (R == 4) dft4<C, -1>(v);
  else if constexpr (R == 8) dft8<C, -1>(v);
  else if constexpr (R == 9) dft_nine<C>(v);
  else if constexpr (R == 6) dft_pfa<C, 2, 3>(v);
  else if constexpr (R == 10) dft_pfa<C, 2, 5>(v);
  else dft_odd<C, R>(v);
}

}  // namespace helm
