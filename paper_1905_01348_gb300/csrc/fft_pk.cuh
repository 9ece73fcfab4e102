// Short-line FFTs on values of one type V with members re and im: packed pairs of FP32 lines
// (pk2) and single FP64 or FP32 lines (cd, cf). Every codelet spells out its fused multiply-adds.
//
// A pk2 holds the same element of two independent lines, (re, re) and (im, im). The
// packed FP32 instructions of sm_100 and later (add / mul / fma on two floats) then do
// two lines per instruction: every rotation by a shared twiddle, +-i or a real constant
// needs no swap inside a register pair, unlike one complex value per register pair.
//
// A line of L = 8 M points (L in {32, 48, 64, 96}, M = 4, 6, 8, 12), n = n1 + M n2,
// k = k2 + 8 k1, takes two steps: 8-point DFTs over n2 with the twiddle W_L^(n1 k2), then
// M-point DFTs over n1. The inverse runs the steps backwards. 6 = 2 x 3 and 12 = 3 x 4 are
// prime-factor DFTs (Good 1958): coprime factors, so an index map takes the place of
// twiddles. An inverse R-point DFT is the forward one with outputs k and R - k exchanged.
#pragma once

#include "common.cuh"

namespace pt {

struct __align__(16) pk2 {
  float2 re, im;
};
struct __align__(16) cd {
  double re, im;
};
struct __align__(8) cf {
  float re, im;
};

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __fadd2_rn(a, vneg(b)); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
// a constant in the component type of V
template <typename V> struct konst;
template <> struct konst<pk2> { __device__ __forceinline__ static float2 of(double a) { return f2((float)a); } };
template <> struct konst<cf> { __device__ __forceinline__ static float of(double a) { return (float)a; } };
template <> struct konst<cd> { __device__ __forceinline__ static double of(double a) { return a; } };
// a b - c d and c - a: the packed fma takes no negated operand for free (two integer
// instructions per pair), a factor of -1 does
__device__ __forceinline__ float2 vminus(float2 c, float2 a) { return __ffma2_rn(a, f2(-1.f), c); }
__device__ __forceinline__ float2 vdet(float2 a, float2 b, float2 c, float2 d) { return vminus(vmul(a, b), vmul(c, d)); }
__device__ __forceinline__ double vminus(double c, double a) { return c - a; }
__device__ __forceinline__ float vminus(float c, float a) { return c - a; }
__device__ __forceinline__ float vdet(float a, float b, float c, float d) { return fmaf(-c, d, a * b); }
__device__ __forceinline__ double vdet(double a, double b, double c, double d) { return fma(-c, d, a * b); }

template <typename V> __device__ __forceinline__ V padd(V a, V b) { return {vadd(a.re, b.re), vadd(a.im, b.im)}; }
template <typename V> __device__ __forceinline__ V psub(V a, V b) { return {vsub(a.re, b.re), vsub(a.im, b.im)}; }
// a - i b and a + i b
template <typename V> __device__ __forceinline__ V psub_i(V a, V b) { return {vadd(a.re, b.im), vsub(a.im, b.re)}; }
template <typename V> __device__ __forceinline__ V padd_i(V a, V b) { return {vsub(a.re, b.im), vadd(a.im, b.re)}; }
// a (c - i s) (forward twiddle) and a (c + i s) (inverse); w = (c, c, s, s)
template <bool INV, typename V> __device__ __forceinline__ V ptwiddle(V a, V w) {
  const auto c = w.re, s = w.im;
  return INV ? V{vdet(a.re, c, a.im, s), vfma(a.re, s, vmul(a.im, c))}
             : V{vfma(a.im, s, vmul(a.re, c)), vdet(a.im, c, a.re, s)};
}

template <typename V> __device__ __forceinline__ void pk_dft4(V& x0, V& x1, V& x2, V& x3) {
  const V a = padd(x0, x2), b = psub(x0, x2), c = padd(x1, x3), d = psub(x1, x3);
  x0 = padd(a, c);
  x2 = psub(a, c);
  x1 = psub_i(b, d);
  x3 = padd_i(b, d);
}

template <typename V> __device__ __forceinline__ void pk_dft3(V& x0, V& x1, V& x2) {
  constexpr double sin60 = 0.86602540378443864676;
  const auto mh = konst<V>::of(-0.5), s3 = konst<V>::of(sin60), n3 = konst<V>::of(-sin60);
  const V s = padd(x1, x2), d = psub(x1, x2);
  const V t = {vfma(s.re, mh, x0.re), vfma(s.im, mh, x0.im)};
  x0 = padd(x0, s);
  x1 = {vfma(d.im, s3, t.re), vfma(d.re, n3, t.im)};
  x2 = {vfma(d.im, n3, t.re), vfma(d.re, s3, t.im)};
}

template <typename V> __device__ __forceinline__ void pk_dft8(V* x) {
  constexpr double r = 0.70710678118654752440;
  const auto h = konst<V>::of(r), nh = konst<V>::of(-r);
  pk_dft4(x[0], x[2], x[4], x[6]);
  pk_dft4(x[1], x[3], x[5], x[7]);
  const V e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
  x[0] = padd(e0, o0);
  x[4] = psub(e0, o0);
  // W8 o1 = h (o1.re + o1.im, o1.im - o1.re), W8^3 o3 = h (o3.im - o3.re, -(o3.re + o3.im))
  const auto p = vadd(o1.re, o1.im), q = vsub(o1.im, o1.re);
  x[1] = {vfma(p, h, e1.re), vfma(q, h, e1.im)};
  x[5] = {vfma(p, nh, e1.re), vfma(q, nh, e1.im)};
  x[2] = psub_i(e2, o2);
  x[6] = padd_i(e2, o2);
  const auto u = vsub(o3.im, o3.re), v = vadd(o3.re, o3.im);
  x[3] = {vfma(u, h, e3.re), vfma(v, nh, e3.im)};
  x[7] = {vfma(u, nh, e3.re), vfma(v, h, e3.im)};
}

// 6 = 2 x 3: n = 3 a + 2 b, k = 3 c + 4 d (mod 6)
template <typename V> __device__ __forceinline__ void pk_dft6(V* x) {
  V y[2][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const V u = x[(2 * b) % 6], v = x[(3 + 2 * b) % 6];
    y[0][b] = padd(u, v);
    y[1][b] = psub(u, v);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    pk_dft3(y[c][0], y[c][1], y[c][2]);
#pragma unroll
    for (int d = 0; d < 3; ++d) x[(3 * c + 4 * d) % 6] = y[c][d];
  }
}

// 12 = 3 x 4: n = 4 a + 3 b, k = 4 c + 9 d (mod 12)
template <typename V> __device__ __forceinline__ void pk_dft12(V* x) {
  V y[3][4];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int b = 0; b < 4; ++b) y[a][b] = x[(4 * a + 3 * b) % 12];
    pk_dft4(y[a][0], y[a][1], y[a][2], y[a][3]);
  }
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    pk_dft3(y[0][d], y[1][d], y[2][d]);
#pragma unroll
    for (int c = 0; c < 3; ++c) x[(4 * c + 9 * d) % 12] = y[c][d];
  }
}

// 16 = 4 x 4: n = a + 4 b, k = 4 c + d with the twiddle W16^(a d)
template <typename V> __device__ __forceinline__ void pk_dft16(V* x) {
  const auto c1 = konst<V>::of(0.92387953251128675613), s1 = konst<V>::of(0.38268343236508977173);
  const auto h = konst<V>::of(0.70710678118654752440), nh = konst<V>::of(-0.70710678118654752440);
  const auto n1 = konst<V>::of(-0.92387953251128675613), m1 = konst<V>::of(-0.38268343236508977173);
  V y[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int b = 0; b < 4; ++b) y[a][b] = x[a + 4 * b];
    pk_dft4(y[a][0], y[a][1], y[a][2], y[a][3]);
  }
  y[1][1] = ptwiddle<false>(y[1][1], V{c1, s1});
  y[1][2] = ptwiddle<false>(y[1][2], V{h, h});
  y[1][3] = ptwiddle<false>(y[1][3], V{s1, c1});
  y[2][1] = ptwiddle<false>(y[2][1], V{h, h});
  y[2][2] = {y[2][2].im, vneg(y[2][2].re)};
  y[2][3] = ptwiddle<false>(y[2][3], V{nh, h});
  y[3][1] = ptwiddle<false>(y[3][1], V{s1, c1});
  y[3][2] = ptwiddle<false>(y[3][2], V{nh, h});
  y[3][3] = ptwiddle<false>(y[3][3], V{n1, m1});
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    pk_dft4(y[0][d], y[1][d], y[2][d], y[3][d]);
#pragma unroll
    for (int c = 0; c < 4; ++c) x[4 * c + d] = y[c][d];
  }
}

// 24 = 3 x 8: n = 8 a + 3 b, k = 16 c + 9 d (mod 24)
template <typename V> __device__ __forceinline__ void pk_dft24(V* x) {
#pragma unroll
  for (int b = 0; b < 8; ++b) pk_dft3(x[(3 * b) % 24], x[(8 + 3 * b) % 24], x[(16 + 3 * b) % 24]);
  V y[3][8];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int b = 0; b < 8; ++b) y[c][b] = x[(8 * c + 3 * b) % 24];
    pk_dft8(y[c]);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int d = 0; d < 8; ++d) x[(16 * c + 9 * d) % 24] = y[c][d];
}

template <int R, bool INV, typename V> __device__ __forceinline__ void pk_dft(V* x) {
  static_assert(R == 1 || R == 2 || R == 3 || R == 4 || R == 6 || R == 8 || R == 12 || R == 16 || R == 24, "radix of a packed DFT");
  if constexpr (R == 1) return;
  else if constexpr (R == 2) {
    const V t = x[1];
    x[1] = psub(x[0], t);
    x[0] = padd(x[0], t);
  } else if constexpr (R == 3) pk_dft3(x[0], x[1], x[2]);
  else if constexpr (R == 4) pk_dft4(x[0], x[1], x[2], x[3]);
  else if constexpr (R == 6) pk_dft6(x);
  else if constexpr (R == 8) pk_dft8(x);
  else if constexpr (R == 12) pk_dft12(x);
  else if constexpr (R == 16) pk_dft16(x);
  else pk_dft24(x);
  if constexpr (INV) {
#pragma unroll
    for (int k = 1; k < (R + 1) / 2; ++k) {
      const V t = x[k];
      x[k] = x[R - k];
      x[R - k] = t;
    }
  }
}

}  // namespace pt
