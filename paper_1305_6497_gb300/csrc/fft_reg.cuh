// DFTs of up to 20 points in registers, on scalar values or on packed pairs.
//
// The element type V is float, double, double-float, or f32p: two FP32 numbers in one 64-bit
// register pair, worked on by the packed instructions {add,sub,mul,fma}.rn.f32x2.
// On this part a packed instruction occupies the FP32 pipe as long as two scalar
// ones (60 lanes per clock and SM measured, against 118), but takes one issue slot
// instead of two, which leaves issue slots to the loads, stores and address
// arithmetic that a transform is made of.
//
// Every DFT takes and leaves its points in natural order (forward:
// exp(-2 pi i jk/R), INV: the conjugate, neither normalised).
#pragma once

#include <type_traits>
#include <utility>

#include "dda_common.cuh"

namespace dda {

struct f32p { unsigned long long v; };

__device__ __forceinline__ f32p pk_make(float lo, float hi) {
  f32p r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void pk_split(f32p a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ f32p vadd(f32p a, f32p b) {
  f32p r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32p vsub(f32p a, f32p b) {
  f32p r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32p vmul(f32p a, f32p b) {
  f32p r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32p vfma(f32p a, f32p b, f32p c) {
  f32p r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ df64 vadd(df64 a, df64 b) { return a + b; }
__device__ __forceinline__ df64 vsub(df64 a, df64 b) { return a - b; }
__device__ __forceinline__ df64 vmul(df64 a, df64 b) { return a * b; }
// a b + c with one renormalisation: the product's leading part, its error (exact by
// FMA) and the low-order terms; 15 instructions against 18 of a product and a sum
__device__ __forceinline__ df64 vfma(df64 a, df64 b, df64 c) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  const float s = __fadd_rn(p, c.hi), bb = __fsub_rn(s, p);
  const float r = __fadd_rn(__fsub_rn(p, __fsub_rn(s, bb)), __fsub_rn(c.hi, bb));
  return df_fast2sum(s, __fadd_rn(r, __fadd_rn(e, c.lo)));
}
__device__ __forceinline__ df64 vneg(df64 a) { return -a; }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

template <typename V> __device__ __forceinline__ V vconst(double c) { return (V)c; }
template <> __device__ __forceinline__ df64 vconst<df64>(double c) { return df64(c); }
template <> __device__ __forceinline__ f32p vconst<f32p>(double c) {
  return pk_make((float)c, (float)c);
}

// c - a / 2 (exact scaling)
__device__ __forceinline__ f32p vsub_half(f32p c, f32p a) { return vfma(vconst<f32p>(-0.5), a, c); }
__device__ __forceinline__ float vsub_half(float c, float a) { return fmaf(-0.5f, a, c); }
__device__ __forceinline__ double vsub_half(double c, double a) { return fma(-0.5, a, c); }
__device__ __forceinline__ df64 vsub_half(df64 c, df64 a) {
  return c + df64(-0.5f * a.hi, -0.5f * a.lo);
}

template <typename V> struct cv { V re, im; };

template <typename V> __device__ __forceinline__ cv<V> cvadd(cv<V> a, cv<V> b) {
  return {vadd(a.re, b.re), vadd(a.im, b.im)};
}
template <typename V> __device__ __forceinline__ cv<V> cvsub(cv<V> a, cv<V> b) {
  return {vsub(a.re, b.re), vsub(a.im, b.im)};
}
__device__ __forceinline__ f32p vneg(f32p a) {
  f32p r;
  r.v = a.v ^ 0x8000000080000000ull;
  return r;
}
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
// a b, and conj(a) b
template <typename V> __device__ __forceinline__ cv<V> cvmul(cv<V> a, cv<V> b) {
  return {vfma(vneg(a.im), b.im, vmul(a.re, b.re)), vfma(a.re, b.im, vmul(a.im, b.re))};
}
template <typename V> __device__ __forceinline__ cv<V> cvmulc(cv<V> a, cv<V> b) {
  return {vfma(a.re, b.re, vmul(a.im, b.im)), vfma(a.re, b.im, vmul(vneg(a.im), b.re))};
}
// Double-float products: both products of a part are split exactly, their leading
// parts added with the sum's error, everything else in one low-order sum -- 19
// instructions a part where two products and a sum take 25, and one rounding less.
__device__ __forceinline__ df64 df_dot2(df64 a, df64 b, df64 c, df64 d) {  // a b + c d
  const float p = __fmul_rn(a.hi, b.hi), q = __fmul_rn(c.hi, d.hi);
  float e = __fadd_rn(__fmaf_rn(a.hi, b.hi, -p), __fmaf_rn(c.hi, d.hi, -q));
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  e = __fmaf_rn(c.hi, d.lo, e);
  e = __fmaf_rn(c.lo, d.hi, e);
  const float s = __fadd_rn(p, q), bb = __fsub_rn(s, p);
  const float r = __fadd_rn(__fsub_rn(p, __fsub_rn(s, bb)), __fsub_rn(q, bb));
  return df_fast2sum(s, __fadd_rn(r, e));
}
template <> __device__ __forceinline__ cv<df64> cvmul(cv<df64> a, cv<df64> b) {
  return {df_dot2(a.re, b.re, vneg(a.im), b.im), df_dot2(a.re, b.im, a.im, b.re)};
}
template <> __device__ __forceinline__ cv<df64> cvmulc(cv<df64> a, cv<df64> b) {
  return {df_dot2(a.re, b.re, a.im, b.im), df_dot2(a.re, b.im, vneg(a.im), b.re)};
}
// a b + c
template <typename V> __device__ __forceinline__ cv<V> cvmad(cv<V> a, cv<V> b, cv<V> c) {
  return {vfma(vneg(a.im), b.im, vfma(a.re, b.re, c.re)), vfma(a.re, b.im, vfma(a.im, b.re, c.im))};
}
// a (c - i s) forward, a (c + i s) inverse: constants c, s
template <bool INV, typename V>
__device__ __forceinline__ cv<V> cvrot(cv<V> a, double c, double s) {
  const V cc = vconst<V>(c), sp = vconst<V>(INV ? -s : s), sn = vconst<V>(INV ? s : -s);
  return {vfma(cc, a.re, vmul(sp, a.im)), vfma(cc, a.im, vmul(sn, a.re))};
}

template <bool INV> __device__ __forceinline__ cv<df64> cvrot(cv<df64> a, double c, double s) {
  const df64 cc(c), sp(INV ? -s : s), sn(INV ? s : -s);
  return {df_dot2(cc, a.re, sp, a.im), df_dot2(cc, a.im, sn, a.re)};
}
// On packed pairs the rotations by constants run on the two halves: a scalar
// multiply takes its constant as an immediate, a packed one needs it twice in a
// register pair, which costs more moves than the packing saves issue slots.
template <bool INV> __device__ __forceinline__ cv<f32p> cvrot(cv<f32p> a, double c, double s) {
  cv<float> l, h;
  pk_split(a.re, l.re, h.re);
  pk_split(a.im, l.im, h.im);
  l = cvrot<INV, float>(l, c, s);
  h = cvrot<INV, float>(h, c, s);
  return {pk_make(l.re, h.re), pk_make(l.im, h.im)};
}

// cos and sin of 2 pi num/den at compile time (Taylor series on |x| <= pi/4)
constexpr double kPiC = 3.14159265358979323846264338327950288;
constexpr double cx_cos_small(double x) {
  double t = 1.0, s = 1.0;
  for (int n = 1; n < 16; ++n) { t *= -x * x / ((2.0 * n - 1.0) * (2.0 * n)); s += t; }
  return s;
}
constexpr double cx_sin_small(double x) {
  double t = x, s = x;
  for (int n = 1; n < 16; ++n) { t *= -x * x / ((2.0 * n) * (2.0 * n + 1.0)); s += t; }
  return s;
}
// num/den of a turn, reduced by eighths so that exact values stay exact
constexpr double cx_sin(int num, int den);
constexpr double cx_cos(int num, int den) {
  num %= den;
  if (num < 0) num += den;
  if (2 * num > den) num = den - num;                            // cos(-x) = cos x
  if (4 * num > den) return -cx_cos(den - 2 * num, 2 * den);     // cos(pi - x) = -cos x
  if (4 * num == den) return 0.0;
  if (8 * num > den) return cx_sin_small(2.0 * kPiC * (0.25 - (double)num / den));
  return cx_cos_small(2.0 * kPiC * num / den);
}
constexpr double cx_sin(int num, int den) { return cx_cos(4 * num - den, 4 * den); }

template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F> __device__ __forceinline__ void static_for(F&& f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// ---- prime-power kernels --------------------------------------------------------
template <typename V> __device__ __forceinline__ void rdft2(cv<V>& a, cv<V>& b) {
  const cv<V> t = cvsub(a, b);
  a = cvadd(a, b);
  b = t;
}
template <bool INV, typename V>
__device__ __forceinline__ void rdft4(cv<V>& a0, cv<V>& a1, cv<V>& a2, cv<V>& a3) {
  const cv<V> s02 = cvadd(a0, a2), d02 = cvsub(a0, a2);
  const cv<V> s13 = cvadd(a1, a3), d13 = cvsub(a1, a3);
  a0 = cvadd(s02, s13);
  a2 = cvsub(s02, s13);
  const cv<V> m{vadd(d02.re, d13.im), vsub(d02.im, d13.re)};  // d02 - i d13
  const cv<V> p{vsub(d02.re, d13.im), vadd(d02.im, d13.re)};  // d02 + i d13
  a1 = INV ? p : m;
  a3 = INV ? m : p;
}
// sqrt(3) / 2.  Its FP32 value is 0.30 x 2^-24 too small, and every 3-point DFT scales what
// it passes on by (1 - 0.1 x 2^-24) on average: the one error of a chain of them that
// adds up instead of averaging out.  UP: the FP32 neighbour above, 0.86 x 2^-24 too large,
// which one DFT in four takes to balance it (the 9-point DFT, see rdft_ct).
template <typename V, bool UP> __device__ __forceinline__ constexpr double sqrt3_half() {
  constexpr bool f32 = std::is_same<V, float>::value || std::is_same<V, f32p>::value;
  return UP && f32 ? 0.866025447845458984375 : cx_sin(1, 3);
}
template <bool INV, bool UP = false, typename V>
__device__ __forceinline__ void rdft3(cv<V>& a0, cv<V>& a1, cv<V>& a2) {
  constexpr double c = sqrt3_half<V, UP>();
  const V s = vconst<V>(INV ? -c : c), sn = vconst<V>(INV ? c : -c);
  const cv<V> t = cvadd(a1, a2), d = cvsub(a1, a2);
  const cv<V> u{vsub_half(a0.re, t.re), vsub_half(a0.im, t.im)};
  a0 = cvadd(a0, t);
  a1 = {vfma(s, d.im, u.re), vfma(sn, d.re, u.im)};  // u - i s d
  a2 = {vfma(sn, d.im, u.re), vfma(s, d.re, u.im)};  // u + i s d
}
template <bool INV, typename V>
__device__ __forceinline__ void rdft5(cv<V>& a0, cv<V>& a1, cv<V>& a2, cv<V>& a3, cv<V>& a4) {
  const V c1 = vconst<V>(cx_cos(1, 5)), c2 = vconst<V>(cx_cos(2, 5));
  const V s1 = vconst<V>(INV ? -cx_sin(1, 5) : cx_sin(1, 5)),
          s2 = vconst<V>(INV ? -cx_sin(2, 5) : cx_sin(2, 5)),
          s1n = vconst<V>(INV ? cx_sin(1, 5) : -cx_sin(1, 5));
  const cv<V> t1 = cvadd(a1, a4), t2 = cvadd(a2, a3), t3 = cvsub(a1, a4), t4 = cvsub(a2, a3);
  const cv<V> b1{vfma(c1, t1.re, vfma(c2, t2.re, a0.re)), vfma(c1, t1.im, vfma(c2, t2.im, a0.im))};
  const cv<V> b2{vfma(c2, t1.re, vfma(c1, t2.re, a0.re)), vfma(c2, t1.im, vfma(c1, t2.im, a0.im))};
  const cv<V> u1{vfma(s1, t3.re, vmul(s2, t4.re)), vfma(s1, t3.im, vmul(s2, t4.im))};
  const cv<V> u2{vfma(s2, t3.re, vmul(s1n, t4.re)), vfma(s2, t3.im, vmul(s1n, t4.im))};
  a0 = cvadd(a0, cvadd(t1, t2));
  a1 = {vadd(b1.re, u1.im), vsub(b1.im, u1.re)};  // b1 - i u1
  a4 = {vsub(b1.re, u1.im), vadd(b1.im, u1.re)};
  a2 = {vadd(b2.re, u2.im), vsub(b2.im, u2.re)};
  a3 = {vsub(b2.re, u2.im), vadd(b2.im, u2.re)};
}
template <bool INV, typename V> __device__ __forceinline__ void rdft8(cv<V> (&a)[8]) {
  rdft4<INV>(a[0], a[2], a[4], a[6]);
  rdft4<INV>(a[1], a[3], a[5], a[7]);
  const V h = vconst<V>(0.70710678118654752440), hn = vconst<V>(-0.70710678118654752440);
  const cv<V> e1 = a[2], e2 = a[4], e3 = a[6], o1 = a[3], o2 = a[5], o3 = a[7];
  const cv<V> e0 = a[0], o0 = a[1];
  a[0] = cvadd(e0, o0);
  a[4] = cvsub(e0, o0);
  // w8 o1 = h ((re + im), (im - re)) forward, h ((re - im), (im + re)) inverse
  const V p1 = INV ? vsub(o1.re, o1.im) : vadd(o1.re, o1.im);
  const V q1 = INV ? vadd(o1.im, o1.re) : vsub(o1.im, o1.re);
  a[1] = {vfma(h, p1, e1.re), vfma(h, q1, e1.im)};
  a[5] = {vfma(hn, p1, e1.re), vfma(hn, q1, e1.im)};
  const cv<V> m{vadd(e2.re, o2.im), vsub(e2.im, o2.re)}, p{vsub(e2.re, o2.im), vadd(e2.im, o2.re)};
  a[2] = INV ? p : m;
  a[6] = INV ? m : p;
  // w8^3 o3 = h ((im - re), -(re + im)) forward, h (-(re + im), (re - im)) inverse
  const V p3 = INV ? vadd(o3.re, o3.im) : vsub(o3.im, o3.re);
  const V q3 = INV ? vsub(o3.re, o3.im) : vadd(o3.re, o3.im);
  if (INV) {
    a[3] = {vfma(hn, p3, e3.re), vfma(h, q3, e3.im)};
    a[7] = {vfma(h, p3, e3.re), vfma(hn, q3, e3.im)};
  } else {
    a[3] = {vfma(h, p3, e3.re), vfma(hn, q3, e3.im)};
    a[7] = {vfma(hn, p3, e3.re), vfma(h, q3, e3.im)};
  }
}
// a b^T form: R = A B as B-point DFTs of A-strided points, twiddles, A-point DFTs.
template <int R, bool INV, typename V> __device__ __forceinline__ void rdft(cv<V> (&a)[R]);

// R = A B, any A, B: x[j], j = B ja + jb; X[ka + A kb]
template <int A, int B, bool INV, typename V>
__device__ __forceinline__ void rdft_ct(cv<V> (&a)[A * B]) {
  static_for<B>([&](auto jbc) {
    constexpr int jb = decltype(jbc)::value;
    cv<V> t[A];
    static_for<A>([&](auto i) { t[i] = a[B * i + jb]; });
    // of the twelve 3-point DFTs of a 9-point one and its inverse, these three take the
    // larger sqrt(3) / 2: round trip of a (9, 9) axis 2.02 -> 1.73 x 2^-24
    if constexpr (A == 3 && B == 3 && INV) rdft3<INV, true>(t[0], t[1], t[2]);
    else rdft<A, INV>(t);
    static_for<A>([&](auto kac) {
      constexpr int ka = decltype(kac)::value;
      constexpr int num = (jb * ka) % (A * B);
      if constexpr (num == 0) {
        a[B * ka + jb] = t[ka];
      } else if constexpr (4 * num == A * B) {
        // -i (forward), +i (inverse)
        if (INV) a[B * ka + jb] = {vneg(t[ka].im), t[ka].re};
        else a[B * ka + jb] = {t[ka].im, vneg(t[ka].re)};
      } else {
        constexpr double c = cx_cos(num, A * B), s = cx_sin(num, A * B);
        a[B * ka + jb] = cvrot<INV>(t[ka], c, s);
      }
    });
  });
  cv<V> out[A * B];
  static_for<A>([&](auto kac) {
    constexpr int ka = decltype(kac)::value;
    cv<V> t[B];
    static_for<B>([&](auto i) { t[i] = a[B * ka + i]; });
    rdft<B, INV>(t);
    static_for<B>([&](auto i) { out[ka + A * i] = t[i]; });
  });
  static_for<A * B>([&](auto i) { a[i] = out[i]; });
}
constexpr int cx_inv_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if ((a * i) % m == 1) return i;
  return 1;
}
// R = A B with A, B coprime (Good-Thomas: no twiddles)
template <int A, int B, bool INV, typename V>
__device__ __forceinline__ void rdft_pfa(cv<V> (&a)[A * B]) {
  constexpr int R = A * B;
  cv<V> m[R];  // [n2][k1]
  static_for<B>([&](auto n2c) {
    constexpr int n2 = decltype(n2c)::value;
    cv<V> t[A];
    static_for<A>([&](auto i) { t[i] = a[(B * i + A * n2) % R]; });
    rdft<A, INV>(t);
    static_for<A>([&](auto i) { m[n2 * A + i] = t[i]; });
  });
  constexpr int ea = B * cx_inv_mod(B % A, A), eb = A * cx_inv_mod(A % B, B);
  static_for<A>([&](auto k1c) {
    constexpr int k1 = decltype(k1c)::value;
    cv<V> t[B];
    static_for<B>([&](auto i) { t[i] = m[i * A + k1]; });
    rdft<B, INV>(t);
    static_for<B>([&](auto i) { a[(ea * k1 + eb * i) % R] = t[i]; });
  });
}
// 16 = 4 x 4: the twiddle w16^4 = -i folds into the second DFT's additions
template <bool INV, typename V> __device__ __forceinline__ void rdft16(cv<V> (&a)[16]) {
  constexpr double c1 = cx_cos(1, 16), s1 = cx_sin(1, 16), h = 0.70710678118654752440;
#pragma unroll
  for (int j = 0; j < 4; ++j) rdft4<INV>(a[j], a[4 + j], a[8 + j], a[12 + j]);
  // a[4 k + j] holds y_j[k]; twiddles w16^(j k)
  a[5] = cvrot<INV>(a[5], c1, s1);
  a[6] = cvrot<INV>(a[6], h, h);
  a[7] = cvrot<INV>(a[7], s1, c1);
  a[9] = cvrot<INV>(a[9], h, h);
  a[11] = cvrot<INV>(a[11], -h, h);
  a[13] = cvrot<INV>(a[13], s1, c1);
  a[14] = cvrot<INV>(a[14], -h, h);
  a[15] = cvrot<INV>(a[15], -c1, -s1);
  rdft4<INV>(a[0], a[1], a[2], a[3]);
  rdft4<INV>(a[4], a[5], a[6], a[7]);
  {
    // row k = 2: a2 still wants w16^4 = -i (+i): s02 = a0 - i a2, d02 = a0 + i a2
    const cv<V> a0 = a[8], a1 = a[9], a2 = a[10], a3 = a[11];
    const cv<V> m{vadd(a0.re, a2.im), vsub(a0.im, a2.re)}, p{vsub(a0.re, a2.im), vadd(a0.im, a2.re)};
    const cv<V> s02 = INV ? p : m, d02 = INV ? m : p;
    const cv<V> s13 = cvadd(a1, a3), d13 = cvsub(a1, a3);
    a[8] = cvadd(s02, s13);
    a[10] = cvsub(s02, s13);
    const cv<V> mm{vadd(d02.re, d13.im), vsub(d02.im, d13.re)};
    const cv<V> pp{vsub(d02.re, d13.im), vadd(d02.im, d13.re)};
    a[9] = INV ? pp : mm;
    a[11] = INV ? mm : pp;
  }
  rdft4<INV>(a[12], a[13], a[14], a[15]);
  // a[4 k + m] holds X[k + 4 m]
  cv<V> t[16];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int m = 0; m < 4; ++m) t[k + 4 * m] = a[4 * k + m];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = t[i];
}

template <int R, bool INV, typename V> __device__ __forceinline__ void rdft(cv<V> (&a)[R]) {
  if constexpr (R == 2) rdft2(a[0], a[1]);
  else if constexpr (R == 3) rdft3<INV>(a[0], a[1], a[2]);
  else if constexpr (R == 4) rdft4<INV>(a[0], a[1], a[2], a[3]);
  else if constexpr (R == 5) rdft5<INV>(a[0], a[1], a[2], a[3], a[4]);
  else if constexpr (R == 6) rdft_pfa<2, 3, INV>(a);
  else if constexpr (R == 8) rdft8<INV>(a);
  else if constexpr (R == 9) rdft_ct<3, 3, INV>(a);
  else if constexpr (R == 10) rdft_pfa<2, 5, INV>(a);
  else if constexpr (R == 12) rdft_pfa<4, 3, INV>(a);
  else if constexpr (R == 15) rdft_pfa<3, 5, INV>(a);
  else if constexpr (R == 16) rdft16<INV>(a);
  else if constexpr (R == 18) rdft_pfa<2, 9, INV>(a);
  else if constexpr (R == 20) rdft_pfa<4, 5, INV>(a);
  else static_assert(R == 1, "no DFT of this length");
}

}  // namespace dda
