// What the register passes of the three axes share (zpass_reg.cuh, xpass_reg.cuh,
// ypass_reg.cuh): the DFTs next to the box, with the halves' packing and the twiddles,
// and the plans of odd lengths.
#pragma once

#include <type_traits>

#include "fft_reg.cuh"
#include "matvec_impl.cuh"

namespace dda {

// ---- R-point DFTs of both halves ------------------------------------------------
// The even half of step 1 is E_k = sum_j x_j w_R^(jk), the odd one
// O_k = sum_j x_j w_2R^(j (2k + 1)).  Rotating x_j by w_2R^j first and running the
// same DFT on both costs the odd half a layer of multiplications, with its roundings,
// more than its value needs.  With R = P M, P a power of two and M odd, a prime factor
// map takes the odd half apart as it does the even one: for each q < P an M-point DFT
// over m of sum_p (+-) x_j w_2P^(p (2q + 1)), j the index that is p mod P and m mod M
// (+-: the sign of w_2P^j / w_2P^p).  So odd R need signs only, R = 2 M exact rotations
// by i, and powers of two one layer of twiddles in both halves.  The frequencies of the
// two halves at one place of the map are k and (k + (M - 1) / 2) mod R: a row of the
// exchange holds that pair (reg_odd_shift), and step 2 counts its odd frequencies from
// there.  Round trip of an (8, 8), (9, 9), (10, 5) and (16, 16) axis against 64 bits,
// rotating first and so: 1.60, 1.81, 1.69, 2.01 and 1.57, 1.73, 1.56, 1.96 x 2^-24 (RMS).
struct eo { cv<float> e, o; };

template <int R> struct EoMap {
  static constexpr int pow2(int r) { return r % 2 ? 1 : 2 * pow2(r / 2); }
  static constexpr int P = pow2(R), M = R / P;
  // 1/R = ale/P + bee/M (mod 1)
  static constexpr int ale = cx_inv_mod(M % P, P), bee = cx_inv_mod(P % M, M);
  static constexpr int j(int p, int m) {
    int i = 0;
    while (i % P != p || i % M != m) ++i;
    return i;
  }
  static constexpr bool neg(int i) { return i % (2 * P) >= P; }
  // the even half's frequency at (q, mu)
  static constexpr int k(int q, int mu) {
    int i = 0;
    while (ale * i % P != q || bee * i % M != mu) ++i;
    return i;
  }
};

// B-point DFTs of both halves, packed
template <int B, bool INV> __device__ __forceinline__ void eo_pair_dft(eo (&t)[B]) {
  cv<f32p> a[B];
#pragma unroll
  for (int i = 0; i < B; ++i) a[i] = {pk_make(t[i].e.re, t[i].o.re), pk_make(t[i].e.im, t[i].o.im)};
  rdft<B, INV>(a);
#pragma unroll
  for (int i = 0; i < B; ++i) {
    pk_split(a[i].re, t[i].e.re, t[i].o.re);
    pk_split(a[i].im, t[i].e.im, t[i].o.im);
  }
}
// a w_DEN^NUM, or a conj(w_DEN^NUM)
template <bool INV, int NUM, int DEN> __device__ __forceinline__ cv<float> eo_rot(cv<float> a) {
  constexpr int n = NUM % DEN;
  if constexpr (n == 0) return a;
  else if constexpr (2 * n == DEN) return {-a.re, -a.im};
  else if constexpr (4 * n == DEN) return INV ? cv<float>{-a.im, a.re} : cv<float>{a.im, -a.re};
  else return cvrot<INV>(a, cx_cos(n, DEN), cx_sin(n, DEN));
}

// P a power of two: t[p] = (x_p, (+-) x_p) in, the halves' frequencies q out
template <int P> __device__ __forceinline__ void eo_dft(eo (&t)[P]) {
  if constexpr (P == 2) {
    const eo a = t[0], b = t[1];
    t[0] = {cvadd(a.e, b.e), {a.o.re + b.o.im, a.o.im - b.o.re}};
    t[1] = {cvsub(a.e, b.e), {a.o.re - b.o.im, a.o.im + b.o.re}};
  } else if constexpr (P > 2) {
    constexpr int A = P == 16 ? 4 : 2, B = P / A;  // x at p = B pa + pb
    static_for<B>([&](auto pbc) {
      constexpr int pb = decltype(pbc)::value;
      eo u[A];
      static_for<A>([&](auto i) { u[i] = t[B * i + pb]; });
      eo_dft<A>(u);
      static_for<A>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        t[B * q + pb] = {eo_rot<false, pb * q, P>(u[q].e),
                         eo_rot<false, pb * (2 * q + 1), 2 * P>(u[q].o)};
      });
    });
    eo out[P];
    static_for<A>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      eo u[B];
      static_for<B>([&](auto i) { u[i] = t[B * q + i]; });
      eo_pair_dft<B, false>(u);
      static_for<B>([&](auto i) { out[q + A * i] = u[i]; });
    });
    static_for<P>([&](auto i) { t[i] = out[i]; });
  }
}
// and back: t[p] = (E part, O part) of x_p = e + (+-) o
template <int P> __device__ __forceinline__ void eo_idft(eo (&t)[P]) {
  if constexpr (P == 2) {
    eo_pair_dft<2, true>(t);
    t[1].o = {-t[1].o.im, t[1].o.re};
  } else if constexpr (P > 2) {
    constexpr int A = P == 16 ? 4 : 2, B = P / A;
    eo v[P];
    static_for<A>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      eo u[B];
      static_for<B>([&](auto i) { u[i] = t[q + A * i]; });
      eo_pair_dft<B, true>(u);
      static_for<B>([&](auto pbc) {
        constexpr int pb = decltype(pbc)::value;
        v[B * q + pb] = {eo_rot<true, pb * q, P>(u[pb].e),
                         eo_rot<true, pb * (2 * q + 1), 2 * P>(u[pb].o)};
      });
    });
    static_for<B>([&](auto pbc) {
      constexpr int pb = decltype(pbc)::value;
      eo u[A];
      static_for<A>([&](auto i) { u[i] = v[B * i + pb]; });
      eo_idft<A>(u);
      static_for<A>([&](auto i) { t[B * i + pb] = u[i]; });
    });
  }
}

// x[0..R) to both halves' spectra: f[k] = (E_k, O at reg_odd_shift from k)
template <int R> __device__ __forceinline__ void eo_step(const float2 (&x)[R], eo (&f)[R]) {
  using K = EoMap<R>;
  eo u[R];  // [m][p]
  static_for<K::M>([&](auto mc) {
    constexpr int m = decltype(mc)::value;
    eo t[K::P];
    static_for<K::P>([&](auto pc) {
      constexpr int j = K::j(decltype(pc)::value, m);
      const cv<float> v{x[j].x, x[j].y};
      t[pc] = {v, K::neg(j) ? cv<float>{-v.re, -v.im} : v};
    });
    eo_dft<K::P>(t);
    static_for<K::P>([&](auto q) { u[m * K::P + q] = t[q]; });
  });
  static_for<K::P>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    eo t[K::M];
    static_for<K::M>([&](auto m) { t[m] = u[m * K::P + q]; });
    eo_pair_dft<K::M, false>(t);
    static_for<K::M>([&](auto muc) {
      constexpr int mu = decltype(muc)::value;
      f[K::k(q, mu)] = t[mu];
    });
  });
}
// and back, the halves joined.  R = 4 rotates the joined odd half instead: the rotation
// fuses with the sum (a round trip of a (4, 4) axis 1.29 against 1.31)
template <int R> __device__ __forceinline__ void eo_step_inv(const eo (&f)[R], float2 (&y)[R]) {
  using K = EoMap<R>;
  if constexpr (R == 4) {
    eo t[R];
    static_for<R>([&](auto i) { t[i] = f[i]; });
    eo_pair_dft<R, true>(t);
    static_for<R>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      constexpr float cw = (float)cx_cos(j, 2 * R), sw = (float)cx_sin(j, 2 * R);
      const cv<float> e = t[j].e, o = t[j].o;
      y[j] = make_float2(fmaf(cw, o.re, fmaf(-sw, o.im, e.re)), fmaf(cw, o.im, fmaf(sw, o.re, e.im)));
    });
  } else {
    eo u[R];
    static_for<K::P>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      eo t[K::M];
      static_for<K::M>([&](auto muc) {
        constexpr int mu = decltype(muc)::value;
        t[mu] = f[K::k(q, mu)];
      });
      eo_pair_dft<K::M, true>(t);
      static_for<K::M>([&](auto m) { u[m * K::P + q] = t[m]; });
    });
    static_for<K::M>([&](auto mc) {
      constexpr int m = decltype(mc)::value;
      eo t[K::P];
      static_for<K::P>([&](auto q) { t[q] = u[m * K::P + q]; });
      eo_idft<K::P>(t);
      static_for<K::P>([&](auto pc) {
        constexpr int j = K::j(decltype(pc)::value, m);
        const cv<float> v = K::neg(j) ? cvsub(t[pc].e, t[pc].o) : cvadd(t[pc].e, t[pc].o);
        y[j] = make_float2(v.re, v.im);
      });
    });
  }
}

// Step 1 of the passes: the R1-point DFTs (both halves') of a thread's inputs
// x[0..NJ), times the twiddles tw[k R2], to dst[k pitch] (elements of EL float2).
template <int R1, int R2, bool EO, int NJ>
__device__ __forceinline__ void reg_step1(const float2 (&x)[NJ], const float4* tw,
                                          float2* dst, int pitch) {
  if constexpr (EO) {
    eo f[R1];
    eo_step<R1>(x, f);
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      const float4 w = tw[k * R2];
      const cv<float> e = cvmul(f[k].e, cv<float>{w.x, w.y});
      const cv<float> o = cvmul(f[k].o, cv<float>{w.z, w.w});
      *reinterpret_cast<float4*>(dst + k * pitch) = make_float4(e.re, e.im, o.re, o.im);
    }
  } else {
    cv<float> a[R1];
#pragma unroll
    for (int j = 0; j < R1; ++j) a[j] = j < NJ ? cv<float>{x[j < NJ ? j : 0].x, x[j < NJ ? j : 0].y} : cv<float>{0.f, 0.f};
    rdft<R1, false>(a);
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      const float4 w = tw[k * R2];
      const cv<float> e = cvmul(a[k], cv<float>{w.x, w.y});
      dst[k * pitch] = make_float2(e.re, e.im);
    }
  }
}
// Its inverse in two parts, of which only the first reads shared memory: the elements
// src[k pitch], times the conjugate twiddles, and from them the outputs y[0..NJ).
template <bool EO> using reg_cv = std::conditional_t<EO, eo, cv<float>>;

template <int R1, int R2, bool EO>
__device__ __forceinline__ void reg_step1_inv_read(const float2* src, int pitch, const float4* tw,
                                                   reg_cv<EO> (&a)[R1]) {
#pragma unroll
  for (int k = 0; k < R1; ++k) {
    const float4 w = tw[k * R2];
    if constexpr (EO) {
      const float4 q = *reinterpret_cast<const float4*>(src + k * pitch);
      a[k] = {cvmulc(cv<float>{w.x, w.y}, cv<float>{q.x, q.y}),
              cvmulc(cv<float>{w.z, w.w}, cv<float>{q.z, q.w})};
    } else {
      const float2 q = src[k * pitch];
      a[k] = cvmulc(cv<float>{w.x, w.y}, cv<float>{q.x, q.y});
    }
  }
}

template <int R1, bool EO, int NJ>
__device__ __forceinline__ void reg_step1_inv_out(reg_cv<EO> (&a)[R1], float2 (&y)[NJ]) {
  if constexpr (EO) {
    eo_step_inv<R1>(a, y);
  } else {
    rdft<R1, true>(a);
#pragma unroll
    for (int j = 0; j < NJ; ++j) y[j] = make_float2(a[j].re, a[j].im);
  }
}

template <int R1, int R2, bool EO, int NJ>
__device__ __forceinline__ void reg_step1_inv(const float2* src, int pitch, const float4* tw,
                                              float2 (&y)[NJ]) {
  reg_cv<EO> a[R1];
  reg_step1_inv_read<R1, R2, EO>(src, pitch, tw, a);
  reg_step1_inv_out<R1, EO>(a, y);
}
// Step 2's threads are numbered q = 2 k1 + parity (or k1, odd lengths).  The frequency that
// the elements at q begin with (the others follow in steps of 2 R1, or R1), and the place
// of the elements that begin with frequency q.
template <int R1, bool EO> __device__ __forceinline__ int reg_freq(int q) {
  constexpr int shift = 2 * reg_odd_shift(R1);
  if (!EO || shift == 0 || !(q & 1)) return q;
  return q + shift < 2 * R1 ? q + shift : q + shift - 2 * R1;
}
template <int R1, bool EO> __device__ __forceinline__ int reg_place(int q) {
  constexpr int shift = 2 * reg_odd_shift(R1);
  if (!EO || shift == 0 || !(q & 1)) return q;
  return q >= shift ? q - shift : q - shift + 2 * R1;
}

// odd lengths R1 R2
#define DDA_XREG_ODD(X) X(5, 3) X(5, 5) X(9, 3) X(9, 5) X(15, 5) X(9, 9) X(15, 9) X(15, 15)
#define DDA_REG_NONE(X)

}  // namespace dda
