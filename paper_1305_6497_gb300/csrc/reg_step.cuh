// What the register passes of the three axes share (zpass_reg.cuh, xpass_reg.cuh,
// ypass_reg.cuh): the DFTs next to the box, with the halves' packing and the twiddles,
// and the plans of odd lengths.
#pragma once

#include <type_traits>

#include "fft_reg.cuh"
#include "matvec_impl.cuh"

namespace dda {

// Step 1 of the passes: the R1-point DFTs (both halves') of a thread's inputs
// x[0..NJ), times the twiddles tw[k R2], to dst[k pitch] (elements of EL float2).
template <int R1, int R2, bool EO, int NJ>
__device__ __forceinline__ void reg_step1(const float2 (&x)[NJ], const float4* tw,
                                          float2* dst, int pitch) {
  if constexpr (EO) {
    cv<f32p> a[R1];
    static_for<R1>([&](auto jc) {
      constexpr int j = decltype(jc)::value;  // w_L^(R2 j) = exp(-i pi j / R1)
      const cv<float> o =
          cvrot<false>(cv<float>{x[j].x, x[j].y}, cx_cos(j, 2 * R1), cx_sin(j, 2 * R1));
      a[j] = {pk_make(x[j].x, o.re), pk_make(x[j].y, o.im)};
    });
    rdft<R1, false>(a);
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      const float4 w = tw[k * R2];
      cv<float> e, o;
      pk_split(a[k].re, e.re, o.re);
      pk_split(a[k].im, e.im, o.im);
      e = cvmul(e, cv<float>{w.x, w.y});
      o = cvmul(o, cv<float>{w.z, w.w});
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
template <bool EO> using reg_cv = cv<std::conditional_t<EO, f32p, float>>;

template <int R1, int R2, bool EO>
__device__ __forceinline__ void reg_step1_inv_read(const float2* src, int pitch, const float4* tw,
                                                   reg_cv<EO> (&a)[R1]) {
#pragma unroll
  for (int k = 0; k < R1; ++k) {
    const float4 w = tw[k * R2];
    if constexpr (EO) {
      const float4 q = *reinterpret_cast<const float4*>(src + k * pitch);
      const cv<float> e = cvmulc(cv<float>{w.x, w.y}, cv<float>{q.x, q.y});
      const cv<float> o = cvmulc(cv<float>{w.z, w.w}, cv<float>{q.z, q.w});
      a[k] = {pk_make(e.re, o.re), pk_make(e.im, o.im)};
    } else {
      const float2 q = src[k * pitch];
      a[k] = cvmulc(cv<float>{w.x, w.y}, cv<float>{q.x, q.y});
    }
  }
}

template <int R1, bool EO, int NJ>
__device__ __forceinline__ void reg_step1_inv_out(reg_cv<EO> (&a)[R1], float2 (&y)[NJ]) {
  rdft<R1, true>(a);
  if constexpr (EO) {
    static_for<R1>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      constexpr float cw = (float)cx_cos(j, 2 * R1), sw = (float)cx_sin(j, 2 * R1);
      float re, im, ro, io;
      pk_split(a[j].re, re, ro);
      pk_split(a[j].im, im, io);
      y[j] = make_float2(fmaf(cw, ro, fmaf(-sw, io, re)), fmaf(cw, io, fmaf(sw, ro, im)));
    });
  } else {
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
// odd lengths R1 R2
#define DDA_XREG_ODD(X) X(5, 3) X(5, 5) X(9, 3) X(9, 5) X(15, 5) X(9, 9) X(15, 9) X(15, 15)
#define DDA_REG_NONE(X)

}  // namespace dda
