// y passes in two register transforms (FP32), for y lengths L = 2n, n = R1 R2, in
// place on a tile of columns: the transform of zpass_reg.cuh with the plans of
// xpass_reg.cuh.  Forward: threads (column, j2) read the ny rows j2 + R2 j1, and
// threads (column, k1, parity) write the L rows 2 (k1 + R1 k2) + parity, in natural
// order; the inverse the other way round.  One exchange through shared memory
// ([k1][j2][column] 16-byte pairs, conflict-free) and one barrier.  A tile is 16
// columns (whole 128-byte lines), except that n = 129..191 takes 8: there 16 leave
// too few CTAs per SM (136 rows: 53 us against 47, 150: 46 against 42), while
// above the whole lines win again (256 rows: 66 against 80, 225: 41 against 49).
//
// What bounds it: HBM on grids larger than L2 (256^3 box: 4.8 GB in 901 us, 0.79 of
// the measured copy rate), latency on smaller ones.  Forward / inverse pass, two
// right-hand sides, before (shared-memory stages, compiled or generic plans) and
// now: 128^3 168 / 203 -> 116 / 105 us, 256^3 1000 / 1013 -> 901 / 939, 100x75x135
// 179 / 142 -> 70 / 60, 60x45x54 31 / 31 -> 12.5 / 12.3, 64^3 19 / 19 -> 18 / 18.
#pragma once

#include "xpass_reg.cuh"

namespace dda {

template <int R1, int R2> struct YRegCfg {
  static constexpr int n = R1 * R2, L = 2 * n;
  static constexpr int TILE = n <= 128 || n >= 192 ? 16 : 8;
  static constexpr int U1 = TILE * R2, U2 = TILE * 2 * R1;
  static constexpr int most = ((U1 > U2 ? U1 : U2) + 31) / 32 * 32;
  static constexpr int NT = most > 320 ? (most / 2 + 31) / 32 * 32 : most;
  static constexpr size_t smem = (size_t)n * TILE * 16;
  static constexpr int regs = (4 * R1 > 2 * R2 ? 4 * R1 : 2 * R2) + 44;
  static constexpr int by_regs = 65536 / (NT * ((regs + 7) / 8 * 8));
  static constexpr int by_smem = (int)(227 * 1024 / (smem + 1024));
  static constexpr int fit = by_regs < by_smem ? by_regs : by_smem;
  static constexpr int MINB = fit < 1 ? 1 : fit > 2048 / NT ? 2048 / NT : fit;
};

template <int R1, int R2, bool INV>
__global__ void __launch_bounds__(YRegCfg<R1, R2>::NT, YRegCfg<R1, R2>::MINB)
k_y_reg(OpView<float> op, float2* __restrict__ buf, const int* __restrict__ active) {
  using K = YRegCfg<R1, R2>;
  constexpr int TILE = K::TILE, NT = K::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* sm = reinterpret_cast<float4*>(smem_raw);
  const int r = blockIdx.z;
  if (active && !active[r]) return;
  const int Lx = op.Lx, ny = op.ny;
  const int col0 = blockIdx.x * TILE;
  const int ncol = min(TILE, Lx - col0);
  float2* base = buf + ((int64_t)r * 3 * op.nz + blockIdx.y) * (int64_t)K::L * Lx + col0;
  const float4* __restrict__ tw = op.twy_reg;
  // step 1's threads hold rows j2 + R2 j1 of one column, step 2's the frequencies
  // 2 (k1 + R1 k2) + p; a half-warp of step 2 covers 8 columns x both parities
  auto place2 = [&](int u, int& t, int& p, int& k1) {
    t = u % 8;
    p = (u / 8) & 1;
    const int h = u / 16;
    t += 8 * (h % (TILE / 8));
    k1 = h / (TILE / 8);
  };
  if (!INV) {
    for (int u = threadIdx.x; u < K::U1; u += NT) {
      const int t = u % TILE, j2 = u / TILE;
      const float2* src = base + (int64_t)j2 * Lx + min(t, ncol - 1);
      const bool last = j2 + R2 * (R1 - 1) < ny;  // row < ny holds for the other j1
      float2 x[R1];
#pragma unroll
      for (int j = 0; j < R1; ++j) x[j] = __ldcg(src + (j < R1 - 1 || last ? j * R2 * Lx : 0));
      if (!last) x[R1 - 1] = make_float2(0.f, 0.f);
      cv<f32p> a[R1];
      static_for<R1>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        const cv<float> o =
            cvrot<false>(cv<float>{x[j].x, x[j].y}, cx_cos(j, 2 * R1), cx_sin(j, 2 * R1));
        a[j] = {pk_make(x[j].x, o.re), pk_make(x[j].y, o.im)};
      });
      rdft<R1, false>(a);
#pragma unroll
      for (int k = 0; k < R1; ++k) {
        const float4 w = __ldg(tw + k * R2 + j2);
        cv<float> e, o;
        pk_split(a[k].re, e.re, o.re);
        pk_split(a[k].im, e.im, o.im);
        e = cvmul(e, cv<float>{w.x, w.y});
        o = cvmul(o, cv<float>{w.z, w.w});
        sm[(k * R2 + j2) * TILE + t] = make_float4(e.re, e.im, o.re, o.im);
      }
    }
    __syncthreads();
    for (int u = threadIdx.x; u < K::U2; u += NT) {
      int t, p, k1;
      place2(u, t, p, k1);
      const float2* s = reinterpret_cast<const float2*>(sm + k1 * R2 * TILE + t) + p;
      cv<float> a[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) {
        const float2 e = s[2 * TILE * j];
        a[j] = {e.x, e.y};
      }
      rdft<R2, false>(a);
      if (t < ncol) {
        float2* dst = base + (int64_t)(2 * k1 + p) * Lx + t;
#pragma unroll
        for (int k = 0; k < R2; ++k) dst[(int64_t)2 * R1 * k * Lx] = make_float2(a[k].re, a[k].im);
      }
    }
  } else {
    for (int u = threadIdx.x; u < K::U2; u += NT) {
      int t, p, k1;
      place2(u, t, p, k1);
      const float2* src = base + (int64_t)(2 * k1 + p) * Lx + min(t, ncol - 1);
      cv<float> a[R2];
#pragma unroll
      for (int k = 0; k < R2; ++k) {
        const float2 e = __ldcg(src + (int64_t)2 * R1 * k * Lx);
        a[k] = {e.x, e.y};
      }
      rdft<R2, true>(a);
      float2* s = reinterpret_cast<float2*>(sm + k1 * R2 * TILE + t) + p;
#pragma unroll
      for (int j = 0; j < R2; ++j) s[2 * TILE * j] = make_float2(a[j].re, a[j].im);
    }
    __syncthreads();
    for (int u = threadIdx.x; u < K::U1; u += NT) {
      const int t = u % TILE, j2 = u / TILE;
      if (t >= ncol) continue;
      const bool last = j2 + R2 * (R1 - 1) < ny;
      cv<f32p> a[R1];
#pragma unroll
      for (int k = 0; k < R1; ++k) {
        const float4 q = sm[(k * R2 + j2) * TILE + t], w = __ldg(tw + k * R2 + j2);
        const cv<float> e = cvmulc(cv<float>{w.x, w.y}, cv<float>{q.x, q.y});
        const cv<float> o = cvmulc(cv<float>{w.z, w.w}, cv<float>{q.z, q.w});
        a[k] = {pk_make(e.re, o.re), pk_make(e.im, o.im)};
      }
      rdft<R1, true>(a);
      float2* dst = base + (int64_t)j2 * Lx + t;
      static_for<R1>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        constexpr float cw = (float)cx_cos(j, 2 * R1), sw = (float)cx_sin(j, 2 * R1);
        float re, im, ro, io;
        pk_split(a[j].re, re, ro);
        pk_split(a[j].im, im, io);
        if (j < R1 - 1 || last)
          dst[(int64_t)j * R2 * Lx] = make_float2(fmaf(cw, ro, fmaf(-sw, io, re)),
                                                  fmaf(cw, io, fmaf(sw, ro, im)));
      });
    }
  }
}

template <int R1, int R2>
void launch_y_reg(bool inv, const OpView<float>& op, int R, float2* buf, const int* active,
                  cudaStream_t st) {
  using K = YRegCfg<R1, R2>;
  const dim3 g((op.Lx + K::TILE - 1) / K::TILE, 3 * op.nz, R);
  if (inv) k_y_reg<R1, R2, true><<<g, K::NT, K::smem, st>>>(op, buf, active);
  else k_y_reg<R1, R2, false><<<g, K::NT, K::smem, st>>>(op, buf, active);
}
template <int R1, int R2> cudaError_t configure_y_reg() {
  const cudaError_t e = cudaFuncSetAttribute(
      k_y_reg<R1, R2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)YRegCfg<R1, R2>::smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_y_reg<R1, R2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)YRegCfg<R1, R2>::smem);
}

// The plans of the x passes, in parts that compile side by side (ypass_reg_*.cu).
#define DDA_YREG_PART0(X) DDA_XREG_PART0(X) DDA_XREG_PART1(X)
#define DDA_YREG_PART1(X) DDA_XREG_PART2(X) DDA_XREG_PART3(X)
#define DDA_YREG_PART2(X) DDA_XREG_PART4(X) DDA_XREG_PART5(X)
#define DDA_YREG_PART3(X) DDA_XREG_PART6(X) DDA_XREG_PART7(X)
#define DDA_YREG_DECLARE(PART)                                                                    \
  bool launch_y_reg_part##PART(bool inv, const OpView<float>& op, int R, float2* buf,             \
                               const int* active, cudaStream_t st);                               \
  cudaError_t configure_y_reg_part##PART(int half);
DDA_YREG_DECLARE(0) DDA_YREG_DECLARE(1) DDA_YREG_DECLARE(2) DDA_YREG_DECLARE(3)

#define DDA_YREG_LAUNCH(A, B) case (A) * (B): launch_y_reg<A, B>(inv, op, R, buf, active, st); return true;
#define DDA_YREG_CONFIG(A, B) case (A) * (B): return configure_y_reg<A, B>();
#define DDA_YREG_DEFINE(PART)                                                                     \
  bool launch_y_reg_part##PART(bool inv, const OpView<float>& op, int R, float2* buf,             \
                               const int* active, cudaStream_t st) {                              \
    switch (op.Ly / 2) { DDA_YREG_PART##PART(DDA_YREG_LAUNCH) }                                   \
    return false;                                                                                 \
  }                                                                                               \
  cudaError_t configure_y_reg_part##PART(int half) {                                               \
    switch (half) { DDA_YREG_PART##PART(DDA_YREG_CONFIG) }                                         \
    return cudaSuccess;                                                                            \
  }

}  // namespace dda
