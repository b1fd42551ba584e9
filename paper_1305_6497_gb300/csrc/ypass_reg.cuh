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
// What bounds it: HBM on grids larger than L2 (256^3 box: 4.8 GB in 875 us, 0.81 of
// the measured copy rate), latency on smaller ones.  Forward / inverse pass, two
// right-hand sides, before (shared-memory stages, compiled or generic plans) and
// now: 128^3 168 / 203 -> 116 / 106 us, 256^3 1000 / 1013 -> 875 / 936, 100x75x135
// 179 / 142 -> 69 / 61, 60x45x54 31 / 31 -> 12.3 / 12.2, 64^3 19 / 19 -> 18 / 18.
#pragma once

#include "xpass_reg.cuh"

namespace dda {

template <int R1, int R2, bool EO = true> struct YRegCfg {
  static constexpr int n = R1 * R2, L = EO ? 2 * n : n;
  static constexpr int NJ = XRegCfg<R1, R2, EO>::NJ, NQ = XRegCfg<R1, R2, EO>::NQ;
  static constexpr int EL = EO ? 2 : 1;  // float2 per element
  static constexpr int TILE = n <= 128 || n >= 192 ? 16 : 8;
  static constexpr int U1 = TILE * R2, U2 = TILE * NQ;
  static constexpr int most = ((U1 > U2 ? U1 : U2) + 31) / 32 * 32;
  static constexpr int NT = most > 320 ? (most / 2 + 31) / 32 * 32 : most;
  static constexpr size_t smem = (size_t)n * TILE * 8 * EL;
  static constexpr int regs = (4 * R1 > 2 * R2 ? 4 * R1 : 2 * R2) + 44;
  static constexpr int by_regs = 65536 / (NT * ((regs + 7) / 8 * 8));
  static constexpr int by_smem = (int)(227 * 1024 / (smem + 1024));
  static constexpr int fit = by_regs < by_smem ? by_regs : by_smem;
  static constexpr int MINB = fit < 1 ? 1 : fit > 2048 / NT ? 2048 / NT : fit;
};

template <int R1, int R2, bool EO, bool INV>
__global__ void __launch_bounds__(YRegCfg<R1, R2, EO>::NT, YRegCfg<R1, R2, EO>::MINB)
k_y_reg(OpView<float> op, float2* buf, const int* active) {
  using K = YRegCfg<R1, R2, EO>;
  constexpr int TILE = K::TILE, NT = K::NT, NJ = K::NJ, NQ = K::NQ, EL = K::EL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  const int r = blockIdx.z;
  chain_next();
  chain_wait();
  active = chained(active);
  buf = chained(buf);
  if (active && !active[r]) return;
  const int Lx = op.Lx, ny = op.ny;
  const int col0 = blockIdx.x * TILE;
  const int ncol = min(TILE, Lx - col0);
  float2* base = buf + ((int64_t)r * 3 * op.nz + blockIdx.y) * (int64_t)K::L * Lx + col0;
  const float4* __restrict__ tw = op.twy_reg;
  // step 1's threads hold rows j2 + R2 j1 of one column, step 2's the frequencies
  // q + NQ k2 (q = 2 k1 + parity, or k1); with two parities a half-warp of step 2
  // covers 8 columns x both
  auto place2 = [&](int u, int& t, int& q) {
    if (EO) {
      const int h = u / 16;
      t = u % 8 + 8 * (h % (TILE / 8));
      q = 2 * (h / (TILE / 8)) + ((u / 8) & 1);
    } else {
      t = u % TILE;
      q = u / TILE;
    }
  };
  auto element = [&](int t, int q) {
    const int at = reg_place<R1, EO>(q);
    return sm + EL * ((EO ? at >> 1 : at) * R2 * TILE + t) + (EO ? at & 1 : 0);
  };
  if (!INV) {
    for (int u = threadIdx.x; u < K::U1; u += NT) {
      const int t = u % TILE, j2 = u / TILE;
      const float2* src = base + (int64_t)j2 * Lx + min(t, ncol - 1);
      const bool last = j2 + R2 * (NJ - 1) < ny;  // row < ny holds for the other j1
      float2 x[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) x[j] = __ldcg(src + (j < NJ - 1 || last ? j * R2 * Lx : 0));
      if (!last) x[NJ - 1] = make_float2(0.f, 0.f);
      reg_step1<R1, R2, EO>(x, tw + j2, sm + EL * (j2 * TILE + t), EL * R2 * TILE);
    }
    __syncthreads();
    for (int u = threadIdx.x; u < K::U2; u += NT) {
      int t, q;
      place2(u, t, q);
      const float2* s = element(t, q);
      cv<float> a[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) {
        const float2 e = s[EL * TILE * j];
        a[j] = {e.x, e.y};
      }
      rdft<R2, false>(a);
      if (t < ncol) {
        float2* dst = base + (int64_t)q * Lx + t;
#pragma unroll
        for (int k = 0; k < R2; ++k) dst[(int64_t)NQ * k * Lx] = make_float2(a[k].re, a[k].im);
      }
    }
  } else {
    for (int u = threadIdx.x; u < K::U2; u += NT) {
      int t, q;
      place2(u, t, q);
      const float2* src = base + (int64_t)q * Lx + min(t, ncol - 1);
      cv<float> a[R2];
#pragma unroll
      for (int k = 0; k < R2; ++k) {
        const float2 e = __ldcg(src + (int64_t)NQ * k * Lx);
        a[k] = {e.x, e.y};
      }
      rdft<R2, true>(a);
      float2* s = element(t, q);
#pragma unroll
      for (int j = 0; j < R2; ++j) s[EL * TILE * j] = make_float2(a[j].re, a[j].im);
    }
    __syncthreads();
    for (int u = threadIdx.x; u < K::U1; u += NT) {
      const int t = u % TILE, j2 = u / TILE;
      if (t >= ncol) continue;
      const bool last = j2 + R2 * (NJ - 1) < ny;
      float2 y[NJ];
      reg_step1_inv<R1, R2, EO>(sm + EL * (j2 * TILE + t), EL * R2 * TILE, tw + j2, y);
      float2* dst = base + (int64_t)j2 * Lx + t;
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (j < NJ - 1 || last) dst[(int64_t)j * R2 * Lx] = y[j];
    }
  }
}

template <int R1, int R2, bool EO>
void launch_y_reg(bool inv, const OpView<float>& op, int R, float2* buf, const int* active,
                  cudaStream_t st) {
  using K = YRegCfg<R1, R2, EO>;
  const dim3 g((op.Lx + K::TILE - 1) / K::TILE, 3 * op.nz, R);
  // the inverse pass of a solve is not chained (see launch_chained)
  launch_chained(inv ? op.chain == 1 : op.chain != 0,
                 inv ? k_y_reg<R1, R2, EO, true> : k_y_reg<R1, R2, EO, false>, g, K::NT, K::smem, st,
                 op, buf, active);
}
template <int R1, int R2, bool EO> cudaError_t configure_y_reg() {
  const int smem = (int)YRegCfg<R1, R2, EO>::smem;
  const cudaError_t e = cudaFuncSetAttribute(
      k_y_reg<R1, R2, EO, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_y_reg<R1, R2, EO, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              smem);
}

// The plans of the x passes, in parts that compile side by side (ypass_reg_*.cu).
#define DDA_YREG_PART0(X) DDA_XREG_PART0(X) DDA_XREG_PART1(X)
#define DDA_YREG_PART1(X) DDA_XREG_PART2(X) DDA_XREG_PART3(X)
#define DDA_YREG_PART2(X) DDA_XREG_PART4(X) DDA_XREG_PART5(X)
#define DDA_YREG_PART3(X) DDA_XREG_PART6(X) DDA_XREG_PART7(X)
#define DDA_YREG_DECLARE(PART)                                                                    \
  bool launch_y_reg_part##PART(bool inv, const OpView<float>& op, int R, float2* buf,             \
                               const int* active, cudaStream_t st);                               \
  cudaError_t configure_y_reg_part##PART(int L);
DDA_YREG_DECLARE(0) DDA_YREG_DECLARE(1) DDA_YREG_DECLARE(2) DDA_YREG_DECLARE(3)

#define DDA_YREG_LAUNCH(A, B) \
  case 2 * (A) * (B): launch_y_reg<A, B, true>(inv, op, R, buf, active, st); return true;
#define DDA_YREG_CONFIG(A, B) case 2 * (A) * (B): return configure_y_reg<A, B, true>();
#define DDA_YREG_LAUNCH_ODD(A, B) \
  case (A) * (B): launch_y_reg<A, B, false>(inv, op, R, buf, active, st); return true;
#define DDA_YREG_CONFIG_ODD(A, B) case (A) * (B): return configure_y_reg<A, B, false>();
// ODDS: the list of odd plans, or nothing
#define DDA_YREG_DEFINE(PART, ODDS)                                                               \
  bool launch_y_reg_part##PART(bool inv, const OpView<float>& op, int R, float2* buf,             \
                               const int* active, cudaStream_t st) {                              \
    switch (op.Ly) { DDA_YREG_PART##PART(DDA_YREG_LAUNCH) ODDS(DDA_YREG_LAUNCH_ODD) }             \
    return false;                                                                                 \
  }                                                                                               \
  cudaError_t configure_y_reg_part##PART(int L) {                                                 \
    switch (L) { DDA_YREG_PART##PART(DDA_YREG_CONFIG) ODDS(DDA_YREG_CONFIG_ODD) }                 \
    return cudaSuccess;                                                                           \
  }
}  // namespace dda
