// x passes in two register transforms (FP32), for x lengths L = 2n, n = R1 R2:
// the transform of zpass_reg.cuh (even and odd frequencies as the halves of packed
// pairs, R1-point and R2-point DFTs in registers with one exchange) on the rows of
// the box, with the vector updates of k_fft_x_fwd and the inner products of
// k_fft_x_inv at its ends.
//
// A warp owns LW rows and needs no other: the exchange goes through the warp's
// own shared memory between two warp barriers, so no warp waits for a CTA.  Step 1
// works on rows x R2 threads, step 2 on rows x 2 R1; LW is chosen so that both fill
// their rounds of 32 lanes.  Spectra leave (and come back) in natural order,
// frequency 2 (k1 + R1 k2) + parity = q + 2 R1 k2 for q = 2 k1 + parity: a row's
// stores for one k2 are 2 R1 consecutive values, its loads of box vectors R2.
//
// Shared memory: [row][k1][j2] 16-byte (even, odd) pairs, k1 rows an odd number of
// pairs apart, so that step 2's half-warps (k1, parity) hit distinct banks.  A row's odd
// half belongs to another k1 (reg_place); the other way round, with natural rows here
// and the odd frequencies permuted in the spectra, a warp's stores fell into more
// 32-byte sectors (216 points: 63.4 us where this takes 60.6).
//
// What bounds it: HBM on grids larger than L2 (256^3 box: the update of p and its
// transform move 4.8 GB in 648 us, all of the measured copy rate, the inverse with its
// inner products 4.1 GB in 661 us, 0.91 of it), load latency on smaller ones.  The
// kernels that keep lines in shared memory ran a third of the warps, each CTA waiting for
// its slowest stage.  Forward / inverse pass, two right-hand sides, before and now: 256^3
// box 1135 / 1319 -> 648 / 661 us, 128^3 164 / 202 -> 87 / 92, 64^3 29 / 43 -> 17 / 23,
// 100x75x135 98 / 121 -> 48 / 64, 16^3 17 / 26 -> 7 / 11.5 us.
#pragma once

#include "reg_step.cuh"

namespace dda {

constexpr int kXRegWarps = 4;  // per CTA

// EO: L = 2 R1 R2, even and odd frequencies as halves; otherwise L = R1 R2 is odd and
// the line is transformed whole, its rows j1 >= NJ zero.
template <int R1, int R2, bool EO = true> struct XRegCfg {
  static constexpr int n = R1 * R2, L = EO ? 2 * n : n;
  static constexpr int NJ = EO ? R1 : ((L + 1) / 2 + R2 - 1) / R2;
  static constexpr int NQ = EO ? 2 * R1 : R1;        // step 2's threads per row
  static constexpr int EL = EO ? 2 : 1;              // float2 per element
  static constexpr int ROW = R2 | 1, LS = R1 * ROW;  // elements per k1 and per line
  // issue slots a row costs with LW rows per warp (a packed R1-point DFT against a
  // scalar R2-point one), the least of LW = 1..4
  static constexpr int cost(int lw) {
    return ((lw * R2 + 31) / 32 * R1 * (EO ? 22 : 14) + (lw * NQ + 31) / 32 * R2 * 14) * 12 / lw;
  }
  static constexpr int pick() {
    int b = 1;
    for (int i = 2; i <= 4; ++i)
      if (cost(i) < cost(b)) b = i;
    return b;
  }
  static constexpr int LW = pick();
  static constexpr int U1 = LW * R2, U2 = LW * NQ;
  static constexpr size_t smem = (size_t)kXRegWarps * LW * LS * 8 * EL;
  static constexpr int regs = (4 * R1 > 2 * R2 ? 4 * R1 : 2 * R2) + 48;
  static constexpr int by_regs = 65536 / (32 * kXRegWarps * ((regs + 7) / 8 * 8));
  static constexpr int MINB = by_regs > 8 ? 8 : by_regs;
};

// CTAs per right-hand side: every warp takes up to 8 groups of LW rows, one while
// that leaves fewer CTAs than the chip holds
inline int x_reg_grid(int rows, int LW) {
  const int per = kXRegWarps * LW, one = (rows + per - 1) / per;
  int loops = one / (152 * 8);
  loops = loops < 1 ? 1 : loops > 8 ? 8 : loops;
  return (one + loops - 1) / loops;
}

template <int R1, int R2, bool EO, int MODE>
__global__ void __launch_bounds__(32 * kXRegWarps, XRegCfg<R1, R2, EO>::MINB)
k_x_fwd_reg(OpView<float> op, const float2* in, float2* buf, const int* active,
            XinArgs<float> xa) {
  using K = XRegCfg<R1, R2, EO>;
  using C = float2;
  constexpr int NJ = K::NJ, NQ = K::NQ, EL = K::EL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int r = blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float2* sm = reinterpret_cast<float2*>(smem_raw) + wid * (EL * K::LW * K::LS);
  const int nx = op.nx, Lx = K::L;
  const int rows = 3 * op.nz * op.ny;
  chain_next();
  chain_wait();
  active = chained(active);
  in = chained(in);
  buf = chained(buf);
  xa = chained(xa);
  if (active && !active[r]) return;
  C s1 = make_float2(0.f, 0.f), s2 = s1, s3 = s1;
  if constexpr (MODE == XIN_P) {
    C sc[2];
    block_scalars<C, 2>({xa.ks[r].beta, xa.ks[r].omega}, sc);
    s1 = sc[0]; s2 = sc[1];
  } else if constexpr (MODE == XIN_S) {
    C sc[1];
    block_scalars<C, 1>({xa.ks[r].alpha}, sc);
    s1 = sc[0];
  } else if constexpr (MODE == XIN_Q) {
    C sc[3];
    block_scalars<C, 3>({xa.ks[r].beta, xa.ks[r].qa1, xa.ks[r].qa2}, sc);
    s1 = sc[0]; s2 = sc[1]; s3 = sc[2];
  }
  const int64_t off = (int64_t)r * rows * nx;
  const int64_t plane_sz = (int64_t)op.Ly * Lx;
  C* dst = buf + (int64_t)r * 3 * op.nz * plane_sz;
  const float4* __restrict__ tw = op.twx_reg;
  for (int row0 = (blockIdx.x * kXRegWarps + wid) * K::LW; row0 < rows;
       row0 += gridDim.x * kXRegWarps * K::LW) {
    for (int u = lane; u < K::U1; u += 32) {
      const int line = u / R2, j2 = u % R2;
      const int row = row0 + line;
      if (row >= rows) break;
      const bool last = j2 + R2 * (NJ - 1) < nx;   // j < nx holds for the other j1
      const int64_t g0 = off + (int64_t)row * nx + j2;
      C x[NJ];
      if constexpr (MODE == XIN_PLAIN) {
#pragma unroll
        for (int j = 0; j < NJ; ++j) x[j] = in[g0 + (j < NJ - 1 || last ? R2 * j : 0)];
      } else {
        C vb[NJ], vc[NJ], vd[NJ];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const int64_t g = g0 + (j < NJ - 1 || last ? R2 * j : 0);
          x[j] = xa.r[g];
          if (MODE != XIN_S) vb[j] = xa.pv[g];
          vc[j] = MODE == XIN_Q ? xa.d[g] : xa.v[g];
          if (MODE == XIN_Q) vd[j] = xa.x[g];
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const int64_t g = g0 + R2 * j;
          const bool st = j < NJ - 1 || last;
          if (MODE == XIN_P) {
            x[j] = cadd(x[j], cmul(s1, csub(vb[j], cmul(s2, vc[j]))));
          } else if (MODE == XIN_Q) {
            const C q = vb[j];
            const C dn = cadd(cmul(s2, vc[j]), cmul(s3, q));
            if (st) {
              xa.d[g] = dn;
              xa.x[g] = cadd(vd[j], dn);
            }
            x[j] = cadd(x[j], cmul(s1, q));
          } else {
            x[j] = csub(x[j], cmul(s1, vc[j]));
          }
          if (st) xa.pv[g] = x[j];
        }
      }
      if (!last) x[NJ - 1] = make_float2(0.f, 0.f);
      reg_step1<R1, R2, EO>(x, tw + j2, sm + EL * (line * K::LS + j2), EL * K::ROW);
    }
    __syncwarp();
    for (int u = lane; u < K::U2; u += 32) {
      const int line = u / NQ, q = u % NQ;  // q = 2 k1 + parity, or k1
      const int row = row0 + line;
      if (row >= rows) break;
      const int at = reg_place<R1, EO>(q);
      const float2* s = sm + EL * (line * K::LS + (EO ? at >> 1 : at) * K::ROW) + (EO ? at & 1 : 0);
      cv<float> a[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) {
        const float2 e = s[EL * j];
        a[j] = {e.x, e.y};
      }
      rdft<R2, false>(a);
      const int plane = fast_div(row, op.div_ny), y = row - plane * op.ny;
      C* drow = dst + plane * plane_sz + (int64_t)y * Lx + q;
#pragma unroll
      for (int k = 0; k < R2; ++k) drow[NQ * k] = make_float2(a[k].re, a[k].im);
    }
    __syncwarp();
  }
}

// a x - s with two roundings a part: the diagonal term is the largest of a product, and
// rounding it before s is taken off it was the largest single error left in one
__device__ __forceinline__ float2 diag_minus(float2 a, float2 x, float2 s) {
  return make_float2(fmaf(a.x, x.x, fmaf(-a.y, x.y, -s.x)), fmaf(a.x, x.y, fmaf(a.y, x.x, -s.y)));
}

template <int R1, int R2, bool EO, int MODE>
__global__ void __launch_bounds__(32 * kXRegWarps, XRegCfg<R1, R2, EO>::MINB)
k_x_inv_reg(OpView<float> op, const float2* buf, const float2* xin, float2* yout,
            const int* active, const float2* rhat, double* partials, FoldArgs fold) {
  using K = XRegCfg<R1, R2, EO>;
  using C = float2;
  constexpr int NJ = K::NJ, NQ = K::NQ, EL = K::EL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kAiSmem = 24;
  __shared__ C sai[kAiSmem];
  const int r = blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float2* sm = reinterpret_cast<float2*>(smem_raw) + wid * (EL * K::LW * K::LS);
  const int nx = op.nx, Lx = K::L;
  const int rows = 3 * op.nz * op.ny;
  chain_next();
  const bool ai_smem = op.ncomp1 * 3 <= kAiSmem;
  const C* ai = op.ainv + (int64_t)r * op.ncomp1 * 3;
  if (ai_smem) {
    for (int i = threadIdx.x; i < op.ncomp1 * 3; i += blockDim.x) sai[i] = ai[i];
    __syncthreads();
    ai = sai;
  }
  chain_wait();
  active = chained(active);
  buf = chained(buf);
  xin = chained(xin);
  yout = chained(yout);
  rhat = chained(rhat);
  partials = chained(partials);
  fold = chained(fold);
  if (active && !active[r]) return;
  const int64_t off = (int64_t)r * rows * nx;
  const int64_t plane_sz = (int64_t)op.Ly * Lx;
  const C* src = buf + (int64_t)r * 3 * op.nz * plane_sz;
  const float4* __restrict__ tw = op.twx_reg;
  LongAcc<4> acc;
  for (int row0 = (blockIdx.x * kXRegWarps + wid) * K::LW; row0 < rows;
       row0 += gridDim.x * kXRegWarps * K::LW) {
    for (int u = lane; u < K::U2; u += 32) {
      const int line = u / NQ, q = u % NQ;
      const int row = row0 + line;
      if (row >= rows) break;
      const int plane = fast_div(row, op.div_ny), y = row - plane * op.ny;
      const C* srow = src + plane * plane_sz + (int64_t)y * Lx + q;
      cv<float> a[R2];
#pragma unroll
      for (int k = 0; k < R2; ++k) {
        const float2 e = __ldcg(srow + NQ * k);
        a[k] = {e.x, e.y};
      }
      rdft<R2, true>(a);
      const int at = reg_place<R1, EO>(q);
      float2* s = sm + EL * (line * K::LS + (EO ? at >> 1 : at) * K::ROW) + (EO ? at & 1 : 0);
#pragma unroll
      for (int j = 0; j < R2; ++j) s[EL * j] = make_float2(a[j].re, a[j].im);
    }
    __syncwarp();
    for (int u = lane; u < K::U1; u += 32) {
      const int line = u / R2, j2 = u % R2;
      const int row = row0 + line;
      if (row >= rows) break;
      const bool last = j2 + R2 * (NJ - 1) < nx;
      // row = (c nz + z) ny + y  ->  sites (z ny + y) nx + j
      const int c = fast_div(fast_div(row, op.div_ny), op.div_nz);
      const uint8_t* cmp = op.comp + (int64_t)(row - c * op.nz * op.ny) * nx + j2;
      const int64_t g0 = off + (int64_t)row * nx + j2;
      C xv[NJ], hv[NJ];
      int cm[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int o = j < NJ - 1 || last ? R2 * j : 0;
        xv[j] = xin[g0 + o];
        if (MODE == XOUT_RV) hv[j] = rhat[g0 + o];
        cm[j] = __ldg(cmp + o);
      }
      C s[NJ];
      reg_step1_inv<R1, R2, EO>(sm + EL * (line * K::LS + j2), EL * K::ROW, tw + j2, s);
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        if (j == NJ - 1 && !last) break;
        C out = make_float2(0.f, 0.f);
        if (cm[j]) out = diag_minus(ai[3 * cm[j] + c], xv[j], s[j]);
        yout[g0 + R2 * j] = out;
        if constexpr (MODE == XOUT_RV) {
          acc.add(0, hv[j].x * out.x + hv[j].y * out.y);
          acc.add(1, hv[j].x * out.y - hv[j].y * out.x);
        } else if constexpr (MODE == XOUT_TS) {
          acc.add(0, out.x * xv[j].x + out.y * xv[j].y);
          acc.add(1, out.x * xv[j].y - out.y * xv[j].x);
          acc.add(2, out.x * out.x + out.y * out.y);
        } else if constexpr (MODE == XOUT_QT) {
          acc.add(0, xv[j].x * out.x - xv[j].y * out.y);
          acc.add(1, xv[j].x * out.y + xv[j].y * out.x);
        }
        if (j == 7 && NJ > 8) acc.flush();
      }
      acc.flush();
    }
    __syncwarp();
  }
  if constexpr (MODE == XOUT_RV || MODE == XOUT_QT) {
    acc.template write<2>(partials);
    if (fold.counter) fold_scalar_step<2>(partials, fold);
  } else if constexpr (MODE == XOUT_TS) {
    acc.template write<4>(partials);
    if (fold.counter) fold_scalar_step<4>(partials, fold);
  }
}

template <int R1, int R2, bool EO, int MODE>
void launch_x_fwd_reg(const OpView<float>& op, int R, const float2* x, float2* buf,
                      const int* active, XinArgs<float> xa, cudaStream_t st) {
  using K = XRegCfg<R1, R2, EO>;
  const dim3 g(x_reg_grid(3 * op.nz * op.ny, K::LW), R);
  launch_chained(op.chain == 2, k_x_fwd_reg<R1, R2, EO, MODE>, g, 32 * kXRegWarps, K::smem, st, op, x,
                 buf, active, xa);
}
template <int R1, int R2, bool EO, int MODE>
void launch_x_inv_reg(const OpView<float>& op, int R, const float2* buf, const float2* x, float2* y,
                      const int* active, const float2* rhat, double* partials, cudaStream_t st,
                      FoldArgs fold) {
  using K = XRegCfg<R1, R2, EO>;
  const dim3 g(x_reg_grid(3 * op.nz * op.ny, K::LW), R);
  launch_chained(op.chain, k_x_inv_reg<R1, R2, EO, MODE>, g, 32 * kXRegWarps, K::smem, st, op, buf, x,
                 y, active, rhat, partials, fold);
}
template <int R1, int R2, bool EO> cudaError_t configure_x_reg() {
  const void* k[] = {(const void*)k_x_fwd_reg<R1, R2, EO, XIN_PLAIN>, (const void*)k_x_fwd_reg<R1, R2, EO, XIN_P>,
                     (const void*)k_x_fwd_reg<R1, R2, EO, XIN_S>, (const void*)k_x_fwd_reg<R1, R2, EO, XIN_Q>,
                     (const void*)k_x_inv_reg<R1, R2, EO, XOUT_PLAIN>, (const void*)k_x_inv_reg<R1, R2, EO, XOUT_RV>,
                     (const void*)k_x_inv_reg<R1, R2, EO, XOUT_TS>, (const void*)k_x_inv_reg<R1, R2, EO, XOUT_QT>};
  for (const void* f : k) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)XRegCfg<R1, R2, EO>::smem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The plans, in parts that compile side by side (xpass_reg_*.cu): X(R1, R2), R1
// about half of R2 so that steps 1 and 2 want about as many threads.
#define DDA_XREG_PART0(X) X(3, 3) X(2, 5) X(3, 4) X(3, 5) X(4, 4) X(3, 6) X(4, 5) X(4, 6) X(5, 5)
#define DDA_XREG_PART1(X) X(3, 9) X(5, 6) X(4, 8) X(4, 9) X(5, 8) X(5, 9) X(6, 8)
#define DDA_XREG_PART2(X) X(5, 10) X(6, 9) X(6, 10) X(8, 8) X(8, 9) X(5, 15)
#define DDA_XREG_PART3(X) X(8, 10) X(9, 9) X(9, 10) X(8, 12) X(10, 10)
#define DDA_XREG_PART4(X) X(9, 12) X(8, 15) X(8, 16) X(9, 15)
#define DDA_XREG_PART5(X) X(9, 16) X(10, 15) X(10, 16) X(9, 18)
#define DDA_XREG_PART6(X) X(12, 15) X(12, 16) X(10, 20) X(12, 18)
#define DDA_XREG_PART7(X) X(15, 15) X(15, 16) X(16, 16)
#define DDA_XREG_ALL(X)                                                                     \
  DDA_XREG_PART0(X) DDA_XREG_PART1(X) DDA_XREG_PART2(X) DDA_XREG_PART3(X) DDA_XREG_PART4(X) \
  DDA_XREG_PART5(X) DDA_XREG_PART6(X) DDA_XREG_PART7(X)

struct XInvArgs {
  const float2* buf;
  const float2* x;
  float2* y;
  const float2* rhat;
  double* partials;
  FoldArgs fold;
};
#define DDA_XREG_DECLARE(PART)                                                               \
  bool launch_x_fwd_reg_part##PART(int mode, const OpView<float>& op, int R, const float2* x, \
                                   float2* buf, const int* active, XinArgs<float> xa,        \
                                   cudaStream_t st);                                         \
  bool launch_x_inv_reg_part##PART(int mode, const OpView<float>& op, int R,                  \
                                   const XInvArgs& a, const int* active, cudaStream_t st);   \
  cudaError_t configure_x_reg_part##PART(int L);
DDA_XREG_DECLARE(0) DDA_XREG_DECLARE(1) DDA_XREG_DECLARE(2) DDA_XREG_DECLARE(3)
DDA_XREG_DECLARE(4) DDA_XREG_DECLARE(5) DDA_XREG_DECLARE(6) DDA_XREG_DECLARE(7)
DDA_XREG_DECLARE(8)

template <int A, int B, bool EO>
void x_fwd_reg_mode(int mode, const OpView<float>& op, int R, const float2* x, float2* buf,
                    const int* active, XinArgs<float> xa, cudaStream_t st) {
  if (mode == XIN_PLAIN) launch_x_fwd_reg<A, B, EO, XIN_PLAIN>(op, R, x, buf, active, xa, st);
  else if (mode == XIN_P) launch_x_fwd_reg<A, B, EO, XIN_P>(op, R, x, buf, active, xa, st);
  else if (mode == XIN_S) launch_x_fwd_reg<A, B, EO, XIN_S>(op, R, x, buf, active, xa, st);
  else launch_x_fwd_reg<A, B, EO, XIN_Q>(op, R, x, buf, active, xa, st);
}
template <int A, int B, bool EO>
void x_inv_reg_mode(int mode, const OpView<float>& op, int R, const XInvArgs& a, const int* active,
                    cudaStream_t st) {
  if (mode == XOUT_PLAIN)
    launch_x_inv_reg<A, B, EO, XOUT_PLAIN>(op, R, a.buf, a.x, a.y, active, a.rhat, a.partials, st, a.fold);
  else if (mode == XOUT_RV)
    launch_x_inv_reg<A, B, EO, XOUT_RV>(op, R, a.buf, a.x, a.y, active, a.rhat, a.partials, st, a.fold);
  else if (mode == XOUT_TS)
    launch_x_inv_reg<A, B, EO, XOUT_TS>(op, R, a.buf, a.x, a.y, active, a.rhat, a.partials, st, a.fold);
  else
    launch_x_inv_reg<A, B, EO, XOUT_QT>(op, R, a.buf, a.x, a.y, active, a.rhat, a.partials, st, a.fold);
}
#define DDA_XREG_FWD(A, B) \
  case 2 * (A) * (B): x_fwd_reg_mode<A, B, true>(mode, op, R, x, buf, active, xa, st); return true;
#define DDA_XREG_INV(A, B) \
  case 2 * (A) * (B): x_inv_reg_mode<A, B, true>(mode, op, R, a, active, st); return true;
#define DDA_XREG_CONFIG(A, B) case 2 * (A) * (B): return configure_x_reg<A, B, true>();
#define DDA_XREG_FWD_ODD(A, B) \
  case (A) * (B): x_fwd_reg_mode<A, B, false>(mode, op, R, x, buf, active, xa, st); return true;
#define DDA_XREG_INV_ODD(A, B) \
  case (A) * (B): x_inv_reg_mode<A, B, false>(mode, op, R, a, active, st); return true;
#define DDA_XREG_CONFIG_ODD(A, B) case (A) * (B): return configure_x_reg<A, B, false>();
// LIST: the lengths' plans, ODD: empty or _ODD
#define DDA_XREG_DEFINE(PART, LIST, ODD)                                                     \
  bool launch_x_fwd_reg_part##PART(int mode, const OpView<float>& op, int R, const float2* x, \
                                   float2* buf, const int* active, XinArgs<float> xa,        \
                                   cudaStream_t st) {                                        \
    switch (op.Lx) { LIST(DDA_XREG_FWD##ODD) }                                               \
    return false;                                                                            \
  }                                                                                          \
  bool launch_x_inv_reg_part##PART(int mode, const OpView<float>& op, int R,                  \
                                   const XInvArgs& a, const int* active, cudaStream_t st) {  \
    switch (op.Lx) { LIST(DDA_XREG_INV##ODD) }                                               \
    return false;                                                                            \
  }                                                                                          \
  cudaError_t configure_x_reg_part##PART(int L) {                                            \
    switch (L) { LIST(DDA_XREG_CONFIG##ODD) }                                                \
    return cudaSuccess;                                                                      \
  }

}  // namespace dda
