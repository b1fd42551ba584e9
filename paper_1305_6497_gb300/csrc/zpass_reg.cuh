// z pass in two register transforms (FP32): forward FFT along z, the 3x3
// complex-symmetric multiply by Ghat, inverse FFT along z, for z lengths
// L = 2n with n = R1 R2, R1 up to 20 and R2 up to 16.
//
// A line holds nz <= n values, zero-padded to L = 2n.  Its spectrum at the even
// frequencies 2k is the n-point DFT of x_j and at the odd ones 2k + 1 that of
// x_j w_L^j, so the padded transform is two n-point transforms of the same input
// that need the same butterflies: they run as the two halves of packed FP32
// pairs (fft_reg.cuh), and no zero is ever transformed.  An n-point transform
// is R1-point DFTs, twiddles, R2-point DFTs, each in the registers of one
// thread, with one exchange through shared memory between them:
//   1. thread (column t, j2, component): x at z = j2 + R2 j1, both halves'
//      R1-point DFTs over j1 (eo_step), twiddles w_L^(j2 (2 k1 + parity)), to shared
//      memory;
//   2. thread (t, k1, parity): the R2-point DFTs over j2 of all three components,
//      which gives them at the frequencies 2 (k1 + R1 k2) + parity (the odd ones' k1
//      counted as reg_freq does); the multiply, and the inverse R2-point DFTs, back in
//      place;
//   3. thread (t, j2, component): conjugate twiddles, inverse R1-point DFTs, the halves
//      joined (eo_step_inv), stored for z < nz.
// Every value crosses shared memory twice (once each way) and a pass meets two
// barriers; the kernels that keep lines in shared memory and transform them stage
// by stage cross it 2 x 3 times for L = 512 and meet ten.
//
// A CTA holds the twiddles and one Ghat tile (its columns of octant row hy) in
// shared memory and runs up to `per` passes on it: both rows ky = hy, Ly - hy of
// every right-hand side.  Ghat columns are contiguous (ghat_f32_offset).
//
// Layout: shared memory [component][k1][j2][t] of 16-byte (even, odd) pairs, the
// columns of the tile fastest.  A quarter-warp's 16-byte accesses (steps 1, 3) and
// a half-warp's 8-byte ones (step 2: columns x parities) cover whole 128-byte rows
// without a conflict, and so do the reads of the Ghat tile (see ROW and GS).
//
// What bounds it: instruction issue and the shared-memory pipe (of the 64x64x256
// brick: 48% and 53% busy, 29% of the measured copy rate, 154 thread instructions per
// stored point against 214 of the column-pair kernel).  8 columns per CTA (64-byte
// rows in global memory) up to n = 96 and 4 above leave room for two to four CTAs.
// Per launch with two right-hand sides, before (the default one-tile or, where
// named, the tuned kernel) and now: 256^3 box 8600 (tuned pair kernel 4460) ->
// 3473 us; 128^3 866 -> 326 us; 64x64x256 582 (tuned 284) -> 206 us; 100x75x135
// 589 -> 179 us; 48x96x144 319 -> 129 us; 64^3 76 (tuned 54) -> 51 us.
#pragma once

#include "reg_step.cuh"

namespace dda {

// EO: L = 2 R1 R2, even and odd frequencies as halves; otherwise L = R1 R2 is odd, the
// line is transformed whole in scalar arithmetic (elements of 8 bytes, rows j1 >= NJ
// zero, no parities in step 2).
template <int R1, int R2, bool EO> struct ZRegCfg {
  static constexpr int n = R1 * R2, L = EO ? 2 * n : n, Hz = L / 2 + 1;
  static constexpr int NJ = EO ? R1 : ((L + 1) / 2 + R2 - 1) / R2;
  static constexpr int EL = EO ? 2 : 1;              // float2 per element
  static constexpr int TILE = !EO || n <= 96 ? 8 : 4;  // columns per CTA
  static constexpr int U1 = 3 * TILE * R2;           // threads at work in steps 1 and 3
  static constexpr int U2 = (EO ? 2 : 1) * TILE * R1;  // in step 2
  static constexpr int NT = ((U1 > U2 ? U1 : U2) + 31) / 32 * 32;
  // elements per (component, k1): with 4 columns a half-warp covers two k1, which
  // half a bank row more keeps apart (odd L: 8 columns and odd R2 do that already)
  static constexpr int ROW = R2 * TILE + (EO && TILE == 4 && R2 % 2 == 0 ? 4 : 0);
  // float4 per column of the Ghat tile: 8 columns want an odd stride, 4 columns
  // (x 2 parities) one of 2 mod 4
  static constexpr int GS = TILE == 8 ? (3 * Hz) | 1 : (3 * Hz + 1) / 4 * 4 + 2;
  static constexpr int ex4 = (3 * R1 * ROW * EL + 1) / 2;  // exchange, in float4
  static constexpr size_t smem = (size_t)(ex4 + TILE * GS + n) * 16;
  static constexpr int regs1 = 4 * R1 + 44, regs2 = 6 * R2 + 44;
  static constexpr int regs = ((regs1 > regs2 ? regs1 : regs2) + 7) / 8 * 8;
  static constexpr int by_regs = 65536 / (NT * regs), by_smem = (int)(227 * 1024 / (smem + 1024));
  static constexpr int fit = by_regs < by_smem ? by_regs : by_smem;
  static constexpr int MINB = fit < 1 ? 1 : fit > 2048 / NT ? 2048 / NT : fit;
};

__device__ __forceinline__ float flip_if(float a, unsigned m) {
  return __uint_as_float(__float_as_uint(a) ^ m);
}

template <int R1, int R2, bool EO, bool ASYNC>
__global__ void __launch_bounds__(ZRegCfg<R1, R2, EO>::NT, ZRegCfg<R1, R2, EO>::MINB)
k_fft_z_reg(OpView<float> op, float2* buf, int R, int per, const int* active) {
  using K = ZRegCfg<R1, R2, EO>;
  constexpr int n = K::n, L = K::L, TILE = K::TILE, NT = K::NT, ROW = K::ROW, Hz = K::Hz;
  constexpr int NJ = K::NJ, EL = K::EL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  float4* gsm = reinterpret_cast<float4*>(smem_raw) + K::ex4;
  float4* tws = gsm + TILE * K::GS;
  const int hy = blockIdx.y;
  const int Lx = op.Lx, Ly = op.Ly, nz = op.nz;
  // the passes of this CTA: v = 2 r + (0: row hy, 1: row Ly - hy)
  const bool self = hy == 0 || 2 * hy == Ly;  // the row is its own mirror image
  const int vend = min(2 * R, ((int)blockIdx.z + 1) * per);
  auto next = [&](int v) {
    while (v < vend && ((self && (v & 1)) || (active && !active[v >> 1]))) ++v;
    return v;
  };
  // a right-hand side frozen before the predecessor has ended stays so
  chain_next();
  if (active) {
    int v = blockIdx.z * per;
    while (v < vend && !static_cast<const volatile int*>(active)[v >> 1]) ++v;
    if (v >= vend) {
      chain_wait();
      return;
    }
  }
  const int col0 = blockIdx.x * TILE;
  const int ncol = min(TILE, Lx - col0);
  const int64_t plane = (int64_t)Ly * Lx, comp = nz * plane;
  // the thread's place in steps 1 and 3
  const int t1 = threadIdx.x % TILE, j2 = (threadIdx.x / TILE) % R2;
  const int c1 = threadIdx.x / (TILE * R2);
  const bool on1 = c1 < 3 && t1 < ncol;
  const bool last = j2 + R2 * (NJ - 1) < nz;  // z < nz holds for the other j1
  // the Ghat tile: columns of 3 x Hz 16-byte pieces, contiguous
  int hx[TILE];
#pragma unroll
  for (int t = 0; t < TILE; ++t) {
    const int kx = op.kx_at[col0 + min(t, ncol - 1)];
    hx[t] = kx > (Lx >> 1) ? Lx - kx : kx;
  }
#pragma unroll
  for (int t = 0; t < TILE; ++t) {
    const float4* src =
        reinterpret_cast<const float4*>(op.ghat) + ((int64_t)hy * op.Hx + hx[t]) * 3 * Hz;
    for (int q = threadIdx.x; q < 3 * Hz; q += NT) cp_async<16>(gsm + t * K::GS + q, src + q);
  }
  for (int e = threadIdx.x; e < n; e += NT) cp_async<16>(tws + e, op.twz_reg + e);
  cp_async_commit();
  chain_wait();
  active = chained(active);
  buf = chained(buf);
  int v = next(blockIdx.z * per);
  if (v >= vend) {
    cp_async_wait_all();
    return;
  }
  float2* const first = buf + col0 + min(t1, ncol - 1) + min(c1, 2) * comp + j2 * plane;
  const int64_t row0 = (int64_t)op.ypos_at[hy] * Lx;
  const int64_t row1 = (int64_t)op.ypos_at[self ? hy : Ly - hy] * Lx;
  auto line = [&](int w) { return first + (w >> 1) * 3 * comp + ((w & 1) ? row1 : row0); };
  float2* own = sm + EL * (c1 * (R1 * ROW) + j2 * TILE + t1);
  // The next pass's input is asked for as soon as step 3 has read the thread's
  // words of shared memory (odd L: both threads' of a pair), and lands in them (ASYNC: 16-byte asynchronous copies
  // past L1, each holding the two columns of a pair of threads for one row; the
  // threads of a pair take the even and the odd rows).  Plain loads need a line of
  // L1 for each of their 32-byte rows until they arrive, and the shared memory
  // leaves L1 room for a fifth of a pass's; they remain for odd Lx, where pairs of
  // columns are not 16-byte aligned.  Every load is unconditional as far as it can
  // be: only the last row (j1 = NJ - 1) may lie beyond nz.  (EO: row j1 lands in word
  // j1 / 2 of the pair's thread of j1's parity; odd L, words of 8 bytes: in word j1 of
  // both.)
  float2 x[NJ];
  auto fetch = [&](int w) {
    if constexpr (ASYNC) {
      if (!on1) return;
      const float2* src = line(w) - (t1 & 1);
#pragma unroll
      for (int i = 0; i < (NJ + 1) / 2; ++i) {
        const int j = 2 * i + (t1 & 1);
        float2* dst = EO ? own + EL * i * ROW : own - (t1 & 1) + j * ROW;
        if (j < NJ - 1 || (j == NJ - 1 && last)) cp_async<16>(dst, src + (int64_t)j * R2 * plane);
      }
      cp_async_commit();
    } else {
      const float2* src = line(w);
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        x[j] = __ldcg(src + (j < NJ - 1 || last ? (int64_t)j * R2 * plane : 0));
    }
  };
  fetch(v);
  // and in step 2
  const int t2 = threadIdx.x % TILE, p2 = EO ? (threadIdx.x / TILE) & 1 : 0;
  const int k2 = threadIdx.x / ((EO ? 2 : 1) * TILE);
  const unsigned mx = op.kx_at[col0 + min(t2, ncol - 1)] > (Lx >> 1) ? 0x80000000u : 0u;
  const float4* tw = tws + j2;

  cp_async_wait_all();
  __syncthreads();
  while (true) {
    const int vn = next(v + 1);
    // ---- 1. both halves' R1-point DFTs
    if constexpr (ASYNC) {
      // every thread of the CTA passes these warp barriers: the two threads of a
      // pair read what either of them copied, and then overwrite it
      cp_async_wait_all();
      __syncwarp();
      if (c1 < 3) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          x[j] = EO ? own[EL * ((j & 1) - (t1 & 1) + (j >> 1) * ROW) + (t1 & 1)] : own[j * ROW];
      }
      __syncwarp();
    }
    if (c1 < 3) {
      if (!last) x[NJ - 1] = make_float2(0.f, 0.f);
      reg_step1<R1, R2, EO>(x, tw, own, EL * ROW);
    }
    __syncthreads();
    if (!ASYNC && vn < vend) fetch(vn);  // lands while step 2 computes

    // ---- 2. R2-point DFTs of the three components, multiply, inverse DFTs
    if (k2 < R1) {
      float2* q = sm + EL * (k2 * ROW + t2) + p2;
      const float4* g = gsm + t2 * K::GS;
      const unsigned my = (v & 1) ? 0x80000000u : 0u;
      cv<float> s[3][R2];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int j = 0; j < R2; ++j) {
          const float2 e = q[EL * (c * (R1 * ROW) + j * TILE)];
          s[c][j] = {e.x, e.y};
        }
        rdft<R2, false>(s[c]);
      }
      // position j holds kz = kf + 2 R1 j (odd L: + R1 j): row kz of the octant up to
      // L / 2, row L - kz (z reflected) above; for even R2 every j is on one side (kz = n
      // sits on both)
      constexpr int KS = EO ? 2 : 1;
      const int kf = reg_freq<R1, EO>(EO ? 2 * k2 + p2 : k2);
      const float4* glo = g + kf;
      const float4* ghi = g + L - kf;
      static_for<R2>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        constexpr bool mid = R2 % 2 == 1 && 2 * j + 1 == R2;
        const bool fz = mid ? kf + KS * R1 * j > L / 2 : 2 * j >= R2;
        const float4* gp = fz ? ghi - KS * R1 * j : glo + KS * R1 * j;
        const float4 g0 = gp[0], g1 = gp[Hz], g2 = gp[2 * Hz];
        // odd components change sign under the reflection of an odd axis
        const cv<float> xx{g0.x, g0.y}, yy{g1.z, g1.w}, zz{g2.z, g2.w};
        const cv<float> xy{flip_if(g0.z, mx ^ my), flip_if(g0.w, mx ^ my)};
        const cv<float> xz{flip_if(g1.x, mx), flip_if(g1.y, mx)};
        const cv<float> yz{flip_if(g2.x, my), flip_if(g2.y, my)};
        const cv<float> a = s[0][j], b = s[1][j];
        const cv<float> c = fz ? cv<float>{-s[2][j].re, -s[2][j].im} : s[2][j];
        s[0][j] = cvmad(xz, c, cvmad(xy, b, cvmul(xx, a)));
        s[1][j] = cvmad(yz, c, cvmad(yy, b, cvmul(xy, a)));
        const cv<float> o = cvmad(zz, c, cvmad(yz, b, cvmul(xz, a)));
        s[2][j] = fz ? cv<float>{-o.re, -o.im} : o;
      });
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        rdft<R2, true>(s[c]);
#pragma unroll
        for (int j = 0; j < R2; ++j)
          q[EL * (c * (R1 * ROW) + j * TILE)] = make_float2(s[c][j].re, s[c][j].im);
      }
    }
    __syncthreads();

    // ---- 3. inverse R1-point DFTs, the halves joined, to global memory.  A thread
    // reads here what it wrote in step 1 and nobody else does, so the next pass's
    // step 1 needs no barrier.  The next pass's copies land in these words: in the
    // thread's own for EO, but in both threads' of a pair for odd L, where neither
    // may ask for them before the other has read its words (a warp barrier that
    // every thread of the CTA passes: the last warp may hold threads with c1 = 3)
    reg_cv<EO> a[R1];
    constexpr bool pair = ASYNC && !EO;
    if constexpr (pair) {
      if (c1 < 3) reg_step1_inv_read<R1, R2, EO>(own, EL * ROW, tw, a);
      __syncwarp();
    }
    if (c1 < 3) {
      if constexpr (!pair) reg_step1_inv_read<R1, R2, EO>(own, EL * ROW, tw, a);
      if (ASYNC && vn < vend) fetch(vn);
      float2 y[NJ];
      reg_step1_inv_out<R1, EO>(a, y);
      float2* dst = line(v);
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (on1 && (j < NJ - 1 || last)) dst[(int64_t)j * R2 * plane] = y[j];
    }
    if (vn >= vend) return;
    v = vn;
  }
}

template <int R1, int R2, bool EO> cudaError_t configure_z_reg() {
  cudaError_t e = cudaFuncSetAttribute(k_fft_z_reg<R1, R2, EO, false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ZRegCfg<R1, R2, EO>::smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fft_z_reg<R1, R2, EO, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)ZRegCfg<R1, R2, EO>::smem);
  return e;
}
template <int R1, int R2, bool EO>
void launch_z_reg(const OpView<float>& op, int R, float2* buf, const int* active, cudaStream_t st) {
  using K = ZRegCfg<R1, R2, EO>;
  const int tiles = (op.Lx + K::TILE - 1) / K::TILE, hy = op.Ly / 2 + 1;
  // passes per CTA: as many as leave four waves of CTAs (more passes save Ghat
  // reads, fewer waves lose to the last one: two right-hand sides, four waves, eight,
  // one pass per CTA: 100x75x135 179, 187, 213 us, 128^3 326, 326, 407, 64x64x256 206,
  // 217, 251)
  int64_t per = (int64_t)tiles * hy * 2 * R / (152 * K::MINB * 4);
  per = per < 1 ? 1 : per > 2 * R ? 2 * R : per;
  const dim3 g(tiles, hy, (unsigned)((2 * R + per - 1) / per));
  if (op.Lx % 2 == 0 && ((uintptr_t)buf & 15) == 0)
    launch_chained(op.chain, k_fft_z_reg<R1, R2, EO, true>, g, K::NT, K::smem, st, op, buf, R, (int)per,
                   active);
  else
    launch_chained(op.chain, k_fft_z_reg<R1, R2, EO, false>, g, K::NT, K::smem, st, op, buf, R,
                   (int)per, active);
}

// The plans, in parts that compile side by side (zpass_reg_*.cu): X(R1, R2).
#define DDA_ZREG_PART0(X) X(3, 3) X(5, 2) X(4, 3) X(5, 3) X(4, 4) X(6, 3) X(5, 4) X(6, 4) X(5, 5) X(9, 3) X(6, 5) X(8, 4)
#define DDA_ZREG_PART1(X) X(6, 6) X(8, 5) X(9, 5) X(8, 6) X(10, 5) X(9, 6) X(10, 6) X(8, 8)
#define DDA_ZREG_PART2(X) X(9, 8) X(15, 5) X(10, 8) X(9, 9) X(10, 9) X(12, 8)
#define DDA_ZREG_PART3(X) X(10, 10) X(12, 9) X(12, 10) X(16, 8) X(15, 9)
#define DDA_ZREG_PART4(X) X(12, 12) X(15, 10) X(16, 10) X(18, 9) X(15, 12)
#define DDA_ZREG_PART5(X) X(16, 12) X(20, 10) X(18, 12) X(15, 15) X(16, 15) X(16, 16)

#define DDA_ZREG_ALL(X)                                                                     \
  DDA_ZREG_PART0(X) DDA_ZREG_PART1(X) DDA_ZREG_PART2(X) DDA_ZREG_PART3(X) DDA_ZREG_PART4(X) \
  DDA_ZREG_PART5(X)
#define DDA_ZREG_DECLARE(PART)                                                                 \
  bool launch_z_reg_part##PART(const OpView<float>& op, int R, float2* buf, const int* active, \
                               cudaStream_t st);                                               \
  cudaError_t configure_z_reg_part##PART(int L);
DDA_ZREG_DECLARE(0) DDA_ZREG_DECLARE(1) DDA_ZREG_DECLARE(2)
DDA_ZREG_DECLARE(3) DDA_ZREG_DECLARE(4) DDA_ZREG_DECLARE(5)

#define DDA_ZREG_LAUNCH(A, B) \
  case 2 * (A) * (B): launch_z_reg<A, B, true>(op, R, buf, active, st); return true;
#define DDA_ZREG_CONFIG(A, B) case 2 * (A) * (B): return configure_z_reg<A, B, true>();
#define DDA_ZREG_LAUNCH_ODD(A, B) \
  case (A) * (B): launch_z_reg<A, B, false>(op, R, buf, active, st); return true;
#define DDA_ZREG_CONFIG_ODD(A, B) case (A) * (B): return configure_z_reg<A, B, false>();
// ODDS: the list of odd plans (DDA_XREG_ODD), or nothing
#define DDA_ZREG_DEFINE(PART, ODDS)                                                            \
  bool launch_z_reg_part##PART(const OpView<float>& op, int R, float2* buf, const int* active, \
                               cudaStream_t st) {                                              \
    switch (op.Lz) { DDA_ZREG_PART##PART(DDA_ZREG_LAUNCH) ODDS(DDA_ZREG_LAUNCH_ODD) }          \
    return false;                                                                              \
  }                                                                                            \
  cudaError_t configure_z_reg_part##PART(int L) {                                              \
    switch (L) { DDA_ZREG_PART##PART(DDA_ZREG_CONFIG) ODDS(DDA_ZREG_CONFIG_ODD) }              \
    return cudaSuccess;                                                                        \
  }

}  // namespace dda
