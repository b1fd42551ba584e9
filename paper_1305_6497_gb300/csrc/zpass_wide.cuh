// z pass in two register transforms for 16-byte complex values (FP64 and
// double-float): the
// transform of zpass_reg.cuh, even and odd frequencies as transforms of their own
// (nothing is packed), each DFT of R1 or R2 points in the registers of one thread
// and every step in place in shared memory:
//   1. thread (column t, j2, parity, component): x at z = j2 + R2 j1 (odd parity:
//      times w_L^(R2 j1)), R1-point DFT, twiddles w_L^(j2 (2 k1 + parity));
//   2. thread (t, k1, parity, component): R2-point DFT;
//   3. thread (t, frequency): the multiply by Ghat;
//   4., 5. the inverses of 2. and 1.; 6. even + odd half, stored for z < nz.
//
// What bounds it: FP32 arithmetic.  A double-float addition is 11 instructions and a
// product 7, and a stored value takes some 100 of them; the run-time plan kernel
// this replaces spent two thirds of its time on the rest (radix dispatch in every
// stage, zeros of the padded half, idle threads of stages with few butterflies).
// Single components per thread keep the registers at 64 of data for 16 points.
// Double-float z pass, two right-hand sides, before and now: 128^3 grid 1237 -> 348
// us, 64x128x128 645 -> 172, 96^3 236 -> 162, 200x150x270 2125 -> 1890, 512^3 35.9 ->
// 30.5 ms (its products are summed with one renormalisation, fft_reg.cuh); the error
// of a product against FP64 stays at 2.5 to 2.9e-15.  FP64 uses it for short lines
// (plan_matvec).
#pragma once

#include "fft_reg.cuh"
#include "matvec_impl.cuh"

namespace dda {

// The multiply w = G v (G symmetric: xx, xy, xz, yy, yz, zz; signs as spectral_mul) in
// double-float: every part is a sum of six products, split exactly and summed with
// the errors of the leading sums, renormalised once (75 instructions where products
// and sums one by one take 97).
__device__ __forceinline__ df64 df_dot6(const df64 (&a)[6], const df64 (&b)[6]) {
  float s = __fmul_rn(a[0].hi, b[0].hi);
  float e = __fmaf_rn(a[0].hi, b[0].hi, -s);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    e = __fmaf_rn(a[i].hi, b[i].lo, e);
    e = __fmaf_rn(a[i].lo, b[i].hi, e);
    if (i > 0) {
      const float p = __fmul_rn(a[i].hi, b[i].hi);
      e = __fadd_rn(e, __fmaf_rn(a[i].hi, b[i].hi, -p));
      const float t = __fadd_rn(s, p), bb = __fsub_rn(t, s);
      e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(p, bb)));
      s = t;
    }
  }
  return df_fast2sum(s, e);
}
__device__ __forceinline__ df64c df_row3(df64c g0, df64c g1, df64c g2, df64c a, df64c b, df64c c) {
  df64c r;
  const df64 gr[6] = {g0.x, -g0.y, g1.x, -g1.y, g2.x, -g2.y};
  const df64 vr[6] = {a.x, a.y, b.x, b.y, c.x, c.y};
  r.x = df_dot6(gr, vr);
  const df64 gi[6] = {g0.x, g0.y, g1.x, g1.y, g2.x, g2.y};
  const df64 vi[6] = {a.y, a.x, b.y, b.x, c.y, c.x};
  r.y = df_dot6(gi, vi);
  return r;
}
template <typename T, bool CROSS>
__device__ __forceinline__ void wide_mul(cplx_t<T> (&g)[6], bool fx, bool fy, bool fz,
                                         cplx_t<T>* w, int stride) {
  if constexpr (std::is_same<T, df64>::value) {
    if (fx != fy) { g[1].x = -g[1].x; g[1].y = -g[1].y; }
    if (fx != fz) { g[2].x = -g[2].x; g[2].y = -g[2].y; }
    if (fy != fz) { g[4].x = -g[4].x; g[4].y = -g[4].y; }
    const df64c a = w[0], b = w[stride], c = w[2 * stride];
    w[0] = df_row3(g[0], g[1], g[2], a, b, c);
    w[stride] = df_row3(g[1], g[3], g[4], a, b, c);
    w[2 * stride] = df_row3(g[2], g[4], g[5], a, b, c);
  } else {
    spectral_mul<T, CROSS>(g, fx, fy, fz, w, stride);
  }
}

template <int R1, int R2> struct ZWideCfg {
  static constexpr int n = R1 * R2, L = 2 * n, TILE = 4;
  static constexpr size_t smem = (size_t)6 * n * TILE * 16;
  static constexpr int most = R1 > R2 ? R1 : R2;
  static constexpr int regs = most > 12 ? 168 : most > 9 ? 128 : 104;
  static constexpr int fit(int nt) {
    const int by_regs = 65536 / (nt * regs), by_smem = (int)(227 * 1024 / (smem + 1024));
    const int f = by_regs < by_smem ? by_regs : by_smem;
    return f < 1 ? 1 : f > 2048 / nt ? 2048 / nt : f;
  }
  // threads: the most CTAs resident per time a CTA takes, counted in rounds of the
  // transform steps (a round of the points of its DFT) and of the multiply
  static constexpr int rounds(int u, int nt) { return (u + nt - 1) / nt; }
  static constexpr int score(int nt) {
    const int t = 2 * rounds(24 * R2, nt) * R1 * 3 + 2 * rounds(24 * R1, nt) * R2 * 2 +
                  rounds(2 * n * TILE, nt) * 8;
    return fit(nt) * 1000000 / t;
  }
  static constexpr int pick() {
    int b = 128;
    for (int nt = 96; nt <= 384; nt += 32)
      if (score(nt) > score(b)) b = nt;
    return b;
  }
  static constexpr int NT = pick(), MINB = fit(NT);
};

template <typename T, bool CROSS, int R1, int R2>
__global__ void __launch_bounds__(ZWideCfg<R1, R2>::NT, ZWideCfg<R1, R2>::MINB)
k_fft_z_wide(OpView<T> op, cplx_t<T>* __restrict__ buf, const int* __restrict__ active) {
  using K = ZWideCfg<R1, R2>;
  using C = cplx_t<T>;
  constexpr int n = K::n, L = K::L, TILE = K::TILE, NT = K::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  // both rows of an octant row and every right-hand side are neighbours in launch
  // order, so that they share the Ghat rows in L2
  const int r = blockIdx.x >> 1, hy = blockIdx.z;
  const bool fy = blockIdx.x & 1;
  if (active && !active[r]) return;
  const int Lx = op.Lx, Ly = op.Ly, nz = op.nz;
  if (fy && (hy == 0 || 2 * hy == Ly)) return;
  const int col0 = blockIdx.y * TILE;
  const int ncol = min(TILE, Lx - col0);
  const int64_t plane = (int64_t)Ly * Lx, comp = nz * plane;
  C* base = buf + r * 3 * comp + (int64_t)op.ypos_at[fy ? Ly - hy : hy] * Lx + col0;
  const C* __restrict__ tw = op.tw_wide;

  for (int u = threadIdx.x; u < 24 * R2; u += NT) {
    const int t = u % 4, j2 = (u / 4) % R2, p = (u / (4 * R2)) & 1, c = u / (8 * R2);
    const C* src = base + c * comp + j2 * plane + min(t, ncol - 1);
    const bool last = j2 + R2 * (R1 - 1) < nz;
    cv<T> a[R1];
    static_for<R1>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      const C v = src[j < R1 - 1 || last ? (int64_t)j * R2 * plane : 0];
      a[j] = {v.x, v.y};
      if (j == R1 - 1 && !last) a[j] = {vconst<T>(0.0), vconst<T>(0.0)};
      if (j > 0 && p) a[j] = cvrot<false>(a[j], cx_cos(j, 2 * R1), cx_sin(j, 2 * R1));
    });
    rdft<R1, false>(a);
    C* d = sm + ((c * 2 + p) * n + j2) * TILE + t;
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      const C w = ldc(tw + (p * R1 + k) * R2 + j2);
      const cv<T> b = cvmul(a[k], cv<T>{w.x, w.y});
      C o;
      o.x = b.re; o.y = b.im;
      d[k * R2 * TILE] = o;
    }
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 24 * R1; u += NT) {
    C* q = sm + (u / 4) * R2 * TILE + u % 4;
    cv<T> a[R2];
#pragma unroll
    for (int j = 0; j < R2; ++j) a[j] = {q[j * TILE].x, q[j * TILE].y};
    rdft<R2, false>(a);
#pragma unroll
    for (int j = 0; j < R2; ++j) { q[j * TILE].x = a[j].re; q[j * TILE].y = a[j].im; }
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 2 * n * TILE; u += NT) {
    const int t = u % 4, pos = u / 4, k2 = pos % R2, k1 = (pos / R2) % R1, p = pos / n;
    if (t >= ncol) continue;
    const int kz = 2 * (k1 + R1 * k2) + p, kx = op.kx_at[col0 + t];
    const bool fz = kz > n, fx = kx > (Lx >> 1);
    C g[6];
    G6<T>::load(ghat_at<T>(op, fz ? L - kz : kz, hy, fx ? Lx - kx : kx), 0, g);
    wide_mul<T, CROSS>(g, fx, fy, fz, sm + u, 2 * n * TILE);
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 24 * R1; u += NT) {
    C* q = sm + (u / 4) * R2 * TILE + u % 4;
    cv<T> a[R2];
#pragma unroll
    for (int j = 0; j < R2; ++j) a[j] = {q[j * TILE].x, q[j * TILE].y};
    rdft<R2, true>(a);
#pragma unroll
    for (int j = 0; j < R2; ++j) { q[j * TILE].x = a[j].re; q[j * TILE].y = a[j].im; }
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 24 * R2; u += NT) {
    const int t = u % 4, j2 = (u / 4) % R2, p = (u / (4 * R2)) & 1, c = u / (8 * R2);
    C* d = sm + ((c * 2 + p) * n + j2) * TILE + t;
    cv<T> a[R1];
#pragma unroll
    for (int k = 0; k < R1; ++k) {
      const C w = ldc(tw + (p * R1 + k) * R2 + j2);
      a[k] = cvmulc(cv<T>{w.x, w.y}, cv<T>{d[k * R2 * TILE].x, d[k * R2 * TILE].y});
    }
    rdft<R1, true>(a);
    static_for<R1>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      if (j > 0 && p) a[j] = cvrot<true>(a[j], cx_cos(j, 2 * R1), cx_sin(j, 2 * R1));
      d[j * R2 * TILE].x = a[j].re;
      d[j * R2 * TILE].y = a[j].im;
    });
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 3 * nz * TILE; u += NT) {
    const int t = u % 4, z = (u / 4) % nz, c = u / (4 * nz);
    if (t >= ncol) continue;
    const C* s = sm + (c * 2 * n + z) * TILE + t;
    base[c * comp + z * plane + t] = cadd(s[0], s[n * TILE]);
  }
}

template <int R1, int R2> cudaError_t configure_z_wide() {
  const void* k[] = {(const void*)k_fft_z_wide<df64, false, R1, R2>,
                     (const void*)k_fft_z_wide<double, false, R1, R2>,
                     (const void*)k_fft_z_wide<double, true, R1, R2>};
  for (const void* f : k) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)ZWideCfg<R1, R2>::smem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
// CROSS: the magnetic near field's vector product (FP64)
template <typename T, int R1, int R2>
void launch_z_wide(bool cross, const OpView<T>& op, int R, cplx_t<T>* buf, const int* active,
                   cudaStream_t st) {
  using K = ZWideCfg<R1, R2>;
  const dim3 g(2 * R, (op.Lx + K::TILE - 1) / K::TILE, op.Ly / 2 + 1);
  if constexpr (std::is_same<T, double>::value) {
    if (cross) {
      k_fft_z_wide<T, true, R1, R2><<<g, K::NT, K::smem, st>>>(op, buf, active);
      return;
    }
  }
  k_fft_z_wide<T, false, R1, R2><<<g, K::NT, K::smem, st>>>(op, buf, active);
}

// The plans of zpass_reg.cuh with R1, R2 <= 16, in parts that compile side by side
// (zpass_wide_*.cu).
#define DDA_ZWIDE_PART0(X) X(3, 3) X(5, 2) X(4, 3) X(5, 3) X(4, 4) X(6, 3) X(5, 4) X(6, 4) X(5, 5) X(9, 3) X(6, 5) X(8, 4) X(6, 6) X(8, 5)
#define DDA_ZWIDE_PART1(X) X(9, 5) X(8, 6) X(10, 5) X(9, 6) X(10, 6) X(8, 8) X(9, 8)
#define DDA_ZWIDE_PART2(X) X(15, 5) X(10, 8) X(9, 9) X(10, 9) X(12, 8) X(10, 10)
#define DDA_ZWIDE_PART3(X) X(12, 9) X(12, 10) X(16, 8) X(15, 9) X(12, 12)
#define DDA_ZWIDE_PART4(X) X(15, 10) X(16, 10) X(15, 12) X(16, 12)
#define DDA_ZWIDE_PART5(X) X(15, 15) X(16, 15) X(16, 16)
#define DDA_ZWIDE_ALL(X)                                                                       \
  DDA_ZWIDE_PART0(X) DDA_ZWIDE_PART1(X) DDA_ZWIDE_PART2(X) DDA_ZWIDE_PART3(X) DDA_ZWIDE_PART4(X) \
  DDA_ZWIDE_PART5(X)
#define DDA_ZWIDE_DECLARE(PART)                                                             \
  bool launch_z_wide_part##PART(bool cross, const OpView<df64>& op, int R, df64c* buf,      \
                                const int* active, cudaStream_t st);                        \
  bool launch_z_wide_part##PART(bool cross, const OpView<double>& op, int R, double2* buf,  \
                                const int* active, cudaStream_t st);                        \
  cudaError_t configure_z_wide_part##PART(int half);
DDA_ZWIDE_DECLARE(0) DDA_ZWIDE_DECLARE(1) DDA_ZWIDE_DECLARE(2)
DDA_ZWIDE_DECLARE(3) DDA_ZWIDE_DECLARE(4) DDA_ZWIDE_DECLARE(5)

#define DDA_ZWIDE_LAUNCH(A, B) case (A) * (B): launch_z_wide<real_t, A, B>(cross, op, R, buf, active, st); return true;
#define DDA_ZWIDE_CONFIG(A, B) case (A) * (B): return configure_z_wide<A, B>();
#define DDA_ZWIDE_DEFINE(PART)                                                              \
  bool launch_z_wide_part##PART(bool cross, const OpView<df64>& op, int R, df64c* buf,      \
                                const int* active, cudaStream_t st) {                       \
    using real_t = df64;                                                                    \
    switch (op.Lz / 2) { DDA_ZWIDE_PART##PART(DDA_ZWIDE_LAUNCH) }                           \
    return false;                                                                           \
  }                                                                                         \
  bool launch_z_wide_part##PART(bool cross, const OpView<double>& op, int R, double2* buf,  \
                                const int* active, cudaStream_t st) {                       \
    using real_t = double;                                                                  \
    switch (op.Lz / 2) { DDA_ZWIDE_PART##PART(DDA_ZWIDE_LAUNCH) }                           \
    return false;                                                                           \
  }                                                                                         \
  cudaError_t configure_z_wide_part##PART(int half) {                                       \
    switch (half) { DDA_ZWIDE_PART##PART(DDA_ZWIDE_CONFIG) }                                \
    return cudaSuccess;                                                                     \
  }

}  // namespace dda
