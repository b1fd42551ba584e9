// Cross sections and scattering amplitudes from the solved dipole moments.
//
//  C_ext = 4 pi k sum_j Im(E_inc,j^* . P_j)
//  C_abs = 4 pi k sum_j sum_a |P_ja|^2 [-Im(1/alpha_ja) - (2/3) k^3]  (a: lattice
//          axis; alpha's diagonal, equal on the axes except for GKDLDR)
//  (Sec. "What Does It Calculate?": Q = C / (pi a_eff^2), Q_ext = Q_sca + Q_abs)
//  F(n) = sum_j P_j exp(-i k n . r_j), f_ml = k^3 e_m . F  (eq. f_ml_def)
//
// On the lattice exp(-i k n.r_j) = ex(ix) ey(iy) ez(iz), so the phases come
// from three short per-axis tables and no transcendental is evaluated per site.
// All sums are FP64, two-stage and deterministic.
#include <algorithm>

#include "dda_ops.h"
#include "reduce.cuh"

namespace dda {

__global__ void k_cross_sections(int nx, int ny, int nz, const uint8_t* __restrict__ comp,
                                 RhsTables tb, const double2* __restrict__ P,
                                 const double* __restrict__ wabs, int ncomp1,
                                 double* partials) {
  const int r = blockIdx.y;
  const int64_t nbox = (int64_t)nx * ny * nz;
  const double2 e0 = tb.pol[r * 3 + 0], e1 = tb.pol[r * 3 + 1], e2 = tb.pol[r * 3 + 2];
  double acc[2] = {0.0, 0.0};
  GRID_LOOP(i, nbox) {
    const int cm = comp[i];
    if (cm) {
      const int ix = (int)(i % nx);
      const int64_t q = i / nx;
      const int iy = (int)(q % ny), iz = (int)(q / ny);
      const double2 ph = cmul(cmul(tb.phx[(int64_t)r * nx + ix], tb.phy[(int64_t)r * ny + iy]),
                              tb.phz[(int64_t)r * nz + iz]);
      const double2 p0 = P[((int64_t)r * 3 + 0) * nbox + i];
      const double2 p1 = P[((int64_t)r * 3 + 1) * nbox + i];
      const double2 p2 = P[((int64_t)r * 3 + 2) * nbox + i];
      // E^* . P = conj(ph) * (conj(e) . P)
      double2 ep = cadd(cadd(cmulc(e0, p0), cmulc(e1, p1)), cmulc(e2, p2));
      ep = cmulc(ph, ep);
      acc[0] += ep.y;
      const double* wa = wabs + ((int64_t)r * ncomp1 + cm) * 3;
      acc[1] += (p0.x * p0.x + p0.y * p0.y) * wa[0] + (p1.x * p1.x + p1.y * p1.y) * wa[1] +
                (p2.x * p2.x + p2.y * p2.y) * wa[2];
    }
  }
  write_partials<2>(acc, partials);
}

cudaError_t launch_cross_sections(int nx, int ny, int nz, const uint8_t* comp, RhsTables tb,
                                  int R, const double2* P, const double* wabs, int ncomp1,
                                  double* partials, int nblk, cudaStream_t st) {
  dim3 g(nblk, R);
  k_cross_sections<<<g, kThreads, 0, st>>>(nx, ny, nz, comp, tb, P, wabs, ncomp1, partials);
  note_launch();
  return cudaGetLastError();
}

// Phase tables exp(-i kd n_a (i - (n_a^box - 1) / 2)) of D directions n (dirs [D][3]) on the
// three axes: [D][nx], then [D][ny], then [D][nz].
__global__ void k_direction_phases(int nx, int ny, int nz, int D, double kd,
                                   const double* __restrict__ dirs, double2* __restrict__ ph) {
  const int per = nx + ny + nz;
  const int64_t entries = (int64_t)D * per;  // 2^31 of them are 34 GB, which the part holds
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < entries;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int d = (int)(e / per), q = (int)(e - (int64_t)d * per);
    const int a = q < nx ? 0 : q < nx + ny ? 1 : 2;
    const int n = a == 0 ? nx : a == 1 ? ny : nz;
    const int i = a == 0 ? q : a == 1 ? q - nx : q - nx - ny;
    double sn, cs;
    sincos(-kd * dirs[3 * (int64_t)d + a] * (i - 0.5 * (n - 1)), &sn, &cs);
    ph[(a == 0 ? (int64_t)d * nx : a == 1 ? (int64_t)D * nx + (int64_t)d * ny
                                          : (int64_t)D * (nx + ny) + (int64_t)d * nz) + i] =
        make_double2(cs, sn);
  }
}

cudaError_t launch_direction_phases(int nx, int ny, int nz, int D, double kd, const double* dirs,
                                    double2* ph, cudaStream_t st) {
  const int64_t n = (int64_t)D * (nx + ny + nz);
  const int blocks = (int)std::min<int64_t>((n + 127) / 128, 152 * 8);
  k_direction_phases<<<blocks, 128, 0, st>>>(nx, ny, nz, D, kd, dirs, ph);
  note_launch();
  return cudaGetLastError();
}

// Far field of R right-hand sides (the polarizations of an incidence) in D directions.
// A thread holds one lattice column (x, y) and DC directions: over its z it sums
// ez_d(z) P, 12 FP64 multiply-adds a site, direction and polarization with a phase
// that is the same for every thread, and only then multiplies by ex_d(x) ey_d(y) and
// joins the block's sum.  P is read once for DC directions and every polarization;
// warps skip planes where none of their sites is occupied.
//
// What bounds it: FP64 arithmetic.  A phase per site and direction (a thread per site,
// two complex products a site) took 20 instructions for each polarization, and the
// tables came from the host: 350 scattering directions of each orientation of the
// 48x96x144 ellipsoid took 83 ms of a 222 ms orientation average, now 29 of 167.
//
// grid: (column blocks x z chunks, direction chunks); partials [(d R + r) nblk + blk][6]
template <int DC, int R>
__global__ void __launch_bounds__(kThreads)
k_farfield(int nx, int ny, int nz, int cols, int zper, int D, const uint8_t* __restrict__ comp,
           const double2* __restrict__ P, const double2* __restrict__ fphx,
           const double2* __restrict__ fphy, const double2* __restrict__ fphz,
           double* __restrict__ partials) {
  const int cb = blockIdx.x % cols, zc = blockIdx.x / cols, d0 = blockIdx.y * DC;
  const int64_t nxy = (int64_t)nx * ny, nbox = nxy * nz;
  const int64_t col = (int64_t)cb * kThreads + threadIdx.x;
  const bool in = col < nxy;
  double2 acc[DC][R][3];
#pragma unroll
  for (int d = 0; d < DC; ++d)
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[d][r][c] = make_double2(0.0, 0.0);
  const int z1 = min(nz, (zc + 1) * zper);
  for (int z = zc * zper; z < z1; ++z) {
    const bool occ = in && comp[z * nxy + col];
    if (!__any_sync(0xffffffffu, occ)) continue;
    double2 p[R][3];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c)  // vacant sites hold zeros
        p[r][c] = in ? P[((int64_t)r * 3 + c) * nbox + z * nxy + col] : make_double2(0.0, 0.0);
#pragma unroll
    for (int d = 0; d < DC; ++d) {
      const double2 e = __ldg(fphz + (int64_t)min(d0 + d, D - 1) * nz + z);
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          double2& a = acc[d][r][c];
          a.x = fma(p[r][c].x, e.x, fma(-p[r][c].y, e.y, a.x));
          a.y = fma(p[r][c].x, e.y, fma(p[r][c].y, e.x, a.y));
        }
    }
  }
  const int ix = in ? (int)(col % nx) : 0, iy = in ? (int)(col / nx) : 0;
#pragma unroll
  for (int d = 0; d < DC; ++d) {
    if (d0 + d >= D) break;
    const double2 xy = cmul(fphx[(int64_t)(d0 + d) * nx + ix], fphy[(int64_t)(d0 + d) * ny + iy]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      double v[6], tot[6];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double2 t = cmul(acc[d][r][c], xy);
        v[2 * c] = t.x;
        v[2 * c + 1] = t.y;
      }
      block_sum<6>(v, tot);
      if (threadIdx.x == 0) {
        double* o = partials + (((int64_t)(d0 + d) * R + r) * gridDim.x + blockIdx.x) * 6;
#pragma unroll
        for (int i = 0; i < 6; ++i) o[i] = tot[i];
      }
    }
  }
}

// Directions per thread: the accumulators of four directions and two polarizations
// take 96 registers; fewer where that wastes less of the last chunk.  z chunks: only
// as many as about four blocks per SM need (every chunk closes with a block sum of
// its own, which costs as much as ten planes), of two planes or more.
static void farfield_grid(int nx, int ny, int nz, int D, int& dc, int& cols, int& zchunks) {
  dc = 4;
  for (int c : {3, 2, 1})
    if ((D + c - 1) / c * c < (D + dc - 1) / dc * dc) dc = c;
  cols = (int)(((int64_t)nx * ny + kThreads - 1) / kThreads);
  const int64_t blocks = (int64_t)cols * ((D + dc - 1) / dc);
  zchunks = (int)std::max<int64_t>(1, std::min<int64_t>((608 + blocks - 1) / blocks, (nz + 1) / 2));
  const int per = (nz + zchunks - 1) / zchunks;
  zchunks = (nz + per - 1) / per;
}

// Directions of one launch.  Every column block leaves six sums per direction and
// right-hand side: 4096 blocks of a 1024 x 1024 box 393 KB per direction.  A chunk's
// partial sums stay within 8 MiB (340 directions of a 256^3 box, still 21,000 blocks)
// and its phase tables within 64 MiB.  Chunks are of equal size and, but for the last,
// hold a multiple of the four directions of a thread.
int farfield_chunk(int nx, int ny, int nz, int D) {
  const int64_t cols = ((int64_t)nx * ny + kThreads - 1) / kThreads;
  const int64_t c = std::min((8ll << 20) / (96 * cols), (64ll << 20) / (16 * (nx + ny + nz)));
  const int64_t most = std::max<int64_t>(4, c / 4 * 4), k = (D + most - 1) / most;
  return (int)std::min<int64_t>(D, ((D + k - 1) / k + 3) / 4 * 4);
}

int farfield_blocks(int nx, int ny, int nz, int D) {
  int dc, cols, zchunks;
  farfield_grid(nx, ny, nz, D, dc, cols, zchunks);
  return cols * zchunks;
}

cudaError_t launch_farfield(int nx, int ny, int nz, const uint8_t* comp, int R, int D, int n,
                            const double2* P, const double2* fphx, const double2* fphy,
                            const double2* fphz, double* partials, cudaStream_t st) {
  int dc, cols, zchunks;
  farfield_grid(nx, ny, nz, D, dc, cols, zchunks);
  const int zper = (nz + zchunks - 1) / zchunks;
  for (int c0 = 0; c0 < (n + dc - 1) / dc; c0 += 65535) {  // grid.y limit
    const int d0 = c0 * dc, m = std::min(n - d0, 65535 * dc);
    const dim3 g(cols * zchunks, (m + dc - 1) / dc);
#define DDA_FAR(DC, RR)                                                                      \
  k_farfield<DC, RR><<<g, kThreads, 0, st>>>(nx, ny, nz, cols, zper, m, comp, P,             \
                                             fphx + (int64_t)d0 * nx, fphy + (int64_t)d0 * ny, \
                                             fphz + (int64_t)d0 * nz,                        \
                                             partials + (int64_t)d0 * R * cols * zchunks * 6)
    if (R == 1) {
      if (dc == 4) DDA_FAR(4, 1);
      else if (dc == 3) DDA_FAR(3, 1);
      else if (dc == 2) DDA_FAR(2, 1);
      else DDA_FAR(1, 1);
    } else {
      if (dc == 4) DDA_FAR(4, 2);
      else if (dc == 3) DDA_FAR(3, 2);
      else if (dc == 2) DDA_FAR(2, 2);
      else DDA_FAR(1, 2);
    }
#undef DDA_FAR
    note_launch();
  }
  return cudaGetLastError();
}

// ---- near field (the guide's NRFLD option, Sec. "Near-Field Calculations") ---------
// E_sca is the field of all dipoles at each box site without the site's own
// dipole; the total microscopic field is E_inc + E_sca, and inside the target
// the macroscopic field is E_macro = 3 / (eps + 2) E_micro (eq. macro_vs_micro),
// in vacuum the two are equal.
// The incident magnetic field of the plane wave is B_inc = khat x E_inc.
__global__ void k_nearfield_post(int nx, int ny, int nz, const uint8_t* __restrict__ comp,
                                 RhsTables tb, const double2* __restrict__ esca,
                                 const double2* __restrict__ fac, const double* __restrict__ khat,
                                 double2* __restrict__ einc, double2* __restrict__ emacro,
                                 double2* __restrict__ binc) {
  const int r = blockIdx.y;
  const int64_t nbox = (int64_t)nx * ny * nz;
  GRID_LOOP(i, nbox) {
    const int ix = (int)(i % nx);
    const int64_t q = i / nx;
    const int iy = (int)(q % ny), iz = (int)(q / ny);
    const double2 ph = cmul(cmul(tb.phx[(int64_t)r * nx + ix], tb.phy[(int64_t)r * ny + iy]),
                            tb.phz[(int64_t)r * nz + iz]);
    const double2 f = fac[comp[i]];
    double2 ei[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int64_t o = ((int64_t)r * 3 + c) * nbox + i;
      ei[c] = cmul(tb.pol[r * 3 + c], ph);
      if (einc) einc[o] = ei[c];
      if (emacro) {
        const double2 es = esca[o];
        emacro[o] = cmul(f, make_double2(ei[c].x + es.x, ei[c].y + es.y));
      }
    }
    if (binc) {
      const double* k = khat + 3 * r;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
        binc[((int64_t)r * 3 + c) * nbox + i] =
            csub(cscale(ei[c2], k[c1]), cscale(ei[c1], k[c2]));
      }
    }
  }
}

cudaError_t launch_nearfield_post(int nx, int ny, int nz, const uint8_t* comp, RhsTables tb,
                                  int R, const double2* esca, const double2* fac,
                                  const double* khat, double2* einc, double2* emacro,
                                  double2* binc, cudaStream_t st) {
  const int64_t nbox = (int64_t)nx * ny * nz;
  dim3 g(reduce_blocks(nbox), R);
  k_nearfield_post<<<g, kThreads, 0, st>>>(nx, ny, nz, comp, tb, esca, fac, khat, einc,
                                           emacro, binc);
  note_launch();
  return cudaGetLastError();
}

}  // namespace dda
