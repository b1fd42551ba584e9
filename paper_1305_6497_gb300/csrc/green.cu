// The lattice Green tensor and its transform on the padded FFT grid.
//
// A_jl = -G(r_j - r_l) for j != l (eq. AP=E).  CM and LDR use the point-dipole
// tensor G = (k^2 I + grad grad) e^{ikr}/r, i.e.
//   G_ab = A(r) delta_ab + B(r) n_a n_b,
//   A = e^{ikr}/r^3 ((kr)^2 - 1 + ikr),  B = e^{ikr}/r^3 (3 - (kr)^2 - 3ikr).
// FCD (Sec. "Filtered Coupled Dipole") uses (k^2 I + grad grad) g_F with g_F
// the outgoing scalar Green function with spatial frequencies above kF = pi/d
// removed; splitting q/(q^2-k^2) into partial fractions gives
//   r g_F = i sin(kr) + [cos(kr) S(r) + sin(kr) C(r)] / pi,
//   S = Si((kF-k)r) + Si((kF+k)r),  C = Ci((kF-k)r) - Ci((kF+k)r),
// and for a radial g: d_a d_b g = n_a n_b g'' + (delta_ab - n_a n_b) g'/r.
//
// G is laid on the periodic grid at offsets |Delta_x| < nx etc. (zero
// elsewhere, zero at Delta = 0), transformed by the same Stockham kernels as
// the matvec (FP64), and one octant of the transform is kept: components xx,
// yy, zz are even in every axis, xy is odd in x and y, xz in x and z, yz in y
// and z, so Ghat(L - k) = +/- Ghat(k) per axis.
#include <cmath>

#include "dda_ops.h"
#include "fft_core.cuh"

namespace dda {

// Si(x), Ci(x) for x > 0: power series below x = 2, and above it the
// continued fraction of E1(ix) = -Ci(x) + i (Si(x) - pi/2) (modified Lentz),
// E1(z) = e^{-z} / (z + 1 - 1/(z + 3 - 4/(z + 5 - ...))).
__device__ void sici(double x, double& si, double& ci) {
  const double kEuler = 0.57721566490153286061;
  const double kPiHalf = 1.57079632679489661923;
  if (x <= 2.0) {
    // Si = sum (-1)^n x^(2n+1) / ((2n+1)(2n+1)!), Ci = gamma + ln x + sum_{n>=1} (-1)^n x^(2n)/(2n (2n)!)
    double term = x;  // x^(2n+1)/(2n+1)! with sign
    double s = x;
    double fact_term = 1.0;  // x^(2n)/(2n)! with sign
    double c = 0.0;
    const double x2 = x * x;
    for (int n = 1; n < 40; ++n) {
      fact_term *= -x2 / ((2.0 * n - 1.0) * (2.0 * n));
      c += fact_term / (2.0 * n);
      term *= -x2 / ((2.0 * n) * (2.0 * n + 1.0));
      const double add = term / (2.0 * n + 1.0);
      s += add;
      if (fabs(add) < 1e-18 * fabs(s) && fabs(fact_term) < 1e-18) break;
    }
    si = s;
    ci = kEuler + log(x) + c;
    return;
  }
  // modified Lentz on b0 + a1/(b1 + a2/(b2 + ...)), b_n = z + 2n + 1, a_n = -n^2
  const double tiny = 1e-300;
  double2 b = make_double2(1.0, x);               // z + 1, z = i x
  double2 cc = make_double2(1.0 / tiny, 0.0);
  double2 d = make_double2(b.x / (b.x * b.x + b.y * b.y), -b.y / (b.x * b.x + b.y * b.y));
  double2 h = d;
  for (int n = 1; n < 400; ++n) {
    const double a = -(double)n * n;
    b.x += 2.0;
    // d = 1/(a d + b), c = b + a/c
    double2 ad = make_double2(a * d.x + b.x, a * d.y + b.y);
    const double dn = ad.x * ad.x + ad.y * ad.y;
    d = make_double2(ad.x / dn, -ad.y / dn);
    const double cn = cc.x * cc.x + cc.y * cc.y;
    cc = make_double2(b.x + a * cc.x / cn, b.y - a * cc.y / cn);
    const double2 del = cmul(cc, d);
    h = cmul(h, del);
    if (fabs(del.x - 1.0) + fabs(del.y) < 1e-16) break;
  }
  // E1(ix) = e^{-ix} h
  double sx, cx;
  sincos(x, &sx, &cx);
  const double2 e1 = cmul(make_double2(cx, -sx), h);
  ci = -e1.x;
  si = kPiHalf + e1.y;
}

// The scalar Green function at r > 0 and its first two radial derivatives:
// point g = e^{ikr}/r, or the filtered g_F (FCD).
__device__ void scalar_green(double r, double k, int filtered, double2& g, double2& g1,
                             double2& g2) {
  const double kr = k * r;
  double skr, ckr;
  sincos(kr, &skr, &ckr);
  const double ir = 1.0 / r, ir2 = ir * ir, ir3 = ir2 * ir;
  if (!filtered) {
    const double2 e = make_double2(ckr, skr);  // e^{ikr}
    g = cscale(e, ir);
    g1 = cscale(cmul(e, make_double2(-1.0, kr)), ir2);                        // (ikr - 1)/r^2
    g2 = cscale(cmul(e, make_double2(2.0 - kr * kr, -2.0 * kr)), ir3);        // (2 - 2ikr - k^2r^2)/r^3
    return;
  }
  const double kf = 3.14159265358979323846;  // pi / d
  const double a = kf - k, b = kf + k;
  double sia, cia, sib, cib;
  sici(a * r, sia, cia);
  sici(b * r, sib, cib);
  double sar, car, sbr, cbr;
  sincos(a * r, &sar, &car);
  sincos(b * r, &sbr, &cbr);
  const double S = sia + sib, Cc = cia - cib;
  const double S1 = (sar + sbr) / r, C1 = (car - cbr) / r;
  const double S2 = (a * car + b * cbr) / r - S1 / r;
  const double C2 = (-a * sar + b * sbr) / r - C1 / r;
  const double ip = 0.31830988618379067154;  // 1/pi
  // h = r g, h', h''
  const double2 h = make_double2(ip * (ckr * S + skr * Cc), skr);
  const double2 h1 = make_double2(ip * (-k * skr * S + ckr * S1 + k * ckr * Cc + skr * C1),
                                  k * ckr);
  const double2 h2 = make_double2(ip * (-k * k * ckr * S - 2.0 * k * skr * S1 + ckr * S2 -
                                        k * k * skr * Cc + 2.0 * k * ckr * C1 + skr * C2),
                                  -k * k * skr);
  g = cscale(h, ir);
  g1 = csub(cscale(h1, ir), cscale(h, ir2));
  g2 = cadd(csub(cscale(h2, ir), cscale(h1, 2.0 * ir2)), cscale(h, 2.0 * ir3));
}

// Tensor at offset (dx, dy, dz) != 0 : out[0..5] = xx, xy, xz, yy, yz, zz
__device__ void green_tensor(double dx, double dy, double dz, double k, int filtered,
                             double2 out[6]) {
  const double r2 = dx * dx + dy * dy + dz * dz;
  const double r = sqrt(r2);
  const double n[3] = {dx / r, dy / r, dz / r};
  double2 A, B;
  if (!filtered) {
    const double kr = k * r;
    double skr, ckr;
    sincos(kr, &skr, &ckr);
    const double inv3 = 1.0 / (r2 * r);
    const double2 e = make_double2(ckr * inv3, skr * inv3);  // e^{ikr}/r^3
    A = cmul(e, make_double2(kr * kr - 1.0, kr));
    B = cmul(e, make_double2(3.0 - kr * kr, -3.0 * kr));
  } else {
    double2 g, g1, g2;
    scalar_green(r, k, 1, g, g1, g2);
    const double ir = 1.0 / r;
    A = cadd(cscale(g, k * k), cscale(g1, ir));
    B = csub(g2, cscale(g1, ir));
  }
  out[0] = cadd(A, cscale(B, n[0] * n[0]));
  out[1] = cscale(B, n[0] * n[1]);
  out[2] = cscale(B, n[0] * n[2]);
  out[3] = cadd(A, cscale(B, n[1] * n[1]));
  out[4] = cscale(B, n[1] * n[2]);
  out[5] = cadd(A, cscale(B, n[2] * n[2]));
}

// Magnetic field of a dipole P at offset r (Gaussian units): B = h(r) x P with
// h = -i k g'(r) rhat (from B = curl A, A = -i k P g), i.e. for the point
// dipole h = k^2 (e^{ikr}/r)(1 + i/(kr)) rhat; FCD uses the filtered g_F.
// out[0..2] = h_x, h_y, h_z.
__device__ void magnetic_vector(double dx, double dy, double dz, double k, int filtered,
                                double2 out[3]) {
  const double r = sqrt(dx * dx + dy * dy + dz * dz);
  double2 g, g1, g2;
  scalar_green(r, k, filtered, g, g1, g2);
  const double2 m = make_double2(k * g1.y, -k * g1.x);  // -i k g'
  out[0] = cscale(m, dx / r);
  out[1] = cscale(m, dy / r);
  out[2] = cscale(m, dz / r);
}

// Parity of each component under the reflection of x, y, z: G xx, xy, xz, yy, yz,
// zz, or h_x, h_y, h_z (odd in their own axis) for the magnetic vector.
__device__ __forceinline__ bool green_odd(bool mag, int c, int axis) {
  if (mag) return c == axis;
  // xy: x, y; xz: x, z; yz: y, z
  return c == 1 ? axis != 2 : c == 2 ? axis != 1 : c == 4 ? axis != 0 : false;
}

// The transform of G on the periodic grid, from the octant of offsets alone.  G is
// even or odd in each axis, so a line of the grid is its first n values and their
// mirror images, its transform is even or odd too, and lines that are mirror
// images of each other need not be transformed: along x the ny nz lines of the
// octant, along y the Hx = Lx/2 + 1 kept frequencies of nz planes, along z the
// Hx Hy kept columns -- a quarter of the full grid's lines on each axis, and one
// array [6][nz][Hy][Hx] instead of two of the full grid.  A mirrored line is put
// together in shared memory and transformed like a full grid's, so the kept values
// are those of the full transform, bit for bit.
//
// What bounds it: FP64 arithmetic.  Build for a new wavelength, before (two full
// grids, allocated and freed each time) and now: 256^3 box 171 -> 41 ms,
// 100x75x135 12.7 -> 3.0, 64^3 2.5 -> 0.59, 70x54x54 2.5 -> 0.59, 16^3 0.35 -> 0.06.

// x pass: rows (y < ny, z < nz), six components a row; the tensor is evaluated
// here.  buf [6][nz][Hy][Hx], rows y < ny.  Shared memory: L x (6 rows) lines.
__global__ void __launch_bounds__(256)
k_green_x(int nx, int ny, int nz, AxisPlan P, const double2* __restrict__ tw,
          const int* __restrict__ pos, int Hx, int Hy, double k, int kind, int per,
          double2* __restrict__ buf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* s = reinterpret_cast<double2*>(smem_raw);
  const int L = P.L, nl = 6 * per;
  const bool mag = (kind & 2) != 0;
  const int row0 = blockIdx.x * per, rows = ny * nz;
  const double2 zero = make_double2(0.0, 0.0);
  // positions nx .. L - nx hold no offset
  for (int e = threadIdx.x; e < (L - 2 * nx + 1) * nl; e += blockDim.x) s[nx * nl + e] = zero;
  for (int e = threadIdx.x; e < nx * per; e += blockDim.x) {
    const int q = e / nx, dx = e - q * nx, row = row0 + q;
    const int dz = row / ny, dy = row - dz * ny;
    double2 g[6] = {zero, zero, zero, zero, zero, zero};
    if (row < rows && (dx | dy | dz) != 0) {
      if (mag) magnetic_vector((double)dx, (double)dy, (double)dz, k, kind & 1, g);
      else green_tensor((double)dx, (double)dy, (double)dz, k, kind & 1, g);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      s[dx * nl + 6 * q + c] = g[c];
      if (dx > 0)
        s[(L - dx) * nl + 6 * q + c] =
            green_odd(mag, c, 0) ? make_double2(-g[c].x, -g[c].y) : g[c];
    }
  }
  __syncthreads();
  fft_smem<double2, false>(s, nl, nl, P, tw);
  for (int e = threadIdx.x; e < Hx * nl; e += blockDim.x) {
    const int line = e / Hx, h = e - line * Hx;
    const int q = line / 6, c = line - 6 * q, row = row0 + q;
    if (row >= rows) continue;
    const int z = row / ny, y = row - z * ny;
    buf[(((int64_t)c * nz + z) * Hy + y) * Hx + h] = s[pos[h] * nl + line];
  }
}

// One line of the y or z pass in shared memory: n values and their mirror images.
__device__ __forceinline__ void green_mirror(double2* s, int tile, int t, int p, int L, double2 v,
                                             bool odd) {
  s[p * tile + t] = v;
  if (p > 0) s[(L - p) * tile + t] = odd ? make_double2(-v.x, -v.y) : v;
}

// y pass, in place: ny rows of each (component, z) plane in, Hy rows out.
// grid: (column tiles, 6 nz)
__global__ void __launch_bounds__(512)
k_green_y(int ny, int nz, AxisPlan P, const double2* __restrict__ tw, const int* __restrict__ pos,
          int Hx, int Hy, int kind, int tile, double2* __restrict__ buf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* s = reinterpret_cast<double2*>(smem_raw);
  const int L = P.L, col0 = blockIdx.x * tile, ncol = min(tile, Hx - col0);
  const int c = blockIdx.y / nz;
  const bool odd = green_odd((kind & 2) != 0, c, 1);
  double2* base = buf + (int64_t)blockIdx.y * Hy * Hx + col0;
  const double2 zero = make_double2(0.0, 0.0);
  for (int e = threadIdx.x; e < (L - 2 * ny + 1) * tile; e += blockDim.x) s[ny * tile + e] = zero;
  for (int e = threadIdx.x; e < ny * tile; e += blockDim.x) {
    const int p = e / tile, t = e - p * tile;
    green_mirror(s, tile, t, p, L, t < ncol ? base[(int64_t)p * Hx + t] : zero, odd);
  }
  __syncthreads();
  fft_smem<double2, false>(s, tile, tile, P, tw);
  for (int e = threadIdx.x; e < Hy * tile; e += blockDim.x) {
    const int h = e / tile, t = e - h * tile;
    if (t < ncol) base[(int64_t)h * Hx + t] = s[pos[h] * tile + t];
  }
}

// z pass: nz planes in, the octant out, scaled by 1/(Lx Ly Lz): FP64, and FP32 and
// double-float where given.  grid: (6, column tiles of Hx Hy), the components of a
// tile neighbours, since they share the lines they are written to.
__global__ void __launch_bounds__(512)
k_green_z(int nz, AxisPlan P, const double2* __restrict__ tw, const int* __restrict__ pos, int Hx,
          int Hy, int kind, int tile, int64_t first, double scale, const double2* __restrict__ buf,
          double2* __restrict__ g64, float2* __restrict__ g32, GhatLayout gl,
          df64c* __restrict__ gdf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* s = reinterpret_cast<double2*>(smem_raw);
  const int L = P.L, Hz = L / 2 + 1, c = blockIdx.x;
  const int64_t plane = (int64_t)Hx * Hy, col0 = first + (int64_t)blockIdx.y * tile;
  const int ncol = (int)min((int64_t)tile, plane - col0);
  const bool odd = green_odd((kind & 2) != 0, c, 2);
  const double2* base = buf + (int64_t)c * nz * plane + col0;
  const double2 zero = make_double2(0.0, 0.0);
  for (int e = threadIdx.x; e < (L - 2 * nz + 1) * tile; e += blockDim.x) s[nz * tile + e] = zero;
  for (int e = threadIdx.x; e < nz * tile; e += blockDim.x) {
    const int p = e / tile, t = e - p * tile;
    green_mirror(s, tile, t, p, L, t < ncol ? base[p * plane + t] : zero, odd);
  }
  __syncthreads();
  fft_smem<double2, false>(s, tile, tile, P, tw);
  for (int e = threadIdx.x; e < Hz * tile; e += blockDim.x) {
    const int hz = e / tile, t = e - hz * tile;
    if (t >= ncol) continue;
    const double2 v = s[pos[hz] * tile + t];
    const double2 w = make_double2(v.x * scale, v.y * scale);
    const int64_t col = col0 + t, o = 6 * (hz * plane + col) + c;
    g64[o] = w;
    if (gdf) gdf[o] = from_io<df64c>(w);
    if (g32)
      g32[hz * gl.sz + col * gl.sxy + (c >> 1) * 2 * gl.piece + (c & 1)] =
          make_float2((float)w.x, (float)w.y);
  }
}

size_t green_scratch_bytes(int nz, int Lx, int Ly) {
  return sizeof(double2) * 6 * (size_t)nz * (Ly / 2 + 1) * (Lx / 2 + 1);
}

cudaError_t launch_green_transform(const OpView<double>& op, const int* posx, const int* posy,
                                   const int* posz, double kd, int kind, double2* scratch,
                                   double2* g64, float2* g32, GhatLayout gl, df64c* gdf,
                                   cudaStream_t st) {
  const int Hx = op.Lx / 2 + 1, Hy = op.Ly / 2 + 1;
  const size_t kLimit = 200 * 1024;
  const void* ks[] = {(const void*)k_green_x, (const void*)k_green_y, (const void*)k_green_z};
  for (const void* k : ks) {
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLimit);
    if (e != cudaSuccess) return e;
  }
  const int rows = op.ny * op.nz;
  int per = 1;  // rows of a CTA: up to 48 KB
  while (per < 8 && (size_t)12 * per * op.Lx * sizeof(double2) <= 48 * 1024) per *= 2;
  k_green_x<<<(rows + per - 1) / per, 256, (size_t)6 * per * op.Lx * sizeof(double2), st>>>(
      op.nx, op.ny, op.nz, op.px, op.twx, posx, Hx, Hy, kd, kind, per, scratch);
  note_launch();
  auto shape = [](int L, int& tile, int& th) {
    tile = 8;
    while (tile > 1 && (size_t)tile * L * sizeof(double2) > 64 * 1024) tile >>= 1;
    th = ((tile * L / 4 + 31) / 32) * 32;
    th = th < 64 ? 64 : (th > 512 ? 512 : th);
  };
  int tile, th;
  shape(op.Ly, tile, th);
  k_green_y<<<dim3((Hx + tile - 1) / tile, 6 * op.nz), th, (size_t)tile * op.Ly * sizeof(double2), st>>>(
      op.ny, op.nz, op.py, op.twy, posy, Hx, Hy, kind, tile, scratch);
  note_launch();
  shape(op.Lz, tile, th);
  const int64_t plane = (int64_t)Hx * Hy, tiles = (plane + tile - 1) / tile;
  // grid.y is limited to 65535 tiles a launch
  for (int64_t t0 = 0; t0 < tiles; t0 += 65535) {
    const int nt = (int)(tiles - t0 < 65535 ? tiles - t0 : 65535);
    k_green_z<<<dim3(6, nt), th, (size_t)tile * op.Lz * sizeof(double2), st>>>(
        op.nz, op.pz, op.twz, posz, Hx, Hy, kind, tile, t0 * tile,
        1.0 / ((double)op.Lx * op.Ly * op.Lz), scratch, g64, g32, gl, gdf);
    note_launch();
  }
  return cudaGetLastError();
}

}  // namespace dda
