// Shared device/host definitions for the GB300 DDA library.
//
// Layouts (all device memory):
//  - box vectors: [R][3][nz][ny][nx] complex (R right-hand sides, 3 Cartesian
//    components), zero on vacant sites;
//  - spectral scratch: [R][3][nz][Ly][Lx] complex.  The x pass fills rows
//    y < ny, the y pass expands each (z, column) to Ly rows in place, the fused
//    z pass transforms along z, multiplies by the Green tensor transform and
//    transforms back in place, and the inverse y and x passes shrink back;
//  - Green tensor transform: one octant [Lz/2+1][Ly/2+1][Lx/2+1][6] complex
//    (components xx, xy, xz, yy, yz, zz side by side; FP32 with a register z pass:
//    [Ly/2+1][Lx/2+1][3][Lz/2+1][2], pairs of components with hz fastest), the
//    rest follows from the parity of each component in each axis.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dda {

constexpr int kMaxStages = 12;
constexpr int kMaxComp = 256;

// ---- double-float ("df64") arithmetic ----------------------------------------
// A value is the unevaluated sum hi + lo of two FP32 numbers (|lo| <= ulp(hi)/2),
// about 48 significant bits.  FP64 runs at 1/58 of the FP32 rate on this part,
// so FFT passes that need FP64-level accuracy (the refinement's residual
// A.x) run in this arithmetic instead.  Sums use Knuth's TwoSum and Dekker's
// Fast2Sum, products the FMA-based exact product (Dekker; Ogita, Rump & Oishi
// 2005); the absolute error of a sum is ~2^-48 (|a| + |b|), enough for an FFT.
// The _rn intrinsics keep the compiler from contracting or reassociating.
struct df64 {
  float hi, lo;
  df64() = default;
  __host__ __device__ constexpr df64(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ df64(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
};
__device__ __forceinline__ df64 df_fast2sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return df64(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ df64 operator+(df64 a, df64 b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return df_fast2sum(s, e);
}
__device__ __forceinline__ df64 operator-(df64 a) { return df64(-a.hi, -a.lo); }
__device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }
__device__ __forceinline__ df64 operator*(df64 a, df64 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_fast2sum(p, e);
}
__host__ __device__ __forceinline__ double df_to_double(df64 a) {
  return (double)a.hi + (double)a.lo;
}
struct __align__(16) df64c { df64 x, y; };

// Complex type for a real type.
template <typename T> struct Cplx;
template <> struct Cplx<float> { using type = float2; };
template <> struct Cplx<double> { using type = double2; };
template <> struct Cplx<df64> { using type = df64c; };
template <typename T> using cplx_t = typename Cplx<T>::type;

// Type of the box vectors a matvec reads and writes (the FFT scratch is
// cplx_t<T>): df64 passes take and return FP64 vectors.
template <typename T> struct IoT { using type = cplx_t<T>; };
template <> struct IoT<df64> { using type = double2; };
template <typename T> using io_t = typename IoT<T>::type;

template <typename C> __host__ __device__ __forceinline__ C mk(double re, double im);
template <> __host__ __device__ __forceinline__ float2 mk<float2>(double re, double im) {
  return make_float2((float)re, (float)im);
}
template <> __host__ __device__ __forceinline__ double2 mk<double2>(double re, double im) {
  return make_double2(re, im);
}
template <> __host__ __device__ __forceinline__ df64c mk<df64c>(double re, double im) {
  df64c r;
  r.x = df64(re);
  r.y = df64(im);
  return r;
}

// box-vector element <-> FFT element
template <typename C, typename IO> __device__ __forceinline__ C from_io(IO v) { return v; }
template <> __device__ __forceinline__ df64c from_io<df64c, double2>(double2 v) {
  df64c r;
  r.x = df64(v.x);
  r.y = df64(v.y);
  return r;
}
template <typename IO, typename C> __device__ __forceinline__ IO to_io(C v) { return v; }
template <> __device__ __forceinline__ double2 to_io<double2, df64c>(df64c v) {
  return make_double2(df_to_double(v.x), df_to_double(v.y));
}

// read-only load of a complex value (tables)
template <typename C> __device__ __forceinline__ C ldc(const C* p) { return __ldg(p); }
template <> __device__ __forceinline__ df64c ldc<df64c>(const df64c* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  df64c r;
  r.x = df64(v.x, v.y);
  r.y = df64(v.z, v.w);
  return r;
}

template <typename C> __host__ __device__ __forceinline__ C cadd(C a, C b) {
  C r; r.x = a.x + b.x; r.y = a.y + b.y; return r;
}
template <typename C> __host__ __device__ __forceinline__ C csub(C a, C b) {
  C r; r.x = a.x - b.x; r.y = a.y - b.y; return r;
}
template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
  C r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
}
// conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cmulc(C a, C b) {
  C r; r.x = a.x * b.x + a.y * b.y; r.y = a.x * b.y - a.y * b.x; return r;
}
template <typename C, typename T> __host__ __device__ __forceinline__ C cscale(C a, T s) {
  C r; r.x = a.x * s; r.y = a.y * s; return r;
}
// multiply by -i (forward) or +i (inverse)
template <bool INV, typename C> __host__ __device__ __forceinline__ C cmul_i(C a) {
  C r;
  if (INV) { r.x = -a.y; r.y = a.x; } else { r.x = a.y; r.y = -a.x; }
  return r;
}

// One 1-D transform of length L = prod(radix[t]), in place.  Stage t works on
// blocks of blk[t] points with span blk[t]/radix[t]; its twiddles are
// tw[tw_off[t] + j*(radix[t]-1) + (m-1)] = exp(-2 pi i j m / blk[t]).
struct AxisPlan {
  int L;
  int nstage;
  int radix[kMaxStages];
  int blk[kMaxStages];
  int tw_off[kMaxStages];
  unsigned long long sdiv[kMaxStages];  // ceil(2^36 / span): q / span = (q * sdiv) >> 36
  int tw_len;
};

// q / d with m = ceil(2^36 / d): exact whenever q d <= 2^36, since m d - 2^36
// is below d.
__host__ __device__ __forceinline__ int fast_div(int q, unsigned long long m) {
  return (int)(((unsigned long long)q * m) >> 36);
}

// Layout of the FP32 Green transform: elements (complex) from one octant point to the
// next in z and, x fastest, in (y, x), and 16-byte pieces from one pair of components (xx
// xy | xz yy | yz zz) to the next.  The register z kernel copies columns whole and wants hz
// fastest; the shared-memory kernels read neighbouring columns at one hz, the components
// side by side (hz fastest cost them up to 10%: z pass of a 50x50x185 box 284 -> 315 us).
struct GhatLayout {
  int64_t sz, sxy;
  int piece;
};
inline GhatLayout ghat_f32_layout(bool z_fastest, int Hx, int Hy, int Hz) {
  if (z_fastest) return {2, 6 * (int64_t)Hz, Hz};
  return {6 * (int64_t)Hx * Hy, 6, 1};
}

// Everything a matvec kernel needs about one target's operator.
template <typename T> struct OpView {
  using C = cplx_t<T>;
  int nx, ny, nz;                 // box
  int Lx, Ly, Lz;                 // FFT grid
  int Hx, Hy, Hz;                 // octant sizes L/2 + 1
  int64_t nbox;                   // nx*ny*nz
  int chain;                      // host, see launch_chained: 0 -- ordinary launches; 1 --
                                  // the passes of a product are chained; 3 -- so they are,
                                  // within a solve; 2 -- and its first pass, which a
                                  // kernel precedes
  int src_z0, src_z1;             // planes outside [src_z0, src_z1) of the input hold zeros:
                                  // the FP64 x and y passes leave them out
  const uint8_t* comp;            // [nbox] 0 = vacant, else composition 1..ncomp
  const C* ghat;                  // octant, already divided by Lx*Ly*Lz: [Hz][Hy][Hx][6],
                                  // FP32 as gl says
  const C* ainv;                  // [R][ncomp+1][3] alpha^{-1} per RHS and lattice axis
                                  // (the polarizability tensor's diagonal), entry 0 unused
  int ncomp1;                     // ncomp + 1
  const C* twx; const C* twy; const C* twz;
  const int* kx_at; const int* ky_at; const int* kz_at;  // frequency held at each
                                                          // digit-reversed position
  const int* ypos_at;             // position holding each y frequency (inverse of ky_at)
  const float4* twz_reg;          // z twiddles of the register kernel (FP32), or null
  const float4* twx_reg;          // x, y twiddles of the register passes (FP32), or null
  const float4* twy_reg;
  const C* tw_wide;               // z twiddles of the 16-byte register kernel, or null
  const float2* twz_pair;         // z twiddles of the column-pair kernel's plan (FP32), or null
  int* zerr;                      // set to 1 by a kernel whose bounded wait on a copy ran out
  unsigned long long div_nx, div_ny, div_nz, div_Lx;     // fast_div magics
  AxisPlan px, py, pz;
  GhatLayout gl;
};

// ---- launches that overlap their predecessor's end ---------------------------
// The passes of a product and the vector updates between them form one chain of short
// kernels (8 to 50 us on boxes of up to 50^3 sites), each of which reads what the one
// before it wrote.  launch_chained lets a kernel's CTAs become resident as soon as the
// last CTAs of its predecessor have started: launch latency, index arithmetic and loads
// of constant tables pass beside the predecessor's end.  The kernel calls
//   chain_next()  first: its own successor may be set up;
//   chain_wait()  in every CTA, before it touches anything a kernel of the chain
//                 writes (and before it returns: a kernel that ends without waiting
//                 would end before its predecessor has);
//   chained(p)    on each pointer to such memory: the compiler knows nothing of p from
//                 before the wait, so no load through it is moved above the wait or
//                 takes the read-only path.
// Ordinary and chained, one GB300: an FP32 product of 16^3 sites 38.5 and 32 us, of
// 75x60x50 77 and 70; in the graph of a solve, whose launches are closer together, 64^3
// 18.05 and 17.5 ms, 36x41x36 6.09 and 5.88.  The FP64 and double-float passes are not
// chained: the 16^3 FP64 solve took 1.56 ms ordinary and 1.73 chained (their CTAs are
// few and large, and those that wait hold the registers of those that work).  Nor is
// the inverse y pass within a solve: behind a z pass of several waves its CTAs cost up
// to 9% of an iteration (100x75x135 1136 us with it chained, 1035 ordinary, 1044 with no
// kernel chained; 128^3 1953, 1817, 1830; 96^3 900, 854, 857; 24^3 74.2, 72.7, 72.1; the
// most it gave was 0.8%, 36x41x36).  A product on its own, launched kernel by kernel,
// gains from it (16^3 23.6 against 26.6 us, 72^3 85.5 against 89.3).
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class P> __device__ __forceinline__ P* chained(P* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
// A view for the products of a solve, and for those inside an iteration, which a kernel
// precedes.
template <typename V> V within_solve(V op) {
  if (op.chain) op.chain = 3;
  return op;
}
template <typename V> V follows_kernel(V op) {
  if (op.chain) op.chain = 2;
  return op;
}
// on: false -- an ordinary launch (profiled solves record an event between the passes)
template <class... K, class... A>
inline void launch_chained(bool on, void (*kernel)(K...), dim3 grid, int threads, size_t smem,
                           cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = on ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, K(args)...);
}

// ---- asynchronous global -> shared copies (cp.async) ------------------------
__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
// BYTES = 4, 8 or 16; both addresses aligned to BYTES
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst_smem, const void* src_gmem) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst_smem)),
                 "l"(src_gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_addr(dst_smem)),
                 "l"(src_gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

}  // namespace dda
