// FFT-convolution matvec with FP64 box vectors and double-float FFT passes:
// the refinement's residual operator.  Kernels: matvec_impl.cuh.
#include "matvec_impl.cuh"
#include "zpass_wide.cuh"

namespace dda {

// the register z pass, instantiated in zpass_wide_*.cu
bool z_wide_plan(int Lz, int nz, int* R1, int* R2) {
  if (Lz % 2) return false;
  switch (Lz / 2) {
#define DDA_ZWIDE_PLAN(A, B) \
  case (A) * (B):            \
    if (R1) *R1 = (A);       \
    if (R2) *R2 = (B);       \
    return nz <= (A) * (B) && nz >= ((A) - 1) * (B);
    DDA_ZWIDE_ALL(DDA_ZWIDE_PLAN)
#undef DDA_ZWIDE_PLAN
  }
  return false;
}

template <typename T>
bool launch_z_wide_any(bool cross, const OpView<T>& op, int R, cplx_t<T>* buf, const int* active,
                       cudaStream_t st) {
  if (!op.tw_wide) return false;
#define DDA_ZWIDE_TRY(P) launch_z_wide_part##P(cross, op, R, buf, active, st)
  return DDA_ZWIDE_TRY(0) || DDA_ZWIDE_TRY(1) || DDA_ZWIDE_TRY(2) || DDA_ZWIDE_TRY(3) ||
         DDA_ZWIDE_TRY(4) || DDA_ZWIDE_TRY(5);
#undef DDA_ZWIDE_TRY
}
template bool launch_z_wide_any<df64>(bool, const OpView<df64>&, int, df64c*, const int*,
                                      cudaStream_t);
template bool launch_z_wide_any<double>(bool, const OpView<double>&, int, double2*, const int*,
                                        cudaStream_t);

cudaError_t launch_matvec_df(const OpView<df64>& op, const MatvecLaunch& L, int R,
                             const double2* x, double2* y, df64c* scratch, const int* active,
                             cudaStream_t st, const cudaEvent_t* ev) {
  // the x and y schedule of the FP64 passes (same element size); the z pass is the
  // register kernel where the length has a plan (launch_z_pass), and otherwise has
  // one variant here: 4 columns, Ghat read from global memory
  MatvecLaunch Ld = L;
  Ld.z_tile = 4;
  Ld.z_gs = false;
  Ld.z_ps = 3 * 4 + 1;
  Ld.z_smem = ((size_t)op.Lz * Ld.z_ps * sizeof(df64c) + 15) & ~(size_t)15;
  return matvec_passes<df64, XIN_PLAIN, XOUT_PLAIN>(op, Ld, R, x, y, scratch, active, st, ev,
                                                    XinArgs<df64>{}, nullptr, nullptr);
}

cudaError_t configure_matvec_kernels_df(int Lz) {
  const void* k[] = {(const void*)k_fft_x_fwd<df64, XIN_PLAIN>,
                     (const void*)k_fft_x_inv<df64, XOUT_PLAIN>,
                     (const void*)k_fft_y<df64, false>, (const void*)k_fft_y<df64, true>,
                     (const void*)k_fft_z_mul<df64, 4, false>};
  for (const void* f : k) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               200 * 1024);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  const int hz = Lz % 2 ? 0 : Lz / 2;
  ok(configure_z_wide_part0(hz)); ok(configure_z_wide_part1(hz)); ok(configure_z_wide_part2(hz));
  ok(configure_z_wide_part3(hz)); ok(configure_z_wide_part4(hz)); ok(configure_z_wide_part5(hz));
  return e;
}

}  // namespace dda
