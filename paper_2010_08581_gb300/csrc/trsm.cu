// Single-problem launches of the triangular solves (trsm_body.cuh), rows a1 and a6.
#include "trsm_body.cuh"

namespace trk {
namespace {

template <typename T, int NV, int VP, int PB>
__global__ void __launch_bounds__(TNT) k_trsm(int n, const double* __restrict__ invdiag,
                                              const int* __restrict__ info, int64_t nvec,
                                              const double* __restrict__ rhs, int64_t ld, int mode,
                                              const T* __restrict__ Limg,
                                              const float* __restrict__ Mimg, int Rl, int Rr,
                                              double* __restrict__ core_out,
                                              double* __restrict__ ell, CdfEpilogue ep) {
  grid_wait();
  extern __shared__ __align__(16) unsigned char trsm_smem[];
  subst_cta<T, NV, VP, PB>(trsm_smem, blockIdx.x, n, invdiag, info, nvec, rhs, ld, mode, Limg, Mimg,
                       Rl, Rr, core_out, ell, ep, gridDim.x);
}

template <typename T>
cudaError_t run(int n, const double* invdiag, const int* info, int64_t nvec, const double* rhs,
                int64_t ld, int mode, const T* Limg, const float* Mimg, int Rl, int Rr,
                double* core_out, double* ell, const CdfEpilogue& ep, cudaStream_t st) {
  // eight vectors a CTA, four while that leaves SMs without one; few: one CTA per SM at most
  const bool four = nvec <= 8 * static_cast<int64_t>(sm_count());
  const bool few = nvec <= 4 * static_cast<int64_t>(sm_count());
  const int nv = four ? 4 : 8;
  const unsigned blocks = static_cast<unsigned>((nvec + nv - 1) / nv);
  const size_t dyn = subst_smem<T>(n, nv, panel_cols<T>(few));
#define TRSM_GO(NV, VP, FEW)                                                                     \
  launch_pdl((k_trsm<T, NV, VP, panel_cols<T>(FEW)>), blocks, TNT, dyn, st, n, invdiag, info,     \
             nvec, rhs, ld, mode, Limg, Mimg, Rl, Rr, core_out, ell, ep)
#define TRSM_8(VP) TRSM_GO(8, VP, false)
#define TRSM_4(VP) TRSM_GO(4, (VP > 1 ? VP / 2 : 1), false)
#define TRSM_FEW(VP) TRSM_GO(4, (VP > 1 ? VP / 2 : 1), true)
  if (few) TRK_SUBST_DISPATCH(n, TRSM_FEW);
  else if (four) TRK_SUBST_DISPATCH(n, TRSM_4);
  else TRK_SUBST_DISPATCH(n, TRSM_8);
#undef TRSM_FEW
#undef TRSM_4
#undef TRSM_8
#undef TRSM_GO
  return cudaGetLastError();
}

template <typename T, int NV, int VP, int PB>
cudaError_t attr_one() {
  return cudaFuncSetAttribute(k_trsm<T, NV, VP, PB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(subst_smem<T>(kMaxL, NV, PB)));
}

template <typename T>
cudaError_t attr() {
  constexpr int PF = panel_cols<T>(true), PM = panel_cols<T>(false);
  cudaError_t e = attr_one<T, 4, 1, PF>();
  if (e == cudaSuccess) e = attr_one<T, 4, 2, PF>();
  if (e == cudaSuccess) e = attr_one<T, 4, 4, PF>();
  if (e == cudaSuccess) e = attr_one<T, 4, 1, PM>();
  if (e == cudaSuccess) e = attr_one<T, 4, 2, PM>();
  if (e == cudaSuccess) e = attr_one<T, 4, 4, PM>();
  if (e == cudaSuccess) e = attr_one<T, 8, 1, PM>();
  if (e == cudaSuccess) e = attr_one<T, 8, 2, PM>();
  if (e == cudaSuccess) e = attr_one<T, 8, 4, PM>();
  if (e == cudaSuccess) e = attr_one<T, 8, 8, PM>();
  return e;
}

}  // namespace

cudaError_t launch_trsm(int mode, bool f32, int n, const double* invdiag, const int* info,
                        int64_t nvec, const double* rhs, int64_t ld, int Rl, int Rr,
                        double* core_out, double* ell, cudaStream_t st, const void* Limg,
                        const float* Mimg, const CdfEpilogue* cdf) {
  if (nvec <= 0) return cudaSuccess;
  if (!Limg || (mode == 2 && (!f32 || !Mimg))) return cudaErrorInvalidValue;
  const CdfEpilogue ep = cdf ? *cdf : CdfEpilogue{};
  if (f32)
    return run<float>(n, invdiag, info, nvec, rhs, ld, mode, static_cast<const float*>(Limg), Mimg,
                      Rl, Rr, core_out, ell, ep, st);
  return run<double>(n, invdiag, info, nvec, rhs, ld, mode, static_cast<const double*>(Limg), Mimg,
                     Rl, Rr, core_out, ell, ep, st);
}

size_t trsm_image_bytes(int n, bool f32) {
  return ((static_cast<size_t>(n) * (n + 1) * (f32 ? 4 : 8) + 15) / 16) * 16;
}

cudaError_t trsm_attributes() {
  const cudaError_t e = attr<float>();
  return e == cudaSuccess ? attr<double>() : e;
}

}  // namespace trk
