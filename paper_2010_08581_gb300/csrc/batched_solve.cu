// Batched triangular solves (trsm_body.cuh): the LS solves of Alg. 2 per instance, FP32 with one
// refinement step (mixed path) or FP64, and the leverage rows with the fused p / CDF step.
#include "batched_kern.cuh"
#include "trsm_body.cuh"

namespace trk {
namespace {

constexpr int BNV = 8;              // vectors per CTA
// Columns per panel: in FP64 and up to 64 unknowns 8, so that a warp solves the diagonal blocks of
// four vectors at once: with many CTAs per SM the FP64 pipe is the bound, where a warp's instruction
// takes 16 clocks however few lanes matter (rows of 512 problems: 250 us with 16 columns, 227 with
// 8). Beyond, where a few large problems have the SMs to themselves, fewer panels count.
template <typename T>
constexpr int batch_cols(int vp) { return sizeof(T) == 4 ? 32 : (vp <= 2 ? 8 : 16); }

template <typename T>
__device__ __forceinline__ void subst_any(unsigned char* sm, int64_t cta, int n,
                                          const double* invdiag, const int* info, int64_t nvec,
                                          const double* rhs, int64_t ld, int mode, const T* Limg,
                                          const float* Mimg, int Rl, int Rr, double* core_out,
                                          double* ell, const CdfEpilogue& ep, int nctas) {
#define SUBST_GO(VP)                                                                          \
  subst_cta<T, BNV, VP, batch_cols<T>(VP)>(sm, cta, n, invdiag, info, nvec, rhs, ld, mode, Limg, Mimg, Rl, Rr,   \
                        core_out, ell, ep, nctas)
  TRK_SUBST_DISPATCH(n, SUBST_GO);
#undef SUBST_GO
}

// (five CTAs per SM: the chains are latency; 512 problems: 269 -> 262 us, the rows 226 -> 215)
template <typename T>
__global__ void __launch_bounds__(TNT, 5) kb_solve(const BInst* __restrict__ tab, int step) {
  extern __shared__ __align__(16) unsigned char sm[];
  const BInst& d = tab[blockIdx.x];
  const Cur cu = current(d, step, 0, false);
  if (!cu.active) return;
  const int nctas = static_cast<int>((cu.I + BNV - 1) / BNV);
  if (static_cast<int>(blockIdx.y) >= nctas) return;
  const CdfEpilogue none{};
  subst_any<T>(sm, blockIdx.y, cu.L, d.invdiag, d.info, cu.I, d.BT, cu.L, sizeof(T) == 4 ? 2 : 1,
               static_cast<const T*>(d.limg), d.mimg, cu.Rl, cu.Rr, d.cores[cu.n], nullptr, none,
               nctas);
}

__global__ void __launch_bounds__(TNT, 5) kb_rows(const BInst* __restrict__ tab, int step, int init_k,
                                               unsigned* err, int from_core) {
  extern __shared__ __align__(16) unsigned char sm[];
  const BInst& d = tab[blockIdx.x];
  const Cur cu = current(d, step, init_k, true);
  if (!cu.active) return;
  const bool tall = cu.I >= cu.L;
  const int nctas = static_cast<int>((cu.I + BNV - 1) / BNV);
  if (static_cast<int>(blockIdx.y) >= nctas) return;
  const double* rhs = tall ? ((cu.init || from_core) ? d.cores[cu.n] : d.BT) : d.L1row;
  const CdfEpilogue ep{d.counter, d.p[cu.n], d.cdf[cu.n], cu.init ? nullptr : d.info, err};
  subst_any<double>(sm, blockIdx.y, tall ? cu.L : static_cast<int>(cu.I), tall ? d.inv1 : d.inv2,
                    nullptr, cu.I, rhs, tall ? cu.L : cu.I, 0, tall ? d.img1 : d.img2, nullptr, 1, 1,
                    nullptr, d.ell, ep, nctas);
}

template <typename T>
size_t smem(int n) { return subst_smem<T>(n, BNV, batch_cols<T>(8)); }
unsigned ctas(int64_t I) { return static_cast<unsigned>((I + BNV - 1) / BNV); }

}  // namespace

cudaError_t bl_solve(const BLaunch& b, int step, cudaStream_t st) {
  const dim3 grid(b.count, ctas(b.Imax));
  if (b.f64) kb_solve<double><<<grid, TNT, smem<double>(b.Lmax), st>>>(b.tab, step);
  else kb_solve<float><<<grid, TNT, smem<float>(b.Lmax), st>>>(b.tab, step);
  return cudaGetLastError();
}

cudaError_t bl_leverage_rows(const BLaunch& b, int step, int init_k, unsigned* err,
                             cudaStream_t st) {
  const int nmax = b.n1max > b.n2max ? b.n1max : b.n2max;
  kb_rows<<<dim3(b.count, ctas(b.Imax)), TNT, smem<double>(nmax), st>>>(
      b.tab, step, init_k, err, b.ls_mode == 1 ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t batched_solve_attributes() {
  const auto a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(kb_solve<float>, a, static_cast<int>(smem<float>(kMaxL)));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kb_solve<double>, a, static_cast<int>(smem<double>(kMaxL)));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kb_rows, a, static_cast<int>(smem<double>(kMaxL)));
  return e;
}

}  // namespace trk
