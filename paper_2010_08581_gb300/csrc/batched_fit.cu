// Serving: the exact relative fit of every slot that completed a sweep (Sec. 5.1) and the
// stop rule of Sec. 4.1, for the batched slot table.
#include "batched_kern.cuh"
#include "fit_tc.cuh"

namespace trk {
namespace {

// ------------------------------------------------------------------------------------
// Serving: relative fit 1 - ||TR - X|| / ||X|| (Sec. 5.1) of every slot that completed a
// sweep in this tick, as kFitParts (or fewer) partial sums in a fixed order, then the stop
// rule (|fit_s - fit_{s-1}| < tol after two or more sweeps, or the sweep cap) and the step
// counters.
// ------------------------------------------------------------------------------------
// The slot's step is the last update of a sweep.
__device__ __forceinline__ bool fit_due(const BInst& d) {
  if (!d.slot) return false;
  const SlotState& s = *d.slot;
  return s.status == kSlotRunning && s.step >= 0 && s.step % d.N == d.N - 1;
}

// Partial sums of one slot's fit: one per CTA, at most kFitParts.
__device__ __forceinline__ int fit_parts(const FitArgs& fa, const FitSplit& f, bool f64_form) {
  const int64_t n = f64_form ? (fit_units(f) + 7) / 8 : fit_tc_parts(fit_tc_plan(fa, f));
  return n < kFitParts ? static_cast<int>(n) : kFitParts;
}

__device__ __forceinline__ void fit_args(const BInst& d, FitArgs& fa) {
  fa.N = d.N;
  for (int m = 0; m < d.N; ++m) {
    fa.core[m] = d.cores[m];
    fa.dims[m] = d.dims[m];
    fa.ranks[m] = d.ranks[m];
  }
}

// The FP32 slice tables of the left and right groups (fit_tc.cuh) live in the slot's fibre
// buffer, which no stage reads between the LS step and the next draws; they are skipped (null)
// where they would not fit (J smaller than about twice the largest L).
__device__ __forceinline__ float* fit_tables(const BInst& d, const FitArgs& fa, const FitSplit& f) {
  int64_t Imax = 0;
  for (int m = 0; m < fa.N; ++m) Imax = fa.dims[m] > Imax ? fa.dims[m] : Imax;
  const int64_t n = fit_tc_tables_floats(fa, f);
  return n > 0 && fit_tc_tables_fit(fa, f) && n <= d.J * Imax ? static_cast<float*>(d.Y) : nullptr;
}

constexpr int kFitRightCtas = 128;  // CTAs per slot forming the right factors

__global__ void __launch_bounds__(256) kb_fit_tables(const BInst* __restrict__ tab) {
  __shared__ FitArgs fa;
  const BInst& d = tab[blockIdx.x];
  if (!fit_due(d)) return;
  if (threadIdx.x == 0) fit_args(d, fa);
  __syncthreads();
  const FitSplit f = fit_split(fa.N, fa.dims, fa.ranks);
  float* out = fit_tables(d, fa, f);
  if (!out) return;
  fit_tables_warps(fa, f, out, (static_cast<int64_t>(blockIdx.y) * blockDim.x + threadIdx.x) >> 5,
                   static_cast<int64_t>(gridDim.y) * (blockDim.x >> 5));
}

// Right factors of the fit: e-major W^T for FP64 X ...
__global__ void __launch_bounds__(FNT) kb_fit_right(const BInst* __restrict__ tab) {
  __shared__ double chain[8][kMaxL];
  __shared__ double slice[8][kMaxL];
  __shared__ FitArgs fa;
  const BInst& d = tab[blockIdx.x];
  if (!fit_due(d)) return;
  if (threadIdx.x == 0) fit_args(d, fa);
  __syncthreads();
  const FitSplit f = fit_split(fa.N, fa.dims, fa.ranks);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t step = static_cast<int64_t>(gridDim.y) * (FNT / 32);
  double* WT = static_cast<double*>(d.fitw);
  for (int64_t q = static_cast<int64_t>(blockIdx.y) * (FNT / 32) + warp; q < f.cols; q += step)
    fit_right_warp(fa, f, q, WT, chain[warp], slice[warp], lane);
}

// ... or the split operand tiles of the tensor-core contraction.
__global__ void __launch_bounds__(32 * FT_RWS) kb_fit_right_tc(const BInst* __restrict__ tab) {
  __shared__ __align__(16) float P[32 * 256];   // 8 chains of kMaxL doubles in the FP64 form
  __shared__ float G[FT_RWS * kMaxL];
  __shared__ FitArgs fa;
  const BInst& d = tab[blockIdx.x];
  if (!fit_due(d)) return;
  if (threadIdx.x == 0) fit_args(d, fa);
  __syncthreads();
  const FitSplit f = fit_split(fa.N, fa.dims, fa.ranks);
  const float* table = fit_tc_right(fa, f, fit_tables(d, fa, f));
  if (d.fit_plain) {        // FP32 W^T for the FP64 form
    double (*chain)[kMaxL] = reinterpret_cast<double (*)[kMaxL]>(P);
    const int warp = threadIdx.x >> 5;
    for (int64_t q = static_cast<int64_t>(blockIdx.y) * FT_RWS + warp; q < f.cols; q += FT_RWS * gridDim.y)
      fit_right_warp(fa, f, q, static_cast<float*>(d.fitw), chain[warp], chain[4 + warp],
                     static_cast<int>(threadIdx.x & 31));
    return;
  }
  const int jobs = fit_right_jobs((f.cols + FT_Q - 1) / FT_Q, (f.K + FT_KS - 1) / FT_KS, 4 * FT_RWS);
  for (int j = blockIdx.y; j < jobs; j += gridDim.y) {
    fit_right_tc_job<FT_RWS, 4>(fa, f, j, table, static_cast<unsigned char*>(d.fitw), P, G);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(FNT) kb_fit(const BInst* __restrict__ tab) {
  extern __shared__ __align__(16) unsigned char fit_dyn[];
  __shared__ double chain[8][kMaxL];
  __shared__ double slice[8][kMaxL];
  __shared__ double red[2 * (FNT / 32)];
  __shared__ FitArgs fa;
  const BInst& d = tab[blockIdx.x];
  if (!fit_due(d)) return;
  if (threadIdx.x == 0) fit_args(d, fa);
  __syncthreads();
  const FitSplit f = fit_split(fa.N, fa.dims, fa.ranks);
  const int parts = fit_parts(fa, f, true);
  if (static_cast<int>(blockIdx.y) >= parts) return;
  const int64_t units = fit_units(f);
  double se = 0.0, sx = 0.0;
  fit_units_f64(fa, f, static_cast<const double*>(d.X), static_cast<const double*>(d.fitw),
                units * blockIdx.y / parts, units * (blockIdx.y + 1) / parts, fit_dyn, chain, slice,
                se, sx);
  fit_block_reduce(se, sx, red);
  if (threadIdx.x == 0) {
    d.fitp[blockIdx.y] = se;
    d.fitp[kFitParts + blockIdx.y] = sx;
  }
}

// Slots with FP32 X: the contraction on the tensor cores (fit_tc.cuh).
__global__ void __launch_bounds__(FT_NT, 1) kb_fit_tc(const BInst* __restrict__ tab,
                                                      unsigned* err) {
  extern __shared__ __align__(128) unsigned char fit_tc_dyn[];
  __shared__ double red[2 * FT_EW];
  __shared__ FitArgs fa;
  __shared__ FitTcShared sh;
  const BInst& d = tab[blockIdx.x];
  if (!fit_due(d)) return;
  if (threadIdx.x == 0) fit_args(d, fa);
  __syncthreads();
  const FitSplit f = fit_split(fa.N, fa.dims, fa.ranks);
  const FitTcPlan pl = fit_tc_plan(fa, f);
  const int parts = fit_parts(fa, f, d.fit_plain);
  if (static_cast<int>(blockIdx.y) >= parts) return;
  double se = 0.0, sx = 0.0;
  if (d.fit_plain) {        // admitted without room for the operand of W
    if (threadIdx.x >= FNT) return;
    double (*chain)[kMaxL] = reinterpret_cast<double (*)[kMaxL]>(fit_tc_dyn + fit_smem_bytes(f.K));
    const int64_t units = fit_units(f);
    fit_units_f64(fa, f, static_cast<const float*>(d.X), static_cast<const float*>(d.fitw),
                  units * blockIdx.y / parts, units * (blockIdx.y + 1) / parts, fit_tc_dyn, chain,
                  chain + FNT / 32, se, sx);
    fit_block_reduce(se, sx, red);
    if (threadIdx.x == 0) {
      d.fitp[blockIdx.y] = se;
      d.fitp[kFitParts + blockIdx.y] = sx;
    }
    return;
  }
  fit_tc_units(fa, f, pl, static_cast<const float*>(d.X),
               static_cast<const unsigned char*>(d.fitw), fit_tc_left(fa, f, fit_tables(d, fa, f)),
               pl.units * blockIdx.y / parts, pl.units * (blockIdx.y + 1) / parts, fit_tc_dyn, sh,
               err, se, sx);
  fit_tc_reduce(se, sx, red);
  if (threadIdx.x == 0) {
    d.fitp[blockIdx.y] = se;
    d.fitp[kFitParts + blockIdx.y] = sx;
  }
}

__global__ void __launch_bounds__(128) kb_advance(const BInst* __restrict__ tab, int count,
                                                  int xf64) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const BInst& d = tab[i];
  if (!d.slot) return;
  SlotState& s = *d.slot;
  if (s.status != kSlotRunning) return;
  const int t = s.step;
  if (t >= 0 && *d.info != 0) s.singular += 1;
  if (fit_due(d)) {
    FitArgs fa;
    fit_args(d, fa);
    const int parts = fit_parts(fa, fit_split(d.N, d.dims, d.ranks), xf64 != 0 || d.fit_plain);
    double se = 0.0, sx = 0.0;
    for (int q = 0; q < parts; ++q) {
      se += d.fitp[q];
      sx += d.fitp[kFitParts + q];
    }
    const double rel = sx > 0.0 ? sqrt(se / sx) : (se > 0.0 ? INFINITY : 0.0);
    const double fit = 1.0 - rel;
    const int sw = s.sweeps + 1;
    s.sweeps = sw;
    s.fit_prev = s.fit;
    s.fit = fit;
    if (sw <= kMaxServedSweeps) d.hist[sw - 1] = fit;
    if (!isfinite(fit)) s.status = kSlotFailed;
    else if (sw >= 2 && fabs(fit - s.fit_prev) < s.tol) s.status = kSlotConverged;
    else if (sw >= s.max_sweeps) s.status = kSlotCapped;
  }
  s.step = t + 1;
}

}  // namespace

cudaError_t bl_fit(const BLaunch& b, unsigned* err, cudaStream_t st) {
  dim3 rgrid(b.count, kFitRightCtas);
  dim3 grid(b.count, kFitParts);
  if (b.xf64) {
    kb_fit_right<<<rgrid, FNT, 0, st>>>(b.tab);
    kb_fit<<<grid, FNT, fit_smem_bytes(b.Lmax), st>>>(b.tab);
  } else {
    kb_fit_tables<<<dim3(b.count, 16), 256, 0, st>>>(b.tab);
    kb_fit_right_tc<<<rgrid, 32 * FT_RWS, 0, st>>>(b.tab);
    kb_fit_tc<<<grid, FT_NT, kFitTcSmem, st>>>(b.tab, err);
  }
  return cudaGetLastError();
}

cudaError_t bl_advance(const BLaunch& b, cudaStream_t st) {
  kb_advance<<<(b.count + 127) / 128, 128, 0, st>>>(b.tab, b.count, b.xf64 ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t batched_fit_attributes() {
  cudaError_t e = cudaFuncSetAttribute(kb_fit, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(fit_smem_bytes(kMaxL)));
  if (e != cudaSuccess) return e;
  e = fit_tc_registers(reinterpret_cast<const void*>(kb_fit_tc));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kb_fit_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kFitTcSmem));
}

}  // namespace trk
