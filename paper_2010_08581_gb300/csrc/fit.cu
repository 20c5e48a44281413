// Relative error ||TR(cores) - X||_F / ||X||_F (Sec. 5.1) of one problem: the right factors
// W^T of the mode split (fit_body.cuh), then partial sums of the squared residual and of
// ||X||^2 per CTA, reduced on the host in a fixed order.
#include "fit_tc.cuh"

namespace trk {
namespace {

template <typename T>
__global__ void __launch_bounds__(FNT) k_fit_right(FitArgs a, FitSplit f, T* __restrict__ WT) {
  __shared__ double chain[8][kMaxL];
  __shared__ double slice[8][kMaxL];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q = static_cast<int64_t>(blockIdx.x) * (FNT / 32) + warp;
  if (q >= f.cols) return;
  fit_right_warp(a, f, q, WT, chain[warp], slice[warp], lane);
}

template <typename T>
__global__ void __launch_bounds__(FNT) k_fit(FitArgs a, FitSplit f, const T* __restrict__ X,
                                             const T* __restrict__ WT,
                                             double* __restrict__ partial, int blocks) {
  extern __shared__ __align__(16) unsigned char fit_smem_raw[];
  __shared__ double chain[8][kMaxL];
  __shared__ double slice[8][kMaxL];
  __shared__ double red[2 * (FNT / 32)];
  const int64_t units = fit_units(f);
  double se = 0.0, sx = 0.0;
  fit_units_f64(a, f, X, WT, units * blockIdx.x / gridDim.x, units * (blockIdx.x + 1) / gridDim.x,
                fit_smem_raw, chain, slice, se, sx);
  fit_block_reduce(se, sx, red);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = se;
    partial[blocks + blockIdx.x] = sx;
  }
}

// FP32 slice tables (fit_tc.cuh), one warp per slice.
__global__ void __launch_bounds__(256) k_fit_tables(FitArgs a, FitSplit f,
                                                    float* __restrict__ out) {
  grid_wait();
  fit_tables_warps(a, f, out, (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5,
                   static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5));
}

template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps) k_fit_right_tc(FitArgs a, FitSplit f, const float* tables,
                                                              unsigned char* __restrict__ WS) {
  grid_wait();
  __shared__ __align__(16) float P[32 * 256];
  __shared__ float G[kWarps * kMaxL];
  fit_right_tc_job<kWarps, 1>(a, f, blockIdx.x, fit_tc_right(a, f, tables), WS, P, G);
}

__global__ void __launch_bounds__(FT_NT, 1) k_fit_tc(FitArgs a, FitSplit f, FitTcPlan pl,
                                                     const float* __restrict__ X,
                                                     const unsigned char* __restrict__ WS,
                                                     const float* tables,
                                                     double* __restrict__ partial, int blocks,
                                                     unsigned* err) {
  grid_wait();
  extern __shared__ __align__(128) unsigned char fit_tc_raw[];
  __shared__ double red[2 * FT_EW];
  __shared__ FitTcShared sh;
  double se = 0.0, sx = 0.0;
  fit_tc_units(a, f, pl, X, WS, fit_tc_left(a, f, tables), pl.units * blockIdx.x / gridDim.x,
               pl.units * (blockIdx.x + 1) / gridDim.x, fit_tc_raw, sh, err, se, sx);
  fit_tc_reduce(se, sx, red);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = se;
    partial[blocks + blockIdx.x] = sx;
  }
}

FitSplit split_of(const FitArgs& a) { return fit_split(a.N, a.dims, a.ranks); }

size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

// CTAs of k_fit<double> per SM (at most 3) by their shared memory: of 228 KB, 1 KB of each CTA's is
// the system's.
int fit_resident(int K) {
  const size_t cta = fit_smem_bytes(K) + (2 * 8 * kMaxL + 2 * (FNT / 32)) * sizeof(double) + 1024;
  const int n = static_cast<int>(228 * 1024 / cta);
  return n < 1 ? 1 : (n > 3 ? 3 : n);
}

template <typename T>
void fit_f64(const FitArgs& a, const FitSplit& f, const void* X, char* wt, double* partial,
             int blocks, cudaStream_t st) {
  const unsigned rb = static_cast<unsigned>((f.cols + FNT / 32 - 1) / (FNT / 32));
  T* WT = reinterpret_cast<T*>(wt);
  // (not as a chain: CTAs placed while the right factors' are still there are spread unevenly, 33 x 37 x
  // 41, rank 9: 87 us a call, 129 so)
  k_fit_right<T><<<rb, FNT, 0, st>>>(a, f, WT);
  k_fit<T><<<blocks, FNT, fit_smem_bytes(f.K), st>>>(a, f, static_cast<const T*>(X), WT, partial,
                                                     blocks);
}

// FP32 X on the FP64 form (fit_body.cuh).
bool fit_plain(const FitSplit& f, bool x_f64, FitRoom room) {
  return room == kFitLeast && !x_f64 && f.K > FKPlain;
}

}  // namespace

size_t fit_workspace(const FitArgs& a, bool x_f64, FitRoom room, int* blocks, size_t* table_bytes) {
  const FitSplit f = split_of(a);
  if (room != kFitRoomy) {   // the room of one CTA per row block
    const bool plain = fit_plain(f, x_f64, room);
    const int64_t edge = x_f64 ? FL : (plain ? 2 * FL : FT_Q);
    const int64_t most = x_f64 || plain ? 4 * sm_count() : sm_count();
    const int64_t rb = (f.rows + edge - 1) / edge;
    *blocks = static_cast<int>(rb < most ? rb : most);
    *table_bytes = 0;
    return round256(static_cast<size_t>(2 * *blocks) * sizeof(double)) +
           (x_f64 || plain ? static_cast<size_t>(f.cols) * f.K * (x_f64 ? 8 : 4)
                           : fit_tc_right_bytes(f));
  }
  int64_t b = x_f64 ? fit_units(f) : fit_tc_plan(a, f).units;
  // the tensor-core form: one CTA per SM. FP64: as many as are resident, three per SM at most (one
  // more is a round of its own: 100000 x 3 x 3, rank 3, with four: 148 us a call, now 132; 7 x 9000 x 11,
  // rank 11, two resident, with three: 940 us a call, now 742), but with a chain of three or more
  // modes a CTA's own V costs more than a tile of products, so the CTAs are then whole row
  // blocks, or equal parts of them while SMs are left over (4^10, rank 10: 279 us with 128 row
  // blocks on as many CTAs, 352 us with 304 CTAs that form V twice each)
  int64_t cap = x_f64 ? fit_resident(f.K) * sm_count() : sm_count();
  if (x_f64 && f.s > 2) {
    const int64_t rb = (f.rows + FL - 1) / FL;
    const int64_t whole = rb * (sm_count() / rb > 1 ? sm_count() / rb : 1);
    cap = whole < cap ? whole : cap;
  }
  // (up to four units per SM one each: the ones beyond the resident CTAs run as others leave; 7 x 900 x 11,
  // rank 11: 310 units, 304 resident: 183 us a call, 210 with 304 CTAs; 40 x 40 x 380, rank 5: 600 units,
  // 456 resident: 110 and 123)
  if (b > cap && !(x_f64 && f.s <= 2 && b <= 4 * sm_count())) b = cap;
  *blocks = static_cast<int>(b);
  const size_t right = x_f64 ? static_cast<size_t>(f.cols) * f.K * 8 : fit_tc_right_bytes(f);
  *table_bytes = x_f64 || !fit_tc_tables_fit(a, f)
                     ? 0 : static_cast<size_t>(fit_tc_tables_floats(a, f)) * sizeof(float);
  return round256(round256(static_cast<size_t>(2 * b) * sizeof(double)) + right);
}

cudaError_t launch_fit(const FitArgs& a, const void* X, bool x_f64, FitRoom room, void* ws,
                       int blocks, float* tables, unsigned* err, cudaStream_t st) {
  const FitSplit f = split_of(a);
  double* partial = static_cast<double*>(ws);
  char* wt = static_cast<char*>(ws) + round256(static_cast<size_t>(2 * blocks) * sizeof(double));
  if (x_f64) {
    fit_f64<double>(a, f, X, wt, partial, blocks, st);
  } else if (fit_plain(f, x_f64, room)) {
    fit_f64<float>(a, f, X, wt, partial, blocks, st);
  } else {
    const FitTcPlan pl = fit_tc_plan(a, f);
    unsigned char* WS = reinterpret_cast<unsigned char*>(wt);
    if (tables) {
      const int64_t n = ((f.s > 1 ? a.dims[f.s - 1] : 0) + (f.s < a.N - 1 ? a.dims[a.N - 1] : 0) + 7) / 8;
      const int64_t tb = n < 8 * sm_count() ? n : 8 * sm_count();
      launch_pdl(k_fit_tables, static_cast<unsigned>(tb), 256, 0, st, a, f, tables);
    }
    const int jobs = fit_right_jobs(pl.tiles, pl.ks, FT_RW);
    if (f.s < a.N - 1 && a.dims[a.N - 1] < 8 && jobs <= 2 * sm_count())
      launch_pdl(k_fit_right_tc<FT_RW>, jobs, 32 * FT_RW, 0, st, a, f, tables, WS);
    else
      launch_pdl(k_fit_right_tc<FT_RWS>, fit_right_jobs(pl.tiles, pl.ks, FT_RWS), 32 * FT_RWS, 0, st, a, f, tables,
                 WS);
    launch_pdl(k_fit_tc, blocks, FT_NT, kFitTcSmem, st, a, f, pl, static_cast<const float*>(X), WS, tables,
               partial, blocks, err);
  }
  return cudaGetLastError();
}

cudaError_t fit_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_fit<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(fit_smem_bytes(kMaxL)));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_fit<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(fit_smem_bytes(kMaxL)));
  if (e != cudaSuccess) return e;
  e = fit_tc_registers(reinterpret_cast<const void*>(k_fit_tc));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_fit_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kFitTcSmem));
}

cudaError_t cholesky_attributes();
cudaError_t trsm_attributes();
cudaError_t normal_eq_tc_attributes();
cudaError_t sample_chain_attributes();
cudaError_t batched_attributes();
cudaError_t jacobi_attributes();
cudaError_t solve_inv_attributes();
cudaError_t merge_attributes();
cudaError_t lev_precond_attributes();

cudaError_t init_kernel_attributes(const char** which) {
  cudaError_t e = cholesky_attributes();
  if (e != cudaSuccess) { *which = "cholesky"; return e; }
  e = trsm_attributes();
  if (e != cudaSuccess) { *which = "trsm"; return e; }
  e = normal_eq_tc_attributes();
  if (e != cudaSuccess) { *which = "normal_eq_tc"; return e; }
  e = sample_chain_attributes();
  if (e != cudaSuccess) { *which = "sample_chain"; return e; }
  e = batched_attributes();
  if (e != cudaSuccess) { *which = "batched"; return e; }
  e = jacobi_attributes();
  if (e != cudaSuccess) { *which = "jacobi"; return e; }
  e = solve_inv_attributes();
  if (e != cudaSuccess) { *which = "solve_inv"; return e; }
  e = merge_attributes();
  if (e != cudaSuccess) { *which = "merge"; return e; }
  e = lev_precond_attributes();
  if (e != cudaSuccess) { *which = "lev_precond"; return e; }
  e = fit_attributes();
  if (e != cudaSuccess) *which = "fit";
  return e;
}

}  // namespace trk
