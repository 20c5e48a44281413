// Relative-error partial sums ||TR(cores) - X||_F^2 and ||X||_F^2 (Sec. 4.1, Sec. 5.1)
// without forming TR(cores), shared by the single-problem kernels and the served fit.
//
// The modes are split at s (1 <= s <= N-1): X is viewed as a rows x cols matrix with
// rows = prod_{m<s} I_m and cols = prod_{m>=s} I_m (row-major X). By eq. 1,
//   TR(p, q) = trace(P_left(p) P_right(q)),
//   P_left(p)  = G^(0)(:, i_0, :) ... G^(s-1)(:, i_{s-1}, :)    (R_{N-1} x R_{s-1}),
//   P_right(q) = G^(s)(:, i_s, :) ... G^(N-1)(:, i_{N-1}, :)    (R_{s-1} x R_{N-1}),
// so TR(p, q) = sum_e V_p[e] W_q[e] over e = b * R_{N-1} + a with V_p[e] = P_left[a][b] and
// W_q[e] = P_right[b][a]: one dense contraction with K = R_{N-1} R_{s-1} <= 256.
//
// The split is chosen so that cols is large enough to amortise the row chains while the right
// factors stay small (fit_split). FP32 X is evaluated on the tensor cores (fit_tc.cuh). This
// file holds the split and the FP64 form: W is formed once per evaluation (fit_right_warp,
// e-major: W^T[e][q]) and V per block of FL rows in shared memory; each thread computes a
// 2 x 2 register tile of TR from two vector loads per e. FP32 X with K > 128 takes it too where a
// budget or an arena has no room for the tensor cores' operand of W (two parts of every entry, in
// whole tiles of 128 columns and 32 terms) but has room for FP32 W^T, half as large: such a call is
// slow rather than refused.
//
// The work is cut into units (row block, column tile), row block by row block, and every CTA
// takes one contiguous range of them, forming V again where its range enters a row block. A
// cube whose first mode alone is the left group has few row blocks (100^3: 4) and thousands of
// columns; with one CTA per row block it ran on 4 SMs (2556 us at 100^3, rank 5), with the
// units spread (105 us) it is bound by the FP64 pipe (2 fused multiply-adds per clock and SM).
#pragma once

#include "common.cuh"

namespace trk {

constexpr int FNT = 256;                       // threads of a fit CTA
constexpr int64_t kFitMinCols = 256;           // grow cols (move s left) up to this
constexpr int64_t kFitMaxRight = 1ll << 22;    // max elements of W^T (cols * K)

constexpr int FKPlain = 128;                   // FP32 X: the longest K without that form
constexpr int FL = 32, FI = 32;                // rows and columns of an FP64 tile
constexpr int FMI = 2, FMJ = 2;                // outputs per thread

struct FitSplit {
  int s;          // first mode of the right group
  int K;          // R_{N-1} * R_{s-1}
  int64_t rows, cols;
};

__host__ __device__ inline FitSplit fit_split(int N, const int64_t* dims, const int* ranks) {
  FitSplit f;
  f.s = N - 1;
  f.cols = dims[N - 1];
  while (f.s > 1 && f.cols < kFitMinCols) {
    const int64_t c2 = f.cols * dims[f.s - 1];
    const int64_t k2 = static_cast<int64_t>(ranks[N - 1]) * ranks[f.s - 2];
    if (c2 * k2 > kFitMaxRight) break;
    f.s -= 1;
    f.cols = c2;
  }
  f.rows = 1;
  for (int m = 0; m < f.s; ++m) f.rows *= dims[m];
  f.K = ranks[N - 1] * ranks[f.s - 1];
  return f;
}

// Dynamic shared memory of an FP64 fit CTA for contraction length K.
__host__ __device__ constexpr size_t fit_smem_bytes(int K) {
  return static_cast<size_t>(K) * (FL + FI) * sizeof(double);
}

// Units of an FP64 evaluation.
__host__ __device__ inline int64_t fit_units(const FitSplit& f) {
  return ((f.rows + FL - 1) / FL) * ((f.cols + FI - 1) / FI);
}

// Product of the lateral slices of modes m0..m1-1 at indices ii[m] into S (row-major
// R_{m0-1} x R_{m1-1}), one warp; G is per-warp scratch. Returns the column count.
__device__ __forceinline__ int warp_slice_product(const FitArgs& a, int m0, int m1,
                                                  const int64_t* ii, double* S, double* G,
                                                  int lane) {
  const int N = a.N;
  int rows = a.ranks[(m0 - 1 + N) % N], cols = a.ranks[m0];
  {
    const double* src = a.core[m0] + ii[m0] * rows * cols;
    for (int e = lane; e < rows * cols; e += 32) S[e] = src[e];
  }
  for (int m = m0 + 1; m < m1; ++m) {
    const int rr = a.ranks[m];
    const double* src = a.core[m] + ii[m] * cols * rr;
    for (int e = lane; e < cols * rr; e += 32) G[e] = src[e];
    __syncwarp();
    double acc[kMaxL / 32];
#pragma unroll
    for (int q = 0; q < kMaxL / 32; ++q) {
      const int e = lane + 32 * q;
      double s = 0.0;
      if (e < rows * rr) {
        const int r = e / rr, c = e - r * rr;
        for (int t = 0; t < cols; ++t) s += S[r * cols + t] * G[t * rr + c];
      }
      acc[q] = s;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kMaxL / 32; ++q) {
      const int e = lane + 32 * q;
      if (e < rows * rr) S[e] = acc[q];
    }
    __syncwarp();
    cols = rr;
  }
  return cols;
}

// W^T[e][q] = P_right(q)[b][a] (e = b * R_{N-1} + a: the row-major index of P_right) for
// column q, one warp; S and G are per-warp scratch of kMaxL elements.
template <typename T>
__device__ __forceinline__ void fit_right_warp(const FitArgs& a, const FitSplit& f, int64_t q,
                                               T* __restrict__ WT, double* S, double* G, int lane) {
  const int N = a.N;
  int64_t ii[kMaxModes];
  int64_t rem = q;
  for (int m = N - 1; m >= f.s; --m) { ii[m] = rem % a.dims[m]; rem /= a.dims[m]; }
  warp_slice_product(a, f.s, N, ii, S, G, lane);
  __syncwarp();
  for (int e = lane; e < f.K; e += 32) WT[e * f.cols + q] = static_cast<T>(S[e]);
  __syncwarp();
}

// Barrier of the first FNT threads of a CTA.
__device__ __forceinline__ void fit_sync() {
  asm volatile("bar.sync 2, %0;" :: "n"(FNT) : "memory");
}

// V_p[e] (e = b * R_{N-1} + a, V_p[e] = P_left(p)[a][b]) for the rows p0 .. p0 + nb - 1 of a
// block and the entries e0 <= e < e1, handed to put(ll, e, value) (rows past the end give
// zeros). The first FNT threads of the CTA call it; it ends with their barrier.
//
// Rows p = pre * J + last (J = I_{s-1}) share the prefix G^(0) .. G^(s-2) of their slice
// chain, and consecutive rows mostly share it: each distinct prefix of the block is formed
// once by one warp (into chain[w]), and every (row, b) item then finishes its column b of
// P_left = prefix * G^(s-1)(:, last, :) in registers. The products and their summation order
// are those of a per-row chain, so V is the same. Blocks with more than 8 prefixes (J < 16)
// form every row's chain with one warp.
template <typename Put>
__device__ void build_left(const FitArgs& a, const FitSplit& f, int64_t p0, int nb, int e0,
                           int e1, double (*chain)[kMaxL], double (*slice)[kMaxL], Put put) {
  const int N = a.N, s = f.s;
  const int K = e1 < f.K ? e1 : f.K;   // entries K .. e1 - 1 are the caller's padding
  const int Rlast = a.ranks[N - 1], Rs = a.ranks[s - 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t rows = f.rows;
  const int64_t pend = (p0 + nb < rows) ? p0 + nb : rows;
  if (s == 1) {   // P_left(p) is the slice G^(0)(:, p, :) itself
    const int w = K - e0;
    for (int it = tid; it < nb * w; it += FNT) {
      const int ll = it / w, e = e0 + (it - ll * w);
      const int64_t p = p0 + ll;
      const int b = e / Rlast, aa = e - b * Rlast;
      put(ll, e, p < rows ? a.core[0][(p * Rlast + aa) * Rs + b] : 0.0);
    }
    fit_sync();
    return;
  }
  const int64_t J = a.dims[s - 1];
  const int64_t pre_lo = p0 / J;
  const int npre = pend > p0 ? static_cast<int>((pend - 1) / J - pre_lo + 1) : 0;
  if (npre > FNT / 32) {
    // many short prefixes: one warp per row forms the whole chain
    for (int ll = warp; ll < nb; ll += FNT / 32) {
      const int64_t p = p0 + ll;
      if (p >= rows) {
        for (int e = e0 + lane; e < K; e += 32) put(ll, e, 0.0);
        continue;
      }
      int64_t ii[kMaxModes];
      int64_t rem = p;
      for (int m = s - 1; m >= 0; --m) { ii[m] = rem % a.dims[m]; rem /= a.dims[m]; }
      double* S = chain[warp];
      const int rs = warp_slice_product(a, 0, s, ii, S, slice[warp], lane);
      __syncwarp();
      for (int e = e0 + lane; e < K; e += 32) {
        const int b = e / Rlast, aa = e - b * Rlast;
        put(ll, e, S[aa * rs + b]);
      }
      __syncwarp();
    }
    fit_sync();
    return;
  }
  const int Rm = a.ranks[s - 2];   // the rank between the prefix and G^(s-1)
  if (warp < npre) {
    int64_t ii[kMaxModes];
    int64_t rem = pre_lo + warp;
    for (int m = s - 2; m >= 0; --m) { ii[m] = rem % a.dims[m]; rem /= a.dims[m]; }
    warp_slice_product(a, 0, s - 1, ii, chain[warp], slice[warp], lane);   // Rlast x Rm
  }
  fit_sync();
  const double* Gs = a.core[s - 1];
  // columns b whose entries b * Rlast .. b * Rlast + Rlast - 1 meet [e0, K)
  const int b0 = e0 / Rlast, b1 = (K + Rlast - 1) / Rlast;
  const int nbc = b1 - b0;
  for (int it = tid; it < nb * nbc; it += FNT) {
    const int ll = it / nbc, b = b0 + (it - ll * nbc);
    const int64_t p = p0 + ll;
    const int a0 = e0 > b * Rlast ? e0 - b * Rlast : 0;
    const int a1 = K < (b + 1) * Rlast ? K - b * Rlast : Rlast;
    if (p >= rows) {
      for (int aa = a0; aa < a1; ++aa) put(ll, b * Rlast + aa, 0.0);
      continue;
    }
    const int64_t pre = p / J, last = p - pre * J;
    const double* P = chain[pre - pre_lo];
    const double* g = Gs + last * Rm * Rs + b;   // column b of G^(s-1)(:, last, :)
    double gc[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) gc[c] = c < Rm ? g[c * Rs] : 0.0;
    for (int aa = a0; aa < a1; ++aa) {
      const double* pr = P + aa * Rm;
      double acc = 0.0;
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (c < Rm) acc += pr[c] * gc[c];
      put(ll, b * Rlast + aa, acc);
    }
  }
  fit_sync();
}

// Accumulates the squared residual (se) and ||X||^2 (sx) over the units lo .. hi - 1 (unit =
// row block * column tiles + tile). The first FNT threads of the CTA call it. `chain` and `slice`
// are per-warp scratch of kMaxL elements (8 warps); `dyn` holds fit_smem_bytes(f.K).
template <typename T>
__device__ inline void fit_units_f64(const FitArgs& a, const FitSplit& f, const T* __restrict__ X,
                                     const T* __restrict__ WT, int64_t lo, int64_t hi,
                                     unsigned char* dyn, double (*chain)[kMaxL],
                                     double (*slice)[kMaxL], double& se, double& sx) {
  constexpr int TX = FI / FMJ;   // threads along the columns (16)
  static_assert((FL / FMI) * (FI / FMJ) == FNT, "one register tile per thread");
  static_assert(FL / FMI == 16, "16 swizzled groups per row of V^T");
  // Row e of V^T stores its 16 groups of FMI entries in the order g ^ (e & 15): the per-row
  // column writes of the chain phase spread over the banks, each group stays contiguous.
  auto vpos = [](int e, int ll) { return e * FL + (((ll / FMI) ^ (e & 15)) * FMI) + ll % FMI; };
  const int K = f.K;
  double* Vt = reinterpret_cast<double*>(dyn);   // [K][FL]
  double* Qt = Vt + K * FL;                      // [K][FI]
  const int64_t rows = f.rows, cols = f.cols, tiles = (cols + FI - 1) / FI;
  const int ty = threadIdx.x / TX, tx = threadIdx.x % TX;
  for (int64_t u = lo; u < hi; ++u) {
    const int64_t p0 = (u / tiles) * FL;
    if (u == lo || u % tiles == 0)   // 1. V^T for the FL rows of the block
      build_left(a, f, p0, FL, 0, K, chain, slice,
                 [&](int ll, int e, double v) { Vt[vpos(e, ll)] = v; });
    // 2. TR(p, q) for FI columns, FMI x FMJ per thread.
    const int64_t q0 = (u % tiles) * FI;
    const int nq = static_cast<int>((cols - q0 < FI) ? cols - q0 : FI);
    for (int o = threadIdx.x; o < K * FI; o += FNT) {
      const int e = o / FI, iq = o - e * FI;
      Qt[o] = iq < nq ? static_cast<double>(WT[e * cols + q0 + iq]) : 0.0;
    }
    // X in flight while the tile of W lands
    double x[FMI][FMJ];
#pragma unroll
    for (int i = 0; i < FMI; ++i)
#pragma unroll
      for (int v = 0; v < FMJ; ++v) {
        const int64_t p = p0 + ty * FMI + i;
        const int iq = tx * FMJ + v;
        x[i][v] = (p < rows && iq < nq) ? static_cast<double>(X[p * cols + q0 + iq]) : 0.0;
      }
    fit_sync();
    double acc[FMI][FMJ] = {};
    const double* qp = Qt + tx * FMJ;
#pragma unroll 4
    for (int e = 0; e < K; ++e) {
      const double2 vv = *reinterpret_cast<const double2*>(Vt + e * FL + (ty ^ (e & 15)) * FMI);
      const double2 qq = *reinterpret_cast<const double2*>(qp + e * FI);
      acc[0][0] += vv.x * qq.x;
      acc[0][1] += vv.x * qq.y;
      acc[1][0] += vv.y * qq.x;
      acc[1][1] += vv.y * qq.y;
    }
#pragma unroll
    for (int i = 0; i < FMI; ++i) {
      if (p0 + ty * FMI + i >= rows) continue;
#pragma unroll
      for (int v = 0; v < FMJ; ++v) {
        if (tx * FMJ + v >= nq) continue;
        const double d = x[i][v] - acc[i][v];
        se += d * d;
        sx += x[i][v] * x[i][v];
      }
    }
    fit_sync();
  }
}

// Sum of (se, sx) over the first FNT threads to thread 0; `red` holds 2 * (FNT / 32) doubles.
__device__ __forceinline__ void fit_block_reduce(double& se, double& sx, double* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    se += __shfl_xor_sync(0xffffffffu, se, o);
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
  }
  if (lane == 0) { red[warp] = se; red[FNT / 32 + warp] = sx; }
  fit_sync();
  if (threadIdx.x == 0) {
    double a0 = 0.0, a1 = 0.0;
    for (int w = 0; w < FNT / 32; ++w) { a0 += red[w]; a1 += red[FNT / 32 + w]; }
    se = a0;
    sx = a1;
  }
}

}  // namespace trk
