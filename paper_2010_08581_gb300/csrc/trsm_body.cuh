// Triangular solves with a Cholesky factor L (n <= 256) for many vectors, shared by the
// single-problem kernel (trsm.cu) and the batched kernels (batched_solve.cu):
//   mode 0 (leverage rows, row a1): ell_v = || L^-1 a_v ||^2 -- row norms of Q = A R^-1 of
//           the Cholesky-based thin QR (Def. 4), optionally followed by p and the CDF;
//   mode 1 (LS solve, row a6):      z_v = L^-T L^-1 b_v, written into the new core;
//   mode 2 (LS solve + one refinement step, row a6):
//           z = L^-T L^-1 b;  r = b - M z;  z += L^-T L^-1 r.
//
// One CTA takes NV vectors through blocked substitutions: the factor's padded image
// (img[c * (n + 1) + r] = L[r][c]) streams through two shared-memory panels of PB columns, the
// vectors stay in shared memory. Per panel, PB lanes solve the diagonal block for one vector
// (lane = row, one shuffle, multiply and multiply-add per column), then every thread takes one of
// the remaining rows and VP vectors through the panel's PB columns, with no dependence between
// rows. The first panel of the next pass is under way while the last one of this pass is used.
// An entry receives its multiply-adds in the order of the columns, one by one, as the
// substitution of one vector by one warp does, so the panel width never changes a result.
//
// What bounds it: the columns' dependent chain (about 40 clocks a column in FP32, 170 in FP64)
// plus a few hundred clocks of barriers a panel; with many vectors in FP64 the FP64 pipe, where a
// warp's instruction takes 16 clocks however few of its lanes matter: hence 16 columns and two
// vectors a warp there. One warp carrying whole vectors through all columns (the form before)
// kept the remaining rows on the same chain, eight register rows at n = 256 behind a switch per
// column. 300 vectors, mode 2 in FP32: n = 224: 569 -> 89 us, n = 256: 747 -> 98 us; mode 1 in FP64:
// n = 100: 50.5 -> 49 us (1300: 152 -> 90), n = 256: 561 -> 153 us.
#pragma once

#include "common.cuh"

namespace trk {

constexpr int TNT = 256;            // threads per CTA
constexpr int TNW = TNT / 32;

// Columns per panel: 32 in FP32, 16 in FP64, and 32 there too where few vectors leave one CTA per
// SM: then a panel's latency counts, not the FP64 pipe (n = 64, 300 vectors: 29 us with 16 columns,
// 26 with 32; 1300 vectors: 45 us with 16 columns and two vectors a warp, 61 with one).
template <typename T>
constexpr int panel_cols(bool few) { return sizeof(T) == 4 || few ? 32 : 16; }

// Block-wide exclusive scan (fixed order) of one double per thread for NW warps.
template <int NW>
__device__ __forceinline__ double block_scan_nw(double v, double* wt, double* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wt[warp] = inc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double run = 0.0;
    for (int q = 0; q < NW; ++q) { const double t = wt[q]; wt[q] = run; run += t; }
    *total = run;
  }
  __syncthreads();
  const double r = wt[warp] + inc - v;
  __syncthreads();
  return r;
}

// p = ell / sum(ell) and its prefix sum, by the CTA that finishes last (mode 0 only), whose
// NW warps all take part.
template <int NW>
__device__ inline void cdf_epilogue_nw(const CdfEpilogue& ep, const double* ell, int64_t I) {
  __shared__ double wt[NW];
  __shared__ double s_total;
  if (ep.skip && *ep.skip) return;
  const int t = threadIdx.x;
  const int64_t chunk = (I + NW * 32 - 1) / (NW * 32);
  const int64_t b = t * chunk, e = (b + chunk < I) ? b + chunk : I;
  double s = 0.0;
  for (int64_t i = b; i < e; ++i) s += __ldcg(ell + i);
  block_scan_nw<NW>(s, wt, &s_total);
  const double total = s_total;
  if (!(total > 0.0) || !isfinite(total)) {
    for (int64_t i = b; i < e; ++i) {
      ep.p[i] = 1.0 / static_cast<double>(I);
      ep.cdf[i] = static_cast<double>(i + 1) / static_cast<double>(I);
    }
    if (t == 0) atomicOr(ep.err, kErrSingular);
    return;
  }
  // one division: p_i = ell_i * (1 / total) (within an ulp of ell_i / total; an FP64 division
  // per entry costs far more than the multiply on this GPU's FP64 pipe)
  const double rt = 1.0 / total;
  double sp = 0.0;
  for (int64_t i = b; i < e; ++i) sp += __ldcg(ell + i) * rt;
  double run = block_scan_nw<NW>(sp, wt, &s_total);
  for (int64_t i = b; i < e; ++i) {
    const double pi = __ldcg(ell + i) * rt;
    ep.p[i] = pi;
    run += pi;
    ep.cdf[i] = run;
  }
}

// Shared memory of a CTA: the inverse diagonal, two panels and two sets of NV vectors.
template <typename T>
__host__ __device__ inline size_t subst_smem(int n, int nv, int PB) {
  return (static_cast<size_t>((n + 3) & ~3) + 2 * static_cast<size_t>(n + 1) * (PB + 1) +
          2 * static_cast<size_t>(n) * nv + 4) * sizeof(T);
}

template <typename T>
__device__ __forceinline__ void copy_async(T* dst, const T* src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" :: "r"(d), "l"(src) : "memory");
}

// Blocked substitutions and products on NV vectors x[row * NV + v] in shared memory.
template <typename T, int NV, int VP, int PB>
struct Subst {
  static constexpr int VPW = 32 / PB;           // vectors per warp in the diagonal blocks
  static constexpr int G = NV / VP;             // groups of vectors
  static constexpr int RT = TNT / G;            // rows the threads cover
  int n, np;
  const T* inv;
  T* panel[2];

  // Panel of columns c0 .. c0 + PB - 1 and rows r0 .. n - 1, as p[k * (n + 1) + row].
  __device__ __forceinline__ void stage_cols(T* p, const T* img, int c0, int r0) const {
    const int w = min(PB, n - c0);
    for (int k = threadIdx.x >> 5; k < w; k += TNW)
      for (int r = r0 + (threadIdx.x & 31); r < n; r += 32)
        copy_async(p + k * np + r, img + static_cast<int64_t>(c0 + k) * np + r);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // Rows c0 .. c0 + PB - 1 of the factor, columns 0 .. r1 - 1, as p[column * (PB + 1) + k].
  __device__ __forceinline__ void stage_rows(T* p, const T* img, int c0, int r1) const {
    const int w = min(PB, n - c0);
    for (int e = threadIdx.x; e < r1 * PB; e += TNT) {
      const int r = e / PB, k = e % PB;
      if (k < w) copy_async(p + r * (PB + 1) + k, img + static_cast<int64_t>(r) * np + c0 + k);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  static __device__ __forceinline__ void landed(bool more) {   // all but the newest group
    if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
  }

  enum Next { kNone, kRows, kCols };   // what the next pass stages first

  // First panel of the next pass, while this pass uses its last one.
  __device__ __forceinline__ bool stage_next(T* p, Next next, const T* img) const {
    if (next == kRows) stage_rows(p, img, (n - 1) / PB * PB, n);
    else if (next == kCols) stage_cols(p, img, 0, 0);
    return next != kNone;
  }

  // x <- L^-1 x. Panel s holds (or receives) the first PB columns; returns the next pass's panel.
  __device__ int forward(T* x, const T* img, int s, Next next) const {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x % PB;
    const int vec = warp * VPW + (threadIdx.x & 31) / PB;
    const int g = threadIdx.x / RT, i = threadIdx.x % RT;
    for (int c0 = 0; c0 < n; c0 += PB, s ^= 1) {
      const int w = min(PB, n - c0);
      bool more = c0 + PB < n;
      if (more) stage_cols(panel[s ^ 1], img, c0 + PB, c0 + PB);
      else more = stage_next(panel[s ^ 1], next, img);
      landed(more);
      const T* p = panel[s];
      if (warp * VPW < NV) {
        T v = lane < w ? x[(c0 + lane) * NV + vec] : T(0);
#pragma unroll 8
        for (int k = 0; k < w; ++k) {
          const T xc = __shfl_sync(0xffffffffu, v, k, PB) * inv[c0 + k];
          const T l = lane > k && lane < w ? p[k * np + c0 + lane] : T(0);
          if (lane == k) v = xc;
          else if (lane > k && lane < w) v -= l * xc;
        }
        if (lane < w) x[(c0 + lane) * NV + vec] = v;
      }
      __syncthreads();
      const int r = c0 + PB + i;
      if (c0 + PB >= n) continue;
      if (r < n) {
        T acc[VP];
#pragma unroll
        for (int v = 0; v < VP; ++v) acc[v] = x[r * NV + g * VP + v];
#pragma unroll 8
        for (int k = 0; k < PB; ++k) {      // more rows follow: the panel is full
          const T l = p[k * np + r];
#pragma unroll
          for (int v = 0; v < VP; ++v) acc[v] -= l * x[(c0 + k) * NV + g * VP + v];
        }
#pragma unroll
        for (int v = 0; v < VP; ++v) x[r * NV + g * VP + v] = acc[v];
      }
      __syncthreads();
    }
    return s;
  }

  // x <- L^-T x, panels and columns in reverse order. Panel s receives the last rows.
  __device__ int backward(T* x, const T* img, int s, Next next, const T* next_img) const {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x % PB;
    const int vec = warp * VPW + (threadIdx.x & 31) / PB;
    const int g = threadIdx.x / RT, i = threadIdx.x % RT;
    for (int c0 = (n - 1) / PB * PB; c0 >= 0; c0 -= PB, s ^= 1) {
      const int w = min(PB, n - c0);
      bool more = c0 > 0;
      if (more) stage_rows(panel[s ^ 1], img, c0 - PB, c0);
      else more = stage_next(panel[s ^ 1], next, next_img);
      landed(more);
      const T* p = panel[s];
      if (warp * VPW < NV) {
        T v = lane < w ? x[(c0 + lane) * NV + vec] : T(0);
#pragma unroll 8
        for (int k = w - 1; k >= 0; --k) {
          const T zc = __shfl_sync(0xffffffffu, v, k, PB) * inv[c0 + k];
          const T l = lane < k ? p[(c0 + lane) * (PB + 1) + k] : T(0);
          if (lane == k) v = zc;
          else if (lane < k) v -= l * zc;
        }
        if (lane < w) x[(c0 + lane) * NV + vec] = v;
      }
      __syncthreads();
      if (c0 == 0) continue;
      if (i < c0) {
        T acc[VP];
#pragma unroll
        for (int v = 0; v < VP; ++v) acc[v] = x[i * NV + g * VP + v];
#pragma unroll 8
        for (int k = w - 1; k >= 0; --k) {
          const T l = p[i * (PB + 1) + k];
#pragma unroll
          for (int v = 0; v < VP; ++v) acc[v] -= l * x[(c0 + k) * NV + g * VP + v];
        }
#pragma unroll
        for (int v = 0; v < VP; ++v) x[i * NV + g * VP + v] = acc[v];
      }
      __syncthreads();
    }
    return s;
  }

  // r <- r - M z (M symmetric, image img[t * (n + 1) + row]); then img2's first columns are staged.
  __device__ int residual(T* r, const T* z, const T* img, int s, const T* img2) const {
    const int g = threadIdx.x / RT, i = threadIdx.x % RT;
    T acc[VP];
#pragma unroll
    for (int v = 0; v < VP; ++v) acc[v] = i < n ? r[i * NV + g * VP + v] : T(0);
    for (int c0 = 0; c0 < n; c0 += PB, s ^= 1) {
      const int w = min(PB, n - c0);
      if (c0 + PB < n) stage_cols(panel[s ^ 1], img, c0 + PB, 0);
      else stage_cols(panel[s ^ 1], img2, 0, 0);
      landed(true);
      const T* p = panel[s];
      if (i < n) {
#pragma unroll 8
        for (int k = 0; k < w; ++k) {
          const T m = p[k * np + i];
#pragma unroll
          for (int v = 0; v < VP; ++v) acc[v] -= m * z[(c0 + k) * NV + g * VP + v];
        }
      }
      __syncthreads();
    }
    if (i < n)
#pragma unroll
      for (int v = 0; v < VP; ++v) r[i * NV + g * VP + v] = acc[v];
    __syncthreads();
    return s;
  }
};

template <typename T, int NV, int VP, int PB>
__device__ __forceinline__ void subst_cta(unsigned char* sm, int64_t cta, int n,
                                          const double* __restrict__ invdiag,
                                          const int* __restrict__ info, int64_t nvec,
                                          const double* __restrict__ rhs, int64_t ld, int mode,
                                          const T* __restrict__ Limg,
                                          const float* __restrict__ Mimg, int Rl, int Rr,
                                          double* __restrict__ core_out,
                                          double* __restrict__ ell, CdfEpilogue ep, int nctas) {
  if ((info && *info) || (ep.run_if && *ep.run_if == 0)) return;
  static_assert(NV <= TNW && NV % Subst<T, NV, VP, PB>::VPW == 0, "vectors a warp");
  T* inv = reinterpret_cast<T*>(sm);
  Subst<T, NV, VP, PB> S;
  S.n = n;
  S.np = n + 1;
  S.inv = inv;
  S.panel[0] = inv + ((n + 3) & ~3);
  S.panel[1] = S.panel[0] + (n + 1) * (PB + 1);
  // (16-byte offset in elements: a pointer rounded as an integer would lose its address space)
  T* x = inv + ((((n + 3) & ~3) + 2 * (n + 1) * (PB + 1) + 3) & ~3);
  T* res = x + n * NV;
  const int64_t v0 = cta * NV;
  S.stage_cols(S.panel[0], Limg, 0, 0);
  for (int c = threadIdx.x; c < n; c += TNT) inv[c] = static_cast<T>(invdiag[c]);
  for (int v = threadIdx.x >> 5; v < NV; v += TNW)
    for (int r = threadIdx.x & 31; r < n; r += 32) {
      const T b = v0 + v < nvec ? static_cast<T>(rhs[(v0 + v) * ld + r]) : T(0);
      x[r * NV + v] = b;
      if (mode == 2) res[r * NV + v] = b;
    }
  int s = S.forward(x, Limg, 0, mode == 0 ? S.kNone : S.kRows);   // (its first barrier covers x)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (mode == 0) {
    if (warp < NV && v0 + warp < nvec) {
      T sq = T(0);
      for (int r = lane; r < n; r += 32) sq += x[r * NV + warp] * x[r * NV + warp];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (lane == 0) ell[v0 + warp] = static_cast<double>(sq);
    }
    if (ep.counter) {      // the last CTA to finish forms p and the CDF
      __shared__ int s_last;
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0)
        s_last = (atomicAdd(ep.counter, 1u) == static_cast<unsigned>(nctas) - 1) ? 1 : 0;
      __syncthreads();
      if (s_last) {
        __threadfence();
        cdf_epilogue_nw<TNW>(ep, ell, nvec);
        if (threadIdx.x == 0) *ep.counter = 0u;
      }
    }
    return;
  }
  if constexpr (sizeof(T) == 4) {
    s = S.backward(x, Limg, s, mode == 2 ? S.kCols : S.kNone, Mimg);
    if (mode == 2) {
      s = S.residual(res, x, Mimg, s, Limg);
      s = S.forward(res, Limg, s, S.kRows);
      S.backward(res, Limg, s, S.kNone, Limg);
    }
  } else {
    S.backward(x, Limg, s, S.kNone, Limg);
  }
  // new core: core[i][a][b] = z[a + Rl*b]
  for (int v = warp; v < NV; v += TNW) {
    if (v0 + v >= nvec) continue;
    for (int r = lane; r < n; r += 32) {
      const T z = mode == 2 ? x[r * NV + v] + res[r * NV + v] : x[r * NV + v];
      core_out[(v0 + v) * n + (r % Rl) * Rr + r / Rl] = static_cast<double>(z);
    }
  }
}

// The vectors per thread follow from the rows the threads have to cover: 256 threads take
// 32 * ceil(n / 32) rows rounded up to a power of two.
#define TRK_SUBST_DISPATCH(n, CASE)      \
  do {                                   \
    if ((n) <= 32) { CASE(1); }          \
    else if ((n) <= 64) { CASE(2); }     \
    else if ((n) <= 128) { CASE(4); }    \
    else { CASE(8); }                    \
  } while (0)

}  // namespace trk
