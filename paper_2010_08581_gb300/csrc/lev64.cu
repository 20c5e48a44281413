// FP32 factor and inverse of a symmetric positive definite n x n matrix for 128 < n <= 256, and
// what is built on an FP32 inverse X of the factor by products that spread over the GPU:
//   * the leverage scores of a tall matrix in FP64 (row a1): with C = X K X^T = I + E (the
//     identity of lev_precond.cu), K^-1 = X'^T X' for X' = C^-1/2 X, so ell_i = ||X' a_i||^2. Every
//     product is in FP64 and C^-1/2 is its binomial series in E, through E^3 for
//     ||E||_F <= 1e-4, E^5 up to 1e-3 and E^7 up to 1e-2: a remainder below 3e-17 each time;
//   * the FP64 LS step (row a6): z = V b with V = M^-1 = X'^T X' and the same X' of M, then one step
//     of refinement, r = b - M z, z += V r: E carries a rounding of eps cond(M), which the products
//     alone would take into z as cond(M)^1/2 times that;
//   * the mixed-precision LS step's solves (row a6) for 160 < L <= 256.
//
// Why: one SM multiplies two FP64 pairs per clock, so the one-CTA FP64 factorisation of a 256 x
// 256 matrix is 0.7 ms of arithmetic (1.85 ms measured), and one chain of 256 columns per
// substitution follows. Here the only serial chains are the FP32 one-CTA passes of chol_inv.cuh;
// the rest are matrix products in small tiles over all SMs: with the factor's, eight short launches
// up to 128 columns and 13 beyond, bound by one tile's FP64 arithmetic and a trip to L2 each, then
// two for the rows (n = 256: 271 us, then 81 for 300 rows).
//
// Every kernel does nothing when the flag in its arguments says that the FP32 factorisation
// failed (a pivot <= n * eps32 * max diag) or that ||E||_F is too large for the series; the
// callers' previous form then runs, gated on the same flag, with no host round trip.
#include "chol_inv.cuh"
#include "trsm_body.cuh"

namespace trk {
namespace {

constexpr int GK = 16;             // terms per shared-memory stage
constexpr int GE = 16;             // tile edge
constexpr int GNT = 64;            // 2 x 2 outputs per thread

// acc(i, j) = sum over kb <= k < ke of a(i, k) * b(k, j) for the GE x GE tile at (i0, j0), in
// order of k; a and b return 0 outside their matrices. kAk / kBk: a (b) is contiguous in k, so
// threads take consecutive k, else consecutive rows (columns). ep(i, j, acc) for every entry.
// Shared memory of one product: two stages of each operand.
template <typename T>
struct Stages {
  T a[2][GK][GE + 1], b[2][GK][GE + 1];
};

template <typename T, bool kAk, bool kBk, typename A, typename B, typename Ep>
__device__ __forceinline__ void tile_product(Stages<T>& sm, int i0, int j0, int kb, int ke, A a, B b,
                                             Ep ep) {
  constexpr int Q = GE * GK / GNT;
  const int t = threadIdx.x, tx = t % (GE / 2), ty = t / (GE / 2);
  T ra[Q], rb[Q];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int e = t + GNT * q;
      const int ak = kAk ? e % GK : e / GE, ar = kAk ? e / GK : e % GE;
      const int bk = kBk ? e % GK : e / GE, bc = kBk ? e / GK : e % GE;
      ra[q] = k0 + ak < ke ? a(i0 + ar, k0 + ak) : T(0);
      rb[q] = k0 + bk < ke ? b(k0 + bk, j0 + bc) : T(0);
    }
  };
  T acc[2][2] = {};
  load(kb);
  int s = 0;
  for (int k0 = kb; k0 < ke; k0 += GK, s ^= 1) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int e = t + GNT * q;
      sm.a[s][kAk ? e % GK : e / GE][kAk ? e / GK : e % GE] = ra[q];
      sm.b[s][kBk ? e % GK : e / GE][kBk ? e / GK : e % GE] = rb[q];
    }
    __syncthreads();
    if (k0 + GK < ke) load(k0 + GK);
#pragma unroll
    for (int k = 0; k < GK; ++k) {
      const T x0 = sm.a[s][k][ty], x1 = sm.a[s][k][ty + GE / 2];
      const T y0 = sm.b[s][k][tx], y1 = sm.b[s][k][tx + GE / 2];
      acc[0][0] += x0 * y0;
      acc[0][1] += x0 * y1;
      acc[1][0] += x1 * y0;
      acc[1][1] += x1 * y1;
    }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) ep(i0 + ty + GE / 2 * u, j0 + tx + GE / 2 * v, acc[u][v]);
}

// ------------------------------------------------------------------------------------
// FP32 factor and inverse, 128 < n <= 256: K = [[A, .], [B, D]] with an n1 x n1 block A,
//   X11 = inv(chol A);  Lb = B X11^T;  S = D - Lb Lb^T;  X22 = inv(chol S);
//   X21 = -X22 Lb X11.
// K[i][j] = pre[j * lda + i] (i >= j). X goes to Ximg[c * np + r], np = n + 1.
// ------------------------------------------------------------------------------------
struct BigInv {
  const float* pre;
  int n, lda, n1;
  float* Ximg;
  float* Lb;         // n2 x n1, row-major
  float* S;          // n2 x n2 lower triangle, S[j * lds + i]; later T = X22 Lb, n2 x n1
  float* T;
  int lds;
  int* bad;          // bad[0] = 1 when the factorisation failed, bad[1] = 1 - bad[0]
};

__global__ void __launch_bounds__(kCiMaxThreads) k_big_factor(BigInv g, float tol, int part,
                                                              int* keep, int* info,
                                                              const unsigned* err) {
  grid_wait();
  __shared__ CiShared cs;
  const int np = g.n + 1, n2 = g.n - g.n1;
  if (part == 0) {
    if (err && (*reinterpret_cast<const volatile unsigned*>(err) & kErrTimeout)) {
      if (threadIdx.x == 0) { *info = -1; g.bad[0] = 2; g.bad[1] = 0; }   // nothing to factor
      return;
    }
    const bool ok = chol_inv_tiles(g.n1, tol, g.pre, g.lda, g.Ximg, np, g.pre, g.n, g.lda, cs);
    if (threadIdx.x == 0) { g.bad[0] = ok ? 0 : 1; g.bad[1] = ok ? 0 : 1; }
    return;
  }
  if (g.bad[0]) return;
  const bool ok = chol_inv_tiles(n2, tol, g.S, g.lds, g.Ximg + static_cast<int64_t>(g.n1) * np + g.n1,
                                 np, g.pre, g.n, g.lda, cs);
  if (ok && keep)
    for (int k = threadIdx.x; k < g.n; k += blockDim.x) keep[k] = 1;
  if (threadIdx.x == 0) {
    if (ok && info) *info = 0;
    if (!ok) { g.bad[0] = 1; g.bad[1] = 1; }
  }
}

__global__ void __launch_bounds__(GNT) k_big_lb(BigInv g) {
  grid_wait();
  __shared__ Stages<float> sm;
  if (g.bad[0]) return;
  const int np = g.n + 1, n1 = g.n1, n2 = g.n - n1;
  const int i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  tile_product<float, false, false>(sm, i0, j0, 0, min(n1, j0 + GE),
      [&](int i, int k) { return i < n2 ? g.pre[static_cast<int64_t>(k) * g.lda + n1 + i] : 0.f; },
      [&](int k, int j) { return j < n1 && k <= j ? g.Ximg[static_cast<int64_t>(k) * np + j] : 0.f; },
      [&](int i, int j, float v) { if (i < n2 && j < n1) g.Lb[i * n1 + j] = v; });
}

__global__ void __launch_bounds__(GNT) k_big_s(BigInv g) {
  grid_wait();
  __shared__ Stages<float> sm;
  const int i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  if (g.bad[0] || i0 + GE <= j0) return;
  const int n1 = g.n1, n2 = g.n - n1;
  tile_product<float, true, true>(sm, i0, j0, 0, n1, [&](int i, int k) { return i < n2 ? g.Lb[i * n1 + k] : 0.f; },
      [&](int k, int j) { return j < n2 ? g.Lb[j * n1 + k] : 0.f; },
      [&](int i, int j, float v) {
        if (i < n2 && j <= i)
          g.S[j * g.lds + i] = g.pre[static_cast<int64_t>(n1 + j) * g.lda + n1 + i] - v;
      });
}

__global__ void __launch_bounds__(GNT) k_big_t(BigInv g) {
  grid_wait();
  __shared__ Stages<float> sm;
  if (g.bad[0]) return;
  const int np = g.n + 1, n1 = g.n1, n2 = g.n - n1;
  const int i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  const float* X22 = g.Ximg + static_cast<int64_t>(n1) * np + n1;
  tile_product<float, false, false>(sm, i0, j0, 0, min(n2, i0 + GE),
      [&](int i, int k) { return i < n2 && k <= i ? X22[static_cast<int64_t>(k) * np + i] : 0.f; },
      [&](int k, int j) { return j < n1 ? g.Lb[k * n1 + j] : 0.f; },
      [&](int i, int j, float v) { if (i < n2 && j < n1) g.T[i * n1 + j] = v; });
}

__global__ void __launch_bounds__(GNT) k_big_x21(BigInv g) {
  grid_wait();
  __shared__ Stages<float> sm;
  if (g.bad[0]) return;
  const int np = g.n + 1, n1 = g.n1, n2 = g.n - n1;
  const int i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  tile_product<float, true, true>(sm, i0, j0, j0, n1, [&](int i, int k) { return i < n2 ? g.T[i * n1 + k] : 0.f; },
      [&](int k, int j) { return j < n1 && k >= j ? g.Ximg[static_cast<int64_t>(j) * np + k] : 0.f; },
      [&](int i, int j, float v) {
        if (i < n2 && j < n1) {
          g.Ximg[static_cast<int64_t>(j) * np + n1 + i] = -v;
          g.Ximg[static_cast<int64_t>(n1 + i) * np + j] = 0.f;     // above the diagonal
        }
      });
}

// ------------------------------------------------------------------------------------
// FP64 products: 8 x 8 outputs per CTA over all terms, loaded at once. One SM's FP64 pipe is the
// bound of a tile (16 x 16 over 100 terms: 6.4 us, 8 x 8: 1.6), one trip to L2 the rest.
// ------------------------------------------------------------------------------------
constexpr int DE = 8, DNT = 64;
constexpr int DLD = kMaxL + 2;

struct Panels {
  double a[DE][DLD], b[DE][DLD];   // a(i0 + r, k), b(k, j0 + r)
  double half[DE * DE];
};

// ep(i, j, sum over kb <= k < ke of a(i, k) * b(k, j)) for the tile at (i0, j0), by the first
// warp: lane = 4 * row + column pair. kAk / kBk: a (b) is contiguous in k. Each warp sums half of
// the terms, in runs of kRun (even).
template <bool kAk, bool kBk, int kRun = DLD, typename A, typename B, typename Ep>
__device__ __forceinline__ void tile8(Panels& sm, int i0, int j0, int kb, int ke, A a, B b, Ep ep) {
  const int t = threadIdx.x, kn = ke - kb, kp = (kn + 3) & ~3;    // padded with zeros to a half
  if constexpr (kAk) {
    for (int r = 0; r < DE; ++r)
      for (int k = t; k < kp; k += DNT) sm.a[r][k] = k < kn ? a(i0 + r, kb + k) : 0.0;
  } else {
    for (int e = t; e < DE * kp; e += DNT) sm.a[e % DE][e / DE] = e / DE < kn ? a(i0 + e % DE, kb + e / DE) : 0.0;
  }
  if constexpr (kBk) {
    for (int r = 0; r < DE; ++r)
      for (int k = t; k < kp; k += DNT) sm.b[r][k] = k < kn ? b(kb + k, j0 + r) : 0.0;
  } else {
    for (int e = t; e < DE * kp; e += DNT) sm.b[e % DE][e / DE] = e / DE < kn ? b(kb + e / DE, j0 + e % DE) : 0.0;
  }
  __syncthreads();
  const int warp = t >> 5, lane = t & 31, r = lane >> 2, c = 2 * (lane & 3);
  double x0 = 0.0, x1 = 0.0, y0 = 0.0, y1 = 0.0;
  const int k0 = warp * (kp / 2), k1 = (warp + 1) * (kp / 2);
  auto terms = [&](int ka, int ke2, double& p0, double& p1, double& q0, double& q1) {
#pragma unroll 4
    for (int k = ka; k < ke2; k += 2) {
      const double2 u = *reinterpret_cast<const double2*>(&sm.a[r][k]);
      const double2 v = *reinterpret_cast<const double2*>(&sm.b[c][k]);
      const double2 w = *reinterpret_cast<const double2*>(&sm.b[c + 1][k]);
      p0 += u.x * v.x;
      q0 += u.x * w.x;
      p1 += u.y * v.y;
      q1 += u.y * w.y;
    }
  };
  if constexpr (kRun >= DLD) {
    terms(k0, k1, x0, x1, y0, y1);
  } else {
    for (int kr = k0; kr < k1; kr += kRun) {
      double p0 = 0.0, p1 = 0.0, q0 = 0.0, q1 = 0.0;
      terms(kr, min(kr + kRun, k1), p0, p1, q0, q1);
      x0 += p0;
      y0 += q0;
      x1 += p1;
      y1 += q1;
    }
  }
  x0 += x1;
  y0 += y1;
  if (warp == 1) { sm.half[r * DE + c] = x0; sm.half[r * DE + c + 1] = y0; }
  __syncthreads();
  if (warp == 0) {
    ep(i0 + r, j0 + c, x0 + sm.half[r * DE + c]);
    ep(i0 + r, j0 + c + 1, y0 + sm.half[r * DE + c + 1]);
  }
}

// Tile (i0, j0), i0 <= j0, number b of the upper triangle of nt x nt tiles.
__device__ __forceinline__ void upper_tile(int b, int nt, int& i0, int& j0) {
  int ti = 0;
  while (b >= nt - ti) { b -= nt - ti; ++ti; }
  i0 = ti * DE;
  j0 = (ti + b) * DE;
}

// ------------------------------------------------------------------------------------
// X' = (X K X^T)^-1/2 X in FP64.
// ------------------------------------------------------------------------------------
struct L64 {
  int n;
  const float* Ximg;
  const double* G;   // K, entries r <= c
  double* E;
  double* U;         // X K, then E2 = E E
  double* P;         // the tiles' shares of ||E||_F^2; c4 + c5 E + E2 (c6 + c7 E); Q
  double* T;         // c2 + c3 E + E2 P; X' = Q X
  int* flag;         // [0]: the FP32 factorisation failed, [1]: the fallback has to run, [2]: degree
  int* keep;         // LS step: set when the series applies (keep = 1, *info = 0); or null
  int* info;
  double tau2;       // largest ||E||_F^2, at most 1e-4
};

// U = X K.
__global__ void __launch_bounds__(DNT) k_l64_u(L64 g) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0]) return;
  const int n = g.n, np = n + 1, i0 = blockIdx.y * DE, j0 = blockIdx.x * DE;
  tile8<false, false>(sm, i0, j0, 0, min(n, i0 + DE),
      [&](int i, int k) { return i < n && k <= i ? static_cast<double>(g.Ximg[k * np + i]) : 0.0; },
      [&](int k, int j) { return j < n ? (k <= j ? g.G[k * n + j] : g.G[j * n + k]) : 0.0; },
      [&](int i, int j, double v) { if (i < n && j < n) g.U[i * n + j] = v; });
}

// E = U X^T - I on the tiles with i0 <= j0, both triangles written, and the tile's share of
// ||E||_F^2 in P[tile].
__global__ void __launch_bounds__(DNT) k_l64_e(L64 g) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0]) return;
  const int n = g.n, np = n + 1;
  int i0, j0;
  upper_tile(blockIdx.x, (n + DE - 1) / DE, i0, j0);
  double sq = 0.0;
  tile8<true, false>(sm, i0, j0, 0, min(n, j0 + DE), [&](int i, int k) { return i < n ? g.U[i * n + k] : 0.0; },
      [&](int k, int j) { return j < n && k <= j ? static_cast<double>(g.Ximg[k * np + j]) : 0.0; },
      [&](int i, int j, double v) {
        if (i >= n || j >= n || i > j) return;
        const double e = i == j ? v - 1.0 : v;
        g.E[i * n + j] = e;
        g.E[j * n + i] = e;
        sq += (i == j ? 1.0 : 2.0) * e * e;
      });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if (threadIdx.x == 0) g.P[blockIdx.x] = sq;
}

// The coefficients of (1 + x)^-1/2, binom(-1/2, k).
__device__ __forceinline__ double l64_c(int k) {
  constexpr double c[8] = {1.0, -1.0 / 2, 3.0 / 8, -5.0 / 16, 35.0 / 128, -63.0 / 256, 231.0 / 1024,
                           -429.0 / 2048};
  return c[k];
}

// Degree of the series by ||E||_F: 3, 5, 7, or 0 when E is too large for it; E2 = E E.
__global__ void __launch_bounds__(DNT) k_l64_e2(L64 g) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0]) return;
  const int n = g.n;
  double f2 = 0.0;
  for (int b = threadIdx.x & 31; b < static_cast<int>(gridDim.x); b += 32) f2 += g.P[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) f2 += __shfl_xor_sync(0xffffffffu, f2, o);
  const int deg = !(f2 <= g.tau2) ? 0 : (f2 <= 1e-8 ? 3 : (f2 <= 1e-6 ? 5 : 7));
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      g.flag[2] = deg;
      if (deg == 0) g.flag[1] = 1;
      else if (g.info) *g.info = 0;
    }
    if (deg && g.info)
      for (int k = threadIdx.x; k < n; k += DNT) g.keep[k] = 1;
  }
  if (deg == 0) return;
  int i0, j0;
  upper_tile(blockIdx.x, (n + DE - 1) / DE, i0, j0);
  tile8<true, true>(sm, i0, j0, 0, n, [&](int i, int k) { return i < n ? g.E[i * n + k] : 0.0; },
      [&](int k, int j) { return j < n ? g.E[j * n + k] : 0.0; },
      [&](int i, int j, double v) {
        if (i >= n || j >= n || i > j) return;
        g.U[i * n + j] = v;
        g.U[j * n + i] = v;
      });
}

// P = c4 + c5 E + E2 (c6 + c7 E) (degree 7 only), T = c2 + c3 E + E2 P (from degree 5 on), Q = 1 + c1 E +
// E2 T into P's place by `which` = 1, 2, 3: polynomials in E, so symmetric; the tiles of the upper
// triangle are formed and both triangles written. which = 4: X' = Q X into T's place, all tiles.
__global__ void __launch_bounds__(DNT) k_l64_poly(L64 g, int which) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0]) return;
  const int deg = g.flag[2];
  if (deg == 0 || (which == 1 && deg < 7) || (which == 2 && deg < 5)) return;
  const int n = g.n, np = n + 1;
  if (which == 4) {
    const int i0 = blockIdx.y * DE, j0 = blockIdx.x * DE;
    tile8<true, true>(sm, i0, j0, j0, n, [&](int i, int k) { return i < n ? g.P[i * n + k] : 0.0; },
        [&](int k, int j) { return j < n && k >= j ? static_cast<double>(g.Ximg[j * np + k]) : 0.0; },
        [&](int i, int j, double v) { if (i < n && j < n) g.T[i * n + j] = v; });
    return;
  }
  int i0, j0;
  upper_tile(blockIdx.x, (n + DE - 1) / DE, i0, j0);
  // the right factor: symmetric, given or c_c + c_(c+1) E
  const double* m = which == 2 && deg == 7 ? g.P : (which == 3 && deg > 3 ? g.T : nullptr);
  const int c = which == 1 ? 6 : (which == 2 ? 4 : 2), out = which == 1 ? 4 : (which == 2 ? 2 : 0);
  const double r0 = l64_c(c), r1 = l64_c(c + 1), o0 = l64_c(out), o1 = l64_c(out + 1);
  double* dst = which == 2 ? g.T : g.P;
  tile8<true, true>(sm, i0, j0, 0, n, [&](int i, int k) { return i < n ? g.U[i * n + k] : 0.0; },
      [&](int k, int j) {
        if (j >= n) return 0.0;
        return m ? m[j * n + k] : (k == j ? r0 : 0.0) + r1 * g.E[j * n + k];
      },
      [&](int i, int j, double v) {
        if (i >= n || j >= n || i > j) return;
        v = (i == j ? o0 : 0.0) + (o1 * g.E[i * n + j] + v);       // smallest terms first
        dst[i * n + j] = v;
        dst[j * n + i] = v;
      });
}

// Partial row norms of A X'^T: the tile's 8 columns of ||X' a_i||^2 into part[column tile][row].
__global__ void __launch_bounds__(DNT) k_l64_rows(L64 g, const double* __restrict__ A, int64_t lda,
                                                  int rows, double* __restrict__ part) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0] || g.flag[2] == 0) return;
  const int n = g.n, i0 = blockIdx.y * DE, j0 = blockIdx.x * DE;
  double sq = 0.0;
  tile8<true, true>(sm, i0, j0, 0, n, [&](int i, int k) { return i < rows ? A[i * lda + k] : 0.0; },
      [&](int k, int j) { return j < n ? g.T[j * n + k] : 0.0; },
      [&](int i, int j, double v) { sq += v * v; });
  if (threadIdx.x >= 32) return;
  sq += __shfl_xor_sync(0xffffffffu, sq, 1);
  sq += __shfl_xor_sync(0xffffffffu, sq, 2);
  const int i = i0 + (threadIdx.x >> 2);
  if ((threadIdx.x & 3) == 0 && i < rows) part[static_cast<int64_t>(blockIdx.x) * rows + i] = sq;
}

// ell of `rows` rows from row0 on, the column tiles' shares added in order; with the last rows
// (ep.p) p and the CDF. One CTA.
constexpr int kFinishThreads = 1024;
__global__ void __launch_bounds__(kFinishThreads) k_l64_finish(L64 g, const double* __restrict__ part,
                                                               int tiles, int rows, int64_t row0,
                                                               double* ell, int64_t I, CdfEpilogue ep) {
  grid_wait();
  if (g.flag[0] || g.flag[2] == 0) return;
  for (int i = threadIdx.x; i < rows; i += kFinishThreads) {
    double s = 0.0;
#pragma unroll 8
    for (int q = 0; q < tiles; ++q) s += part[static_cast<int64_t>(q) * rows + i];
    ell[row0 + i] = s;
  }
  __threadfence();
  __syncthreads();
  if (ep.p) cdf_epilogue_nw<kFinishThreads / 32>(ep, ell, I);
}

// The FP64 LS step: V = X'^T X' into E2's place (the tiles of the upper triangle, both written).
// z = X'^T (X' b) twice would be five products of a right-hand side instead of three and two
// launches more (L = 256, 300 right-hand sides: 314 us a solve, 242 with V).
__global__ void __launch_bounds__(DNT) k_l64_inv(L64 g) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0] || g.flag[2] == 0) return;
  const int n = g.n;
  int i0, j0;
  upper_tile(blockIdx.x, (n + DE - 1) / DE, i0, j0);
  tile8<false, false>(sm, i0, j0, 0, n, [&](int i, int k) { return i < n ? g.T[k * n + i] : 0.0; },
      [&](int k, int j) { return j < n ? g.T[k * n + j] : 0.0; },
      [&](int i, int j, double v) {
        if (i >= n || j >= n || i > j) return;
        g.U[i * n + j] = v;
        g.U[j * n + i] = v;
      });
}

// The place of unknown k in a row of the core.
__device__ __forceinline__ int core_entry(int k, int Rl, int Rr) { return (k % Rl) * Rr + k / Rl; }

// z = V b for `rows` right-hand sides (rows of b) into the new core, or z there + V b (add).
__global__ void __launch_bounds__(DNT) k_l64_z(L64 g, const double* __restrict__ b, int64_t ld,
                                               int rows, int Rl, int Rr, double* __restrict__ core,
                                               bool add) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0] || g.flag[2] == 0) return;
  const int n = g.n;
  tile8<true, true>(sm, blockIdx.y * DE, blockIdx.x * DE, 0, n,
      [&](int i, int k) { return i < rows ? b[i * ld + k] : 0.0; },
      [&](int k, int j) { return j < n ? g.U[j * n + k] : 0.0; },
      [&](int i, int j, double v) {
        if (i >= rows || j >= n) return;
        double* at = core + static_cast<int64_t>(i) * n + core_entry(j, Rl, Rr);
        *at = add ? *at + v : v;
      });
}

// r = b - M z, summed in runs of 16 terms: the rounding of r is what is left in the result, and
// one chain of 256 terms carries about twice as much of it.
__global__ void __launch_bounds__(DNT) k_l64_r(L64 g, const double* __restrict__ b, int64_t ld,
                                               int rows, int Rl, int Rr,
                                               const double* __restrict__ core, double* __restrict__ r) {
  grid_wait();
  __shared__ __align__(16) Panels sm;
  if (g.flag[0] || g.flag[2] == 0) return;
  const int n = g.n;
  tile8<true, false, 16>(sm, blockIdx.y * DE, blockIdx.x * DE, 0, n,
      [&](int i, int k) { return i < rows ? core[static_cast<int64_t>(i) * n + core_entry(k, Rl, Rr)] : 0.0; },
      [&](int k, int j) { return j < n ? (k <= j ? g.G[k * n + j] : g.G[j * n + k]) : 0.0; },
      [&](int i, int j, double v) {
        if (i < rows && j < n) r[static_cast<int64_t>(i) * n + j] = b[i * ld + j] - v;
      });
}

// ------------------------------------------------------------------------------------
// The mixed LS step's solves, 160 < n <= 256, `rows` right-hand sides b (rows of B^T): with
// W = X: y = W b, z = W^T y, r = b - M z, y = W r, z += W^T y, in FP32, as solve_inv.cu.
// ------------------------------------------------------------------------------------
// out = src W^T (lower: out_j = sum_{k <= j} W[j][k] src_k).
template <typename TS>
__global__ void __launch_bounds__(GNT) k_sv_lower(int n, const float* __restrict__ Wimg,
                                                  const int* bad, int rows,
                                                  const TS* __restrict__ src, int64_t ld,
                                                  float* __restrict__ out) {
  grid_wait();
  __shared__ Stages<float> sm;
  if (*bad) return;
  const int np = n + 1, i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  tile_product<float, true, false>(sm, i0, j0, 0, min(n, j0 + GE),
      [&](int i, int k) { return i < rows ? static_cast<float>(src[i * ld + k]) : 0.f; },
      [&](int k, int j) { return j < n && k <= j ? Wimg[k * np + j] : 0.f; },
      [&](int i, int j, float v) { if (i < rows && j < n) out[static_cast<int64_t>(i) * n + j] = v; });
}

// z_j = sum_{k >= j} W[k][j] y_k; with core the new core's entries z + add, else z.
__global__ void __launch_bounds__(GNT) k_sv_upper(int n, const float* __restrict__ Wimg,
                                                  const int* bad, int rows,
                                                  const float* __restrict__ y,
                                                  const float* __restrict__ add,
                                                  float* __restrict__ z, int Rl, int Rr,
                                                  double* __restrict__ core) {
  grid_wait();
  __shared__ Stages<float> sm;
  if (*bad) return;
  const int np = n + 1, i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  tile_product<float, true, true>(sm, i0, j0, j0, n, [&](int i, int k) { return i < rows ? y[static_cast<int64_t>(i) * n + k] : 0.f; },
      [&](int k, int j) { return j < n && k >= j ? Wimg[j * np + k] : 0.f; },
      [&](int i, int j, float v) {
        if (i >= rows || j >= n) return;
        const int64_t o = static_cast<int64_t>(i) * n + j;
        if (core) core[static_cast<int64_t>(i) * n + (j % Rl) * Rr + j / Rl] = static_cast<double>(add[o] + v);
        else z[o] = v;
      });
}

// r = b - M z (M symmetric, FP32 image M[k * np + j]).
__global__ void __launch_bounds__(GNT) k_sv_residual(int n, const float* __restrict__ Mimg,
                                                     const int* bad, int rows,
                                                     const double* __restrict__ b, int64_t ld,
                                                     const float* __restrict__ z,
                                                     float* __restrict__ r) {
  grid_wait();
  __shared__ Stages<float> sm;
  if (*bad) return;
  const int np = n + 1, i0 = blockIdx.y * GE, j0 = blockIdx.x * GE;
  tile_product<float, true, false>(sm, i0, j0, 0, n, [&](int i, int k) { return i < rows ? z[static_cast<int64_t>(i) * n + k] : 0.f; },
      [&](int k, int j) { return j < n ? Mimg[k * np + j] : 0.f; },
      [&](int i, int j, float v) {
        if (i < rows && j < n) r[static_cast<int64_t>(i) * n + j] = static_cast<float>(b[i * ld + j]) - v;
      });
}

constexpr double kEps32 = 1.1920928955078125e-07;

__global__ void __launch_bounds__(kCiMaxThreads) k_small_factor(int n, float tol,
                                                                const float* pre, int lda,
                                                                float* Ximg, int* bad) {
  grid_wait();
  __shared__ CiShared cs;
  const bool ok = chol_inv_tiles(n, tol, pre, lda, Ximg, n + 1, pre, n, lda, cs);
  if (threadIdx.x == 0) { bad[0] = ok ? 0 : 1; bad[1] = ok ? 0 : 1; }
}

// From about here on the products beat the one-CTA FP64 factorisation and the FP64 substitutions. Whole
// calls, 300 rows: n = 88: 191 -> 151 us, 100: 224 -> 160, 144: 402 -> 230, 256: 2285 -> 402. Where the
// products are refused the call pays for both forms: a few us when a pivot is too small, the
// FP32 inverse, U and E when ||E|| is too large (cond(K) of 1e5 and more): 240, 277, 507 and 1995 us.
constexpr int kLev64MinN = 88;

constexpr int64_t kMaxRows = 1 << 18;      // rows per launch: tiles in a grid's second dimension
unsigned dtiles(int64_t n) { return static_cast<unsigned>((n + DE - 1) / DE); }

L64 args_of(const Lev64& w, int n) {
  const size_t nn = static_cast<size_t>(n) * n;
  return L64{n, w.Ximg, w.G, w.E, w.partial, w.partial + nn, w.partial + 2 * nn, w.bad, w.keep,
             w.info, w.tau * w.tau};
}

unsigned tiles_of(int64_t n) { return static_cast<unsigned>((n + GE - 1) / GE); }

}  // namespace

// The one-CTA panel factorisation holds up to 160 columns in registers (L = 144: 61 us and 59 us of
// substitutions, 77 and 55 here); beyond it works from L2 (L = 224: 399 + 89, here 104 + 72).
constexpr int kSolveBigMin = 160;
bool solve_big_fits(int L) { return L > kSolveBigMin && L <= kMaxL; }

bool inv256_fits(int n) { return n > kCiMaxN && n <= kMaxL; }

cudaError_t launch_inv256(int n, double tol_scale, const float* pre, int lda, float* Ximg,
                          float* scratch, int* bad, int* keep, int* info, const unsigned* err,
                          cudaStream_t st) {
  if (!inv256_fits(n)) return cudaErrorInvalidValue;
  BigInv g{};
  g.pre = pre;
  g.n = n;
  g.lda = lda;
  g.n1 = n - kCiMaxN >= 4 ? kCiMaxN : kCiMaxN - 4;      // both blocks have at least 4 rows
  const int n2 = n - g.n1;
  g.Ximg = Ximg;
  g.lds = (n2 + 3) & ~3;
  g.S = scratch;                                         // 16-byte aligned columns
  g.Lb = scratch + static_cast<int64_t>(n2) * g.lds;
  g.T = g.Lb + static_cast<int64_t>(n2) * g.n1;
  g.bad = bad;
  const float tol = static_cast<float>(tol_scale);
  const dim3 lb(tiles_of(g.n1), tiles_of(n2));
  launch_pdl(k_big_factor, 1, chol_inv_threads(g.n1), 0, st, g, tol, 0, nullptr, info, err);
  launch_pdl(k_big_lb, lb, GNT, 0, st, g);
  launch_pdl(k_big_s, dim3(tiles_of(n2), tiles_of(n2)), GNT, 0, st, g);
  launch_pdl(k_big_factor, 1, chol_inv_threads(n2), 0, st, g, tol, 1, keep, info, nullptr);
  launch_pdl(k_big_t, lb, GNT, 0, st, g);
  launch_pdl(k_big_x21, lb, GNT, 0, st, g);
  return cudaGetLastError();
}

cudaError_t launch_solve_big(int n, const float* Wimg, const float* Mimg, const int* bad,
                             int64_t nvec, const double* rhs, int64_t ld, int Rl, int Rr,
                             double* core_out, float* scratch, int64_t rows, cudaStream_t st) {
  if (rows > kMaxRows) rows = kMaxRows;
  for (int64_t r0 = 0; r0 < nvec; r0 += rows) {
    const int m = static_cast<int>(nvec - r0 < rows ? nvec - r0 : rows);
    float* y = scratch;
    float* z = y + static_cast<int64_t>(m) * n;
    float* r = z + static_cast<int64_t>(m) * n;
    const double* b = rhs + r0 * ld;
    const dim3 grid(tiles_of(n), tiles_of(m));
    launch_pdl(k_sv_lower<double>, grid, GNT, 0, st, n, Wimg, bad, m, b, ld, y);
    launch_pdl(k_sv_upper, grid, GNT, 0, st, n, Wimg, bad, m, y, nullptr, z, Rl, Rr, nullptr);
    launch_pdl(k_sv_residual, grid, GNT, 0, st, n, Mimg, bad, m, b, ld, z, r);
    launch_pdl(k_sv_lower<float>, grid, GNT, 0, st, n, Wimg, bad, m, r, n, y);
    launch_pdl(k_sv_upper, grid, GNT, 0, st, n, Wimg, bad, m, y, z, nullptr, Rl, Rr, core_out + r0 * n);
  }
  return cudaGetLastError();
}

// (The same line for the FP64 LS step, whole calls of 30 right-hand sides, J = 9 L, substitutions
// against V: L = 88: 210 -> 188 us, L = 100: 253 -> 203, L = 256: 2645 -> 563; L = 81 was equal.)
// A right-hand side costs three products here and one in the substitutions, which many of them keep
// busy: the forms break even at about 550 right-hand sides for L = 88 and 90, 830 for 100, 900 for
// 121, 1160 for 144, and, where the factor no longer fits one SM's shared memory, 2260 for 169, 3400
// for 196, 5400 for 225 and 8600 for 256 (I = 1000: L = 90: 349 us by substitutions, 384 with V,
// L = 169: 1194 and 997; I = 10000: L = 256: 13.8 and 14.1 ms).
bool solve_f64_fits(int64_t I, int n, int splits) {
  return n >= kLev64MinN && n <= kMaxL && I <= (n > kSolveBigMin ? 12 : 6) * n &&
         static_cast<int64_t>(splits) * (n + I) >= 3 * static_cast<int64_t>(n) + 1;
}

cudaError_t launch_solve_f64(const Lev64& w, int n, const double* rhs, int64_t ld, int64_t I, int Rl,
                             int Rr, double* core_out, cudaStream_t st) {
  const L64 g = args_of(w, n);
  const unsigned nt = dtiles(n);
  launch_pdl(k_l64_inv, nt * (nt + 1) / 2, DNT, 0, st, g);
  double* r = g.P;        // behind V: room for splits * (n + I) - n >= I rows
  const int m = static_cast<int>(I);
  const dim3 grid(nt, dtiles(m));
  launch_pdl(k_l64_z, grid, DNT, 0, st, g, rhs, ld, m, Rl, Rr, core_out, false);
  launch_pdl(k_l64_r, grid, DNT, 0, st, g, rhs, ld, m, Rl, Rr, core_out, r);
  launch_pdl(k_l64_z, grid, DNT, 0, st, g, r, static_cast<int64_t>(n), m, Rl, Rr, core_out, true);
  return cudaGetLastError();
}

// A row costs one product here (n^2 multiply-adds, in tiles) and half of that in the substitutions,
// which many rows keep busy. Break-even by whole calls: I = 3000 for n = 90, 5800 for 100, 7000 for 121
// and 144 (I = 20000, n = 100: 1157 us here, 977 by substitutions), and, where the factor no longer
// fits one SM's shared memory, 10500 for 169, 12500 for 196, 19000 for 225 and 32000 for 256
// (I = 5000: 877 us here and 1081 for 169, 1453 and 2838 for 256; I = 50000: 6.8 and 5.2 ms, 11.1 and
// 10.2).
bool leverage_f64_fits(int64_t I, int n, int splits) {
  return n >= kLev64MinN && n <= kMaxL && I >= n && I <= (n > kSolveBigMin ? 64 : 32) * n && splits >= 4;
}

cudaError_t launch_leverage_f64(int part, const Lev64& w, const double* A, int64_t I, int n,
                                int64_t lda, double* ell, const CdfEpilogue& ep, cudaStream_t st) {
  const double tol = n * kEps32;
  const size_t nn = static_cast<size_t>(n) * n;
  const L64 g = args_of(w, n);
  const unsigned nt = dtiles(n), up = nt * (nt + 1) / 2;
  if (part == 1) {
    // rows per launch by the room for their partial sums, behind X'
    double* sums = w.partial + 3 * nn;
    const int64_t room = static_cast<int64_t>((w.splits - 3) * nn / nt) / DE * DE;
    const int64_t most = room < kMaxRows ? room : kMaxRows;
    for (int64_t r0 = 0; r0 < I; r0 += most) {
      const int m = static_cast<int>(I - r0 < most ? I - r0 : most);
      CdfEpilogue e2 = ep;
      if (r0 + m < I) e2.p = nullptr;
      launch_pdl(k_l64_rows, dim3(nt, dtiles(m)), DNT, 0, st, g, A + r0 * lda, lda, m, sums);
      launch_pdl(k_l64_finish, 1, kFinishThreads, 0, st, g, sums, static_cast<int>(nt), m, r0, ell, I, e2);
    }
    return cudaGetLastError();
  }
  if (inv256_fits(n)) {
    const cudaError_t e = launch_inv256(n, tol, w.K32, w.ldk, w.Ximg, reinterpret_cast<float*>(g.U),
                                        w.bad, nullptr, nullptr, nullptr, st);
    if (e != cudaSuccess) return e;
  } else {
    launch_pdl(k_small_factor, 1, chol_inv_threads(n), 0, st, n, static_cast<float>(tol), w.K32,
               w.ldk, w.Ximg, w.bad);
  }
  launch_pdl(k_l64_u, dim3(nt, nt), DNT, 0, st, g);
  launch_pdl(k_l64_e, up, DNT, 0, st, g);
  launch_pdl(k_l64_e2, up, DNT, 0, st, g);
  for (int k = 1; k < 4; ++k) launch_pdl(k_l64_poly, up, DNT, 0, st, g, k);
  launch_pdl(k_l64_poly, dim3(nt, nt), DNT, 0, st, g, 4);
  return cudaGetLastError();
}

}  // namespace trk
