// Row a5: normal-equation contractions of the sampled LS (Alg. 2, LS step):
//   M = A~^T A~ (L x L),  B = A~^T Y~ (L x I),
// computed together as C = A~^T [A~ | Y~] with the J rows split into chunks; each chunk
// writes its own partial C so that the reduction order downstream is fixed (results do
// not depend on scheduling).
//
// SIMT tiles: 64 x 64 outputs per CTA in FP32, 32 x 32 or 16 x 16 in FP64, 16 rows of J per
// shared-memory stage, the next stage's values in flight while one is multiplied. T = float
// accumulates in FP32 within a chunk; T = double in FP64, where the FP64 pipe (2 multiply-adds
// per clock and SM) is the bound: work on padding and idle SMs cost directly. With 64 x 64 tiles
// J = 2000, L = 25, I = 100 ran on 64 of 152 SMs with 61% of the rows padding (78 us); with
// 32 x 32 on 128 (23 us). A tile below M's diagonal is not computed but written by its mirror
// image. 16 x 16 where that leaves the busiest SM less to do: J = 2000, L = 100, I = 4 is 160
// tiles of 32 x 32, two on 8 of the SMs (74 us), or 560 of 16 x 16, four at most (28 us). The
// chunks, and with them every sum, are the same.
#include "common.cuh"

namespace trk {
namespace {

constexpr int BK = 16;

// Threads along an edge of a BM x BM tile.
constexpr int tile_threads(int bm) { return bm < 32 ? 8 : 16; }

template <typename T, int BM>
__global__ void __launch_bounds__(tile_threads(BM) * tile_threads(BM)) k_normal_eq(const T* __restrict__ A,
                                                  const T* __restrict__ Y, int64_t J, int L,
                                                  int64_t I, int64_t chunk,
                                                  T* __restrict__ partial,
                                                  const int64_t* __restrict__ jdev) {
  grid_wait();
  constexpr int BN = BM, TE = tile_threads(BM), NT = TE * TE, U = BM / TE, V = BN / TE;
  __shared__ T As[2][BK][BM];
  __shared__ T Bs[2][BK][BN];
  const int64_t ldc = L + I;
  const int r0 = blockIdx.y * BM;
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * BN;
  // FP64: entirely below the diagonal of M (the mirror tile writes it)
  constexpr bool kMirror = sizeof(T) == 8;
  if (kMirror && c0 + BN <= r0) return;
  const int64_t j0 = static_cast<int64_t>(blockIdx.z) * chunk;
  const int64_t Jr = jdev ? (*jdev < J ? *jdev : J) : J;
  const int64_t j1 = (j0 + chunk < Jr) ? j0 + chunk : Jr;
  const int tx = threadIdx.x % TE, ty = threadIdx.x / TE;
  T acc[U][V];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < V; ++v) acc[u][v] = T(0);
  constexpr int NA = (BK * BM) / NT, NB = (BK * BN) / NT;
  T ra[NA], rb[NB];                       // the next stage, in flight
  auto load = [&](int64_t jb) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = threadIdx.x + q * NT;
      const int64_t j = jb + e / BM;
      const int r = r0 + e % BM;
      ra[q] = (j < j1 && r < L) ? A[j * L + r] : T(0);
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = threadIdx.x + q * NT;
      const int64_t j = jb + e / BN, c = c0 + e % BN;
      rb[q] = T(0);
      if (j < j1) {
        if (c < L) rb[q] = A[j * L + c];
        else if (c < ldc) rb[q] = Y[j * I + (c - L)];
      }
    }
  };
  if (j0 < j1) load(j0);
  int s = 0;
  for (int64_t jb = j0; jb < j1; jb += BK, s ^= 1) {
#pragma unroll
    for (int q = 0; q < NA; ++q) (&As[s][0][0])[threadIdx.x + q * NT] = ra[q];
#pragma unroll
    for (int q = 0; q < NB; ++q) (&Bs[s][0][0])[threadIdx.x + q * NT] = rb[q];
    __syncthreads();       // the stage is written; its previous readers passed the last barrier
    if (jb + BK < j1) load(jb + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[U], b[V];
#pragma unroll
      for (int u = 0; u < U; ++u) a[u] = As[s][kk][ty + TE * u];
#pragma unroll
      for (int v = 0; v < V; ++v) b[v] = Bs[s][kk][tx + TE * v];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[u][v] += a[u] * b[v];
    }
  }
  T* out = partial + static_cast<int64_t>(blockIdx.z) * L * ldc;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = r0 + ty + TE * u;
    if (r >= L) continue;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int64_t c = c0 + tx + TE * v;
      if (c < ldc) out[static_cast<int64_t>(r) * ldc + c] = acc[u][v];
      // the mirror image of an entry whose own tile was not computed
      if (kMirror && c < L && r / BN * BN + BN <= c / BM * BM)
        out[c * ldc + r] = acc[u][v];
    }
  }
}

// Chunks of the samples, laid down for 64 x 64 tiles (four CTAs per SM, at least 64 rows).
void plan(int64_t J, int L, int64_t I, int* splits, int64_t* chunk) {
  const int64_t tiles = ((L + 63) / 64) * ((L + I + 63) / 64);
  int64_t s = (4 * sm_count() + tiles - 1) / tiles;
  const int64_t maxs = (J + 63) / 64;  // at least 64 rows per chunk
  if (s > maxs) s = maxs;
  if (s < 1) s = 1;
  int64_t c = (J + s - 1) / s;
  c = (c + BK - 1) / BK * BK;
  s = (J + c - 1) / c;
  *splits = static_cast<int>(s);
  *chunk = c;
}

template <typename T, int BM>
void go(const void* A, const void* Y, int64_t J, int L, int64_t I, int64_t chunk, void* partial,
        int splits, cudaStream_t st, const int64_t* jdev) {
  const dim3 grid(static_cast<unsigned>((L + I + BM - 1) / BM), (L + BM - 1) / BM, splits);
  launch_pdl((k_normal_eq<T, BM>), grid, tile_threads(BM) * tile_threads(BM), 0, st,
             static_cast<const T*>(A), static_cast<const T*>(Y), J, L, I, chunk,
             static_cast<T*>(partial), jdev);
}

}  // namespace

size_t normal_eq_workspace(int64_t J, int L, int64_t I, bool f64, int* splits) {
  int64_t chunk;
  plan(J, L, I, splits, &chunk);
  return static_cast<size_t>(*splits) * L * (L + I) * (f64 ? 8 : 4);
}

cudaError_t launch_normal_eq(const void* A, const void* Y, bool f64, int64_t J, int L,
                             int64_t I, void* partial, int splits, cudaStream_t st,
                             const int64_t* jdev) {
  int s;
  int64_t chunk;
  plan(J, L, I, &s, &chunk);
  if (s != splits) return cudaErrorInvalidValue;
  if (f64) {
    // the busiest SM's multiply-adds with tiles of edge b (those below M's diagonal left out)
    auto share = [&](int64_t b) {
      const int64_t rows = (L + b - 1) / b, ctas = (rows * ((L + I + b - 1) / b) - rows * (rows - 1) / 2) * s;
      return (ctas + sm_count() - 1) / sm_count() * b * b;
    };
    if (share(16) < share(32)) go<double, 16>(A, Y, J, L, I, chunk, partial, s, st, jdev);
    else go<double, 32>(A, Y, J, L, I, chunk, partial, s, st, jdev);
  } else {
    go<float, 64>(A, Y, J, L, I, chunk, partial, s, st, jdev);
  }
  return cudaGetLastError();
}

}  // namespace trk
