// Row a5: normal-equation contractions of the sampled LS (Alg. 2, LS step):
//   M = A~^T A~ (L x L),  B = A~^T Y~ (L x I),
// computed together as C = A~^T [A~ | Y~] with the J rows split into chunks; each chunk
// writes its own partial C so that the reduction order downstream is fixed (results do
// not depend on scheduling).
//
// SIMT tiles: 64 x 64 outputs per CTA in FP32, 32 x 32 in FP64, 16 rows of J per shared-memory
// stage, the next stage's values in flight while one is multiplied. T = float accumulates in
// FP32 within a chunk; T = double in FP64, where the FP64 pipe (2 multiply-adds per clock and
// SM) is the bound: work on padding and idle SMs cost directly. With 64 x 64 tiles J = 2000,
// L = 25, I = 100 ran on 64 of 152 SMs with 61% of the rows padding (78 us); with 32 x 32 on 128
// (23 us). A tile below M's diagonal is not computed but written by its mirror image
// (J = 2000, L = 100, I = 4: 77 -> 74 us). The chunks, and with them every sum, are the same.
#include "common.cuh"

namespace trk {
namespace {

constexpr int BK = 16, NT = 256;

// Edge of an output tile, by type.
constexpr int tile_edge(bool f64) { return f64 ? 32 : 64; }

template <typename T>
__global__ void __launch_bounds__(NT) k_normal_eq(const T* __restrict__ A,
                                                  const T* __restrict__ Y, int64_t J, int L,
                                                  int64_t I, int64_t chunk,
                                                  T* __restrict__ partial,
                                                  const int64_t* __restrict__ jdev) {
  constexpr int BM = tile_edge(sizeof(T) == 8), BN = BM, U = BM / 16, V = BN / 16;
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
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // 16 x 16 threads
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
      for (int u = 0; u < U; ++u) a[u] = As[s][kk][ty + 16 * u];
#pragma unroll
      for (int v = 0; v < V; ++v) b[v] = Bs[s][kk][tx + 16 * v];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[u][v] += a[u] * b[v];
    }
  }
  T* out = partial + static_cast<int64_t>(blockIdx.z) * L * ldc;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = r0 + ty + 16 * u;
    if (r >= L) continue;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int64_t c = c0 + tx + 16 * v;
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
  const int b = tile_edge(f64);
  dim3 grid(static_cast<unsigned>((L + I + b - 1) / b), (L + b - 1) / b, s);
  if (f64)
    k_normal_eq<double><<<grid, NT, 0, st>>>(static_cast<const double*>(A),
                                             static_cast<const double*>(Y), J, L, I, chunk,
                                             static_cast<double*>(partial), jdev);
  else
    k_normal_eq<float><<<grid, NT, 0, st>>>(static_cast<const float*>(A),
                                            static_cast<const float*>(Y), J, L, I, chunk,
                                            static_cast<float*>(partial), jdev);
  return cudaGetLastError();
}

}  // namespace trk
