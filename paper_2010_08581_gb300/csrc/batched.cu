// Batched stages of TR-ALS-Sampled (Alg. 2 per instance, Alg. 3 + Alg. 4 for the sketch):
// one launch per stage for every instance of the table; see batched.cuh. This file holds
// the initial cores, the draws with their rows and fibres, the normal-equation contraction
// and the leverage Grams; the factorisations, solves and fit live in batched_chol.cu,
// batched_solve.cu and batched_fit.cu.
#include "batched_kern.cuh"
#include "draw.cuh"

namespace trk {
namespace {

// ------------------------------------------------------------------------------------
// Initial cores N(0,1) (same stream as launch_init_normal: stream id = core index).
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) kb_init_cores(const BInst* __restrict__ tab) {
  const BInst& d = tab[blockIdx.x];
  if (!d.draw_init) return;
  if (d.slot) {
    if (d.slot->status != kSlotRunning || d.slot->step != 1 - d.N) return;
  } else if (d.nupd <= 0) {
    return;
  }
  const uint32_t k0 = static_cast<uint32_t>(d.seed), k1 = static_cast<uint32_t>(d.seed >> 32);
  for (int k = 1; k < d.N; ++k) {
    const int64_t count = d.dims[k] * d.ranks[(k - 1 + d.N) % d.N] * d.ranks[k];
    const int64_t pairs = (count + 1) / 2;
    double* out = d.cores[k];
    for (int64_t q = static_cast<int64_t>(blockIdx.y) * blockDim.x + threadIdx.x; q < pairs;
         q += static_cast<int64_t>(gridDim.y) * blockDim.x) {
      double z0, z1;
      normal_pair(q, static_cast<uint32_t>(k), k0, k1, &z0, &z1);
      out[2 * q] = z0;
      if (2 * q + 1 < count) out[2 * q + 1] = z1;
    }
  }
}

// ------------------------------------------------------------------------------------
// Draws (Alg. 3), sampled subchain rows (Alg. 4) and sampled fibres (Alg. 2) for one chunk
// of one instance's samples: first one thread per draw (a binary search is a chain of dependent
// loads, about 5 us: all of a CTA's run at once), then one warp per sample, the fibre's scattered
// loads in flight while the slices are multiplied. 512 problems of I = 32 .. 200, J = 160 .. 640:
// 522 us with each warp drawing, multiplying and loading in turn (this and the Gram below took
// 340 us off a step of 1.9 ms).
// ------------------------------------------------------------------------------------
constexpr int SW = 8;     // warps per CTA
constexpr int kSpwMax = 8;   // samples per warp: a launch parameter in [1, 8] (tiles)
constexpr int kFibre = 8;    // fibre entries per lane that are loaded ahead

template <typename T, typename TX>
__global__ void __launch_bounds__(SW * 32) kb_sample(const BInst* __restrict__ tab, int step,
                                                     int spw) {
  __shared__ T sS[SW][kMaxL];
  __shared__ T sG[SW][kMaxL];
  __shared__ ChainArgs ca;
  __shared__ int idx[SW * kSpwMax][kMaxModes];       // the draws of each sample
  __shared__ double prob[SW * kSpwMax][kMaxModes];
  __shared__ int64_t fibre[SW * kSpwMax];
  __shared__ T weight[SW * kSpwMax];
  const BInst& d = tab[blockIdx.x];
  const Cur cu = current(d, step, 0, false);
  if (!cu.active) return;
  const int64_t j0 = static_cast<int64_t>(blockIdx.y) * SW * spw;
  if (j0 >= d.J) return;
  const int N = d.N, npos = N - 1, n = cu.n;
  if (threadIdx.x == 0) {
    ca.npos = npos;
    for (int m = 0; m < npos; ++m) {
      const int mode = (n + 1 + m) % N;
      ca.core[m] = d.cores[mode];
      ca.I[m] = d.dims[mode];
      ca.rl[m] = d.ranks[(mode - 1 + N) % N];
      ca.rr[m] = d.ranks[mode];
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t k0 = static_cast<uint32_t>(d.seed), k1 = static_cast<uint32_t>(d.seed >> 32);
  const uint32_t u0 = static_cast<uint32_t>(cu.t), u1 = 0u;
  const int count = d.J - j0 < SW * spw ? static_cast<int>(d.J - j0) : SW * spw;
  for (int e = threadIdx.x; e < count * npos; e += SW * 32) {
    const int s = e / npos, m = e - s * npos;
    const int mode = (n + 1 + m) % N;
    const double u = draw_uniform(j0 + s, m, k0, k1, u0, u1);
    int64_t i;
    double pi = 1.0;
    if (d.uniform) {
      i = uniform_index(d.dims[mode], u);
    } else {
      i = inverse_cdf(d.cdf[mode], d.p[mode], d.dims[mode], u);
      pi = d.p[mode][i];
    }
    idx[s][m] = static_cast<int>(i);
    prob[s][m] = pi;
  }
  __syncthreads();
  if (threadIdx.x < static_cast<unsigned>(count)) {
    const int s = threadIdx.x;
    int64_t off = 0;
    for (int m = 0; m < npos; ++m) off += idx[s][m] * d.stride[(n + 1 + m) % N];
    fibre[s] = off;
    const double w = d.uniform ? uniform_weight(d.J, ca.I, npos) : sample_weight(d.J, prob[s], npos);
    weight[s] = static_cast<T>(w);
  }
  __syncthreads();
  const TX* __restrict__ X = static_cast<const TX*>(d.X);
  T* A = static_cast<T*>(d.A);
  T* Y = static_cast<T*>(d.Y);
  const int L = cu.L;
  const int64_t I = cu.I, sn = d.stride[n];
  for (int s = warp; s < count; s += SW) {
    const int64_t j = j0 + s;
    const TX* src = X + fibre[s];
    TX ahead[kFibre];
#pragma unroll
    for (int q = 0; q < kFibre; ++q) {
      const int64_t e = lane + 32 * q;
      ahead[q] = e < I ? src[e * sn] : TX(0);
    }
    auto index = [&](int m) -> int64_t { return idx[s][m]; };
    warp_slice_chain<T>(ca, index, sS[warp], sG[warp], lane);
    const T scale = weight[s];
    for (int e = lane; e < L; e += 32) A[j * L + e] = sS[warp][e] * scale;
#pragma unroll
    for (int q = 0; q < kFibre; ++q) {
      const int64_t e = lane + 32 * q;
      if (e < I) Y[j * I + e] = static_cast<T>(static_cast<T>(ahead[q]) * scale);
    }
    for (int64_t e = lane + 32 * kFibre; e < I; e += 32)
      Y[j * I + e] = static_cast<T>(static_cast<T>(src[e * sn]) * scale);
    __syncwarp();
  }
}

// ------------------------------------------------------------------------------------
// Normal equations C = A^T [A | Y] per instance, square output tiles over all samples
// (no split: one fixed summation order per entry); M = C[:, :L], B^T = C[:, L:]^T in FP64.
// ------------------------------------------------------------------------------------
// 4 x 4 outputs per thread over a TILE x TILE tile (2 x 4 over TILE / 2 rows where the instance
// has no more unknowns than that). The next 16 samples are in registers while the current ones
// are multiplied from one of two shared-memory stages: with one stage and no prefetch every 16
// samples waited for their loads (J = 2560: 459 us of 16 CTA-rows that ran alone on an SM).
// Every entry is one chain of multiply-adds over the samples in order whatever the tile (a
// launch parameter), so the tile never changes results.
constexpr int BK = 16;

template <typename T, int TILE, int U>
__device__ __forceinline__ void contract_tile_cta(const BInst& d, const Cur& cu, T* smem) {
  constexpr int TXN = TILE / 4, CT = TXN * TXN, BM = TXN * U, BN = TILE;
  constexpr int NA = (BK * BM + CT - 1) / CT, NB = (BK * BN) / CT;
  T* As = smem;                       // [2][BK][BM]
  T* Bs = smem + 2 * BK * TILE;       // [2][BK][BN]
  const int L = cu.L;
  const int64_t I = cu.I, ldc = L + I;
  const int ntr = (L + BM - 1) / BM;
  const int ntc = static_cast<int>((ldc + BN - 1) / BN);
  const int t = blockIdx.y;
  if (t >= ntr * ntc) return;
  const int r0 = (t / ntc) * BM;
  const int64_t c0 = static_cast<int64_t>(t % ntc) * BN;
  const T* __restrict__ A = static_cast<const T*>(d.A);
  const T* __restrict__ Y = static_cast<const T*>(d.Y);
  const int64_t J = d.J;
  const int tx = threadIdx.x % TXN, ty = threadIdx.x / TXN;
  T ra[NA], rb[NB];
  auto load = [&](int64_t jb) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = threadIdx.x + q * CT;
      const int kk = e / BM, r = r0 + e % BM;
      const int64_t j = jb + kk;
      ra[q] = (kk < BK && j < J && r < L) ? A[j * L + r] : T(0);
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = threadIdx.x + q * CT;
      const int64_t j = jb + e / BN, c = c0 + e % BN;
      rb[q] = T(0);
      if (j < J) {
        if (c < L) rb[q] = A[j * L + c];
        else if (c < ldc) rb[q] = Y[j * I + (c - L)];
      }
    }
  };
  T acc[U][4];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = T(0);
  load(0);
  int s = 0;
  for (int64_t jb = 0; jb < J; jb += BK, s ^= 1) {
    T* as = As + s * (BK * TILE);
    T* bs = Bs + s * (BK * TILE);
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = threadIdx.x + q * CT;
      if (NA * CT == BK * BM || e < BK * BM) as[e] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) bs[threadIdx.x + q * CT] = rb[q];
    __syncthreads();       // the stage is written; its previous readers passed the last barrier
    if (jb + BK < J) load(jb + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[U], b[4];
#pragma unroll
      for (int u = 0; u < U; ++u) a[u] = as[kk * BM + ty * U + u];
#pragma unroll
      for (int v = 0; v < 4; ++v) b[v] = bs[kk * BN + tx * 4 + v];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] += a[u] * b[v];
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = r0 + ty * U + u;
    if (r >= L) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int64_t c = c0 + tx * 4 + v;
      if (c < L) d.M[static_cast<int64_t>(r) * L + c] = static_cast<double>(acc[u][v]);
      else if (c < ldc) d.BT[(c - L) * L + r] = static_cast<double>(acc[u][v]);
    }
  }
}

template <typename T, int TILE>
__global__ void __launch_bounds__((TILE / 4) * (TILE / 4)) kb_contract(
    const BInst* __restrict__ tab, int step) {
  __shared__ __align__(16) T smem[4 * BK * TILE];
  const BInst& d = tab[blockIdx.x];
  const Cur cu = current(d, step, 0, false);
  if (!cu.active) return;
  if (cu.L <= TILE / 2) contract_tile_cta<T, TILE, 2>(d, cu, smem);
  else contract_tile_cta<T, TILE, 4>(d, cu, smem);
}

// ------------------------------------------------------------------------------------
// Gram matrices of the leverage passes (FP64, full square, 32 x 32 tiles over all rows).
//   pass 1, tall (I >= L): G1 = S^T S (L x L); wide: G1 = S S^T (I x I), S = the I x L rows
//           (the core at initialisation and, under the column-dropping LS rule, after each
//           update; B^T during the updates otherwise);
//   pass 2 (wide modes only): G2 = C^T C (I x I), C = the pass-1 factor.
// ------------------------------------------------------------------------------------
constexpr int GK = 16, GNT = 256;     // a thread holds at most one 2 x 2 block; all of them load

// The 2 x 2 blocks of G's upper triangle, row by row, are dealt out to the CTAs of blockIdx.y, `per`
// each, and their threads, GK rows of the matrix at a time in shared memory;
// the lower triangle is written by its mirror image. The FP64 pipe is the bound, so there is no
// work on padding beyond the last warp: 32 x 32 tiles of the whole square took 174 .. 310 us for
// 512 cores of L = 9 .. 64, I = 32 .. 200. Every entry is one chain over the rows
// in order, as before.
__host__ __device__ inline int gram_blocks(int n) { const int h = (n + 1) / 2; return h * (h + 1) / 2; }

__global__ void __launch_bounds__(GNT) kb_gram(const BInst* __restrict__ tab, int step, int init_k,
                                               int pass, int from_core, int per) {
  __shared__ __align__(16) double P[GK * kMaxL];
  const BInst& d = tab[blockIdx.x];
  const Cur cu = current(d, step, init_k, true);
  if (!cu.active) return;
  const bool tall = cu.I >= cu.L;
  if (pass == 2 && tall) return;
  const double* S = (cu.init || from_core) ? d.cores[cu.n] : d.BT;
  const double* src;
  int64_t K, lda;
  int n;
  bool trans;
  double* G;
  if (pass == 1) {
    src = S; lda = cu.L; G = d.G1;
    if (tall) { n = cu.L; K = cu.I; trans = false; }
    else { n = static_cast<int>(cu.I); K = cu.L; trans = true; }
  } else {
    src = d.L1row; lda = cu.I; G = d.G2;
    n = static_cast<int>(cu.I); K = cu.I; trans = false;
  }
  const int h = (n + 1) / 2, blocks = gram_blocks(n);
  const int parts = (blocks + per - 1) / per;
  if (static_cast<int>(blockIdx.y) >= parts) return;
  const int b0 = static_cast<int>(static_cast<int64_t>(blocks) * blockIdx.y / parts);
  const int b1 = static_cast<int>(static_cast<int64_t>(blocks) * (blockIdx.y + 1) / parts);
  const int ld = 2 * h;               // an even row length: aligned pairs
  int row = -1, col = 0, rest = b0 + static_cast<int>(threadIdx.x);
  double acc[2][2] = {};
  if (rest < b1) {
    int r = 0;
    while (rest >= h - r) { rest -= h - r; ++r; }
    row = 2 * r;
    col = 2 * (r + rest);
  }
  for (int64_t kb = 0; kb < K; kb += GK) {
    for (int e = threadIdx.x; e < GK * ld; e += GNT) {
      int kk, c;
      if (!trans) { kk = e / ld; c = e - kk * ld; } else { c = e / GK; kk = e % GK; }
      const int64_t k = kb + kk;
      P[kk * ld + c] = k < K && c < n ? (trans ? src[c * lda + k] : src[k * lda + c]) : 0.0;
    }
    __syncthreads();
    if (row >= 0) {
#pragma unroll 4
      for (int kk = 0; kk < GK; ++kk) {
        const double2 x = *reinterpret_cast<const double2*>(P + kk * ld + row);
        const double2 y = *reinterpret_cast<const double2*>(P + kk * ld + col);
        acc[0][0] += x.x * y.x;
        acc[0][1] += x.x * y.y;
        acc[1][0] += x.y * y.x;
        acc[1][1] += x.y * y.y;
      }
    }
    __syncthreads();
  }
  if (row < 0) return;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = row + u, c = col + v;
      if (r >= n || c >= n) continue;
      G[static_cast<int64_t>(r) * n + c] = acc[u][v];
      G[static_cast<int64_t>(c) * n + r] = acc[u][v];
    }
}

}  // namespace

cudaError_t bl_init_cores(const BLaunch& b, cudaStream_t st) {
  dim3 grid(b.count, 16);
  kb_init_cores<<<grid, 256, 0, st>>>(b.tab);
  return cudaGetLastError();
}

cudaError_t bl_sample_chain_gather(const BLaunch& b, int step, cudaStream_t st) {
  const int spw = b.spw >= 1 && b.spw <= kSpwMax ? b.spw : 4;
  const int64_t per = SW * spw;
  dim3 grid(b.count, static_cast<unsigned>((b.Jmax + per - 1) / per));
  if (b.f64 && b.xf64) kb_sample<double, double><<<grid, SW * 32, 0, st>>>(b.tab, step, spw);
  else if (b.f64) kb_sample<double, float><<<grid, SW * 32, 0, st>>>(b.tab, step, spw);
  else if (b.xf64) kb_sample<float, double><<<grid, SW * 32, 0, st>>>(b.tab, step, spw);
  else kb_sample<float, float><<<grid, SW * 32, 0, st>>>(b.tab, step, spw);
  return cudaGetLastError();
}

template <int TILE>
cudaError_t contract_tile(const BLaunch& b, int step, cudaStream_t st) {
  const int ntr = (b.Lmax + TILE - 1) / TILE;
  const int64_t ntc = (b.Lmax + b.Imax + TILE - 1) / TILE;
  dim3 grid(b.count, static_cast<unsigned>(ntr * ntc));
  constexpr int CT = (TILE / 4) * (TILE / 4);
  if (b.f64) kb_contract<double, TILE><<<grid, CT, 0, st>>>(b.tab, step);
  else kb_contract<float, TILE><<<grid, CT, 0, st>>>(b.tab, step);
  return cudaGetLastError();
}

cudaError_t bl_contract(const BLaunch& b, int step, cudaStream_t st) {
  return b.ctile == 32 ? contract_tile<32>(b, step, st) : contract_tile<64>(b, step, st);
}

cudaError_t bl_gram(const BLaunch& b, int step, int init_k, int pass, cudaStream_t st) {
  const int nmax = pass == 1 ? b.n1max : b.n2max;
  if (nmax <= 0) return cudaSuccess;
  // 128 blocks a CTA, 64 where the problems alone do not fill the SMs: one SM's FP64 pipe takes
  // 150 us for 512 blocks of 300 rows, 19 us for 64, and the largest problems of a batch end last
  // (512 problems: 180 us with 512 blocks, 135 with 128)
  const int per = b.count >= 2 * sm_count() ? 128 : 64;
  dim3 grid(b.count, (gram_blocks(nmax) + per - 1) / per);
  kb_gram<<<grid, GNT, 0, st>>>(b.tab, step, init_k, pass, b.ls_mode == 1 ? 1 : 0, per);
  return cudaGetLastError();
}

cudaError_t batched_attributes() {
  cudaError_t e = batched_chol_attributes();
  if (e != cudaSuccess) return e;
  e = batched_solve_attributes();
  if (e != cudaSuccess) return e;
  return batched_fit_attributes();
}

}  // namespace trk
