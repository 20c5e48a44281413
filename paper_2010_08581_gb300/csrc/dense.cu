// Dense TR-ALS (Alg. 1) on the same least-squares path as the sampled method: every row of
// G_[2]^{!=n} and of X_[n]^T, each with weight 1, instead of J sampled ones (Def. 5 with
// S = I). Rows are taken in the row-major order of the modes other than n (the last mode
// fastest), which is the memory order of X: row r = pre * P_post + post, where X is viewed as
// [P_pre][I_n][P_post].
#include "common.cuh"

namespace trk {
namespace {

// Every row of G_[2]^{!=n} (Alg. 4 with every multi-index, weight 1) in the same order. A run is
// the I_f rows that differ only in the fastest mode f; all other factors of the slice chain are
// fixed along it. One CTA per run (or per part of one, where runs are few): the fixed factors,
// and the product `pre` of those before f in ring order, are formed in shared memory once; then
// for `rb` rows at a time thread (i, c) multiplies pre by column c of G^(f)(:, i, :), and thread
// (i, r) carries row r through the factors after f, the fixed factor broadcast from shared
// memory, four entries per load (zeros beyond a rank). Products are summed in the order of the
// per-sample chain (warp_slice_chain), so the rows are the same bit for bit.
// The per-sample kernel read every factor of every row in FP64 and converted it on the FP64
// pipe: 240 us for 250,000 rows of rank 10, now 70 us (15 us to write them).
constexpr int DENSE_NT = 256;
constexpr int DENSE_TILE = 16 * 256;   // entries of a CTA's rows: rb * R_0 * max columns

struct DenseRows {
  const float* core[kMaxModes];    // ring order, slice-major
  int64_t I[kMaxModes];
  int rl[kMaxModes], rr[kMaxModes];
  int slow[kMaxModes];          // ring positions of the fixed modes, fastest first
  int npos, mf;                 // positions; that of f
  int rb;                       // rows at a time: DENSE_NT / the widest of R_0 and R_f
  int64_t runs;
};

__global__ void __launch_bounds__(DENSE_NT) k_dense_rows(DenseRows a, float* __restrict__ A) {
  extern __shared__ __align__(16) float F[];   // [npos][16][16] fixed factors, zero-padded
  float* pre = F + a.npos * 256;               // [16][16]
  float* tile = pre + 256;                     // [rb][R_0][columns]
  __shared__ int64_t ii[kMaxModes];
  const int tid = threadIdx.x;
  const int R0 = a.rl[0], L = R0 * a.rr[a.npos - 1], rb = a.rb;
  const int fr = a.rl[a.mf], fc = a.rr[a.mf];
  const int64_t If = a.I[a.mf];
  const int ic = tid / fc, c0 = tid - ic * fc, ir = tid / R0, r0 = tid - ir * R0;
  for (int64_t run = blockIdx.x; run < a.runs; run += gridDim.x) {
    if (tid == 0) {
      int64_t rest = run;
      for (int k = 0; k < a.npos - 1; ++k) {
        const int m = a.slow[k];
        ii[m] = rest % a.I[m];
        rest /= a.I[m];
      }
    }
    __syncthreads();
    for (int m = 0; m < a.npos; ++m) {
      if (m == a.mf) continue;
      const int r = tid >> 4, c = tid & 15;
      F[m * 256 + tid] = r < a.rl[m] && c < a.rr[m]
                             ? a.core[m][(ii[m] * a.rl[m] + r) * a.rr[m] + c] : 0.f;
    }
    __syncthreads();
    for (int m = 0; m < a.mf; ++m) {         // pre = F[0] F[1] ... F[mf - 1]
      const int r = tid >> 4, c = tid & 15;
      float s = 0.f;
      if (r < R0 && c < a.rr[m]) {
        if (m == 0) s = F[tid];
        else
          for (int t = 0; t < a.rl[m]; ++t) s += pre[r * 16 + t] * F[m * 256 + t * 16 + c];
      }
      __syncthreads();
      pre[tid] = s;
      __syncthreads();
    }
    for (int64_t i0 = static_cast<int64_t>(blockIdx.y) * rb; i0 < If;
         i0 += static_cast<int64_t>(gridDim.y) * rb) {
      const int nb = If - i0 < rb ? static_cast<int>(If - i0) : rb;
      const float* src = a.core[a.mf] + i0 * fr * fc;
      if (a.mf > 0) {
        if (ic < nb) {
          float g[16];
#pragma unroll
          for (int t = 0; t < 16; ++t)
            g[t] = t < fr ? src[(ic * fr + t) * fc + c0] : 0.f;
          for (int r = 0; r < R0; ++r) {
            const float4* p = reinterpret_cast<const float4*>(pre + r * 16);
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (4 * q >= fr) continue;
              const float4 x = p[q];
              s += x.x * g[4 * q];
              s += x.y * g[4 * q + 1];
              s += x.z * g[4 * q + 2];
              s += x.w * g[4 * q + 3];
            }
            tile[(ic * R0 + r) * fc + c0] = s;
          }
        }
      } else {
        for (int e = tid; e < nb * fr * fc; e += DENSE_NT) tile[e] = src[e];
      }
      int cols = fc;
      for (int m = a.mf + 1; m < a.npos; ++m) {
        __syncthreads();
        const int cc = a.rr[m];
        const bool on = ir < nb;
        float* row = tile + (ir * R0 + r0) * cols;
        float v[16], s[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          v[t] = (on && t < cols) ? row[t] : 0.f;
          s[t] = 0.f;
        }
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          if (t >= cols) continue;
          const float4* p = reinterpret_cast<const float4*>(F + m * 256 + t * 16);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (4 * q >= cc) continue;
            const float4 x = p[q];
            s[4 * q] += v[t] * x.x;
            s[4 * q + 1] += v[t] * x.y;
            s[4 * q + 2] += v[t] * x.z;
            s[4 * q + 3] += v[t] * x.w;
          }
        }
        __syncthreads();
        row = tile + (ir * R0 + r0) * cc;
        if (on)
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (c < cc) row[c] = s[c];
        cols = cc;
      }
      __syncthreads();
      float* out = A + (run * If + i0) * L;
      for (int e = tid; e < nb * L; e += DENSE_NT) out[e] = tile[e];
      __syncthreads();
    }
  }
}

// FP32 copies of the cores at every ring position, one after another.
__global__ void __launch_bounds__(256) k_cores_f32(ChainArgs a, float* __restrict__ out) {
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int m = 0; m < a.npos; ++m) {
    const int64_t n = a.I[m] * a.rl[m] * a.rr[m];
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < n; e += step)
      out[e] = static_cast<float>(a.core[m][e]);
    out += n;
  }
}

// Row r -> its multi-index in ring order (position m holds mode (n + 1 + m) % N).
__global__ void __launch_bounds__(256) k_enumerate(int N, int n, DenseDims d, int64_t P,
                                                   int32_t* __restrict__ idx) {
  const int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= P) return;
  int64_t rest = r;
  for (int mode = N - 1; mode >= 0; --mode) {
    if (mode == n) continue;
    const int64_t i = rest % d.I[mode];
    rest /= d.I[mode];
    const int m = (mode - n - 1 + N) % N;
    idx[r * (N - 1) + m] = static_cast<int32_t>(i);
  }
}

// Y[pre * P_post + q][i] = X[pre][i][q] (a batched transpose of the I_n x P_post slabs),
// through 32 x 32 shared-memory tiles: reads coalesced along q, writes along i.
template <typename TX, typename TY>
__global__ void __launch_bounds__(256) k_unfold(const TX* __restrict__ X, int64_t Ppre,
                                                int64_t In, int64_t Ppost, TY* __restrict__ Y) {
  __shared__ TY tile[32][33];
  const int64_t q0 = static_cast<int64_t>(blockIdx.x) * 32, i0 = static_cast<int64_t>(blockIdx.y) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 8 rows of 32 per pass
  for (int64_t pre = blockIdx.z; pre < Ppre; pre += gridDim.z) {
    const TX* src = X + pre * In * Ppost;
    TY* dst = Y + pre * Ppost * In;
    for (int r = ty; r < 32; r += 8) {
      const int64_t i = i0 + r, q = q0 + tx;
      if (i < In && q < Ppost) tile[r][tx] = static_cast<TY>(src[i * Ppost + q]);
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
      const int64_t q = q0 + r, i = i0 + tx;
      if (q < Ppost && i < In) dst[q * In + i] = tile[tx][r];
    }
    __syncthreads();
  }
}

// Y = X with a type change (the last mode: X is already [P][I_n]).
template <typename TX, typename TY>
__global__ void __launch_bounds__(256) k_convert(const TX* __restrict__ X, int64_t count,
                                                 TY* __restrict__ Y) {
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < count;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x)
    Y[e] = static_cast<TY>(X[e]);
}

template <typename TX, typename TY>
cudaError_t unfold_t(const TX* X, int64_t Ppre, int64_t In, int64_t Ppost, TY* Y,
                     cudaStream_t st) {
  if (Ppost == 1) {
    const int64_t count = Ppre * In;
    const unsigned blocks = static_cast<unsigned>(count / 256 + 1 < sm_count() * 16 ? count / 256 + 1 : sm_count() * 16);
    k_convert<TX, TY><<<blocks, 256, 0, st>>>(X, count, Y);
    return cudaGetLastError();
  }
  dim3 grid(static_cast<unsigned>((Ppost + 31) / 32), static_cast<unsigned>((In + 31) / 32),
            static_cast<unsigned>(Ppre < 65535 ? Ppre : 65535));
  k_unfold<TX, TY><<<grid, 256, 0, st>>>(X, Ppre, In, Ppost, Y);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_enumerate(int N, int n, const DenseDims& d, int32_t* idx, cudaStream_t st) {
  int64_t P = 1;
  for (int m = 0; m < N; ++m)
    if (m != n) P *= d.I[m];
  if (P <= 0) return cudaSuccess;
  k_enumerate<<<static_cast<unsigned>((P + 255) / 256), 256, 0, st>>>(N, n, d, P, idx);
  return cudaGetLastError();
}

// A run costs a chain of barriers whatever its length, and a CTA: short ones are only worth it while
// they are few or their products large (the kernel that takes row by row reads longer chains from
// global memory from 100 columns on). All updates of 400 x 400 x f x f, by runs and row by row: f = 3,
// rank 8: 1887 and 818 us; f = 5, rank 10: 2188 and 2318; f = 6, rank 8: 1985 and 1596, rank 9: 2116 and 2067, of
// 50 x 50 x 40 x f x f: f = 7, rank 8: 2016 and 1915; 30 x 30 x 3 x 3, rank 8: 59 and 66; 8^6, rank 8: 54 and
// 58 an update; 2^16, rank 2: 349 and 120.
bool dense_by_runs(int N, int n, const ChainArgs& ca) {
  const int f = ((n == N - 1 ? N - 2 : N - 1) - n - 1 + N) % N;     // ring position of the runs' mode
  const int L = ca.rl[0] * ca.rr[ca.npos - 1];
  int64_t runs = 1;
  for (int m = 0; m < ca.npos; ++m)
    if (m != f) runs *= ca.I[m];
  return ca.I[f] >= (L >= 100 ? 5 : (L > 64 ? 6 : 8)) || runs <= 2 * sm_count();
}

cudaError_t launch_dense_rows(int N, int n, const ChainArgs& ca, float* f32_cores, float* A,
                              cudaStream_t st) {
  k_cores_f32<<<2 * static_cast<unsigned>(sm_count()), 256, 0, st>>>(ca, f32_cores);
  DenseRows a{};
  a.npos = ca.npos;
  a.runs = 1;
  for (int m = 0; m < ca.npos; ++m) {
    a.core[m] = f32_cores;
    a.I[m] = ca.I[m];
    a.rl[m] = ca.rl[m];
    a.rr[m] = ca.rr[m];
    f32_cores += ca.I[m] * ca.rl[m] * ca.rr[m];
  }
  const int f = n == N - 1 ? N - 2 : N - 1;
  int k = 0;
  a.mf = (f - n - 1 + N) % N;
  for (int mode = f - 1; mode >= 0; --mode) {
    if (mode == n) continue;
    a.slow[k] = (mode - n - 1 + N) % N;
    a.runs *= ca.I[a.slow[k]];
    ++k;
  }
  int cols = 0;
  for (int m = a.mf; m < a.npos; ++m) cols = a.rr[m] > cols ? a.rr[m] : cols;
  a.rb = DENSE_NT / (a.rl[0] > a.rr[a.mf] ? a.rl[0] : a.rr[a.mf]);
  if (a.rb * a.rl[0] * cols > DENSE_TILE) a.rb = DENSE_TILE / (a.rl[0] * cols);
  const int64_t most = 64 * sm_count();
  const int64_t steps = (ca.I[a.mf] + a.rb - 1) / a.rb;
  int64_t parts = 8 * sm_count() / a.runs;
  parts = parts < 1 ? 1 : (parts < steps ? parts : steps);
  const size_t smem = (static_cast<size_t>(a.npos + 1) * 256 + a.rb * a.rl[0] * cols) * sizeof(float);
  const dim3 grid(static_cast<unsigned>(a.runs < most ? a.runs : most), static_cast<unsigned>(parts));
  k_dense_rows<<<grid, DENSE_NT, smem, st>>>(a, A);
  return cudaGetLastError();
}

cudaError_t launch_unfold(const void* X, bool x_f64, int N, int n, const DenseDims& d, void* Y,
                          bool y_f64, cudaStream_t st) {
  int64_t Ppre = 1, Ppost = 1;
  for (int m = 0; m < n; ++m) Ppre *= d.I[m];
  for (int m = n + 1; m < N; ++m) Ppost *= d.I[m];
  const int64_t In = d.I[n];
  // grid.x, grid.y <= 65535 tiles: checked by the caller (dense_fits)
  if (x_f64 && y_f64)
    return unfold_t(static_cast<const double*>(X), Ppre, In, Ppost, static_cast<double*>(Y), st);
  if (x_f64)
    return unfold_t(static_cast<const double*>(X), Ppre, In, Ppost, static_cast<float*>(Y), st);
  if (y_f64)
    return unfold_t(static_cast<const float*>(X), Ppre, In, Ppost, static_cast<double*>(Y), st);
  return unfold_t(static_cast<const float*>(X), Ppre, In, Ppost, static_cast<float*>(Y), st);
}

}  // namespace trk
