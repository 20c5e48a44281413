// Row a5 on the 5th-generation tensor cores: C = A~^T [A~ | Y~] (M = A~^T A~ and B = A~^T Y~
// of the sampled LS, Alg. 2 LS step) with tcgen05.mma kind::tf32 and FP32 accumulation in
// tensor memory.
//
// Each FP32 operand x is split into TF32 parts hi = rna_tf32(x), lo = rna_tf32(x - hi), and
// every k-step issues hi*hi + hi*lo + lo*hi into the same accumulator, which recovers
// close to FP32 accuracy (Markidis et al., "NVIDIA Tensor Core Programmability,
// Performance & Precision", 2018; Ootomo & Yokota, 2022).
//
// One CTA = one 128 x TN output tile over one chunk of the J samples (split-K, partials
// reduced downstream in a fixed order). All 256 threads load the chunk from global memory
// (16-byte vectors along the feature / fibre index), two 32-sample stages ahead in registers,
// split it and store it into K-major, 128-byte-swizzled shared-memory tiles; one elected thread
// issues the MMAs and commits them to an mbarrier per pipeline stage; TMEM is read back with
// tcgen05.ld. The dense method's right-hand sides (X_[n]^T of a strided mode) are read from X
// where it lies: there 32 consecutive samples of one column are consecutive words of X.
//
// A stage is latency: loads, conversion, two barriers and twelve MMAs follow one another. With
// 128 columns per CTA (129 KB of shared memory) one CTA runs per SM, and 155 CTAs on 152 SMs took
// two rounds at J = 250,000 (1134 us). With 64 or 80 columns two CTAs share an SM and one's loads
// and conversions cover the other's MMAs (788 us). One CTA of 128 columns per SM converts A's rows
// half as often and is the best where it is one round (launch_normal_eq_tc).
// The column tile does not change a result: an entry is the same sequence of FP32
// accumulations over the same chunk of samples whatever the tile. Every
// mbarrier wait is bounded: a wait of the main loop polls at most `wait_limit` times; on
// expiry the CTA records an error, stops issuing, waits (bounded by the default limit) for
// the MMAs it has committed, frees its TMEM and returns without writing its partials.
#include <type_traits>

#include "common.cuh"
#include "tc_common.cuh"

namespace trk {
namespace {

constexpr int TM = 128;          // UMMA M
constexpr int TK = 32;           // samples per pipeline stage (one 128-byte swizzle row)
constexpr int NT = 256;
static_assert(TK == 32 && TM == 4 * (NT / 32) * 4,
              "operand loader: one sample per lane, 4 groups of 4 rows per warp");
constexpr int STAGES = 2;
constexpr int A_BYTES = TM * TK * 4;   // 16 KB
constexpr uint32_t TMEM_COLS = 128;    // FP32 accumulator: 128 lanes x TN <= 128 columns

template <int TN>
constexpr int stage_bytes() { return 2 * A_BYTES + 2 * TN * TK * 4; }   // hi and lo of both
template <int TN>
constexpr int smem_bytes() { return STAGES * stage_bytes<TN>() + 1024; }

using namespace tc;

// TN output columns per CTA (MMA N). kDense: the columns from L on are X viewed as
// [J / post][I][post] (Y points to X, post > 1): Y[r][i] = X[r / post][i][r % post].
template <int TN, bool kDense>
__global__ void __launch_bounds__(NT, TN > 80 ? 1 : 2) k_normal_eq_tc(const float* __restrict__ A,
                                                        const float* __restrict__ Y, int64_t J,
                                                        int L, int64_t I, int64_t post,
                                                        int64_t chunk,
                                                        float* __restrict__ partial,
                                                        unsigned* err, long long wait_limit,
                                                        const int64_t* __restrict__ jdev) {
  grid_wait();
  constexpr uint32_t kIdesc = idesc_tf32(TM, TN);
  constexpr int B_BYTES = TN * TK * 4;
  constexpr int STAGE_BYTES = stage_bytes<TN>();
  constexpr int NG = TN / 4;                        // column groups of 4
  constexpr int NQ = (NG + NT / 32 - 1) / (NT / 32);   // groups per warp, rounded up
  static_assert(TN % 16 == 0 && TN <= static_cast<int>(TMEM_COLS), "MMA N");
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  // 1024-byte alignment of the tiles (required by the 128-byte swizzle atoms)
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t mbar[STAGES];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t ldc = L + I;
  const int m0 = blockIdx.y * TM;
  const int64_t n0 = static_cast<int64_t>(blockIdx.x) * TN;
  const int64_t j0 = static_cast<int64_t>(blockIdx.z) * chunk;
  const int64_t Jr = jdev ? (*jdev < J ? *jdev : J) : J;
  const int64_t j1 = (j0 + chunk < Jr) ? j0 + chunk : Jr;
  const int nchunks = j1 > j0 ? static_cast<int>((j1 - j0 + TK - 1) / TK) : 0;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(smem_u32(&mbar[s]), 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_slot;

  // Loaders. Groups of 4 consecutive tile rows (features for A, output columns for B) at one
  // sample: with rows of A and Y that are multiples of 16 bytes long (and 16-byte aligned
  // bases) a group is one 16-byte load, otherwise four scalar loads with bounds. Group q of
  // thread t: sample k = lane, tile rows 4 g .. 4 g + 3 with g = warp + 8 q. Lanes cover
  // consecutive samples, so the stores into the K-major swizzled tile below hit 32 different
  // banks (consecutive k of one row span the whole 128-byte line).
  const bool vec_a = (L % 4) == 0 && (reinterpret_cast<uintptr_t>(A) % 16) == 0;
  const bool vec_y = !kDense && vec_a && (I % 4) == 0 && (reinterpret_cast<uintptr_t>(Y) % 16) == 0;
  auto load_chunk = [&](int c, float (&ra)[TK / 2], float (&rb)[4 * NQ]) {
    if (c >= nchunks) return;
    const int64_t j = j0 + static_cast<int64_t>(c) * TK + lane;
    const bool in = j < j1;
    const float* arow = A + j * L;
    const float* yrow = Y + (kDense ? 0 : j * I);
    if constexpr (kDense) {
      int64_t pre, at;
      if (J <= INT32_MAX) {
        const uint32_t p = static_cast<uint32_t>(j) / static_cast<uint32_t>(post);
        pre = p;
        at = static_cast<uint32_t>(j) - p * static_cast<uint32_t>(post);
      } else {
        pre = j / post;
        at = j - pre * post;
      }
      yrow = Y + pre * I * post + at;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int am = m0 + 4 * (warp + (NT / 32) * q);
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      if (in) {
        if (vec_a) {
          if (am < L) a = __ldg(reinterpret_cast<const float4*>(arow + am));
        } else {
          if (am < L) a.x = __ldg(arow + am);
          if (am + 1 < L) a.y = __ldg(arow + am + 1);
          if (am + 2 < L) a.z = __ldg(arow + am + 2);
          if (am + 3 < L) a.w = __ldg(arow + am + 3);
        }
      }
      ra[4 * q] = a.x; ra[4 * q + 1] = a.y; ra[4 * q + 2] = a.z; ra[4 * q + 3] = a.w;
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int g = warp + (NT / 32) * q;
      const int64_t bn = n0 + 4 * g;
      float b[4] = {0.f, 0.f, 0.f, 0.f};
      if (in && g < NG && bn < ldc) {
        if (vec_a && bn < L) {             // L % 4 == 0: the whole group is in A
          const float4 v = __ldg(reinterpret_cast<const float4*>(arow + bn));
          b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
        } else if (vec_y) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(yrow + (bn - L)));
          b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int64_t c2 = bn + i;
            if (c2 < L) b[i] = __ldg(arow + c2);
            else if (c2 < ldc) b[i] = __ldg(yrow + (c2 - L) * (kDense ? post : 1));
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) rb[4 * q + i] = b[i];
    }
  };
  int issued = 0;
  // Splits chunk c's values, stores them into its stage and issues its MMAs; false when a
  // bounded wait expired.
  auto run_chunk = [&](int c, const float (&ra)[TK / 2], const float (&rb)[4 * NQ]) -> bool {
    if (c >= nchunks) return false;
    const int s = c % STAGES;
    unsigned char* st = base + s * STAGE_BYTES;
    if (c >= STAGES) {   // wait until the MMAs that read this stage have finished
      const bool ok = mbar_wait(smem_u32(&mbar[s]), ((c / STAGES) - 1) & 1, wait_limit);
      if (!ok) atomicExch(&s_abort, 1);
    }
    __syncthreads();
    if (s_abort) return false;
#pragma unroll
    for (int u = 0; u < TK / 2; ++u) {
      const int row = 4 * (warp + (NT / 32) * (u / 4)) + (u % 4);
      const float ah = tf32_rna(ra[u]);
      const uint32_t o = sw128_offset(row, lane);
      *reinterpret_cast<float*>(st + o) = ah;
      *reinterpret_cast<float*>(st + A_BYTES + o) = tf32_rna(ra[u] - ah);
    }
#pragma unroll
    for (int u = 0; u < 4 * NQ; ++u) {
      const int g = warp + (NT / 32) * (u / 4);
      if (g < NG) {
        const float bh = tf32_rna(rb[u]);
        const uint32_t o = sw128_offset(4 * g + (u % 4), lane);
        *reinterpret_cast<float*>(st + 2 * A_BYTES + o) = bh;
        *reinterpret_cast<float*>(st + 2 * A_BYTES + B_BYTES + o) = tf32_rna(rb[u] - bh);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a_hi = smem_u32(st), a_lo = a_hi + A_BYTES;
      const uint32_t b_hi = a_hi + 2 * A_BYTES, b_lo = b_hi + B_BYTES;
#pragma unroll
      for (int ks = 0; ks < TK / 8; ++ks) {
        const uint32_t koff = ks * 32;   // 8 TF32 = 32 bytes along K inside the swizzle row
        const uint32_t acc0 = (c > 0 || ks > 0) ? 1u : 0u;
        mma_tf32(tmem_d, make_desc(a_hi + koff), make_desc(b_hi + koff), kIdesc, acc0);
        mma_tf32(tmem_d, make_desc(a_hi + koff), make_desc(b_lo + koff), kIdesc, 1u);
        mma_tf32(tmem_d, make_desc(a_lo + koff), make_desc(b_hi + koff), kIdesc, 1u);
      }
      mma_commit(smem_u32(&mbar[s]));
    }
    issued = c + 1;
    return true;
  };
  {
    float a0[TK / 2], b0[4 * NQ], a1[TK / 2], b1[4 * NQ], a2[TK / 2], b2[4 * NQ];
    load_chunk(0, a0, b0);
    load_chunk(1, a1, b1);
    for (int c = 0; c < nchunks; c += 3) {   // two chunks in flight while one is stored
      load_chunk(c + 2, a2, b2);
      if (!run_chunk(c, a0, b0)) break;
      load_chunk(c + 3, a0, b0);
      if (!run_chunk(c + 1, a1, b1)) break;
      load_chunk(c + 4, a1, b1);
      if (!run_chunk(c + 2, a2, b2)) break;
    }
  }
  __syncthreads();
  const int aborted = s_abort;
  // `issued` counts the chunks whose MMAs were committed: all of them, or, after an expired
  // wait at chunk c, chunks 0 .. c-1.
  // Wait for the last commit of each stage that was used (bounded by the default limit,
  // so that no MMA is in flight when TMEM is freed).
  bool ok = true;
  if (issued > 0) {
    const int last = issued - 1;
    ok = mbar_wait(smem_u32(&mbar[last % STAGES]), (last / STAGES) & 1);
    if (issued > 1) {
      const int prev = issued - 2;
      ok = mbar_wait(smem_u32(&mbar[prev % STAGES]), (prev / STAGES) & 1) && ok;
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!ok) atomicExch(&s_abort, 1);
  __syncthreads();
  const bool failed = aborted || s_abort != 0;     // the same for every thread
  if (failed) {
    if (tid == 0) atomicOr(err, kErrTimeout);
  } else if (issued == 0) {
    // no rows in this chunk (beyond the device-side row count): zero partials
    for (int e = tid; e < TM * TN; e += NT) {
      const int m = m0 + e / TN;
      const int64_t col = n0 + e % TN;
      if (m < L && col < ldc)
        partial[(static_cast<int64_t>(blockIdx.z) * L + m) * ldc + col] = 0.0f;
    }
  } else {
    // Epilogue through shared memory (every MMA has completed, so the stage buffers are
    // free): warp w moves TMEM lanes 32*(w%4).. (tile rows) of every other 16-column piece
    // into a [TM][TN + 1] tile (odd stride: no bank conflicts), then the warps write whole
    // rows, 32 consecutive columns per store instruction.
    float* tile = reinterpret_cast<float*>(base);
    const int quad = warp & 3, half = warp >> 2;
    const int rl = quad * 32 + lane;
    for (int col = half * 16; col < TN; col += 32) {
      float v[16];
      tmem_load16(tmem_d + (static_cast<uint32_t>(quad * 32) << 16) + col, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) tile[rl * (TN + 1) + col + i] = v[i];
    }
    __syncthreads();
    for (int r = warp; r < TM; r += NT / 32) {
      const int m = m0 + r;
      if (m >= L) break;
      float* out = partial + (static_cast<int64_t>(blockIdx.z) * L + m) * ldc + n0;
#pragma unroll
      for (int q = 0; q < (TN + 31) / 32; ++q) {
        const int c = lane + 32 * q;
        if (c < TN && n0 + c < ldc) out[c] = tile[r * (TN + 1) + c];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 :: "r"(tmem_d), "r"(TMEM_COLS) : "memory");
}

// The split of the samples: every entry of the result is summed within these chunks, in
// order. It was laid down for 128-column tiles, one CTA per SM, and is kept because it fixes
// the result's rounding; the launch below chooses the column tile.
void plan_tc(int64_t J, int L, int64_t I, int* splits, int64_t* chunk) {
  const int64_t tiles = ((L + TM - 1) / TM) * ((L + I + 127) / 128);
  int64_t s = (sm_count() + tiles - 1) / tiles;
  const int64_t maxs = (J + 4 * TK - 1) / (4 * TK);   // at least 4 stages per CTA
  if (s > maxs) s = maxs;
  if (s < 1) s = 1;
  int64_t c = (J + s - 1) / s;
  c = (c + TK - 1) / TK * TK;
  s = (J + c - 1) / c;
  *splits = static_cast<int>(s);
  *chunk = c;
}

template <int TN, bool kDense>
cudaError_t launch_tn(const float* A, const float* Y, int64_t J, int L, int64_t I, int64_t post,
                      int64_t chunk, int splits, float* partial, unsigned* err, cudaStream_t st,
                      long long wait_limit, const int64_t* jdev) {
  dim3 grid(static_cast<unsigned>((L + I + TN - 1) / TN), (L + TM - 1) / TM, splits);
  launch_pdl((k_normal_eq_tc<TN, kDense>), grid, NT, smem_bytes<TN>(), st, A, Y, J,
             L, I, post, chunk, partial, err, wait_limit < 0 ? kTcSpinLimit : wait_limit, jdev);
  return cudaGetLastError();
}

}  // namespace

size_t normal_eq_tc_workspace(int64_t J, int L, int64_t I, int* splits) {
  int64_t chunk;
  plan_tc(J, L, I, splits, &chunk);
  return static_cast<size_t>(*splits) * L * (L + I) * sizeof(float);
}

cudaError_t launch_normal_eq_tc(const float* A, const float* Y, int64_t J, int L, int64_t I,
                                float* partial, int splits, unsigned* err, cudaStream_t st,
                                long long wait_limit, const int64_t* jdev, int64_t post) {
  int s;
  int64_t chunk;
  plan_tc(J, L, I, &s, &chunk);
  if (s != splits) return cudaErrorInvalidValue;
  // The busiest SM's share: its CTAs times the work of a stage (the tile's columns plus A's 128
  // rows, which every column tile converts again) times their stages. The last chunk of the samples
  // is the shorter one and its CTAs are launched last: where only they are left over for one more
  // round, that round is as short. 800 sizes (L = 9 to 256, I = 3 to 4000, J = 300 to 40000): on average
  // 0.3 % slower than the fastest tile of each, 7 % without the 128-column tile (whose CTA, alone on
  // its SM, counts 250). J = 4000, L = 100, I = 500: 125 CTAs of 128 columns, 250 of 64: 15.6 us and 20.6; J = 250,000:
  // 310 CTAs of 64 or 248 of 80, three or two on an SM; J = 4000, L = 121, I = 300: 22.4 us with 128 columns,
  // 31.2 with 64.
  const int64_t mt = (L + TM - 1) / TM, sms = sm_count();
  const int64_t last = J - (splits - 1) * chunk;
  auto share = [&](int tn) {
    const int64_t of_chunk = mt * ((L + I + tn - 1) / tn), ctas = of_chunk * splits;
    const int64_t rounds = (ctas + sms - 1) / sms, over = ctas - (rounds - 1) * sms;
    const int64_t rows = rounds > 1 && over <= of_chunk ? (rounds - 1) * chunk + last : rounds * chunk;
    return rows * (tn < 128 ? tn + TM : 250);
  };
  auto go = [&](auto tn) {
    constexpr int N = decltype(tn)::value;
    return post > 1 ? launch_tn<N, true>(A, Y, J, L, I, post, chunk, splits, partial, err, st,
                                         wait_limit, jdev)
                    : launch_tn<N, false>(A, Y, J, L, I, 1, chunk, splits, partial, err, st,
                                          wait_limit, jdev);
  };
  const int64_t s64 = share(64), s80 = share(80), s128 = share(128);
  if (s128 < s64 && s128 < s80) return go(std::integral_constant<int, 128>{});
  if (s80 < s64) return go(std::integral_constant<int, 80>{});
  return go(std::integral_constant<int, 64>{});
}

cudaError_t normal_eq_tc_attributes() {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_normal_eq_tc<64, false>, attr, smem_bytes<64>());
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_normal_eq_tc<80, false>, attr, smem_bytes<80>());
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_normal_eq_tc<128, false>, attr, smem_bytes<128>());
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_normal_eq_tc<64, true>, attr, smem_bytes<64>());
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_normal_eq_tc<80, true>, attr, smem_bytes<80>());
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_normal_eq_tc<128, true>, attr, smem_bytes<128>());
  return e;
}

}  // namespace trk
