// The relative-error contraction of fit_body.cuh (the error ||TR - X|| / ||X|| of Sec. 5
// and the stop rule of Sec. 4.1) on the 5th-generation tensor cores, for X in FP32.
//
// TR(p, q) = sum_e V_p[e] W_q[e], K = R_{N-1} R_{s-1} <= 256 terms, for rows p and columns q
// of X's mode split. Each FP32 factor is split into TF32 parts hi + lo, and per 8 terms hi*hi,
// (V) hi*lo and lo*hi go into one FP32 accumulator, in order of the terms. (Two FP16 parts per
// factor, scaled per row and column, take half the MMA time and shared memory and truncate the
// accumulator half as often, but the error's systematic part, about 5e-7 of TR, is then another
// one: the fit of a stalled decomposition, 1 - error with the error near 1, moves by 1e-4 of
// itself. The tensor pipe is not what bounds this kernel, so the products stay as they were.)
//
// One tile is 128 columns q (the MMA's M: W is the A operand) times NB rows p (N: V is the
// B operand). A tensor-memory lane is then a column of X, so a warp reads 32 consecutive
// entries of a row of X per load, whatever the alignment of the rows. The units (row block,
// column tile), row block by row block, are cut into one contiguous range per CTA, so every
// CTA has the same number of tiles within one, for tall, wide and small X alike.
//
// Warps of a CTA (640 threads, one CTA per SM; registers are shared out by setmaxnreg):
//   0-7   epilogue: 32-row chunks of X loaded one ahead, TR from tensor memory, squares;
//   8-15  build V of the next row block, k-step by k-step, as the MMAs release it;
//   16    streams W (formed once per evaluation in operand layout) through a ring of 8 KB
//         slots, one bulk copy per k-step;
//   17    issues the MMAs, two accumulators in tensor memory (epilogue of one tile overlaps
//         the MMAs of the next).
// Operands are K-major without swizzle: 8-row x 16-byte core matrices, rows 16 bytes apart, so
// a thread that owns a row writes its own words.
//
// What bounds it: the builder's short dependent chains where a row block has few column tiles,
// then the epilogue's loads of X; the tensor pipe is busy about a sixth of the time. Per call,
// with the two preparing launches (before: one CTA formed V, contracted and read X in turn):
// 500^3 rank 10: 755 -> 435 us; 256 x 256 x 3 x 2000 rank 10: 2526 -> 1031 us;
// 37 x 33 x 41 x 29 x 26, ranks 12, 8, 14, 6, 10: 490 -> 217 us.
//
// Every mbarrier wait is bounded and also ends when another warp gave up: the CTA then
// records the timeout bit, waits (bounded) for its MMAs and copies in flight, frees its
// tensor memory and stops.
#pragma once

#include "fit_body.cuh"
#include "tc_common.cuh"

namespace trk {

constexpr int FT_Q = 128;                      // columns of X per tile (MMA M)
constexpr int FT_KS = 8;                       // terms per k-step (MMA K)
constexpr int FT_SLOT = 2 * 2 * FT_Q * 16;     // W of one tile and k-step: 8 KB
constexpr int FT_MAXKS = kMaxL / FT_KS;        // 32
constexpr int FT_MAXSLOTS = 8;
constexpr int FT_EW = 8, FT_BW = 8;            // epilogue and builder warps
constexpr int FT_NT = 32 * (FT_EW + FT_BW + 4);
// registers a thread at launch, and of the epilogue, builder and control warpgroups: two, two
// and one of 128 threads, (2 * 128 + 2 * 88 + 40) * 128 <= 640 * 96
constexpr int FT_REGS = 96, FT_REGS_E = 128, FT_REGS_B = 88, FT_REGS_C = 40;
static_assert(2 * FT_REGS_E + 2 * FT_REGS_B + FT_REGS_C <= 5 * FT_REGS, "register shares");
// setmaxnreg.inc draws on what the CTA was launched with and waits for it without limit, so a kernel
// that the compiler gave fewer registers than the shares add up to must never be launched: checked
// when a context or a server is created.
inline cudaError_t fit_tc_registers(const void* kernel) {
  cudaFuncAttributes at;
  const cudaError_t e = cudaFuncGetAttributes(&at, kernel);
  if (e != cudaSuccess) return e;
  return at.numRegs < FT_REGS ? cudaErrorInvalidConfiguration : cudaSuccess;
}
constexpr size_t kFitTcSmem = 220 * 1024;      // dynamic shared memory of a CTA

// Bytes of the right factors of a split (whole chunks of 32 terms).
__host__ __device__ inline size_t fit_tc_right_bytes(const FitSplit& f) {
  const int64_t tiles = (f.cols + FT_Q - 1) / FT_Q;
  return static_cast<size_t>(tiles) * ((f.K + 31) / 32) * (32 / FT_KS) * FT_SLOT;
}

// FP32 slice tables of the last mode of each group, entry-major: t[(r * Rc + c) * I + i], so
// that threads that own consecutive indices i read consecutive words. Optional: without them
// the FP64 cores are read (one conversion per use, on the FP64 pipe). A group of one mode has none:
// its entries are read once (100000 x 3 x 3, rank 3: 102 us a call with a table, 89 without).
__host__ __device__ inline int64_t fit_tc_table_floats(const FitArgs& a, int mode) {
  return a.dims[mode] * a.ranks[(mode - 1 + a.N) % a.N] * a.ranks[mode];
}
__host__ __device__ inline int64_t fit_tc_left_floats(const FitArgs& a, const FitSplit& f) {
  return f.s > 1 ? fit_tc_table_floats(a, f.s - 1) : 0;
}
__host__ __device__ inline int64_t fit_tc_right_floats(const FitArgs& a, const FitSplit& f) {
  return f.s < a.N - 1 ? fit_tc_table_floats(a, a.N - 1) : 0;
}
__host__ __device__ inline int64_t fit_tc_tables_floats(const FitArgs& a, const FitSplit& f) {
  return fit_tc_left_floats(a, f) + fit_tc_right_floats(a, f);
}
// Table offsets are 32-bit. Where the right group alone has one, few entries read with a conversion
// each cost less than the launch that forms it (20 x 20 x 20, rank 8, 2e5 of them: 77 us a call with
// the table, 74 without; 60 x 60 x 60, rank 16, 1.5e7: 142 and 176).
__host__ __device__ inline bool fit_tc_tables_fit(const FitArgs& a, const FitSplit& f) {
  return (f.s > 1 || f.cols * a.ranks[a.N - 2] * f.K >= (1 << 20)) &&
         fit_tc_tables_floats(a, f) < (1ll << 31);
}
// The two tables behind `tables` (null where there is none).
__host__ __device__ inline const float* fit_tc_left(const FitArgs& a, const FitSplit& f, const float* tables) {
  return f.s > 1 ? tables : nullptr;
}
__host__ __device__ inline const float* fit_tc_right(const FitArgs& a, const FitSplit& f, const float* tables) {
  return tables && f.s < a.N - 1 ? tables + fit_tc_left_floats(a, f) : nullptr;
}

struct FitTcPlan {
  int NB;              // rows per block: 256, 128 or 64 (MMA N)
  int ks;              // k-steps
  int slots;           // ring slots of W
  int npre;            // prefix products held per block (0: the left group is one mode)
  int64_t tiles, units;
};

// NB is the largest that leaves a ring of four slots, then
// halved while the units are fewer than two per SM: a function of the problem alone, so a
// served request's sums do not depend on what runs beside it.
__host__ __device__ inline FitTcPlan fit_tc_plan(const FitArgs& a, const FitSplit& f) {
  FitTcPlan p;
  p.ks = (f.K + FT_KS - 1) / FT_KS;
  p.tiles = (f.cols + FT_Q - 1) / FT_Q;
  const int64_t J = a.dims[f.s - 1];
  const int rlast = a.ranks[a.N - 1];
  p.NB = 256;
  for (;;) {
    int64_t np = f.s > 1 ? (p.NB - 1) / J + 2 : 0;
    if (np > p.NB) np = p.NB;
    p.npre = static_cast<int>(np);
    const size_t need = static_cast<size_t>(p.ks) * 64 * p.NB + np * rlast * 64 +
                        (f.s > 2 ? FT_BW * kMaxL * 4 : 0);
    const size_t room = kFitTcSmem;
    const int64_t s = need < room ? static_cast<int64_t>((room - need) / FT_SLOT) : 0;
    p.slots = static_cast<int>(s < FT_MAXSLOTS ? s : FT_MAXSLOTS);
    p.units = (f.rows + p.NB - 1) / p.NB * p.tiles;
    const bool fits = p.slots >= 4;
    if (p.NB == 64 || (fits && p.units >= 304)) break;
    p.NB /= 2;
  }
  return p;
}

// Partial sums of one served evaluation (one per CTA): about eight units each.
__host__ __device__ inline int64_t fit_tc_parts(const FitTcPlan& p) { return (p.units + 7) / 8; }

struct FitTcShared {
  uint64_t vfull[FT_MAXKS], vfree[FT_MAXKS];      // V k-step written / released by the MMAs
  uint64_t wfull[FT_MAXSLOTS], wempty[FT_MAXSLOTS];
  uint64_t accfull[2], accfree[2];
  uint64_t drain;
  uint32_t tmem_slot;
  int abort;
};

namespace ft {

// One group's last mode: entry (r, c) of the slice at index i.
struct Slices {
  const double* core;
  const float* table;
  int64_t I;
  int Rm, Rc;
  __device__ __forceinline__ float at(int r, int c, int64_t i) const {
    return table ? __ldg(table + static_cast<int64_t>(r * Rc + c) * I + i)
                 : static_cast<float>(__ldg(core + (i * Rm + r) * Rc + c));
  }
};

__device__ __forceinline__ Slices slices(const FitArgs& a, int mode, const float* table) {
  return Slices{a.core[mode], table, a.dims[mode], a.ranks[(mode - 1 + a.N) % a.N], a.ranks[mode]};
}

// Pairs of FP32 values in one 64-bit register: one instruction for two multiply-adds.
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// Dot product of a prefix row (16 floats in shared memory, zeros beyond Rm) and a slice column.
__device__ __forceinline__ float dot_row(const float* row, const float (&g)[16], int Rm) {
  const ulonglong2* P = reinterpret_cast<const ulonglong2*>(row);
  uint64_t x = 0, y = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (4 * t < Rm) {
      const ulonglong2 p = P[t];
      x = fma2(p.x, pack2(g[4 * t], g[4 * t + 1]), x);
      y = fma2(p.y, pack2(g[4 * t + 2], g[4 * t + 3]), y);
    }
  }
  const float2 a = unpack2(x), b = unpack2(y);
  return (a.x + a.y) + (b.x + b.y);
}

// Product of the slices of modes m0 .. m1 - 1 at the mixed-radix index `pre` (the last mode
// fastest) into dst (row stride 16, zeros beyond the last rank), one warp; G is scratch of
// kMaxL floats, used when the product has more than one factor. kAhead: a factor's loads are in
// flight while the one before it is multiplied (16 registers; a long chain is their latency).
template <bool kAhead>
__device__ inline void prefix_product(const FitArgs& a, int m0, int m1, int64_t pre, float* dst,
                                      float* G, int lane) {
  int64_t div = 1;
  for (int m = m0 + 1; m < m1; ++m) div *= a.dims[m];
  const int rows = a.ranks[(m0 - 1 + a.N) % a.N];
  int cols = a.ranks[m0];
  double next[kAhead ? kMaxL / 32 : 1];
  auto fetch = [&](int m, int left) {        // the slice of mode m, left x ranks[m]
    pre %= div;
    div /= a.dims[m];
    const int n = left * a.ranks[m];
    const double* src = a.core[m] + (pre / div) * n;
    if constexpr (kAhead) {
#pragma unroll
      for (int q = 0; q < kMaxL / 32; ++q) next[q] = lane + 32 * q < n ? src[lane + 32 * q] : 0.0;
    } else {
      __syncwarp();
      for (int e = lane; e < n; e += 32) G[e] = static_cast<float>(src[e]);
    }
  };
  {
    const double* src = a.core[m0] + (pre / div) * rows * cols;
    if (kAhead && m0 + 1 < m1) fetch(m0 + 1, cols);
    for (int e = lane; e < rows * 16; e += 32) {
      const int r = e >> 4, c = e & 15;
      dst[e] = c < cols ? static_cast<float>(src[r * cols + c]) : 0.f;
    }
  }
  for (int m = m0 + 1; m < m1; ++m) {
    const int rr = a.ranks[m];
    if constexpr (kAhead) {
      __syncwarp();
#pragma unroll
      for (int q = 0; q < kMaxL / 32; ++q)
        if (lane + 32 * q < cols * rr) G[lane + 32 * q] = static_cast<float>(next[q]);
      if (m + 1 < m1) fetch(m + 1, rr);
    } else {
      fetch(m, cols);
    }
    __syncwarp();
    float acc[8];                    // rows * 16 <= 256 entries, 8 per lane
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = lane + 32 * q, r = e >> 4, c = e & 15;
      float s = 0.f;
      if (r < rows && c < rr)
        for (int t = 0; t < cols; ++t) s = fmaf(dst[r * 16 + t], G[t * rr + c], s);
      acc[q] = s;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = lane + 32 * q;
      if ((e >> 4) < rows) dst[e] = acc[q];
    }
    cols = rr;
  }
  __syncwarp();
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, 8-row groups 128 bytes
// apart (stride), k-groups of 4 terms `lbo` bytes apart (leading).
__device__ __forceinline__ uint64_t desc_plain(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>(128u >> 4) << 32;
  d |= static_cast<uint64_t>(1u) << 46;
  return d;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mbar) : "memory");
}

// Bounded wait that also ends when another warp of the CTA gave up; false then. Each poll may
// sleep up to the hint: warps that spin take issue slots from the ones that work.
__device__ __forceinline__ bool wait_for(uint32_t mbar, uint32_t parity, int* abort) {
  constexpr int kPolls = 1 << 18;
  constexpr uint32_t kSleepNs = 20000;
  for (int it = 0; it < kPolls; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(mbar), "r"(parity), "r"(kSleepNs) : "memory");
    if (done) return true;
    if (*reinterpret_cast<volatile int*>(abort)) return false;
  }
  *reinterpret_cast<volatile int*>(abort) = 1;
  return false;
}

// The builder warps' part of fit_tc_units: thread = row of V; with fewer rows than builder
// threads the k-steps are split between the groups of NB threads. The slice column in use and
// the next one are in registers, so a column's loads are in flight while the one before is
// multiplied. One short loop on purpose: unrolled over the entries of a k-step it spilled and
// outgrew the instruction cache (110 us a block against 22 us for everything else).
template <bool kTable>
__device__ __forceinline__ void build_v(const FitArgs& a, const FitSplit& f, const FitTcPlan& pl,
                                        const float* ltable, int64_t lo, int64_t hi,
                                        unsigned char* vt, float* prefix, float* scratch,
                                        FitTcShared& sh) {
  constexpr int kThreads = 32 * FT_BW;
  const int bt = threadIdx.x - 32 * FT_EW, bw = bt >> 5, lane = bt & 31;
  const int NB = pl.NB, nks = pl.ks;
  const int vstep = 64 * NB, vpart = 32 * NB, vgroup = 16 * NB;
  const int Rlast = a.ranks[a.N - 1], K = f.K;
  const int pstride = Rlast * 16;
  const int groups = kThreads / NB, row = bt % NB, part = bt / NB;
  const int e0 = nks * part / groups * FT_KS, e1 = nks * (part + 1) / groups * FT_KS;
  const Slices g = slices(a, f.s - 1, ltable);
  const int Rm = g.Rm, Rc = g.Rc;
  const int64_t I = g.I;
  const bool pre = f.s > 1;
  // entry offsets, 32 bits (a table has less than 2^31 entries, or there is none)
  const int cstep = kTable ? Rc * static_cast<int>(I) : Rc;   // from row t to t + 1
  const int bstep = kTable ? static_cast<int>(I) : 1;         // from column b to b + 1
  int seg = 0;
  for (int64_t u = lo; u < hi; ++seg) {
    const int64_t rb = u / pl.tiles;
    const int64_t p0 = rb * NB;
    const int64_t pend = p0 + NB < f.rows ? p0 + NB : f.rows;
    const int64_t pre0 = p0 / I;
    if (pre) {
      const int np = static_cast<int>((pend - 1) / I - pre0 + 1);
      for (int x = bw; x < np; x += FT_BW) {
        float* dst = prefix + x * pstride;
        prefix_product<false>(a, 0, f.s - 1, pre0 + x, dst, scratch + bw * kMaxL, lane);
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    // the row's slice and prefix
    const int64_t p = p0 + row;
    const bool live = p < pend;
    const int64_t mine = live ? p / I : pre0, i = live ? p - mine * I : 0;
    const float* tp = ltable + i;
    const double* dp = g.core + i * Rm * Rc;
    const float* P = prefix + (mine - pre0) * pstride;
    auto entry = [&](int o) -> float {
      if constexpr (kTable) return __ldg(tp + o);
      else return static_cast<float>(__ldg(dp + o));
    };
    auto column = [&](int b, float (&col)[16]) {
      const int n = b < Rc ? Rm : 0;
      int o = b * bstep;
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        col[t] = 0.f;
        if (t < n) col[t] = entry(o);
        o += cstep;
      }
    };
    bool ok = true;
    int e = e0, b = e0 / Rlast, c = e0 - b * Rlast;
    float gc[16], gn[16];
    unsigned char* vrow = vt + row * 16;
    if (pre) column(b, gc);
    while (e < e1 && ok) {
      if (pre) column(b + 1, gn);
#pragma unroll 2
      for (; c < Rlast && e < e1; ++c, ++e) {
        const int ks = e / FT_KS;
        if ((e & (FT_KS - 1)) == 0 && seg > 0) {
          ok = wait_for(tc::smem_u32(&sh.vfree[ks]), static_cast<uint32_t>((seg - 1) & 1), &sh.abort);
          if (!ok) break;
        }
        float x = 0.f;
        if (live && e < K) x = pre ? dot_row(P + c * 16, gc, Rm) : entry(c * cstep + b * bstep);
        const float h = tc::tf32_rna(x);
        unsigned char* at = vrow + ks * vstep + ((e >> 2) & 1) * vgroup + (e & 3) * 4;
        *reinterpret_cast<float*>(at) = h;
        *reinterpret_cast<float*>(at + vpart) = tc::tf32_rna(x - h);
        if ((e & (FT_KS - 1)) == FT_KS - 1) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(tc::smem_u32(&sh.vfull[ks]));
        }
      }
      c = 0;
      ++b;
#pragma unroll
      for (int t = 0; t < 16; ++t) gc[t] = gn[t];
    }
    if (pre) {   // this block's prefixes are read; the builder warps leave together
      int all;
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
                   "bar.red.and.pred q, 1, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                   : "=r"(all) : "r"(ok ? 1 : 0) : "memory");
      ok = all != 0;
    }
    if (!ok) break;
    u = (rb + 1) * pl.tiles;
  }
}

}  // namespace ft

// The slice tables, one warp per slice: warp w of n.
__device__ inline void fit_tables_warps(const FitArgs& a, const FitSplit& f, float* out, int64_t w,
                                        int64_t n) {
  const int lane = threadIdx.x & 31;
  const int64_t I0 = f.s > 1 ? a.dims[f.s - 1] : 0, I1 = f.s < a.N - 1 ? a.dims[a.N - 1] : 0;
  for (; w < I0 + I1; w += n) {
    const int mode = w < I0 ? f.s - 1 : a.N - 1;
    const int64_t i = w < I0 ? w : w - I0, I = w < I0 ? I0 : I1;
    float* t = w < I0 ? out : out + fit_tc_left_floats(a, f);
    const int L = a.ranks[(mode - 1 + a.N) % a.N] * a.ranks[mode];
    for (int e = lane; e < L; e += 32) t[e * I + i] = static_cast<float>(a.core[mode][i * L + e]);
  }
}

// The right factors are formed in jobs of 32 columns and kWarps * kPer k-steps: thread = column, and
// kPer k-steps one after another. What bounds a job is chains: of its at most 32 prefix products
// (modes s .. N-2), dealt out to the warps, of the loads of an entry's slice column, and of the
// instructions themselves, hence one short loop over the entries (unrolled, with 128 columns and two
// k-steps a CTA: 10 x 10 x 10, rank 3: 20 us, now 9; 2^12, rank 3, with 64 prefixes of six products:
// 110, now 17). One problem: 4 warps and one k-step each, or 16 where 32 columns span more than four
// prefixes and the jobs leave SMs idle (2^12 with 4: 39 us; 20 x 20 x 20, rank 8, with 16: 17 us, with
// 4: 11, the conversions of one SM's FP64 pipe); served requests share the SMs: 4 warps and 4 k-steps
// each, so that a prefix product serves more entries.
constexpr int FT_RC = 32, FT_RW = 16, FT_RWS = 4;
__host__ __device__ inline int fit_right_jobs(int64_t tiles, int ks, int per_job) {
  return static_cast<int>(tiles) * (FT_Q / FT_RC) * ((ks + per_job - 1) / per_job);
}

template <bool kTable>
__device__ __forceinline__ void fit_right_entries(const ft::Slices& g, bool pre, const float* P,
                                                  int Rlast, int e0, int e1, bool valid, int64_t i,
                                                  unsigned char* dst) {
  const float* tp = g.table + i;
  const double* dp = g.core + i * g.Rm * g.Rc;
  const int cstep = kTable ? g.Rc * static_cast<int>(g.I) : g.Rc;
  const int bstep = kTable ? static_cast<int>(g.I) : 1;
  auto entry = [&](int o) -> float {
    if constexpr (kTable) return __ldg(tp + o);
    else return static_cast<float>(__ldg(dp + o));
  };
  int b = e0 / Rlast, c = e0 - b * Rlast;
  const int end = (e1 + FT_KS - 1) / FT_KS * FT_KS;       // the last k-step is padded with zeros
#pragma unroll 1
  for (int e = e0; e < end; ++e) {
    float v = 0.f;
    if (valid && e < e1) {
      if (pre) {
        float gc[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) gc[t] = t < g.Rm ? entry(t * cstep + c * bstep) : 0.f;
        v = ft::dot_row(P + b * 16, gc, g.Rm);
      } else {
        v = entry(b * cstep + c * bstep);
      }
    }
    const float h = tc::tf32_rna(v);
    unsigned char* at = dst + static_cast<size_t>((e - e0) / FT_KS) * FT_SLOT +
                        ((e >> 2) & 1) * (FT_Q * 16) + (e & 3) * 4;
    *reinterpret_cast<float*>(at) = h;
    *reinterpret_cast<float*>(at + 2 * FT_Q * 16) = tc::tf32_rna(v - h);
    if (++c == Rlast) { c = 0; ++b; }
  }
}

// Job `job` of them, in operand layout: WS[tile][k-step][part][k-group][column][4]; entry
// e = b * Rlast + a holds P_right(q)[b][a]. P: 32 * 256 floats, G: kWarps * kMaxL floats of shared
// memory.
template <int kWarps, int kPer>
__device__ inline void fit_right_tc_job(const FitArgs& a, const FitSplit& f, int64_t job,
                                        const float* table, unsigned char* WS, float* P, float* G) {
  constexpr int kJob = kWarps * kPer;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nks = (f.K + FT_KS - 1) / FT_KS, nkj = (nks + kJob - 1) / kJob;
  const int Rlast = a.ranks[a.N - 1];
  const ft::Slices g = ft::slices(a, a.N - 1, table);
  const bool pre = f.s < a.N - 1;
  const int64_t part = job / nkj, tile = part / (FT_Q / FT_RC);
  const int ks = static_cast<int>(job - part * nkj) * kJob + warp * kPer;
  const int64_t q = part * FT_RC + lane;
  const bool valid = q < f.cols;
  const int64_t mine = q / g.I, pre0 = part * FT_RC / g.I;
  if (pre && part * FT_RC < f.cols) {
    const int64_t last = (part * FT_RC + FT_RC < f.cols ? part * FT_RC + FT_RC : f.cols) - 1;
    for (int64_t x = pre0 + warp; x <= last / g.I; x += kWarps)
      ft::prefix_product<true>(a, f.s, a.N - 1, x, P + (x - pre0) * 256, G + warp * kMaxL, lane);
  }
  __syncthreads();
  if (ks >= nks) return;
  const int e0 = ks * FT_KS, most = (ks + kPer) * FT_KS, e1 = most < f.K ? most : f.K;
  unsigned char* dst = WS + (static_cast<size_t>(tile) * nks + ks) * FT_SLOT + (q - tile * FT_Q) * 16;
  const float* Pq = P + (valid ? mine - pre0 : 0) * 256;
  const int64_t i = valid ? q - mine * g.I : 0;
  if (table) fit_right_entries<true>(g, pre, Pq, Rlast, e0, e1, valid, i, dst);
  else fit_right_entries<false>(g, pre, Pq, Rlast, e0, e1, valid, i, dst);
}

// Accumulates (se, sx) over the units lo .. hi - 1 (unit = row block * tiles + tile). All
// FT_NT threads of the CTA call it; `dyn` holds kFitTcSmem bytes of
// dynamic shared memory, 128-byte aligned; se
// and sx are meaningful in the epilogue warps (zero elsewhere).
__device__ inline void fit_tc_units(const FitArgs& a, const FitSplit& f, const FitTcPlan& pl,
                                    const float* __restrict__ X,
                                    const unsigned char* __restrict__ WS, const float* ltable,
                                    int64_t lo, int64_t hi, unsigned char* dyn, FitTcShared& sh,
                                    unsigned* err, double& se, double& sx) {
  using namespace tc;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NB = pl.NB, nks = pl.ks, slots = pl.slots;
  // (no pointer is rounded through an integer: the compiler keeps 32-bit shared addresses)
  unsigned char* ring = dyn;
  unsigned char* vt = ring + slots * FT_SLOT;          // V: [k-step][part][k-group][row][8]
  const int vstep = 64 * NB, vpart = 32 * NB, vgroup = 16 * NB;
  float* prefix = reinterpret_cast<float*>(vt + nks * vstep);
  const int pstride = a.ranks[a.N - 1] * 16;
  float* scratch = prefix + pl.npre * pstride;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&sh.tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int k = 0; k < FT_MAXKS; ++k) {
      mbar_init(smem_u32(&sh.vfull[k]), NB / 32);
      mbar_init(smem_u32(&sh.vfree[k]), 1);
    }
    for (int k = 0; k < FT_MAXSLOTS; ++k) {
      mbar_init(smem_u32(&sh.wfull[k]), 1);
      mbar_init(smem_u32(&sh.wempty[k]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(smem_u32(&sh.accfull[k]), 1);
      mbar_init(smem_u32(&sh.accfree[k]), FT_EW);
    }
    mbar_init(smem_u32(&sh.drain), 1);
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh.tmem_slot;
  const int64_t tiles = pl.tiles;

  if (warp < FT_EW) {
    // ---- epilogue: lane = column of the tile's quarter, half of the block's rows per warp
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(FT_REGS_E));
    const int quad = warp & 3, half = warp >> 2;
    const int nch = NB / 64;                           // 32-row chunks of this warp
    const int ntile = static_cast<int>(tiles);
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    const uint32_t total = static_cast<uint32_t>(hi - lo) * nch;
    // the next chunk to load: its lane's first entry, the rows and the column left there
    const float* src = X + ((lo / tiles) * NB + half * (NB / 2)) * f.cols + quad * 32 + lane;
    int64_t lp = (lo / tiles) * NB + half * (NB / 2);
    int lt = static_cast<int>(lo % tiles), lc = 0;
    const int lastq = static_cast<int>(f.cols - (tiles - 1) * FT_Q) - quad * 32 - lane;
    uint32_t nload = 0;
    auto load = [&](float (&x)[32]) {
      if (nload == total) return;
      ++nload;
      const float* s = src + lt * FT_Q;
      int n = static_cast<int>(f.rows - lp < 32 ? f.rows - lp : 32);
      if (lt + 1 == ntile && lastq <= 0) n = 0;
      if (n >= 32) {
#pragma unroll
        for (int i = 0; i < 32; ++i) { x[i] = __ldcs(s); s += f.cols; }
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) { x[i] = i < n ? __ldcs(s) : 0.f; s += f.cols; }
      }
      lp += 32;
      src += 32 * f.cols;
      if (++lc == nch) {       // next tile: back to the block's first row, or the next block
        lc = 0;
        lp -= NB / 2;
        src -= (NB / 2) * f.cols;
        if (++lt == ntile) { lt = 0; lp += NB; src += NB * f.cols; }
      }
    };
    int ch = 0;                                        // the chunk in use
    uint32_t ul = 0, done = 0;                         // its tile, counted from lo
    uint64_t se_t = 0, sx_t = 0;
    auto take = [&](const float (&x)[32]) -> bool {
      if (done == total) return false;
      ++done;
      const int buf = static_cast<int>(ul & 1);
      const int r0 = half * (NB / 2) + ch * 32;
      if (ch == 0) {
        if (!ft::wait_for(smem_u32(&sh.accfull[buf]), (ul >> 1) & 1, &sh.abort)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      }
      __syncwarp();
      float v[32];
      tmem_load32(lane_addr + static_cast<uint32_t>(buf * 256 + r0), v);
      const uint64_t minus = ft::pack2(-1.f, -1.f);
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const uint64_t x2 = ft::pack2(x[i], x[i + 1]);
        const uint64_t d2 = ft::fma2(ft::pack2(v[i], v[i + 1]), minus, x2);
        se_t = ft::fma2(d2, d2, se_t);
        sx_t = ft::fma2(x2, x2, sx_t);
      }
      if (++ch == nch) {        // at most 64 squares per FP32 sum, then FP64
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) ft::mbar_arrive(smem_u32(&sh.accfree[buf]));
        ch = 0;
        ++ul;
        const float2 p = ft::unpack2(se_t), q = ft::unpack2(sx_t);
        se += static_cast<double>(p.x + p.y);
        sx += static_cast<double>(q.x + q.y);
        se_t = sx_t = 0;
      }
      return true;
    };
    float xa[32], xb[32];
    load(xa);
    for (;;) {
      load(xb);
      if (!take(xa)) break;
      load(xa);
      if (!take(xb)) break;
    }
  } else if (warp < FT_EW + FT_BW) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(FT_REGS_B));
    if (ltable)
      ft::build_v<true>(a, f, pl, ltable, lo, hi, vt, prefix, scratch, sh);
    else
      ft::build_v<false>(a, f, pl, ltable, lo, hi, vt, prefix, scratch, sh);
  } else if (warp == FT_EW + FT_BW) {
    // ---- W producer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(FT_REGS_C));
    if (lane == 0) {
      long long n = 0;
      int s = 0;
      uint32_t phase = 0;                  // of slot s: its use count's parity
      bool ok = true;
      for (int64_t u = lo; u < hi && ok; ++u) {
        const unsigned char* src = WS + static_cast<size_t>(u % tiles) * nks * FT_SLOT;
        for (int ks = 0; ks < nks; ++ks, ++n) {
          if (n >= slots && !ft::wait_for(smem_u32(&sh.wempty[s]), phase ^ 1, &sh.abort)) {
            ok = false;
            break;
          }
          const uint32_t full = smem_u32(&sh.wfull[s]);
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                       :: "r"(full), "r"(static_cast<uint32_t>(FT_SLOT)) : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
              :: "r"(smem_u32(ring + s * FT_SLOT)), "l"(src + static_cast<size_t>(ks) * FT_SLOT),
                 "r"(static_cast<uint32_t>(FT_SLOT)), "r"(full) : "memory");
          if (++s == slots) { s = 0; phase ^= 1; }
        }
      }
      // no copy is in flight when the CTA leaves (bounded; after an abort some were not consumed)
      for (long long m = n > slots ? n - slots : 0; m < n; ++m)
        mbar_wait(smem_u32(&sh.wfull[m % slots]), static_cast<uint32_t>((m / slots) & 1));
    }
  } else if (warp == FT_EW + FT_BW + 1) {
    // ---- MMA issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(FT_REGS_C));
    if (lane == 0) {
      const uint32_t idesc = idesc_tf32(FT_Q, NB);
      int s = 0, seg = 0;
      uint32_t phase = 0;
      const int ntile = static_cast<int>(tiles);
      int t = static_cast<int>(lo % tiles);
      bool ok = true;
      const uint32_t count = static_cast<uint32_t>(hi - lo);
      for (uint32_t ul = 0; ul < count && ok; ++ul) {
        const int buf = static_cast<int>(ul & 1);
        const bool first = ul == 0 || t == 0;
        const bool last = ul + 1 < count && t + 1 == ntile;     // V is rebuilt after this tile
        if (first && ul > 0) ++seg;
        if (++t == ntile) t = 0;
        if (ul >= 2)
          ok = ft::wait_for(smem_u32(&sh.accfree[buf]), (ul / 2 - 1) & 1, &sh.abort);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem + static_cast<uint32_t>(buf * 256);
        for (int ks = 0; ks < nks; ++ks) {
          if (first && !ft::wait_for(smem_u32(&sh.vfull[ks]), static_cast<uint32_t>(seg & 1),
                                     &sh.abort)) {
            ok = false;
            break;
          }
          if (!ft::wait_for(smem_u32(&sh.wfull[s]), phase, &sh.abort)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t wb = smem_u32(ring + s * FT_SLOT), vb = smem_u32(vt + ks * vstep);
          constexpr int wp[3] = {0, 1, 0}, vp[3] = {0, 0, 1};
#pragma unroll
          for (int m = 0; m < 3; ++m)
            mma_tf32(acc, ft::desc_plain(wb + wp[m] * (2 * FT_Q * 16), FT_Q * 16),
                         ft::desc_plain(vb + vp[m] * vpart, vgroup), idesc,
                         (ks > 0 || m > 0) ? 1u : 0u);
          mma_commit(smem_u32(&sh.wempty[s]));
          if (last) mma_commit(smem_u32(&sh.vfree[ks]));
          if (++s == slots) { s = 0; phase ^= 1; }
        }
        if (ok) mma_commit(smem_u32(&sh.accfull[buf]));
      }
      mma_commit(smem_u32(&sh.drain));
      if (!mbar_wait(smem_u32(&sh.drain), 0)) *reinterpret_cast<volatile int*>(&sh.abort) = 1;
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(FT_REGS_C));
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 :: "r"(tmem), "r"(512u) : "memory");
  if (tid == 0 && sh.abort) atomicOr(err, kErrTimeout);
}

// Block sum of the epilogue warps' (se, sx) to thread 0; red holds 2 * FT_EW doubles.
__device__ __forceinline__ void fit_tc_reduce(double& se, double& sx, double* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < FT_EW) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      se += __shfl_xor_sync(0xffffffffu, se, o);
      sx += __shfl_xor_sync(0xffffffffu, sx, o);
    }
    if (lane == 0) { red[warp] = se; red[FT_EW + warp] = sx; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    se = sx = 0.0;
    for (int w = 0; w < FT_EW; ++w) { se += red[w]; sx += red[FT_EW + w]; }
  }
}

}  // namespace trk
