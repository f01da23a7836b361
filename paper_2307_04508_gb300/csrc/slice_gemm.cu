// FP64-accurate contractions on the tensor cores (tcgen05 + TMEM) from integer
// digits of fixed-point operand rows.
//
// Every operand row X_r is written as X_r ~ 2^(e_r) sum_i a_i 2^(-b i) with
// NS balanced digits a_1 .. a_NS in base 2^b (a BF16 value holds an integer of
// up to 8 bits exactly), and
//
//   D = sum_{i + j <= NL + 1} 2^(-b (i + j)) (a_i b_j^T) 2^(e_A + e_B),
//
// NL = NS levels, or (base 256, short contractions) NS + 1.
//
// All digit pairs of one level i + j add into ONE accumulator: the products
// are integers, and their FP32 sums stay exact below 2^24, which bounds the
// contraction length between drains (`drain_kb` blocks of 16).  So the kernel
// brings each digit of both operands in once for all the pairs it takes part
// in (28 pairs of 7 + 7 digits: a quarter of the operand bytes that one
// contraction per pair reads), and a drain reads NS level accumulators, not
// one per pair.
//
// The B digits of a 64-row tile lie one after the other in shared memory, so
// for one A digit i the digits 1 .. NS + 1 - i of B are ONE operand of
// N = 64 (NS + 1 - i) rows whose products fall into consecutive level columns
// of tensor memory: 10 MMA instructions of N = 64 .. 256 per 16 of K instead of
// 28 of N = 64 (NL = 7), each A tile read from shared memory at most twice (N = 64
// MMAs would be bound by the A operand's shared-memory reads).
//
// Accumulators: NL x 64 columns of 128 lanes (448 or all of the 512 TMEM
// columns for NS = 7).  Sixteen epilogue warps add each drain into two 64-bit integers per
// output element (the four lowest levels; the others), exact over the whole
// contraction, release the accumulators, and only then turn the sum into FP64 (one
// rounding), while the next tile's MMAs run.  The conversion is integer code:
// this part issues two FP64 instructions per clock and SM, and a tile of
// 128 x 64 outputs would hold the FP64 pipe for 4096 clocks per FP64
// instruction per output.
//
// Bound: the tensor pipe (28 BF16 products per useful one).  Measured, Pi's
// eight moments at N = 453, 27,000 pairs: 1.2 ms of MMAs and drains, 70 % of the
// tensor pipe's cycles (28 products: 1.0 PFLOP/s; useful 37 TFLOP/s), where the
// FP64 tiles of gemm_f64.cu took 56 ms at 95 % of the FP64 pipe.  Issuing the
// upper and the lower levels from two threads: 2.60 -> 2.46 ms for the whole
// call, one copy per lane of the producer: 2.37 ms.
//
// The 128-row operand A indexes the contiguous dimension of the output, so a
// warp's 32 lanes write (and read, when accumulating) 256 contiguous bytes.
#include <cuda_bf16.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "per_device.h"
#include "tc_ptx.cuh"

namespace ltgw {
namespace {

constexpr int SG_M = 128, SG_N = 64;                // output tile: A rows x B rows
constexpr uint32_t SG_DIG = SL_ROWS * SL_K * 2;     // one digit of a 64-row, 16-k block: 2 KB
constexpr int SG_EPI_WARPS = 16;
// Warps: 0 bulk-copy producer, 1 and 2 MMA issue (the lower and the upper levels:
// separate accumulators, so one issuer's MMAs run while the other's levels are
// drained, and the two share the issue overhead), then the epilogue: sixteen warps
// of 16 columns each (two 64-bit sums per output: eight warps of 32 columns
// would need 128 registers for the sums alone).  608 threads leave 96 registers;
// ptxas spills 44 bytes of <7, 8, 7>, 256 of <7, 8, 8>, 172 of <6, 7, 6> and 136 of
// <7, 7, 7> around the drain.
constexpr int SG_EPI0 = 3, SG_CW = SG_N * 4 / SG_EPI_WARPS;
constexpr int SG_THREADS = 32 * (SG_EPI0 + SG_EPI_WARPS);
static_assert(SG_CW == 16, "one 16-column load per level");
constexpr int SG_MAX_STAGES = 8;
// stages of (2 + 1) x NS digit blocks that fit 216 KB
__host__ __device__ constexpr int sg_stages(int ns) {
  return (int)((216u * 1024) / (3u * ns * SG_DIG)) < SG_MAX_STAGES ? (int)((216u * 1024) / (3u * ns * SG_DIG))
                                                                   : SG_MAX_STAGES;
}
__host__ __device__ constexpr uint32_t sg_smem(int ns) { return (uint32_t)sg_stages(ns) * 3u * ns * SG_DIG + 1024; }

struct SgBars {
  uint64_t full[SG_MAX_STAGES], empty[SG_MAX_STAGES], acc_full[2], acc_empty[2], fin;   // [1]: the upper levels
  uint32_t tmem_base;
  int abort;
};

// K-major operand with the 32-byte swizzle: rows of 16 BF16 (32 bytes), groups
// of 8 rows every 256 bytes.
__device__ __forceinline__ uint64_t sg_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);   // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused, swizzled K-major)
  d |= (uint64_t)(256 >> 4) << 32;          // stride byte offset: 8 rows x 32 B
  d |= (uint64_t)1 << 46;                   // descriptor version
  d |= (uint64_t)6 << 61;                   // 32-byte swizzle
  return d;
}

// kind::f16, D = FP32, A = B = BF16, both K-major, M = 128.
__host__ __device__ constexpr uint32_t sg_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(SG_M >> 4) << 24);
}

__device__ __forceinline__ void sg_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// The MMAs of one 16-k block in two parts: the upper levels (0-based LO ..
// NL - 1) and the lower ones (0 .. LO - 1).  A digit i meets the B digits
// j0 .. j1 that land in the part.  The digit that reaches every level of the part
// comes first: with acc = 0 its MMAs overwrite them (digit 0; with NL = NS + 1
// levels digit 1 for the upper part, as digit 0 ends at level NS - 1).
template <int NL> struct SgLevels { static constexpr int LO = NL > 4 ? (NL + 1) / 2 : NL / 2; };

template <int NS, int NL, bool UPPER>
__device__ __forceinline__ void sg_part(uint32_t tmem, uint64_t a0, uint64_t b0, uint32_t acc) {
  constexpr int L0 = UPPER ? SgLevels<NL>::LO : 0, L1 = UPPER ? NL : SgLevels<NL>::LO;   // levels [L0, L1)
  constexpr int FIRST = UPPER && NL > NS ? 1 : 0;
#pragma unroll
  for (int q = 0; q < (L1 < NS ? L1 : NS); ++q) {
    const int i = q <= FIRST ? FIRST - q : q;
    const int j0 = L0 > i ? L0 - i : 0, j1 = L1 - i < NS ? L1 - i : NS, nj = j1 - j0;   // at most four digits: N <= 256
    sg_mma(tmem + (i + j0) * SG_N, a0 + (uint64_t)(i * (2 * SG_DIG >> 4)), b0 + (uint64_t)(j0 * (SG_DIG >> 4)),
           sg_idesc(nj * SG_N), q == 0 ? acc : 1u);
  }
}

// The unit of work u: (batch entry, K split, tile I of 128 A rows, tile J of
// 64 B rows), tiles fastest.  Symmetric products: J <= 2 I + 1 (the tiles that
// hold an entry with A row >= B row), row I starting at I (I + 1).
struct SgUnit {
  int b, sp, I, J, tile;
  bool valid;
};
__device__ __forceinline__ SgUnit sg_unit(const SliceGemmArgs &g, int64_t u) {
  SgUnit w;
  w.tile = (int)(u % g.n_tiles);
  const int64_t q = u / g.n_tiles;
  w.sp = (int)(q % g.splits);
  w.b = (int)(q / g.splits);
  if (g.sym) {
    int I = (int)((sqrtf(4.0f * (float)w.tile + 1.0f) - 1.0f) * 0.5f);
    while ((int64_t)(I + 1) * (I + 2) <= w.tile) ++I;
    while ((int64_t)I * (I + 1) > w.tile) --I;
    w.I = I;
    w.J = w.tile - I * (I + 1);
  } else {
    w.J = w.tile % g.tiles_n;
    w.I = w.tile / g.tiles_n;
  }
  w.valid = w.J < g.tiles_n;
  return w;
}

// (hi 2^S + lo) 2^E in FP64, negated with neg, rounded once (ties away from
// zero).  |hi 2^S + lo| < 2^95.  About thirty integer instructions, where
// three FP64 ones would take the time of a hundred.
__device__ __noinline__ double sg_value_rare(uint32_t w2, uint32_t w1, uint32_t w0, int E, bool negative) {
  if (E >= SL_NONFINITE / 2) return __longlong_as_double(0x7ff8000000000000ll);   // an operand row was not finite
  double v = 0.0;
  if (E > -SL_NONFINITE / 2)
    v = ldexp((double)w2, E + 64) + ldexp((double)w1, E + 32) + ldexp((double)w0, E);
  return negative ? -v : v;
}

template <int S>
__device__ __forceinline__ double sg_value(long long hi, long long lo, int E, uint32_t neg) {
  uint32_t w0, w1, w2;
  if constexpr (S == 0) {
    w0 = (uint32_t)lo; w1 = (uint32_t)((unsigned long long)lo >> 32); w2 = (uint32_t)(lo >> 63);
  } else {
    const unsigned long long h0 = (unsigned long long)hi << S;
    const unsigned long long t0 = h0 + (unsigned long long)lo;
    w2 = (uint32_t)(hi >> (64 - S)) + (uint32_t)(lo >> 63) + (t0 < h0 ? 1u : 0u);
    w0 = (uint32_t)t0; w1 = (uint32_t)(t0 >> 32);
  }
  const uint32_t sgn = (uint32_t)((int)w2 >> 31);   // all ones for a negative sum
  const unsigned long long mag = ((unsigned long long)(w1 ^ sgn) << 32 | (w0 ^ sgn)) + (sgn & 1u);
  const uint32_t a0 = (uint32_t)mag, a1 = (uint32_t)(mag >> 32), a2 = (w2 ^ sgn) + (sgn && mag == 0ull ? 1u : 0u);
  const uint32_t sign = (sgn ^ neg) & 0x80000000u;
  uint32_t m2 = a2, m1 = a1, m0 = a0;
  int be = E + 1023 + 95;                           // biased exponent of a leading one at bit 95
  if (m2 == 0u) { m2 = m1; m1 = m0; m0 = 0u; be -= 32; }
  if (m2 == 0u) { m2 = m1; m1 = 0u; be -= 32; }
  const int lz = __clz((int)m2);
  m2 = __funnelshift_l(m1, m2, lz);
  m1 = __funnelshift_l(m0, m1, lz);
  be -= lz;
  if (m2 == 0u || (unsigned)(be - 1) >= 2045u) {   // zero, not finite, or outside the normal range
    if (m2 == 0u && E < SL_NONFINITE / 2) return 0.0;
    return sg_value_rare(a2, a1, a0, E, sign != 0u);
  }
  // the leading one adds 1 to the exponent field; a rounding carry goes there too
  const unsigned long long m = ((unsigned long long)(m2 >> 11) << 32 | __funnelshift_r(m1, m2, 11)) + ((m1 >> 10) & 1u);
  return __longlong_as_double((long long)(m + ((unsigned long long)((uint32_t)(be - 1) << 20 | sign) << 32)));
}

// MMA issue of one part's levels (one thread).
template <int NS, int NL, bool UPPER>
__device__ __forceinline__ void sg_issue(const SliceGemmArgs &g, uint8_t *smem, SgBars &bars, uint32_t tmem,
                                         int64_t n_units, int lane) {
  constexpr int ST = sg_stages(NS);
  constexpr uint32_t STAGE = 3u * NS * SG_DIG, A_BYTES = 2u * NS * SG_DIG;
  if (lane == 0) {
    const uint64_t d0 = sg_desc(smem_u32(smem));
    int js = 0;
    uint32_t ps = 0, pe = 1;
    bool ok = true;
    for (int64_t u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
      const SgUnit w = sg_unit(g, u);
      if (!w.valid) continue;
      const int kb0 = g.kb_first + w.sp * g.kb_per_split, kb1 = min(g.nkb, kb0 + g.kb_per_split);
      for (int kb = kb0; kb < kb1 && ok; kb += g.drain_kb) {
        const int ke = min(kb1, kb + g.drain_kb);
        ok = mbar_wait(&bars.acc_empty[UPPER], pe, &bars.abort, g.err);
        pe ^= 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        for (int k = kb; k < ke && ok; ++k) {
          ok = mbar_wait(&bars.full[js], ps, &bars.abort, g.err);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint64_t a0 = d0 + (uint64_t)((js * STAGE) >> 4);
          sg_part<NS, NL, UPPER>(tmem, a0, a0 + (uint64_t)(A_BYTES >> 4), k == kb ? 0u : 1u);
          mma_commit(&bars.empty[js]);
          if (++js == ST) { js = 0; ps ^= 1; }
        }
        if (ok) mma_commit(&bars.acc_full[UPPER]);
      }
    }
    // all issued MMAs complete before the CTA tears down
    mma_commit(&bars.fin);
    mbar_wait(&bars.fin, 0, &bars.abort, g.err, false);
  }
  __syncwarp();
}

template <int NS, int BITS, int NL>
__global__ void __launch_bounds__(SG_THREADS, 1) slice_gemm_kernel(SliceGemmArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(16) SgBars bars;
  constexpr int ST = sg_stages(NS);
  constexpr uint32_t STAGE = 3u * NS * SG_DIG;   // A digits (128 rows each), then B digits
  constexpr uint32_t A_BYTES = 2u * NS * SG_DIG;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int LO = SgLevels<NL>::LO;
  const int64_t n_units = (int64_t)g.batch * g.splits * g.n_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) { mbar_init(&bars.full[s], 1); mbar_init(&bars.empty[s], 2); }
    for (int h = 0; h < 2; ++h) { mbar_init(&bars.acc_full[h], 1); mbar_init(&bars.acc_empty[h], SG_EPI_WARPS); }
    mbar_init(&bars.fin, 2);
    bars.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32(&bars.tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = bars.tmem_base;

  if (warp == 0) {
    // ---------------------------------------------------------------- bulk-copy producer
    // One copy per lane (lane 0: the B digits; lanes 1 .. 2 NS: one digit of
    // one 64-row half of A each): issued by one thread, the fifteen copies
    // of a stage took longer than its MMAs.
    const uint8_t *Bsel = (g.b_sel && *g.b_sel) ? g.B_alt : g.B;
    const int piece = lane - 1, dig = piece >> 1, ah = piece & 1;
    const bool act = lane <= 2 * NS;
    const uint32_t dst_off = lane == 0 ? A_BYTES : (uint32_t)(dig * 2 + ah) * SG_DIG;
    const uint32_t bytes = lane == 0 ? NS * SG_DIG : SG_DIG;
    int64_t issued = 0;
    int js = 0;
    uint32_t ps = 0;
    bool ok = true;
    for (int64_t u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
      const SgUnit w = sg_unit(g, u);
      if (!w.valid) continue;
      const int kb0 = g.kb_first + w.sp * g.kb_per_split, kb1 = min(g.nkb, kb0 + g.kb_per_split);
      const uint8_t *src = lane == 0 ? Bsel + (int64_t)w.b * g.b_batch + (int64_t)w.J * g.nkb * (NS * SG_DIG)
                                     : g.A + (int64_t)w.b * g.a_batch +
                                           (int64_t)(2 * w.I + ah) * g.nkb * (NS * SG_DIG) + dig * SG_DIG;
      for (int kb = kb0; kb < kb1; ++kb) {
        ok = __all_sync(0xffffffffu, mbar_wait(&bars.empty[js], ps ^ 1, &bars.abort, g.err));
        if (!ok) break;
        if (lane == 0) mbar_expect_tx(&bars.full[js], STAGE);
        __syncwarp();
        if (act) bulk_load(smem + js * STAGE + dst_off, src + (int64_t)kb * (NS * SG_DIG), bytes, &bars.full[js]);
        if (++js == ST) { js = 0; ps ^= 1; }
        ++issued;
      }
    }
    if (!ok)   // given up: let the copies in flight land before the CTA's shared memory goes away
      for (int64_t q = max((int64_t)0, issued - ST); q < issued; ++q)
        mbar_wait(&bars.full[q % ST], (uint32_t)(q / ST) & 1, &bars.abort, g.err, false);
    __syncwarp();
  } else if (warp == 1) {
    sg_issue<NS, NL, false>(g, smem, bars, tmem, n_units, lane);
  } else if (warp == 2) {
    sg_issue<NS, NL, true>(g, smem, bars, tmem, n_units, lane);
  } else {
    // ---------------------------------------------------------------- epilogue
    const int ew = warp & 3;              // TMEM lane quarter this warp may read
    const int cq = (warp - SG_EPI0) >> 2;       // columns cq * 16 .. + 15 of every level
    const uint32_t tbase = tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)(cq * SG_CW);
    constexpr int HS = NL > 4 ? 4 * BITS : 0;   // weight of the upper sum
    uint32_t pf = 0;
    bool ok = true;
    for (int64_t u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
      const SgUnit w = sg_unit(g, u);
      if (!w.valid) continue;
      const int kb0 = g.kb_first + w.sp * g.kb_per_split, kb1 = min(g.nkb, kb0 + g.kb_per_split);
      long long lo[SG_CW], hi[NL > 4 ? SG_CW : 1];
#pragma unroll
      for (int q = 0; q < SG_CW; ++q) { lo[q] = 0; if (NL > 4) hi[NL > 4 ? q : 0] = 0; }
      if (g.C && g.beta != 0.0 && !g.partial && (lane & 15) == 0) {
        // the output's lines, read after the contraction: on their way to L2 meanwhile
        const int m0 = w.I * SG_M + ew * 32 + lane, nn = w.J * SG_N + cq * SG_CW;
        if (m0 < g.M)
          for (int q = 0; q < SG_CW && nn + q < g.N; ++q)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(g.C + (int64_t)w.b * g.c_batch + (int64_t)(nn + q) * g.ldc + m0));
      }
      for (int kb = kb0; kb < kb1 && ok; kb += g.drain_kb) {
#pragma unroll
        for (int part = 1; part >= 0; --part) {   // the upper levels are complete first
          ok = mbar_wait(&bars.acc_full[part], pf, &bars.abort, g.err);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
          for (int l = part ? LO : 0; l < (part ? NL : LO); ++l) {
            const bool up = l < NL - 4;
            const int wgt = 1 << (BITS * ((up ? NL - 5 : NL - 1) - l));
            uint32_t r[SG_CW];
            tmem_ld16(r, tbase + (uint32_t)(l * SG_N));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int q = 0; q < SG_CW; ++q) {
              const long long v = (long long)__float2int_rn(__uint_as_float(r[q])) * (long long)wgt;
              if (up) hi[NL > 4 ? q : 0] += v; else lo[q] += v;
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;");
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars.acc_empty[part]);
        }
        pf ^= 1;
      }
      if (!ok) break;
      // ---- the tile's values: A row m (contiguous in the output), B rows n0 ..
      const int m = w.I * SG_M + ew * 32 + lane, n0 = w.J * SG_N + cq * SG_CW;
      const int em = g.ea[(int64_t)w.b * g.ea_batch + m];
      const int e0 = em + g.alpha_exp - BITS * (NL + 1);
      const uint32_t neg = g.alpha_neg ? 0xffffffffu : 0u;
      const int4 *ebp = reinterpret_cast<const int4 *>(g.eb + (int64_t)w.b * g.eb_batch + n0);   // n0 is a multiple of 16
      double val[SG_CW];
#pragma unroll
      for (int q = 0; q < SG_CW; q += 4) {
        const int4 en = __ldg(ebp + q / 4);
        val[q] = sg_value<HS>(NL > 4 ? hi[NL > 4 ? q : 0] : 0ll, lo[q], e0 + en.x, neg);
        val[q + 1] = sg_value<HS>(NL > 4 ? hi[NL > 4 ? q + 1 : 0] : 0ll, lo[q + 1], e0 + en.y, neg);
        val[q + 2] = sg_value<HS>(NL > 4 ? hi[NL > 4 ? q + 2 : 0] : 0ll, lo[q + 2], e0 + en.z, neg);
        val[q + 3] = sg_value<HS>(NL > 4 ? hi[NL > 4 ? q + 3 : 0] : 0ll, lo[q + 3], e0 + en.w, neg);
      }
      if (g.partial) {
        double *o = g.partial + (((int64_t)w.b * g.splits + w.sp) * g.n_tiles + w.tile) * (SG_M * SG_N) +
                    (int64_t)(cq * SG_CW) * SG_M + ew * 32 + lane;
#pragma unroll
        for (int q = 0; q < SG_CW; ++q) o[(int64_t)q * SG_M] = val[q];
      } else if (g.cd_out) {
        // column dot: sum over this tile's B rows n of D[m][n] cd_B[n][m]
        double acc = 0.0;
        if (m < g.M) {
          const int t = m / g.cd_cols;
          const double *cb = g.cd_B + (int64_t)t * g.cd_stride + (m - t * g.cd_cols) + (int64_t)n0 * g.cd_ld;
#pragma unroll
          for (int q = 0; q < SG_CW; ++q)
            if (n0 + q < g.N) acc = fma(val[q], cb[(int64_t)q * g.cd_ld], acc);
          g.cd_out[((int64_t)w.b * (4 * g.tiles_n) + 4 * w.J + cq) * g.cd_ldo + m] = acc;
        }
      } else if (m < g.M) {
        double *o = g.C + (int64_t)w.b * g.c_batch + (int64_t)n0 * g.ldc + m;
        if (g.beta != 0.0) {
#pragma unroll
          for (int q0 = 0; q0 < SG_CW; q0 += 8) {
            double c[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) c[q] = n0 + q0 + q < g.N ? o[(int64_t)(q0 + q) * g.ldc] : 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (n0 + q0 + q < g.N) o[(int64_t)(q0 + q) * g.ldc] = fma(g.beta, c[q], val[q0 + q]);
          }
        } else {
#pragma unroll
          for (int q = 0; q < SG_CW; ++q)
            if (n0 + q < g.N) o[(int64_t)q * g.ldc] = val[q];
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

// C[n][m] = beta C[n][m] + sum over splits of the partial tiles; symmetric
// products: the entries with m >= n, each written to (n, m) and (m, n).
__global__ void __launch_bounds__(256) slice_reduce_kernel(SliceGemmArgs g, const double *__restrict__ partial) {
  const int b = blockIdx.y;
  const int64_t tile_elems = SG_M * SG_N;
  const int64_t total = (int64_t)g.n_tiles * tile_elems;
  const double *p0 = partial + (int64_t)b * g.splits * total;
  double *C = g.C + (int64_t)b * g.c_batch;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const SgUnit w = sg_unit(g, e / tile_elems);
    const int in = (int)(e % tile_elems);
    const int m = w.I * SG_M + in % SG_M, n = w.J * SG_N + in / SG_M;
    if (!w.valid || m >= g.M || n >= g.N || (g.sym && m < n)) continue;
    double a = 0.0;
    for (int sp = 0; sp < g.splits; ++sp) a += p0[(int64_t)sp * total + e];
    double *o = C + (int64_t)n * g.ldc + m;
    if (g.beta != 0.0) a = fma(g.beta, *o, a);
    *o = a;
    if (g.sym && m != n) C[(int64_t)m * g.ldc + n] = a;
  }
}

// C[m][n] = C[n][m] for m > n (batched, 32 x 32 tiles through shared memory).
__global__ void __launch_bounds__(256) mirror_upper_kernel(double *__restrict__ C, int N, int64_t ldc, int64_t batch_stride) {
  __shared__ double t[32][33];
  const int bi = blockIdx.y, bj = blockIdx.x;   // source tile rows bi, columns bj >= bi
  if (bj < bi) return;
  double *Cb = C + (int64_t)blockIdx.z * batch_stride;
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int r = bi * 32 + q, c = bj * 32 + threadIdx.x;
    if (r < N && c < N) t[q][threadIdx.x] = Cb[(int64_t)r * ldc + c];
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int r = bj * 32 + q, c = bi * 32 + threadIdx.x;   // destination (r, c), r > c
    if (r < N && c < N && r > c) Cb[(int64_t)r * ldc + c] = t[threadIdx.x][q];
  }
}

// W[b][m] = sum over the 4 tiles_n part rows of cd_out.
__global__ void slice_coldot_reduce_kernel(const double *__restrict__ cd, int parts, int64_t ldo, int M,
                                           double *__restrict__ W, int64_t ldw) {
  const int b = blockIdx.y;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
    double a = 0.0;
    for (int q = 0; q < parts; ++q) a += cd[((int64_t)b * parts + q) * ldo + m];
    W[(int64_t)b * ldw + m] = a;
  }
}

// ---- operand digits ----
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// Stored exponent of a row whose largest magnitude has the bits mb: the
// smallest e with max < 2^e, plus one in base 256 (its leading digit stays
// within 128); SL_ZERO for a zero row, SL_NONFINITE when an entry is not finite.
__device__ __forceinline__ int slice_exponent(unsigned long long mb, int bits) {
  if (mb == 0ull) return SL_ZERO;
  const int E = (int)(mb >> 52);
  if (E == 2047) return SL_NONFINITE;
  const int e = E ? E - 1022 : 64 - __clzll((long long)mb) - 1074;
  return e + (bits == 8 ? 1 : 0);
}

// rint(x 2^S) to a 64-bit integer, ties to even (integer code; |x| 2^S < 2^63).
__device__ __forceinline__ long long to_fixed(double x, int S) {
  const unsigned long long xb = (unsigned long long)__double_as_longlong(x);
  int E = (int)(xb >> 52) & 0x7ff;
  unsigned long long m = xb & 0xfffffffffffffull;
  if (E) m |= 0x10000000000000ull; else E = 1;
  const int sh = E - 1075 + S;
  unsigned long long q;
  if (sh >= 0) {
    q = sh < 11 ? m << sh : 0ull;
  } else {
    const int r = -sh;
    if (r > 54) {
      q = 0ull;
    } else {
      q = m >> r;
      const unsigned long long rem = m & ((1ull << r) - 1ull), half = 1ull << (r - 1);
      q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
    }
  }
  return (long long)xb < 0 ? -(long long)q : (long long)q;
}

// The digits of eight consecutive k of one row (fixed point), one 16-byte store per digit.
template <int NS, int BITS>
__device__ __forceinline__ void store_fixed(const long long fixed[8], uint8_t *dst) {
  constexpr unsigned long long BIAS = [] {
    unsigned long long b = 0;
    for (int i = 0; i < NS - 1; ++i) b |= (1ull << (BITS - 1)) << (BITS * i);
    return b;
  }();
  unsigned long long Q[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) Q[k] = (unsigned long long)fixed[k] + BIAS;
#pragma unroll
  for (int d = 0; d < NS; ++d) {   // digit d + 1, the leading one first
    uint32_t p[4];
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      float f[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (d == 0)
          f[h] = (float)(int)((long long)Q[k + h] >> (BITS * (NS - 1)));
        else   // an unsigned field minus its bias, through the mantissa of 2^23
          f[h] = __uint_as_float(0x4B000000u |
                                 ((uint32_t)(Q[k + h] >> (BITS * (NS - 1 - d))) & ((1u << BITS) - 1u))) -
                 (8388608.0f + (float)(1 << (BITS - 1)));
      }
      p[k / 2] = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);   // exact in BF16
    }
    *reinterpret_cast<uint4 *>(dst + d * SG_DIG) = make_uint4(p[0], p[1], p[2], p[3]);
  }
}

template <int NS, int BITS>
__device__ __forceinline__ void store_digits(const double x[8], int e, uint8_t *dst) {
  const bool zero = e == SL_ZERO || e >= SL_NONFINITE;
  long long q[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) q[k] = zero ? 0ll : to_fixed(x[k], BITS * NS - e);
  store_fixed<NS, BITS>(q, dst);
}

// Destination of the 16-byte chunk (row r, k 8 g .. 8 g + 7), digit 0.
template <int NS>
__device__ __forceinline__ uint8_t *digit_chunk(uint8_t *dig, int r, int g, int nkb) {
  const int rl = r & (SL_ROWS - 1);
  return dig + ((int64_t)(r / SL_ROWS) * nkb + (g >> 1)) * (NS * SG_DIG) + rl * 32 +
         (((g & 1) ^ ((rl >> 2) & 1)) << 4);
}

__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Largest magnitude of every row over a chunk of its columns (grid: row,
// chunk, batch), its exponent merged into exps (initialised to SL_ZERO).
__global__ void __launch_bounds__(256) slice_max_rows_kernel(SliceSrc a, int bits, int64_t chunk) {
  __shared__ unsigned long long red[8];
  if (a.only_if && !*a.only_if) return;
  const int r = blockIdx.x, b = blockIdx.z;
  const double *x = a.X + (int64_t)b * a.x_batch + (int64_t)r * a.ld;
  const double *f = a.colscale ? a.colscale + (int64_t)b * a.cs_batch : nullptr;
  const int64_t k0 = blockIdx.y * chunk, k1 = min(a.K, k0 + chunk);
  unsigned long long mb = 0ull;
  for (int64_t k = k0 + threadIdx.x; k < k1; k += 256)
    mb = max(mb, mag_bits(f ? __dmul_rn(x[k], f[k]) : x[k]));
  mb = warp_max(mb);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mb;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mb = max(mb, red[w]);
    if (mb) atomicMax(a.exps + (int64_t)b * a.exp_batch + r, slice_exponent(mb, bits));
  }
}

// Digits of rows r < rows_p (zero past `rows`), k < 16 nkb (zero past K):
// one thread per row and eight k, consecutive lanes along k.
template <int NS, int BITS>
__global__ void __launch_bounds__(256) slice_rows_tiles_kernel(SliceSrc a) {
  if (a.only_if && !*a.only_if) return;
  const int b = blockIdx.z;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  uint8_t *dig = a.dig + (int64_t)b * a.dig_batch;
  const double *x = a.X + (int64_t)b * a.x_batch + (int64_t)r * a.ld;
  const double *f = a.colscale ? a.colscale + (int64_t)b * a.cs_batch : nullptr;
  const bool live = r < a.rows;
  const int e = live ? a.exps[(int64_t)b * a.exp_batch + r] : SL_ZERO;
  for (int g = blockIdx.y * 32 + (threadIdx.x & 31); g < 2 * a.nkb; g += gridDim.y * 32) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t k = (int64_t)g * 8 + q;
      v[q] = (live && k < a.K) ? (f ? __dmul_rn(x[k], f[k]) : x[k]) : 0.0;
    }
    store_digits<NS, BITS>(v, e, digit_chunk<NS>(dig, r, g, a.nkb));
  }
}

// ---- rows scaled by several factor rows (Pi's frequencies or Laplace points) ----
// The products X_rk f_k are formed in integer arithmetic (the 128-bit product of
// the mantissas, rounded once to the digits): two FP64 multiplications per
// entry and factor row, one for the maximum and one for the digits, would keep
// the FP64 pipe busy for longer than the digits take to write.
struct Scaled {
  unsigned long long hi;   // upper 64 bits of the mantissas' product, both shifted to bit 63
  int ex;                  // |x f| = hi 2^(ex - 64) up to the dropped lower bits
};
// A zero or subnormal factor: the FP64 product (not inlined, so that the
// multiplication is not issued for every entry).
__device__ __noinline__ Scaled scaled_product_rare(unsigned long long xb, unsigned long long fb) {
  const unsigned long long vb = mag_bits(__dmul_rn(__longlong_as_double((long long)xb), __longlong_as_double((long long)fb)));
  const int E = (int)(vb >> 52);
  Scaled p;
  p.hi = E == 2047 ? ~0ull : E ? (vb << 11) | 0x8000000000000000ull : 0ull;
  p.ex = E == 2047 ? SL_NONFINITE : E - 1022;
  return p;
}
__device__ __forceinline__ Scaled scaled_product(double x, double f) {
  const unsigned long long xb = mag_bits(x), fb = mag_bits(f);
  const int Ex = (int)(xb >> 52), Ef = (int)(fb >> 52);
  Scaled p;
  if (xb == 0ull) {
    p.hi = 0ull;
    p.ex = 0;
    if (Ef == 2047) p = scaled_product_rare(xb, fb);
  } else if (Ex == 0 || Ef == 0) {
    p = scaled_product_rare(xb, fb);
  } else {
    p.hi = __umul64hi((xb << 11) | 0x8000000000000000ull, (fb << 11) | 0x8000000000000000ull);
    p.ex = (Ex == 2047 || Ef == 2047) ? SL_NONFINITE : Ex + Ef - 2044;
  }
  return p;
}

// Exponent of the largest |X_rk f_bk| over a chunk of k, for every factor row
// b (grid: row, chunk); X is read from memory once.
__global__ void __launch_bounds__(256) slice_max_scaled_kernel(SliceSrc a, int batch, int64_t chunk) {
  __shared__ int red[8];
  if (a.only_if && !*a.only_if) return;
  const int r = blockIdx.x;
  const double *x = a.X + (int64_t)r * a.ld;
  const int64_t k0 = blockIdx.y * chunk, k1 = min(a.K, k0 + chunk);
  for (int b = 0; b < batch; ++b) {
    const double *f = a.colscale + (int64_t)b * a.cs_batch;
    int m = SL_ZERO;
    for (int64_t k = k0 + threadIdx.x; k < k1; k += 256) {
      const Scaled p = scaled_product(x[k], f[k]);
      if (p.hi) m = max(m, p.ex - (p.hi >> 63 ? 0 : 1));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) m = max(m, red[w]);
      if (m > SL_ZERO) atomicMax(a.exps + (int64_t)b * a.exp_batch + r, m >= SL_NONFINITE - 1 ? SL_NONFINITE : m + 1);
    }
  }
}

// Digits (7 in base 256) of every scaled row; one thread per row and eight k
// for all factor rows.
__global__ void __launch_bounds__(256) slice_rows_scaled_kernel(SliceSrc a, int batch) {
  if (a.only_if && !*a.only_if) return;
  constexpr int NS = 7, BITS = 8;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  const double *x = a.X + (int64_t)r * a.ld;
  const bool live = r < a.rows;
  for (int g = blockIdx.y * 32 + (threadIdx.x & 31); g < 2 * a.nkb; g += gridDim.y * 32) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = (live && (int64_t)g * 8 + q < a.K) ? x[(int64_t)g * 8 + q] : 0.0;
    for (int b = 0; b < batch; ++b) {
      const int e = live ? a.exps[(int64_t)b * a.exp_batch + r] : SL_ZERO;
      const bool zero = e == SL_ZERO || e >= SL_NONFINITE;
      const double *f = a.colscale + (int64_t)b * a.cs_batch + (int64_t)g * 8;
      long long Q[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const double fk = (live && (int64_t)g * 8 + q < a.K) ? f[q] : 0.0;
        const Scaled p = scaled_product(v[q], fk);
        const int sh = e - BITS * NS - p.ex + 64;   // Q = hi 2^-sh, at least 8 (|x f| < 2^(e - 1))
        const unsigned long long m = (zero || sh > 64) ? 0ull : ((p.hi >> (sh - 1)) + 1ull) >> 1;
        Q[q] = ((__double_as_longlong(v[q]) ^ __double_as_longlong(fk)) < 0) ? -(long long)m : (long long)m;
      }
      store_fixed<NS, BITS>(Q, digit_chunk<NS>(a.dig + (int64_t)b * a.dig_batch, r, g, a.nkb));
    }
  }
}

// Short rows (K <= 128 W): W half-warps' worth of lanes (16 W) hold one row in
// registers, so the exponent and the digits need one pass.  Aligned rows are
// read 16 bytes at a time.
template <int NS, int BITS, int W>
__global__ void __launch_bounds__(256) slice_rows_short_kernel(SliceSrc a, int aligned) {
  if (a.only_if && !*a.only_if) return;
  constexpr int LANES = W >= 2 ? 32 : 16, H = W >= 2 ? W / 2 : 1;   // lanes per row, groups of eight k per lane
  const int b = blockIdx.z, sub = threadIdx.x & (LANES - 1);
  const int r = blockIdx.x * (256 / LANES) + threadIdx.x / LANES;
  uint8_t *dig = a.dig + (int64_t)b * a.dig_batch;
  const double *x = a.X + (int64_t)b * a.x_batch + (int64_t)r * a.ld;
  const double *f = a.colscale ? a.colscale + (int64_t)b * a.cs_batch : nullptr;
  const bool live = r < a.rows;
  double v[H][8];
  unsigned long long mb = 0ull;
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const int64_t k0 = (int64_t)(sub + LANES * h) * 8;
    if (aligned && live && k0 + 8 <= a.K && !f) {
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        const double2 t = *reinterpret_cast<const double2 *>(x + k0 + q);
        v[h][q] = t.x;
        v[h][q + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        v[h][q] = (live && k0 + q < a.K) ? (f ? __dmul_rn(x[k0 + q], f[k0 + q]) : x[k0 + q]) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) mb = max(mb, mag_bits(v[h][q]));
  }
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  const int e = slice_exponent(mb, BITS);
  if (r >= a.rows_p) return;
  if (sub == 0) a.exps[(int64_t)b * a.exp_batch + r] = e;
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const int g = sub + LANES * h;
    if (g < 2 * a.nkb) store_digits<NS, BITS>(v[h], e, digit_chunk<NS>(dig, r, g, a.nkb));
  }
}

// First entry of operand column c of batch entry b.
__device__ __forceinline__ const double *column_source(const SliceSrc &a, int b, int c) {
  const double *x = a.X + (int64_t)b * a.x_batch;
  if (!a.col_group) return x + c;
  const int t = c / a.col_group;
  return x + (int64_t)t * a.col_stride + (c - t * a.col_group);
}

// Column operands (operand row = column of the row-major X): largest
// magnitude of 32 columns over a chunk of X's rows (grid: column block, chunk,
// batch).
__global__ void __launch_bounds__(256) slice_max_cols_kernel(SliceSrc a, int bits, int64_t chunk) {
  __shared__ unsigned long long red[8][32];
  const int c = blockIdx.x * 32 + (threadIdx.x & 31), ty = threadIdx.x >> 5, b = blockIdx.z;
  const double *x = column_source(a, b, c);
  const int64_t k0 = blockIdx.y * chunk, k1 = min(a.K, k0 + chunk);
  unsigned long long mb = 0ull;
  if (c < a.rows)
    for (int64_t k = k0 + ty; k < k1; k += 8) mb = max(mb, mag_bits(x[k * a.ld]));
  red[ty][threadIdx.x & 31] = mb;
  __syncthreads();
  if (ty == 0) {
    for (int w = 1; w < 8; ++w) mb = max(mb, red[w][threadIdx.x]);
    if (mb) atomicMax(a.exps + (int64_t)b * a.exp_batch + c, slice_exponent(mb, bits));
  }
}

// Digits of column operands: one thread per column and 16 k (both chunks of
// its 32-byte row), consecutive lanes along the columns.
template <int NS, int BITS>
__global__ void __launch_bounds__(256) slice_cols_tiles_kernel(SliceSrc a) {
  const int b = blockIdx.z;
  const int r = blockIdx.x * 64 + (threadIdx.x & 63);
  uint8_t *dig = a.dig + (int64_t)b * a.dig_batch;
  const double *x = column_source(a, b, r);
  const bool live = r < a.rows;
  const int e = live ? a.exps[(int64_t)b * a.exp_batch + r] : SL_ZERO;
  for (int kb = a.kb_first + blockIdx.y * 4 + (threadIdx.x >> 6); kb < a.nkb; kb += gridDim.y * 4)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int64_t k = (int64_t)kb * 16 + h * 8 + q;
        v[q] = (live && k < a.K) ? x[k * a.ld] : 0.0;
      }
      store_digits<NS, BITS>(v, e, digit_chunk<NS>(dig, r, 2 * kb + h, a.nkb));
    }
}

// One block per 64 rows, one thread per row and 16 k: both operands of a
// symmetric rank-2 nk update in one pass.
__global__ void __launch_bounds__(512) slice_pair_kernel(SlicePairSrc a) {
  __shared__ unsigned long long red[8][SL_ROWS];
  constexpr int NS = 7, BITS = 8;
  const int rl = threadIdx.x & 63, kb = threadIdx.x >> 6, half = a.nk / SL_K, nkb = 2 * half;
  const int r = blockIdx.x * SL_ROWS + rl;
  const unsigned long long yb = *a.ymax;
  const int c = yb ? max(-1000, min(1000, 1022 - (int)(yb >> 52))) : 0;   // |Y| 2^c < 1
  const double f = __longlong_as_double((long long)(1023 + c) << 52);
  double v[2][8];
  unsigned long long mb = 0ull;
  if (kb < nkb) {
    const bool y = kb >= half;
    const double *src = (y ? a.Y + (int64_t)(kb - half) * SL_K * a.ld : a.X + (int64_t)kb * SL_K * a.ld) + r;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      double t = r < a.rows ? src[(int64_t)q * a.ld] : 0.0;
      if (y) t *= f;
      v[q >> 3][q & 7] = t;
      mb = max(mb, mag_bits(t));
    }
    red[kb][rl] = mb;
  }
  __syncthreads();
  if (kb >= nkb) return;
  for (int q = 0; q < nkb; ++q) mb = max(mb, red[q][rl]);
  const int e = slice_exponent(mb, BITS);
  const int kq = kb >= half ? kb - half : kb + half;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    store_digits<NS, BITS>(v[h], e, digit_chunk<NS>(a.dig_p, r, 2 * kb + h, nkb));
    store_digits<NS, BITS>(v[h], e, digit_chunk<NS>(a.dig_q, r, 2 * kq + h, nkb));
  }
  if (kb == 0) {
    a.exp_q[r] = e;
    a.exp_p[r] = (e == SL_ZERO || e >= SL_NONFINITE) ? e : e - c;
  }
}

__global__ void fill_int_kernel(int *p, int64_t n, int v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = v;
}

template <int NS, int BITS>
cudaError_t slice_operand(const SliceSrc &a, int batch, cudaStream_t s) {
  if (!a.cols && a.nkb <= 32) {
    const int al = a.ld % 2 == 0 && a.x_batch % 2 == 0 && ((uintptr_t)a.X & 15) == 0;
    if (a.nkb <= 8)
      slice_rows_short_kernel<NS, BITS, 1><<<dim3(a.rows_p / 16, 1, batch), 256, 0, s>>>(a, al);
    else if (a.nkb <= 16)
      slice_rows_short_kernel<NS, BITS, 2><<<dim3(a.rows_p / 8, 1, batch), 256, 0, s>>>(a, al);
    else
      slice_rows_short_kernel<NS, BITS, 4><<<dim3(a.rows_p / 8, 1, batch), 256, 0, s>>>(a, al);
    return cudaGetLastError();
  }
  if (a.cols && a.fixed_exp) {
    const int gy = (int)std::min<int64_t>(((int64_t)(a.nkb - a.kb_first) + 3) / 4, 64);
    slice_cols_tiles_kernel<NS, BITS><<<dim3(a.rows_p / 64, gy, batch), 256, 0, s>>>(a);
    return cudaGetLastError();
  }
  const int64_t n_exp = (int64_t)batch * a.exp_batch;
  fill_int_kernel<<<(int)std::min<int64_t>((n_exp + 255) / 256, 152 * 4), 256, 0, s>>>(a.exps, n_exp, SL_ZERO);
  if (NS == 7 && BITS == 8 && a.colscale && a.x_batch == 0) {
    const int64_t want = std::max<int64_t>(1, 152 * 16 / std::max<int64_t>(1, a.rows));
    const int64_t nch = std::max<int64_t>(std::min<int64_t>(want, (a.K + 2047) / 2048), (a.K + 8191) / 8192);
    slice_max_scaled_kernel<<<dim3(a.rows, (unsigned)nch), 256, 0, s>>>(a, batch, (a.K + nch - 1) / nch);
    const int gx = (int)std::min<int64_t>((2 * (int64_t)a.nkb + 31) / 32, 1024);
    slice_rows_scaled_kernel<<<dim3(a.rows_p / 8, gx), 256, 0, s>>>(a, batch);
  } else if (!a.cols) {
    // about eight blocks per SM over rows, chunks and the batch
    const int64_t want = std::max<int64_t>(1, 152 * 8 / std::max<int64_t>(1, (int64_t)a.rows * batch));
    const int64_t nch = std::min<int64_t>(want, (a.K + 2047) / 2048);
    const int64_t chunk = (a.K + nch - 1) / nch;
    slice_max_rows_kernel<<<dim3(a.rows, (unsigned)nch, batch), 256, 0, s>>>(a, BITS, chunk);
    const int gx = (int)std::min<int64_t>((2 * (int64_t)a.nkb + 31) / 32, 64);
    slice_rows_tiles_kernel<NS, BITS><<<dim3(a.rows_p / 8, gx, batch), 256, 0, s>>>(a);
  } else {
    const int64_t want = std::max<int64_t>(1, 152 * 8 / std::max<int64_t>(1, (int64_t)((a.rows + 31) / 32) * batch));
    const int64_t nch = std::min<int64_t>(want, (a.K + 63) / 64);
    const int64_t chunk = (a.K + nch - 1) / nch;
    slice_max_cols_kernel<<<dim3((a.rows + 31) / 32, (unsigned)nch, batch), 256, 0, s>>>(a, BITS, chunk);
    const int gy = (int)std::min<int64_t>(((int64_t)a.nkb + 3) / 4, 64);
    slice_cols_tiles_kernel<NS, BITS><<<dim3(a.rows_p / 64, gy, batch), 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

template <int NS, int BITS, int NL = NS>
cudaError_t launch_ns(const SliceGemmArgs &g, int blocks, cudaStream_t s) {
  static OncePerDevice smem_limit;
  const cudaError_t e = smem_limit([] {
    return cudaFuncSetAttribute(slice_gemm_kernel<NS, BITS, NL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sg_smem(NS));
  });
  if (e != cudaSuccess) return e;
  slice_gemm_kernel<NS, BITS, NL><<<blocks, SG_THREADS, sg_smem(NS), s>>>(g);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_slice_operand(const SliceSrc &a, int ns, int bits, int batch, cudaStream_t s) {
  if (a.rows < 1 || a.K < 1 || batch < 1 || batch > 65535 || a.rows > a.rows_p || a.rows_p % 128 ||
      (int64_t)a.nkb * 16 < a.K || a.exp_batch < a.rows_p || (a.cols && (a.colscale || a.only_if)) ||
      (!a.cols && a.col_group) || a.kb_first < 0 || a.kb_first >= a.nkb || ((a.kb_first || a.fixed_exp) && !a.cols))
    return cudaErrorInvalidValue;
  if (bits == 8) return ns == 7 ? slice_operand<7, 8>(a, batch, s) : cudaErrorInvalidValue;
  switch (bits == 7 ? ns : 0) {
    case 2: return slice_operand<2, 7>(a, batch, s);
    case 3: return slice_operand<3, 7>(a, batch, s);
    case 4: return slice_operand<4, 7>(a, batch, s);
    case 5: return slice_operand<5, 7>(a, batch, s);
    case 6: return slice_operand<6, 7>(a, batch, s);
    case 7: return slice_operand<7, 7>(a, batch, s);
    case 8: return slice_operand<8, 7>(a, batch, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_fill_int(int *p, int64_t n, int v, cudaStream_t s) {
  fill_int_kernel<<<(int)std::min<int64_t>((n + 255) / 256, 152 * 4), 256, 0, s>>>(p, n, v);
  return cudaGetLastError();
}

cudaError_t launch_slice_pair(const SlicePairSrc &a, cudaStream_t s) {
  if (a.rows < 1 || a.rows > a.rows_p || a.rows_p % 128 || a.nk < SL_K || a.nk > 64 || a.nk % SL_K) return cudaErrorInvalidValue;
  slice_pair_kernel<<<a.rows_p / SL_ROWS, 512, 0, s>>>(a);
  return cudaGetLastError();
}

void slice_gemm_tiles(SliceGemmArgs *g) {
  const int tm = (g->M + SG_M - 1) / SG_M;
  g->tiles_n = (g->N + SG_N - 1) / SG_N;
  g->n_tiles = g->sym ? tm * (tm + 1) : tm * g->tiles_n;
  // FP32 sums of one level stay below 2^24: in base 256 a level adds at most
  // ns products of 2^14 per k; in base 128 only the leading digits reach 128
  // (two of a level's products, or the leading level's one of 2^14)
  const int per_k = g->bits == 8 ? g->ns << 14 : std::max(1 << 14, (g->ns + 2) << 12);
  g->drain_kb = (1 << 24) / per_k / SL_K;
  // base 256: the products of level 9 (six per k, about 2^-57.6 sqrt(6 K) of the
  // rows' scales together) stay below an FP64 sum's own rounding, which grows
  // with K, from a few thousand on; shorter contractions take them too
  if (!g->levels) g->levels = g->bits == 8 && (g->nkb - g->kb_first) < 256 ? g->ns + 1 : g->ns;
}

size_t slice_gemm_piece(SliceGemmArgs *g) {
  slice_gemm_tiles(g);
  return g->splits > 1 ? (size_t)g->splits * g->batch * g->n_tiles * SG_M * SG_N * sizeof(double) : 0;
}

size_t slice_gemm_plan(SliceGemmArgs *g, int n_sm, size_t max_partial) {
  slice_gemm_tiles(g);
  const int nkb = g->nkb - g->kb_first;
  const int64_t units = (int64_t)g->batch * g->n_tiles;
  int best = 1;
  double cost_best = 1e300;
  const size_t part1 = (size_t)units * SG_M * SG_N * sizeof(double);
  for (int sp = 1; sp <= 64; ++sp) {
    if (sp > 1 && (g->cd_out || nkb / sp < 8 || (size_t)sp * part1 > max_partial)) break;
    const int64_t waves = (units * sp + n_sm - 1) / n_sm;
    // per unit: its blocks, and about five blocks' time for the exposed drain
    // and store; a split also pays the reduction's pass over its partials
    const double cost = (double)waves * (5.0 + (double)((nkb + sp - 1) / sp)) + (sp > 1 ? 6.0 + 2.0 * sp * units / n_sm : 0.0);
    if (cost < cost_best) { cost_best = cost; best = sp; }
  }
  g->kb_per_split = (nkb + best - 1) / best;
  g->splits = (nkb + g->kb_per_split - 1) / g->kb_per_split;
  return slice_gemm_piece(g);
}

cudaError_t launch_slice_gemm(const SliceGemmArgs &g, int n_sm, cudaStream_t s) {
  const int64_t units = (int64_t)g.batch * g.splits * g.n_tiles;
  if (g.M < 1 || g.N < 1 || g.batch < 1 || g.kb_first < 0 || g.nkb <= g.kb_first || g.splits < 1 ||
      g.kb_per_split < 1 || g.drain_kb < 1 || g.n_tiles < 1 || (g.splits > 1 && !g.partial) ||
      (g.splits == 1 && g.partial) || (g.b_sel && !g.B_alt) || (g.sym && g.M != g.N) || !g.A || !g.B || !g.ea || !g.eb || !g.err || (!g.cd_out && !g.C) || (g.cd_out && (g.sym || g.partial)))
    return cudaErrorInvalidValue;
  const int blocks = (int)std::min<int64_t>(units, n_sm);
  cudaError_t e = cudaErrorInvalidValue;
  switch (g.bits == 8 ? (g.ns == 7 ? 78 : 0) : (g.bits == 7 ? g.ns : 0)) {
    case 2: e = launch_ns<2, 7>(g, blocks, s); break;
    case 3: e = launch_ns<3, 7>(g, blocks, s); break;
    case 4: e = launch_ns<4, 7>(g, blocks, s); break;
    case 5: e = launch_ns<5, 7>(g, blocks, s); break;
    case 6: e = launch_ns<6, 7>(g, blocks, s); break;
    case 7: e = launch_ns<7, 7>(g, blocks, s); break;
    case 8: e = launch_ns<8, 7>(g, blocks, s); break;
    case 78: e = g.levels == 8 ? launch_ns<7, 8, 8>(g, blocks, s) : launch_ns<7, 8>(g, blocks, s); break;
  }
  if (e != cudaSuccess) return e;
  if (g.partial) {
    const int64_t total = (int64_t)g.n_tiles * SG_M * SG_N;
    const int bx = (int)std::min<int64_t>((total + 255) / 256, 152 * 8);
    slice_reduce_kernel<<<dim3(bx, g.batch), 256, 0, s>>>(g, g.partial);
    e = cudaGetLastError();
  } else if (g.sym && g.mirror) {
    e = launch_mirror_upper(g.C, g.M, g.ldc, g.c_batch, g.batch, s);
  }
  return e;
}

cudaError_t launch_mirror_upper(double *C, int N, int64_t ldc, int64_t batch_stride, int batch, cudaStream_t s) {
  const int t = (N + 31) / 32;
  mirror_upper_kernel<<<dim3(t, t, batch), dim3(32, 8), 0, s>>>(C, N, ldc, batch_stride);
  return cudaGetLastError();
}

cudaError_t launch_slice_coldot_reduce(const SliceGemmArgs &g, double *W, int64_t ldw, cudaStream_t s) {
  slice_coldot_reduce_kernel<<<dim3(std::min((g.M + 127) / 128, 256), g.batch), 128, 0, s>>>(
      g.cd_out, 4 * g.tiles_n, g.cd_ldo, g.M, W, ldw);
  return cudaGetLastError();
}

}  // namespace ltgw
