// Entries of Pi that the digit contraction (slice_gemm.cu) may hold with fewer
// bits than an FP64 sum: found from the leading digits, and summed in FP64.
//
// Digits are integers of a row's common scale, so an entry (i, j) of K terms is
// off by up to K 2^-57 2^(e_i + e_j) with eight levels of digit pairs, where an FP64
// sum is off by up to K 2^-53 S, S = sum_k |a_ik| |a_jk|: less, where the rows are
// large on different pairs and S lies far below their scales.  (Seven levels drop
// products of 2^-58.3 in the mean square, sqrt(K) 2^-58.3 in all: no more beside an
// FP64 sum's mean error sqrt(K) 2^-54.7 S from the same S on, 2^-4 of the scales.)
// Since |a| 2^(8 - e) >= |d| - 1/2 for the leading digit d (exact in BF16), one BF16
// product
//   sum_k (|d_i| - 1/2) (|d_j| - 1/2) <= S 2^(16 - e_i - e_j)
// bounds S from below; an entry is weak while this has not reached 2^16 / 16, and
// entries of rows that are not finite are (their FP64 sums keep the sign of an
// infinity).
//
// One block per 64 x 64 tile of the lower triangle: four groups of 16 rows by four
// of every fourth 16-k block.  The groups' sums are added up at growing intervals
// and the scan ends when every entry has passed: rows of Gaussian entries take a
// few hundred k whatever K is, so the scan's latency is its cost and not its
// products; mma.sync needs no tensor memory and reads the fragments straight from
// the digits' blocks.  Measured: 0.03 of 2.22 ms for eight moments of N = 453 and
// 27,000 pairs (eight groups, one block per SM: 0.04; two groups 0.11), 0.02 of 0.30
// at N = 200 and 5,000 pairs, 0.012 of 0.08 at N = 48 and 64 pairs (32 frequencies).
//
// Weak entries: up to PW_WHOLE of a tile one per warp at a time (a clock of the
// FP64 pipe per entry and pair), more by the whole tile (2048 clocks per pair).
// Rows localised so that nearly every entry is weak: N = 453, 27,000 pairs, eight
// moments 60 ms, the FP64 tiles alone 56.
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"
#include "kernels.cuh"
#include "pair_scale.cuh"

namespace ltgw {
namespace {

constexpr int PW_STRIP = 256, PW_WHOLE = 1024, PW_BK = 16;

// |d| - 1/2, at least 0, of two digits.
__device__ __forceinline__ uint32_t digit_floor(uint32_t d2) {
  const uint32_t a = d2 & 0x7fff7fffu;
  const __nv_bfloat162 v = __hmax2(__hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&a), __float2bfloat162_rn(0.5f)),
                                   __float2bfloat162_rn(0.0f));
  return *reinterpret_cast<const uint32_t *>(&v);
}

struct PwSmem {
  union {
    float S[64][66];
    struct { double a[PW_BK][65], b[PW_BK][65]; } tile;
  };
  double sc[PW_STRIP];
  unsigned bits[64][2];
  unsigned short list[PW_WHOLE];
  int exi[64], exj[64], n_list;
};

constexpr int KG = 4, THREADS = 128 * KG, WARPS = 4 * KG;

__global__ void __launch_bounds__(THREADS, 2) pi_weak_kernel(PiWeakArgs g) {
  __shared__ PwSmem sm;
  const int b = blockIdx.y, t = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int I = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((I + 1) * (I + 2) / 2 <= t) ++I;
  while (I * (I + 1) / 2 > t) --I;
  const int i0 = I * 64, j0 = (t - I * (I + 1) / 2) * 64;
  const int *ex = g.exps + (int64_t)b * g.exp_batch;
  if (tid < 64) sm.exi[tid] = i0 + tid < g.N ? ex[i0 + tid] : SL_ZERO;
  else if (tid < 128) sm.exj[tid - 64] = j0 + tid - 64 < g.N ? ex[j0 + tid - 64] : SL_ZERO;
  for (int e = tid; e < 64 * 64; e += THREADS) sm.S[e >> 6][e & 63] = 0.0f;
  if (tid == 0) sm.n_list = 0;
  __syncthreads();

  // ---- the scan
  constexpr int64_t BLK = SL_ROWS * SL_K * 2;   // one digit of a 64-row, 16-k block
  constexpr float thr = 3968.0f;   // 0.97 of 2^16 / 16: a row's square passes with one entry, (64 - 1/2)^2
  const int64_t row_bytes = (int64_t)g.nkb * 7 * BLK;
  const uint8_t *A = g.dig + (int64_t)b * g.dig_batch + (i0 / 64) * row_bytes;
  const uint8_t *B = g.dig + (int64_t)b * g.dig_batch + (j0 / 64) * row_bytes;
  // a row's 32 bytes, their halves exchanged where bit 2 of the row is set (the same for rows 8 apart)
  const int kg = warp >> 2, r = (warp & 3) * 16 + (lane >> 2), rb0 = lane >> 2, c = lane & 3;
  const int ra = r * 32 + (((r >> 2) & 1) << 4) + 4 * c, rb = rb0 * 32 + (((rb0 >> 2) & 1) << 4) + 4 * c;
  int kb = kg;
  bool open = true;
  for (int steps = 3; open; steps *= 3) {
    float acc[8][4] = {};
    for (int s = 0; s < steps && kb < g.nkb; ++s, kb += KG) {
      const uint8_t *a = A + (int64_t)kb * 7 * BLK, *p = B + (int64_t)kb * 7 * BLK;
      uint32_t fa[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)   // rows r, r + 8, then their upper eight k
        fa[u] = digit_floor(__ldg(reinterpret_cast<const uint32_t *>(a + ((ra + (u & 1) * 256) ^ ((u >> 1) << 4)))));
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        const uint32_t b0 = digit_floor(__ldg(reinterpret_cast<const uint32_t *>(p + rb + n * 256)));
        const uint32_t b1 = digit_floor(__ldg(reinterpret_cast<const uint32_t *>(p + ((rb + n * 256) ^ 16))));
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(acc[n][0]), "+f"(acc[n][1]), "+f"(acc[n][2]), "+f"(acc[n][3])
            : "r"(fa[0]), "r"(fa[1]), "r"(fa[2]), "r"(fa[3]), "r"(b0), "r"(b1));
      }
    }
    for (int q = 0; q < KG; ++q) {   // the groups one after the other: exact sums below 2^22
      if (q == kg)
#pragma unroll
        for (int n = 0; n < 8; ++n)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float2 *d = reinterpret_cast<float2 *>(&sm.S[r + 8 * h][8 * n + 2 * c]);
            float2 v = *d;
            v.x += acc[n][2 * h];
            v.y += acc[n][2 * h + 1];
            *d = v;
          }
      __syncthreads();
    }
    bool waits = false;   // an entry that further k could pass
    for (int e = tid; e < 64 * 64; e += THREADS) {
      const int ei = sm.exi[e >> 6], ej = sm.exj[e & 63];
      waits |= j0 + (e & 63) <= i0 + (e >> 6) && ei != SL_ZERO && ej != SL_ZERO && ei < SL_NONFINITE && ej < SL_NONFINITE &&
               !(sm.S[e >> 6][e & 63] >= thr);
    }
    // every round that follows takes at least one group on
    const bool left = __syncthreads_or(kb < g.nkb);
    open = __syncthreads_or(waits) && left;
  }

  // ---- the weak entries
  int mine = 0;
  for (int q = 0; q < 4096 / THREADS; ++q) {
    const int e = tid + q * THREADS, i = e >> 6, j = e & 63, ei = sm.exi[i], ej = sm.exj[j];
    bool weak = false;
    if (i0 + i < g.N && j0 + j <= i0 + i) {
      if (ei >= SL_NONFINITE || ej >= SL_NONFINITE) weak = true;
      else weak = ei != SL_ZERO && ej != SL_ZERO && !(sm.S[i][j] >= thr);
    }
    const unsigned m = __ballot_sync(0xffffffffu, weak);
    if (lane == 0) sm.bits[i][j >> 5] = m;
    mine += weak;
  }
  if (!__syncthreads_or(mine)) return;
  if (mine) atomicAdd(&sm.n_list, mine);
  __syncthreads();
  const int total = sm.n_list;
  const double p0 = g.p0[b], p1 = g.p1 ? g.p1[b] : 0.0;
  const double *sgn = g.sgn ? g.sgn + (int64_t)b * g.f_batch : nullptr, *mag = g.mag ? g.mag + (int64_t)b * g.f_batch : nullptr;
  auto scale = [&](int64_t k) { return sgn ? sgn[k] * mag[k] : pair_scale(g.mode, g.delta[k], p0, p1); };
  double *C = g.C + (int64_t)b * g.N * g.N;
  if (total > PW_WHOLE) {
    constexpr int U = 64 / WARPS;   // rows per thread
    double acc[U][2] = {};
    for (int64_t k0 = 0; k0 < g.K; k0 += PW_BK) {
      __syncthreads();
#pragma unroll
      for (int e = tid; e < 64 * PW_BK; e += THREADS) {
        const int k = e % PW_BK, rr = e / PW_BK;
        const int64_t kk = k0 + k;
        const bool in = kk < g.K;
        sm.tile.a[k][rr] = in && i0 + rr < g.N ? g.X[(int64_t)(i0 + rr) * g.ld + kk] * scale(kk) : 0.0;
        sm.tile.b[k][rr] = in && j0 + rr < g.N ? g.X[(int64_t)(j0 + rr) * g.ld + kk] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < PW_BK; ++k) {
        const double b0 = sm.tile.b[k][lane], b1 = sm.tile.b[k][lane + 32];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const double x = sm.tile.a[k][warp + WARPS * u];
          acc[u][0] = fma(x, b0, acc[u][0]);
          acc[u][1] = fma(x, b1, acc[u][1]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int i = warp + WARPS * u, j = lane + 32 * v;
        if (i0 + i < g.N && j0 + j <= i0 + i) {
          C[(int64_t)(i0 + i) * g.N + j0 + j] = g.alpha * acc[u][v];
          C[(int64_t)(j0 + j) * g.N + i0 + i] = g.alpha * acc[u][v];
        }
      }
    return;
  }
  __syncthreads();
  if (tid == 0) sm.n_list = 0;
  __syncthreads();
  for (int e = tid; e < 64 * 64; e += THREADS)
    if (sm.bits[e >> 6][(e & 63) >> 5] >> (e & 31) & 1u) sm.list[atomicAdd(&sm.n_list, 1)] = (unsigned short)e;
  __syncthreads();
  for (int q0 = 0; q0 < total; q0 += WARPS) {
    const int q = q0 + warp;
    const int i = i0 + (sm.list[min(q, total - 1)] >> 6), j = j0 + (sm.list[min(q, total - 1)] & 63);
    double v = 0.0;
    for (int64_t k0 = 0; k0 < g.K; k0 += PW_STRIP) {
      __syncthreads();
      for (int k = tid; k < PW_STRIP && k0 + k < g.K; k += THREADS) sm.sc[k] = scale(k0 + k);
      __syncthreads();
      const int len = (int)min((int64_t)PW_STRIP, g.K - k0);
      const double *x = g.X + (int64_t)i * g.ld + k0, *y = g.X + (int64_t)j * g.ld + k0;
#pragma unroll 2
      for (int k = lane; k < len; k += 32) v = fma(x[k] * sm.sc[k], y[k], v);
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && q < total) {
      C[(int64_t)i * g.N + j] = g.alpha * v;
      C[(int64_t)j * g.N + i] = g.alpha * v;
    }
  }
}

}  // namespace

cudaError_t launch_pi_weak(const PiWeakArgs &a, int batch, cudaStream_t s) {
  if (a.N < 1 || batch < 1 || batch > 65535 || a.nkb < 1 || a.K < 1 || !a.dig || !a.exps ||
      !a.X || !a.C || !a.delta || !a.p0 || (!a.sgn != !a.mag))
    return cudaErrorInvalidValue;
  const int t = (a.N + 63) / 64;
  pi_weak_kernel<<<dim3(t * (t + 1) / 2, batch), THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace ltgw
