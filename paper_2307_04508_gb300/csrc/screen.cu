// Screening of Eq. ScreenedCoulombOrbital: C(i w_j) = [1 - Pi(i w_j)]^-1 - 1
// for every frequency, by the symmetric sweep operator (Gauss-Jordan without
// pivoting, stable here because 1 - Pi is symmetric positive definite with all
// eigenvalues >= 1).  After sweeping every pivot the matrix holds -A^-1.
//
// Two forms:
//  * launch_screen: one launch per pivot k for all frequencies, ping-ponging
//    between two buffers (first step forms A = 1 - Pi, last writes C = -X - 1);
//  * launch_screen_blocked: pivot blocks of 64 - the block is inverted by a
//    4-CTA cluster, and the rank-64 update A -= A[:,P] A_PP^-1 A[P,:] runs on
//    the FP64 tiled GEMM (about N/64 x 5 launches instead of N);
//  * launch_screen_digits: pivot blocks of 128, the update from integer digits
//    on the tensor cores (FP64-accurate, slice_gemm.cu).
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace ltgw {
namespace {

constexpr int SW_ROWS = 4;  // rows of one matrix per block

// grid: x = row group of SW_ROWS rows, y = frequency.  Threads stride over columns.
__global__ void __launch_bounds__(256) sweep_step_kernel(const double *__restrict__ in,
                                                         double *__restrict__ out, int N, int k,
                                                         int first, int last, int *flags) {
  const int b = blockIdx.y;
  const int64_t NN = (int64_t)N * N;
  const double *X = in + b * NN;
  double *Y = out + b * NN;
  const double *rowk = X + (int64_t)k * N;
  double p = rowk[k];
  if (first) p = 1.0 - p;
  if (blockIdx.x == 0 && threadIdx.x == 0 && !(p > 0.0 && isfinite(p)))
    atomicExch(&flags[FLAG_NOT_SPD], 1);
  const double rp = 1.0 / p;
  const double sg = first ? -1.0 : 1.0;  // first step reads 1 - Pi
  for (int q = 0; q < SW_ROWS; ++q) {
    const int i = blockIdx.x * SW_ROWS + q;
    if (i >= N) break;
    const double *rowi = X + (int64_t)i * N;
    double *yi = Y + (int64_t)i * N;
    double aik = sg * rowi[k];
    if (i == k && first) aik = p;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      double akj = sg * rowk[j] + ((first && j == k) ? 1.0 : 0.0);
      double aij = sg * rowi[j] + ((first && i == j) ? 1.0 : 0.0);
      double r;
      if (i == k && j == k) r = -rp;
      else if (i == k) r = akj * rp;
      else if (j == k) r = aik * rp;
      else r = aij - aik * akj * rp;
      if (last) r = -r - (i == j ? 1.0 : 0.0);
      yi[j] = r;
    }
  }
}

// ---- blocked sweep: pivot blocks of SB_B, rank-SB_B updates on the tiled GEMM ----
constexpr int SB_B = 64;

// X = I - Pi
template <typename T>
__global__ void form_a_kernel(const double *__restrict__ Pi, T *__restrict__ X, int N, int64_t total) {
  const int64_t NN = (int64_t)N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = e % NN;
    const int i = (int)(f / N), j = (int)(f - (int64_t)i * N);
    X[e] = (T)((i == j ? 1.0 : 0.0) - Pi[e]);
  }
}

// Z = X[P,P]^-1 for each frequency, by the sweep on a cluster of B / SB_RPC CTAs
// (one CTA per frequency would leave most SMs idle through the bs pivots).
// CTA c of the cluster holds rows SB_RPC*c .. SB_RPC*c + SB_RPC - 1 of the
// block in registers: warp w rows 4w .. 4w + 3 of them, lane l the column pairs
// 2l, 2l + 64, ... (B = 32: column l; the FP64 pipe's time is a warp's whatever its
// lanes hold, so a matrix of up to 32 rows does not take B = 64: N = 32, 32
// frequencies 138 us for the screening, 148 so).  Four pivots form a round: the warp that holds their rows
// sweeps those four rows alone (no other row changes them), writes the four
// rows, each scaled by its pivot's reciprocal at its turn, and the reciprocals
// into every CTA's shared memory; one cluster barrier; then every other row
// takes the four rank-1 updates in order.  The arithmetic per entry is that of
// one pivot at a time.  The buffers alternate with the round's parity, so the
// writes of one round never meet the reads of the round before.  UPPER: only
// the block's upper triangle is read (the matrix is known to be symmetric).
// Bound: the owner warp's chain of division, scaled row and three rank-1 rows
// per pivot (B = 64: 90 us for 32 blocks, 85 us with one pivot per barrier),
// and for B = 128 the FP64 pipe beside it (2.1e6 multiply-adds a block, two CTAs
// on most SMs: 276 us for 32 blocks, 460 us with one pivot per barrier).
constexpr int SB_RPC = 16;                   // rows per CTA
constexpr int SB_PR = 4;                     // pivots per round = rows per warp
constexpr int SB_THREADS = SB_RPC / SB_PR * 32;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void st_cluster_2f64(uint32_t local_addr, unsigned rank, double v0, double v1) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(remote), "d"(v0), "d"(v1) : "memory");
}

__device__ __forceinline__ void st_cluster_f64(uint32_t local_addr, unsigned rank, double v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}

template <int B, bool UPPER>
__global__ void __cluster_dims__(B / SB_RPC, 1, 1) __launch_bounds__(SB_THREADS)
    block_inverse_kernel(const double *__restrict__ X, int N, int p0, int bs, double *__restrict__ Z, int *flags) {
  constexpr int NC = B / 32;          // columns per lane, in pairs (B = 32: one)
  constexpr int LDZ = B == 32 ? 64 : B;
  static_assert(B == 32 || B == 64 || B == 128, "one column or one or two column pairs per lane");
  __shared__ __align__(16) double rowk[2][SB_PR][B];
  __shared__ __align__(16) double rpk[2][SB_PR];
  unsigned crank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
  const int b = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = (int)crank * SB_RPC + SB_PR * warp;
  const double *Xb = X + (int64_t)b * N * N;
  auto col = [&](int h) { return NC == 1 ? lane : 2 * lane + 64 * (h >> 1) + (h & 1); };
  // entry (row r of the warp, block column c), in every lane
  auto at = [&](const double (&v)[SB_PR][NC], int r, int c) {
    if (NC == 1) return __shfl_sync(0xffffffffu, v[r][0], c);
    double x = (c & 1) ? v[r][NC > 1] : v[r][0];
    if (NC > 2) {
      const double y = (c & 1) ? v[r][NC - 1] : v[r][NC > 1 ? NC - 2 : 0];
      if (c >= 64) x = y;
    }
    return __shfl_sync(0xffffffffu, x, (c & 63) >> 1);
  };
  double v[SB_PR][NC];
#pragma unroll
  for (int r = 0; r < SB_PR; ++r)
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const int i = i0 + r, j = col(h);
      const int a = UPPER ? min(i, j) : i, c = UPPER ? max(i, j) : j;
      v[r][h] = (i < bs && j < bs) ? Xb[(int64_t)(p0 + a) * N + (p0 + c)] : 0.0;
    }
  const uint32_t rowk_addr = (uint32_t)__cvta_generic_to_shared(&rowk[0][0][0]);
  const uint32_t rpk_addr = (uint32_t)__cvta_generic_to_shared(&rpk[0][0]);
  cluster_sync();   // every CTA of the cluster is running before the first remote write
  for (int k0 = 0; k0 < bs; k0 += SB_PR) {
    const int par = (k0 / SB_PR) & 1, np = min(SB_PR, bs - k0);
    const bool owner = (int)crank == k0 / SB_RPC && warp == (k0 % SB_RPC) / SB_PR;
    if (owner) {
      double rps[SB_PR] = {};
#pragma unroll
      for (int j = 0; j < SB_PR; ++j) {
        if (j < np) {
          const int k = k0 + j;
          const double piv = at(v, j, k);
          if (lane == 0 && !(piv > 0.0 && isfinite(piv))) atomicExch(&flags[FLAG_NOT_SPD], 1);
          const double rp = 1.0 / piv;
          rps[j] = rp;
          double a[NC], c[SB_PR];
#pragma unroll
          for (int r = 0; r < SB_PR; ++r) c[r] = r == j ? 0.0 : at(v, r, k);
#pragma unroll
          for (int h = 0; h < NC; ++h) a[h] = v[j][h] * rp;
          const uint32_t row = rowk_addr + (uint32_t)((par * SB_PR + j) * B + col(0)) * sizeof(double);
#pragma unroll
          for (unsigned cta = 0; cta < B / SB_RPC; ++cta) {
            if constexpr (NC == 1) {
              st_cluster_f64(row, cta, a[0]);
            } else {
#pragma unroll
              for (int h = 0; h < NC; h += 2) st_cluster_2f64(row + 32 * h * sizeof(double), cta, a[h], a[h + 1]);
            }
          }
#pragma unroll
          for (int h = 0; h < NC; ++h) {
            const bool at_k = col(h) == k;
#pragma unroll
            for (int r = 0; r < SB_PR; ++r) {
              if (r == j) v[r][h] = at_k ? -rp : a[h];
              else v[r][h] = at_k ? c[r] * rp : fma(-c[r], a[h], v[r][h]);
            }
          }
        }
      }
      if (lane < B / SB_RPC) {   // one CTA per lane
        st_cluster_2f64(rpk_addr + par * SB_PR * sizeof(double), lane, rps[0], rps[1]);
        st_cluster_2f64(rpk_addr + (par * SB_PR + 2) * sizeof(double), lane, rps[2], rps[3]);
      }
    }
    cluster_sync();
    if (!owner) {
#pragma unroll
      for (int j = 0; j < SB_PR; ++j) {
        const int k = k0 + j;
        if (j < np) {
          const double rp = rpk[par][j];
          double c[SB_PR], ck[SB_PR];
#pragma unroll
          for (int r = 0; r < SB_PR; ++r) { c[r] = at(v, r, k); ck[r] = c[r] * rp; }
          if constexpr (NC == 1) {
            const double a = rowk[par][j][lane];
#pragma unroll
            for (int r = 0; r < SB_PR; ++r) v[r][0] = lane == k ? ck[r] : fma(-c[r], a, v[r][0]);
          } else {
#pragma unroll
            for (int h = 0; h < NC; h += 2) {
              const double2 a = *reinterpret_cast<const double2 *>(&rowk[par][j][2 * lane + 32 * h]);
#pragma unroll
              for (int r = 0; r < SB_PR; ++r) {
                v[r][h] = col(h) == k ? ck[r] : fma(-c[r], a.x, v[r][h]);
                v[r][h + 1] = col(h + 1) == k ? ck[r] : fma(-c[r], a.y, v[r][h + 1]);
              }
            }
          }
        }
      }
    }
  }
  cluster_sync();   // no CTA leaves while another may still write to it
  double *Zb = Z + (int64_t)b * LDZ * LDZ;
#pragma unroll
  for (int r = 0; r < SB_PR; ++r)
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const int i = i0 + r, j = col(h);
      if (i < bs && j < bs) Zb[i * LDZ + j] = -v[r][h];
    }
}

// rowsP[b][r][j] = X[b][p0 + r][j]
template <typename T>
__global__ void copy_rows_kernel(const T *__restrict__ X, int N, int p0, int bs, T *__restrict__ rowsP) {
  const int b = blockIdx.z, r = blockIdx.y;
  const T *src = X + (int64_t)b * N * N + (int64_t)(p0 + r) * N;
  T *dst = rowsP + ((int64_t)b * SB_B + r) * N;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) dst[j] = src[j];
}

// X[:, P] = R, X[P, :] = R^T, X[P, P] = -Z
template <typename T>
__global__ void fix_block_kernel(T *__restrict__ X, int N, int p0, int bs, const T *__restrict__ R,
                                 const T *__restrict__ Z) {
  const int b = blockIdx.y;
  T *Xb = X + (int64_t)b * N * N;
  const T *Rb = R + (int64_t)b * N * SB_B;
  const T *Zb = Z + (int64_t)b * SB_B * SB_B;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (int64_t)N * bs;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(q / bs), c = (int)(q % bs);
    const bool inP = i >= p0 && i < p0 + bs;
    const T v = inP ? -Zb[(i - p0) * SB_B + c] : Rb[(int64_t)i * SB_B + c];
    Xb[(int64_t)i * N + p0 + c] = v;
    if (!inP) Xb[(int64_t)(p0 + c) * N + i] = v;   // the P x P block is written once
  }
}

// C = -X - I
template <typename T>
__global__ void finish_c_kernel(const T *__restrict__ X, double *__restrict__ C, int N, int64_t total) {
  const int64_t NN = (int64_t)N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = e % NN;
    const int i = (int)(f / N), j = (int)(f - (int64_t)i * N);
    C[e] = -(double)X[e] - (i == j ? 1.0 : 0.0);
  }
}

template <typename T>
cudaError_t screen_blocked_impl(const double *Pi, int N, int n_omega, T *work, double *C, int *flags,
                                cudaStream_t s, int *launches) {
  const int64_t NN = (int64_t)N * N, total = NN * n_omega;
  T *X = work;
  T *R = X + total;
  T *rowsP = R + (int64_t)n_omega * N * SB_B;
  T *Z = rowsP + (int64_t)n_omega * SB_B * N;
  int eb = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  form_a_kernel<T><<<eb, 256, 0, s>>>(Pi, X, N, total);
  ++*launches;
  for (int p0 = 0; p0 < N; p0 += SB_B) {
    const int bs = std::min(SB_B, N - p0);
    if (N <= 32)
      block_inverse_kernel<32, false><<<dim3(32 / SB_RPC, n_omega), SB_THREADS, 0, s>>>(X, N, p0, bs, Z, flags);
    else
      block_inverse_kernel<SB_B, false><<<dim3(SB_B / SB_RPC, n_omega), SB_THREADS, 0, s>>>(X, N, p0, bs, Z, flags);
    dim3 cg((N + 255) / 256 < 8 ? (N + 255) / 256 : 8, bs, n_omega);
    copy_rows_kernel<T><<<cg, 256, 0, s>>>(X, N, p0, bs, rowsP);
    GemmArgs<T> g;   // R = X[:, P] Z
    g.M = N; g.N = bs; g.K = bs;
    g.A = X + p0; g.lda = N; g.strideA = NN;
    g.B = Z; g.ldb = SB_B; g.strideB = (int64_t)SB_B * SB_B;
    g.C = R; g.ldc = SB_B; g.strideC = (int64_t)N * SB_B;
    cudaError_t e = launch_gemm<T>(g, n_omega, true, false, s);
    if (e != cudaSuccess) return e;
    GemmArgs<T> u;   // X -= R X[P, :]  (= X[:, P] Z X[P, :], symmetric: lower tiles, mirrored)
    u.M = N; u.N = N; u.K = bs; u.syrk = 1;
    u.A = R; u.lda = SB_B; u.strideA = (int64_t)N * SB_B;
    u.B = rowsP; u.ldb = N; u.strideB = (int64_t)SB_B * N;
    u.C = X; u.ldc = N; u.strideC = NN;
    u.alpha = -1.0; u.beta = 1.0;
    e = launch_gemm<T>(u, n_omega, true, false, s);
    if (e != cudaSuccess) return e;
    dim3 fg((int)std::min<int64_t>(((int64_t)N * bs + 255) / 256, 64), n_omega);
    fix_block_kernel<T><<<fg, 256, 0, s>>>(X, N, p0, bs, R, Z);
    *launches += 5;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  finish_c_kernel<T><<<eb, 256, 0, s>>>(X, C, N, total);
  ++*launches;
  return cudaGetLastError();
}

// ---- blocked sweep with the updates from digits (slice_gemm.cu) ----
// Pivot blocks of SD_B; only the upper triangle (row <= column) of X is kept
// up to date.  Per block: Z = X[P,P]^-1, the panel X[:,P] as digits, R = X[:,P] Z,
// X -= R X[P,:] (the tiles with an upper entry), then X[:,P] = R, X[P,P] = -Z.
// Blocks of 128 and not 64: an update tile costs about 17,000 cycles whatever
// the block's length up to 144 (its drain, conversion and the sum with X), so
// half as many updates beat the dearer pivot blocks.  What bounds the step at
// N = 2258 (32 frequencies): the updates' epilogue, 0.65 of 1.3 ms per block;
// the pivot blocks 0.28 ms; digits 0.09 ms.  The whole step: 23.1 ms against
// 360.7 ms on the FP64 tiles (81 % of the FP64 pipe); N = 453: 1.71 against
// 5.58 ms, N = 160: 0.59 against 0.85 ms, error against 64-bit torch not larger
// at any size from 130 to 2258.
constexpr int SD_B = 128;
constexpr int SD_NS = 7, SD_BITS = 8;   // the FP64 digits; levels up to 8 (the ninth: error 1 % less, time 16 % more)

// X = I - Pi on the upper triangle (and what of the lower its 32-column blocks cover)
__global__ void form_upper_kernel(const double *__restrict__ Pi, double *__restrict__ X, int N) {
  const int i = blockIdx.y;
  const int64_t o = (int64_t)blockIdx.z * N * N + (int64_t)i * N;
  for (int j = (i & ~31) + blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x)
    X[o + j] = (i == j ? 1.0 : 0.0) - Pi[o + j];
}

// The same for a Pi that need not be symmetric: *asym is set where two mirrored
// entries differ by more than the rounding of a product of rows, 4 N u
// sqrt((1 - Pi_ii) (1 - Pi_jj)), or are not both numbers.  FP64 instructions run
// only where the bits differ.  Grid: 32 x 32 tiles (column, row, frequency).
__global__ void __launch_bounds__(256) form_upper_checked_kernel(const double *__restrict__ Pi, double *__restrict__ X,
                                                                 int N, int *__restrict__ asym) {
  __shared__ double t[32][33];
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  const double *P = Pi + (int64_t)blockIdx.z * N * N;
  double *Xb = X + (int64_t)blockIdx.z * N * N;
  const int tx = threadIdx.x, ty = threadIdx.y;
  double m[4], v[4];   // the mirrored tile and this one: eight loads at once
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = bj * 32 + ty + 8 * u, c = bi * 32 + tx, i = bi * 32 + ty + 8 * u, j = bj * 32 + tx;
    m[u] = r < N && c < N ? __ldcs(P + (int64_t)r * N + c) : 0.0;
    v[u] = i < N && j < N ? __ldcs(P + (int64_t)i * N + j) : 0.0;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) t[ty + 8 * u][tx] = m[u];
  __syncthreads();
  bool bad = false;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int q = ty + 8 * u, i = bi * 32 + q, j = bj * 32 + tx;
    if (i >= N || j >= N) continue;
    const double a = v[u], b = t[tx][q];
    Xb[(int64_t)i * N + j] = (i == j ? 1.0 : 0.0) - a;
    if (__double_as_longlong(a) != __double_as_longlong(b) || (__double2hiint(a) & 0x7ff00000) == 0x7ff00000) {
      const double di = 1.0 - P[(int64_t)i * N + i], dj = 1.0 - P[(int64_t)j * N + j];
      bad |= !(fabs(a - b) <= 4.0 * N * 0x1p-53 * sqrt(di * dj));
    }
  }
  if (bad) *asym = 1;
}

// P[b][i][c] = X[i][p0 + c] from the upper triangle, i < N, c < bs (ld SD_B).
// grid: (32-row blocks of i, 32-column blocks of c, frequency).
__global__ void __launch_bounds__(256) gather_panel_kernel(const double *__restrict__ X, int N, int p0, int bs,
                                                           double *__restrict__ P) {
  __shared__ double t[32][33];
  const int i0 = blockIdx.x * 32, c0 = blockIdx.y * 32, b = blockIdx.z;
  const double *Xb = X + (int64_t)b * N * N;
  double *Pb = P + (int64_t)b * N * SD_B;
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (i0 >= p0) {   // at or below the diagonal: row p0 + c, column i, through the tile
    for (int q = ty; q < 32; q += 8) {
      const int c = c0 + q, i = i0 + tx;
      if (c < bs && i < N) t[q][tx] = Xb[(int64_t)min(p0 + c, i) * N + max(p0 + c, i)];
    }
    __syncthreads();
    for (int q = ty; q < 32; q += 8) {
      const int i = i0 + q, c = c0 + tx;
      if (i < N && c < bs) Pb[(int64_t)i * SD_B + c] = t[tx][q];
    }
  } else {
    for (int q = ty; q < 32; q += 8) {
      const int i = i0 + q, c = c0 + tx;
      if (i < N && c < bs) Pb[(int64_t)i * SD_B + c] = Xb[(int64_t)i * N + p0 + c];
    }
  }
}

// The upper triangle's entries of X[:, P] = R, X[P, P] = -Z.
__global__ void __launch_bounds__(256) scatter_panel_kernel(double *__restrict__ X, int N, int p0, int bs,
                                                            const double *__restrict__ R,
                                                            const double *__restrict__ Z) {
  __shared__ double t[32][33];
  const int i0 = blockIdx.x * 32, c0 = blockIdx.y * 32, b = blockIdx.z;
  double *Xb = X + (int64_t)b * N * N;
  const double *Rb = R + (int64_t)b * N * SD_B, *Zb = Z + (int64_t)b * SD_B * SD_B;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int q = ty; q < 32; q += 8) {
    const int i = i0 + q, c = c0 + tx;
    double v = 0.0;
    if (i < N && c < bs) v = (i >= p0 && i < p0 + bs) ? -Zb[(i - p0) * SD_B + c] : Rb[(int64_t)i * SD_B + c];
    if (i < p0) {
      if (i < N && c < bs) Xb[(int64_t)i * N + p0 + c] = v;
    } else {
      t[q][tx] = v;
    }
  }
  if (i0 + 31 < p0) return;   // p0 is a multiple of 32: the whole block is above the panel
  __syncthreads();
  for (int q = ty; q < 32; q += 8) {
    const int c = c0 + q, i = i0 + tx;
    if (c < bs && i < N && i >= p0 + c) Xb[(int64_t)(p0 + c) * N + i] = t[tx][q];
  }
}

// C = -X - I, both triangles from the upper one.
__global__ void __launch_bounds__(256) finish_upper_kernel(const double *__restrict__ X, double *__restrict__ C, int N) {
  __shared__ double t[32][33];
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  const int64_t o = (int64_t)blockIdx.z * N * N;
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int r = bi * 32 + q, c = bj * 32 + threadIdx.x;
    if (r < N && c < N && r <= c) {
      const double v = -X[o + (int64_t)r * N + c] - (r == c ? 1.0 : 0.0);
      C[o + (int64_t)r * N + c] = v;
      t[q][threadIdx.x] = v;
    }
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int r = bj * 32 + q, c = bi * 32 + threadIdx.x;
    if (r < N && c < N && r > c) C[o + (int64_t)r * N + c] = t[threadIdx.x][q];
  }
}

struct SdScratch {
  double *Z;
  uint8_t *dP, *dR, *dZ;
  int *eP, *eR, *eZ;
  int64_t bP, bZ;   // digit bytes per frequency
  int Np;
};

size_t sd_layout(int N, int n_omega, void *base, SdScratch *o) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    void *p = base ? (char *)base + off : nullptr;
    off += (bytes + 255) / 256 * 256;
    return p;
  };
  o->Np = (int)slice_rows_padded(N);
  o->bP = slice_digit_bytes(N, SD_B / SL_K, SD_NS);
  o->bZ = slice_digit_bytes(SD_B, SD_B / SL_K, SD_NS);
  o->Z = (double *)take((size_t)n_omega * SD_B * SD_B * sizeof(double));
  o->dP = (uint8_t *)take((size_t)n_omega * o->bP);
  o->dR = (uint8_t *)take((size_t)n_omega * o->bP);
  o->dZ = (uint8_t *)take((size_t)n_omega * o->bZ);
  o->eP = (int *)take((size_t)n_omega * o->Np * sizeof(int));
  o->eR = (int *)take((size_t)n_omega * o->Np * sizeof(int));
  o->eZ = (int *)take((size_t)n_omega * SD_B * sizeof(int));
  return off;
}

}  // namespace

size_t screen_digit_bytes(int N, int n_omega) {
  SdScratch o;
  return sd_layout(N, n_omega, nullptr, &o);
}

cudaError_t launch_screen_digits(const double *Pi, int N, int n_omega, double *work, void *digits, double *C,
                                 int *flags, int n_sm, int *asym, cudaStream_t s, int *launches) {
  if (N <= 0 || n_omega <= 0) return cudaSuccess;
  if (n_omega > 65535 || N > 65535) return cudaErrorInvalidValue;
  const int64_t NN = (int64_t)N * N;
  double *X = work, *P = X + NN * n_omega;   // P, then R: [n_omega][N][SD_B]
  SdScratch o;
  sd_layout(N, n_omega, digits, &o);
  const int nt = (N + 31) / 32;
  if (asym)
    form_upper_checked_kernel<<<dim3(nt, nt, n_omega), dim3(32, 8), 0, s>>>(Pi, X, N, asym);
  else
    form_upper_kernel<<<dim3(std::min((N + 255) / 256, 8), N, n_omega), 256, 0, s>>>(Pi, X, N);
  ++*launches;
  for (int p0 = 0; p0 < N; p0 += SD_B) {
    const int bs = std::min(SD_B, N - p0), nkb = (bs + SL_K - 1) / SL_K;
    const dim3 pg((N + 31) / 32, (bs + 31) / 32, n_omega), tb(32, 8);
    block_inverse_kernel<SD_B, true><<<dim3(SD_B / SB_RPC, n_omega), SB_THREADS, 0, s>>>(X, N, p0, bs, o.Z, flags);
    gather_panel_kernel<<<pg, tb, 0, s>>>(X, N, p0, bs, P);
    SliceSrc a;
    a.X = P; a.ld = SD_B; a.x_batch = (int64_t)N * SD_B; a.rows = N; a.rows_p = o.Np; a.K = bs; a.nkb = nkb;
    a.dig = o.dP; a.dig_batch = o.bP; a.exps = o.eP; a.exp_batch = o.Np;
    cudaError_t e = launch_slice_operand(a, SD_NS, SD_BITS, n_omega, s);
    if (e != cudaSuccess) return e;
    SliceSrc z;
    z.X = o.Z; z.ld = SD_B; z.x_batch = SD_B * SD_B; z.rows = bs; z.rows_p = SD_B; z.K = bs; z.nkb = nkb;
    z.dig = o.dZ; z.dig_batch = o.bZ; z.exps = o.eZ; z.exp_batch = SD_B;
    e = launch_slice_operand(z, SD_NS, SD_BITS, n_omega, s);
    if (e != cudaSuccess) return e;
    SliceGemmArgs r;   // R[i][c] = sum_k Z[c][k] P[i][k] (over P: its digits are taken)
    r.A = o.dZ; r.a_batch = o.bZ; r.ea = o.eZ; r.ea_batch = SD_B;
    r.B = o.dP; r.b_batch = o.bP; r.eb = o.eP; r.eb_batch = o.Np;
    r.ns = SD_NS; r.bits = SD_BITS; r.nkb = nkb; r.batch = n_omega;
    r.levels = SD_NS; r.M = bs; r.N = N; r.C = P; r.ldc = SD_B; r.c_batch = (int64_t)N * SD_B; r.err = flags;
    slice_gemm_plan(&r, n_sm, 0);
    e = launch_slice_gemm(r, n_sm, s);
    if (e != cudaSuccess) return e;
    a.dig = o.dR; a.exps = o.eR;
    e = launch_slice_operand(a, SD_NS, SD_BITS, n_omega, s);
    if (e != cudaSuccess) return e;
    if (bs < N) {
      SliceGemmArgs u;   // X -= R X[P, :] on the tiles with an upper entry
      u.A = o.dP; u.a_batch = o.bP; u.ea = o.eP; u.ea_batch = o.Np;
      u.B = o.dR; u.b_batch = o.bP; u.eb = o.eR; u.eb_batch = o.Np;
      u.ns = SD_NS; u.bits = SD_BITS; u.nkb = nkb; u.batch = n_omega;
      u.levels = SD_NS; u.M = u.N = N; u.sym = 1; u.mirror = 0; u.C = X; u.ldc = N; u.c_batch = NN;
      u.beta = 1.0; u.alpha_neg = 1; u.err = flags;
      slice_gemm_plan(&u, n_sm, 0);
      e = launch_slice_gemm(u, n_sm, s);
      if (e != cudaSuccess) return e;
    }
    scatter_panel_kernel<<<pg, tb, 0, s>>>(X, N, p0, bs, P, o.Z);
    *launches += 8;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  finish_upper_kernel<<<dim3(nt, nt, n_omega), dim3(32, 8), 0, s>>>(X, C, N);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_screen(const double *Pi, int N, int n_omega, double *X0, double *X1,
                          double *C, int *flags, cudaStream_t s, int *launches) {
  if (N <= 0 || n_omega <= 0) return cudaSuccess;
  dim3 grid((N + SW_ROWS - 1) / SW_ROWS, n_omega);
  const int threads = N >= 256 ? 256 : (N >= 128 ? 128 : (N >= 64 ? 64 : 32));
  const double *in = Pi;
  for (int k = 0; k < N; ++k) {
    int last = (k == N - 1);
    double *out = last ? C : ((k & 1) ? X1 : X0);
    sweep_step_kernel<<<grid, threads, 0, s>>>(in, out, N, k, k == 0, last, flags);
    ++*launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    in = out;
  }
  return cudaSuccess;
}

}  // namespace ltgw

namespace ltgw {

size_t screen_blocked_scratch(int N, int n_omega) {
  return (size_t)n_omega * ((size_t)N * N + 2 * (size_t)N * SB_B + (size_t)SB_B * SB_B);
}

cudaError_t launch_screen_blocked(const double *Pi, int N, int n_omega, double *work, double *C, int *flags,
                                  cudaStream_t s, int *launches) {
  if (N <= 0 || n_omega <= 0) return cudaSuccess;
  return screen_blocked_impl<double>(Pi, N, n_omega, work, C, flags, s, launches);
}

}  // namespace ltgw
