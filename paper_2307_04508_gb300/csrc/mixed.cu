// Bandwidth-bound helpers of the mixed-precision (split-BF16) path: FP32
// padded operand copies, the per-pair scale table of the polarisability
// (fused into the tensor-core operand load), and the FP64 reduction of the
// split-K partial tiles into full symmetric matrices.
#include <math.h>

#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <climits>
#include <cuda_fp8.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace ltgw {
namespace {

__global__ void to_f32_padded_kernel(const double *__restrict__ src, int64_t lds, int rows, int64_t cols,
                                     float *__restrict__ dst, int64_t cols_p) {
  const int r = blockIdx.y;
  const double *s = src + (int64_t)r * lds;
  float *d = dst + (int64_t)r * cols_p;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cols_p;
       c += (int64_t)gridDim.x * blockDim.x)
    d[c] = (r < rows && c < cols) ? (float)s[c] : 0.0f;
}

__global__ void scale_table_kernel(const double *__restrict__ delta, int64_t K, int64_t Kp,
                                   const double *__restrict__ p0, const double *__restrict__ p1,
                                   int mode, float *__restrict__ scale) {
  const int t = blockIdx.y;
  const double a = p0 ? p0[t] : 0.0, b = p1 ? p1[t] : 0.0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < Kp;
       k += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    if (k < K) {
      const double d = delta ? delta[k] : 0.0;
      v = (mode == SCALE_DIRECT) ? d / (a * a + d * d)
          : (mode == SCALE_LAPLACE) ? b * d * exp(-d * d * a)
          : (mode == SCALE_EXPTAU) ? exp(-d * a) : 1.0;
    }
    scale[(int64_t)t * Kp + k] = (float)v;
  }
}

// Sum of FP32 partials as an unevaluated pair hi + lo of FP32 numbers
// (Knuth's TwoSum per term; about 48 significant bits): the FP32 partials
// carry errors of 2^-24 of their own, so the pair's sum equals their FP64 sum
// far below that, and FP32 additions run many times faster than FP64 ones on
// this part (where the FP64 sum made the reductions FP64-bound).
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  lo += (hi - (s - bp)) + (x - bp);
  hi = s;
}

// Sums of the partial tiles, scaled, into both triangles of M, t = blockIdx.y.
// Small matrices: one thread per element (i >= j) of the lower triangle.  The
// FP64 conversions bound this step there, and the blocks below convert whole
// 128 x 128 tiles: 32 matrices of N = 130, 7.8 us against 11.5; N = 100 with 35
// partials per element, 13 against 19.  From RS_SMALL on the blocks are no slower
// (whole Pi, 70,000 pairs: N = 200 626 us by elements, 621 by blocks; N = 300 1104
// and 1098).
constexpr int RS_SMALL = 160;
__global__ void tc_reduce_sym_small_kernel(const double *__restrict__ partial, const float *__restrict__ partial32,
                                           int splits, int groups, int n_tiles, const int *__restrict__ tile_index,
                                           int nJ, int N, int nt_group, int colmajor, double alpha, double beta,
                                           double *__restrict__ M) {
  const int t = blockIdx.y, grp = t / nt_group, slot = t % nt_group;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * (N + 1) / 2) return;
  // e -> (a, b), a >= b, b fastest (an FP32 estimate corrected by integer tests);
  // column-major tiles take (i, j) = (N-1-b, N-1-a) so that consecutive threads
  // read consecutive rows of one column
  int a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while ((a + 1) * (a + 2) / 2 <= e) ++a;
  while (a * (a + 1) / 2 > e) --a;
  const int b = e - a * (a + 1) / 2;
  const int i = colmajor ? N - 1 - b : a, j = colmajor ? N - 1 - a : b;
  const int64_t step = (int64_t)groups * nt_group * n_tiles * (128 * 128);
  const int64_t at = (((int64_t)grp * nt_group + slot) * n_tiles + tile_index[(i / 128) * nJ + j / 128]) * (128 * 128) +
                     (colmajor ? (j % 128) * 128 + i % 128 : (i % 128) * 128 + j % 128);
  double acc = 0.0;
  if (partial32) {
    float hi = 0.0f, lo = 0.0f;
    for (int s = 0; s < splits; ++s) two_sum_acc(hi, lo, partial32[at + s * step]);
    acc = (double)hi + (double)lo;
  } else {
    for (int s = 0; s < splits; ++s) acc += partial[at + s * step];
  }
  acc *= alpha;
  double *m = M + (int64_t)t * N * N;
  if (beta != 0.0) acc += beta * m[(int64_t)i * N + j];
  m[(int64_t)i * N + j] = acc;
  m[(int64_t)j * N + i] = acc;
}

// Larger ones: a block takes a strip of 16 x 64 entries of a 128 x 128 tile
// (tiles I >= J, elements i >= j).  Bound by memory: the partials are read four
// entries of one column (row, unless colmajor) at a time, and the strip goes
// through shared memory so that the stores of both triangles run along M's rows.
// Ten matrices of N = 2258: with 35 partials per entry 908 us by elements, 700
// here (reading the partials alone takes about 580); with 5 partials 341 and 220.
// Strips of 64 x 64 are as fast there, but too few blocks for N of a few hundred
// (N = 400, 20,000 pairs, 10 points: 306 us for the whole Pi against 294).
template <bool colmajor>
__global__ void __launch_bounds__(256) tc_reduce_sym_kernel(const double *__restrict__ partial,
                                                            const float *__restrict__ partial32, int splits,
                                                            int groups, int n_tiles,
                                                            const int *__restrict__ tile_index, int nJ, int N,
                                                            int nt_group, double alpha, double beta,
                                                            double *__restrict__ M) {
  constexpr int SLOW = 16, FAST = 64;
  __shared__ double sm[SLOW][FAST + 1];   // [slow][fast]: fast runs along the partials
  const int t = blockIdx.y, grp = t / nt_group, slot = t % nt_group;
  const int strip = blockIdx.x & 7, half = (blockIdx.x >> 3) & 1, pair = blockIdx.x >> 4;
  int I = (int)((sqrtf(8.0f * (float)pair + 1.0f) - 1.0f) * 0.5f);   // corrected by integer tests
  while ((I + 1) * (I + 2) / 2 <= pair) ++I;
  while (I * (I + 1) / 2 > pair) --I;
  const int J = pair - I * (I + 1) / 2;
  constexpr int EI = colmajor ? FAST : SLOW, EJ = colmajor ? SLOW : FAST;   // the block's rows and columns of M
  const int i0 = I * 128 + (colmajor ? half : strip) * EI, j0 = J * 128 + (colmajor ? strip : half) * EJ;
  if (i0 >= N || j0 >= N || i0 + EI <= j0) return;
  const int tile = tile_index[I * nJ + J], tid = threadIdx.x;
  const int f = (tid & 15) * 4, sl = tid >> 4;
  const int64_t step = (int64_t)groups * nt_group * n_tiles * (128 * 128);
  const int64_t base = (((int64_t)grp * nt_group + slot) * n_tiles + tile) * (128 * 128) +
                       (strip * SLOW + sl) * 128 + half * FAST + f;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  if (partial32) {
    float hi[4] = {}, lo[4] = {};
#pragma unroll 4
    for (int s = 0; s < splits; ++s) {
      const float4 x = __ldcs(reinterpret_cast<const float4 *>(partial32 + base + s * step));
      two_sum_acc(hi[0], lo[0], x.x);
      two_sum_acc(hi[1], lo[1], x.y);
      two_sum_acc(hi[2], lo[2], x.z);
      two_sum_acc(hi[3], lo[3], x.w);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = (double)hi[u] + (double)lo[u];
  } else {
    for (int s = 0; s < splits; ++s)
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] += partial[base + s * step + u];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) sm[sl][f + u] = acc[u] * alpha;
  __syncthreads();
  double *Mt = M + (int64_t)t * N * N;
#pragma unroll
  for (int r = tid / EJ; r < EI; r += 256 / EJ) {   // (i, j), j along the threads
    const int c = tid % EJ, i = i0 + r, j = j0 + c;
    if (i < N && i >= j) {
      double &v = colmajor ? sm[c][r] : sm[r][c];
      double *d = Mt + (int64_t)i * N + j;
      if (beta != 0.0) v += beta * *d;
      *d = v;
    }
  }
  if (beta != 0.0) __syncthreads();
#pragma unroll
  for (int r = tid / EI; r < EJ; r += 256 / EI) {   // (j, i), i along the threads
    const int c = tid % EI, i = i0 + c, j = j0 + r;
    if (i < N && i > j) Mt[(int64_t)j * N + i] = colmajor ? sm[r][c] : sm[c][r];
  }
}

// dst[c][r] = src[r][c0 + c] (FP64 -> FP32), zero padding, 32 x 32 tiles through smem.
__global__ void to_f32_transposed_kernel(const double *__restrict__ src, int64_t lds, int64_t c0, int rows,
                                         int cols, float *__restrict__ dst, int rows_p, int cols_p,
                                         int64_t strideS, int64_t strideD) {
  __shared__ float tile[32][33];
  const int b = blockIdx.z;
  const double *S = src + b * strideS + c0;
  float *D = dst + b * strideD;
  const int r0 = blockIdx.y * 32, cb = blockIdx.x * 32;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = r0 + q, c = cb + threadIdx.x;
    tile[q][threadIdx.x] = (r < rows && c < cols) ? (float)S[(int64_t)r * lds + c] : 0.0f;
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int c = cb + q, r = r0 + threadIdx.x;
    if (c < cols_p && r < rows_p) D[(int64_t)c * rows_p + r] = tile[threadIdx.x][q];
  }
}

// dst[c][r] = src[r][c0 + c] in FP64, r < rows, c < cols (batched).
__global__ void transpose_f64_kernel(const double *__restrict__ src, int64_t lds, int64_t c0, int rows, int cols,
                                     double *__restrict__ dst, int64_t ldd, int64_t strideS, int64_t strideD) {
  __shared__ double tile[32][33];
  const int b = blockIdx.z;
  const double *S = src + b * strideS + c0;
  double *D = dst + b * strideD;
  const int r0 = blockIdx.y * 32, cb = blockIdx.x * 32;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = r0 + q, c = cb + threadIdx.x;
    if (r < rows && c < cols) tile[q][threadIdx.x] = S[(int64_t)r * lds + c];
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int c = cb + q, r = r0 + threadIdx.x;
    if (c < cols && r < rows) D[(int64_t)c * ldd + r] = tile[threadIdx.x][q];
  }
}

// Full-grid partial tiles -> FP64 and/or FP32 padded output, per group.
__global__ void tc_reduce_full_kernel(const double *__restrict__ partial, const float *__restrict__ partial32,
                                      int splits, int groups, int n_tiles, int nJ, int rows, int cols,
                                      double alpha, double *__restrict__ out64, int64_t ld64, int64_t stride64,
                                      float *__restrict__ out32, int64_t ld32, int64_t cols32, int rows_p32,
                                      int64_t stride32) {
  const int g = blockIdx.z;
  const int r = blockIdx.y;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < (out32 ? cols32 : cols);
       c += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    if (r < rows && c < cols) {
      const int tile = (r / 128) * nJ + (int)(c / 128);
      const int64_t off = (int64_t)(r % 128) * 128 + (c % 128);
      if (partial32) {
        float hi = 0.0f, lo = 0.0f;
        for (int s = 0; s < splits; ++s)
          two_sum_acc(hi, lo, partial32[(((int64_t)s * groups + g) * n_tiles + tile) * (128 * 128) + off]);
        acc = (double)hi + (double)lo;
      } else {
        for (int s = 0; s < splits; ++s) acc += partial[(((int64_t)s * groups + g) * n_tiles + tile) * (128 * 128) + off];
      }
      acc *= alpha;
      if (out64) out64[g * stride64 + (int64_t)r * ld64 + c] = acc;
    }
    if (out32 && r < rows_p32) out32[g * stride32 + (int64_t)r * ld32 + c] = (float)acc;
  }
}

__global__ void tc_reduce_coldot_kernel(const float *__restrict__ cd, int splits, int groups, int n_tile_rows,
                                        int cols_p, int cols, double *__restrict__ W, int64_t ldw) {
  const int g = blockIdx.y;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += gridDim.x * blockDim.x) {
    float hi = 0.0f, lo = 0.0f;
    for (int s = 0; s < splits; ++s)
      for (int I = 0; I < n_tile_rows; ++I) two_sum_acc(hi, lo, cd[(((int64_t)s * groups + g) * n_tile_rows + I) * cols_p + c]);
    W[(int64_t)g * ldw + c] = (double)hi + (double)lo;
  }
}

}  // namespace

cudaError_t launch_to_f32_padded(const double *src, int64_t lds, int rows, int64_t cols, float *dst,
                                 int rows_p, int64_t cols_p, cudaStream_t s) {
  if (rows_p <= 0 || cols_p <= 0) return cudaSuccess;
  int bx = (int)((cols_p + 255) / 256);
  if (bx > 64) bx = 64;
  dim3 grid(bx, rows_p);
  to_f32_padded_kernel<<<grid, 256, 0, s>>>(src, lds, rows, cols, dst, cols_p);
  return cudaGetLastError();
}

cudaError_t launch_scale_table(const double *delta, int64_t K, int64_t Kp, int n_t, const double *p0,
                               const double *p1, int mode, float *scale, cudaStream_t s) {
  if (n_t <= 0) return cudaSuccess;
  int bx = (int)((Kp + 255) / 256);
  if (bx > 152) bx = 152;
  dim3 grid(bx, n_t);
  scale_table_kernel<<<grid, 256, 0, s>>>(delta, K, Kp, p0, p1, mode, scale);
  return cudaGetLastError();
}

cudaError_t launch_tc_reduce_sym(const double *partial, const float *partial32, int splits, int groups,
                                 int n_tiles, const int *tile_index, int nJ, int n_t, int N, double alpha,
                                 double *M, cudaStream_t s, double beta, int nt_group, int colmajor) {
  if (N <= 0 || n_t <= 0) return cudaSuccess;
  const int nI = (N + 127) / 128;
  if (nt_group < 1 || (n_t + nt_group - 1) / nt_group != groups) return cudaErrorInvalidValue;
  if (N < RS_SMALL) {
    tc_reduce_sym_small_kernel<<<dim3((N * (N + 1) / 2 + 255) / 256, n_t), 256, 0, s>>>(
        partial, partial32, splits, groups, n_tiles, tile_index, nJ, N, nt_group, colmajor, alpha, beta, M);
  } else {
    const auto kernel = colmajor ? tc_reduce_sym_kernel<true> : tc_reduce_sym_kernel<false>;
    kernel<<<dim3(nI * (nI + 1) / 2 * 16, n_t), 256, 0, s>>>(partial, partial32, splits, groups, n_tiles, tile_index,
                                                             nJ, N, nt_group, alpha, beta, M);
  }
  return cudaGetLastError();
}

}  // namespace ltgw

namespace ltgw {

cudaError_t launch_to_f32_transposed(const double *src, int64_t lds, int64_t c0, int rows, int cols,
                                     float *dst, int rows_p, int cols_p, int batch, int64_t strideS,
                                     int64_t strideD, cudaStream_t s) {
  if (rows_p <= 0 || cols_p <= 0 || batch <= 0) return cudaSuccess;
  dim3 block(32, 8), grid((cols_p + 31) / 32, (rows_p + 31) / 32, batch);
  to_f32_transposed_kernel<<<grid, block, 0, s>>>(src, lds, c0, rows, cols, dst, rows_p, cols_p, strideS, strideD);
  return cudaGetLastError();
}

cudaError_t launch_tc_reduce_full(const double *partial, const float *partial32, int splits, int groups,
                                  int n_tiles, int nJ, int rows, int cols, double alpha, double *out64,
                                  int64_t ld64, int64_t stride64, float *out32, int64_t ld32,
                                  int rows_p32, int64_t stride32, cudaStream_t s, int64_t cols32) {
  if (cols32 < 0) cols32 = ld32;
  const int nrows = out32 ? std::max(rows, rows_p32) : rows;
  const int64_t ncols = out32 ? cols32 : cols;
  if (nrows <= 0 || ncols <= 0 || groups <= 0) return cudaSuccess;
  int bx = (int)((ncols + 255) / 256);
  if (bx > 64) bx = 64;
  dim3 grid(bx, nrows, groups);
  tc_reduce_full_kernel<<<grid, 256, 0, s>>>(partial, partial32, splits, groups, n_tiles, nJ, rows, cols, alpha,
                                             out64, ld64, stride64, out32, ld32, cols32, rows_p32, stride32);
  return cudaGetLastError();
}

cudaError_t launch_transpose_f64(const double *src, int64_t lds, int64_t c0, int rows, int cols, double *dst,
                                 int64_t ldd, int batch, int64_t strideS, int64_t strideD, cudaStream_t s) {
  if (rows <= 0 || cols <= 0 || batch <= 0) return cudaSuccess;
  dim3 block(32, 8), grid((cols + 31) / 32, (rows + 31) / 32, batch);
  transpose_f64_kernel<<<grid, block, 0, s>>>(src, lds, c0, rows, cols, dst, ldd, strideS, strideD);
  return cudaGetLastError();
}

cudaError_t launch_tc_reduce_coldot(const float *cd_out, int splits, int groups, int n_tile_rows, int cols_p,
                                    int cols, double *W, int64_t ldw, cudaStream_t s) {
  if (cols <= 0 || groups <= 0) return cudaSuccess;
  int bx = (cols + 255) / 256;
  if (bx > 64) bx = 64;
  dim3 grid(bx, groups);
  tc_reduce_coldot_kernel<<<grid, 256, 0, s>>>(cd_out, splits, groups, n_tile_rows, cols_p, cols, W, ldw);
  return cudaGetLastError();
}


namespace {
__global__ void split_bf16_kernel(const float *__restrict__ x, __nv_bfloat16 *__restrict__ hi,
                                  __nv_bfloat16 *__restrict__ lo, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float v = x[i];
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    hi[i] = h;
    lo[i] = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}
}  // namespace

cudaError_t launch_split_bf16(const float *x, __nv_bfloat16 *hi, __nv_bfloat16 *lo, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 152 * 16);
  split_bf16_kernel<<<(int)blocks, 256, 0, s>>>(x, hi, lo, n);
  return cudaGetLastError();
}

namespace {
constexpr int Q8_THREADS = 256;
constexpr float E4M3_MAX = 448.0f;   // largest finite FP8 E4M3 value

__device__ __forceinline__ float block_max(float v, float *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float m = 0.0f;
#pragma unroll
  for (int i = 0; i < Q8_THREADS / 32; ++i) m = fmaxf(m, red[i]);
  return m;
}

// four E4M3 codes (round to nearest even, saturating) of x * inv, packed low byte first
__device__ __forceinline__ uint32_t e4m3x4(float4 x, float inv) {
  const __nv_fp8x2_storage_t lo = __nv_cvt_float2_to_fp8x2(make_float2(x.x * inv, x.y * inv), __NV_SATFINITE, __NV_E4M3);
  const __nv_fp8x2_storage_t hi = __nv_cvt_float2_to_fp8x2(make_float2(x.z * inv, x.w * inv), __NV_SATFINITE, __NV_E4M3);
  return (uint32_t)lo | ((uint32_t)hi << 16);
}

// E4M3 values of four packed codes (exact in FP32)
__device__ __forceinline__ float4 e4m3x4_value(uint32_t c) {
  const __half2_raw a = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(c & 0xffffu), __NV_E4M3);
  const __half2_raw b = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(c >> 16), __NV_E4M3);
  const float2 fa = __half22float2(__half2(a)), fb = __half22float2(__half2(b));
  return make_float4(fa.x, fa.y, fb.x, fb.y);
}

// Codes of xs = x * inv (one term), or (split) of its two-term expansion h + l
// with h = e4m3(xs) and l = e4m3(xs - h) (exact in FP32), both in the
// row's scaled units: the row's three segments of Kq codes are written as
// pattern[0..2] of {h, l} (A operands h | l | h, B operands h | h | l, so that
// one accumulator sums h_a h_b + l_a h_b + h_a l_b).
__device__ __forceinline__ void codes_of(float4 x, float inv, uint32_t *h, uint32_t *l) {
  *h = e4m3x4(x, inv);
  const float4 hv = e4m3x4_value(*h);
  *l = e4m3x4(make_float4(__fsub_rn(__fmul_rn(x.x, inv), hv.x), __fsub_rn(__fmul_rn(x.y, inv), hv.y),
                          __fsub_rn(__fmul_rn(x.z, inv), hv.z), __fsub_rn(__fmul_rn(x.w, inv), hv.w)),
              1.0f);
}
__device__ __forceinline__ void write_codes(uint32_t *row, int64_t k, int64_t q4, float4 x, float inv, int split,
                                            bool a_pattern) {
  uint32_t h, l;
  codes_of(x, inv, &h, &l);
  row[k] = h;
  if (!split) return;
  row[q4 + k] = a_pattern ? l : h;
  row[2 * q4 + k] = a_pattern ? h : l;
}
// The same for 16 consecutive values, 16 bytes per segment.
__device__ __forceinline__ void write_codes4(uint32_t *row, int64_t k, int64_t q4, const float4 x[4], float inv,
                                             int split, bool a_pattern) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) codes_of(x[v], inv, &h[v], &l[v]);
  const uint4 hh = make_uint4(h[0], h[1], h[2], h[3]), ll = make_uint4(l[0], l[1], l[2], l[3]);
  *reinterpret_cast<uint4 *>(row + k) = hh;
  if (!split) return;
  *reinterpret_cast<uint4 *>(row + q4 + k) = a_pattern ? ll : hh;
  *reinterpret_cast<uint4 *>(row + 2 * q4 + k) = a_pattern ? hh : ll;
}

// Row r of X [rows][Kp] (FP32; Kp a multiple of 16): the row's scale inv = 448 /
// max_k |X_rk| and codes qb[r][k] = e4m3(X_rk inv); for each of the n_t factor
// rows S[t] the products p = X_rk S_tk (FP32) get their own scale and codes
// qa[t][r][k].  De-scales 1 / inv (0 for a zero row) go to ds_b[r] and
// ds_a[t][r]; code columns Kp..Kq-1 are zero.  split: each code row holds three
// segments of Kq (the two-term expansion, write_codes).
//
// Two kernels over (8 rows, a chunk of k, T factor rows): the maxima, then the
// codes.  A warp takes one row, so the eight warps of a block share the factor
// rows' chunk through L1, and the grid fills the SMs whatever the row count.
// Bound: HBM, n_t times three code bytes per value.  N = 611, 20,001 pairs, 32
// frequencies (1.2 GB of codes): 0.55 ms with the maxima; one block per row with all 32 factor
// rows in its registers took 1.09 ms.  Few rows: a block's chain of loads bounds
// it, so fewer factor rows and a shorter chunk per block where those of eight
// rows and 512 float4 would not fill the SMs (whole Pi, 32 frequencies: N = 120, 4,000
// pairs 121 -> 107 us, N = 300, 1,500 pairs 147 -> 133; N = 611, 20,001 pairs would be
// 1262 instead of 1191).
constexpr int Q8_ROWS = Q8_THREADS / 32;
constexpr int Q8_CHUNK = 512, Q8_CHUNK_FEW = 128;   // float4 per row and block (more for rows past 1.3e8 values)
constexpr int64_t Q8_FEW = 152 * 8;                 // blocks

// maxima (float bits, zeroed beforehand) [n_t][rows] of |X_rk S_tk|, then [rows] of |X_rk|
template <int T>
__global__ void __launch_bounds__(Q8_THREADS)
    fp8_max_kernel(const float *__restrict__ X, int64_t Kp, const float *__restrict__ S, int n_t, int rows,
                   int64_t chunk, int *__restrict__ maxima) {
  const int r = blockIdx.x * Q8_ROWS + (threadIdx.x >> 5), lane = threadIdx.x & 31, t0 = blockIdx.z * T;
  if (r >= rows) return;
  const float4 *xr = reinterpret_cast<const float4 *>(X + (int64_t)r * Kp);
  const int64_t n4 = Kp / 4, k0 = (int64_t)blockIdx.y * chunk, k1 = min(n4, k0 + chunk);
  float mb = 0.0f, ma[T] = {};
  for (int64_t k = k0 + lane; k < k1; k += 32) {
    const float4 x = xr[k];
    mb = fmaxf(mb, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
#pragma unroll
    for (int u = 0; u < T; ++u)
      if (t0 + u < n_t) {
        const float4 sv = __ldg(reinterpret_cast<const float4 *>(S + (int64_t)(t0 + u) * Kp) + k);
        ma[u] = fmaxf(ma[u], fmaxf(fmaxf(fabsf(x.x * sv.x), fabsf(x.y * sv.y)), fmaxf(fabsf(x.z * sv.z), fabsf(x.w * sv.w))));
      }
  }
#pragma unroll
  for (int u = 0; u < T; ++u) {   // magnitudes order as their bits
    const int m = __reduce_max_sync(0xffffffffu, __float_as_int(ma[u]));
    if (lane == 0 && t0 + u < n_t && m) atomicMax(maxima + (int64_t)(t0 + u) * rows + r, m);
  }
  const int m = __reduce_max_sync(0xffffffffu, __float_as_int(mb));
  if (lane == 0 && t0 == 0 && m) atomicMax(maxima + (int64_t)n_t * rows + r, m);
}

__device__ __forceinline__ float e4m3_inv(int max_bits) {
  const float m = __int_as_float(max_bits);
  return m > 0.0f ? E4M3_MAX / m : 0.0f;
}

template <int T>
__global__ void __launch_bounds__(Q8_THREADS)
    fp8_quantize_kernel(const float *__restrict__ X, int64_t Kp, int64_t Kq, const float *__restrict__ S, int n_t,
                        int rows, int64_t chunk, const int *__restrict__ maxima, uint8_t *__restrict__ qa, uint8_t *__restrict__ qb,
                        float *__restrict__ ds_a, float *__restrict__ ds_b, int split) {
  const int r = blockIdx.x * Q8_ROWS + (threadIdx.x >> 5), lane = threadIdx.x & 31, t0 = blockIdx.z * T;
  if (r >= rows) return;
  const float4 *xr = reinterpret_cast<const float4 *>(X + (int64_t)r * Kp);
  const int64_t n4 = Kp / 4, q4 = Kq / 4, k0 = (int64_t)blockIdx.y * chunk, k1 = min(q4, k0 + chunk);
  const int64_t Ks = split ? 3 * Kq : Kq;   // codes per row
  const float invb = e4m3_inv(maxima[(int64_t)n_t * rows + r]);
  float inv[T];
#pragma unroll
  for (int u = 0; u < T; ++u) inv[u] = t0 + u < n_t ? e4m3_inv(maxima[(int64_t)(t0 + u) * rows + r]) : 0.0f;
  if (blockIdx.y == 0 && lane == 0) {
    if (t0 == 0) ds_b[r] = invb > 0.0f ? 1.0f / invb : 0.0f;
#pragma unroll
    for (int u = 0; u < T; ++u)
      if (t0 + u < n_t) ds_a[(int64_t)(t0 + u) * rows + r] = inv[u] > 0.0f ? 1.0f / inv[u] : 0.0f;
  }
  uint32_t *qbr = qb && t0 == 0 ? reinterpret_cast<uint32_t *>(qb + (int64_t)r * Ks) : nullptr;
  for (int64_t k = k0 + 4 * lane; k < k1; k += 128) {   // 16 values per lane: n4, q4 and the chunks are multiples of 4
    const bool in = k < n4;   // past the data: zero codes
    float4 x[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) x[v] = in ? xr[k + v] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (qbr) write_codes4(qbr, k, q4, x, invb, split, false);
#pragma unroll
    for (int u = 0; u < T; ++u)
      if (t0 + u < n_t) {
        float4 p[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const float4 sv = in ? __ldg(reinterpret_cast<const float4 *>(S + (int64_t)(t0 + u) * Kp) + k + v)
                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          p[v] = make_float4(x[v].x * sv.x, x[v].y * sv.y, x[v].z * sv.z, x[v].w * sv.w);
        }
        write_codes4(reinterpret_cast<uint32_t *>(qa + ((int64_t)(t0 + u) * rows + r) * Ks), k, q4, p, inv[u], split, true);
      }
  }
}

// The same with one block per row, which keeps the maxima of all factor rows (MAXT at
// most): one launch, and X and the factor rows stay in L1 between its two passes.
// For up to 12 factor rows of up to Q8_ROW_K codes; whole Pi with eight points,
// against the two kernels above: N = 200, 2,000 pairs 97 us (105), 8,000 130 (137),
// 15,000 181 (176); N = 2000, 8,000 pairs 1114 (1152), 15,000 1738 (1700).
constexpr int Q8_ROW_T = 12;
constexpr int64_t Q8_ROW_K = 12288;
template <int MAXT>
__global__ void __launch_bounds__(Q8_THREADS)
    fp8_quantize_rows_kernel(const float *__restrict__ X, int64_t Kp, int64_t Kq, const float *__restrict__ S, int n_t,
                        int rows, uint8_t *__restrict__ qa, uint8_t *__restrict__ qb, float *__restrict__ ds_a,
                        float *__restrict__ ds_b, int split) {
  __shared__ float red[Q8_THREADS / 32];
  __shared__ float inv_s[MAXT + 1];
  const int r = blockIdx.x;
  const float4 *xr = reinterpret_cast<const float4 *>(X + (int64_t)r * Kp);
  const int64_t n4 = Kp / 4, q4 = Kq / 4;
  float mb = 0.0f, ma[MAXT];
#pragma unroll
  for (int t = 0; t < MAXT; ++t) ma[t] = 0.0f;
  for (int64_t k = threadIdx.x; k < n4; k += Q8_THREADS) {
    const float4 x = xr[k];
    mb = fmaxf(mb, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
#pragma unroll
    for (int t = 0; t < MAXT; ++t) {
      if (t < n_t) {
        const float4 sv = reinterpret_cast<const float4 *>(S + (int64_t)t * Kp)[k];
        ma[t] = fmaxf(ma[t], fmaxf(fmaxf(fabsf(x.x * sv.x), fabsf(x.y * sv.y)),
                                   fmaxf(fabsf(x.z * sv.z), fabsf(x.w * sv.w))));
      }
    }
  }
  mb = block_max(mb, red);
  if (threadIdx.x == 0) inv_s[MAXT] = mb > 0.0f ? E4M3_MAX / mb : 0.0f;
#pragma unroll
  for (int t = 0; t < MAXT; ++t) {
    if (t < n_t) {
      const float m = block_max(ma[t], red);
      if (threadIdx.x == 0) inv_s[t] = m > 0.0f ? E4M3_MAX / m : 0.0f;
    }
  }
  __syncthreads();
  const float invb = inv_s[MAXT];
  if (threadIdx.x == 0) {
    ds_b[r] = invb > 0.0f ? 1.0f / invb : 0.0f;
    for (int t = 0; t < n_t; ++t) ds_a[(int64_t)t * rows + r] = inv_s[t] > 0.0f ? 1.0f / inv_s[t] : 0.0f;
  }
  const int64_t Ks = split ? 3 * Kq : Kq;   // codes per row
  uint32_t *qbr = qb ? reinterpret_cast<uint32_t *>(qb + (int64_t)r * Ks) : nullptr;
  for (int64_t k = threadIdx.x; k < q4; k += Q8_THREADS) {
    if (k >= n4) {
      for (int seg = 0; seg < (split ? 3 : 1); ++seg) {
        if (qbr) qbr[seg * q4 + k] = 0u;
        for (int t = 0; t < n_t; ++t) reinterpret_cast<uint32_t *>(qa + ((int64_t)t * rows + r) * Ks)[seg * q4 + k] = 0u;
      }
      continue;
    }
    const float4 x = xr[k];
    if (qbr) write_codes(qbr, k, q4, x, invb, split, false);
#pragma unroll
    for (int t = 0; t < MAXT; ++t) {
      if (t < n_t) {
        const float4 sv = reinterpret_cast<const float4 *>(S + (int64_t)t * Kp)[k];
        const float4 p = make_float4(x.x * sv.x, x.y * sv.y, x.z * sv.z, x.w * sv.w);
        write_codes(reinterpret_cast<uint32_t *>(qa + ((int64_t)t * rows + r) * Ks), k, q4, p, inv_s[t], split, true);
      }
    }
  }
}
// One block per row r of X [rows][Kp]: codes of X itself as an A operand
// (split: segments h | l | h), de-scale to ds[r].
__global__ void __launch_bounds__(Q8_THREADS)
    fp8_quantize_a_kernel(const float *__restrict__ X, int64_t Kp, int64_t Kq, int rows, uint8_t *__restrict__ q,
                          float *__restrict__ ds, int split) {
  __shared__ float red[Q8_THREADS / 32];
  const int r = blockIdx.x;
  const float4 *xr = reinterpret_cast<const float4 *>(X + (int64_t)r * Kp);
  const int64_t n4 = Kp / 4, q4 = Kq / 4;
  float m = 0.0f;
  for (int64_t k = threadIdx.x; k < n4; k += Q8_THREADS) {
    const float4 x = xr[k];
    m = fmaxf(m, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
  }
  m = block_max(m, red);
  const float inv = m > 0.0f ? E4M3_MAX / m : 0.0f;
  if (threadIdx.x == 0) ds[r] = inv > 0.0f ? 1.0f / inv : 0.0f;
  const int64_t Ks = split ? 3 * Kq : Kq;
  uint32_t *qr = reinterpret_cast<uint32_t *>(q + (int64_t)r * Ks);
  for (int64_t k = threadIdx.x; k < q4; k += Q8_THREADS) {
    if (k >= n4) {
      for (int seg = 0; seg < (split ? 3 : 1); ++seg) qr[seg * q4 + k] = 0u;
      continue;
    }
    write_codes(qr, k, q4, xr[k], inv, split, true);
  }
}
// FP64 per-pair factors f[t][k] of the Pi contraction, each operation rounded
// once (no fused multiply-add): Delta / (w_t^2 + Delta^2) (direct, p0 = w),
// (w_t Delta) exp(-Delta Delta x_t) (Laplace, p0 = x, p1 = w), exp(-Delta tau_t)
// (imaginary time, p0 = tau).
__device__ __forceinline__ double pi_factor64(int mode, double d, double a, double b) {
  if (mode == SCALE_DIRECT) return __ddiv_rn(d, __dadd_rn(__dmul_rn(a, a), __dmul_rn(d, d)));
  if (mode == SCALE_LAPLACE) return __dmul_rn(__dmul_rn(b, d), exp(__dmul_rn(__dmul_rn(-d, d), a)));
  return exp(__dmul_rn(-d, a));   // SCALE_EXPTAU: e^{-Delta tau_t}
}

__global__ void pi_factor64_kernel(const double *__restrict__ delta, int64_t K, const double *__restrict__ p0,
                                   const double *__restrict__ p1, int mode, double *__restrict__ f) {
  const int t = blockIdx.y;
  const double a = p0[t], b = p1 ? p1[t] : 0.0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.x * blockDim.x)
    f[(int64_t)t * K + k] = pi_factor64(mode, delta[k], a, b);
}

// sgn = sign(f) sqrt|f|, mag = sqrt|f| of the same factors; *neg is set if any f < 0.
__global__ void pi_root_factor_kernel(const double *__restrict__ delta, int64_t K, const double *__restrict__ p0,
                                      const double *__restrict__ p1, int mode, double *__restrict__ sgn,
                                      double *__restrict__ mag, int *__restrict__ neg) {
  const int t = blockIdx.y;
  const double a = p0[t], b = p1 ? p1[t] : 0.0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.x * blockDim.x) {
    const double f = pi_factor64(mode, delta[k], a, b);
    const double r = sqrt(fabs(f));
    if (f < 0.0) *neg = 1;
    sgn[(int64_t)t * K + k] = f < 0.0 ? -r : r;
    mag[(int64_t)t * K + k] = r;
  }
}
}  // namespace

cudaError_t launch_fp8_quantize(const float *X, int64_t Kp, int64_t Kq, const float *S, int n_t, int rows,
                                uint8_t *qa, uint8_t *qb, float *ds_a, float *ds_b, int *maxima, cudaStream_t s,
                                int split) {
  if (rows <= 0) return cudaSuccess;
  if (Kp % 16 || Kq % 16 || Kq < Kp || n_t < 0 || n_t > 32) return cudaErrorInvalidValue;   // Kp is padded to 64
  if (n_t > 0 && n_t <= Q8_ROW_T && Kq <= Q8_ROW_K) {
    const auto kernel = n_t <= 8 ? fp8_quantize_rows_kernel<8> : fp8_quantize_rows_kernel<Q8_ROW_T>;
    kernel<<<rows, Q8_THREADS, 0, s>>>(X, Kp, Kq, S, n_t, rows, qa, qb, ds_a, ds_b, split);
    return cudaGetLastError();
  }
  cudaError_t e = cudaMemsetAsync(maxima, 0, (size_t)(n_t + 1) * rows * sizeof(int), s);
  if (e != cudaSuccess) return e;
  const int64_t q4 = Kq / 4, least = ((q4 + 65534) / 65535 + 3) / 4 * 4;
  const int gx = (rows + Q8_ROWS - 1) / Q8_ROWS;
  auto run = [&](auto max_kernel, auto code_kernel, int64_t chunk, int t) {
    const dim3 grid(gx, (unsigned)((q4 + chunk - 1) / chunk), std::max(1, (n_t + t - 1) / t));
    max_kernel<<<grid, Q8_THREADS, 0, s>>>(X, Kp, S, n_t, rows, chunk, maxima);
    code_kernel<<<grid, Q8_THREADS, 0, s>>>(X, Kp, Kq, S, n_t, rows, chunk, maxima, qa, qb, ds_a, ds_b, split);
  };
  if (gx * ((q4 + Q8_CHUNK - 1) / Q8_CHUNK) * std::max(1, (n_t + 7) / 8) >= Q8_FEW)
    run(fp8_max_kernel<8>, fp8_quantize_kernel<8>, std::max<int64_t>(Q8_CHUNK, least), 8);
  else
    run(fp8_max_kernel<2>, fp8_quantize_kernel<2>, std::max<int64_t>(Q8_CHUNK_FEW, least), 2);
  return cudaGetLastError();
}

cudaError_t launch_pi_factor64(const double *delta, int64_t K, int n_t, const double *p0, const double *p1,
                               int mode, double *f, cudaStream_t st) {
  if (n_t <= 0 || K <= 0) return cudaSuccess;
  int bx = (int)((K + 255) / 256);
  if (bx > 152) bx = 152;
  pi_factor64_kernel<<<dim3(bx, n_t), 256, 0, st>>>(delta, K, p0, p1, mode, f);
  return cudaGetLastError();
}

cudaError_t launch_pi_root_factor(const double *delta, int64_t K, int n_t, const double *p0, const double *p1,
                                  int mode, double *sgn, double *mag, int *neg, cudaStream_t st) {
  if (n_t <= 0 || K <= 0) return cudaSuccess;
  int bx = (int)((K + 255) / 256);
  if (bx > 152) bx = 152;
  pi_root_factor_kernel<<<dim3(bx, n_t), 256, 0, st>>>(delta, K, p0, p1, mode, sgn, mag, neg);
  return cudaGetLastError();
}

cudaError_t launch_fp8_quantize_a(const float *X, int64_t Kp, int64_t Kq, int rows, uint8_t *q, float *ds,
                                  cudaStream_t s, int split) {
  if (rows <= 0) return cudaSuccess;
  if (Kp % 4 || Kq % 16 || Kq < Kp) return cudaErrorInvalidValue;
  fp8_quantize_a_kernel<<<rows, Q8_THREADS, 0, s>>>(X, Kp, Kq, rows, q, ds, split);
  return cudaGetLastError();
}

}  // namespace ltgw
