// Symmetric eigensolver for the natural auxiliary functions (Sec. 2:
// diagonalise K, keep the eigenvectors whose eigenvalue exceeds eps_NAF).
//
//  1. Householder reduction K = Q T Q^T to tridiagonal T.  From n = 1000 on in
//     panels of 64 steps, whose rank-128 update comes from integer digits on the
//     tensor cores; the last 800 or so columns, and smaller matrices, in one
//     kernel that applies a rank-2 update per step;
//  2. Sturm-sequence count of the eigenvalues of T above the threshold;
//  3. multisection for the kept eigenvalues, with T in shared memory, its points
//     placed by an FP32 estimate and by secants;
//  4. their eigenvectors from twisted factorisations of T; inverse iteration
//     (tridiagonal LU with row interchanges, modified Gram-Schmidt inside groups
//     of nearly equal eigenvalues) for those that these leave, and where T does
//     not fit in shared memory;
//  5. one symmetric re-orthonormalisation X <- X (3 - X^T X)/2, which squares the
//     small non-orthogonality left between close eigenvalues without leaving the
//     span of X;
//  6. back-transformation U = Q X in compact-WY blocks of 64 reflectors, written
//     transposed as the rows of Ut.  Steps 5 and 6 from digits from n = 200 on, as
//     long as their scratch holds the digits (up to about 70 % of the vectors
//     kept), else on the FP64 units.
//
// FP64 accuracy in norm throughout (both the plain and the mixed-precision solve:
// only the dense contractions around the eigensolver change precision).  Only the
// kept eigenvectors are formed.  Householder convention: H = 1 - tau v v^T,
// v_0 = 1, H x = beta e_1.
//
// On this part an FP64 FMA has a dependent latency of about 64 cycles and an
// IEEE FP64 division about 400 (FP32 FMA: 4), so the sequential recurrences
// (Sturm counts, tridiagonal LU) are written to keep as few operations as
// possible on their dependency chains.
#include <float.h>

#include <algorithm>
#include <math.h>

#include "common.cuh"
#include "fast_fp64.cuh"
#include "kernels.cuh"
#include "per_device.h"

namespace ltgw {
namespace {

constexpr int RB = 1024;        // threads of the single-block kernels
constexpr int HH_MIN_ROWS = 4;  // fewest rows per block of the fused reduction

template <typename T> struct Lim;
template <> struct Lim<double> {
  static __device__ __forceinline__ double eps() { return DBL_EPSILON; }
  static __device__ __forceinline__ double tiny() { return DBL_MIN; }
  static constexpr double group_tol = 1e-7;   // inverse-iteration groups, relative to ||T||
};

__device__ __forceinline__ double block_sum(double v, double *sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    r = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    if (lane == 0) sh[0] = r;
  }
  __syncthreads();
  r = sh[0];
  __syncthreads();
  return r;
}

// ---- per-step kernels (FP64; used when a cooperative launch is not possible)
// Reflector for column k: x = A[k+1:n, k].
__global__ void __launch_bounds__(RB) hh_reflector_kernel(const double *A, double *V, double *d,
                                                          double *e, double *tau, double *scal,
                                                          int n, int k) {
  __shared__ double sh[32];
  const int L = n - k - 1;
  double s = 0.0;
  for (int i = 1 + threadIdx.x; i < L; i += blockDim.x) {
    double x = A[(int64_t)(k + 1 + i) * n + k];
    s = fma(x, x, s);
  }
  const double sigma = block_sum(s, sh);
  const double alpha = A[(int64_t)(k + 1) * n + k];
  double t, beta, sc;
  if (sigma == 0.0) {
    t = 0.0; beta = alpha; sc = 0.0;
  } else {
    double nrm = sqrt(alpha * alpha + sigma);
    beta = (alpha >= 0.0) ? -nrm : nrm;
    t = (beta - alpha) / beta;
    sc = 1.0 / (alpha - beta);
  }
  double *v = V + (int64_t)k * n + (k + 1);
  for (int i = threadIdx.x; i < L; i += blockDim.x)
    v[i] = (i == 0) ? 1.0 : A[(int64_t)(k + 1 + i) * n + k] * sc;
  if (threadIdx.x == 0) {
    d[k] = A[(int64_t)k * n + k];
    e[k] = beta;
    tau[k] = t;
    scal[0] = t;
  }
}

// p = tau * A22 v, one warp per row of the trailing block.
__global__ void hh_symv_kernel(const double *__restrict__ A, const double *__restrict__ V,
                               double *__restrict__ p, const double *__restrict__ scal, int n,
                               int k) {
  const int L = n - k - 1;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= L) return;
  const double *row = A + (int64_t)(k + 1 + warp) * n + (k + 1);
  const double *v = V + (int64_t)k * n + (k + 1);
  double s = 0.0;
  for (int j = lane; j < L; j += 32) s = fma(row[j], v[j], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) p[warp] = scal[0] * s;
}

// w = p - (tau/2)(p.v) v
__global__ void __launch_bounds__(RB) hh_w_kernel(const double *V, const double *p, double *w,
                                                  const double *scal, int n, int k) {
  __shared__ double sh[32];
  const int L = n - k - 1;
  const double *v = V + (int64_t)k * n + (k + 1);
  double s = 0.0;
  for (int i = threadIdx.x; i < L; i += blockDim.x) s = fma(p[i], v[i], s);
  const double gamma = 0.5 * scal[0] * block_sum(s, sh);
  for (int i = threadIdx.x; i < L; i += blockDim.x) w[i] = p[i] - gamma * v[i];
}

// A22 -= v w^T + w v^T
__global__ void hh_update_kernel(double *__restrict__ A, const double *__restrict__ V,
                                 const double *__restrict__ w, int n, int k) {
  const int L = n - k - 1;
  const double *v = V + (int64_t)k * n + (k + 1);
  const int64_t LL = (int64_t)L * L;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < LL;
       e += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(e / L), j = (int)(e - (int64_t)i * L);
    double *a = A + (int64_t)(k + 1 + i) * n + (k + 1 + j);
    *a -= v[i] * w[j] + w[i] * v[j];
  }
}

// Last diagonal / off-diagonal entries once every reflector is applied.
__global__ void hh_finalize_kernel(const double *A, double *d, double *e, int n) {
  if (threadIdx.x != 0) return;
  if (n >= 2) {
    d[n - 2] = A[(int64_t)(n - 2) * n + (n - 2)];
    e[n - 2] = A[(int64_t)(n - 1) * n + (n - 2)];
  }
  d[n - 1] = A[(int64_t)(n - 1) * n + (n - 1)];
  e[n - 1] = 0.0;
}

// ---- fused Householder reduction (one cooperative launch) ----
// All n-2 reflector steps in one kernel with ONE grid barrier per step.
// Writing A^(k) for the matrix after the first k rank-2 updates, reflector k
// comes from row k of A^(k) (= column k by symmetry), p_k = tau_k A^(k)_22 v_k,
// w_k = p_k - (tau_k/2)(p_k.v_k) v_k and A^(k+1)_22 = A^(k)_22 - v_k w_k^T - w_k v_k^T.
// Row r belongs to block r mod G for the whole reduction and stays in its
// shared memory.
// Step k:
//  phase 1 (every block, identical arithmetic, so every block holds the same
//    vectors): normalise v_{k-1}; p_{k-1}.v_{k-1} from the full p_{k-1} (so
//    no per-block partial sums are exchanged); w_{k-1}; row k of A^(k) from
//    row k of A^(k-1), which its owner published during step k-1, minus
//    update k-1; the coefficients of reflector k.  The reflector is kept
//    unnormalised, x = (alpha, x_{k+2}, ...), with v = (1, sc x_{k+2}, ...) and
//    sc = 1/(alpha - beta), so no extra pass is needed before phase 2;
//  phase 2 (own rows r > k): one pass that applies update k-1 and accumulates
//    s_r = sum_j A^(k)[r][j] x_j, then p_k[r] = tau sc (s_r - beta A^(k)[r][k+1]);
//    the owner of row k+1 copies that row to the published buffer;
//  grid barrier.
// p and the published row are double-buffered by step parity, so a block
// still reading step k-1's copies never sees step k's writes.  Data crossing
// blocks goes through L2 (ld.global.cg).  The barrier is bounded (about two
// seconds) and reports through flags.
struct GridBar {
  unsigned count;   // arrivals so far; barrier j (0-based) is passed at count >= G (j + 1)
  int abort;
};

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_add_release(unsigned *p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// Grid barrier number j: one release-add per block, then an acquire poll of
// the counter (bounded: about two seconds, then the abort flag and FLAG_EIG).
__device__ bool grid_barrier(GridBar *gb, unsigned j, int *flags) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = gridDim.x * (j + 1);
    red_add_release(&gb->count, 1u);
    if (ld_acquire(&gb->count) < target) {
      const uint64_t t0 = gtimer();
      unsigned it = 0;
      while (ld_acquire(&gb->count) < target) {
        if ((++it & 1023) == 0) {
          if (*(volatile int *)&gb->abort) { ok = 0; break; }
          if (gtimer() - t0 > 2000000000ull) {
            atomicExch(&flags[FLAG_EIG], 1);
            atomicExch(&gb->abort, 1);
            ok = 0;
            break;
          }
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <typename A>
__device__ __forceinline__ A warp_sum(A v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;   // in lane 0
}

template <typename T>
struct HhFusedArgs {
  const double *A0;   // the input matrix (row 0 is read from here at step 0)
  T *V;               // [n][n] reflectors, row k = v_k (columns k+1..n-1 written)
  double *d, *e, *tau;
  T *P;               // [2][n] p of the step, by parity
  T *pub;             // [2][n] the next reflector's row, by parity
  double *tail;       // [2] A^(n-3)[n-1][n-2 .. n-1], for the last 2 x 2 block
  GridBar *gb;
  int *flags;
  int n, R;           // R = rows per block
  int64_t ld;         // row stride of A0 and V
};

// One lane-strided pass over row[j0:j1): optional update a -= v_r w + w_r v
// (UPD) and the dot with vc.  Eight loads are issued before their use so that
// rows streamed from L2/HBM keep enough requests in flight.
template <typename T, bool UPD>
__device__ __forceinline__ T row_pass(T *row, int j0, int j1, const T *vp, const T *wv, const T *vc, T vr, T wr) {
  const int lane = threadIdx.x & 31;
  T acc0 = 0, acc1 = 0;
  int j = j0 + lane;
  for (; j + 7 * 32 < j1; j += 8 * 32) {
    T x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = row[j + u * 32];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int q = j + u * 32;
      T a = x[u];
      if (UPD) {
        a = fma(-vr, wv[q], fma(-wr, vp[q], a));
        row[q] = a;
      }
      if (u & 1) acc1 = fma(a, vc[q], acc1); else acc0 = fma(a, vc[q], acc0);
    }
  }
  for (; j < j1; j += 32) {
    T a = row[j];
    if (UPD) {
      a = fma(-vr, wv[j], fma(-wr, vp[j], a));
      row[j] = a;
    }
    acc0 = fma(a, vc[j], acc0);
  }
  return acc0 + acc1;
}

// FP64 instructions are scarce on this part (about 2 per clock per SM), so
// the per-step bookkeeping keeps them off paths that every thread runs: the
// scalars are computed by one thread, and in the FP64 form phase 1 runs on
// HH_P1_FP64 threads only (the FP32 form does all of it in FP32).
constexpr int HH_P1_FP64 = 128;

template <typename T>
__global__ void __launch_bounds__(512, 1) hh_fused_kernel(HhFusedArgs<T> g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *smem = reinterpret_cast<T *>(smem_raw);
  __shared__ T wbuf[2][16];       // per-warp partials: p.v, |x|^2
  __shared__ T s_seg[16], s_a1[16];
  __shared__ T s_st[5];           // x[k], alpha; tau, beta, sc of the step
  const int n = g.n, G = gridDim.x, b = blockIdx.x, R = g.R;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int p1 = (sizeof(T) == 8) ? min(HH_P1_FP64, (int)blockDim.x) : (int)blockDim.x;  // phase-1 team
  const int p1w = p1 >> 5;
  T *wv = smem + 2 * n;
  T *rows = smem + 3 * n;   // [R][n], local row lr is global row lr * G + b
  const int n_own = (b < n) ? min(R, (n - 1 - b) / G + 1) : 0;
  for (int lr = 0; lr < n_own; ++lr) {
    const double *src = g.A0 + (int64_t)(lr * G + b) * g.ld;
    for (int j = threadIdx.x; j < n; j += blockDim.x) rows[(int64_t)lr * n + j] = (T)src[j];
  }
  T *vprev = smem + n, *vcur = smem;
  T tau_prev = 0, sc_prev = 0;
  for (int k = 0; k + 2 < n; ++k) {
    // ---- phase 1.  Team thread t owns element j = k + t + m * p1 of every
    // vector it touches, so the loops below need no barrier between them.
    T *x = vcur;
    T s2 = 0;
    if (k == 0) {
      if (threadIdx.x < p1)
        for (int j = threadIdx.x; j < n; j += p1) {
          const T xj = (T)__ldcg(g.A0 + j);
          x[j] = xj;
          if (j >= 2) s2 = fma(xj, xj, s2);
          if (j < 2) s_st[j] = xj;
        }
    } else {
      const T *Pk = g.P + (size_t)((k - 1) & 1) * n;
      const T *pb = g.pub + (size_t)(k & 1) * n;
      // p of step k-1 and the published row k into wv and x by every thread,
      // its loads issued together: one L2 round trip, where the team's loop
      // below (a global store between its loads) would wait once per element
      for (int j0 = k + threadIdx.x; j0 < n; j0 += 4 * blockDim.x) {
        T pv[4], xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = j0 + u * blockDim.x;
          if (j < n) { pv[u] = __ldcg(Pk + j); xv[u] = __ldcg(pb + j); }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = j0 + u * blockDim.x;
          if (j < n) { wv[j] = pv[u]; x[j] = xv[u]; }
        }
      }
      __syncthreads();
      const T pkk = wv[k];   // read before the team's second loop rewrites wv
      T dsum = 0;
      if (threadIdx.x < p1)
        for (int j = k + threadIdx.x; j < n; j += p1) {
          const T vj = (j == k) ? (T)1 : vprev[j] * sc_prev;   // normalise v_{k-1}
          vprev[j] = vj;
          if (b == 0) g.V[(int64_t)(k - 1) * g.ld + j] = vj;
          dsum = fma(wv[j], vj, dsum);
        }
      if (warp < p1w) {
        dsum = warp_sum(dsum);
        if (lane == 0) wbuf[0][warp] = dsum;
      }
      __syncthreads();
      if (threadIdx.x < p1) {
        T pv = 0;
        for (int q = 0; q < p1w; ++q) pv += wbuf[0][q];
        const T gam = (T)0.5 * tau_prev * pv;
        const T wk = pkk - gam;   // v_{k-1}[k] = 1
        for (int j = k + threadIdx.x; j < n; j += p1) {
          const T wj = wv[j] - gam * vprev[j];
          wv[j] = wj;
          const T xj = x[j] - wj - wk * vprev[j];
          x[j] = xj;
          if (j >= k + 2) s2 = fma(xj, xj, s2);
          if (j < k + 2) s_st[j - k] = xj;
        }
      }
    }
    if (warp < p1w) {
      s2 = warp_sum(s2);
      if (lane == 0) wbuf[1][warp] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {   // the reflector's scalars, once
      T sigma = 0;
      for (int q = 0; q < p1w; ++q) sigma += wbuf[1][q];
      double t, beta, sc;
      reflector_scalars(s_st[1], sigma, &t, &beta, &sc);
      s_st[2] = t; s_st[3] = beta; s_st[4] = sc;
      if (b == 0) {
        g.d[k] = s_st[0];
        g.e[k] = beta;
        g.tau[k] = t;
      }
    }
    __syncthreads();
    const T t = s_st[2], beta = s_st[3], sc = s_st[4], tsc = t * sc;
    // ---- phase 2: own rows r > k: update k-1 (k > 0) fused with s_r
    const int lr0 = (k + 1 > b) ? (k + 1 - b + G - 1) / G : 0;
    const int nact = n_own - lr0;
    // warps per row when rows are few: a row's pass is a chain of about 6 L / wpr
    // clocks, and every warp's sum holds the FP64 pipe for 80
    const int wpr = nact > 0 ? max(1, min(nwarp / nact, (int)(sqrtf(0.075f * (float)(n - k - 1) / (float)nact) + 0.5f))) : 1;
    T *Pk = g.P + (size_t)(k & 1) * n;
    if (nact > 0) {
      const int L = n - k - 1;
      const int seglen = (((L + wpr - 1) / wpr) + 31) & ~31;
      for (int task = warp; task < nact * wpr; task += nwarp) {
        const int lr = lr0 + task / wpr, seg = task % wpr;
        const int r = lr * G + b;
        T *row = rows + (int64_t)lr * n;
        const int j0 = k + 1 + seg * seglen, j1 = min(n, j0 + seglen);
        T acc = 0, a1 = 0;
        if (j0 < j1) {
          if (k == 0) acc = row_pass<T, false>(row, j0, j1, vprev, wv, x, (T)0, (T)0);
          else acc = row_pass<T, true>(row, j0, j1, vprev, wv, x, vprev[r], wv[r]);
        }
        acc = warp_sum(acc);
        if (seg == 0) {   // A^(k)[r][k+1], written by this warp's lane 0
          __syncwarp();
          a1 = row[k + 1];
        }
        if (wpr == 1) {
          if (lane == 0) Pk[r] = tsc * (acc - beta * a1);
        } else if (lane == 0) {
          s_seg[task] = acc;
          if (seg == 0) s_a1[task / wpr] = a1;
        }
      }
    }
    __syncthreads();   // every row update of this step is complete
    if (nact > 0 && wpr > 1 && threadIdx.x < nact) {
      const int r = (lr0 + threadIdx.x) * G + b;
      T a = 0;
      for (int q = 0; q < wpr; ++q) a += s_seg[threadIdx.x * wpr + q];
      Pk[r] = tsc * (a - beta * s_a1[threadIdx.x]);
    }
    // the owner of row k+1 publishes it (A^(k) values, columns k+1..n-1); at the
    // last step the owner of row n-1 also hands over that row's last two entries
    if ((k + 1) % G == b) {
      const int lr = (k + 1) / G;
      const T *rp = rows + (int64_t)lr * n;
      T *pubp = g.pub + (size_t)((k + 1) & 1) * n;
      for (int j = k + 1 + threadIdx.x; j < n; j += blockDim.x) pubp[j] = rp[j];
    }
    if (k == n - 3 && (n - 1) % G == b && threadIdx.x == 0) {
      const T *rp = rows + (int64_t)((n - 1) / G) * n;
      g.tail[0] = rp[n - 2];
      g.tail[1] = rp[n - 1];
    }
    if (!grid_barrier(g.gb, (unsigned)k, g.flags)) return;
    tau_prev = t;
    sc_prev = sc;
    T *tmp = vprev; vprev = vcur; vcur = tmp;
  }
  // ---- the last 2 x 2 block: normalise v_{n-3}, apply update n-3 to rows n-2, n-1
  if (b == 0 && n >= 3 && threadIdx.x == 0) {
    const int kl = n - 3;
    const T *Pk = g.P + (size_t)(kl & 1) * n;
    const T *pb = g.pub + (size_t)((kl + 1) & 1) * n;
    const T v2 = 1, v1 = vprev[n - 1] * sc_prev;
    g.V[(int64_t)kl * g.ld + n - 2] = v2;
    g.V[(int64_t)kl * g.ld + n - 1] = v1;
    const T p2 = __ldcg(Pk + n - 2), p1v = __ldcg(Pk + n - 1);
    const T gam = (T)0.5 * tau_prev * (p2 * v2 + p1v * v1);
    const T w2 = p2 - gam * v2, w1 = p1v - gam * v1;
    const T a22 = __ldcg(pb + n - 2), a21 = __ldcg(pb + n - 1), a11 = (T)__ldcg(g.tail + 1);
    g.d[n - 2] = fma(-v2, w2, fma(-w2, v2, a22));
    g.e[n - 2] = fma(-v2, w1, fma(-w2, v1, a21));
    g.d[n - 1] = fma(-v1, w1, fma(-w1, v1, a11));
    g.e[n - 1] = 0.0;
  }
}

// Number of eigenvalues of T below x (Sturm): the sign changes along the
// leading principal minors p_0 = 1, p_i = det(T_i - x) with
// p_i = (d_{i-1} - x) p_{i-1} - e_{i-2}^2 p_{i-2}.  This is the LDL^T pivot
// count q_i = p_i / p_{i-1} without the division: one FMA per step sits on the
// dependency chain (e^2 p_{i-2} is ready a step early), against a reciprocal
// and its Newton steps in the quotient form.  The pair (p_{i-1}, p_i) is
// rescaled by an exact power of two whenever the larger exponent leaves
// [-400, 400] (integer operations on the high words), and a minor that comes
// out exactly zero is replaced by pivmin with the sign opposite to p_{i-1}
// (counted as a sign change, like the quotient form's pivot -pivmin).  The range check runs every 8 steps, off
// the chain.
__device__ __forceinline__ bool is_zero_bits(double v) {   // +0 or -0, on the integer pipe
  return ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) == 0;
}

__device__ int sturm_count(const double *d, const double *e2, int n, double x, double pivmin) {
  double pm = 1.0, p = d[0] - x;
  if (p == 0.0) p = -pivmin;
  bool neg = __double2hiint(p) < 0;
  int c = neg;
  int i = 1;
  while (i < n) {
    // 8 steps between range checks: |p| grows at most 2 (|d| + |e| + |x|) per
    // step and shrinks by at most e^2 per two, so +-400 stays far from overflow.
    // The block's d_i - x and e^2 are formed first, off the FMA chain.
    double dx[8], ee[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = min(i + u, n - 1);
      dx[u] = d[j] - x;
      ee[u] = e2[j - 1];
    }
    const int m = min(8, n - i);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (u < m) {
        double pn = fma(dx[u], p, -(ee[u] * pm));
        if (is_zero_bits(pn))   // -pivmin with the sign opposite to p, on the integer pipe
          pn = __longlong_as_double((~__double_as_longlong(p) & (long long)0x8000000000000000ull) |
                                    __double_as_longlong(pivmin));
        const bool nn = __double2hiint(pn) < 0;
        c += (nn != neg);
        neg = nn;
        pm = p;
        p = pn;
      }
    }
    i += m;
    const int em = max((__double2hiint(p) >> 20) & 0x7ff, (__double2hiint(pm) >> 20) & 0x7ff);
    if (em > 1023 + 400 || em < 1023 - 400) {
      const double f = __hiloint2double((2046 - em) << 20, 0);   // 2^(1023 - em), exact
      p *= f;
      pm *= f;
    }
  }
  return c;
}

// 1/q from the hardware reciprocal estimate and Newton steps y <- y (2 - q y)
// (each squares the relative error): two give a few ulps, one about 2^-46, at
// a fraction of the latency of the IEEE division on this part.  |q| is kept
// away from zero and subnormals by the caller.
template <int STEPS = 2>
__device__ __forceinline__ double recip_nr(double q) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(q));
#pragma unroll
  for (int s = 0; s < STEPS; ++s) y = y * fma(-q, y, 2.0);
  return y;
}

// ---- blocked Householder reduction (one cooperative launch per panel) ----
// The fused reduction above spends three FP64 multiply-adds per matrix entry
// and step, two of them on the rank-2 updates.  Here a panel of HP_NB steps
// leaves the trailing matrix as it was at the panel's start (A) and keeps the
// reflectors V and their w (W) beside it; each step applies
//   A^(k) = A - sum_t (v_t w_t^T + w_t v_t^T)
// to the one column and the one product that it needs, so the matrix pays one
// multiply-add per entry and step, and the panel's updates reach it together,
// as one product of length 2 HP_NB from digits on the tensor cores.
// Row r belongs to block r mod G.  Step k = k0 + j, two grid barriers:
//   own rows' entries of column k, x_r (known from the step before) -> barrier 1;
//   every block: the whole x into shared memory; the own rows' products
//     S_r = sum_c A[r][c] x_c and their share of T = x^T S; block b < 2 j also the
//     product of x with the one earlier vector v_t (b = 2 t) or w_t (b = 2 t + 1);
//     one warp meanwhile the reflector's scalars                   -> barrier 2;
//   every block: with v = sc (x - beta e_{k+1}): a_t = v_t.v and b_t = w_t.v from those
//     products, v.Av = sc^2 (T - 2 beta S_{k+1} + beta^2 A_{k+1,k+1}),
//     p.v = tau (v.Av - 2 sum a_t b_t); the own rows' p_r = tau (y_r - sum_t (v_t[r] b_t
//     + w_t[r] a_t)), y = sc (S - beta A e_{k+1}), their w_r and their entries of
//     column k + 1 (w_{k+1} from S_{k+1}, which its owner published).
// Own rows' v_t, w_t stay in shared memory.  What crosses blocks goes through
// L2; the barriers are bounded as above.
// On this part an FP64 instruction holds the SM's pipe for 16 clocks whether 1
// or 32 lanes need it, and one warp's FP64 instructions follow each other at
// about 64: so nothing between the barriers waits for the scalars (only the
// unscaled products are published), and the sums over the panel's vectors
// reduce four rows per warp together.
// Bound: the step's chain, two barriers with their L2 round trips (3.5 of
// about 10 us per step at n = 1000), beside one multiply-add per entry on the FP64
// pipe.  Tried and slower: values in self-validating 16-byte packets that their
// readers poll, without barriers (every block polls every packet: 4 to 6 us per
// exchange where a barrier and the loads take 2.5).
constexpr int HP_NB = 64;         // steps per panel: the update's length is 128
constexpr int HP_THREADS = 512;
constexpr int HP_MAX_ROWS = 128;  // rows per block
constexpr int HP_SIGMA_WARPS = 4; // the last warps: sum of squares of x, then (but the last) rows

struct HhPanelArgs {
  const double *A;     // [n][n] the matrix as of step k0
  double *V;           // [n][n] reflectors, row k = v_k
  double *W;           // [HP_NB][n] w of the panel's steps
  double *d, *e, *tau;
  double *xbuf;        // [2][n] column k, by parity
  double *part;        // [2][G] the blocks' shares of T, by parity
  double *dots;        // [2][2 HP_NB] products of x with the earlier vectors, by parity
  double *snext;       // [2][2] S_{k+1}, A[k+1][k+1]
  unsigned long long *wmax;   // bits of the panel's largest |w| (zeroed)
  GridBar *gb;
  unsigned bar0;       // barriers passed before this launch
  int *flags;
  int n, k0, R;
};

__device__ __forceinline__ void grid_arrive(GridBar *gb) { red_add_release(&gb->count, 1u); }

// One thread's bounded wait for barrier number j; false after a time-out anywhere.
__device__ bool grid_wait(GridBar *gb, unsigned j, int *flags) {
  const unsigned target = gridDim.x * (j + 1);
  if (ld_acquire(&gb->count) >= target) return true;
  const uint64_t t0 = gtimer();
  unsigned it = 0;
  while (ld_acquire(&gb->count) < target) {
    if ((++it & 1023) == 0) {
      if (*(volatile int *)&gb->abort) return false;
      if (gtimer() - t0 > 2000000000ull) {
        atomicExch(&flags[FLAG_EIG], 1);
        atomicExch(&gb->abort, 1);
        return false;
      }
    }
  }
  return true;
}

// Named barriers: `sync` waits, `arrive` does not.
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ double warp_sum_all(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// sum over j0 <= j < j1 of row[j] x[j], lane-strided, eight loads in flight.
template <bool L2>
__device__ __forceinline__ double dot_pass(const double *row, int j0, int j1, const double *x) {
  const int lane = threadIdx.x & 31;
  double acc0 = 0.0, acc1 = 0.0;
  int j = j0 + lane;
  for (; j + 7 * 32 < j1; j += 8 * 32) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = L2 ? __ldcg(row + j + u * 32) : row[j + u * 32];
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      acc0 = fma(v[u], x[j + u * 32], acc0);
      acc1 = fma(v[u + 1], x[j + (u + 1) * 32], acc1);
    }
  }
  double v[8];
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (j + u * 32 < j1) v[u] = L2 ? __ldcg(row + j + u * 32) : row[j + u * 32];
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (j + u * 32 < j1) acc0 = fma(v[u], x[j + u * 32], acc0);
  return acc0 + acc1;
}

// Sums over the warp of four values at once: lane l returns the total of
// value l / 8 (two exchanges halve the values held per lane, three more add up
// the eight lanes that hold the same value).
__device__ __forceinline__ double warp_sum4(double a0, double a1, double a2, double a3) {
  const int lane = threadIdx.x & 31;
  const bool hi = lane & 16, h8 = lane & 8;
  double m0 = hi ? a2 : a0, m1 = hi ? a3 : a1;                 // kept: values 0, 1 or 2, 3
  m0 += __shfl_xor_sync(0xffffffffu, hi ? a0 : a2, 16);
  m1 += __shfl_xor_sync(0xffffffffu, hi ? a1 : a3, 16);
  double m = (h8 ? m1 : m0) + __shfl_xor_sync(0xffffffffu, h8 ? m0 : m1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  return m;
}

// sum over t < j of o_i[t] c[t] + o_i[HP_NB + t] c[HP_NB + t] for the rows i0 .. i0 + 3
// of `own` (below n_i), four per warp: lane l returns row i0 + l / 8's.
__device__ __forceinline__ double own_products(const double *own, int i0, int n_i, int j, const double *c) {
  const int lane = threadIdx.x & 31;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int t = lane; t < j; t += 32) {
    const double c0 = c[t], c1 = c[HP_NB + t];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < n_i) {
        const double *o = own + (size_t)(i0 + u) * 2 * HP_NB + t;
        acc[u] = fma(o[0], c0, fma(o[HP_NB], c1, acc[u]));
      }
  }
  return warp_sum4(acc[0], acc[1], acc[2], acc[3]);
}

__global__ void __launch_bounds__(HP_THREADS, 1) hh_panel_kernel(HhPanelArgs g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = g.n, G = gridDim.x, b = blockIdx.x, R = g.R;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = HP_THREADS / 32, LAST = NW - 1;   // the last warp has the scalars
  double *xs = reinterpret_cast<double *>(smem_raw);   // [n] column k
  double *own = xs + n;                                // [R][2 HP_NB]: v_t[r], w_t[r]
  __shared__ double ab[2 * HP_NB], rk[2 * HP_NB];      // b_t, a_t; w_t[k+1], v_t[k+1]
  __shared__ double xo[HP_MAX_ROWS], ty[HP_MAX_ROWS], vo[HP_MAX_ROWS], qo[HP_MAX_ROWS], co[HP_MAX_ROWS];
  __shared__ double seg_acc[HP_MAX_ROWS + NW], row_a1[HP_MAX_ROWS + 1], sig[HP_SIGMA_WARPS];
  __shared__ double s_sc[4], s_vy, s_wk;               // tau, beta, sc, tau^2 / 2; v.Av; tau y_{k+1}
  __shared__ int s_ok;
  const int n_own = b < n ? (n - 1 - b) / G + 1 : 0;
  unsigned bar = g.bar0;
  unsigned long long wmax = 0ull;
  if (warp == 0)
    for (int lr = lane; lr < n_own; lr += 32) {
      const int r = lr * G + b;
      if (r >= g.k0) {
        const double x = g.A[(int64_t)r * n + g.k0];
        xo[lr] = x;
        if (r > g.k0) g.xbuf[r] = x;
        else g.d[r] = x;
      }
    }
  for (int j = 0; j < HP_NB; ++j) {
    const int k = g.k0 + j, par = j & 1;
    const int lr1 = (k + 1 > b) ? (k + 1 - b + G - 1) / G : 0;   // first own row > k
    const int nrow = n_own - lr1;
    const double *xb = g.xbuf + (size_t)par * n;
    double *part = g.part + (size_t)par * G, *dots = g.dots + par * 2 * HP_NB, *snext = g.snext + 2 * par;
    // ---- barrier 1: x and the vectors of the step before are published
    __syncthreads();
    if (tid == 0) { grid_arrive(g.gb); s_ok = grid_wait(g.gb, bar, g.flags); }
    ++bar;
    __syncthreads();
    if (!s_ok) return;
    {
      double t[4], rkv = 0.0;
      // row k + 1 of the earlier vectors
      if (tid < 2 * j) rkv = (tid & 1) ? __ldcg(g.V + (int64_t)(g.k0 + (tid >> 1)) * n + k + 1)
                                       : __ldcg(g.W + (int64_t)(tid >> 1) * n + k + 1);
      for (int c0 = k + 1 + tid; c0 < n; c0 += 4 * HP_THREADS) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u * HP_THREADS < n) t[u] = __ldcg(xb + c0 + u * HP_THREADS);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (c0 + u * HP_THREADS < n) xs[c0 + u * HP_THREADS] = t[u];
      }
      if (tid < 2 * j) rk[(tid & 1) * HP_NB + (tid >> 1)] = rkv;
    }
    __syncthreads();
    // ---- own rows' products with x, and one earlier vector's
    const int ndot = b < 2 * j ? 1 : 0, tot = nrow + ndot;
    const int S = max(1, LAST / tot);   // warps per row when rows are few
    const int seglen = ((n - k - 1 + S - 1) / S + 31) & ~31;
    if (warp >= NW - HP_SIGMA_WARPS) {   // sum of squares of x_{k+2 ..}
      const int w4 = warp - (NW - HP_SIGMA_WARPS);
      double s0 = 0.0;
      for (int c = k + 2 + w4 * 32 + lane; c < n; c += 32 * HP_SIGMA_WARPS) s0 = fma(xs[c], xs[c], s0);
      s0 = warp_sum_all(s0);
      if (lane == 0) sig[w4] = s0;
      if (warp != LAST) bar_arrive(1, 32 * HP_SIGMA_WARPS);
    }
    if (warp != LAST) {
      for (int task = warp; task < tot * S; task += LAST) {
        const int item = task / S, seg = task - item * S;
        const int j0 = k + 1 + seg * seglen, j1 = min(n, j0 + seglen);
        double acc;
        if (item < nrow) {
          const double *row = g.A + (int64_t)((lr1 + item) * G + b) * n;
          acc = dot_pass<false>(row, j0, j1, xs);
          if (seg == 0 && lane == 0) row_a1[item] = row[k + 1];
        } else {
          acc = dot_pass<true>((b & 1) ? g.W + (int64_t)(b >> 1) * n : g.V + (int64_t)(g.k0 + (b >> 1)) * n, j0, j1, xs);
        }
        acc = warp_sum_all(acc);
        if (lane == 0) seg_acc[task] = acc;
      }
      bar_sync(2, 32 * LAST);
      if (warp == 0) {
        double T = 0.0;
        for (int i = lane; i < nrow; i += 32) {
          double S_r = seg_acc[i * S];
          for (int q = 1; q < S; ++q) S_r += seg_acc[i * S + q];
          seg_acc[i * S] = S_r;
          T = fma(xo[lr1 + i], S_r, T);
          if ((lr1 + i) * G + b == k + 1) { snext[0] = S_r; snext[1] = row_a1[i]; }
        }
        T = warp_sum_all(T);
        if (lane == 0) part[b] = T;
        bar_arrive(3, 64);   // the rows' sums are there
        bar_sync(4, 64);     // warp 1's product is written
        if (lane == 0) grid_arrive(g.gb);
      } else if (warp == 1) {
        if (lane == 0 && ndot) {
          double S_t = seg_acc[nrow * S];
          for (int q = 1; q < S; ++q) S_t += seg_acc[nrow * S + q];
          dots[b] = S_t;
        }
        bar_arrive(4, 64);
      }
      // the own rows' column k + 1 without this step's update
      for (int i0 = 4 * (warp - 1); warp > 0 && i0 < nrow; i0 += 4 * (LAST - 1)) {
        const double q = own_products(own, lr1 + i0, lr1 + nrow, j, rk);
        const int i = i0 + (lane >> 3);
        if ((lane & 7) == 0 && i < nrow) qo[lr1 + i] = row_a1[i] - q;
      }
    } else {
      bar_sync(1, 32 * HP_SIGMA_WARPS);
      double tau, beta, sc;
      reflector_scalars(xs[k + 1], (sig[0] + sig[1]) + (sig[2] + sig[3]), &tau, &beta, &sc);
      if (lane == 0) {
        s_sc[0] = tau; s_sc[1] = beta; s_sc[2] = sc; s_sc[3] = 0.5 * tau * tau;
        if (b == 0) { g.e[k] = beta; g.tau[k] = tau; }
      }
      bar_sync(3, 64);
      for (int i = lane; i < nrow; i += 32) {   // the own rows' v and tau y
        const int lr = lr1 + i, r = lr * G + b;
        const double v = r == k + 1 ? 1.0 : sc * xo[lr];
        vo[lr] = v;
        ty[lr] = tau * (sc * fma(-beta, row_a1[i], seg_acc[i * S]));
        g.V[(int64_t)k * n + r] = v;
      }
    }
    __syncthreads();
    const double tau = s_sc[0], beta = s_sc[1], sc = s_sc[2];
    // ---- barrier 2
    if (tid == 0) s_ok = grid_wait(g.gb, bar, g.flags);
    ++bar;
    __syncthreads();
    if (!s_ok) return;
    if (tid < 2 * j) {   // a_t = sc (v_t.x - beta v_t[k+1]), b_t likewise: ab = (b_t | a_t)
      const int odd = tid & 1, t = tid >> 1;
      ab[(odd ^ 1) * HP_NB + t] = sc * fma(-beta, rk[(odd ^ 1) * HP_NB + t], __ldcg(dots + tid));
    }
    if (warp == LAST) {
      double t[5], T = 0.0;
      const double S1 = __ldcg(snext), a11 = __ldcg(snext + 1);
      for (int q0 = lane; q0 < G; q0 += 5 * 32) {
#pragma unroll
        for (int u = 0; u < 5; ++u) t[u] = q0 + u * 32 < G ? __ldcg(part + q0 + u * 32) : 0.0;
#pragma unroll
        for (int u = 0; u < 5; ++u) T += t[u];
      }
      T = warp_sum_all(T);
      if (lane == 0) {
        s_vy = sc * sc * fma(beta, fma(beta, a11, -2.0 * S1), T);
        s_wk = tau * (sc * fma(-beta, a11, S1));
      }
    }
    __syncthreads();
    double abs_ = 0.0, c1 = 0.0;
    if (warp == 0) {   // sum a_t b_t and row k + 1's correction, in warp 0
      for (int t = lane; t < j; t += 32) {
        abs_ = fma(ab[t], ab[HP_NB + t], abs_);
        c1 = fma(rk[HP_NB + t], ab[t], fma(rk[t], ab[HP_NB + t], c1));   // v_t[k+1] b_t + w_t[k+1] a_t
      }
      const double m = warp_sum4(abs_, c1, 0.0, 0.0);
      abs_ = __shfl_sync(0xffffffffu, m, 0);
      c1 = __shfl_sync(0xffffffffu, m, 8);
    } else {
      for (int i0 = 4 * (warp - 1); i0 < nrow; i0 += 4 * (NW - 1)) {
        const double c = own_products(own, lr1 + i0, lr1 + nrow, j, ab);
        if ((lane & 7) == 0 && i0 + (lane >> 3) < nrow) co[lr1 + i0 + (lane >> 3)] = c;
      }
    }
    __syncthreads();
    if (warp == 0) {   // w, and column k + 1 of the own rows
      const double gam = s_sc[3] * fma(-2.0, abs_, s_vy);
      const double wk1 = fma(-tau, c1, s_wk) - gam;
      for (int i = lane; i < nrow; i += 32) {
        const int lr = lr1 + i, r = lr * G + b;
        const double v = vo[lr], w = fma(-gam, v, fma(-tau, co[lr], ty[lr]));
        const double x = fma(-v, wk1, qo[lr]) - w;
        if (r > k + 1) g.xbuf[(size_t)(par ^ 1) * n + r] = x;
        else g.d[r] = x;
        own[(size_t)lr * 2 * HP_NB + j] = v;
        own[(size_t)lr * 2 * HP_NB + HP_NB + j] = w;
        g.W[(int64_t)j * n + r] = w;
        xo[lr] = x;
        wmax = max(wmax, (unsigned long long)__double_as_longlong(w) & 0x7fffffffffffffffull);
      }
    }
  }
  if (warp == 0) {
    for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
    if (lane == 0 && wmax) atomicMax(g.wmax, wmax);
  }
}

// |a| < |b| on the integer pipe (finite doubles: magnitude order = bit order)
__device__ __forceinline__ bool abs_less(double a, double b) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffll) < (__double_as_longlong(b) & 0x7fffffffffffffffll);
}

// scal[1..3] = lower / upper Gershgorin bound, pivmin; scal[4] = ||T|| bound;
// scal[5] = max e^2; count[0] = #eig > thresh, count[1] = #eig within
// 1e-12 ||T|| of it.
__global__ void __launch_bounds__(RB) tridiag_bounds_kernel(const double *dg, const double *e,
                                                            int n, double thresh, double *scal,
                                                            double *e2g, int *count, bool staged) {
  __shared__ double s_lo[RB], s_hi[RB], s_e[RB];
  // the Sturm counts below walk d and e^2 sequentially: staged in shared
  // memory when they fit, so that each step is not an L2 round trip
  extern __shared__ double s_de[];
  double *sd = staged ? s_de : nullptr, *se2 = staged ? s_de + n : e2g;
  const double *d = staged ? sd : dg;
  double *e2 = se2;
  if (staged)
    for (int i = threadIdx.x; i < n; i += blockDim.x) sd[i] = dg[i];
  double lo = DBL_MAX, hi = -DBL_MAX, em = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < n - 1 ? fabs(e[i]) : 0.0);
    lo = fmin(lo, dg[i] - r);
    hi = fmax(hi, dg[i] + r);
    if (i < n - 1) {
      const double ee = e[i] * e[i];
      e2[i] = ee;
      if (staged) e2g[i] = ee;
      em = fmax(em, ee);
    }
  }
  s_lo[threadIdx.x] = lo; s_hi[threadIdx.x] = hi; s_e[threadIdx.x] = em;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      s_lo[threadIdx.x] = fmin(s_lo[threadIdx.x], s_lo[threadIdx.x + s]);
      s_hi[threadIdx.x] = fmax(s_hi[threadIdx.x], s_hi[threadIdx.x + s]);
      s_e[threadIdx.x] = fmax(s_e[threadIdx.x], s_e[threadIdx.x + s]);
    }
    __syncthreads();
  }
  // the three counts (at the threshold and at thresh -/+ tol) run in three warps at once
  __shared__ int s_cnt[3];
  const double pivmin = DBL_MIN * fmax(1.0, s_e[0]);
  const double tn = fmax(fabs(s_lo[0]), fabs(s_hi[0]));  // ||T|| bound
  const double tol = 1e-12 * tn;
  const int w = threadIdx.x >> 5;
  if (w < 3 && (threadIdx.x & 31) == 0) {
    const double x = thresh + (w == 0 ? 0.0 : (w == 1 ? tol : -tol));
    s_cnt[w] = sturm_count(d, e2, n, x, pivmin);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    scal[1] = s_lo[0] - 2.0 * DBL_EPSILON * fabs(s_lo[0]) - 4.0 * pivmin - 1e-300;
    scal[2] = s_hi[0] + 2.0 * DBL_EPSILON * fabs(s_hi[0]) + 4.0 * pivmin + 1e-300;
    scal[3] = pivmin;
    scal[4] = tn;
    scal[5] = s_e[0];
    count[0] = n - s_cnt[0];
    // eigenvalues within tol of the threshold (tie diagnostics)
    count[1] = s_cnt[1] - s_cnt[2];
  }
}

// lam[r] = (n-1-r)-th smallest eigenvalue (r-th largest), r < k, one warp per
// eigenvalue: a sweep counts the eigenvalues below 32 points, one per lane,
// inside a bracket [lo, hi] whose ends the counts have proven, and the bracket
// becomes the interval between two neighbouring points.  What the sweeps cost
// is FP64 instructions: three per row, 16 clocks of the SM's FP64 pipe each and
// about 64 clocks apart within a warp, whatever their dependences.  So few
// sweeps: their points may lie anywhere, and lie where the eigenvalue is likely:
//   - FP32 sweeps first (quotient form, T scaled to norm 1), which cost a tenth;
//     the first FP64 sweep spans their bracket and its error bound;
//   - with the eigenvalue alone in the bracket, p_n = det(T - x) at both ends
//     gives a secant point, and the points close in on it geometrically (the
//     distances to both ends divided by 4, 16, ...);
//   - evenly spaced otherwise, and after any sweep that did less than an even one.
// Measured, bisection to transposition with a quarter of the vectors kept,
// against evenly spaced FP64 sweeps in blocks of four warps: n = 264 1.43 -> 1.11
// ms, n = 800 3.81 -> 2.95, n = 1800 9.7 -> 8.0, n = 3300 22.7 -> 16.8.
// (Ending at eps ||T|| instead of eps |lambda| would save 0.03 to 0.4 ms of these and
// lose the small eigenvalues' last bits.)
constexpr int BS_PRE = 4;                      // FP32 sweeps: 2 / 33^4 of ||T||
constexpr double BS_PRE_ERR = 1.0 / 524288.0;  // 2^-19 ||T||: above the FP32 counts' error

// p_n = det(T - x) as p 2^ex beside the count; t[i] = (d_i, e_{i-1}^2).
__device__ __forceinline__ int sturm_value(const double2 *t, int n, double x, double pivmin, double *pv, int *ex) {
  double pm = 1.0, p = t[0].x - x;
  if (p == 0.0) p = -pivmin;
  bool neg = __double2hiint(p) < 0;
  int c = neg, E = 0;
  for (int i = 1; i < n; i += 8) {
    double dx[8], ee[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double2 v = t[min(i + u, n - 1)];
      dx[u] = v.x - x;
      ee[u] = v.y;
    }
    const int m = n - i;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (u < m) {
        double pn = fma(dx[u], p, -(ee[u] * pm));
        if (is_zero_bits(pn))   // -pivmin with the sign opposite to p
          pn = __longlong_as_double((~__double_as_longlong(p) & (long long)0x8000000000000000ull) |
                                    __double_as_longlong(pivmin));
        const bool nn = __double2hiint(pn) < 0;
        c += (nn != neg);
        neg = nn;
        pm = p;
        p = pn;
      }
    }
    const int em = max((__double2hiint(p) >> 20) & 0x7ff, (__double2hiint(pm) >> 20) & 0x7ff);
    if (em > 1023 + 400 || em < 1023 - 400) {
      const double f = __hiloint2double((2046 - em) << 20, 0);   // 2^(1023 - em), exact
      p *= f;
      pm *= f;
      E += em - 1023;
    }
  }
  *pv = p;
  *ex = E;
  return c;
}

// The FP32 count: pivots q_i = (d_i - x) - e_{i-1}^2 / q_{i-1}, kept away from zero.
__device__ __forceinline__ int sturm_count32(const float2 *t, int n, float x) {
  float q = 1.0f;
  int c = 0;
#pragma unroll 8
  for (int i = 0; i < n; ++i) {
    const float2 v = t[i];   // t[0].y = 0
    q = fmaf(-v.y, __fdividef(1.0f, q), v.x - x);
    if (fabsf(q) < 1e-20f) q = -1e-20f;
    c += q < 0.0f;
  }
  return c;
}

// pre: the block's shared memory also holds T in FP32.
__global__ void bisect_kernel(const double *d, const double *e2g, const double *scal, int n, int k, bool pre,
                              double *lam) {
  extern __shared__ __align__(16) unsigned char bis_raw[];
  double2 *t = reinterpret_cast<double2 *>(bis_raw);
  float2 *tf = reinterpret_cast<float2 *>(t + n);
  const double tn = scal[4], pivmin = scal[3];
  pre = pre && tn > 0.0 && isfinite(tn);
  const double rt = pre ? 1.0 / tn : 0.0;
  pre = pre && isfinite(rt);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double2 v = make_double2(d[i], i > 0 ? e2g[i - 1] : 0.0);
    t[i] = v;
    if (pre) tf[i] = make_float2((float)(v.x * rt), (float)(v.y * rt * rt));
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= k) return;
  const int idx = n - 1 - r;  // ascending index of the wanted eigenvalue
  constexpr unsigned ALL = 0xffffffffu;
  double lo = scal[1], hi = scal[2], hl = lo, hh = hi;
  bool hint = false;
  if (pre) {
    float a = (float)(lo * rt), b = (float)(hi * rt);
    for (int it = 0; it < BS_PRE; ++it) {
      const float x = a + (b - a) * ((float)(lane + 1) * (1.0f / 33.0f));
      const unsigned m = __ballot_sync(ALL, sturm_count32(tf, n, x) > idx);
      const int j = m ? __ffs(m) - 1 : 32;
      const float xl = __shfl_sync(ALL, x, max(j - 1, 0)), xh = __shfl_sync(ALL, x, min(j, 31));
      if (j > 0) a = xl;
      if (j < 32) b = xh;
    }
    hl = fmax(lo, ((double)a - BS_PRE_ERR) * tn);
    hh = fmin(hi, ((double)b + BS_PRE_ERR) * tn);
    hint = hl < hh;
  }
  // p 2^E and the count at the ends (count -1: not known), both from lanes of a sweep
  double pl = 0.0, ph = 0.0;
  int El = 0, Eh = 0, cl = -1, ch = -1;
  bool even = false;   // the next sweep's points are evenly spaced
  int misses = 0;      // placed sweeps that did less: below the counts' resolution none are placed any more
  for (int it = 0; it < 200; ++it) {
    const double w = hi - lo;
    // relative to the eigenvalue: the small ones of a graded T are as well
    // determined by its entries
    if (w <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + pivmin) break;
    double x = lo + w * ((double)(lane + 1) * (1.0 / 33.0));
    bool placed = false;
    if (hint) {
      x = lane == 31 ? hh : hl + (hh - hl) * ((double)lane * (1.0 / 31.0));
      placed = true;
    } else if (!even && misses < 2 && cl >= 0 && ch == cl + 1) {
      const int sh = min(max(Eh - El, -1000), 1000);
      const double q = scalbn(fabs(ph / pl), sh), c = lo + w / (1.0 + q);
      if (c > lo && c < hi) {
        x = lane < 16 ? c - (c - lo) * __hiloint2double((1023 - 2 * (lane + 1)) << 20, 0)
                      : c + (hi - c) * __hiloint2double((1023 - 2 * (32 - lane)) << 20, 0);
        placed = true;
      }
    }
    hint = false;
    double p;
    int E;
    const int c = sturm_value(t, n, x, pivmin, &p, &E);
    const unsigned m = __ballot_sync(ALL, c > idx);   // eigenvalue idx < x
    const int j = m ? __ffs(m) - 1 : 32, jl = max(j - 1, 0), jh = min(j, 31);
    const double xl = __shfl_sync(ALL, x, jl), xh = __shfl_sync(ALL, x, jh);
    const double p0 = __shfl_sync(ALL, p, jl), p1 = __shfl_sync(ALL, p, jh);
    const int E0 = __shfl_sync(ALL, E, jl), E1 = __shfl_sync(ALL, E, jh);
    const int c0 = __shfl_sync(ALL, c, jl), c1 = __shfl_sync(ALL, c, jh);
    bool moved = false;
    if (j > 0 && xl >= lo) {
      moved = xl > lo;
      lo = xl; pl = p0; El = E0; cl = c0;
    }
    if (j < 32 && xh <= hi) {
      moved = moved || xh < hi;
      hi = xh; ph = p1; Eh = E1; ch = c1;
    }
    if (!placed && !moved) break;   // no progress at this resolution
    even = placed && !(hi - lo <= w * (1.0 / 32.0));
    misses += even;
  }
  if (lane == 0) lam[r] = 0.5 * (lo + hi);
}

// Inverse iteration for those eigenvectors of T that the twisted
// factorisations below leave (need; null: all), one thread per group of
// consecutive eigenvalues closer than gtol (groups are orthogonalised
// internally).  X[i*k + r] receives the vector of lam[r].
//
// The LU factorisation of T - lambda (row interchanges) runs with its
// recurrence carried in registers, so it only reads T and writes the factors:
// multipliers, reciprocals of U's diagonal, U's two super-diagonals and the
// interchange flags.  SMEM: those five arrays and the working vector live in
// shared memory, interleaved by thread (TPB threads per block); otherwise in
// the global scratch lu (strided by k) and X.  The start vector comes from an
// integer hash of (i, r).
constexpr int IV_DL = 0, IV_RDD = 1, IV_DU = 2, IV_DU2 = 3, IV_PV = 4, IV_X = 5;

__device__ __forceinline__ unsigned mix32(unsigned x) {
  x ^= x >> 16; x *= 0x7feb352du;
  x ^= x >> 15; x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

template <typename T>
__device__ __forceinline__ T iv_start(int i, int r) {
  return (T)0.5 + (T)(mix32((unsigned)i * 0x9e3779b9u ^ mix32((unsigned)r + 0x632be5abu)) >> 8) * (T)(1.0 / 16777216.0);
}

template <typename T, bool SMEM>
__global__ void inverse_iteration_kernel(const double *dg, const double *eg, const double *lam,
                                         const double *scal, int n, int k, T *X, T *lu, const int *need,
                                         int *flags) {
  extern __shared__ __align__(16) unsigned char sde_raw[];
  // need: the vectors that are left to this kernel (null: all of them)
  {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (!__syncthreads_or(r < k && (need == nullptr || need[r]))) return;
  }
  T *d = reinterpret_cast<T *>(sde_raw), *e = d + n;
  T *ws = e + n;                                   // SMEM: [6][n][blockDim.x]
  for (int i = threadIdx.x; i < n; i += blockDim.x) { d[i] = (T)dg[i]; e[i] = (i < n - 1) ? (T)eg[i] : (T)0; }
  __syncthreads();
  const int tl = threadIdx.x, tpb = blockDim.x;
  const int r0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (r0 >= k) return;
  const double tnorm = scal[4];
  const double gtol = Lim<T>::group_tol * tnorm;
  if (r0 > 0 && lam[r0 - 1] - lam[r0] <= gtol) return;  // not the first of its group
  int r1 = r0 + 1;
  while (r1 < k && lam[r1 - 1] - lam[r1] <= gtol) ++r1;
  if (need && !need[r0]) return;   // members of a group all have it set
  const T tiny = Lim<T>::eps() * fmax((T)tnorm, Lim<T>::tiny());
  // pivots below tiny in magnitude (zero included) become +-tiny; integer compare
  const long long tiny_bits = __double_as_longlong(tiny);
  auto fix = [&](T x) -> T {
    const long long xb = __double_as_longlong(x);
    return ((xb & 0x7fffffffffffffffll) < tiny_bits) ? __longlong_as_double((xb & (long long)0x8000000000000000ull) | tiny_bits)
                                                   : x;
  };
  double prev = 0.0;
  for (int r = r0; r < r1; ++r) {
    // element i of array a of this thread's vector
#define S(a, i) (SMEM ? ws[((int64_t)(a) * n + (i)) * tpb + tl] : lu[((int64_t)(a) * n + (i)) * k + r])
#define XV(i) (SMEM ? ws[((int64_t)IV_X * n + (i)) * tpb + tl] : X[(int64_t)(i) * k + r])
    double lmd = lam[r];
    if (r > r0) {
      double pert = 10.0 * (double)Lim<T>::eps() * fmax(fabs(lmd), tnorm * 1e-3);
      if (prev - lmd < pert) lmd = prev - pert;
    }
    prev = lmd;
    const T lm = (T)lmd;
    // LU of T - lm with row interchanges; a, b = current diagonal and super-diagonal.
    // One reciprocal per step (of the pivot); U's super-diagonals are stored
    // pre-scaled by it, so the backward sweep has one FMA on its chain.
    {
      // chain per step: pivot choice (integer compare), reciprocal, one FMA;
      // the block's d - lm, c b and a dn are formed beside it
      T a = d[0] - lm, b = e[0];
      for (int i0 = 0; i0 < n - 1; i0 += 8) {
        T dn8[8], c8[8], bn8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = min(i0 + u, n - 2);
          dn8[u] = d[i + 1] - lm;
          c8[u] = e[i];
          bn8[u] = e[i + 1];   // e[n-1] = 0
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = i0 + u;
          if (i < n - 1) {
            const T c = c8[u], dn = dn8[u], bn = bn8[u];
            const T cb = c * b, adn = a * dn;
            const bool sw = abs_less(a, c);
            const T piv = fix(sw ? c : a);
            const T rp = recip_nr<1>(piv);   // 2^-46: ample for an iteration that refines itself
            const T f = (sw ? a : c) * rp;
            S(IV_DL, i) = f;
            S(IV_RDD, i) = rp;
            S(IV_DU, i) = (sw ? dn : b) * rp;
            S(IV_DU2, i) = sw ? bn * rp : (T)0;
            S(IV_PV, i) = sw ? (T)1 : (T)0;
            const T an = sw ? fma(-adn, rp, b) : fma(-cb, rp, dn);
            b = sw ? -f * bn : bn;
            a = an;
          }
        }
      }
      S(IV_RDD, n - 1) = recip_nr<1>(fix(a));
      S(IV_DU, n - 1) = 0;
      S(IV_DU2, n - 1) = 0;
    }
    for (int iter = 0; iter < 2; ++iter) {
      // forward: apply L^-1 with the interchanges (the start vector on the first
      // pass).  Eight steps' factors and entries are loaded before the chain.
      T xc = (iter == 0) ? iv_start<T>(0, r) : XV(0);
      for (int i0 = 0; i0 < n - 1; i0 += 8) {
        T f8[8], p8[8], x8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = min(i0 + u, n - 2);
          f8[u] = S(IV_DL, i);
          p8[u] = S(IV_PV, i);
          x8[u] = (iter == 0) ? iv_start<T>(i + 1, r) : XV(i + 1);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = i0 + u;
          if (i < n - 1) {
            T xn = x8[u], out;
            if (p8[u] == (T)0) { out = xc; xn = xn - f8[u] * xc; }
            else { out = xn; xn = xc - f8[u] * xn; }
            XV(i) = out;
            xc = xn;
          }
        }
      }
      XV(n - 1) = xc;
      // backward: U^-1 (rows scaled by 1 / pivot), eight steps' data loaded first
      T x1 = 0, x2 = 0;
      for (int i0 = n - 1; i0 >= 0; i0 -= 8) {
        T du8[8], dv8[8], rd8[8], xv8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = max(i0 - u, 0);
          du8[u] = S(IV_DU, i);
          dv8[u] = S(IV_DU2, i);
          rd8[u] = S(IV_RDD, i);
          xv8[u] = XV(i);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = i0 - u;
          if (i >= 0) {
            const T sv = fma(-du8[u], x1, fma(-dv8[u], x2, xv8[u] * rd8[u]));
            XV(i) = sv;
            x2 = x1;
            x1 = sv;
          }
        }
      }
      // orthogonalise against the earlier vectors of this group (already in X)
      for (int q = r0; q < r; ++q) {
        double dot = 0.0;
        for (int i = 0; i < n; ++i) dot += (double)X[(int64_t)i * k + q] * (double)XV(i);
        const T dt = (T)dot;
        for (int i = 0; i < n; ++i) XV(i) -= dt * X[(int64_t)i * k + q];
      }
      T s0 = 0, s1 = 0, s2 = 0, s3 = 0;   // four chains: FP64 FMA latency is long here
      int i = 0;
      for (; i + 3 < n; i += 4) {
        s0 = fma(XV(i), XV(i), s0); s1 = fma(XV(i + 1), XV(i + 1), s1);
        s2 = fma(XV(i + 2), XV(i + 2), s2); s3 = fma(XV(i + 3), XV(i + 3), s3);
      }
      for (; i < n; ++i) s0 = fma(XV(i), XV(i), s0);
      const double nrm = sqrt((double)((s0 + s1) + (s2 + s3)));
      if (!(nrm > 0.0) || !isfinite(nrm)) { atomicExch(&flags[FLAG_EIG], 1); break; }
      const T inv = (T)(1.0 / nrm);
      if (SMEM && iter == 1) {
        for (int i = 0; i < n; ++i) X[(int64_t)i * k + r] = XV(i) * inv;
      } else {
        for (int i = 0; i < n; ++i) XV(i) *= inv;
      }
    }
#undef S
#undef XV
  }
}

// ---- eigenvectors from twisted factorisations ----
// T - lam = (top-down pivots D+) = (bottom-up pivots D-); with the row r where
// gamma_r = D+_r + D-_r - (d_r - lam) is smallest in magnitude, the two
// factorisations joined at r give (T - lam) z = gamma_r e_r with z_r = 1,
//   z_i = -(e_i / D+_i) z_{i+1} above r,  z_i = -(e_{i-1} / D-_i) z_{i-1} below
// (Fernando's double factorisation; Parlett and Dhillon, Linear Algebra Appl.
// 267 (1997) 247).  Bound by the FP64 chains: five instructions per row for the
// pivots and two for z, about 64 clocks each, against about 22 for LU with
// interchanges and two solves; the two directions run in two warps at once.
// One lane per vector there, V vectors per block so that the blocks make one
// wave; gamma, the residual and the norm use the whole block.
// The residual is formed from the entries of T: a vector whose residual is above
// TW_TOL ||T||, or whose eigenvalue is closer than the group tolerance to another,
// goes to inverse iteration (need[r] = 1).  SM: pivots and z in shared memory.
// Measured, n = 3300 with 883 vectors: 1.6 ms (1.06 M clocks of it the pivots' chain)
// against 7.2 for inverse iteration; bisection to transposition n = 264 1.11 ->
// 0.89 ms, n = 800 2.95 -> 2.18, n = 1800 8.0 -> 5.1, n = 3300 16.8 -> 11.2.  The
// vectors are closer to those of an FP64 eigensolver as well: 1e-13 instead of
// 2e-11 (relative 2-norm over all kept) at n = 3300.
constexpr double TW_TOL = 8.0 * DBL_EPSILON;
constexpr int TW_THREADS = 256;

template <bool SM>
__global__ void __launch_bounds__(TW_THREADS) twisted_kernel(const double *dg, const double *eg, const double *lam,
                                                             const double *scal, int n, int k, int V, double *X,
                                                             double *lu, int *need) {
  extern __shared__ __align__(16) unsigned char tw_raw[];
  double *d = reinterpret_cast<double *>(tw_raw), *e = d + n, *e2 = e + n;   // e[i], e2[i] couple rows i and i + 1
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = blockIdx.x * V, nv = min(V, k - r0);
  // pivots' reciprocals [n][ld]; z replaces those of D+
  const int64_t ld = SM ? V : k;
  double *F = SM ? e2 + n : lu + r0, *Bk = SM ? F + (int64_t)n * V : lu + (int64_t)n * k + r0;
  __shared__ double s_a[TW_THREADS], s_b[TW_THREADS];
  __shared__ int s_i[TW_THREADS];
  for (int i = tid; i < n; i += TW_THREADS) {
    const double ei = i < n - 1 ? eg[i] : 0.0;
    d[i] = dg[i];
    e[i] = ei;
    e2[i] = ei * ei;
  }
  __syncthreads();
  const double tn = scal[4];
  const long long tiny_bits = __double_as_longlong(fmax(DBL_EPSILON * DBL_EPSILON * tn, 1e-290));
  auto fix = [&](double x) -> double {
    const long long xb = __double_as_longlong(x);
    return ((xb & 0x7fffffffffffffffll) < tiny_bits)
               ? __longlong_as_double((xb & (long long)0x8000000000000000ull) | tiny_bits) : x;
  };
  if (warp < 2 && lane < nv) {
    const double lm = lam[r0 + lane];
    double rp = 0.0;
    for (int i0 = 0; i0 < n; i0 += 8) {
      double dx[8], ee[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = min(i0 + u, n - 1), i = warp == 0 ? t : n - 1 - t;
        dx[u] = d[i] - lm;
        ee[u] = warp == 0 ? (i > 0 ? e2[i - 1] : 0.0) : e2[i];
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = i0 + u;
        if (t < n) {
          rp = recip_cubic(fix(fma(-ee[u], rp, dx[u])));
          if (warp == 0) F[t * ld + lane] = rp;
          else Bk[(n - 1 - t) * ld + lane] = rp;
        }
      }
    }
  }
  __syncthreads();
  // the twist row of each vector (the first of equal ones)
  const int v = tid & (V - 1), g = tid / V, ng = TW_THREADS / V;
  const double lmv = v < nv ? lam[r0 + v] : 0.0;
  {
    double best = DBL_MAX;
    int bi = 0;
    if (v < nv)
#pragma unroll 4
      for (int i = g; i < n; i += ng) {
        double x = d[i] - lmv;
        if (i > 0) x = fma(-e2[i - 1], F[(i - 1) * ld + v], x);
        if (i + 1 < n) x = fma(-e2[i], Bk[(i + 1) * ld + v], x);
        if (fabs(x) < best) { best = fabs(x); bi = i; }
      }
    s_a[tid] = best;
    s_i[tid] = bi;
    __syncthreads();
    for (int o = TW_THREADS / 2; o >= V; o >>= 1) {
      if (tid < o && (s_a[tid + o] < s_a[tid] || (s_a[tid + o] == s_a[tid] && s_i[tid + o] < s_i[tid]))) {
        s_a[tid] = s_a[tid + o];
        s_i[tid] = s_i[tid + o];
      }
      __syncthreads();
    }
  }
  if (warp < 2 && lane < nv) {
    // outwards from r; eight rows' factors are loaded a block ahead
    const int r = s_i[lane];
    const double *src = warp == 0 ? F : Bk;
    const int len = warp == 0 ? r : n - 1 - r;
    double z = 1.0, a[8], b[8];
    auto row = [&](int t) { return warp == 0 ? r - 1 - t : r + 1 + t; };
    auto load = [&](int t0) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = t0 + u;
        if (t < len) {
          const int i = row(t);
          b[u] = -(warp == 0 ? e[i] : e[i - 1]) * src[i * ld + lane];
        }
      }
    };
    load(0);
    for (int t0 = 0; t0 < len; t0 += 8) {
#pragma unroll
      for (int u = 0; u < 8; ++u) a[u] = b[u];
      load(t0 + 8);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = t0 + u;
        if (t < len) {
          z *= a[u];
          F[row(t) * ld + lane] = z;
        }
      }
    }
  }
  __syncthreads();
  if (tid < nv) F[s_i[tid] * ld + tid] = 1.0;
  __syncthreads();
  double zz = 0.0, rr = 0.0;
  if (v < nv)
#pragma unroll 4
    for (int i = g; i < n; i += ng) {
      const double z = F[i * ld + v];
      double x = (d[i] - lmv) * z;
      if (i > 0) x = fma(e[i - 1], F[(i - 1) * ld + v], x);
      if (i + 1 < n) x = fma(e[i], F[(i + 1) * ld + v], x);
      zz = fma(z, z, zz);
      rr = fma(x, x, rr);
    }
  s_a[tid] = zz;
  s_b[tid] = rr;
  __syncthreads();
  for (int o = TW_THREADS / 2; o >= V; o >>= 1) {
    if (tid < o) {
      s_a[tid] += s_a[tid + o];
      s_b[tid] += s_b[tid + o];
    }
    __syncthreads();
  }
  if (v >= nv) return;
  const double nrm = sqrt(s_a[v]), inv = 1.0 / nrm;
  if (g == 0) {
    const int r = r0 + v;
    const double gtol = Lim<double>::group_tol * tn;
    const bool good = nrm >= 1.0 && isfinite(nrm) && sqrt(s_b[v]) <= TW_TOL * tn * nrm;
    need[r] = !good || (r > 0 && lam[r - 1] - lmv <= gtol) || (r + 1 < k && lmv - lam[r + 1] <= gtol);
  }
  for (int i = g; i < n; i += ng) X[(int64_t)i * k + r0 + v] = F[i * ld + v] * inv;
}

// F = (3 I - G) / 2 for a k x k Gram matrix G (in place).
template <typename T>
__global__ void lowdin_factor_kernel(T *G, int k) {
  int64_t kk = (int64_t)k * k;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < kk;
       e += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(e / k), j = (int)(e - (int64_t)i * k);
    G[e] = (T)(((i == j) ? 1.5 : 0.0) - 0.5 * (double)G[e]);
  }
}

// ---- compact-WY back-transformation: U = H_0 H_1 ... H_{n-3} X ----
// For a block of nb consecutive reflectors j0..j0+nb-1 (rows of V, zero
// outside j+1..n-1), H_j0 ... H_{j0+nb-1} = 1 - V_b T V_b^T with T upper
// triangular (T_ii = tau_i, T[0:l, l] = -tau_l T[0:l, 0:l] G[0:l, l],
// G = V_b^T V_b).  Blocks are applied from the last to the first:
// Y <- Y - V_b (T (V_b^T Y)).
constexpr int WY_NB = 64;
constexpr int64_t WY_KSPLIT = 64;

// dst[i] = sum_s src[s * stride + i]
template <typename T>
__global__ void sum_partials_kernel(const T *__restrict__ src, int nsplit, int64_t stride,
                                    int64_t n, T *__restrict__ dst) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    T a = 0;
    for (int q = 0; q < nsplit; ++q) a += src[q * stride + i];
    dst[i] = a;
  }
}

// T (row-major, upper, zero-padded to WY_NB x WY_NB) of reflector block b (one
// CTA each) from G_b = V_b^T V_b (Gg + b*WY_NB^2, ld nb) and tau[j0..j0+nb),
// j0 = b*WY_NB.
// Column l: T[0:l, l] = -tau_l T[0:l, 0:l] G[0:l, l]; four threads share
// each row's sum (shorter FMA chains).
template <typename T>
__global__ void wy_build_t_kernel(const T *__restrict__ Gall, const double *__restrict__ tau, int nref,
                                  T *__restrict__ Tall) {
  // dynamic: [2][WY_NB][WY_NB + 1] (over the static limit in FP64)
  extern __shared__ __align__(16) unsigned char wy_raw[];
  T (*sT)[WY_NB + 1] = reinterpret_cast<T (*)[WY_NB + 1]>(wy_raw);
  T (*Gt)[WY_NB + 1] = sT + WY_NB;   // G transposed: column l of G is read along a row
  const int j0 = blockIdx.x * WY_NB, nb = min(WY_NB, nref - j0);
  const T *Gg = Gall + (int64_t)blockIdx.x * WY_NB * WY_NB;
  T *Tm = Tall + (int64_t)blockIdx.x * WY_NB * WY_NB;
  for (int q = threadIdx.x; q < WY_NB * WY_NB; q += blockDim.x) {
    sT[q / WY_NB][q % WY_NB] = 0;
    if (q < nb * nb) Gt[q % nb][q / nb] = Gg[q];
  }
  __syncthreads();
  if (threadIdx.x < nb) sT[threadIdx.x][threadIdx.x] = (T)tau[j0 + threadIdx.x];
  __syncthreads();
  const int i = threadIdx.x >> 2, part = threadIdx.x & 3;   // blockDim = 4 * WY_NB
  for (int l = 1; l < nb; ++l) {
    T v = 0;
    if (i < l)
      for (int m = i + part; m < l; m += 4) v = fma(sT[i][m], Gt[l][m], v);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    __syncthreads();
    if (i < l && part == 0) sT[i][l] = -(T)tau[j0 + l] * v;
    __syncthreads();
  }
  for (int q = threadIdx.x; q < WY_NB * WY_NB; q += blockDim.x) Tm[q] = sT[q / WY_NB][q % WY_NB];   // zero-padded
}

// ---- the compact-WY blocks applied by one cooperative kernel ----
// Launched as G CTAs for each of the S column slices (columns 64 s .. 64 s +
// 63 of Y).  CTA (s, c) owns the row chunks ch = c, c + G, c + 2G, ... of
// WA_RC rows.  For each block b, last to first (rows r0 = 64 b + 1 .. n-1):
//   1. the partial of W1 = V_b Y[r0:, slice] over the own chunks -> Wp[s][c];
//   2. grid barrier; CTA c sums entries c*256 + t (+ G*256 ...) of the
//      slice's partials                                            -> W1[s];
//   3. grid barrier; Y[own rows, slice] -= M_b[own rows] W1[s].
// A CTA reads and writes only its own rows of Y, so step 3 of one block and
// step 1 of the next need no barrier between them.  Each step does
// WA_RC x 64 x 64 FMAs per chunk (64 rows of V_b by the slice, or the chunk's
// rows by 64 columns), so the FP64 work spreads over every SM in units a
// quarter of a 64 x 64 x 64 tile.
constexpr int WA_RC = 32;
constexpr size_t WA_SMEM = (size_t)(64 * (WA_RC + 1) + 64 * 64) * sizeof(double);   // step 3 (the larger)

struct WyApplyArgs {
  const double *V;   // [n + 64][n] reflectors (rows)
  const double *M;   // [nblk][n - 1][64]: M_b[r - 1][i] = (V_b^T T_b)[r][i]
  double *Y;         // [n][k], updated in place
  double *Wp;        // [S * G][64 * 64] partials of W1
  double *W1;        // [S][64 * 64]
  GridBar *gb;
  int *flags;
  int n, k, nref, nblk, G;
};

__global__ void __launch_bounds__(256) wy_apply_kernel(WyApplyArgs g) {
  extern __shared__ __align__(16) double wa_sm[];
  const int s = blockIdx.x / g.G, c = blockIdx.x % g.G;
  const int n = g.n, k = g.k, col0 = 64 * s, ncol = min(64, k - col0);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double *W1s = g.W1 + (int64_t)s * 4096;
  unsigned bar = 0;
  for (int b = g.nblk - 1; b >= 0; --b) {
    const int j0 = 64 * b, nb = min(64, g.nref - j0), r0 = j0 + 1;
    // ---- 1: Vs[r][i] = V_b[i][a + r] (transposed), Ys[r][cc] = Y[a + r][col0 + cc]
    double *Vs = wa_sm, *Ys = wa_sm + WA_RC * 65;
    double acc[4][4] = {};
    for (int ch = c; ch * WA_RC < n; ch += g.G) {
      const int a = max(ch * WA_RC, r0), e = min(n, ch * WA_RC + WA_RC);
      if (a >= e) continue;   // the same for the whole CTA
      const int len = e - a;
      for (int q = tid; q < 64 * WA_RC; q += 256) {
        const int i = q / WA_RC, r = q % WA_RC;
        Vs[r * 65 + i] = (i < nb && r < len) ? g.V[(int64_t)(j0 + i) * n + a + r] : 0.0;
        const int r2 = q >> 6, cc = q & 63;
        Ys[r2 * 64 + cc] = (r2 < len && cc < ncol) ? g.Y[(int64_t)(a + r2) * k + col0 + cc] : 0.0;
      }
      __syncthreads();
      for (int r = 0; r < len; ++r) {
        double av[4], bv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) av[u] = Vs[r * 65 + ty + 16 * u];
#pragma unroll
        for (int v = 0; v < 4; ++v) bv[v] = Ys[r * 64 + tx + 16 * v];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
      }
      __syncthreads();
    }
    double *Wpc = g.Wp + (int64_t)blockIdx.x * 4096;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) Wpc[(ty + 16 * u) * 64 + tx + 16 * v] = acc[u][v];
    if (!grid_barrier(g.gb, bar++, g.flags)) return;
    // ---- 2: the slice's partials summed, 256 entries per CTA at a time
    const double *Wps = g.Wp + (int64_t)s * g.G * 4096;
    for (int q = c * 256 + tid; q < 4096; q += g.G * 256) {
      double t = 0.0;
      for (int m = 0; m < g.G; ++m) t += __ldcg(Wps + (int64_t)m * 4096 + q);
      W1s[q] = t;
    }
    if (!grid_barrier(g.gb, bar++, g.flags)) return;
    // ---- 3: Ms[i][r] = M_b[a + r - 1][i] (transposed), Ws = W1[s]
    double *Ms = wa_sm, *Ws = wa_sm + 64 * (WA_RC + 1);
    for (int q = tid; q < 4096; q += 256) Ws[q] = __ldcg(W1s + q);
    __syncthreads();
    for (int ch = c; ch * WA_RC < n; ch += g.G) {
      const int a = max(ch * WA_RC, r0), e = min(n, ch * WA_RC + WA_RC);
      if (a >= e) continue;
      const int len = e - a;
      for (int q = tid; q < WA_RC * 64; q += 256) {
        const int r = q >> 6, i = q & 63;
        Ms[i * (WA_RC + 1) + r] = (r < len && i < nb) ? g.M[((int64_t)b * (n - 1) + (a + r - 1)) * 64 + i] : 0.0;
      }
      __syncthreads();
      double upd[2][4] = {};
      for (int i = 0; i < nb; ++i) {
        double av[2], bv[4];
#pragma unroll
        for (int u = 0; u < 2; ++u) av[u] = Ms[i * (WA_RC + 1) + ty + 16 * u];
#pragma unroll
        for (int v = 0; v < 4; ++v) bv[v] = Ws[i * 64 + tx + 16 * v];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) upd[u][v] = fma(av[u], bv[v], upd[u][v]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int r = ty + 16 * u;
        if (r >= len) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int cc = tx + 16 * v;
          if (cc < ncol) g.Y[(int64_t)(a + r) * k + col0 + cc] -= upd[u][v];
        }
      }
      __syncthreads();
    }
  }
}

// Ut[c][r] = X[r][c]
template <typename T>
__global__ void transpose_kernel(const T *__restrict__ X, int n, int k, double *__restrict__ Ut) {
  __shared__ T tile[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    int r = r0 + q, c = c0 + threadIdx.x;
    if (r < n && c < k) tile[q][threadIdx.x] = X[(int64_t)r * k + c];
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    int c = c0 + q, r = r0 + threadIdx.x;
    if (r < n && c < k) Ut[(int64_t)c * n + r] = tile[threadIdx.x][q];
  }
}

// Raise a kernel's dynamic shared-memory limit once per device, to the most any
// call may use; setting it per call races between host threads (one thread could
// lower it between another thread's set and launch).
cudaError_t allow_max_dynamic_smem(const void *kernel, OncePerDevice &once) {
  return once([&] {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  });
}
OncePerDevice g_smem_hh, g_smem_hp, g_smem_bisect, g_smem_invit[2], g_smem_tw[2], g_smem_bounds, g_smem_wy, g_smem_wa;

// Try the fused reduction of the trailing block from row and column k0 on in
// arithmetic T; false when it cannot be launched.
template <typename T>
bool launch_fused(EigWork &w, int n_all, int k0, cudaStream_t s, int *launches, cudaError_t *err) {
  const int n = n_all - k0;
  int dev = 0, nsm = 0, coop = 0, optin = 0;
  *err = cudaSuccess;
  bool ok = n > 2 && w.grid_ws != nullptr && cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess;
  cudaGetLastError();
  if (!ok) return false;
  const int G = std::min(nsm, std::max(1, (n + HH_MIN_ROWS - 1) / HH_MIN_ROWS));
  const int R = (n + G - 1) / G;
  const size_t reserve = 1024;   // static shared memory of the kernel
  const size_t smem = (size_t)(3 + R) * n * sizeof(T);
  if (smem + reserve > (size_t)optin) return false;
  const void *kern = (const void *)hh_fused_kernel<T>;
  int per_sm = 0;
  ok = allow_max_dynamic_smem(kern, g_smem_hh) == cudaSuccess &&
       cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 512, smem) == cudaSuccess && per_sm >= 1;
  cudaGetLastError();
  if (!ok) return false;
  HhFusedArgs<T> g;
  const int64_t off = (int64_t)k0 * n_all + k0;
  g.A0 = w.A + off;
  g.V = reinterpret_cast<T *>(w.V) + off;
  g.d = w.d + k0; g.e = w.e + k0; g.tau = w.tau + k0;
  g.ld = n_all;
  g.P = reinterpret_cast<T *>(w.grid_ws);
  g.pub = g.P + 2 * (size_t)n;
  double *after = w.grid_ws + (4 * (size_t)n_all * sizeof(T) + sizeof(double) - 1) / sizeof(double);
  g.tail = after;
  g.gb = reinterpret_cast<GridBar *>(after + 2);
  g.flags = w.flags;
  g.n = n; g.R = R;
  *err = cudaMemsetAsync(g.gb, 0, sizeof(GridBar), s);
  if (*err != cudaSuccess) return true;
  void *args[] = {&g};
  *err = cudaLaunchCooperativeKernel(kern, dim3(G), dim3(512), args, smem, s);
  if (*err == cudaSuccess) *launches += 1;
  return true;
}

// Panels of the blocked reduction from the front, as long as they pay; *k0 is
// the first column left to the fused kernel (0: none, or not available here).
// The panel's arrays and digits live in the inverse-iteration scratch.
// Sizes: measured at n = 900 both take 8.0 ms, n = 1100 10.3 against 10.8, n = 1800
// 20.0 against 25.4, n = 3300 58.7 against 107 ms; leaving the last 800 columns to
// the fused kernel is 0.1 to 0.5 ms better than 500, 0.6 better than 1100 (all
// before the fused kernel's scalars were shortened: 0.7 ms off its 6.7 at n = 800).
constexpr int HP_MIN_N = 1000, HP_TAIL = 800;

cudaError_t launch_blocked(EigWork &w, int n, cudaStream_t s, int *launches, int *k0_out) {
  *k0_out = 0;
  int dev = 0, nsm = 0, coop = 0, optin = 0, per_sm = 0;
  bool ok = n >= HP_MIN_N && w.grid_ws != nullptr && w.flags != nullptr && cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess;
  cudaGetLastError();
  if (!ok) return cudaSuccess;
  const int G = nsm, R = (n + G - 1) / G;
  const size_t smem = ((size_t)n + (size_t)R * 2 * HP_NB) * sizeof(double);
  ok = G >= 2 * HP_NB && R <= HP_MAX_ROWS && smem + 12 * 1024 <= (size_t)optin &&
       allow_max_dynamic_smem((const void *)hh_panel_kernel, g_smem_hp) == cudaSuccess &&
       cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)hh_panel_kernel, HP_THREADS, smem) ==
           cudaSuccess && per_sm >= 1;
  cudaGetLastError();
  if (!ok) return cudaSuccess;
  // scratch: 5 n^2 doubles, of which this takes about (64 + 448) n + small
  char *base = reinterpret_cast<char *>(w.lu);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    void *p = base + off;
    off += (bytes + 255) / 256 * 256;
    return p;
  };
  const int n_panels_max = n / HP_NB + 1, nkb = 2 * HP_NB / SL_K, np = (int)slice_rows_padded(n);
  HhPanelArgs a;
  a.W = (double *)take((size_t)HP_NB * n * sizeof(double));
  a.xbuf = (double *)take((size_t)2 * n * sizeof(double));
  a.part = (double *)take((size_t)2 * G * sizeof(double));
  a.dots = (double *)take((size_t)4 * HP_NB * sizeof(double));
  a.snext = (double *)take(4 * sizeof(double));
  const size_t zero0 = off;
  a.gb = (GridBar *)take(sizeof(GridBar));
  unsigned long long *wmax = (unsigned long long *)take((size_t)n_panels_max * sizeof(unsigned long long));
  const size_t zero1 = off;
  SlicePairSrc ps;
  const int64_t dig = slice_digit_bytes(n, nkb, 7);
  ps.dig_p = (uint8_t *)take(dig);
  ps.dig_q = (uint8_t *)take(dig);
  ps.exp_p = (int *)take((size_t)np * sizeof(int));
  ps.exp_q = (int *)take((size_t)np * sizeof(int));
  if (off > (size_t)5 * n * n * sizeof(double)) return cudaSuccess;
  a.A = w.A; a.V = w.V; a.d = w.d; a.e = w.e; a.tau = w.tau;
  a.flags = w.flags; a.n = n; a.R = R; a.bar0 = 0;
  cudaError_t e = cudaMemsetAsync(base + zero0, 0, zero1 - zero0, s);
  if (e != cudaSuccess) return e;
  int k0 = 0;
  for (int q = 0; n - k0 >= HP_TAIL + HP_NB; ++q, k0 += HP_NB) {
    a.k0 = k0;
    a.wmax = wmax + q;
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel((const void *)hh_panel_kernel, dim3(G), dim3(HP_THREADS), args, smem, s);
    if (e != cudaSuccess) return e;
    a.bar0 += 2 * HP_NB;
    // A22 -= V W^T + W V^T on the rows and columns past the panel
    const int k1 = k0 + HP_NB, m = n - k1;
    ps.X = w.V + (int64_t)k0 * n + k1; ps.Y = a.W + k1; ps.ld = n; ps.nk = HP_NB;
    ps.rows = m; ps.rows_p = (int)slice_rows_padded(m); ps.ymax = a.wmax;
    e = launch_slice_pair(ps, s);
    if (e != cudaSuccess) return e;
    SliceGemmArgs g;
    g.A = ps.dig_p; g.ea = ps.exp_p; g.B = ps.dig_q; g.eb = ps.exp_q; g.nkb = nkb;
    g.M = g.N = m; g.sym = 1; g.C = w.A + (int64_t)k1 * n + k1; g.ldc = n; g.beta = 1.0; g.alpha_neg = 1;
    g.err = w.flags;
    slice_gemm_plan(&g, nsm, 0);
    e = launch_slice_gemm(g, nsm, s);
    if (e != cudaSuccess) return e;
    *launches += 4;
  }
  *k0_out = k0;
  return cudaSuccess;
}

// ---- the eigenvectors' dense products from digits (slice_gemm.cu) ----
// From VD_MIN_N on: the re-orthonormalisation X (3 - X^T X) / 2 and the compact-WY
// blocks.  The vectors' columns have unit length all along, so their digits
// take one fixed exponent (2^-56 beside the entries of a column of length 1; the
// FP64 sums round at about that) and need no pass for the maxima.
// V's digits are formed once; per block of 64 reflectors (last to first, rows
// r > 64 b): the vectors' digits, W1 = V_b Y, its digits, Y -= M_b W1.
// Measured (bisection to the transposition; a quarter of the vectors kept): n = 3300
// 46.7 -> 22.7 ms, n = 1800 13.1 -> 9.7, n = 800 4.16 -> 3.81, n = 264 1.56 -> 1.43; the blocks
// alone took 21.9 ms of FP64 tiles at n = 3300 and 1.5 from digits.  All eight
// levels of digit pairs are kept: with seven the vectors' orthogonality falls
// from 2e-15 to 2e-14 (V's rows hold a 1 beside entries of 1/sqrt(n), so their
// scale is far above what the sums carry); with eight it is the FP64 form's.
constexpr int VD_MIN_N = 200;
constexpr int VD_EXP = 2;   // |x| < 2: stored exponents carry one more bit in base 256

struct VecDigits {
  int n, k, nsm;
  int np, kp, nkb;        // padded rows, 16-k blocks of length n
  uint8_t *dV, *dY, *dM, *dW;
  int *eV, *eY, *eM, *eW;
  int *flags;
  size_t bytes;
};

// Arrays in `base` (counted only when base is null).
VecDigits vec_digits(int n, int k, int nsm, int *flags, void *base) {
  VecDigits d;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    uint8_t *p = base ? (uint8_t *)base + off : nullptr;
    off += (bytes + 255) / 256 * 256;
    return p;
  };
  d.n = n; d.k = k; d.nsm = nsm; d.flags = flags;
  d.np = (int)slice_rows_padded(n); d.kp = (int)slice_rows_padded(k);
  d.nkb = (n + SL_K - 1) / SL_K;
  d.dV = take(slice_digit_bytes(n, d.nkb, 7));    // V's rows; before that X's rows (K = k) and F's
  d.dY = take(slice_digit_bytes(k, d.nkb, 7));    // the vectors' columns (K = n)
  d.dM = take(slice_digit_bytes(n, WY_NB / SL_K, 7));
  d.dW = take(slice_digit_bytes(k, std::max(WY_NB / SL_K, (k + SL_K - 1) / SL_K), 7));
  d.eV = (int *)take(d.np * sizeof(int));
  d.eY = (int *)take(d.kp * sizeof(int));
  d.eM = (int *)take(d.np * sizeof(int));
  d.eW = (int *)take(d.kp * sizeof(int));
  d.bytes = off;
  return d;
}

SliceSrc digit_rows(const double *X, int64_t ld, int rows, int64_t K, uint8_t *dig, int *exps) {
  SliceSrc a;
  a.X = X; a.ld = ld; a.rows = rows; a.rows_p = (int)slice_rows_padded(rows); a.K = K; a.nkb = (int)((K + SL_K - 1) / SL_K);
  a.dig = dig; a.exps = exps; a.exp_batch = a.rows_p;
  return a;
}

// Digits of the vectors' columns (X [n][k]) from row 16 kb_first on.
cudaError_t slice_vectors(const VecDigits &d, const double *X, int kb_first, cudaStream_t s) {
  SliceSrc a = digit_rows(X, d.k, d.k, d.n, d.dY, d.eY);
  a.cols = 1; a.fixed_exp = VD_EXP; a.kb_first = kb_first;
  return launch_slice_operand(a, 7, 8, 1, s);
}

cudaError_t run_slice(SliceGemmArgs &g, const VecDigits &d, double *partial, size_t partial_bytes, cudaStream_t s) {
  g.err = d.flags;
  g.levels = 8;
  const size_t need = slice_gemm_plan(&g, d.nsm, partial_bytes);
  g.partial = need ? partial : nullptr;
  return launch_slice_gemm(g, d.nsm, s);
}

// X <- X (3 - X^T X) / 2 in place; G, Xn: k x k and n x k scratch.
cudaError_t lowdin_digits(const VecDigits &d, double *X, double *G, double *Xn, double *partial, size_t partial_bytes,
                          cudaStream_t s) {
  const int n = d.n, k = d.k;
  cudaError_t e = slice_vectors(d, X, 0, s);
  if (e != cudaSuccess) return e;
  SliceGemmArgs g;   // G = X^T X
  g.A = g.B = d.dY; g.ea = g.eb = d.eY; g.nkb = d.nkb; g.M = g.N = k; g.sym = 1; g.C = G; g.ldc = k;
  if ((e = run_slice(g, d, partial, partial_bytes, s)) != cudaSuccess) return e;
  lowdin_factor_kernel<double><<<152, 256, 0, s>>>(G, k);
  if ((e = launch_slice_operand(digit_rows(G, k, k, k, d.dW, d.eW), 7, 8, 1, s)) != cudaSuccess) return e;
  if ((e = launch_slice_operand(digit_rows(X, k, n, k, d.dV, d.eV), 7, 8, 1, s)) != cudaSuccess) return e;
  SliceGemmArgs h;   // Xn[r][c] = sum F[c][j] X[r][j] (F symmetric)
  h.A = d.dW; h.ea = d.eW; h.B = d.dV; h.eb = d.eV; h.nkb = (k + SL_K - 1) / SL_K; h.M = k; h.N = n; h.C = Xn; h.ldc = k;
  if ((e = run_slice(h, d, partial, partial_bytes, s)) != cudaSuccess) return e;
  return cudaMemcpyAsync(X, Xn, (size_t)n * k * sizeof(double), cudaMemcpyDeviceToDevice, s);
}

// Every block Y <- Y - M_b (V_b Y), last to first; W1: 64 x k scratch.
cudaError_t wy_digits(const VecDigits &d, const double *V, const double *Mall, int nblk, double *Y, double *W1,
                      double *partial, size_t partial_bytes, cudaStream_t s, int *launches) {
  const int n = d.n, k = d.k;
  cudaError_t e = launch_slice_operand(digit_rows(V, n, n, n, d.dV, d.eV), 7, 8, 1, s);
  if (e != cudaSuccess) return e;
  for (int b = nblk - 1; b >= 0; --b) {
    const int j0 = b * WY_NB, nb = std::min(WY_NB, n - 2 - j0), kb0 = j0 / SL_K;
    if ((e = slice_vectors(d, Y, kb0, s)) != cudaSuccess) return e;
    SliceGemmArgs g;   // W1[i][c] = sum_r V[j0 + i][r] Y[r][c]
    g.A = d.dY; g.ea = d.eY;
    g.B = d.dV + (int64_t)b * d.nkb * (SL_ROWS * SL_K * 2 * 7); g.eb = d.eV + j0;
    g.nkb = d.nkb; g.kb_first = kb0; g.M = k; g.N = nb; g.C = W1; g.ldc = k;
    if ((e = run_slice(g, d, partial, partial_bytes, s)) != cudaSuccess) return e;
    SliceSrc w = digit_rows(W1, k, k, nb, d.dW, d.eW);
    w.cols = 1;
    if ((e = launch_slice_operand(w, 7, 8, 1, s)) != cudaSuccess) return e;
    const int rows = n - 1 - j0;   // M_b's rows j0 .. n - 2 stand for Y's rows j0 + 1 ..
    if ((e = launch_slice_operand(digit_rows(Mall + ((int64_t)b * (n - 1) + j0) * WY_NB, WY_NB, rows, nb, d.dM, d.eM), 7,
                                  8, 1, s)) != cudaSuccess)
      return e;
    SliceGemmArgs u;   // Y[j0 + 1 + r][c] -= sum_i M_b[j0 + r][i] W1[i][c]
    u.A = d.dW; u.ea = d.eW; u.B = d.dM; u.eb = d.eM; u.nkb = (nb + SL_K - 1) / SL_K;
    u.M = k; u.N = rows; u.C = Y + (int64_t)(j0 + 1) * k; u.ldc = k; u.beta = 1.0; u.alpha_neg = 1;
    if ((e = run_slice(u, d, nullptr, 0, s)) != cudaSuccess) return e;
    *launches += 8;
  }
  return cudaSuccess;
}

// Steps 3-6 in arithmetic T.
template <typename T>
cudaError_t eig_vectors_impl(EigWork &w, int n, int k, double *Ut, int *flags, cudaStream_t s, int *launches) {
  const size_t smem = 2 * (size_t)n * sizeof(T);
  {
    cudaError_t e = allow_max_dynamic_smem((const void *)bisect_kernel, g_smem_bisect);
    if (e != cudaSuccess) return e;
    e = allow_max_dynamic_smem((const void *)inverse_iteration_kernel<T, true>, g_smem_invit[0]);
    if (e != cudaSuccess) return e;
    e = allow_max_dynamic_smem((const void *)inverse_iteration_kernel<T, false>, g_smem_invit[1]);
    if (e != cudaSuccess) return e;
    e = allow_max_dynamic_smem((const void *)twisted_kernel<true>, g_smem_tw[0]);
    if (e != cudaSuccess) return e;
    e = allow_max_dynamic_smem((const void *)twisted_kernel<false>, g_smem_tw[1]);
    if (e != cudaSuccess) return e;
    e = allow_max_dynamic_smem((const void *)wy_build_t_kernel<T>, g_smem_wy);
    if (e != cudaSuccess) return e;
  }
  {
    // One warp per eigenvalue, four or more per block, one or more per scheduler
    // of the SM (the warps of one-warp blocks can share a scheduler, and each
    // FP64 instruction holds it for the whole warp); just enough for one wave of
    // blocks, up to 16: 825 warps in blocks of four put eight on some SMs.
    int dev = 0, nsm = 148, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      nsm = 148;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) optin = 0;
    cudaGetLastError();
    const int wpb = std::min(16, std::max(4, (k + nsm - 1) / nsm));
    const size_t b64 = (size_t)n * sizeof(double2), b32 = (size_t)n * sizeof(float2);
    const bool pre = b64 + b32 + 1024 <= (size_t)optin;
    bisect_kernel<<<(k + wpb - 1) / wpb, wpb * 32, pre ? b64 + b32 : b64, s>>>(w.d, w.p, w.scal, n, k, pre, w.lam);
  }
  T *X = reinterpret_cast<T *>(w.X), *lu = reinterpret_cast<T *>(w.lu), *V = reinterpret_cast<T *>(w.V);
  {
    // the twisted factorisations, where T fits in a block's shared memory
    int dev = 0, optin = 0, nsm_iv = 148;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
      optin = 48 * 1024;
    if (cudaDeviceGetAttribute(&nsm_iv, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) nsm_iv = 148;
    cudaGetLastError();
    int *need = nullptr;
    const size_t tw_static = 6 * 1024, tw_t = 3 * (size_t)n * sizeof(double);
    if (tw_t + tw_static <= (size_t)optin) {
      int V = 4;   // few vectors per block, as long as the blocks make one wave
      while (V < 32 && (k + V - 1) / V > nsm_iv) V *= 2;
      const size_t tw_all = tw_t + 2 * (size_t)n * V * sizeof(double);
      need = reinterpret_cast<int *>(w.w);
      const int blocks = (k + V - 1) / V;
      if (tw_all + tw_static <= (size_t)optin && blocks <= nsm_iv)
        twisted_kernel<true><<<blocks, TW_THREADS, tw_all, s>>>(w.d, w.e, w.lam, w.scal, n, k, V, X, lu, need);
      else
        twisted_kernel<false><<<blocks, TW_THREADS, tw_t, s>>>(w.d, w.e, w.lam, w.scal, n, k, V, X, lu, need);
      *launches += 1;
    }
    // inverse iteration for what is left: factors in shared memory when at least
    // one thread's share fits
    // shared-memory factors only when every vector then runs in one wave; FP64
    // instructions cost a warp the same with 2 active lanes as with 32, so
    // otherwise 32 vectors per warp with the factors in L2 is faster
    const size_t budget = (size_t)optin - 1024, per_thread = 6 * (size_t)n * sizeof(T);
    int tpb = smem + per_thread <= budget ? (int)std::min<size_t>(32, (budget - smem) / per_thread) : 0;
    if (tpb >= 1 && (k + tpb - 1) / tpb > nsm_iv) tpb = 0;
    if (tpb >= 1)
      inverse_iteration_kernel<T, true><<<(k + tpb - 1) / tpb, tpb, smem + tpb * per_thread, s>>>(
          w.d, w.e, w.lam, w.scal, n, k, X, lu, need, flags);
    else
      inverse_iteration_kernel<T, false><<<(k + 31) / 32, 32, smem, s>>>(w.d, w.e, w.lam, w.scal, n, k, X, lu, need, flags);
  }
  *launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // re-orthonormalise: G = X^T X, F = (3 - G)/2, X <- X F.  One pass squares
  // the non-orthogonality inverse iteration leaves (about 1e-12 here).  X^T X
  // is split over its length-n sum (partials in the free inverse-iteration
  // scratch): a 64 x 64 FP64 tile over all n rows would keep one SM busy for
  // milliseconds.
  T *G = lu;                       // k*k scratch (inverse-iteration scratch is free now)
  T *Xn = lu + (int64_t)k * k;     // n*k scratch
  // digits where the vectors are large enough and the scratch holds them: the
  // factor F and X F first, then the digits (5 n^2 doubles in all)
  VecDigits vd{};
  bool digits = false;
  double *vd_part = w.wy;
  const size_t vd_part_bytes = (size_t)w.wy_r0 * sizeof(double);
  if (n >= VD_MIN_N) {
    int dev = 0, nsm = 0;
    digits = cudaGetDevice(&dev) == cudaSuccess &&
             cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
    cudaGetLastError();
    const size_t head = (((size_t)k * k + (size_t)n * k) * sizeof(double) + 255) / 256 * 256;
    vd = vec_digits(n, k, nsm, flags, (char *)w.lu + head);
    digits = digits && head + vd.bytes <= (size_t)5 * n * n * sizeof(double);
  }
  if (digits) {
    if ((e = launch_fill_int(vd.eY, vd.kp, VD_EXP, s)) != cudaSuccess) return e;
    e = lowdin_digits(vd, reinterpret_cast<double *>(X), reinterpret_cast<double *>(G), reinterpret_cast<double *>(Xn),
                      vd_part, vd_part_bytes, s);
    if (e != cudaSuccess) return e;
    *launches += 14;
  } else {
    T *Gpart = Xn + (int64_t)n * k;
    const int64_t room = 5 * (int64_t)n * n - (int64_t)k * k - (int64_t)n * k;
    int nsp = (int)std::min<int64_t>((n + 63) / 64, std::max<int64_t>(1, room / ((int64_t)k * k)));
    const int64_t ks = (n + nsp - 1) / nsp;
    nsp = (int)((n + ks - 1) / ks);
    GemmArgs<T> g;
    g.M = k; g.N = k; g.K = n; g.ksplit = ks;
    g.A = X; g.lda = k;   // A[kidx][m] = X[i][m]  (M-major)
    g.B = X; g.ldb = k;   // B[kidx][n] = X[i][n]  (N-major)
    g.C = Gpart; g.ldc = k; g.strideC = (int64_t)k * k;
    g.syrk = 1;
    e = launch_gemm<T>(g, nsp, false, false, s);
    if (e != cudaSuccess) return e;
    sum_partials_kernel<T><<<152, 256, 0, s>>>(Gpart, nsp, (int64_t)k * k, (int64_t)k * k, G);
    lowdin_factor_kernel<T><<<152, 256, 0, s>>>(G, k);
    GemmArgs<T> h;
    h.M = n; h.N = k; h.K = k;
    h.A = X; h.lda = k;   // K-major rows of X
    h.B = G; h.ldb = k;   // N-major
    h.C = Xn; h.ldc = k;
    e = launch_gemm<T>(h, 1, true, false, s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(X, Xn, (size_t)n * k * sizeof(T), cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    *launches += 4;
  }
  // compact-WY back-transformation, blocks of WY_NB reflectors from the last:
  // Y <- Y - M_b (V_b^T Y) with M_b = V_b T_b.  Every block's G, T and M_b are
  // formed first (every G in one launch, the T recurrences in one launch, all
  // M_b in one batched GEMM over rows 1..n-1; V carries WY_NB zero rows past
  // its end for the last block), then the blocks are applied in order: by one
  // cooperative kernel, or two GEMMs each where that kernel cannot launch.
  const int nref = n - 2;  // reflectors 0 .. n-3
  if (nref > 0) {
    const int nblk = (nref + WY_NB - 1) / WY_NB;
    const int nsplit_max = (int)((n + WY_KSPLIT - 1) / WY_KSPLIT);
    // region 0 (w.wy_r0 doubles): W1's split partials and W1 for the
    // block-at-a-time form, or the cooperative kernel's partials and W1
    T *W1p = reinterpret_cast<T *>(w.wy);                        // [nsplit][nb][k]
    T *W1 = W1p + (int64_t)nsplit_max * WY_NB * k;               // [nb][k]
    T *Gs = reinterpret_cast<T *>(w.wy) + w.wy_r0;               // [nblk][nb][nb]
    T *Tm = Gs + (int64_t)nblk * WY_NB * WY_NB;                  // [nblk][WY_NB][WY_NB]
    T *Mall = Tm + (int64_t)nblk * WY_NB * WY_NB;                // [nblk][n-1][WY_NB]
    {
      // every block's G = V_b V_b^T in one launch (column chunks of WY_KSPLIT;
      // a block-at-a-time GEMM keeps only ~n/64 SMs busy), the chunk partials
      // in the M_b region, which is written only after the T recurrences
      T *Gp = Mall;                                              // [nchunk][nblk][nb][nb]
      const int64_t nchunk = (n - 1 + WY_KSPLIT - 1) / WY_KSPLIT;
      e = launch_gram_panels(V, n, nref, WY_NB, WY_KSPLIT, Gp, s);
      if (e != cudaSuccess) return e;
      sum_partials_kernel<T><<<152, 256, 0, s>>>(Gp, (int)nchunk, (int64_t)nblk * WY_NB * WY_NB,
                                                 (int64_t)nblk * WY_NB * WY_NB, Gs);
      *launches += 2;
    }
    wy_build_t_kernel<T><<<nblk, 4 * WY_NB, 2 * WY_NB * (WY_NB + 1) * sizeof(T), s>>>(Gs, w.tau, nref, Tm);
    {
      GemmArgs<T> m;                      // M_b[r-1][c] = sum_i V[j0+i][r] T_b[i][c], r = 1..n-1
      m.M = n - 1; m.N = WY_NB; m.K = WY_NB;
      m.A = V + 1; m.lda = n; m.strideA = (int64_t)WY_NB * n;        // A[kidx=i][m] = V[j0+i][1+m]
      m.B = Tm; m.ldb = WY_NB; m.strideB = (int64_t)WY_NB * WY_NB;
      m.C = Mall; m.ldc = WY_NB; m.strideC = (int64_t)(n - 1) * WY_NB;
      e = launch_gemm<T>(m, nblk, false, false, s);
      if (e != cudaSuccess) return e;
    }
    *launches += 2;
    // the blocks applied from digits; or by one cooperative kernel when its CTAs
    // fit at once and region 0 holds their partials; otherwise two GEMMs per block
    bool applied = false;
    if (digits) {
      const size_t w1 = ((size_t)WY_NB * k + 31) / 32 * 32;   // W1 in front of the partials
      e = wy_digits(vd, reinterpret_cast<const double *>(V), reinterpret_cast<const double *>(Mall), nblk,
                    reinterpret_cast<double *>(X), w.wy, w.wy + w1, vd_part_bytes - w1 * sizeof(double), s, launches);
      if (e != cudaSuccess) return e;
      applied = true;
    }
    if (!applied && sizeof(T) == sizeof(double)) {
      int dev = 0, nsm = 0, coop = 0, per_sm = 0;
      const int S = (k + 63) / 64;
      if (cudaGetDevice(&dev) == cudaSuccess &&
          cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
          cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop && S <= nsm &&
          allow_max_dynamic_smem((const void *)wy_apply_kernel, g_smem_wa) == cudaSuccess &&
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)wy_apply_kernel, 256, WA_SMEM) ==
              cudaSuccess && per_sm >= 1) {
        int G = nsm / S;
        while (G > 1 && (int64_t)(S * G + S) * 4096 > w.wy_r0) --G;
        if ((int64_t)(S * G + S) * 4096 <= w.wy_r0) {
          WyApplyArgs a;
          a.V = reinterpret_cast<const double *>(V);
          a.M = reinterpret_cast<const double *>(Mall);
          a.Y = reinterpret_cast<double *>(X);
          a.Wp = w.wy;
          a.W1 = w.wy + (int64_t)S * G * 4096;
          // the fused reduction's barrier word (that kernel has finished)
          a.gb = reinterpret_cast<GridBar *>(w.grid_ws + 4 * (size_t)n + 2);
          a.flags = flags;
          a.n = n; a.k = k; a.nref = nref; a.nblk = nblk; a.G = G;
          e = cudaMemsetAsync(a.gb, 0, sizeof(GridBar), s);
          if (e != cudaSuccess) return e;
          void *args[] = {&a};
          e = cudaLaunchCooperativeKernel((const void *)wy_apply_kernel, dim3((unsigned)(S * G)), dim3(256), args,
                                          WA_SMEM, s);
          if (e != cudaSuccess) return e;
          *launches += 1;
          applied = true;
        }
      }
      cudaGetLastError();
    }
    for (int bi = nblk - 1; bi >= 0 && !applied; --bi) {
      const int j0 = bi * WY_NB, nb = std::min(WY_NB, nref - j0);
      const int r0 = j0 + 1;
      const int64_t len = n - r0;
      const int nsplit = (int)((len + WY_KSPLIT - 1) / WY_KSPLIT);
      GemmArgs<T> h;                      // W1 partials = V_b^T Y over row chunks
      h.M = nb; h.N = k; h.K = len; h.ksplit = WY_KSPLIT;
      h.A = V + (int64_t)j0 * n + r0; h.lda = n;
      h.B = X + (int64_t)r0 * k; h.ldb = k;
      h.C = W1p; h.ldc = k; h.strideC = (int64_t)nb * k;
      e = launch_gemm<T>(h, nsplit, true, false, s);
      if (e != cudaSuccess) return e;
      sum_partials_kernel<T><<<152, 256, 0, s>>>(W1p, nsplit, (int64_t)nb * k, (int64_t)nb * k, W1);
      GemmArgs<T> u;                      // Y[r0:, :] -= M_b[r0:, 0:nb] W1
      u.M = (int)len; u.N = k; u.K = nb;
      u.A = Mall + (int64_t)bi * (n - 1) * WY_NB + (int64_t)(r0 - 1) * WY_NB; u.lda = WY_NB;   // K-major
      u.B = W1; u.ldb = k;
      u.C = X + (int64_t)r0 * k; u.ldc = k;
      u.alpha = -1.0; u.beta = 1.0;
      e = launch_gemm<T>(u, 1, true, false, s);
      if (e != cudaSuccess) return e;
      *launches += 3;
    }
  }
  dim3 tb(32, 8), tg((k + 31) / 32, (n + 31) / 32);
  transpose_kernel<T><<<tg, tb, 0, s>>>(X, n, k, Ut);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_eig_tridiag(EigWork &w, int n, double thresh, cudaStream_t s, int *launches) {
  cudaError_t e = cudaSuccess;
  int k0 = 0;
  e = launch_blocked(w, n, s, launches, &k0);
  if (e != cudaSuccess) return e;
  const bool fused = launch_fused<double>(w, n, k0, s, launches, &e);
  if (e != cudaSuccess) return e;
  if (!fused && k0 > 0) return cudaErrorNotSupported;   // not reached: the tail's rows fit in shared memory
  if (!fused) {
    for (int k = 0; k + 2 < n; ++k) {
      const int L = n - k - 1;
      hh_reflector_kernel<<<1, RB, 0, s>>>(w.A, w.V, w.d, w.e, w.tau, w.scal, n, k);
      int symv_blocks = (L * 32 + 255) / 256;
      hh_symv_kernel<<<symv_blocks, 256, 0, s>>>(w.A, w.V, w.p, w.scal, n, k);
      hh_w_kernel<<<1, RB, 0, s>>>(w.V, w.p, w.w, w.scal, n, k);
      int64_t LL = (int64_t)L * L;
      int ub = (int)((LL + 255) / 256);
      if (ub > 152 * 8) ub = 152 * 8;
      hh_update_kernel<<<ub, 256, 0, s>>>(w.A, w.V, w.w, n, k);
      *launches += 4;
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    hh_finalize_kernel<<<1, 32, 0, s>>>(w.A, w.d, w.e, n);
    *launches += 1;
  }
  // e2 reuses w.p (length n)
  {
    const size_t st = 2 * (size_t)n * sizeof(double);
    const bool staged = st <= 180 * 1024 &&
                        allow_max_dynamic_smem((const void *)tridiag_bounds_kernel, g_smem_bounds) == cudaSuccess;
    cudaGetLastError();
    tridiag_bounds_kernel<<<1, RB, staged ? st : 0, s>>>(w.d, w.e, n, thresh, w.scal, w.p, w.count, staged);
  }
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_eig_vectors(EigWork &w, int n, int k, double *Ut, int *flags, cudaStream_t s,
                               int *launches) {
  if (k <= 0) return cudaSuccess;
  return eig_vectors_impl<double>(w, n, k, Ut, flags, s, launches);
}

}  // namespace ltgw
