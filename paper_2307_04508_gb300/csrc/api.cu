// C ABI of the LT-GW library: argument checking, workspace, host/device
// staging and the order of the steps of Sec. 2 (frozen-core slice -> NAF ->
// Pi -> screening -> W_nm -> Sigma(i w) -> Pade -> Newton).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <functional>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "digit_memory.h"
#include "kernels.cuh"

namespace ltgw {
int g_launch_count = 0;
}

using namespace ltgw;

namespace {

// Device bump allocator; grows (free + malloc) only between calls.
struct Arena {
  char *base = nullptr;
  size_t cap = 0, off = 0;
  bool sizing = false;
  size_t need = 0;
  void begin_sizing() { sizing = true; need = 0; off = 0; }
  template <class T>
  T *take(size_t n) {
    off = (off + 255) & ~(size_t)255;
    T *p = sizing ? nullptr : reinterpret_cast<T *>(base + off);
    off += std::max<size_t>(n, 1) * sizeof(T);
    if (sizing) need = off;
    return p;
  }
  cudaError_t commit() {
    sizing = false;
    size_t want = need;
    off = 0;
    if (want <= cap) return cudaSuccess;
    if (base) cudaFree(base);
    base = nullptr;
    cap = 0;
    cudaError_t e = cudaMalloc(&base, want);
    if (e != cudaSuccess) { cudaGetLastError(); return e; }
    cap = want;
    return cudaSuccess;
  }
  void release() {
    if (base) cudaFree(base);
    base = nullptr;
    cap = 0;
  }
};

bool is_device_ptr(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

enum Stage { EV_START = 0, EV_NAF, EV_PI0, EV_PI1, EV_PI, EV_SCREEN, EV_WNM, EV_SIGQP, EV_END, EV_TRI0, EV_TRI1,
             EV_K0, EV_VEC1, EV_COUNT };

}  // namespace

struct ltgw_ctx {
  int device = 0;
  ltgw_status st = LTGW_OK;
  std::string err;
  Arena a1, a2, a3;  // a1: inputs; a2: after the NAF count is known; a3: NAF scratch
  int *flags = nullptr;
  bool timing = false;
  cudaEvent_t ev[EV_COUNT] = {};
  // side stream for the copy of inputs first read late in the solve (B_tgt),
  // forked from and joined back to the caller's stream by two events
  cudaStream_t side = nullptr;
  cudaEvent_t fork_ev = nullptr, join_ev = nullptr;
  // streamed solve: the block callback fills one of two block buffers on its
  // own stream while the caller's stream consumes the other; per buffer, an
  // event when its block has arrived and one when its consumers are done
  cudaStream_t fill_stream = nullptr;
  cudaEvent_t blk_ready[2] = {}, blk_done[2] = {};
  ltgw_stats stats{};
  int launches = 0;
  double pi_tc_flops = 0.0;
  int tri_n = 0;
  double gen_ms = 0.0;
  int n_sm = 148;
  Arena a4;  // tensor-core scratch: tile lists and partial tiles
  Arena a5;  // tensor-core operand copies consumed by the next contraction
  size_t digit_max = kSliceHold;   // digits and partials held at a time (ltgw_set_digit_memory)
  // Autotuner of the tensor-core contractions (off by default): per shape, the
  // (scales per CTA, K-splits) configuration that timed fastest on this GPU.
  struct TcKey {
    int kind, n_tiles, n_t, out_mode;
    int64_t Kp, rows_a, rows_b;
    bool operator<(const TcKey &o) const {
      return std::tie(kind, n_tiles, n_t, out_mode, Kp, rows_a, rows_b) <
             std::tie(o.kind, o.n_tiles, o.n_t, o.out_mode, o.Kp, o.rows_a, o.rows_b);
    }
  };
  struct TcChoice { int nt_group; int64_t splits; };
  bool autotune = false;
  std::map<TcKey, TcChoice> tuned;

  void fail(ltgw_status c, const std::string &m) {
    if (st == LTGW_OK) { st = c; err = m; }
  }
  ltgw_status status() const { return st; }
  void reset() { st = LTGW_OK; err.clear(); launches = 0; }
  void mark(Stage s, cudaStream_t stream) {
    if (timing) cudaEventRecord(ev[s], stream);
  }
  double ms(Stage a, Stage b) {
    float t = 0.f;
    if (!timing) return 0.0;
    if (cudaEventElapsedTime(&t, ev[a], ev[b]) != cudaSuccess) { cudaGetLastError(); return 0.0; }
    return (double)t;
  }
};

#define CHECK_LAUNCH(ctx, expr, nk)                                                              \
  do {                                                                                           \
    cudaError_t _e = (expr);                                                                     \
    (ctx)->launches += (nk);                                                                     \
    if (_e != cudaSuccess) {                                                                     \
      (ctx)->fail(LTGW_ERR_DEVICE, std::string(#expr) + ": " + cudaGetErrorString(_e));          \
      return (ctx)->status();                                                                    \
    }                                                                                            \
  } while (0)

#define REQUIRE(ctx, cond, msg)                                                                  \
  do {                                                                                           \
    if (!(cond)) {                                                                               \
      (ctx)->fail(LTGW_ERR_BAD_ARG, msg);                                                        \
      return (ctx)->status();                                                                    \
    }                                                                                            \
  } while (0)

namespace {

ltgw_status copy_in(ltgw_ctx *ctx, void *dst, const void *src, size_t bytes, cudaStream_t s) {
  if (bytes == 0) return LTGW_OK;
  LTGW_CUDA(ctx, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, s));
  return LTGW_OK;
}

ltgw_status read_small(ltgw_ctx *ctx, void *dst, const void *src, size_t bytes, cudaStream_t s) {
  if (bytes == 0) return LTGW_OK;
  LTGW_CUDA(ctx, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, s));
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  return LTGW_OK;
}

ltgw_status check_flags(ltgw_ctx *ctx, cudaStream_t s) {
  int h[FLAG_COUNT];
  if (read_small(ctx, h, ctx->flags, sizeof(h), s) != LTGW_OK) return ctx->status();
  if (h[FLAG_EIG]) ctx->fail(LTGW_ERR_EIG, "NAF eigensolver: a vector was not finite, or a wait in the reduction timed out");
  if (h[FLAG_NOT_SPD]) ctx->fail(LTGW_ERR_NOT_SPD, "screening: a pivot of 1 - Pi(iw) was not positive");
  if (h[FLAG_TC_TIMEOUT]) ctx->fail(LTGW_ERR_DEVICE, "tensor-core kernel: a pipeline wait timed out");
  return ctx->status();
}

// NAF basis on device data: K = B B^T, eigenvectors with eigenvalue > thresh
// as rows of Ut (descending eigenvalue), their eigenvalues in lam.
ltgw_status naf_metric_tc(ltgw_ctx *ctx, int n, int64_t n_pairs, const double *B, int64_t ld, double *K,
                          cudaStream_t s, double beta = 0.0);

// ---- FP64 contractions on the tensor cores from integer digits (slice_gemm.cu)
// The FP64 form's products: 7 digits in base 256 hold 55 bits relative to each
// operand row's largest magnitude (2^e a power of two 2 to 4 times that), and with
// the products kept (levels i + j <= 8, or 9) an entry is off by at most K 2^-55
// 2^(e_i + e_j).  In norm that is an FP64 sum's error or less; an entry whose terms are
// all small beside its rows' largest ones loses what lies below, where an FP64
// sum (K 2^-53 sum |a||b|) would keep it.  So the polarisability as a result has
// those entries summed in FP64 (pi_weak.cu); inside a solve, in the NAF metric and
// in the inverse they are summed over or mixed by factorisations whose own error
// is one of the norm.
// The emulated FP64 forms: n_slices digits in base 128, one exponent per whole
// operand row, and no CUDA-core kernel to fall back to.
struct SliceForm {
  int ns, bits;
  bool required;   // LTGW_ERR_NOMEM when the digits do not fit
};
constexpr SliceForm kFp64Digits{7, 8, false};
constexpr int kEmuSlices = 6;   // slices per operand row in the LTGW_FP64_EMU solve
constexpr SliceForm emu_digits(int n_slices) { return {n_slices, 7, true}; }
// A product's digits and K-split partials are held in pieces (matrices of a batch,
// columns, frequencies): as many at a time as the context's limit
// (ltgw_set_digit_memory) and half of what is free on the device allow.  The
// lengths of the sums (pair chunks, K splits) follow from the product's sizes
// alone (the splits from those of a piece of kSliceHold bytes), so a result has
// the same bits whatever piece fits.  A pair chunk costs another conversion of the
// sums and pass over the output, 0.5 ms for ten moments of N = 2258: in chunks of
// 12,000 pairs (768 MiB) 4 % of the time, of 25,000 2 %.
constexpr size_t kSliceTermMax = (size_t)1536 << 20;   // digits of one matrix's operands (sets its pair chunk)
constexpr size_t kSlicePartialMax = (size_t)1 << 30;   // K-split partial tiles of a piece
constexpr int64_t kSliceMinCols = 1024;                // columns of a projection's smallest piece

// Products this small stay on the CUDA-core kernels.  Digits take two to four
// launches (about 20 us), which a 64 x 64 FP64 tile passes at a length of a few
// hundred however few tiles there are: request of 8 occupied orbitals, metric
// (264^2 x 560) 0.587 -> 0.042 ms, Pi (65^2 x 560 x 8) 0.616 -> 0.071, projection
// (65 x 560 x 264) 0.58 -> 0.10, W_nm 0.211 -> 0.057; without NAF 48^2 x 64 x 24
// 0.062 -> 0.042.  A limit of 2e5 changes no case measured.
bool slices_pay(int64_t m, int64_t n, int64_t k, int64_t batch) {
  return k >= 48 && (double)m * (double)n * (double)k * (double)batch >= 2e6;
}

int slice_blocks(int64_t K) { return (int)((K + SL_K - 1) / SL_K); }

struct SliceOperand {
  uint8_t *dig = nullptr;
  int *exps = nullptr;
  int rows_p = 0, nkb = 0;
  int64_t dig_batch = 0;
  void layout(Arena &A, int64_t rows, int64_t K, int batch, SliceForm f) {
    rows_p = (int)slice_rows_padded(rows);
    nkb = slice_blocks(K);
    dig_batch = slice_digit_bytes(rows, nkb, f.ns);
    dig = A.take<uint8_t>((size_t)dig_batch * batch);
    exps = A.take<int>((size_t)rows_p * batch);
  }
  SliceSrc source(const double *X, int64_t ld, int64_t x_batch, int rows, int64_t K, bool cols) const {
    SliceSrc a;
    a.X = X; a.ld = ld; a.x_batch = x_batch; a.cols = cols; a.rows = rows; a.rows_p = rows_p; a.K = K; a.nkb = nkb;
    a.dig = dig; a.dig_batch = dig_batch; a.exps = exps; a.exp_batch = rows_p;
    return a;
  }
};

// The next smaller equal pieces of n items; false when they are single already.
bool next_piece(int n, int *blk) {
  if (*blk == 1) return false;
  int pieces = (n + *blk - 1) / *blk, b = *blk;
  while (b >= *blk) b = (n + pieces) / (pieces + 1), ++pieces;
  *blk = b;
  return true;
}

// The next fewer columns of one matrix.
bool next_columns(int64_t *cols) {
  if (*cols <= kSliceMinCols) return false;
  *cols = (*cols / 2 + 127) / 128 * 128;
  return true;
}

// Each product below has a struct of its piece: layout(arena) takes its digits,
// partial() is the bytes of its K-split partials (pointer `part`), shrink() takes
// the next smaller piece and is false at the smallest.
template <class P>
size_t piece_bytes(Arena &ar, P &p) {
  ar.begin_sizing();
  p.layout(ar);
  if (const size_t pb = p.partial()) ar.take<double>(pb / sizeof(double));
  ar.sizing = false;
  return ar.need;
}

// Memory (arena a5) for the largest piece that fits.  False when the smallest one
// does not either: an error in the forms that need the digits, else the product is
// left to the CUDA-core kernels.  Other contexts' solves size their own workspace
// from what is free, so more than half of it is taken for the smallest piece only.
template <class P>
bool slice_fit(ltgw_ctx *ctx, bool required, P &p) {
  Arena &ar = ctx->a5;
  for (;;) {
    const size_t need = piece_bytes(ar, p);
    const bool allowed = required || need <= ctx->digit_max;
    bool ok = need <= ctx->digit_max;
    if (ok && need > ar.cap) {
      size_t free_b = 0, total_b = 0;
      if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) cudaGetLastError();
      else ok = need <= (free_b + ar.cap) / 2;
    }
    if (!ok && p.shrink()) continue;
    if (allowed && ar.commit() == cudaSuccess) {
      p.layout(ar);
      const size_t pb = p.partial();
      p.part = pb ? ar.take<double>(pb / sizeof(double)) : nullptr;
      return true;
    }
    if (ok && p.shrink()) continue;
    if (required) ctx->fail(LTGW_ERR_NOMEM, "slice operand allocation failed");
    return false;
  }
}

// One piece of a digit contraction planned by slice_plan.
ltgw_status slice_run(ltgw_ctx *ctx, SliceGemmArgs &g, double *part, cudaStream_t s) {
  g.err = ctx->flags;
  g.partial = slice_gemm_piece(&g) ? part : nullptr;
  CHECK_LAUNCH(ctx, launch_slice_gemm(g, ctx->n_sm, s), g.partial || (g.sym && g.mirror) ? 2 : 1);
  return LTGW_OK;
}

// Matrices in a piece of kSliceHold bytes, `each` per matrix.
int planned_piece(int n, size_t each, size_t shared) {
  int blk = n;
  while (shared + blk * each > kSliceHold && next_piece(n, &blk)) {}
  return blk;
}

// The plan of a product (M, N, nkb, sym, matrices of a piece): its K splits hold
// for every piece.
SliceGemmArgs slice_plan(int n_sm, int M, int N, int nkb, int sym, int batch, SliceForm f) {
  SliceGemmArgs g;
  g.ns = f.ns; g.bits = f.bits;
  g.M = M; g.N = N; g.nkb = nkb; g.sym = sym; g.batch = batch;
  slice_gemm_plan(&g, n_sm, kSlicePartialMax);
  return g;
}
// Bytes of its partials for a piece of `batch` matrices and M columns.
size_t slice_partial(SliceGemmArgs g, int batch, int M) {
  g.batch = batch; g.M = M;
  return slice_gemm_piece(&g);
}

// Chunk of the contraction length so that `rows` operand rows stay within
// kSliceTermMax (the emulated forms' exponents belong to whole rows: one chunk).
int64_t slice_k_chunk(int64_t rows, int64_t K, SliceForm f) {
  if (f.required) return K;
  const int64_t per_k = slice_rows_padded(rows) * 2 * f.ns;
  const int64_t most = std::max<int64_t>(2048, (int64_t)kSliceTermMax / per_k);
  const int64_t n = (K + most - 1) / most;
  return std::min(K, ((K + n - 1) / n + 63) / 64 * 64);
}

struct SyrkPiece {   // C = X X^T: one pair chunk
  SliceForm f;
  int n;
  int64_t chunk;
  SliceGemmArgs plan;
  SliceOperand o;
  double *part = nullptr;
  SyrkPiece(int n_sm, int n_, int64_t K, SliceForm f_) : f(f_), n(n_), chunk(slice_k_chunk(n_, K, f_)) {
    plan = slice_plan(n_sm, n, n, slice_blocks(chunk), 1, 1, f);
  }
  void layout(Arena &A) { o.layout(A, n, chunk, 1, f); }
  size_t partial() const { return slice_partial(plan, 1, n); }
  bool shrink() { return false; }
};

// C = beta C + X X^T (full, symmetric bit for bit), X [n][ld] with K columns.
// *done is false when the product was left to the caller (no memory).
ltgw_status slice_syrk(ltgw_ctx *ctx, int n, int64_t K, const double *X, int64_t ld, double *C, double beta,
                       SliceForm f, cudaStream_t s, bool *done) {
  SyrkPiece p(ctx->n_sm, n, K, f);
  *done = slice_fit(ctx, f.required, p);
  if (!*done) return ctx->status();
  for (int64_t k0 = 0; k0 < K; k0 += p.chunk) {
    const int64_t kc = std::min(p.chunk, K - k0);
    CHECK_LAUNCH(ctx, launch_slice_operand(p.o.source(X + k0, ld, 0, n, kc, false), f.ns, f.bits, 1, s), 3);
    SliceGemmArgs g = p.plan;
    g.A = g.B = p.o.dig; g.ea = g.eb = p.o.exps; g.C = C; g.ldc = n; g.beta = k0 ? 1.0 : beta;
    if (slice_run(ctx, g, p.part, s) != LTGW_OK) return ctx->status();
  }
  return LTGW_OK;
}

struct ProjectPiece {   // some of the matrices X_b, or some columns of one
  SliceForm f;
  int N, n_aux, batch, nb;
  int64_t chunk;
  SliceGemmArgs plan;
  SliceOperand u, x;
  double *part = nullptr;
  ProjectPiece(int n_sm, int N_, int n_aux_, int64_t cols, int batch_, SliceForm f_)
      : f(f_), N(N_), n_aux(n_aux_), batch(batch_), nb(batch_), chunk(cols) {
    const int nkb = slice_blocks(n_aux);
    plan = slice_plan(n_sm, (int)cols, N, nkb, 0, planned_piece(batch, slice_digit_bytes(cols, nkb, f.ns), 0), f);
  }
  void layout(Arena &A) {
    u.layout(A, N, n_aux, 1, f);
    x.layout(A, chunk, n_aux, nb, f);
  }
  size_t partial() const { return slice_partial(plan, nb, (int)chunk); }
  bool shrink() { return next_piece(batch, &nb) || next_columns(&chunk); }
};

// out_b [N][ld_out] = Ut X_b for the columns of X_b [n_aux][ld] (Ut rows [N][n_aux]).
ltgw_status slice_project(ltgw_ctx *ctx, int N, int n_aux, const double *Ut, const double *X, int64_t ld,
                          int64_t x_batch, int64_t cols, int batch, double *out, int64_t ld_out, int64_t out_batch,
                          SliceForm f, cudaStream_t s, bool *done) {
  ProjectPiece p(ctx->n_sm, N, n_aux, cols, batch, f);
  *done = slice_fit(ctx, f.required, p);
  if (!*done) return ctx->status();
  const SliceOperand &u = p.u, &x = p.x;
  CHECK_LAUNCH(ctx, launch_slice_operand(u.source(Ut, n_aux, 0, N, n_aux, false), f.ns, f.bits, 1, s), 3);
  for (int t0 = 0; t0 < batch; t0 += p.nb) {
    for (int64_t c0 = 0; c0 < cols; c0 += p.chunk) {
      const int cc = (int)std::min(p.chunk, cols - c0), bb = std::min(p.nb, batch - t0);
      CHECK_LAUNCH(ctx, launch_slice_operand(x.source(X + t0 * x_batch + c0, ld, x_batch, cc, n_aux, true), f.ns,
                                             f.bits, bb, s), 3);
      SliceGemmArgs g = p.plan;
      g.A = x.dig; g.a_batch = x.dig_batch; g.ea = x.exps; g.ea_batch = x.rows_p;
      g.B = u.dig; g.eb = u.exps; g.batch = bb; g.M = cc;
      g.C = out + t0 * out_batch + c0; g.ldc = ld_out; g.c_batch = out_batch;
      if (slice_run(ctx, g, p.part, s) != LTGW_OK) return ctx->status();
    }
  }
  return LTGW_OK;
}

struct WnmPiece {   // some frequencies, then some targets, then some columns of one
  SliceForm f;
  int N, n_omega, T, blk, tb;
  int64_t cc;
  SliceOperand r, c;
  double *cd = nullptr, *part = nullptr;   // the column dot takes no K splits
  WnmPiece(int N_, int n_omega_, int T_, int cols, SliceForm f_)
      : f(f_), N(N_), n_omega(n_omega_), T(T_), blk(n_omega_), tb(T_), cc(cols) {}
  void layout(Arena &A) {
    r.layout(A, tb * cc, N, 1, f);
    c.layout(A, N, N, blk, f);
    cd = A.take<double>((size_t)blk * 4 * ((N + 63) / 64) * tb * cc);
  }
  size_t partial() const { return 0; }
  bool shrink() { return next_piece(n_omega, &blk) || next_piece(T, &tb) || next_columns(&cc); }
};

// W_j[t][c] = sum_PQ Btt[t][P][c] C_j[P][Q] Btt[t][Q][c] (Eq. ScreenedCoulombOrbital)
// with the column dot in the contraction's epilogue; pieces of frequencies,
// then of targets, then of one target's columns.
ltgw_status slice_wnm(ltgw_ctx *ctx, int N, int n_omega, const double *C, int T, int n_orb_act, const double *Btt,
                      int64_t ld_btt, int64_t stride_btt, double *W, SliceForm f, cudaStream_t s, bool *done) {
  const int cols = T * n_orb_act;
  WnmPiece p(N, n_omega, T, n_orb_act, f);
  *done = slice_fit(ctx, f.required, p);
  if (!*done) return ctx->status();
  const SliceOperand &r = p.r, &c = p.c;
  const int blk = p.blk, tb = p.tb;
  const int64_t cc = p.cc;
  for (int t0 = 0; t0 < T; t0 += tb)
    for (int64_t c0 = 0; c0 < n_orb_act; c0 += cc) {
      const int nc = (int)std::min<int64_t>(cc, n_orb_act - c0), m = std::min(tb, T - t0) * nc;
      const double *B = Btt + t0 * stride_btt + c0;
      SliceSrc rs = r.source(B, ld_btt, 0, m, N, true);
      rs.col_group = nc; rs.col_stride = stride_btt;
      CHECK_LAUNCH(ctx, launch_slice_operand(rs, f.ns, f.bits, 1, s), 3);
      for (int j0 = 0; j0 < n_omega; j0 += blk) {
        const int nb = std::min(blk, n_omega - j0);
        CHECK_LAUNCH(ctx, launch_slice_operand(c.source(C + (int64_t)j0 * N * N, N, (int64_t)N * N, N, N, false), f.ns,
                                               f.bits, nb, s), 3);
        SliceGemmArgs g;
        g.A = r.dig; g.ea = r.exps;
        g.B = c.dig; g.b_batch = c.dig_batch; g.eb = c.exps; g.eb_batch = c.rows_p;
        g.ns = f.ns; g.bits = f.bits; g.nkb = r.nkb; g.batch = nb; g.M = m; g.N = N;
        g.cd_B = B; g.cd_ld = ld_btt; g.cd_stride = stride_btt; g.cd_cols = nc; g.cd_out = p.cd; g.cd_ldo = m;
        slice_gemm_plan(&g, ctx->n_sm, 0);
        if (slice_run(ctx, g, nullptr, s) != LTGW_OK) return ctx->status();
        CHECK_LAUNCH(ctx, launch_slice_coldot_reduce(g, W + (int64_t)j0 * cols + (int64_t)t0 * n_orb_act + c0, cols, s), 1);
      }
    }
  return LTGW_OK;
}

struct PiPiece {   // some of the factor rows, one pair chunk
  SliceForm f;
  int N, n_t, blk;
  int64_t chunk;
  SliceGemmArgs plan;
  SliceOperand o, o2;   // o2: the unsigned operand, written and read only where some factor is negative
  double *fac = nullptr, *part = nullptr;
  int *neg = nullptr;
  PiPiece(int n_sm, int N_, int64_t n_pairs, int n_t_, SliceForm f_)
      : f(f_), N(N_), n_t(n_t_), blk(n_t_), chunk(slice_k_chunk(2 * slice_rows_padded(N_), n_pairs, f_)) {
    const int nkb = slice_blocks(chunk);
    plan = slice_plan(n_sm, N, N, nkb, 1, planned_piece(n_t, 2 * slice_digit_bytes(N, nkb, f.ns), 0), f);
  }
  void layout(Arena &A) {
    o.layout(A, N, chunk, blk, f);
    o2.layout(A, N, chunk, blk, f);
    fac = A.take<double>((size_t)n_t * 2 * chunk);
    neg = A.take<int>(1);
  }
  size_t partial() const { return slice_partial(plan, blk, N); }
  bool shrink() { return next_piece(n_t, &blk); }
};

// M_t = alpha (Bt diag(f_t)) Bt^T for t < n_t (full, symmetric).  Both operands
// are Bt diag(sqrt |f_t|), the sign of f_t with the first one: an entry's error
// then follows the pairs that carry it, also where a factor singles out few of
// them (a factor on one side only would weigh that side's rounding with every
// pair of the other).  Entries whose terms are all small beside their rows' largest
// ones (rows that are large on different pairs) would still lose bits to the
// rows' common scales: with `entries` these are found and summed in FP64 (pi_weak.cu).
ltgw_status slice_pi(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, int64_t ldb, const double *delta,
                     int n_t, const double *p0, const double *p1, int mode, int alpha_exp, int alpha_neg, double *M,
                     bool entries, SliceForm f, cudaStream_t s, bool *done) {
  PiPiece p(ctx->n_sm, N, n_pairs, n_t, f);
  *done = slice_fit(ctx, f.required, p);
  if (!*done) return ctx->status();
  const SliceOperand &o = p.o, &o2 = p.o2;
  double *const fac = p.fac;
  int *const neg = p.neg;
  const int64_t chunk = p.chunk;
  const int blk = p.blk;
  for (int64_t k0 = 0; k0 < n_pairs; k0 += chunk) {
    const int64_t kc = std::min(chunk, n_pairs - k0);
    LTGW_CUDA(ctx, cudaMemsetAsync(neg, 0, sizeof(int), s));
    CHECK_LAUNCH(ctx, launch_pi_root_factor(delta + k0, kc, n_t, p0, p1, mode, fac, fac + (int64_t)n_t * kc, neg, s), 1);
    for (int t0 = 0; t0 < n_t; t0 += blk) {
      const int nb = std::min(blk, n_t - t0);
      SliceSrc a = o.source(Bt + k0, ldb, 0, N, kc, false);
      a.colscale = fac + (int64_t)t0 * kc; a.cs_batch = kc;
      CHECK_LAUNCH(ctx, launch_slice_operand(a, f.ns, f.bits, nb, s), 3);
      SliceSrc b = o2.source(Bt + k0, ldb, 0, N, kc, false);
      b.colscale = fac + (int64_t)(n_t + t0) * kc; b.cs_batch = kc; b.only_if = neg;
      CHECK_LAUNCH(ctx, launch_slice_operand(b, f.ns, f.bits, nb, s), 3);
      SliceGemmArgs g = p.plan;
      g.A = g.B = o.dig; g.a_batch = g.b_batch = o.dig_batch; g.ea = g.eb = o.exps; g.ea_batch = g.eb_batch = o.rows_p;
      g.B_alt = o2.dig; g.b_sel = neg;   // |sqrt| rows have the same exponents
      g.batch = nb;
      g.C = M + (int64_t)t0 * N * N; g.ldc = N; g.c_batch = (int64_t)N * N;
      g.beta = k0 ? 1.0 : 0.0; g.alpha_exp = alpha_exp; g.alpha_neg = alpha_neg;
      if (slice_run(ctx, g, p.part, s) != LTGW_OK) return ctx->status();
      if (!entries) continue;
      PiWeakArgs w;   // a chunk's weak entries: the sum so far
      w.dig = o.dig; w.dig_batch = o.dig_batch; w.exps = o.exps; w.exp_batch = o.rows_p; w.nkb = o.nkb;
      w.N = N; w.mode = mode; w.K = k0 + kc; w.X = Bt; w.ld = ldb;
      w.delta = delta; w.p0 = p0 + t0; w.p1 = p1 ? p1 + t0 : nullptr;
      if (k0 == 0) { w.sgn = a.colscale; w.mag = b.colscale; w.f_batch = kc; }
      w.alpha = ldexp(alpha_neg ? -1.0 : 1.0, alpha_exp); w.C = g.C;
      CHECK_LAUNCH(ctx, launch_pi_weak(w, nb, s), 1);
    }
  }
  return LTGW_OK;
}

struct GemmPiece {   // the whole product
  SliceForm f;
  int m, n;
  int64_t K;
  SliceGemmArgs plan;
  SliceOperand a, b;
  double *part = nullptr;
  GemmPiece(int n_sm, int m_, int n_, int64_t K_, SliceForm f_) : f(f_), m(m_), n(n_), K(K_) {
    plan = slice_plan(n_sm, n, m, slice_blocks(K), 0, 1, f);
  }
  void layout(Arena &A) {
    a.layout(A, m, K, 1, f);
    b.layout(A, n, K, 1, f);
  }
  size_t partial() const { return slice_partial(plan, 1, n); }
  bool shrink() { return false; }
};

// C [m][ldc] = A B^T from slices (sym: C = A A^T, whole).
ltgw_status emu_gemm(ltgw_ctx *ctx, int m, int n, int64_t K, const double *A, int64_t lda, const double *B,
                     int64_t ldb, double *C, int64_t ldc, bool sym, SliceForm f, cudaStream_t s) {
  bool done = false;
  if (sym) return slice_syrk(ctx, m, K, A, lda, C, 0.0, f, s, &done);
  GemmPiece p(ctx->n_sm, m, n, K, f);
  if (!slice_fit(ctx, f.required, p)) return ctx->status();
  const SliceOperand &a = p.a, &b = p.b;
  CHECK_LAUNCH(ctx, launch_slice_operand(a.source(A, lda, 0, m, K, false), f.ns, f.bits, 1, s), 3);
  CHECK_LAUNCH(ctx, launch_slice_operand(b.source(B, ldb, 0, n, K, false), f.ns, f.bits, 1, s), 3);
  SliceGemmArgs g = p.plan;   // the contiguous dimension of C is B's rows
  g.A = b.dig; g.ea = b.exps; g.B = a.dig; g.eb = a.exps; g.C = C; g.ldc = ldc;
  return slice_run(ctx, g, p.part, s);
}

struct PiEmuPiece {   // some of the factor rows, one chunk of at most 131072 pairs
  SliceForm f;
  int N, n_t, blk;
  int64_t chunk;
  SliceGemmArgs plan;
  SliceOperand a, b;
  double *fac = nullptr, *part = nullptr;
  PiEmuPiece(int n_sm, int N_, int64_t n_pairs, int n_t_, SliceForm f_) : f(f_), N(N_), n_t(n_t_), blk(n_t_) {
    const int64_t max_chunk = (int64_t)1 << 17, n_chunks = (n_pairs + max_chunk - 1) / max_chunk;
    chunk = std::min(n_pairs, ((n_pairs + n_chunks - 1) / n_chunks + 63) / 64 * 64);   // balanced
    const int nkb = slice_blocks(chunk);
    const size_t each = slice_digit_bytes(N, nkb, f.ns);
    plan = slice_plan(n_sm, N, N, nkb, 1, planned_piece(n_t, each, each), f);
  }
  void layout(Arena &A) {
    a.layout(A, N, chunk, blk, f);
    b.layout(A, N, chunk, 1, f);
    fac = A.take<double>((size_t)n_t * chunk);
  }
  size_t partial() const { return slice_partial(plan, blk, N); }
  bool shrink() { return next_piece(n_t, &blk); }
};

// Pi from slices (the emulated FP64 form): per frequency (n_tau == 0, Pi_j =
// -2 s M_j written directly) or moment t (lt_form 1: Laplace factors; 2:
// e^{-Delta tau_t}) M_t = (Bt diag(f_t)) Bt^T, the lower triangle (rows scaled)
// mirrored, then the recombination with d_E [n_omega][n_tau].  Pairs in equal
// chunks of at most 131072, each with its own row exponents, their products added.
ltgw_status polarizability_emu(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, int64_t ldb,
                               const double *delta, int n_omega, const double *d_om, int n_tau, const double *d_x,
                               const double *d_w, const double *d_E, double *d_M, int spin, double *Pi,
                               cudaStream_t s, int lt_form, SliceForm f) {
  const int n_t = n_tau ? n_tau : n_omega;
  PiEmuPiece p(ctx->n_sm, N, n_pairs, n_t, f);
  if (!slice_fit(ctx, f.required, p)) return ctx->status();
  const SliceOperand &a = p.a, &b = p.b;
  double *const fac = p.fac;
  const int64_t chunk = p.chunk;
  const int blk = p.blk;
  ctx->mark(EV_PI0, s);
  const int mode = n_tau ? (lt_form == 2 ? SCALE_EXPTAU : SCALE_LAPLACE) : SCALE_DIRECT;
  double *out = n_tau ? d_M : Pi;
  for (int64_t k0 = 0; k0 < n_pairs; k0 += chunk) {
    const int64_t kc = std::min(chunk, n_pairs - k0);
    CHECK_LAUNCH(ctx, launch_pi_factor64(delta + k0, kc, n_t, n_tau ? d_x : d_om,
                                         mode == SCALE_LAPLACE ? d_w : nullptr, mode, fac, s), 1);
    CHECK_LAUNCH(ctx, launch_slice_operand(b.source(Bt + k0, ldb, 0, N, kc, false), f.ns, f.bits, 1, s), 3);
    for (int t0 = 0; t0 < n_t; t0 += blk) {
      const int nb = std::min(blk, n_t - t0);
      SliceSrc sa = a.source(Bt + k0, ldb, 0, N, kc, false);
      sa.colscale = fac + (int64_t)t0 * kc; sa.cs_batch = kc;
      CHECK_LAUNCH(ctx, launch_slice_operand(sa, f.ns, f.bits, nb, s), 3);
      SliceGemmArgs g = p.plan;
      g.A = a.dig; g.a_batch = a.dig_batch; g.ea = a.exps; g.ea_batch = a.rows_p;
      g.B = b.dig; g.eb = b.exps; g.batch = nb; g.C = out + (int64_t)t0 * N * N; g.ldc = N; g.c_batch = (int64_t)N * N;
      g.beta = k0 ? 1.0 : 0.0; g.alpha_exp = n_tau ? 0 : spin; g.alpha_neg = n_tau ? 0 : 1;   // -2 s: -2 or -4
      if (slice_run(ctx, g, p.part, s) != LTGW_OK) return ctx->status();
    }
  }
  ctx->mark(EV_PI1, s);
  if (n_tau)
    CHECK_LAUNCH(ctx, launch_recombine(d_M, n_tau, d_E, n_omega, (int64_t)N * N, -2.0 * spin, Pi, s),
                 (n_omega + 63) / 64);
  return LTGW_OK;
}

// K builder for the streamed solve: fills w.A (n x n) itself.
using KBuilder = std::function<ltgw_status(double *K)>;

ltgw_status naf_basis_dev(ltgw_ctx *ctx, Arena &ar, int n, int64_t n_pairs, const double *B,
                          int64_t ld, double thresh, double *Ut, double *lam_out, int *k_out,
                          int *near_out, cudaStream_t s, bool mixed = false, const KBuilder *build_K = nullptr,
                          int emu_slices = 0) {
  EigWork w;
  auto layout = [&](Arena &A) {
    w.A = A.take<double>((size_t)n * n);
    w.V = A.take<double>((size_t)(n + 64) * n);   // 64 zero rows past the last reflector (compact-WY blocks)
    w.d = A.take<double>(n);
    w.e = A.take<double>(n);
    w.tau = A.take<double>(n);
    w.p = A.take<double>(n);
    w.w = A.take<double>(n);
    w.scal = A.take<double>(8);
    w.lam = A.take<double>(n);
    w.X = A.take<double>((size_t)n * n);
    w.lu = A.take<double>((size_t)5 * n * n);
    w.count = A.take<int>(2);
    const int64_t nsplit = (n + 63) / 64, nblk = (n + 63) / 64;
    // compact-WY scratch: W1 and its partials (block-at-a-time form: split
    // partials of 64 x n and W1 64 x n; cooperative form: one 64 x 64 partial
    // per CTA and one W1 per 64-column slice), every block's G and T, and
    // every block's M_b (before the T recurrences: the split partials of G)
    w.wy_r0 = (int64_t)std::max((size_t)nsplit * 64 * (size_t)n + 64 * (size_t)n,
                                ((size_t)ctx->n_sm + (size_t)nsplit) * 64 * 64);
    w.wy = A.take<double>((size_t)w.wy_r0 + 2 * (size_t)nblk * 64 * 64 +
                          (size_t)nblk * std::max((size_t)n * 64, (size_t)nsplit * 64 * 64));
    w.grid_ws = A.take<double>((size_t)4 * n + 2 * (size_t)ctx->n_sm + 8);
  };
  ar.begin_sizing();
  layout(ar);
  if (ar.commit() != cudaSuccess) {
    ctx->fail(LTGW_ERR_NOMEM, "NAF workspace allocation failed");
    return ctx->status();
  }
  layout(ar);
  w.flags = ctx->flags;
  ctx->mark(EV_K0, s);
  if (build_K) {
    if ((*build_K)(w.A) != LTGW_OK) return ctx->status();
  } else if (mixed) {
    if (naf_metric_tc(ctx, n, n_pairs, B, ld, w.A, s) != LTGW_OK) return ctx->status();
  } else if (emu_slices) {
    if (emu_gemm(ctx, n, n, n_pairs, B, ld, B, ld, w.A, n, true, emu_digits(emu_slices), s) != LTGW_OK) return ctx->status();
  } else {
    bool done = false;
    if (slices_pay(n, n, n_pairs, 1) && slice_syrk(ctx, n, n_pairs, B, ld, w.A, 0.0, kFp64Digits, s, &done) != LTGW_OK)
      return ctx->status();
    if (!done) {
      GemmF64Args g;
      g.M = n; g.N = n; g.K = n_pairs;
      g.A = B; g.lda = ld; g.B = B; g.ldb = ld;
      g.C = w.A; g.ldc = n;
      g.syrk = 1;
      CHECK_LAUNCH(ctx, launch_gemm_f64(g, 1, true, true, s), 1);
    }
  }
  LTGW_CUDA(ctx, cudaMemsetAsync(w.V, 0, (size_t)(n + 64) * n * sizeof(double), s));
  int nl = 0;
  ctx->mark(EV_TRI0, s);
  cudaError_t e = launch_eig_tridiag(w, n, thresh, s, &nl);
  ctx->mark(EV_TRI1, s);
  ctx->tri_n = n;
  ctx->launches += nl;
  if (e != cudaSuccess) { ctx->fail(LTGW_ERR_DEVICE, std::string("eig_tridiag: ") + cudaGetErrorString(e)); return ctx->status(); }
  int cnt[2] = {0, 0};
  if (read_small(ctx, cnt, w.count, sizeof(cnt), s) != LTGW_OK) return ctx->status();
  const int k = cnt[0];
  *k_out = k;
  if (near_out) *near_out = cnt[1];
  if (k <= 0) { ctx->fail(LTGW_ERR_NO_NAF, "NAF threshold kept no auxiliary function"); return ctx->status(); }
  nl = 0;
  e = launch_eig_vectors(w, n, k, Ut, ctx->flags, s, &nl);
  ctx->mark(EV_VEC1, s);
  ctx->launches += nl;
  if (e != cudaSuccess) { ctx->fail(LTGW_ERR_DEVICE, std::string("eig_vectors: ") + cudaGetErrorString(e)); return ctx->status(); }
  if (lam_out) LTGW_CUDA(ctx, cudaMemcpyAsync(lam_out, w.lam, (size_t)k * sizeof(double), cudaMemcpyDeviceToDevice, s));
  return LTGW_OK;
}

// Pi at the GL frequencies, direct (n_tau == 0) or through moments M^k and the
// recombination d_E [n_omega][n_tau]: lt_form 1 = the M^m form of Eq. LT
// (factors w_m Delta e^{-Delta^2 x_m}), 2 = imaginary time (factors e^{-Delta tau_k},
// tau_k in d_x).  entries: Pi itself is the result, each entry to an FP64 sum's
// accuracy; within a solve it is summed over, and the rows' scales are enough.
ltgw_status polarizability_dev(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, int64_t ldb,
                               const double *delta, int n_omega, const double *d_omega,
                               int n_tau, const double *d_x, const double *d_w, const double *d_E,
                               double *M, int spin, double *Pi, cudaStream_t s, int lt_form, bool entries) {
  const int mode = n_tau == 0 ? SCALE_DIRECT : (lt_form == 2 ? SCALE_EXPTAU : SCALE_LAPLACE);
  const int n_t = n_tau ? n_tau : n_omega;
  const double *p0 = n_tau ? d_x : d_omega, *p1 = mode == SCALE_LAPLACE ? d_w : nullptr;
  double *out = n_tau ? M : Pi;
  ctx->mark(EV_PI0, s);
  bool done = false;
  // alpha: 1 for the moments, -2 spin = -2 or -4 for Pi itself
  if (slices_pay(N, N, n_pairs, n_t) &&
      slice_pi(ctx, N, n_pairs, Bt, ldb, delta, n_t, p0, p1, mode, n_tau ? 0 : spin, n_tau ? 0 : 1, out, entries,
               kFp64Digits, s, &done) != LTGW_OK)
    return ctx->status();
  if (!done) {
    GemmF64Args g;
    g.M = N; g.N = N; g.K = n_pairs;
    g.A = Bt; g.lda = ldb; g.B = Bt; g.ldb = ldb;
    g.ldc = N; g.strideC = (int64_t)N * N;
    g.syrk = 1;
    g.delta = delta;
    g.C = out;
    g.alpha = n_tau ? 1.0 : -2.0 * spin;
    g.scale_mode = mode;
    g.batch_p0 = p0;
    g.batch_p1 = p1;
    CHECK_LAUNCH(ctx, launch_gemm_f64(g, n_t, true, true, s), 1);
  }
  ctx->mark(EV_PI1, s);
  if (n_tau)
    CHECK_LAUNCH(ctx, launch_recombine(M, n_tau, d_E, n_omega, (int64_t)N * N, -2.0 * spin, Pi, s),
                 (n_omega + 63) / 64);
  return LTGW_OK;
}

// Split-K plan: one CTA per SM, so choose the split count that fills whole
// waves best while keeping at least 1024 pairs per CTA.
// K-split count for a tensor-core contraction of `units` output tiles x groups:
// the CTAs of one wave run in lockstep, so the time is about waves x (per-CTA
// overhead + K chunks per CTA); the overhead (TMEM and barrier setup, pipeline
// fill, draining the accumulators) costs about as much as ten 64-pair chunks.
// At least Kp / drain_k splits (up to 64) keep each CTA to one FP32 drain; the
// split length is a multiple of `align` pairs.
int64_t tc_splits(const ltgw_ctx *ctx, int64_t units, int64_t Kp, int64_t drain_k, int64_t align, int64_t *kps_out) {
  const int64_t max_split = std::min<int64_t>(64, std::max<int64_t>(1, Kp / 1024));
  const int64_t min_split = std::min<int64_t>(max_split, (Kp + drain_k - 1) / drain_k);
  const int64_t nchunk = Kp / 64;
  int64_t splits = min_split;
  double best = 1e300;
  for (int64_t sp = min_split; sp <= max_split; ++sp) {
    const int64_t waves = (units * sp + ctx->n_sm - 1) / ctx->n_sm;
    const double cost = (double)waves * (10.0 + (double)((nchunk + sp - 1) / sp));
    if (cost < best) { best = cost; splits = sp; }   // fewer splits on ties
  }
  int64_t kps = ((Kp + splits - 1) / splits + align - 1) / align * align;
  *kps_out = kps;
  return (Kp + kps - 1) / kps;
}

std::vector<int> lower_tiles(int nI, std::vector<int> *tindex) {
  std::vector<int> tiles;
  if (tindex) tindex->assign((size_t)nI * nI, -1);
  for (int I = 0; I < nI; ++I)
    for (int J = 0; J <= I; ++J) {
      if (tindex) (*tindex)[(size_t)I * nI + J] = (int)(tiles.size() / 2);
      tiles.push_back(I);
      tiles.push_back(J);
    }
  return tiles;
}

std::vector<int> full_tiles(int nI, int nJ) {
  std::vector<int> tiles;
  for (int I = 0; I < nI; ++I)
    for (int J = 0; J < nJ; ++J) { tiles.push_back(I); tiles.push_back(J); }
  return tiles;
}

// One split-BF16 contraction on the tensor cores.  Scratch (tile list,
// partials) comes from `ar`; the caller reduces the partials (returned).
struct TcRun {
  double *partial = nullptr;
  float *partial32 = nullptr;
  float *cd_out = nullptr;
  int splits = 1, groups = 1, n_tiles = 0, nt_group = 1;
};

// One configuration of a contraction: scales per CTA, K-split length, output precision.
struct TcPlan {
  int nt_group, groups;
  int64_t splits, kps;
  int out_mode;
};

TcPlan tc_plan(const ltgw_ctx *ctx, const TcGemmArgs &g, int n_tiles, int nt_group, int64_t want_splits) {
  TcPlan p;
  p.nt_group = nt_group;
  p.groups = (g.n_t + nt_group - 1) / nt_group;
  const int64_t align = g.A8 ? 128 : 64;
  const int64_t klen = (g.k_end ? g.k_end : g.Kp) - g.k_begin;   // pairs contracted
  if (g.out_mode == TC_OUT_COLDOT) {
    // the column dot needs the whole contraction (K = the NAF count) in one drain
    p.kps = klen; p.splits = 1; p.out_mode = TC_OUT_COLDOT;
    return p;
  }
  if (want_splits > 0) {
    p.kps = ((klen + want_splits - 1) / want_splits + align - 1) / align * align;
    p.splits = (klen + p.kps - 1) / p.kps;
  } else {
    p.splits = tc_splits(ctx, (int64_t)n_tiles * p.groups, klen, g.drain_k, align, &p.kps);
  }
  p.out_mode = p.kps <= g.drain_k ? TC_OUT_F32 : TC_OUT_F64;
  return p;
}

// Run a contraction.  Scratch (tile list, partials) comes from `ar`; the
// caller reduces the partials (returned with the configuration used).  With
// the autotuner on, the first contraction of a shape times its candidate
// configurations (scales per CTA where the kernel and the caller's reduction
// allow several; the heuristic's K-split count, half and twice it, each
// keeping one FP32 drain per CTA where one can) with CUDA events on the
// stream, keeps the fastest for this context and then runs it.
ltgw_status tc_run(ltgw_ctx *ctx, Arena &ar, TcGemmArgs g, const std::vector<int> &tiles, int coldot_rows,
                   TcRun *run, cudaStream_t s) {
  const int n_tiles = (int)(tiles.size() / 2);
  if (g.out_mode == TC_OUT_COLDOT) g.drain_k = std::max<int64_t>(g.drain_k, (g.k_end ? g.k_end : g.Kp) - g.k_begin);
  const int kind = g.A8 ? 2 : (g.B_hi ? 1 : 0);
  TcPlan plan = tc_plan(ctx, g, n_tiles, g.nt_group, 0);
  std::vector<TcPlan> cands{plan};
  const ltgw_ctx::TcKey key{kind, n_tiles, g.n_t, g.out_mode, (g.k_end ? g.k_end : g.Kp) - g.k_begin, g.rows_a,
                            g.rows_b};
  bool tune = false;
  if (ctx->autotune && g.out_mode != TC_OUT_COLDOT) {
    auto it = ctx->tuned.find(key);
    if (it != ctx->tuned.end()) {
      plan = tc_plan(ctx, g, n_tiles, it->second.nt_group, it->second.splits);
      cands = {plan};
    } else {
      tune = true;
      cands.clear();
      std::vector<int> ntgs{g.nt_group};
      // scales per CTA vary only where the caller reduces with reduce_sym (column-major partials)
      if (g.out_colmajor && g.n_t > 1 && kind == 1) ntgs = {2, 1};
      if (g.out_colmajor && g.n_t > 1 && kind == 2) ntgs = {4, 2, 1};
      const int64_t min_split = std::min<int64_t>(64, ((g.k_end ? g.k_end : g.Kp) - g.k_begin + g.drain_k - 1) / g.drain_k);
      for (int ntg : ntgs) {
        const TcPlan base = tc_plan(ctx, g, n_tiles, ntg, 0);
        for (int64_t sp : {base.splits, base.splits / 2, base.splits * 2}) {
          sp = std::max<int64_t>(std::max<int64_t>(sp, min_split), 1);
          const TcPlan c = tc_plan(ctx, g, n_tiles, ntg, sp);
          if (c.splits > 256) continue;
          bool dup = false;
          for (const TcPlan &o : cands) dup |= (o.nt_group == c.nt_group && o.splits == c.splits);
          if (!dup) cands.push_back(c);
        }
      }
    }
  }
  size_t part64_n = 0, part32_n = 0, cd_n = 0;
  for (const TcPlan &c : cands) {
    const size_t n_part = (size_t)c.splits * c.groups * c.nt_group * n_tiles * 128 * 128;
    if (c.out_mode == TC_OUT_F64) part64_n = std::max(part64_n, n_part);
    if (c.out_mode == TC_OUT_F32) part32_n = std::max(part32_n, n_part);
    if (c.out_mode == TC_OUT_COLDOT) cd_n = (size_t)c.splits * c.groups * coldot_rows * (size_t)g.cd_cols_p;
  }
  int *d_tiles;
  double *part64;
  float *part32, *cd;
  auto layout = [&](Arena &A) {
    d_tiles = A.take<int>(tiles.size());
    part64 = part64_n ? A.take<double>(part64_n) : nullptr;
    part32 = part32_n ? A.take<float>(part32_n) : nullptr;
    cd = cd_n ? A.take<float>(cd_n) : nullptr;
  };
  ar.begin_sizing();
  layout(ar);
  if (ar.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "tensor-core workspace allocation failed"); return ctx->status(); }
  layout(ar);
  copy_in(ctx, d_tiles, tiles.data(), tiles.size() * sizeof(int), s);
  g.tiles = d_tiles;
  g.n_tile_rows = coldot_rows;
  g.err = ctx->flags;
  auto launch = [&](const TcPlan &c) {
    TcGemmArgs h = g;
    h.nt_group = c.nt_group;
    h.k_per_split = c.kps;
    h.out_mode = c.out_mode;
    h.partial = c.out_mode == TC_OUT_F64 ? part64 : nullptr;
    h.partial32 = c.out_mode == TC_OUT_F32 ? part32 : nullptr;
    h.cd_out = c.out_mode == TC_OUT_COLDOT ? cd : nullptr;
    return h.A8 ? launch_tc_fp8_gemm(h, n_tiles, s) : launch_tc_split_gemm(h, n_tiles, s);
  };
  if (tune) {
    cudaEvent_t e0, e1;
    LTGW_CUDA(ctx, cudaEventCreate(&e0));
    LTGW_CUDA(ctx, cudaEventCreate(&e1));
    float best = 1e30f;
    for (const TcPlan &c : cands) {
      float ms = 0.0f;
      CHECK_LAUNCH(ctx, launch(c), 1);   // warm
      cudaEventRecord(e0, s);
      CHECK_LAUNCH(ctx, launch(c), 1);
      cudaEventRecord(e1, s);
      LTGW_CUDA(ctx, cudaEventSynchronize(e1));
      LTGW_CUDA(ctx, cudaEventElapsedTime(&ms, e0, e1));
      if (ms < best) { best = ms; plan = c; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    ctx->tuned[key] = ltgw_ctx::TcChoice{plan.nt_group, plan.splits};
  }
  ctx->stats.tc_autotuned = (int)ctx->tuned.size();
  CHECK_LAUNCH(ctx, launch(plan), 1);
  run->partial = plan.out_mode == TC_OUT_F64 ? part64 : nullptr;
  run->partial32 = plan.out_mode == TC_OUT_F32 ? part32 : nullptr;
  run->cd_out = plan.out_mode == TC_OUT_COLDOT ? cd : nullptr;
  run->splits = (int)plan.splits;
  run->groups = plan.groups;
  run->n_tiles = n_tiles;
  run->nt_group = plan.nt_group;
  return LTGW_OK;
}

// Pi (direct) or the Laplace moments M^k on the tensor cores, split-BF16 or
// (fp8) FP8 E4M3 with per-row scales.  Operand: Af (FP32
// [roundup(N,128)][roundup(n_pairs,64)]) when given, else converted from the
// FP64 block Bt.  Scale table: the per-pair factor of Eq. Pi or of the M^m
// form, applied by the converter warps (split-BF16) or before quantisation (FP8).
ltgw_status polarizability_tc(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, int64_t ldb,
                              const float *Af_in, const double *delta, int n_omega, const double *d_omega,
                              int n_tau, const double *d_x, const double *d_w, const double *d_E,
                              double *M, int spin, double *Pi, cudaStream_t s, bool fp8, int lt_form) {
  const int64_t Kp = (n_pairs + 63) / 64 * 64, Kq = (n_pairs + 127) / 128 * 128;
  const int nI = (N + 127) / 128, Mp = nI * 128;
  const int n_t = n_tau ? n_tau : n_omega;
  std::vector<int> tindex;
  std::vector<int> tiles = lower_tiles(nI, &tindex);
  float *Af = nullptr, *scale;
  __nv_bfloat16 *Bhi = nullptr, *Blo = nullptr;   // the unscaled operand, pre-split for the TMA-fed kernel
  uint8_t *qa = nullptr, *qb = nullptr;           // FP8 codes: scaled operands [n_t][Mp][3 Kq], B [Mp][3 Kq]
  float *ds_a = nullptr, *ds_b = nullptr;         // FP8 per-row de-scales
  int *maxima = nullptr;                          // FP8 per-row largest magnitudes
  int *d_tindex;
  auto layout = [&](Arena &A) {
    Af = Af_in ? nullptr : A.take<float>((size_t)Mp * Kp);
    scale = A.take<float>((size_t)n_t * Kp);
    if (fp8) {
      qa = A.take<uint8_t>((size_t)n_t * Mp * 3 * Kq);
      qb = A.take<uint8_t>((size_t)Mp * 3 * Kq);
      ds_a = A.take<float>((size_t)n_t * Mp);
      ds_b = A.take<float>((size_t)Mp);
      maxima = A.take<int>((size_t)(n_t + 1) * Mp);
    } else {
      Bhi = A.take<__nv_bfloat16>((size_t)Mp * Kp);
      Blo = A.take<__nv_bfloat16>((size_t)Mp * Kp);
    }
    d_tindex = A.take<int>(tindex.size());
  };
  ctx->a5.begin_sizing();
  layout(ctx->a5);
  if (ctx->a5.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "tensor-core operand allocation failed"); return ctx->status(); }
  layout(ctx->a5);
  const float *A = Af_in ? Af_in : Af;
  copy_in(ctx, d_tindex, tindex.data(), tindex.size() * sizeof(int), s);
  if (!Af_in) CHECK_LAUNCH(ctx, launch_to_f32_padded(Bt, ldb, N, n_pairs, Af, Mp, Kp, s), 1);
  const int mode = n_tau ? (lt_form == 2 ? SCALE_EXPTAU : SCALE_LAPLACE) : SCALE_DIRECT;
  CHECK_LAUNCH(ctx, launch_scale_table(delta, n_pairs, Kp, n_t, n_tau ? d_x : d_omega,
                                       mode == SCALE_LAPLACE ? d_w : nullptr, mode, scale, s), 1);
  TcGemmArgs g;
  if (fp8) {
    // two-term E4M3 expansions of both operands (three products over 3 Kq codes)
    CHECK_LAUNCH(ctx, launch_fp8_quantize(A, Kp, Kq, scale, n_t, Mp, qa, qb, ds_a, ds_b, maxima, s, 1), 2);
    // FP32 sums of exact E4M3 products: a 4096-code drain keeps the accumulation
    // bias (about 4e-6) below the expansion's rounding error
    g.A8 = qa; g.B8 = qb; g.ds_a = ds_a; g.ds_b = ds_b; g.Kp = 3 * Kq; g.nt_group = 2; g.drain_k = 4096;
  } else {
    CHECK_LAUNCH(ctx, launch_split_bf16(A, Bhi, Blo, (int64_t)Mp * Kp, s), 1);
    g.A = A; g.B = A; g.scale = scale; g.Kp = Kp; g.nt_group = 2; g.B_hi = Bhi; g.B_lo = Blo;
  }
  g.n_t = n_t; g.rows_a = Mp; g.rows_b = Mp; g.out_colmajor = 1;
  // Pairs go in blocks of at most 64 K-splits x drain_k (one FP32 drain per
  // CTA, partials bounded); each block's partials are added to Pi or M^k.
  TcRun run;
  const int64_t kblk = 64 * g.drain_k;
  ctx->mark(EV_PI0, s);
  for (int64_t k0 = 0; k0 < g.Kp; k0 += kblk) {
    TcGemmArgs gb = g;
    gb.k_begin = k0;
    gb.k_end = std::min(g.Kp, k0 + kblk);
    if (tc_run(ctx, ctx->a4, gb, tiles, 0, &run, s) != LTGW_OK) return ctx->status();
    if (gb.k_end == g.Kp) ctx->mark(EV_PI1, s);
    CHECK_LAUNCH(ctx, launch_tc_reduce_sym(run.partial, run.partial32, run.splits, run.groups, run.n_tiles, d_tindex,
                                           nI, n_t, N, n_tau ? 1.0 : -2.0 * spin, n_tau ? M : Pi, s,
                                           k0 ? 1.0 : 0.0, run.nt_group, 1), 1);
  }
  ctx->pi_tc_flops = (fp8 ? 1.0 : 3.0) * 2.0 * (double)run.n_tiles * 128 * 128 * (double)g.Kp * n_t;   // FP8: Kp = 3 Kq
  if (n_tau) {
    CHECK_LAUNCH(ctx, launch_recombine(M, n_tau, d_E, n_omega, (int64_t)N * N, -2.0 * spin, Pi, s, true),
                 (n_omega + 63) / 64);
  }
  return LTGW_OK;
}

// NAF metric K = B B^T (Eq. nafeq) in the split-BF16 form; K: device [n][n] FP64.
ltgw_status naf_metric_tc(ltgw_ctx *ctx, int n, int64_t n_pairs, const double *B, int64_t ld, double *K,
                          cudaStream_t s, double beta) {
  const int64_t Kp = (n_pairs + 63) / 64 * 64;
  const int nI = (n + 127) / 128, Mp = nI * 128;
  std::vector<int> tindex;
  std::vector<int> tiles = lower_tiles(nI, &tindex);
  float *Af, *ones;
  __nv_bfloat16 *Bhi, *Blo;   // the operand pre-split for the TMA-fed kernel
  int *d_tindex;
  auto layout = [&](Arena &A) {
    Af = A.take<float>((size_t)Mp * Kp);
    ones = A.take<float>((size_t)Kp);
    Bhi = A.take<__nv_bfloat16>((size_t)Mp * Kp);
    Blo = A.take<__nv_bfloat16>((size_t)Mp * Kp);
    d_tindex = A.take<int>(tindex.size());
  };
  ctx->a5.begin_sizing();
  layout(ctx->a5);
  if (ctx->a5.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "tensor-core operand allocation failed"); return ctx->status(); }
  layout(ctx->a5);
  copy_in(ctx, d_tindex, tindex.data(), tindex.size() * sizeof(int), s);
  CHECK_LAUNCH(ctx, launch_to_f32_padded(B, ld, n, n_pairs, Af, Mp, Kp, s), 1);
  CHECK_LAUNCH(ctx, launch_scale_table(nullptr, n_pairs, Kp, 1, nullptr, nullptr, SCALE_NONE, ones, s), 1);
  CHECK_LAUNCH(ctx, launch_split_bf16(Af, Bhi, Blo, (int64_t)Mp * Kp, s), 1);
  TcGemmArgs g;
  g.A = Af; g.B = Af; g.scale = ones; g.Kp = Kp; g.n_t = 1; g.nt_group = 1;
  g.B_hi = Bhi; g.B_lo = Blo; g.rows_a = Mp; g.rows_b = Mp; g.out_colmajor = 1;
  TcRun run;
  if (tc_run(ctx, ctx->a4, g, tiles, 0, &run, s) != LTGW_OK) return ctx->status();
  CHECK_LAUNCH(ctx, launch_tc_reduce_sym(run.partial, run.partial32, run.splits, run.groups, run.n_tiles, d_tindex,
                                         nI, 1, n, 1.0, K, s, beta, run.nt_group, 1), 1);
  return LTGW_OK;
}

// C_j = [1 - Pi_j]^-1 - 1 (Eq. ScreenedCoulombOrbital): the blocked sweep with
// its updates from digits where N is past one pivot block of 128 by more than a
// sliver (N = 130: 0.76 ms, FP64 tiles 0.56; N = 160: 0.59 against 0.85) and the
// digits of one frequency fit, else on the FP64 tiles.
constexpr int kScreenDigitsMinN = 144;

struct ScreenPiece {   // some of the frequencies
  int N, n_omega, blk;
  void *digits = nullptr;
  double *part = nullptr;
  ScreenPiece(int N_, int n_omega_) : N(N_), n_omega(n_omega_), blk(n_omega_) {}
  void layout(Arena &A) { digits = A.take<uint8_t>(screen_digit_bytes(N, blk)); }
  size_t partial() const { return 0; }
  bool shrink() { return next_piece(n_omega, &blk); }
};

// check: Pi comes from the caller; one that is not symmetric goes to the FP64 tiles,
// which read both triangles (the solves' own Pi is symmetric bit for bit).
ltgw_status screen_step(ltgw_ctx *ctx, int N, int n_omega, const double *Pi, double *work, double *C, cudaStream_t s,
                        bool check = false) {
  int nl = 0;
  ScreenPiece p(N, n_omega);
  const bool use = N >= kScreenDigitsMinN && N <= 65535 && n_omega <= 65535 && slice_fit(ctx, false, p);
  cudaError_t e = cudaSuccess;
  bool general = !use;
  if (use) {
    for (int j0 = 0; j0 < n_omega && e == cudaSuccess; j0 += p.blk)
      e = launch_screen_digits(Pi + (int64_t)j0 * N * N, N, std::min(p.blk, n_omega - j0), work, p.digits,
                               C + (int64_t)j0 * N * N, ctx->flags, ctx->n_sm,
                               check ? ctx->flags + FLAG_ASYM : nullptr, s, &nl);
    int asym = 0;
    if (check && e == cudaSuccess) {
      if (read_small(ctx, &asym, ctx->flags + FLAG_ASYM, sizeof(int), s) != LTGW_OK) return ctx->status();
      if (asym) LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
      general = asym != 0;
    }
  }
  if (general && e == cudaSuccess) e = launch_screen_blocked(Pi, N, n_omega, work, C, ctx->flags, s, &nl);
  ctx->launches += nl;
  if (e != cudaSuccess) ctx->fail(LTGW_ERR_DEVICE, std::string("screen: ") + cudaGetErrorString(e));
  return ctx->status();
}

// Operands of the mixed form after the NAF step (Eq. naftrafo in split BF16):
//   Bf       FP32 [roundup(N,128)][roundup(n_ov,64)]   R~_ov, the Pi operand
//   BtT64    FP64 [T][n_orb_act][N]                      R~_tgt transposed (column dot)
//   BtT32    FP32 [roundup(T n_orb_act,128)][roundup(N,64)]  the W_nm operand
// With Ut == nullptr (no NAF) they are copies of the active blocks of B_ov, B_tgt.
// With `window` set, only the ov part runs, for n_ov columns of B_act written
// into columns [col0, col0 + n_ov) of Bf (row stride ld_bf); padding is left
// to the caller.  With Bh_in / Bl_in set (and B_act NULL), the ov block comes
// already transposed and split: BF16 hi / lo [roundup(n_ov,128)][roundup(n_aux,64)].
struct OvWindow {
  int64_t col0 = 0, ld_bf = 0;
};

ltgw_status naf_project_tc(ltgw_ctx *ctx, int N, int n_aux, const double *Ut, const double *B_act, int64_t ld_act,
                           int64_t n_ov, const double *B_tgt, int n_orb, int n_fc, int T, int n_orb_act, float *Bf,
                           double *BtT64, float *BtT32, cudaStream_t s, const OvWindow *window = nullptr,
                           const __nv_bfloat16 *Bh_in = nullptr, const __nv_bfloat16 *Bl_in = nullptr) {
  const int64_t Kp_ov = (n_ov + 63) / 64 * 64;
  const int MpN = (N + 127) / 128 * 128, KpN = (N + 63) / 64 * 64;
  const int64_t rowsT = (int64_t)T * n_orb_act, rowsTp = (rowsT + 127) / 128 * 128;
  if (!Ut) {
    CHECK_LAUNCH(ctx, launch_to_f32_padded(B_act, ld_act, N, n_ov, Bf, MpN, Kp_ov, s), 1);
    CHECK_LAUNCH(ctx, launch_transpose_f64(B_tgt, n_orb, n_fc, n_aux, n_orb_act, BtT64, N, T,
                                           (int64_t)n_aux * n_orb, (int64_t)n_orb_act * N, s), 1);
    CHECK_LAUNCH(ctx, launch_to_f32_transposed(B_tgt, n_orb, n_fc, n_aux, n_orb_act, BtT32, KpN, n_orb_act, T,
                                               (int64_t)n_aux * n_orb, (int64_t)n_orb_act * KpN, s), 1);
    if (rowsTp > rowsT)
      LTGW_CUDA(ctx, cudaMemsetAsync(BtT32 + rowsT * KpN, 0, (size_t)(rowsTp - rowsT) * KpN * sizeof(float), s));
    return LTGW_OK;
  }
  const int Kpa = (n_aux + 63) / 64 * 64;
  const int nI_ov = (int)((n_ov + 127) / 128);
  const int MpT = (n_orb_act + 127) / 128 * 128;
  float *UtF, *BactT, *BtgT, *ones;
  __nv_bfloat16 *Bh, *Bl, *Uh = nullptr, *Ul = nullptr;   // B operands pre-split for the TMA-fed kernel
  const bool pre = Bh_in != nullptr;
  auto layout = [&](Arena &A) {
    UtF = A.take<float>((size_t)MpN * Kpa);
    BactT = (B_act && !pre) ? A.take<float>((size_t)nI_ov * 128 * Kpa) : nullptr;
    BtgT = window ? nullptr : A.take<float>((size_t)T * MpT * Kpa);
    ones = A.take<float>((size_t)std::max(T, 1) * Kpa);
    Bh = (B_act && !pre) ? A.take<__nv_bfloat16>((size_t)nI_ov * 128 * Kpa) : nullptr;
    Bl = (B_act && !pre) ? A.take<__nv_bfloat16>((size_t)nI_ov * 128 * Kpa) : nullptr;
    if (!window) {
      Uh = A.take<__nv_bfloat16>((size_t)MpN * Kpa);
      Ul = A.take<__nv_bfloat16>((size_t)MpN * Kpa);
    }
  };
  ctx->a5.begin_sizing();
  layout(ctx->a5);
  if (ctx->a5.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "tensor-core operand allocation failed"); return ctx->status(); }
  layout(ctx->a5);
  CHECK_LAUNCH(ctx, launch_to_f32_padded(Ut, n_aux, N, n_aux, UtF, MpN, Kpa, s), 1);
  if (B_act && !pre)
    CHECK_LAUNCH(ctx, launch_to_f32_transposed(B_act, ld_act, 0, n_aux, (int)n_ov, BactT, Kpa, nI_ov * 128, 1, 0, 0, s),
                 1);
  if (!window)
    CHECK_LAUNCH(ctx, launch_to_f32_transposed(B_tgt, n_orb, n_fc, n_aux, n_orb_act, BtgT, Kpa, MpT, T,
                                               (int64_t)n_aux * n_orb, (int64_t)MpT * Kpa, s), 1);
  CHECK_LAUNCH(ctx, launch_scale_table(nullptr, n_aux, Kpa, std::max(T, 1), nullptr, nullptr, SCALE_NONE, ones, s), 1);
  // R~_ov = U^T R_ov: rows N (A = U^T), columns n_ov (B rows = R_ov^T)
  if (B_act || pre) {
    if (!pre) CHECK_LAUNCH(ctx, launch_split_bf16(BactT, Bh, Bl, (int64_t)nI_ov * 128 * Kpa, s), 1);
    TcGemmArgs g;
    g.A = UtF; g.B = BactT; g.scale = ones; g.Kp = Kpa; g.n_t = 1; g.nt_group = 1;
    g.B_hi = pre ? Bh_in : Bh; g.B_lo = pre ? Bl_in : Bl; g.rows_a = MpN; g.rows_b = (int64_t)nI_ov * 128;
    TcRun run;
    const int nI = (N + 127) / 128;
    if (tc_run(ctx, ctx->a4, g, full_tiles(nI, nI_ov), 0, &run, s) != LTGW_OK) return ctx->status();
    if (window) {
      CHECK_LAUNCH(ctx, launch_tc_reduce_full(run.partial, run.partial32, run.splits, run.groups, run.n_tiles, nI_ov,
                                              N, (int)n_ov, 1.0, nullptr, 0, 0, Bf + window->col0, window->ld_bf,
                                              MpN, 0, s, n_ov), 1);
      return LTGW_OK;
    }
    CHECK_LAUNCH(ctx, launch_tc_reduce_full(run.partial, run.partial32, run.splits, run.groups, run.n_tiles, nI_ov, N,
                                            (int)n_ov, 1.0, nullptr, 0, 0, Bf, Kp_ov, MpN, 0, s), 1);
  }
  // R~_tgt[t]^T = R_tgt[t]^T U: per target t, rows n_orb_act (A), columns N (B rows = U^T)
  {
    CHECK_LAUNCH(ctx, launch_split_bf16(UtF, Uh, Ul, (int64_t)MpN * Kpa, s), 1);
    TcGemmArgs g;
    g.A = BtgT; g.a_group_stride = (int64_t)MpT * Kpa; g.B = UtF; g.scale = ones; g.Kp = Kpa;
    g.n_t = T; g.nt_group = 1;
    g.B_hi = Uh; g.B_lo = Ul; g.rows_a = MpT; g.rows_b = MpN;
    TcRun run;
    const int nJ = (N + 127) / 128;
    if (tc_run(ctx, ctx->a4, g, full_tiles(MpT / 128, nJ), 0, &run, s) != LTGW_OK) return ctx->status();
    CHECK_LAUNCH(ctx, launch_tc_reduce_full(run.partial, run.partial32, run.splits, run.groups, run.n_tiles, nJ,
                                            n_orb_act, N, 1.0, BtT64, N, (int64_t)n_orb_act * N, BtT32, KpN,
                                            n_orb_act, (int64_t)n_orb_act * KpN, s), 1);
    if (rowsTp > rowsT)
      LTGW_CUDA(ctx, cudaMemsetAsync(BtT32 + rowsT * KpN, 0, (size_t)(rowsTp - rowsT) * KpN * sizeof(float), s));
  }
  return LTGW_OK;
}

// W_nm(i w_j) (Eq. ScreenedCoulombOrbital) on the tensor cores: Y_j = C_j R~_tgt
// with the column dot against R~_tgt fused into the epilogue; split BF16, or
// (fp8) FP8 E4M3 codes of C_j's and R~_tgt^T's rows, each row with its own
// scale (C_j's rows are auxiliary functions).
ltgw_status wnm_tc(ltgw_ctx *ctx, int N, int n_omega, const double *C, int T, int n_orb_act, const double *BtT64,
                   const float *BtT32, double *W, cudaStream_t s, bool fp8) {
  const int KpN = (N + 63) / 64 * 64, MpN = (N + 127) / 128 * 128, nI = MpN / 128, Kq = (N + 127) / 128 * 128;
  const int ncols = T * n_orb_act, nJ = (ncols + 127) / 128, rowsTp = nJ * 128;
  float *Cf, *ones = nullptr, *dsC = nullptr, *dsR = nullptr;
  uint8_t *qC = nullptr, *qR = nullptr;
  int *maxima = nullptr;
  __nv_bfloat16 *Rh = nullptr, *Rl = nullptr;   // R~_tgt^T pre-split for the TMA-fed kernel
  auto layout = [&](Arena &A) {
    Cf = A.take<float>((size_t)n_omega * MpN * KpN);
    if (fp8) {
      qC = A.take<uint8_t>((size_t)n_omega * MpN * 3 * Kq);
      qR = A.take<uint8_t>((size_t)rowsTp * 3 * Kq);
      dsC = A.take<float>((size_t)n_omega * MpN);
      dsR = A.take<float>((size_t)rowsTp);
      maxima = A.take<int>((size_t)rowsTp);
    } else {
      ones = A.take<float>((size_t)n_omega * KpN);
      Rh = A.take<__nv_bfloat16>((size_t)rowsTp * KpN);
      Rl = A.take<__nv_bfloat16>((size_t)rowsTp * KpN);
    }
  };
  ctx->a5.begin_sizing();
  layout(ctx->a5);
  if (ctx->a5.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "tensor-core operand allocation failed"); return ctx->status(); }
  layout(ctx->a5);
  // C_j is symmetric, so its transpose is its padded copy
  CHECK_LAUNCH(ctx, launch_to_f32_transposed(C, N, 0, N, N, Cf, KpN, MpN, n_omega, (int64_t)N * N,
                                             (int64_t)MpN * KpN, s), 1);
  TcGemmArgs g;
  if (fp8) {
    // two-term E4M3 expansions: C_j's rows as A operands, R~_tgt^T's as B
    CHECK_LAUNCH(ctx, launch_fp8_quantize_a(Cf, KpN, Kq, n_omega * MpN, qC, dsC, s, 1), 1);
    CHECK_LAUNCH(ctx, launch_fp8_quantize(BtT32, KpN, Kq, nullptr, 0, rowsTp, nullptr, qR, nullptr, dsR, maxima, s, 1), 2);
    g.A8 = qC; g.B8 = qR; g.ds_a = dsC; g.ds_b = dsR; g.Kp = 3 * Kq; g.rows_a = MpN; g.rows_b = rowsTp;
  } else {
    CHECK_LAUNCH(ctx, launch_scale_table(nullptr, N, KpN, n_omega, nullptr, nullptr, SCALE_NONE, ones, s), 1);
    CHECK_LAUNCH(ctx, launch_split_bf16(BtT32, Rh, Rl, (int64_t)rowsTp * KpN, s), 1);
    g.A = Cf; g.a_group_stride = (int64_t)MpN * KpN; g.B = BtT32; g.scale = ones; g.Kp = KpN;
    g.B_hi = Rh; g.B_lo = Rl; g.rows_a = MpN; g.rows_b = rowsTp;   // C_j stacked by frequency
  }
  g.n_t = n_omega; g.nt_group = 1;
  g.out_mode = TC_OUT_COLDOT;
  g.cd_B = BtT64; g.cd_ld = N; g.cd_rows = N; g.cd_cols = ncols; g.cd_cols_p = nJ * 128;
  TcRun run;
  if (tc_run(ctx, ctx->a4, g, full_tiles(nI, nJ), nI, &run, s) != LTGW_OK) return ctx->status();
  CHECK_LAUNCH(ctx, launch_tc_reduce_coldot(run.cd_out, run.splits, run.groups, nI, nJ * 128, ncols, W, ncols, s), 1);
  return LTGW_OK;
}

ltgw_status validate(ltgw_ctx *ctx, const ltgw_params *p) {
  REQUIRE(ctx, p != nullptr, "params is NULL");
  REQUIRE(ctx, p->n_occ >= 1 && p->n_virt >= 1 && p->n_aux >= 1, "n_occ, n_virt, n_aux must be >= 1");
  REQUIRE(ctx, p->n_frozen >= 0 && p->n_frozen < p->n_occ, "need 0 <= n_frozen < n_occ");
  REQUIRE(ctx, p->n_omega >= 1 && p->n_omega <= 256, "n_omega must be in [1, 256]");
  REQUIRE(ctx, p->omega0 > 0.0 && isfinite(p->omega0), "omega0 must be positive");
  REQUIRE(ctx, p->spin == 1 || p->spin == 2, "spin must be 1 or 2");
  REQUIRE(ctx, p->use_laplace >= 0 && p->use_laplace <= 2, "use_laplace must be 0, 1 or 2");
  REQUIRE(ctx, !p->use_laplace || (p->n_tau >= 1 && p->n_tau <= 32), "n_tau must be in [1, 32]");
  REQUIRE(ctx, p->precision >= LTGW_FP64 && p->precision <= LTGW_FP64_EMU,
          "precision must be LTGW_FP64, LTGW_BF16X3, LTGW_FP8, LTGW_FP8_PI or LTGW_FP64_EMU");
  REQUIRE(ctx, p->reserved == 0, "reserved must be 0");
  REQUIRE(ctx, isfinite(p->naf_thresh), "naf_thresh must be finite");
  return LTGW_OK;
}

}  // namespace

size_t ltgw::solve_digit_bytes(const ltgw_params &p, int n_tgt, int N, size_t limit) {
  const int n_sm = 152, n_act = p.n_occ - p.n_frozen, n_orb_act = n_act + p.n_virt;
  const int n_t = p.use_laplace && p.n_tau > 0 ? p.n_tau : p.n_omega;
  if (n_act < 1 || p.n_virt < 1 || p.n_aux < 1 || n_t < 1 || p.n_omega < 1 || N < 1 || n_tgt < 1) return 0;
  const int64_t n_ov = (int64_t)n_act * p.n_virt;
  const bool emu = p.precision == LTGW_FP64_EMU;
  Arena ar;
  size_t most = 0;
  auto add = [&](auto piece) {
    size_t b = piece_bytes(ar, piece);
    if (b > limit) {
      while (piece.shrink()) b = piece_bytes(ar, piece);
      b = std::max(b, limit);
    }
    most = std::max(most, b);
  };
  if (emu || p.precision == LTGW_FP64) {
    const SliceForm f = emu ? emu_digits(kEmuSlices) : kFp64Digits;
    if (p.naf_thresh >= 0.0) {
      add(SyrkPiece(n_sm, p.n_aux, n_ov, f));
      add(ProjectPiece(n_sm, N, p.n_aux, std::min<int64_t>(n_ov, INT32_MAX), 1, f));
      add(ProjectPiece(n_sm, N, p.n_aux, n_orb_act, n_tgt, f));
    }
    if (emu) add(PiEmuPiece(n_sm, N, n_ov, n_t, f));
    else add(PiPiece(n_sm, N, n_ov, n_t, f));
    add(WnmPiece(N, p.n_omega, n_tgt, n_orb_act, f));
  }
  if (N >= kScreenDigitsMinN) add(ScreenPiece(N, p.n_omega));
  return most;
}

void ltgw::release_products(ltgw_ctx *ctx) {
  ctx->a4.release();
  ctx->a5.release();
}


extern "C" {

const char *ltgw_status_string(ltgw_status s) {
  switch (s) {
    case LTGW_OK: return "ok";
    case LTGW_ERR_BAD_ARG: return "bad argument";
    case LTGW_ERR_NOMEM: return "out of memory";
    case LTGW_ERR_NOT_SPD: return "1 - Pi not positive definite";
    case LTGW_ERR_NO_CONVERGE: return "quasi-particle solve did not converge";
    case LTGW_ERR_DEVICE: return "CUDA error";
    case LTGW_ERR_EIG: return "eigensolver failure";
    case LTGW_ERR_NO_NAF: return "no natural auxiliary function kept";
    case LTGW_ERR_TIMEOUT: return "timed out";
  }
  return "unknown status";
}

ltgw_status ltgw_create(ltgw_ctx **out, int device) {
  if (!out) return LTGW_ERR_BAD_ARG;
  *out = nullptr;
  int n = 0;
  if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) {
    cudaGetLastError();
    return LTGW_ERR_DEVICE;
  }
  if (cudaSetDevice(device) != cudaSuccess) return LTGW_ERR_DEVICE;
  ltgw_ctx *c = new ltgw_ctx();
  c->device = device;
  if (cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || c->n_sm < 1) {
    cudaGetLastError();
    c->n_sm = 148;
  }
  if (cudaMalloc(&c->flags, FLAG_COUNT * sizeof(int)) != cudaSuccess) {
    delete c;
    return LTGW_ERR_NOMEM;
  }
  for (auto &e : c->ev) cudaEventCreate(&e);
  if (cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->fork_ev, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->join_ev, cudaEventDisableTiming) != cudaSuccess ||
      cudaStreamCreateWithFlags(&c->fill_stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->blk_ready[0], cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->blk_ready[1], cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->blk_done[0], cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->blk_done[1], cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    ltgw_destroy(c);
    return LTGW_ERR_DEVICE;
  }
  *out = c;
  return LTGW_OK;
}

void ltgw_destroy(ltgw_ctx *ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  ctx->a1.release();
  ctx->a2.release();
  ctx->a3.release();
  ctx->a4.release();
  ctx->a5.release();
  if (ctx->flags) cudaFree(ctx->flags);
  for (auto &e : ctx->ev) if (e) cudaEventDestroy(e);
  if (ctx->side) cudaStreamDestroy(ctx->side);
  if (ctx->fork_ev) cudaEventDestroy(ctx->fork_ev);
  if (ctx->join_ev) cudaEventDestroy(ctx->join_ev);
  if (ctx->fill_stream) cudaStreamDestroy(ctx->fill_stream);
  for (int b = 0; b < 2; ++b) {
    if (ctx->blk_ready[b]) cudaEventDestroy(ctx->blk_ready[b]);
    if (ctx->blk_done[b]) cudaEventDestroy(ctx->blk_done[b]);
  }
  delete ctx;
}

const char *ltgw_last_error(const ltgw_ctx *ctx) { return ctx ? ctx->err.c_str() : "no context"; }

ltgw_status ltgw_set_timing(ltgw_ctx *ctx, int on) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->timing = (on != 0);
  return LTGW_OK;
}

size_t ltgw_workspace_bytes(const ltgw_ctx *ctx) {
  if (!ctx) return 0;
  return ctx->a1.cap + ctx->a2.cap + ctx->a3.cap + ctx->a4.cap + ctx->a5.cap;
}

ltgw_status ltgw_trim(ltgw_ctx *ctx) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  ctx->a1.release();
  ctx->a2.release();
  ctx->a3.release();
  ctx->a4.release();
  ctx->a5.release();
  return LTGW_OK;
}

ltgw_status ltgw_set_autotune(ltgw_ctx *ctx, int on) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->autotune = (on != 0);
  return LTGW_OK;
}

ltgw_status ltgw_set_digit_memory(ltgw_ctx *ctx, size_t bytes) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->digit_max = bytes;
  return LTGW_OK;
}

ltgw_status ltgw_get_stats(const ltgw_ctx *ctx, ltgw_stats *out) {
  if (!ctx || !out) return LTGW_ERR_BAD_ARG;
  *out = ctx->stats;
  return LTGW_OK;
}

}  // extern "C"

namespace {

// One solve; with `fill` set, B_ov is not given and the occupied blocks are
// requested from the caller twice (NAF metric, then projection).
// One solve; ev_cycles > 0 adds evGW cycles (Sec. 3): Pi, W and Sigma rebuilt
// from the previous quasi-particle energies (targets) and the scissor shift of
// the nearest target (other active orbitals), the NAF basis and the projected
// tensors kept, until the HOMO/LUMO quasi-particle gap changes by less than
// ev_gap_tol (> 0; both states among the targets) or ev_cycles cycles ran.
ltgw_status solve_impl(ltgw_ctx *ctx, const ltgw_params *p, const double *eps, const double *B_ov,
                       ltgw_block_fn fill, void *user, int occ_block, const double *B_tgt, const int *targets,
                       int n_tgt, const double *shift, const double *tau_x, const double *tau_w,
                       double *sigma_iw, double *e_qp, int *qp_status, void *stream, int ev_cycles = 0,
                       double ev_gap_tol = 0.0, int *ev_done = nullptr) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  if (validate(ctx, p) != LTGW_OK) return ctx->status();
  const bool streamed = fill != nullptr;
  REQUIRE(ctx, eps && (B_ov || streamed) && B_tgt && targets && shift && sigma_iw && e_qp && qp_status,
          "a required pointer is NULL");
  REQUIRE(ctx, !streamed || (p->naf_thresh >= 0.0 && occ_block >= 1),
          "the streamed solve needs NAF (naf_thresh >= 0) and occ_block >= 1");
  REQUIRE(ctx, n_tgt >= 1, "n_tgt must be >= 1");
  REQUIRE(ctx, (tau_x == nullptr) == (tau_w == nullptr), "tau_x and tau_w must both be given or both NULL");
  REQUIRE(ctx, ev_cycles >= 0 && ev_cycles <= 100 && ev_gap_tol >= 0.0, "need 0 <= ev_cycles <= 100, ev_gap_tol >= 0");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  const int n_occ = p->n_occ, n_virt = p->n_virt, n_fc = p->n_frozen, n_aux = p->n_aux;
  const int n_orb = n_occ + n_virt, n_act = n_occ - n_fc, n_orb_act = n_orb - n_fc;
  const int64_t n_ov_all = (int64_t)n_occ * n_virt, n_ov = (int64_t)n_act * n_virt;
  const int n_omega = p->n_omega, T = n_tgt;
  const int n_tau = p->use_laplace ? p->n_tau : 0;
  const bool naf = p->naf_thresh >= 0.0;
  // emulated FP64 form: the FP64 form's data flow with K, the projections, Pi
  // and W_nm FP64-accurate from integer slices on the tensor cores
  const bool emu = p->precision == LTGW_FP64_EMU;
  const SliceForm emu_f = emu_digits(kEmuSlices);
  const bool mixed = p->precision != LTGW_FP64 && !emu;   // split-BF16 / FP8 contractions
  const bool fp8 = p->precision == LTGW_FP8 || p->precision == LTGW_FP8_PI;   // Pi build in FP8 E4M3
  const bool fp8_w = p->precision == LTGW_FP8;                                // W_nm in FP8 E4M3
  ctx->stats = ltgw_stats{};
  ctx->mark(EV_START, s);

  // small inputs on the host
  std::vector<double> h_eps(n_orb), h_shift(T);
  std::vector<int> h_tg(T);
  if (read_small(ctx, h_eps.data(), eps, n_orb * sizeof(double), s) != LTGW_OK) return ctx->status();
  if (read_small(ctx, h_tg.data(), targets, T * sizeof(int), s) != LTGW_OK) return ctx->status();
  if (read_small(ctx, h_shift.data(), shift, T * sizeof(double), s) != LTGW_OK) return ctx->status();
  for (int i = 0; i < n_orb; ++i) REQUIRE(ctx, isfinite(h_eps[i]), "eps has a non-finite entry");
  for (int i = 1; i < n_orb; ++i) REQUIRE(ctx, h_eps[i] >= h_eps[i - 1], "eps must be ascending");
  REQUIRE(ctx, h_eps[n_occ] > h_eps[n_occ - 1], "need eps_LUMO > eps_HOMO");
  for (int t = 0; t < T; ++t)
    REQUIRE(ctx, h_tg[t] >= n_fc && h_tg[t] < n_orb, "target outside the active orbitals");
  double eF = 0.5 * (h_eps[n_occ - 1] + h_eps[n_occ]);
  std::vector<double> h_om(n_omega), h_wt(n_omega);
  if (ltgw_gl_grid(n_omega, p->omega0, h_om.data(), h_wt.data()) != LTGW_OK) {
    ctx->fail(LTGW_ERR_BAD_ARG, "GL grid");
    return ctx->status();
  }
  std::vector<double> h_x(n_tau), h_w(n_tau), h_E((size_t)n_omega * std::max(n_tau, 1));
  ctx->stats.lt_max_rel_err = NAN;
  // The library's grid for orbital energies e: Eq. LT's bounds of Sec. 3
  // (a = gap^2 + w_min^2, b = max(span^2, 1e4)), or the imaginary-time fit on
  // [gap, span] (the tensor-core forms carry ~1e-5 relative error in M^k: a
  // larger ridge keeps the recombination from magnifying it).
  auto fit_grid = [&](const std::vector<double> &e) -> ltgw_status {
    const double gap = e[n_occ] - e[n_occ - 1];
    const double span = *std::max_element(e.begin() + n_fc, e.end()) - *std::min_element(e.begin() + n_fc, e.end());
    double err = 0.0;
    if (p->use_laplace == 2) {
      if (ltgw_cosine_grid(n_tau, gap, span, n_omega, h_om.data(), mixed ? 1e-10 : 1e-14, h_x.data(), h_E.data(),
                           &err, nullptr) != LTGW_OK) {
        ctx->fail(LTGW_ERR_BAD_ARG, "imaginary-time grid fit");
        return ctx->status();
      }
    } else {
      if (ltgw_laplace_grid(n_tau, gap * gap + h_om[0] * h_om[0], std::max(span * span, 1e4), h_x.data(), h_w.data(),
                            &err) != LTGW_OK) {
        ctx->fail(LTGW_ERR_BAD_ARG, "Laplace grid fit");
        return ctx->status();
      }
      for (int j = 0; j < n_omega; ++j)
        for (int k = 0; k < n_tau; ++k) h_E[(size_t)j * n_tau + k] = exp(-h_om[j] * h_om[j] * h_x[k]);
    }
    ctx->stats.lt_max_rel_err = err;
    return LTGW_OK;
  };
  if (n_tau && tau_x) {
    // caller's grid: Eq. LT (x, w), or imaginary time (tau_k, gamma [n_omega][n_tau])
    if (read_small(ctx, h_x.data(), tau_x, n_tau * sizeof(double), s) != LTGW_OK) return ctx->status();
    if (p->use_laplace == 2) {
      if (read_small(ctx, h_E.data(), tau_w, h_E.size() * sizeof(double), s) != LTGW_OK) return ctx->status();
    } else {
      if (read_small(ctx, h_w.data(), tau_w, n_tau * sizeof(double), s) != LTGW_OK) return ctx->status();
      for (int j = 0; j < n_omega; ++j)
        for (int k = 0; k < n_tau; ++k) h_E[(size_t)j * n_tau + k] = exp(-h_om[j] * h_om[j] * h_x[k]);
    }
  } else if (n_tau && fit_grid(h_eps) != LTGW_OK) {
    return ctx->status();
  }
  std::vector<double> h_epsn(T);
  for (int t = 0; t < T; ++t) h_epsn[t] = h_eps[h_tg[t]];

  const bool bov_dev = streamed || is_device_ptr(B_ov), btg_dev = is_device_ptr(B_tgt);
  // a streamed solve that fails leaves no callback work in flight behind it
  struct FillDrain {
    ltgw_ctx *ctx;
    bool on;
    ~FillDrain() {
      if (on) cudaStreamSynchronize(ctx->fill_stream);
    }
  } fill_drain{ctx, streamed};
  const int blk = streamed ? std::min(occ_block, n_act) : 0;
  double *d_blk[2] = {nullptr, nullptr};
  // streamed tensor-core forms: every block, transposed and split into BF16
  // hi / lo as the projection's operand, is kept from the metric's pass, so
  // that the callback is asked for each block once
  const bool keep_split = streamed && mixed;
  const int64_t n_ov_p = (n_ov + 127) / 128 * 128, Kpa_aux = (n_aux + 63) / 64 * 64;
  __nv_bfloat16 *d_Rh = nullptr, *d_Rl = nullptr;
  float *d_Rt = nullptr;   // one block, transposed, FP32
  ctx->gen_ms = 0.0;
  // ---- phase-1 workspace: inputs, grids, NAF
  double *d_eps, *d_delta, *d_om, *d_wt, *d_x, *d_w, *d_E, *d_epsn, *d_shift, *d_Bov, *d_Btg, *d_Ut, *d_lam;
  auto layout1 = [&](Arena &A) {
    d_eps = A.take<double>(n_orb);
    d_delta = A.take<double>(n_ov);
    d_om = A.take<double>(n_omega);
    d_wt = A.take<double>(n_omega);
    d_x = A.take<double>(std::max(n_tau, 1));
    d_w = A.take<double>(std::max(n_tau, 1));
    d_E = A.take<double>(h_E.size());
    d_epsn = A.take<double>(T);
    d_shift = A.take<double>(T);
    d_Bov = bov_dev ? const_cast<double *>(B_ov) : A.take<double>((size_t)n_aux * n_ov_all);
    d_blk[0] = streamed ? A.take<double>((size_t)n_aux * blk * n_virt) : nullptr;
    d_blk[1] = streamed ? A.take<double>((size_t)n_aux * blk * n_virt) : nullptr;
    d_Rh = keep_split ? A.take<__nv_bfloat16>((size_t)n_ov_p * Kpa_aux) : nullptr;
    d_Rl = keep_split ? A.take<__nv_bfloat16>((size_t)n_ov_p * Kpa_aux) : nullptr;
    d_Rt = keep_split ? A.take<float>((size_t)blk * n_virt * Kpa_aux) : nullptr;
    d_Btg = btg_dev ? const_cast<double *>(B_tgt) : A.take<double>((size_t)T * n_aux * n_orb);
    d_Ut = naf ? A.take<double>((size_t)n_aux * n_aux) : nullptr;
    d_lam = naf ? A.take<double>(n_aux) : nullptr;
  };
  ctx->a1.begin_sizing();
  layout1(ctx->a1);
  if (ctx->a1.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "input workspace allocation failed"); return ctx->status(); }
  layout1(ctx->a1);
  LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  copy_in(ctx, d_eps, h_eps.data(), n_orb * sizeof(double), s);
  copy_in(ctx, d_om, h_om.data(), n_omega * sizeof(double), s);
  copy_in(ctx, d_wt, h_wt.data(), n_omega * sizeof(double), s);
  if (n_tau) {
    copy_in(ctx, d_x, h_x.data(), n_tau * sizeof(double), s);
    copy_in(ctx, d_w, h_w.data(), n_tau * sizeof(double), s);
    copy_in(ctx, d_E, h_E.data(), h_E.size() * sizeof(double), s);
  }
  copy_in(ctx, d_epsn, h_epsn.data(), T * sizeof(double), s);
  copy_in(ctx, d_shift, h_shift.data(), T * sizeof(double), s);
  // a solve that fails from here on waits for its stream before it returns,
  // so that no copy from the caller's (possibly pinned) B_ov or B_tgt is
  // still in flight when the call returns
  struct SyncOnError {
    ltgw_ctx *ctx;
    cudaStream_t s;
    bool active;
    ~SyncOnError() {
      if (active && ctx->status() != LTGW_OK) cudaStreamSynchronize(s);
    }
  } sync_on_error{ctx, s, !bov_dev || !btg_dev};
  // host B_ov: only the active pairs' columns cross the link (the frozen
  // columns are never read)
  if (!bov_dev && n_fc == 0) copy_in(ctx, d_Bov, B_ov, (size_t)n_aux * n_ov_all * sizeof(double), s);
  if (!bov_dev && n_fc > 0)
    LTGW_CUDA(ctx, cudaMemcpy2DAsync(d_Bov + (int64_t)n_fc * n_virt, (size_t)n_ov_all * sizeof(double),
                                     B_ov + (int64_t)n_fc * n_virt, (size_t)n_ov_all * sizeof(double),
                                     (size_t)n_ov * sizeof(double), (size_t)n_aux, cudaMemcpyDefault, s));
  // host B_tgt is first read by the projections, after the NAF: its copy runs
  // on the side stream meanwhile.  A solve that fails before the join waits
  // for the copy, so the caller may release B_tgt when the call returns.
  struct SideJoin {
    ltgw_ctx *ctx = nullptr;
    bool pending = false;
    ltgw_status join(cudaStream_t s) {
      if (!pending) return LTGW_OK;
      pending = false;
      LTGW_CUDA(ctx, cudaStreamWaitEvent(s, ctx->join_ev, 0));
      return LTGW_OK;
    }
    ~SideJoin() {
      if (pending) cudaStreamSynchronize(ctx->side);
    }
  } btg_join;
  btg_join.ctx = ctx;
  if (!btg_dev) {
    LTGW_CUDA(ctx, cudaEventRecord(ctx->fork_ev, s));
    LTGW_CUDA(ctx, cudaStreamWaitEvent(ctx->side, ctx->fork_ev, 0));
    LTGW_CUDA(ctx, cudaMemcpyAsync(d_Btg, B_tgt, (size_t)T * n_aux * n_orb * sizeof(double), cudaMemcpyDefault,
                                   ctx->side));
    btg_join.pending = true;
    LTGW_CUDA(ctx, cudaEventRecord(ctx->join_ev, ctx->side));
  }
  if (ctx->status() != LTGW_OK) return ctx->status();
  CHECK_LAUNCH(ctx, launch_pair_gaps(d_eps, n_occ, n_virt, n_fc, d_delta, s), 1);

  // ---- frozen-core slice: the active pairs are the trailing columns
  const double *B_act = streamed ? nullptr : d_Bov + (int64_t)n_fc * n_virt;
  const int64_t ld_act = n_ov_all;
  // streamed: ask the caller for occupied block [i0, i1) into the next of the
  // two block buffers (*dst).  The buffer's previous consumers are waited for
  // on the host first, so the callback may write it by any means; its work,
  // issued on the fill stream, then overlaps the consumers of the other
  // buffer on `s`, which waits for the block's arrival.  block_done() marks
  // the block's consumers issued.
  int blk_next = 0;
  auto get_block = [&](int i0, int i1, double **dst) -> ltgw_status {
    const int b = blk_next;
    LTGW_CUDA(ctx, cudaEventSynchronize(ctx->blk_done[b]));
    const auto t0 = std::chrono::steady_clock::now();
    const int rc = fill(user, i0, i1, d_blk[b], (void *)ctx->fill_stream);
    ctx->gen_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    if (rc != 0) {
      cudaStreamSynchronize(ctx->fill_stream);
      ctx->fail(LTGW_ERR_BAD_ARG, "the block callback reported an error");
      return ctx->status();
    }
    LTGW_CUDA(ctx, cudaEventRecord(ctx->blk_ready[b], ctx->fill_stream));
    LTGW_CUDA(ctx, cudaStreamWaitEvent(s, ctx->blk_ready[b], 0));
    *dst = d_blk[b];
    return LTGW_OK;
  };
  auto block_done = [&]() -> ltgw_status {
    LTGW_CUDA(ctx, cudaEventRecord(ctx->blk_done[blk_next], s));
    blk_next ^= 1;
    return LTGW_OK;
  };
  KBuilder build_K = [&](double *K) -> ltgw_status {
    LTGW_CUDA(ctx, cudaMemsetAsync(K, 0, (size_t)n_aux * n_aux * sizeof(double), s));
    for (int i0 = n_fc; i0 < n_occ; i0 += blk) {
      const int i1 = std::min(n_occ, i0 + blk);
      const int64_t cols = (int64_t)(i1 - i0) * n_virt;
      double *B_blk = nullptr;
      if (get_block(i0, i1, &B_blk) != LTGW_OK) return ctx->status();
      if (mixed) {
        if (naf_metric_tc(ctx, n_aux, cols, B_blk, cols, K, s, 1.0) != LTGW_OK) return ctx->status();
        // the projection's operand rows (i0 - n_fc) n_virt .. + cols, transposed and split
        const int64_t off = (int64_t)(i0 - n_fc) * n_virt * Kpa_aux;
        CHECK_LAUNCH(ctx, launch_to_f32_transposed(B_blk, cols, 0, n_aux, (int)cols, d_Rt, (int)Kpa_aux, (int)cols,
                                                   1, 0, 0, s), 1);
        CHECK_LAUNCH(ctx, launch_split_bf16(d_Rt, d_Rh + off, d_Rl + off, cols * Kpa_aux, s), 1);
      } else if (emu) {
        bool done = false;   // K += B_blk B_blk^T from slices
        if (slice_syrk(ctx, n_aux, cols, B_blk, cols, K, 1.0, emu_f, s, &done) != LTGW_OK) return ctx->status();
      } else {
        bool done = false;   // K += B_blk B_blk^T
        if (slices_pay(n_aux, n_aux, cols, 1) &&
            slice_syrk(ctx, n_aux, cols, B_blk, cols, K, 1.0, kFp64Digits, s, &done) != LTGW_OK)
          return ctx->status();
        if (!done) {
          GemmF64Args g;
          g.M = n_aux; g.N = n_aux; g.K = cols;
          g.A = B_blk; g.lda = cols; g.B = B_blk; g.ldb = cols;
          g.C = K; g.ldc = n_aux; g.syrk = 1; g.beta = 1.0;
          CHECK_LAUNCH(ctx, launch_gemm_f64(g, 1, true, true, s), 1);
        }
      }
      if (block_done() != LTGW_OK) return ctx->status();
    }
    if (keep_split && n_ov_p > n_ov) {
      LTGW_CUDA(ctx, cudaMemsetAsync(d_Rh + n_ov * Kpa_aux, 0, (size_t)(n_ov_p - n_ov) * Kpa_aux * 2, s));
      LTGW_CUDA(ctx, cudaMemsetAsync(d_Rl + n_ov * Kpa_aux, 0, (size_t)(n_ov_p - n_ov) * Kpa_aux * 2, s));
    }
    return LTGW_OK;
  };

  // ---- NAF (Eqs. nafeq, naftrafo) on a separate arena for its scratch
  int N = n_aux, near = 0;
  if (naf) {
    if (naf_basis_dev(ctx, ctx->a3, n_aux, n_ov, B_act, ld_act, p->naf_thresh, d_Ut, d_lam, &N, &near, s,
                      mixed, streamed ? &build_K : nullptr, emu ? kEmuSlices : 0) != LTGW_OK)
      return ctx->status();
  }
  ctx->stats.n_naf = N;
  ctx->stats.naf_near_threshold = near;
  if (btg_join.join(s) != LTGW_OK) return ctx->status();   // B_tgt is read from here on

  // ---- phase-2 workspace
  double *d_Bt = nullptr, *d_Btt = nullptr, *d_M = nullptr, *d_Pi, *d_X0, *d_X1, *d_C, *d_W, *d_sig, *d_eqp;
  int *d_st;
  float *d_Bf = nullptr, *d_BtT32 = nullptr;
  double *d_BtT64 = nullptr;
  const int64_t Kp_ov = (n_ov + 63) / 64 * 64;
  auto layout2 = [&](Arena &A) {
    d_Bt = (naf && !mixed) ? A.take<double>((size_t)N * n_ov) : nullptr;
    d_Btt = (naf && !mixed) ? A.take<double>((size_t)T * N * n_orb_act) : nullptr;
    if (mixed) {
      d_Bf = A.take<float>((size_t)((N + 127) / 128 * 128) * Kp_ov);
      d_BtT64 = A.take<double>((size_t)T * n_orb_act * N);
      d_BtT32 = A.take<float>((size_t)(((int64_t)T * n_orb_act + 127) / 128 * 128) * ((N + 63) / 64 * 64));
    }
    d_M = n_tau ? A.take<double>((size_t)n_tau * N * N) : nullptr;
    d_Pi = A.take<double>((size_t)n_omega * N * N);
    d_X0 = A.take<double>(screen_blocked_scratch(N, n_omega));
    d_X1 = nullptr;
    d_C = A.take<double>((size_t)n_omega * N * N);
    d_W = A.take<double>((size_t)n_omega * T * n_orb_act);
    d_sig = A.take<double>((size_t)T * n_omega * 2);
    d_eqp = A.take<double>(T);
    d_st = A.take<int>(T);
  };
  ctx->a2.begin_sizing();
  layout2(ctx->a2);
  if (ctx->a2.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "solve workspace allocation failed"); return ctx->status(); }
  layout2(ctx->a2);

  // out_b = U^T X_b over `cols` columns of X_b (FP64 form)
  auto project_f64 = [&](const double *X, int64_t ld, int64_t x_batch, int64_t cols, int batch, double *out,
                         int64_t ld_out, int64_t out_batch) -> ltgw_status {
    bool done = false;
    if (slices_pay(N, cols, n_aux, batch) &&
        slice_project(ctx, N, n_aux, d_Ut, X, ld, x_batch, cols, batch, out, ld_out, out_batch, kFp64Digits, s,
                      &done) != LTGW_OK)
      return ctx->status();
    if (done) return LTGW_OK;
    GemmF64Args g;
    g.M = N; g.N = (int)cols; g.K = n_aux;
    g.A = d_Ut; g.lda = n_aux;
    g.B = X; g.ldb = ld; g.strideB = x_batch;
    g.C = out; g.ldc = ld_out; g.strideC = out_batch;
    CHECK_LAUNCH(ctx, launch_gemm_f64(g, batch, true, false, s), 1);
    return LTGW_OK;
  };

  const double *Bt = B_act;
  int64_t ld_bt = ld_act;
  const double *Btt = d_Btg + n_fc;
  int64_t ld_btt = n_orb, stride_btt = (int64_t)n_aux * n_orb;
  if (mixed && streamed) {
    // one projection over every block's kept operand: no second pass of the callback
    if (naf_project_tc(ctx, N, n_aux, d_Ut, nullptr, 0, n_ov, d_Btg, n_orb, n_fc, T, n_orb_act, d_Bf, d_BtT64,
                       d_BtT32, s, nullptr, d_Rh, d_Rl) != LTGW_OK)
      return ctx->status();
  } else if (mixed) {
    if (naf_project_tc(ctx, N, n_aux, naf ? d_Ut : nullptr, B_act, ld_act, n_ov, d_Btg, n_orb, n_fc, T, n_orb_act,
                       d_Bf, d_BtT64, d_BtT32, s) != LTGW_OK)
      return ctx->status();
  } else if (naf) {
    if (streamed) {
      for (int i0 = n_fc; i0 < n_occ; i0 += blk) {
        const int i1 = std::min(n_occ, i0 + blk);
        const int64_t cols = (int64_t)(i1 - i0) * n_virt;
        double *B_blk = nullptr;
        if (get_block(i0, i1, &B_blk) != LTGW_OK) return ctx->status();
        if (emu) {
          bool done = false;
          if (slice_project(ctx, N, n_aux, d_Ut, B_blk, cols, 0, cols, 1, d_Bt + (int64_t)(i0 - n_fc) * n_virt, n_ov, 0,
                            emu_f, s, &done) != LTGW_OK)
            return ctx->status();
        } else {
          // R~_ov[:, block] = U^T R_blk
          if (project_f64(B_blk, cols, 0, cols, 1, d_Bt + (int64_t)(i0 - n_fc) * n_virt, n_ov, 0) != LTGW_OK)
            return ctx->status();
        }
        if (block_done() != LTGW_OK) return ctx->status();
      }
    } else if (emu) {
      REQUIRE(ctx, n_ov <= INT32_MAX, "too many pairs for one emulated projection");
      bool done = false;
      if (slice_project(ctx, N, n_aux, d_Ut, B_act, ld_act, 0, n_ov, 1, d_Bt, n_ov, 0, emu_f, s, &done) != LTGW_OK)
        return ctx->status();
    } else {
      // R~_ov = U^T R_ov
      if (project_f64(B_act, ld_act, 0, std::min<int64_t>(n_ov, INT32_MAX), 1, d_Bt, n_ov, 0) != LTGW_OK)
        return ctx->status();
    }
    if (emu) {
      bool done = false;   // R~_tgt[t] = U^T R_tgt[t][:, active]
      if (slice_project(ctx, N, n_aux, d_Ut, d_Btg + n_fc, n_orb, (int64_t)n_aux * n_orb, n_orb_act, T, d_Btt, n_orb_act,
                        (int64_t)N * n_orb_act, emu_f, s, &done) != LTGW_OK)
        return ctx->status();
    } else {
      // R~_tgt[t] = U^T R_tgt[t][:, active]
      if (project_f64(d_Btg + n_fc, n_orb, (int64_t)n_aux * n_orb, n_orb_act, T, d_Btt, n_orb_act,
                      (int64_t)N * n_orb_act) != LTGW_OK)
        return ctx->status();
    }
    Bt = d_Bt; ld_bt = n_ov;
    Btt = d_Btt; ld_btt = n_orb_act; stride_btt = (int64_t)N * n_orb_act;
  }
  ctx->mark(EV_NAF, s);

  // evGW: the quasi-particle energies of the previous cycle (targets) and the
  // scissor shift of the nearest target by orbital index (other active orbitals)
  auto ev_energies = [&](const std::vector<double> &hq) {
    std::vector<double> e = h_eps;
    std::vector<std::pair<int, double>> ts(T);
    for (int t = 0; t < T; ++t) ts[t] = {h_tg[t], hq[t] - h_eps[h_tg[t]]};
    std::sort(ts.begin(), ts.end());
    for (int q = n_fc; q < n_orb; ++q) {
      int best = 0;
      for (int t = 1; t < T; ++t)
        if (abs(ts[t].first - q) < abs(ts[best].first - q)) best = t;   // ties keep the lower target
      e[q] = h_eps[q] + ts[best].second;
    }
    return e;
  };
  int ih = -1, il = -1;
  for (int t = 0; t < T; ++t) {
    if (h_tg[t] == n_occ - 1) ih = t;
    if (h_tg[t] == n_occ) il = t;
  }
  std::vector<double> hq_prev;
  int cycles = 0;
  for (int cyc = 0;; ++cyc) {
    // ---- Pi (Eq. Pi or the Laplace form)
    if (mixed) {
      if (polarizability_tc(ctx, N, n_ov, nullptr, 0, d_Bf, d_delta, n_omega, d_om, n_tau, d_x, d_w, d_E,
                            d_M, p->spin, d_Pi, s, fp8, p->use_laplace) != LTGW_OK)
        return ctx->status();
    } else if (emu) {
      if (polarizability_emu(ctx, N, n_ov, Bt, ld_bt, d_delta, n_omega, d_om, n_tau, d_x, d_w, d_E, d_M, p->spin,
                             d_Pi, s, p->use_laplace, emu_f) != LTGW_OK)
        return ctx->status();
    } else if (polarizability_dev(ctx, N, n_ov, Bt, ld_bt, d_delta, n_omega, d_om, n_tau, d_x, d_w, d_E, d_M,
                                  p->spin, d_Pi, s, p->use_laplace, false) != LTGW_OK) {
      return ctx->status();
    }
    ctx->mark(EV_PI, s);

    // ---- screening
    if (screen_step(ctx, N, n_omega, d_Pi, d_X0, d_C, s) != LTGW_OK) return ctx->status();
    ctx->mark(EV_SCREEN, s);

    // ---- W_nm(i w_j)
    if (mixed) {
      if (wnm_tc(ctx, N, n_omega, d_C, T, n_orb_act, d_BtT64, d_BtT32, d_W, s, fp8_w) != LTGW_OK) return ctx->status();
    } else if (emu) {
      bool done = false;
      if (slice_wnm(ctx, N, n_omega, d_C, T, n_orb_act, Btt, ld_btt, stride_btt, d_W, emu_f, s, &done) != LTGW_OK)
        return ctx->status();
    } else {
      bool done = false;
      if (slices_pay(N, T * n_orb_act, N, n_omega) &&
          slice_wnm(ctx, N, n_omega, d_C, T, n_orb_act, Btt, ld_btt, stride_btt, d_W, kFp64Digits, s, &done) != LTGW_OK)
        return ctx->status();
      if (!done) {
        ColDotArgs cd;
        cd.N = N; cd.ncols = n_orb_act; cd.n_tgt = T;
        cd.C = d_C; cd.ldc = N; cd.strideC = (int64_t)N * N;
        cd.Bt = Btt; cd.ldb = ld_btt; cd.strideBt = stride_btt;
        cd.W = d_W; cd.ldw = n_orb_act;
        CHECK_LAUNCH(ctx, launch_gemm_coldot(cd, n_omega, s), 1);
      }
    }
    ctx->mark(EV_WNM, s);

    // ---- Sigma(i w), Pade, Newton
    SigmaArgs sa;
    sa.n_tgt = T; sa.n_omega = n_omega; sa.n_orb = n_orb_act;
    sa.W = d_W; sa.eps_m = d_eps + n_fc; sa.omega = d_om; sa.weight = d_wt;
    sa.eps_F = eF; sa.sigma = d_sig;
    CHECK_LAUNCH(ctx, launch_sigma(sa, s), 1);
    QpArgs q;
    q.n_tgt = T; q.n_omega = n_omega; q.pade_stride = 2;
    q.sigma = d_sig; q.omega = d_om; q.eps_n = d_epsn; q.shift = d_shift;
    q.eps_F = eF; q.eta = 0.0; q.tol = 1e-12; q.max_iter = 100;
    q.e_qp = d_eqp; q.status = d_st;
    CHECK_LAUNCH(ctx, launch_qp(q, s), 1);
    ctx->mark(EV_SIGQP, s);

    if (cyc == ev_cycles) break;
    // ---- next evGW cycle
    std::vector<double> hq(T);
    if (read_small(ctx, hq.data(), d_eqp, T * sizeof(double), s) != LTGW_OK) return ctx->status();
    if (cyc > 0 && ev_gap_tol > 0.0 && ih >= 0 && il >= 0 &&
        fabs((hq[il] - hq[ih]) - (hq_prev[il] - hq_prev[ih])) < ev_gap_tol)
      break;
    const std::vector<double> e_next = ev_energies(hq);
    REQUIRE(ctx, e_next[n_occ] > e_next[n_occ - 1], "evGW: the quasi-particle HOMO/LUMO gap closed");
    eF = 0.5 * (e_next[n_occ - 1] + e_next[n_occ]);
    copy_in(ctx, d_eps, e_next.data(), n_orb * sizeof(double), s);
    CHECK_LAUNCH(ctx, launch_pair_gaps(d_eps, n_occ, n_virt, n_fc, d_delta, s), 1);
    if (n_tau && !tau_x) {
      if (fit_grid(e_next) != LTGW_OK) return ctx->status();
      copy_in(ctx, d_x, h_x.data(), n_tau * sizeof(double), s);
      copy_in(ctx, d_w, h_w.data(), n_tau * sizeof(double), s);
      copy_in(ctx, d_E, h_E.data(), h_E.size() * sizeof(double), s);
    }
    if (ctx->status() != LTGW_OK) return ctx->status();
    hq_prev = hq;
    ++cycles;
  }
  if (ev_done) *ev_done = cycles;

  // ---- outputs
  LTGW_CUDA(ctx, cudaMemcpyAsync(sigma_iw, d_sig, (size_t)T * n_omega * 2 * sizeof(double), cudaMemcpyDefault, s));
  LTGW_CUDA(ctx, cudaMemcpyAsync(e_qp, d_eqp, (size_t)T * sizeof(double), cudaMemcpyDefault, s));
  LTGW_CUDA(ctx, cudaMemcpyAsync(qp_status, d_st, (size_t)T * sizeof(int), cudaMemcpyDefault, s));
  ctx->mark(EV_END, s);
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  if (check_flags(ctx, s) != LTGW_OK) return ctx->status();

  ltgw_stats &st = ctx->stats;
  st.n_pade = (n_omega + 1) / 2;
  st.n_tau = n_tau;
  st.kernel_launches = ctx->launches;
  st.pi_kernel_launches = 1;
  st.ms_naf = ctx->ms(EV_START, EV_NAF);
  st.ms_pi = ctx->ms(EV_NAF, EV_PI);
  st.ms_pi_kernel = ctx->ms(EV_PI0, EV_PI1);
  st.ms_screen = ctx->ms(EV_PI, EV_SCREEN);
  st.ms_wnm = ctx->ms(EV_SCREEN, EV_WNM);
  st.ms_sigma_qp = ctx->ms(EV_WNM, EV_SIGQP);
  st.ms_total = ctx->ms(EV_START, EV_END);
  st.ms_tridiag = naf ? ctx->ms(EV_TRI0, EV_TRI1) : 0.0;
  st.ms_naf_metric = naf ? ctx->ms(EV_K0, EV_TRI0) : 0.0;
  st.ms_eig_vectors = naf ? ctx->ms(EV_TRI1, EV_VEC1) : 0.0;
  st.ms_naf_project = naf ? ctx->ms(EV_VEC1, EV_NAF) : 0.0;

  st.ms_generate = ctx->gen_ms;
  std::vector<int> hs(T);
  if (read_small(ctx, hs.data(), qp_status, T * sizeof(int), s) != LTGW_OK) return ctx->status();
  for (int t = 0; t < T; ++t)
    if (hs[t] != 0) ctx->fail(LTGW_ERR_NO_CONVERGE, "a quasi-particle Newton solve did not converge");
  return ctx->status();
}

ltgw_status polarizability_dev_api(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, const double *delta,
                                   int n_omega, const double *omegas, int n_tau, const double *x, const double *w,
                                   int spin, double *Pi, void *stream, int lt_form, const double *gamma) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  REQUIRE(ctx, N >= 1 && n_pairs >= 1 && n_omega >= 1 && n_omega <= 256, "bad sizes");
  REQUIRE(ctx, n_tau >= 0 && n_tau <= 32, "n_tau must be in [0, 32]");
  REQUIRE(ctx, spin == 1 || spin == 2, "spin must be 1 or 2");
  REQUIRE(ctx, Bt && delta && omegas && Pi && (n_tau == 0 || (x && (lt_form == 2 ? gamma : w) != nullptr)),
          "a required pointer is NULL");
  REQUIRE(ctx, is_device_ptr(Bt) && is_device_ptr(delta) && is_device_ptr(Pi), "Bt, delta, Pi must be device pointers");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<double> h_om(omegas, omegas + n_omega), h_E((size_t)n_omega * std::max(n_tau, 1));
  for (int j = 0; j < n_omega; ++j)
    for (int k = 0; k < n_tau; ++k)
      h_E[(size_t)j * n_tau + k] = lt_form == 2 ? gamma[(size_t)j * n_tau + k] : exp(-h_om[j] * h_om[j] * x[k]);
  double *d_om, *d_x, *d_w, *d_E, *d_M;
  auto layout = [&](Arena &A) {
    d_om = A.take<double>(n_omega);
    d_x = A.take<double>(std::max(n_tau, 1));
    d_w = A.take<double>(std::max(n_tau, 1));
    d_E = A.take<double>(h_E.size());
    d_M = n_tau ? A.take<double>((size_t)n_tau * N * N) : nullptr;
  };
  ctx->a2.begin_sizing();
  layout(ctx->a2);
  if (ctx->a2.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "workspace allocation failed"); return ctx->status(); }
  layout(ctx->a2);
  copy_in(ctx, d_om, h_om.data(), n_omega * sizeof(double), s);
  if (n_tau) {
    copy_in(ctx, d_x, x, n_tau * sizeof(double), s);
    if (lt_form != 2) copy_in(ctx, d_w, w, n_tau * sizeof(double), s);
    copy_in(ctx, d_E, h_E.data(), h_E.size() * sizeof(double), s);
  }
  // only the digit kernels set flags
  const bool flags = slices_pay(N, N, n_pairs, n_tau ? n_tau : n_omega);
  if (flags) LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  if (ctx->status() != LTGW_OK) return ctx->status();
  if (polarizability_dev(ctx, N, n_pairs, Bt, n_pairs, delta, n_omega, d_om, n_tau, d_x, d_w, d_E, d_M,
                         spin, Pi, s, lt_form, true) != LTGW_OK)
    return ctx->status();
  if (flags) return check_flags(ctx, s);   // synchronises: the staged grid lives in the workspace
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  return LTGW_OK;
}

// lt_form 1: x, w are the Laplace grid of Eq. LT; 2: x holds tau_k and gamma
// [n_omega][n_tau] the imaginary-time recombination (w unused).
ltgw_status polarizability_tc_api(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, const double *delta,
                                  int n_omega, const double *omegas, int n_tau, const double *x, const double *w,
                                  int spin, double *Pi, void *stream, bool fp8, int lt_form = 1,
                                  const double *gamma = nullptr) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  REQUIRE(ctx, N >= 1 && n_pairs >= 1 && n_omega >= 1 && n_omega <= 256, "bad sizes");
  REQUIRE(ctx, n_tau >= 0 && n_tau <= 32, "n_tau must be in [0, 32]");
  REQUIRE(ctx, spin == 1 || spin == 2, "spin must be 1 or 2");
  REQUIRE(ctx, Bt && delta && omegas && Pi && (n_tau == 0 || (x && (lt_form == 2 ? gamma : w) != nullptr)),
          "a required pointer is NULL");
  REQUIRE(ctx, is_device_ptr(Bt) && is_device_ptr(delta) && is_device_ptr(Pi), "Bt, delta, Pi must be device pointers");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<double> h_om(omegas, omegas + n_omega), h_E((size_t)n_omega * std::max(n_tau, 1));
  for (int j = 0; j < n_omega; ++j)
    for (int k = 0; k < n_tau; ++k)
      h_E[(size_t)j * n_tau + k] = lt_form == 2 ? gamma[(size_t)j * n_tau + k] : exp(-h_om[j] * h_om[j] * x[k]);
  double *d_om, *d_x, *d_w, *d_E, *d_M;
  auto layout = [&](Arena &A) {
    d_om = A.take<double>(n_omega);
    d_x = A.take<double>(std::max(n_tau, 1));
    d_w = A.take<double>(std::max(n_tau, 1));
    d_E = A.take<double>(h_E.size());
    d_M = n_tau ? A.take<double>((size_t)n_tau * N * N) : nullptr;
  };
  ctx->a2.begin_sizing();
  layout(ctx->a2);
  if (ctx->a2.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "workspace allocation failed"); return ctx->status(); }
  layout(ctx->a2);
  LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  copy_in(ctx, d_om, h_om.data(), n_omega * sizeof(double), s);
  if (n_tau) {
    copy_in(ctx, d_x, x, n_tau * sizeof(double), s);
    if (lt_form != 2) copy_in(ctx, d_w, w, n_tau * sizeof(double), s);
    copy_in(ctx, d_E, h_E.data(), h_E.size() * sizeof(double), s);
  }
  if (ctx->status() != LTGW_OK) return ctx->status();
  if (polarizability_tc(ctx, N, n_pairs, Bt, n_pairs, nullptr, delta, n_omega, d_om, n_tau, d_x, d_w, d_E, d_M,
                        spin, Pi, s, fp8, lt_form) != LTGW_OK)
    return ctx->status();
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  ctx->stats.ms_pi_kernel = ctx->ms(EV_PI0, EV_PI1);
  ctx->stats.pi_kernel_launches = 1;
  return check_flags(ctx, s);
}

}  // namespace

extern "C" {

ltgw_status ltgw_solve(ltgw_ctx *ctx, const ltgw_params *p, const double *eps, const double *B_ov,
                       const double *B_tgt, const int *targets, int n_tgt, const double *shift,
                       const double *tau_x, const double *tau_w, double *sigma_iw, double *e_qp,
                       int *qp_status, void *stream) {
  return solve_impl(ctx, p, eps, B_ov, nullptr, nullptr, 0, B_tgt, targets, n_tgt, shift, tau_x, tau_w, sigma_iw,
                    e_qp, qp_status, stream);
}

ltgw_status ltgw_solve_ev(ltgw_ctx *ctx, const ltgw_params *p, const double *eps, const double *B_ov,
                          const double *B_tgt, const int *targets, int n_tgt, const double *shift,
                          const double *tau_x, const double *tau_w, int n_cycles, double gap_tol,
                          double *sigma_iw, double *e_qp, int *qp_status, int *cycles_done, void *stream) {
  return solve_impl(ctx, p, eps, B_ov, nullptr, nullptr, 0, B_tgt, targets, n_tgt, shift, tau_x, tau_w, sigma_iw,
                    e_qp, qp_status, stream, n_cycles, gap_tol, cycles_done);
}

ltgw_status ltgw_solve_streamed(ltgw_ctx *ctx, const ltgw_params *p, const double *eps, ltgw_block_fn fill,
                                void *user, int occ_block, const double *B_tgt, const int *targets, int n_tgt,
                                const double *shift, const double *tau_x, const double *tau_w, double *sigma_iw,
                                double *e_qp, int *qp_status, void *stream) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  if (!fill) {
    ctx->reset();
    ctx->fail(LTGW_ERR_BAD_ARG, "fill callback is NULL");
    return ctx->status();
  }
  return solve_impl(ctx, p, eps, nullptr, fill, user, occ_block, B_tgt, targets, n_tgt, shift, tau_x, tau_w,
                    sigma_iw, e_qp, qp_status, stream);
}

static ltgw_status naf_basis_api(ltgw_ctx *ctx, int n_aux, int64_t n_pairs, const double *B, int64_t ld,
                                 double thresh, double *Ut, double *lambda, int *n_naf, void *stream, bool mixed) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  REQUIRE(ctx, n_aux >= 1 && n_pairs >= 1 && ld >= n_pairs, "bad sizes");
  REQUIRE(ctx, B && Ut && lambda && n_naf, "a required pointer is NULL");
  REQUIRE(ctx, is_device_ptr(B) && is_device_ptr(Ut) && is_device_ptr(lambda), "B, Ut, lambda must be device pointers");
  REQUIRE(ctx, isfinite(thresh), "thresh must be finite");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  int k = 0, near = 0;
  if (naf_basis_dev(ctx, ctx->a3, n_aux, n_pairs, B, ld, thresh, Ut, lambda, &k, &near, s, mixed) != LTGW_OK)
    return ctx->status();
  *n_naf = k;
  ctx->stats = ltgw_stats{};
  ctx->stats.n_naf = k;
  ctx->stats.naf_near_threshold = near;
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  ctx->stats.ms_naf_metric = ctx->ms(EV_K0, EV_TRI0);
  ctx->stats.ms_tridiag = ctx->ms(EV_TRI0, EV_TRI1);
  ctx->stats.ms_eig_vectors = ctx->ms(EV_TRI1, EV_VEC1);
  ctx->stats.kernel_launches = ctx->launches;
  return check_flags(ctx, s);
}

ltgw_status ltgw_naf_basis(ltgw_ctx *ctx, int n_aux, int64_t n_pairs, const double *B, int64_t ld,
                           double thresh, double *Ut, double *lambda, int *n_naf, void *stream) {
  return naf_basis_api(ctx, n_aux, n_pairs, B, ld, thresh, Ut, lambda, n_naf, stream, false);
}

ltgw_status ltgw_naf_basis_mixed(ltgw_ctx *ctx, int n_aux, int64_t n_pairs, const double *B, int64_t ld,
                                 double thresh, double *Ut, double *lambda, int *n_naf, void *stream) {
  return naf_basis_api(ctx, n_aux, n_pairs, B, ld, thresh, Ut, lambda, n_naf, stream, true);
}

ltgw_status ltgw_polarizability(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt,
                                const double *delta, int n_omega, const double *omegas, int n_tau,
                                const double *x, const double *w, int spin, double *Pi, void *stream) {
  return polarizability_dev_api(ctx, N, n_pairs, Bt, delta, n_omega, omegas, n_tau, x, w, spin, Pi, stream, 1,
                                nullptr);
}

ltgw_status ltgw_polarizability_tau(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt, const double *delta,
                                    int n_omega, const double *omegas, int n_tau, const double *tau,
                                    const double *gamma, int spin, int precision, double *Pi, void *stream) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  if (n_tau < 1) { ctx->reset(); ctx->fail(LTGW_ERR_BAD_ARG, "n_tau must be >= 1"); return ctx->status(); }
  if (precision == LTGW_FP64)
    return polarizability_dev_api(ctx, N, n_pairs, Bt, delta, n_omega, omegas, n_tau, tau, nullptr, spin, Pi,
                                  stream, 2, gamma);
  if (precision < LTGW_FP64 || precision > LTGW_FP8_PI) {
    ctx->reset();
    ctx->fail(LTGW_ERR_BAD_ARG, "unknown precision");
    return ctx->status();
  }
  return polarizability_tc_api(ctx, N, n_pairs, Bt, delta, n_omega, omegas, n_tau, tau, nullptr, spin, Pi, stream,
                               precision == LTGW_FP8 || precision == LTGW_FP8_PI, 2, gamma);
}

ltgw_status ltgw_polarizability_mixed(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt,
                                      const double *delta, int n_omega, const double *omegas, int n_tau,
                                      const double *x, const double *w, int spin, double *Pi,
                                      void *stream) {
  return polarizability_tc_api(ctx, N, n_pairs, Bt, delta, n_omega, omegas, n_tau, x, w, spin, Pi, stream, false);
}

ltgw_status ltgw_polarizability_fp8(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt,
                                    const double *delta, int n_omega, const double *omegas, int n_tau,
                                    const double *x, const double *w, int spin, double *Pi, void *stream) {
  return polarizability_tc_api(ctx, N, n_pairs, Bt, delta, n_omega, omegas, n_tau, x, w, spin, Pi, stream, true);
}

ltgw_status ltgw_gemm_emulated(ltgw_ctx *ctx, int m, int n, int64_t k, const double *A, int64_t lda,
                               const double *B, int64_t ldb, double *C, int64_t ldc, int sym, int n_slices,
                               void *stream) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  REQUIRE(ctx, m >= 1 && n >= 1 && k >= 1 && lda >= k && ldb >= k && ldc >= n, "bad sizes");
  REQUIRE(ctx, n_slices >= 2 && n_slices <= 8, "n_slices must be in [2, 8]");
  REQUIRE(ctx, A && C && (sym || B), "a required pointer is NULL");
  REQUIRE(ctx, !sym || (m == n && ldc == n), "sym needs m == n and ldc == n");
  REQUIRE(ctx, m <= 65535, "m must be <= 65535");
  REQUIRE(ctx, is_device_ptr(A) && is_device_ptr(C) && (sym || is_device_ptr(B)), "A, B, C must be device pointers");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  ctx->stats = ltgw_stats{};
  ctx->mark(EV_START, s);
  if (emu_gemm(ctx, m, n, k, A, lda, sym ? A : B, sym ? lda : ldb, C, ldc, sym != 0, emu_digits(n_slices), s) != LTGW_OK)
    return ctx->status();
  ctx->mark(EV_END, s);
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  ctx->stats.ms_total = ctx->ms(EV_START, EV_END);
  ctx->stats.kernel_launches = ctx->launches;
  return check_flags(ctx, s);
}

ltgw_status ltgw_polarizability_emulated(ltgw_ctx *ctx, int N, int64_t n_pairs, const double *Bt,
                                         const double *delta, int n_omega, const double *omegas, int n_tau,
                                         const double *x, const double *w, int spin, int n_slices, double *Pi,
                                         void *stream) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  REQUIRE(ctx, N >= 1 && n_pairs >= 1 && n_omega >= 1 && n_omega <= 256, "bad sizes");
  REQUIRE(ctx, n_tau >= 0 && n_tau <= 32, "n_tau must be in [0, 32]");
  REQUIRE(ctx, spin == 1 || spin == 2, "spin must be 1 or 2");
  REQUIRE(ctx, n_slices >= 2 && n_slices <= 8, "n_slices must be in [2, 8]");
  REQUIRE(ctx, Bt && delta && omegas && Pi && (n_tau == 0 || (x && w)), "a required pointer is NULL");
  REQUIRE(ctx, is_device_ptr(Bt) && is_device_ptr(delta) && is_device_ptr(Pi), "Bt, delta, Pi must be device pointers");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  ctx->stats = ltgw_stats{};
  ctx->mark(EV_START, s);
  std::vector<double> h_om(omegas, omegas + n_omega), h_E((size_t)n_omega * std::max(n_tau, 1));
  for (int j = 0; j < n_omega; ++j)
    for (int k = 0; k < n_tau; ++k) h_E[(size_t)j * n_tau + k] = exp(-h_om[j] * h_om[j] * x[k]);
  double *d_om, *d_x, *d_w, *d_E, *d_M;
  auto layout = [&](Arena &A) {
    d_om = A.take<double>(n_omega);
    d_x = A.take<double>(std::max(n_tau, 1));
    d_w = A.take<double>(std::max(n_tau, 1));
    d_E = A.take<double>(h_E.size());
    d_M = n_tau ? A.take<double>((size_t)n_tau * N * N) : nullptr;
  };
  ctx->a2.begin_sizing();
  layout(ctx->a2);
  if (ctx->a2.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "workspace allocation failed"); return ctx->status(); }
  layout(ctx->a2);
  copy_in(ctx, d_om, h_om.data(), n_omega * sizeof(double), s);
  if (n_tau) {
    copy_in(ctx, d_x, x, n_tau * sizeof(double), s);
    copy_in(ctx, d_w, w, n_tau * sizeof(double), s);
    copy_in(ctx, d_E, h_E.data(), h_E.size() * sizeof(double), s);
  }
  if (ctx->status() != LTGW_OK) return ctx->status();
  if (polarizability_emu(ctx, N, n_pairs, Bt, n_pairs, delta, n_omega, d_om, n_tau, d_x, d_w, d_E, d_M, spin, Pi, s,
                         1, emu_digits(n_slices)) != LTGW_OK)
    return ctx->status();
  ctx->mark(EV_END, s);
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));   // the staged grid lives in the workspace
  ctx->stats.ms_total = ctx->ms(EV_START, EV_END);
  ctx->stats.ms_pi_kernel = ctx->ms(EV_PI0, EV_PI1);
  ctx->stats.kernel_launches = ctx->launches;
  return check_flags(ctx, s);
}

ltgw_status ltgw_screen(ltgw_ctx *ctx, int N, int n_omega, const double *Pi, double *C, void *stream) {
  if (!ctx) return LTGW_ERR_BAD_ARG;
  ctx->reset();
  REQUIRE(ctx, N >= 1 && n_omega >= 1, "bad sizes");
  REQUIRE(ctx, Pi && C && Pi != C, "Pi and C must be distinct non-NULL pointers");
  REQUIRE(ctx, is_device_ptr(Pi) && is_device_ptr(C), "Pi and C must be device pointers");
  LTGW_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t s = (cudaStream_t)stream;
  double *X0;
  auto layout = [&](Arena &A) { X0 = A.take<double>(screen_blocked_scratch(N, n_omega)); };
  ctx->a2.begin_sizing();
  layout(ctx->a2);
  if (ctx->a2.commit() != cudaSuccess) { ctx->fail(LTGW_ERR_NOMEM, "workspace allocation failed"); return ctx->status(); }
  layout(ctx->a2);
  LTGW_CUDA(ctx, cudaMemsetAsync(ctx->flags, 0, FLAG_COUNT * sizeof(int), s));
  if (screen_step(ctx, N, n_omega, Pi, X0, C, s, true) != LTGW_OK) return ctx->status();
  LTGW_CUDA(ctx, cudaStreamSynchronize(s));
  return check_flags(ctx, s);
}

}  // extern "C"
