// solve.cu -- back-substitution R X = C with the R of an H12 factorization.
//
// The paper (Section 1, abstract) names the back-substitution that SLSQP runs
// on the stored factorization at each iteration; it is the textbook
// substitution x_i = (c_i - sum_{j>i} R_ij x_j) / R_ii, i = n-1 .. 0.  An
// exact zero on the diagonal sets x_i = 0 and records SLQR_ERANK.
//
// GPU form: blocks of kTB rows from the bottom.  One launch first inverts
// every diagonal block (independent, one CTA each).  Launch b then updates
// every row block above block b with the now known x of block b (a tiled FP64
// GEMV or GEMM over the right-hand sides), and the CTA of the row block just
// above multiplies its updated right-hand sides by its block's inverse, so
// each launch advances the substitution by one block with no sequential chain
// inside it.  An exact zero R_ii gets a zero row and column in the block
// inverse, which sets x_i = 0 and leaves c_i unused: the same result as the
// substitution that sets x_i = 0 and carries on.
#include "slqr_internal.cuh"

#include <algorithm>

namespace slqr {

constexpr int kTB = 64;    // rows per block of R

// Rinv[b] = inverse of the upper-triangular diagonal block b (kTB x kTB,
// column-major, zero-padded).  Thread j computes column j by back-substitution
// of R y = e_j with the diagonal reciprocals (0 for an exact zero R_ii).
__global__ void __launch_bounds__(kTB)
trsm_inv_kernel(const double *__restrict__ A, int lda, int n, double *__restrict__ Rinv,
                int *status) {
  __shared__ double Rs[kTB][kTB + 1];
  __shared__ double rd[kTB];
  const int b = blockIdx.x, j = threadIdx.x;
  const int row_begin = b * kTB;
  const int rows = min(kTB, n - row_begin);
  for (int c = 0; c < kTB; ++c)
    Rs[j][c] = (j < rows && c < rows && j <= c) ? A[SLQR_IDX(row_begin + j, row_begin + c, lda)]
                                                : 0.0;
  __syncthreads();
  const double d = Rs[j][j];
  rd[j] = (j < rows && d != 0.0) ? 1.0 / d : 0.0;
  const bool zero = (j < rows && d == 0.0);
  __syncthreads();
  double *out = Rinv + (size_t)b * kTB * kTB + (size_t)j * kTB;   // column j
  double y[kTB];
#pragma unroll
  for (int i = 0; i < kTB; ++i) y[i] = 0.0;
  if (j < rows) {
#pragma unroll
    for (int i = kTB - 1; i >= 0; --i) {
      if (i <= j) {
        double t = (i == j) ? 1.0 : 0.0;
#pragma unroll
        for (int k = i + 1; k < kTB; ++k)
          if (k <= j) t = fma(-Rs[i][k], y[k], t);
        y[i] = t * rd[i];
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kTB; ++i) out[i] = y[i];
  if (zero) atomicCAS(status, 0, SLQR_ERANK);
}

// grid: (blocks, ceil(nrhs / RC)), row block t = t_first + blockIdx.x.
// CTA t updates row block t with the x of block b_src (when b_src >= 0), and
// CTA t == b_diag then replaces its right-hand sides by Rinv[t] times them.
// A step is a chain of loads and of FP64 instructions (16 clocks of the SM's
// FP64 pipe each), so a CTA takes few right-hand sides: RC = 4, a thread for
// each row and right-hand side, or RC = 1, a thread for each row and quarter of
// the columns (16 right-hand sides a CTA: 47 us a step whatever their number).
template <int RC>
__global__ void __launch_bounds__(kThreads)
trsm_step_kernel(const double *__restrict__ A, int lda, int n, int nrhs, double *__restrict__ B,
                 int ldb, int t_first, int b_src, int b_diag, const double *__restrict__ Rinv) {
  constexpr int CQ = kThreads / kTB / RC;      // column splits
  constexpr int CW = kTB / CQ;                 // columns of a split
  constexpr int PER = kTB * kTB / kThreads;
  __shared__ double Rs[kTB][kTB + 1];   // R tile (or the block inverse) [col][row]
  __shared__ double Xs[RC][kTB];        // x of block b_src, or the rhs being solved
  __shared__ double part[CQ][kTB];
  const int t = t_first + blockIdx.x;
  const int r0 = blockIdx.y * RC;
  const int tid = threadIdx.x;
  const int row_begin = t * kTB;
  const int rows = min(kTB, n - row_begin);
  const int r = tid & (kTB - 1), g = tid >> 6;
  const int q = RC > 1 ? g : 0, cs = RC > 1 ? 0 : g;
  const bool rhs_ok = r0 + q < nrhs;
  const bool diag = t == b_diag;
  // everything this step reads of R, its inverse and B, in flight at once
  double tile[PER], inv[PER];
  double rhs = 0.0, xsrc = 0.0;
  const int col_begin = b_src * kTB;
  const int cols = b_src >= 0 ? min(kTB, n - col_begin) : 0;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int c = g + u * (kThreads / kTB);
    tile[u] = (r < rows && c < cols) ? A[SLQR_IDX(row_begin + r, col_begin + c, lda)] : 0.0;
  }
  if (diag) {
#pragma unroll
    for (int u = 0; u < PER; ++u)
      inv[u] = Rinv[(size_t)t * kTB * kTB + tid + u * kThreads];
  }
  if (rhs_ok && cs == 0) {
    if (r < rows) rhs = B[SLQR_IDX(row_begin + r, r0 + q, ldb)];
    if (r < cols) xsrc = B[SLQR_IDX(col_begin + r, r0 + q, ldb)];
  }
  // this thread's part of row r of the tile times the vectors in Xs
  auto product = [&]() {
    double a0 = 0.0, a1 = 0.0;
#pragma unroll
    for (int c = 0; c < CW; c += 2) {
      a0 = fma(Rs[cs * CW + c][r], Xs[q][cs * CW + c], a0);
      a1 = fma(Rs[cs * CW + c + 1][r], Xs[q][cs * CW + c + 1], a1);
    }
    a0 += a1;
    if (CQ > 1) {
      part[cs][r] = a0;
      __syncthreads();
      a0 = part[0][r];
#pragma unroll
      for (int s = 1; s < CQ; ++s) a0 += part[s][r];
    }
    return a0;
  };
  if (b_src >= 0) {
#pragma unroll
    for (int u = 0; u < PER; ++u) Rs[g + u * (kThreads / kTB)][r] = tile[u];
    if (cs == 0) Xs[q][r] = xsrc;
    __syncthreads();
    rhs -= product();
    if (!diag && rhs_ok && cs == 0 && r < rows) B[SLQR_IDX(row_begin + r, r0 + q, ldb)] = rhs;
    __syncthreads();
  }
  if (!diag) return;
  // x of the diagonal block = Rinv[t] * (its updated right-hand sides)
#pragma unroll
  for (int u = 0; u < PER; ++u) Rs[g + u * (kThreads / kTB)][r] = inv[u];
  if (cs == 0) Xs[q][r] = (rhs_ok && r < rows) ? rhs : 0.0;
  __syncthreads();
  const double x = product();
  if (rhs_ok && cs == 0 && r < rows) B[SLQR_IDX(row_begin + r, r0 + q, ldb)] = x;
}

}  // namespace slqr

using namespace slqr;

extern "C" slqr_status slqr_solve_r(slqr_ctx *ctx, int n, const double *A, int lda, int nrhs,
                                    double *B, int ldb, void *stream) {
  NvtxRange nvtx_range("slqr_solve_r");
  if (!ctx) return SLQR_EINVAL;
  std::lock_guard<std::recursive_mutex> lk(ctx->mu);
  if (n < 0 || nrhs < 0) return fail(ctx, SLQR_EINVAL, "n=%d nrhs=%d must be >= 0", n, nrhs);
  if (n == 0 || nrhs == 0) return SLQR_OK;
  if (lda < std::max(1, n)) return fail(ctx, SLQR_EINVAL, "lda=%d < n=%d", lda, n);
  if (ldb < std::max(1, n)) return fail(ctx, SLQR_EINVAL, "ldb=%d < n=%d", ldb, n);
  if (!A || !B) return fail(ctx, SLQR_EINVAL, "NULL A or B");
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return fail(ctx, SLQR_ECUDA, "cudaSetDevice: %s", cudaGetErrorString(e));
  cudaStream_t s = (cudaStream_t)stream;
  const int nblk = (n + kTB - 1) / kTB;
  const int RC = nrhs <= 2 ? 1 : 4;
  const int gy = (nrhs + RC - 1) / RC;
  auto step = [&](int blocks, int b_src, int b_diag, double fl) {
    int slot = prof_begin(ctx, s);
    const int first = b_src < 0 ? b_diag : 0;
    if (RC == 1)
      trsm_step_kernel<1><<<dim3(blocks, gy), kThreads, 0, s>>>(
          A, lda, n, nrhs, B, ldb, first, b_src, b_diag, (const double *)ctx->ws.ptr);
    else
      trsm_step_kernel<4><<<dim3(blocks, gy), kThreads, 0, s>>>(
          A, lda, n, nrhs, B, ldb, first, b_src, b_diag, (const double *)ctx->ws.ptr);
    prof_end(ctx, s, slot, kTrsm, fl);
  };
  slqr_status st = ensure_workspace(ctx, (size_t)nblk * kTB * kTB * sizeof(double));
  if (st != SLQR_OK) return st;
  double *Rinv = (double *)ctx->ws.ptr;
  auto rows_of = [&](int blk) { return std::min(kTB, n - blk * kTB); };
  int slot = prof_begin(ctx, s);
  trsm_inv_kernel<<<nblk, kTB, 0, s>>>(A, lda, n, Rinv, ctx->d_status);
  prof_end(ctx, s, slot, kTrsm, 0.0);
  // first launch: only the last diagonal block
  step(1, -1, nblk - 1, (double)rows_of(nblk - 1) * rows_of(nblk - 1) * nrhs);
  // update of rows [0, b*kTB) by block b, then the diagonal block b-1
  for (int b = nblk - 1; b >= 1; --b)
    step(b, b, b - 1, 2.0 * b * kTB * rows_of(b) * nrhs + (double)kTB * kTB * nrhs);
  return check_launch(ctx, "solve_r");
}
