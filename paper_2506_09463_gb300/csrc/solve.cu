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
// inside it.  For few right-hand sides one launch does all of them: a CTA for
// every row block takes the x of the blocks below it as they come
// (trsm_chain_kernel).  An exact zero R_ii gets a zero row and column in the block
// inverse, which sets x_i = 0 and leaves c_i unused: the same result as the
// substitution that sets x_i = 0 and carries on.
#include "slqr_internal.cuh"

#include <algorithm>

namespace slqr {

constexpr int kTB = 64;    // rows per block of R

// The values of x of a block pass between the CTAs of trsm_chain_kernel as their
// own message: a slot holds this signalling-NaN pattern, which no arithmetic result
// has, until its value is there.
constexpr unsigned long long kTrsmUnset = 0x7ff0dead5a5a5a5aull;

// Rinv[b] = inverse of the upper-triangular diagonal block b (kTB x kTB,
// column-major, zero-padded), by back-substitution of R y = e_j with the diagonal
// reciprocals (0 for an exact zero R_ii).  Eight lanes take a column j, lane l the
// entries y_l, y_(l+8), ..; grid (blocks, column groups).  A chain of FP64
// instructions, each 64 clocks after the last: at most 12 for a row of a block
// instead of 64 with a thread to a column (30 us a launch against 115; the SM's pipe is idle
// then).
constexpr int kInvCols = 16;
constexpr int kInvThreads = 8 * kInvCols;
__global__ void __launch_bounds__(kInvThreads)
trsm_inv_kernel(const double *__restrict__ A, int lda, int n, double *__restrict__ Rinv,
                int *status, double *slots, int nslots) {
  __shared__ double Rs[kTB][kTB + 1];          // above the diagonal (zero elsewhere)
  __shared__ double rd[kTB];
  const int b = blockIdx.x, tid = threadIdx.x, l = tid & 7;
  const int j = blockIdx.y * kInvCols + (tid >> 3), top = blockIdx.y * kInvCols + kInvCols;
  // the slots of trsm_chain_kernel back to unset
  if (blockIdx.y == 0)
    for (int i = b * kInvThreads + tid; i < nslots; i += gridDim.x * kInvThreads)
      slots[i] = __longlong_as_double((long long)kTrsmUnset);
  const int row_begin = b * kTB;
  const int rows = min(kTB, n - row_begin);
  for (int idx = tid; idx < kTB * top; idx += kInvThreads) {
    const int i = idx & (kTB - 1), c = idx / kTB;
    const double v = i <= c && c < rows ? A[SLQR_IDX(row_begin + i, row_begin + c, lda)] : 0.0;
    if (i == c) {
      rd[i] = v != 0.0 ? 1.0 / v : 0.0;
      if (blockIdx.y == i / kInvCols && i < rows && v == 0.0) atomicCAS(status, 0, SLQR_ERANK);
    }
    Rs[i][c] = i < c ? v : 0.0;
  }
  __syncthreads();
  double y[kTB / 8];
#pragma unroll
  for (int u = 0; u < kTB / 8; ++u) y[u] = 0.0;
#pragma unroll
  for (int i = kTB - 1; i >= 0; --i) {
    if (i >= top) continue;                    // (uniform)
    double t = (i == j && l == 0) ? 1.0 : 0.0;
#pragma unroll
    for (int u = i / 8; u < kTB / 8; ++u)      // (y is zero up to row i and past row j)
      if (8 * u < top) t = fma(l + 8 * u <= j ? -Rs[i][l + 8 * u] : 0.0, y[u], t);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    t = t * rd[i];
    if ((i & 7) == l && i <= j) y[i / 8] = t;
  }
  double *out = Rinv + (size_t)b * kTB * kTB + (size_t)j * kTB;   // column j
#pragma unroll
  for (int u = 0; u < kTB / 8; ++u) out[l + 8 * u] = y[u];
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
  // this thread's part of row r of the tile times the vectors in Xs, from column
  // `from` on: row r of a block inverse takes no part of the values above it (zero
  // times one that is not finite would reach the rows below)
  auto product = [&](int from) {
    double a0 = 0.0, a1 = 0.0;
#pragma unroll
    for (int c = 0; c < CW; c += 2) {
      const int col = cs * CW + c;
      if (col >= from) a0 = fma(Rs[col][r], Xs[q][col], a0);
      if (col + 1 >= from) a1 = fma(Rs[col + 1][r], Xs[q][col + 1], a1);
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
    rhs -= product(0);
    if (!diag && rhs_ok && cs == 0 && r < rows) B[SLQR_IDX(row_begin + r, r0 + q, ldb)] = rhs;
    __syncthreads();
  }
  if (!diag) return;
  // x of the diagonal block = Rinv[t] * (its updated right-hand sides)
#pragma unroll
  for (int u = 0; u < PER; ++u) Rs[g + u * (kThreads / kTB)][r] = inv[u];
  if (cs == 0) Xs[q][r] = (rhs_ok && r < rows) ? rhs : 0.0;
  __syncthreads();
  const double x = product(r);
  if (rhs_ok && cs == 0 && r < rows) B[SLQR_IDX(row_begin + r, r0 + q, ldb)] = x;
}

__device__ __forceinline__ bool trsm_unset(double v) {
  return (unsigned long long)__double_as_longlong(v) == kTrsmUnset;
}

// The whole substitution of few right-hand sides in one cooperative launch, grid
// (row blocks, right-hand sides): CTA t takes the x of the blocks below it as they
// come, from the last one up, with the next tile of R and its own block's inverse
// already in registers, and hands on its own.  What bounds it is the chain from
// one block to the next: two products of 4096 terms on the SM's FP64 pipe (2048
// clocks each) and the way through L2, about 3 us a block; a launch for every block
// took 12.4 us.
__global__ void __launch_bounds__(kThreads, 1)
trsm_chain_kernel(const double *__restrict__ A, int lda, int n, double *__restrict__ B, int ldb,
                  const double *__restrict__ Rinv, double *slots, int *status, unsigned spin) {
  constexpr int CW = kTB * kTB / kThreads;     // columns of a thread
  __shared__ double Xs[2][kTB];
  __shared__ double part[kThreads / kTB][kTB];
  const int nblk = gridDim.x, t = nblk - 1 - (int)blockIdx.x, q = blockIdx.y;
  const int tid = threadIdx.x, r = tid & (kTB - 1), g = tid >> 6;
  const int row_begin = t * kTB, rows = min(kTB, n - row_begin);
  double *xs = slots + (size_t)q * nblk * kTB;
  double tile[CW], next[CW], inv[CW], rhs = 0.0, acc = 0.0;
  auto load = [&](int b, double (&dst)[CW]) {
    const int cols = min(kTB, n - b * kTB);
#pragma unroll
    for (int u = 0; u < CW; ++u) {
      const int c = g * CW + u;
      dst[u] = (r < rows && c < cols) ? A[SLQR_IDX(row_begin + r, b * kTB + c, lda)] : 0.0;
    }
  };
  if (t < nblk - 1) load(nblk - 1, tile);
#pragma unroll
  for (int u = 0; u < CW; ++u) inv[u] = Rinv[(size_t)t * kTB * kTB + (g * CW + u) * kTB + r];
  if (g == 0 && r < rows) rhs = B[SLQR_IDX(row_begin + r, q, ldb)];
  bool dead = false;
  for (int b = nblk - 1; b > t; --b) {
    if (b - 1 > t) load(b - 1, next);
    if (g == 0) {
      const double *slot = xs + (size_t)b * kTB + r;
      double v;
      for (unsigned it = 0;; ++it) {
        asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(slot) : "memory");
        if (!trsm_unset(v) || dead) break;
        // (past the context's limit it reports and goes on waiting, as the blocks above
        // wait for this one's x)
        if (it == spin) record_status(status, SLQR_ETIMEOUT);
        if (it > kSpinLimit) dead = true;
      }
      Xs[b & 1][r] = v;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < CW; ++u) acc = fma(tile[u], Xs[b & 1][g * CW + u], acc);
#pragma unroll
    for (int u = 0; u < CW; ++u) tile[u] = next[u];
  }
  auto total = [&](double v) {                 // over the quarters of the columns
    part[g][r] = v;
    __syncthreads();
    return g == 0 ? part[0][r] + part[1][r] + (part[2][r] + part[3][r]) : 0.0;
  };
  const double below = total(acc);
  if (g == 0) Xs[t & 1][r] = rhs - below;
  __syncthreads();
  acc = 0.0;
#pragma unroll
  for (int u = 0; u < CW; ++u)                 // (from the diagonal on, as in the steps)
    if (g * CW + u >= r) acc = fma(inv[u], Xs[t & 1][g * CW + u], acc);
  const double x = total(acc);
  if (g == 0) {
    const double v = trsm_unset(x) ? __longlong_as_double(0x7fffffffffffffffll) : x;
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(xs + (size_t)t * kTB + r), "d"(v)
                 : "memory");
    if (r < rows) B[SLQR_IDX(row_begin + r, q, ldb)] = x;
  }
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
  // Up to four right-hand sides go in one launch where a CTA for every block and
  // right-hand side is resident and the slots fit beside the inverses (2048 rows,
  // one right-hand side: 139 us with the inverses against 409 in a launch a block).  More of them
  // share the tiles of a launch a block.
  const size_t inv_bytes = (size_t)nblk * kTB * kTB * sizeof(double);
  const int nslots = nblk * kTB * nrhs;
  bool chain = nblk > 1 && nrhs <= 4 && nblk * nrhs <= ctx->num_sms;
  slqr_status st = ensure_workspace(ctx, inv_bytes + (chain ? nslots * sizeof(double) : 0));
  if (st != SLQR_OK && chain) {
    chain = false;
    st = ensure_workspace(ctx, inv_bytes);
  }
  if (st != SLQR_OK) return st;
  double *Rinv = (double *)ctx->ws.ptr;
  double *slots = Rinv + (size_t)nblk * kTB * kTB;
  auto rows_of = [&](int blk) { return std::min(kTB, n - blk * kTB); };
  int slot = prof_begin(ctx, s);
  trsm_inv_kernel<<<dim3(nblk, kTB / kInvCols), kInvThreads, 0, s>>>(A, lda, n, Rinv, ctx->d_status, slots, chain ? nslots : 0);
  prof_end(ctx, s, slot, kTrsm, 0.0);
  if (chain) {
    slot = prof_begin(ctx, s);
    int *status = ctx->d_status;
    unsigned spin = ctx->spin_limit;
    void *args[] = {&A, &lda, &n, &B, &ldb, &Rinv, &slots, &status, &spin};
    e = cudaLaunchCooperativeKernel((const void *)trsm_chain_kernel, dim3(nblk, nrhs),
                                    dim3(kThreads), args, 0, s);
    if (e != cudaSuccess)
      return fail(ctx, SLQR_ECUDA, "back-substitution launch: %s", cudaGetErrorString(e));
    prof_end(ctx, s, slot, kTrsm, (double)n * n * nrhs);
    return check_launch(ctx, "solve_r");
  }
  // first launch: only the last diagonal block
  step(1, -1, nblk - 1, (double)rows_of(nblk - 1) * rows_of(nblk - 1) * nrhs);
  // update of rows [0, b*kTB) by block b, then the diagonal block b-1
  for (int b = nblk - 1; b >= 1; --b)
    step(b, b, b - 1, 2.0 * b * kTB * rows_of(b) * nrhs + (double)kTB * kTB * nrhs);
  return check_launch(ctx, "solve_r");
}
