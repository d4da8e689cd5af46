// tc_fp64.cu -- the two FP64 products of the compact-WY trailing update
//   W = V^T X   and   X -= V W'
// on the 5th-generation tensor cores, by error-free splitting (the scheme of
// Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59, 2012): every operand
// is written as an integer times a power of two per vector, the integer in
// balanced base-256 digits, and products of digit matrices are summed exactly.
//
//   x = 2^(e-55) sum_i d_i 256^(6-i),   d_i in [-128, 127], i = 0..6
//
// e is the exponent of the vector's largest entry, so the rounding of x to
// this grid is at most 2^(e-56): a quarter of the half-ulp that one FP64
// operation on that largest entry commits, but more than FP64's on entries far
// below it.  Results whose terms are all far below the product of the scales are
// formed again in FP64 (fx_digits.cuh has the rule, each kernel its bound).  The
// digits are exact in FP16.  A product
// of two digits is an integer of at most 2^14 in magnitude; the tensor core
// sums them in FP32, which is exact while the sum stays below 2^24: at most
// 7 pairs of digits of the same order i + j, over at most 128 terms.  The 34
// pairs with i + j <= 7 are kept (the first dropped ones are 2^-8 times the
// rounding above), one accumulator per order in tensor memory, and the eight
// orders are put together in integer arithmetic before one rounding to FP64.
// The residual ||A - Q R|| / ||A|| in 128-bit arithmetic: 3.73e-16 with these
// kernels, 4.92e-16 with the DFMA kernels of factor.cu (700 x 300 Gaussian),
// 3.08e-16 against 3.38e-16 (3000 x 260), 2.96e-16 against 2.98e-16
// (16384 x 260).
//
// Why: the FP64 pipe of GB300 does 2 DFMA per SM and clock, 1.2 TFLOP/s, and
// the products ran at 82-91% of that.  34 FP16 products cost 34/1834 of the
// same work at the tensor rate, so the products are bound by memory, by the
// digit extraction and by the reassembly instead.  Both products over a whole
// 8192 x 8192 factorization: 663 ms on the FP64 pipe, 50 ms here.
//
// Operand layout: K-major shared-memory images of the digit matrices, written
// by the producing kernel in the exact (swizzled) form the MMA reads, so that
// a tile is one bulk copy:
//   V1  per 32 rows:     [digit][reflector a][32 rows]   64-byte rows, SWIZZLE_64B
//   V2  per 128 rows:    [digit][row][64 reflectors]    128-byte rows, SWIZZLE_128B
//   W   per 32 columns:  [digit][column][64 reflectors] 128-byte rows, SWIZZLE_128B
// The digit matrices of one operand are stacked, so A_i times all B_j with
// j <= 7 - i is one MMA (N = 64 or 32 per digit) whose result columns are the
// accumulators of the orders i, i + 1, ...
#include "fx_digits.cuh"
#include "tc_common.cuh"

#include <cuda_fp16.h>
#include <algorithm>
#include <climits>

namespace slqr {

constexpr int kFxWorkers = 16;                // warps that split and reassemble; one more issues MMAs
constexpr int kFxThreads = 32 * (kFxWorkers + 1);
constexpr int kFxV1Chunk = kFxD * 64 * 64;            // 28672 B: 32 rows
constexpr int kFxV2Tile = kFxD * 128 * 128;           // 114688 B: 128 rows
constexpr int kFxWTile = kFxD * 32 * 128;             // 28672 B: 32 columns
constexpr int kFxXStage = kFxD * 128 * 64;            // 57344 B: 128 columns x 32 rows
constexpr int kFxStage = kFxXStage + kFxV1Chunk;
constexpr size_t kFxVtxSmem = 2 * (size_t)kFxStage + 1024;
constexpr int kFxMaxPer = 32;                // column tiles of a CTA of the update
constexpr int kFxLostWords = kFxWorkers * 8; // of a column tile: a warp's 8 columns, a bit a row
constexpr size_t kFxUpdSmem =
    (size_t)kFxV2Tile + 2 * kFxWTile + 1024 + kFxMaxPer * kFxLostWords * sizeof(unsigned);

// D = F32, A = B = F16, both K-major, M = 128; N is added per MMA
constexpr uint32_t kIdescF16 = (1u << 4) | ((128u >> 4) << 24);

__device__ __forceinline__ uint32_t fx_idesc(int n) { return kIdescF16 | ((uint32_t)(n >> 3) << 17); }

// The panel's V in FP64: rows < nbw in Vtop (ld 64, zero above the diagonal), the
// others at tail[i + a ld]
struct FxPanel {
  const double *Vtop, *tail;
  int ld, nbw, M, skip;                // skip > 0: [L^T; C], the top rows hold the pivots only
};

// out[k] = sum_i V(i, a0 + k) x_i for k < 8 on the FP64 pipe, by a warp, for C columns x
// (at the panel's first row, ldx apart; their results 64 apart).  Bound by the pipe: eight
// loads of V (coalesced) to 8 C FMAs of 16 clocks each, where V comes from L2 ([L^T; C] of
// 4000 + 1000 with L's rows over 10^6: 37 ms with one column, 31 with two).
template <int C>
static __device__ __noinline__ void fx_dots8(FxPanel p, const double *x, size_t ldx, int a0,
                                             double *out) {
  const int lane = threadIdx.x & 31, na = min(8, p.nbw - a0);
  double acc[C][8];
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[c][k] = 0.0;
  auto add = [&](const double *v, size_t ld, const double (&xi)[C]) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < na) {
        const double t = v[k * ld];
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c][k] = fma(t, xi[c], acc[c][k]);
      }
  };
  if (p.skip > 0) {                                    // (the pivots only)
    if (lane < na) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k == lane)
#pragma unroll
          for (int c = 0; c < C; ++c) acc[c][k] = p.Vtop[(a0 + k) * 65] * x[c * ldx + a0 + k];
    }
  } else {
    for (int i = lane; i < p.nbw; i += 32) {
      double xi[C];
#pragma unroll
      for (int c = 0; c < C; ++c) xi[c] = x[c * ldx + i];
      add(p.Vtop + a0 * 64 + i, 64, xi);
    }
  }
  // (128 rows of x at a time: where they are zero, as in a banded or block matrix, V is
  // not read)
  const double *v = p.tail + (size_t)a0 * p.ld;
  for (int i0 = p.nbw + lane; i0 - lane < p.M; i0 += 128) {
    double xi[4][C];
    bool any = false;
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        xi[t][c] = i0 + 32 * t < p.M ? x[c * ldx + p.skip + i0 + 32 * t] : 0.0;
        any |= (unsigned long long)__double_as_longlong(xi[t][c]) << 1 != 0;
      }
    if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
    for (int t = 0; t < 4; ++t) add(v + min(i0 + 32 * t, p.M - 1), p.ld, xi[t]);
  }
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int k = 0; k < 8; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[c][k] += __shfl_xor_sync(0xffffffffu, acc[c][k], o);
      if (lane == 0) out[c * 64 + k] = acc[c][k];
    }
  __syncwarp();
}
// the same for this thread's reflector a, of a panel of few rows
constexpr int kFxFewRows = 192;
static __device__ __noinline__ double fx_dot1(FxPanel p, const double *x, int a) {
  double s = p.Vtop[a * 65] * x[a];
  if (p.skip == 0) {
#pragma unroll 4
    for (int i = a + 1; i < p.nbw; ++i) s = fma(p.Vtop[a * 64 + i], x[i], s);
  }
  const double *v = p.tail + (size_t)a * p.ld;
#pragma unroll 4
  for (int i = p.nbw; i < p.M; ++i) s = fma(v[i], x[p.skip + i], s);
  return s;
}

// sum_a V(i, a) W'(a, c) for four columns c .. c + 3 (w: W' of column c, nc of them) and
// this thread's row
struct FxFour { double v[4]; };
static __device__ __noinline__ FxFour fx_row4(FxPanel p, const double *w, int nc, int i) {
  FxFour s = {{0.0, 0.0, 0.0, 0.0}};
  const double *v = i < p.nbw ? p.Vtop + i : p.tail + min(i, p.M - 1);
  const size_t ld = i < p.nbw ? 64 : p.ld;
#pragma unroll 4
  for (int a = 0; a < p.nbw; a += 2) {                 // (W' is zero past nbw, V not read there)
    const double t0 = v[a * ld], t1 = a + 1 < p.nbw ? v[(a + 1) * ld] : 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double2 u = *(const double2 *)(w + min(k, nc - 1) * 64 + a);
      s.v[k] = fma(t1, u.y, fma(t0, u.x, s.v[k]));
    }
  }
  return s;
}

// The entries of X -= V W' that fx_upd_kernel's digits left out, by the warp (of its 32
// rows, i this thread's) that found them: rows[t * kFxLostWords + k] for column c0 + 32 t + k.
static __device__ __noinline__ void fx_lost_entries(FxPanel p, const double *Wf, double *X, int ldx,
                                                    int N, int i, int c0, int T,
                                                    const unsigned *rows, unsigned *cnext) {
  const int lane = threadIdx.x & 31;
  for (int b = 0; b < 2 * T; b += 32) {                  // a lane to a tile's four columns
    const int mine = b + lane;
    const uint4 m = mine < 2 * T
                        ? *(const uint4 *)(rows + (mine >> 1) * kFxLostWords + (mine & 1) * 4)
                        : make_uint4(0, 0, 0, 0);
    unsigned todo = __ballot_sync(0xffffffffu, (m.x | m.y | m.z | m.w) != 0);
    for (; todo; todo &= todo - 1) {
      const int src = __ffs(todo) - 1, t = (b + src) >> 1, u = (b + src) & 1;
      const int c = c0 + 32 * t + 4 * u;
      unsigned w[4] = {m.x, m.y, m.z, m.w};
      double *xp = X + i + (i >= p.nbw ? p.skip : 0) + (size_t)c * ldx;
      int n = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        w[k] = __shfl_sync(0xffffffffu, w[k], src);
        n += __popc(w[k]);
      }
      auto store = [&](int k, double s) {
        const double v = xp[(size_t)k * ldx] - s;
        xp[(size_t)k * ldx] = v;
        if (cnext && i >= 64) atomicMax(cnext + c + k, fx_hi(v));
      };
      if (n > 16) {
        const FxFour s = fx_row4(p, Wf + (size_t)c * 64, min(4, N - c), i);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (w[k] >> lane & 1) store(k, s.v[k]);
      } else {
        // four entries at a time, two reflectors a lane: one round trip of loads
        for (; n > 0; n -= 4) {
          int row[4], col[4];
          double s[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            row[e] = -1;
            col[e] = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (row[e] < 0 && w[k]) {
                row[e] = __ffs(w[k]) - 1;
                col[e] = k;
                w[k] &= w[k] - 1;
              }
            const int r = i - lane + max(row[e], 0);
            const double *v = r < p.nbw ? p.Vtop + r : p.tail + min(r, p.M - 1);
            const size_t ld = r < p.nbw ? 64 : p.ld;
            const double *wc = Wf + (size_t)min(c + col[e], N - 1) * 64;
            s[e] = 0.0;
            if (row[e] >= 0) {
              if (lane < p.nbw) s[e] = v[lane * ld] * wc[lane];
              if (lane + 32 < p.nbw) s[e] = fma(v[(lane + 32) * ld], wc[lane + 32], s[e]);
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], o);
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (lane == row[e]) store(col[e], s[e]);
        }
      }
    }
  }
}

// The Gram terms of a panel beside (or, with no columns, instead of) V^T X
struct FxGram {
  unsigned long long *sum;             // [c][a], zero before; NULL: none
  unsigned *arrived;                   // zero before
  FxPanel p;
  double *part;                        // [slice][c (c - 1) / 2 + a]: terms formed in FP64
  double *G;                           // the compact-WY store's G (tau follows it)
  double *Gt;                          // Gt and tau for the substitution (kFxGt doubles)
  int slices, RS;                      // CTAs, rows of each (a multiple of 128)
  int vtx_slices;                      // row slices of V^T X
};

// K-major operand with 64-byte rows, SWIZZLE_64B, 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;                    // SWIZZLE_64B
  return d;
}

__device__ __forceinline__ void fx_mma(uint32_t d, uint64_t ad, uint64_t bd, int n, bool accum) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
               " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
               :: "r"(d), "l"(ad), "l"(bd), "r"(fx_idesc(n)), "r"(accum ? 1u : 0u) : "memory");
}

__device__ __forceinline__ void fx_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               :: "r"(smem_u32(bar)) : "memory");
}

// Row (of 32) of slot 8 rg + k along K in V1 and in the digits of X: a thread of
// V^T X reads 8 rows of a column, two at a time, and its four neighbours' pairs
// are adjacent, so that a load covers whole sectors.
__device__ __forceinline__ int fx_row(int rg, int k) { return (k >> 1) * 8 + rg * 2 + (k & 1); }

// 1-D bulk copy (16-byte aligned, a multiple of 16 bytes) counted on an mbarrier
__device__ __forceinline__ void fx_bulk(uint32_t dst, const void *src, uint32_t bytes,
                                        uint64_t *bar) {
  const uint32_t b = smem_u32(bar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes"
               " [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(b) : "memory");
}

// Four accumulators of every order for this thread's TMEM lane: order o at
// addr + o * stride columns.
__device__ __forceinline__ void fx_ld_orders(uint32_t (&r)[kFxOrders][4], uint32_t addr,
                                             uint32_t stride) {
#pragma unroll
  for (int o = 0; o < kFxOrders; ++o)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[o][0]), "=r"(r[o][1]), "=r"(r[o][2]), "=r"(r[o][3])
                 : "r"(addr + (uint32_t)o * stride));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// --------------------------------------------------------------------------
// Column maxima (high words) of the rows each panel sees: cmax[p][c] over the
// rows [k0, m) of panel p that no earlier panel changes.  A dense matrix: all
// rows for panel 0 (later panels' maxima come from the update kernel).  A
// stacked [L^T; C]: panel p's diagonal rows, panel 0 also all rows of C.
// grid: (columns, row slices); columns from c_first.
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
fx_colmax_kernel(const double *__restrict__ X, int ldx, int r0, int r1, int c_first, int n,
                 unsigned *__restrict__ cmax) {
  const int c = c_first + blockIdx.x;
  if (c >= n) return;
  const int rows = r1 - r0;
  const int per = (rows + gridDim.y - 1) / gridDim.y;
  const int lo = r0 + blockIdx.y * per, hi = min(r1, lo + per);
  unsigned mx = 0;
  for (int i = lo + threadIdx.x; i < hi; i += 256) mx = max(mx, fx_hi(X[SLQR_IDX(i, c, ldx)]));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(cmax + c, mx);
}

// stacked: panel p's rows 64 p .. 64 p + 63 of the top block of `top` rows;
// upper: of its upper triangle only (the rest is zero and not read)
__global__ void __launch_bounds__(256)
fx_colmax_diag_kernel(const double *__restrict__ A, int lda, int n, int top, int upper,
                      unsigned *__restrict__ cmax) {
  const int p = blockIdx.y, c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n) return;
  unsigned mx = 0;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int r = p * 64 + lane + 32 * t;
    if (r < top && (!upper || r <= c)) mx = max(mx, fx_hi(A[SLQR_IDX(r, c, lda)]));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0 && mx) atomicMax(cmax + (size_t)p * n + c, mx);
}

// --------------------------------------------------------------------------
// Digits of the panel's V: both images and the row exponents of the second.
// Reflector a is scaled by its pivot entry: |up| >= the norm of the tail, so it
// is the largest entry, and for a tall panel far above all others.  For V^T X
// it may therefore stick out of the leading digit by three bits (1024 instead
// of 128), which leaves the tail 8 times finer steps.  The sums stay exact:
// the leading digits of one reflector have a 2-norm of at most sqrt(2) 1024,
// so by Cauchy-Schwarz their absolute sum over 128 rows is at most 128^2, what
// 128 rows of ordinary digits may have.  For X -= V W' each row is scaled once
// more by its own largest (scaled) entry.
// One CTA per 32 rows.  Bound by latency (one pass over M x 64 doubles).
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
fx_vsplit_kernel(const double *__restrict__ A, int lda, const double *__restrict__ Vtop, int k0,
                 int nbw, int M, int skip, unsigned char *__restrict__ V1,
                 unsigned char *__restrict__ V2, int *__restrict__ erow) {
  __shared__ double t[64][33];
  __shared__ int s_f[64];
  const int tid = threadIdx.x, i0 = blockIdx.x * 32;
  {
    const int r = tid & 31, i = i0 + r;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int a = (tid >> 5) + 8 * u;
      v[u] = 0.0;
      if (i < M && a < nbw)
        v[u] = (i < nbw) ? Vtop[i + a * 64] : A[SLQR_IDX(k0 + skip + i, k0 + a, lda)];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) t[(tid >> 5) + 8 * u][r] = v[u];
  }
  if (tid < 64) {
    const double up = Vtop[tid * 65];
    // a skipped reflector (up = 0) takes no part: all digits zero
    s_f[tid] = (up == 0.0) ? kFxNonFinite : fx_exp_of_hi(fx_hi(up));
  }
  __syncthreads();
  {
    const int a = tid >> 2, rg = tid & 3;
    const int f = s_f[a];
    unsigned long long y[8];
    __align__(16) __half lead[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      int d0;
      y[k] = fx_digits_wide(f == kFxNonFinite ? 0.0 : t[a][fx_row(rg, k)], f - 3, &d0);
      lead[k] = __int2half_rn(d0);
    }
    unsigned char *dst = V1 + (size_t)blockIdx.x * kFxV1Chunk + a * 64 +
                         ((rg * 16) ^ (((a >> 1) & 3) << 4));
    *(uint4 *)dst = *(const uint4 *)lead;
#pragma unroll
    for (int i = 1; i < kFxD; ++i) *(uint4 *)(dst + i * 4096) = fx_pack8(y, i);
  }
  {
    const int r = tid >> 3, ag = tid & 7;
    int key = kFxZero;
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int f = s_f[ag * 8 + k];
      v[k] = f == kFxNonFinite ? 0.0 : t[ag * 8 + k][r];
      const int kk = fx_key(v[k], 0);
      if (kk != kFxZero) key = max(key, kk - f * (1 << 20));
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    const int e = (key == kFxZero) ? kFxZeroExp : fx_exp(key);
    unsigned long long y[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int f = s_f[ag * 8 + k];
      y[k] = fx_digits(v[k], (f == kFxNonFinite ? 0 : f) + e);
    }
    const int rr = (i0 + r) & 127;
    unsigned char *dst = V2 + (size_t)((i0 + r) >> 7) * kFxV2Tile + rr * 128 +
                         ((ag * 16) ^ ((rr & 7) << 4));
#pragma unroll
    for (int i = 0; i < kFxD; ++i) *(uint4 *)(dst + i * 16384) = fx_pack8(y, i);
    if (ag == 0) erow[i0 + r] = e;
  }
}

__device__ __forceinline__ void fx_mbar_init(uint64_t *bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void fx_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// whole-warp wait (the lanes leave together)
__device__ __forceinline__ bool fx_wait(uint64_t *bar, int phase) {
  return __all_sync(0xffffffffu, mbar_wait(smem_u32(bar), (uint32_t)(phase & 1)));
}

// --------------------------------------------------------------------------
// Strict upper triangle of G = V^T V of the panel, from the digit images V1 on
// both sides: gram[c][a] += the sums over this CTA's rows (integers, so the
// order of the atomic adds does not matter), and the CTA that arrives last
// writes G to the compact-WY store and tau G for the substitution.  Digits i and i + 1 of V are the two halves
// of the M side (rows 64 .. 127 of A are digit i + 1, one order up), the stacked
// digits the N side.  With V's wide leading digits the sums are still exact: by
// Cauchy-Schwarz a product with them is at most (sqrt(2) 1024)^2 over all rows.
// G is known to 2^-58 of |up_a up_c|; the panel's own sums in FP64 cost it 0.5
// us of each column step.  That is below FP64's own error in a sum of products unless
// their magnitudes add up to far less (columns whose large entries are in different
// rows).  Every CTA forms the sums of |products| over the panel's first kFxGramSample
// rows from the leading digits (mma.sync), a lower bound; the terms whose bound is below
// 2^-7 |up_a up_c| (for M > 512 rows 512 / M of it, as of the sum of all) are formed in
// FP64, each CTA's rows by itself, and added by the last one.  Without structure the
// sample holds 0.16 to 0.64 of 256 / M.
// Called by every thread of CTAs (gridDim.x - 1, y), y < slices.
// --------------------------------------------------------------------------
constexpr int kFxGramSample = 256;
// the line in products of leading digits: with the sample's share of M rows
__device__ __forceinline__ float fx_gram_line(int M) {
  return (float)(1 << (20 - 7)) * 512.f / (float)max(M, 512);
}
constexpr int kFxGramChunk = kFxV1Chunk + 4096;       // (a zero digit 7 behind each chunk)
constexpr int kFxGramShift = 56;                      // units of 2^56 digit products

__device__ __noinline__ void fx_gram_block(const FxGram &gr, int nbw, int M,
                                           const unsigned char *V1, unsigned char *base,
                                           uint32_t taddr, uint64_t *s_full, uint64_t *s_acc,
                                           uint64_t *s_sample, const int *s_fa, int *status) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i_begin = blockIdx.y * gr.RS, i_end = min(M, i_begin + gr.RS);
  const int B = (i_end - i_begin + 127) / 128;
  for (int idx = tid; idx < 4 * 4096 / 16; idx += kFxThreads)
    *(uint4 *)(base + (idx >> 8) * kFxGramChunk + kFxV1Chunk + (idx & 255) * 16) =
        make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __shared__ unsigned s_low[64][2], s_any;              // terms to be formed in FP64, by column
  unsigned char *sample = base + 4 * kFxGramChunk;
  const int chunks = min(kFxGramSample / 32, (M + 127) / 128 * 4);
  if (tid < 128) s_low[tid >> 1][tid & 1] = 0;
  if (tid == 128) s_any = 0;
  if (tid == 0) {
    const uint32_t bar = smem_u32(s_sample);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 ::"r"(bar), "r"(chunks * 4096) : "memory");
    for (int u = 0; u < chunks; ++u)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes"
                   " [%0], [%1], %2, [%3];"
                   ::"r"(smem_u32(sample + u * 4096)), "l"(V1 + (size_t)u * kFxV1Chunk), "r"(4096),
                   "r"(bar) : "memory");
  }
  __syncthreads();
  const int q = warp & 3, h = warp >> 2;               // workers: TMEM lanes, 16 columns
  const int a = (q * 32 + lane) & 63;
  const bool upper = q >= 2;                            // lanes of digit i + 1
  long long tot[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) tot[k] = 0;
  bool ok = true;
  for (int b = 0; b < B && ok; ++b) {
    if (tid == 0) {
      const uint32_t bar = smem_u32(s_full);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                   ::"r"(bar), "r"(4 * kFxV1Chunk) : "memory");
      for (int u = 0; u < 4; ++u)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes"
                     " [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(base + u * kFxGramChunk)),
                     "l"(V1 + (size_t)(i_begin / 32 + b * 4 + u) * kFxV1Chunk), "r"(kFxV1Chunk),
                     "r"(bar) : "memory");
      if (mbar_wait(bar, (uint32_t)(b & 1))) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int u = 0; u < 4; ++u) {
          const uint32_t v = smem_u32(base + u * kFxGramChunk);
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            const bool acc = u > 0 || ks > 0;
            auto piece = [&](int i, int n0, int n, bool ac) {
              fx_mma(taddr + (uint32_t)(i * 64 + n0), sw64_desc(v + i * 4096 + ks * 32),
                     sw64_desc(v + n0 * 64 + ks * 32), n, ac);
            };
            piece(0, 0, 256, acc);  piece(0, 256, 192, acc);
            piece(2, 0, 192, true); piece(2, 192, 128, true); piece(2, 320, 64, acc);
            piece(4, 0, 256, true);
            piece(6, 0, 128, true);
          }
        }
        fx_commit(s_acc);
      }
    }
    __syncwarp();
    if (b == 0) ok = fx_wait(s_sample, 0);
    if (b == 0 && ok && warp < kFxWorkers) {
      // beside the first MMAs: 16 x 16 of the 64 x 64 sums to a warp (at most 2^21 by
      // Cauchy-Schwarz, so exact)
      const int gid = lane >> 2, tq = lane & 3, ar = q * 16 + gid, cr = h * 16 + gid;
      const float line = fx_gram_line(M);
      float mag[2][4] = {};
      for (int u = 0; u < chunks; ++u) {
        auto pair = [&](int row, int grp) {
          return fx_abs2(*(const uint32_t *)(sample + u * 4096 + row * 64 +
                                             ((grp * 16) ^ (((row >> 1) & 3) << 4)) + tq * 4));
        };
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          const uint32_t fa[4] = {pair(ar, 2 * ks), pair(ar + 8, 2 * ks), pair(ar, 2 * ks + 1),
                                  pair(ar + 8, 2 * ks + 1)};
#pragma unroll
          for (int t = 0; t < 2; ++t)
            fx_mma16816(mag[t], fa, pair(cr + 8 * t, 2 * ks), pair(cr + 8 * t, 2 * ks + 1));
        }
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = q * 16 + gid + 8 * ((k >> 1) & 1), c = h * 16 + 8 * (k >> 2) + 2 * tq + (k & 1);
        if (r < c && c < nbw && mag[k >> 2][k & 3] < line)
          atomicOr(&s_low[c][r >> 5], 1u << (r & 31)), s_any = 1;
      }
    }
    ok = fx_wait(s_acc, b) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok && warp < kFxWorkers) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        uint32_t r[kFxOrders][4];
        fx_ld_orders(r, taddr + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * 16 + u * 4), 64);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          // lower lanes: block t is order t; upper lanes: order t + 1 (8 dropped)
          if (upper) r[7][k] = 0;
          const long long x = fx_four(r, 0, k), y = fx_four(r, 4, k);
          tot[u * 4 + k] += upper ? (x << 8) + ((y + (1 << 23)) >> 24)
                                  : (x << 16) + ((y + (1 << 15)) >> 16);
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  if (!ok && tid == 0) {
    mbar_wait(smem_u32(s_sample), 0);                       // let the copies in flight land
    mbar_wait(smem_u32(s_full), (uint32_t)((B - 1) & 1));
    atomicCAS(status, 0, SLQR_ETIMEOUT);
  }
  // (s_low is complete: a barrier ended each block)
  if (warp < kFxWorkers) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int c = h * 16 + k;
      if (a < c && !(s_low[c][a >> 5] >> (a & 31) & 1))
        atomicAdd(gr.sum + c * 64 + a, (unsigned long long)tot[k]);
    }
  }
  if (s_any) {
    // this CTA's rows of those terms in FP64: 64 rows at a time through shared memory (the
    // chunks are used up), a thread for column c and the a = a8, a8 + 8, ..
    double *vs = (double *)base;                        // [64][65]
    const int c = tid >> 3, a8 = tid & 7;
    double g[8];
    unsigned mine = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      g[k] = 0.0;
      if (warp < kFxWorkers) mine |= (s_low[c][k >> 2] >> (a8 + 8 * (k & 3)) & 1) << k;
    }
    // ([L^T; C]: no two reflectors meet in the top rows)
    for (int i0 = gr.p.skip > 0 ? max(i_begin, nbw) : i_begin; i0 < i_end; i0 += 64) {
      const int rows = min(64, i_end - i0);
      __syncthreads();
      for (int idx = tid; idx < 64 * 64; idx += kFxThreads) {
        const int r = idx & 63, aa = idx >> 6, i = i0 + r;
        double v = 0.0;
        if (r < rows && aa < nbw)
          v = i < nbw ? gr.p.Vtop[aa * 64 + i] : gr.p.tail[(size_t)aa * gr.p.ld + i];
        vs[r * 65 + aa] = v;
      }
      __syncthreads();
      if (mine)
        for (int r = 0; r < rows; ++r) {
          const double x = vs[r * 65 + c];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (mine >> k & 1) g[k] = fma(vs[r * 65 + a8 + 8 * k], x, g[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (mine >> k & 1)
        gr.part[(size_t)blockIdx.y * 2016 + c * (c - 1) / 2 + a8 + 8 * k] = g[k];
  }
  __threadfence();
  __syncthreads();
  __shared__ int s_last;
  if (tid == 0) s_last = atomicAdd(gr.arrived, 1u) == (unsigned)gr.slices - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int idx = tid; idx < 64 * 64; idx += kFxThreads) {
    const int c = idx >> 6, aa = idx & 63;
    double g = 0.0;
    if (aa < c && c < nbw) {
      const int fa = s_fa[aa], fc = s_fa[c];
      const long long t = (long long)__ldcg(gr.sum + idx);
      g = (fa == kFxNonFinite || fc == kFxNonFinite)
              ? __longlong_as_double(0x7ff8000000000000ll)
              : fx_scale((double)t, fa + fc - 110 + kFxGramShift);
      if (s_low[c][aa >> 5] >> (aa & 31) & 1)            // (a NaN stays one)
        for (int s = 0; s < gr.slices; ++s)
          g += __ldcg(gr.part + (size_t)s * 2016 + c * (c - 1) / 2 + aa);
    }
    gr.G[idx] = g;
    const double tau = gr.G[64 * 64 + aa];               // (of the panel's own kernel)
    gr.Gt[aa * 64 + c] = (aa < c && c < nbw) ? tau * g : 0.0;
    if (c == 0) gr.Gt[64 * 64 + aa] = aa < nbw ? tau : 0.0;
  }
}

// --------------------------------------------------------------------------
// W_part[s][c][a] = sum over the rows i of slice s of X(i, c) V(i, a):
// 128 columns of X on the M side, the digits of the 64 reflectors stacked on
// the N side, 32 rows per stage, two stages.  The sixteen worker warps read X
// as FP64 and split it (a thread owns 8 consecutive rows of a column); V's
// digits come by bulk copy; warp 16 issues the MMAs.  Every 128 rows the eight
// accumulators (all of tensor memory) are drained into 96-bit integer totals;
// the workers split the first chunk of the next 128 rows before they wait for
// that, so the splitting of a chunk runs beside the MMAs of the one before.
// grid: (ceil(N / 128), S), slices of RS rows (a multiple of 128); with gr.sum
// one more column of CTAs for the Gram terms (fx_gram_block).
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(kFxThreads, 1)
fx_vtx_kernel(const double *__restrict__ X, int ldx, int k0, int nbw, int skip, int M, int N,
              int RS, const unsigned char *__restrict__ V1, const double *__restrict__ Vtop,
              const unsigned *__restrict__ cmax, double *__restrict__ Wp, FxGram gr, int *status) {
  extern __shared__ __align__(1024) unsigned char fx_smem_raw[];
  unsigned char *base = (unsigned char *)(((uintptr_t)fx_smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint32_t s_taddr;
  // V's copy landed, X's digits written, a stage's MMAs done; accumulators
  // complete, accumulators drained
  __shared__ __align__(8) uint64_t s_full[2], s_xfull[2], s_empty[2], s_acc, s_drained;
  __shared__ int s_fa[64];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = blockIdx.x * 128, s = blockIdx.y;
  const bool gram = gr.sum != nullptr && blockIdx.x == gridDim.x - 1;
  if ((int)blockIdx.y >= (gram ? gr.slices : gr.vtx_slices)) return;
  const int i_begin = s * RS, i_end = min(M, i_begin + RS);
  const int T = (i_end - i_begin + 31) / 32;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                 :: "r"(smem_u32(&s_taddr)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int st = 0; st < 2; ++st) {
      fx_mbar_init(&s_full[st], 1);
      fx_mbar_init(&s_xfull[st], kFxWorkers);
      fx_mbar_init(&s_empty[st], 1);
    }
    fx_mbar_init(&s_acc, 1);
    fx_mbar_init(&s_drained, kFxWorkers);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (tid < 64) {
    const double up = Vtop[tid * 65];
    s_fa[tid] = (fx_hi(up) >= 0x7ff00000u) ? kFxNonFinite : fx_exp_of_hi(fx_hi(up)) - 3;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t taddr = s_taddr;

  if (gram) {
    fx_gram_block(gr, nbw, M, V1, base, taddr, &s_full[0], &s_acc, &s_empty[0], s_fa, status);
  } else if (warp == kFxWorkers) {                      // ---- the MMAs --------------------
    if (lane == 0) {
      bool ok = true;
      for (int t = 0; t < T; ++t) {
        const int st = t & 1;
        ok = mbar_wait(smem_u32(&s_full[st]), (uint32_t)((t >> 1) & 1)) &&
             mbar_wait(smem_u32(&s_xfull[st]), (uint32_t)((t >> 1) & 1));
        if (ok && (t & 3) == 0 && t > 0)
          ok = mbar_wait(smem_u32(&s_drained), (uint32_t)((t / 4 - 1) & 1));
        if (!ok) break;                                 // (the workers' waits run out too)
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t xa = smem_u32(base + st * kFxStage), vb = xa + kFxXStage;
        const bool fresh = (t & 3) == 0;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          const bool acc = !(fresh && ks == 0);
          // digit i of X times the stacked digits 0 .. min(6, 7 - i) of V, in
          // pieces of at most 256 columns; the last 64 of i = 1 open order 7
          auto piece = [&](int i, int n0, int n, bool ac) {
            fx_mma(taddr + (uint32_t)(i * 64 + n0), sw64_desc(xa + i * 8192 + ks * 32),
                   sw64_desc(vb + n0 * 64 + ks * 32), n, ac);
          };
          piece(0, 0, 256, acc);   piece(0, 256, 192, acc);
          piece(1, 0, 256, true);  piece(1, 256, 128, true); piece(1, 384, 64, acc);
          piece(2, 0, 192, true);  piece(2, 192, 192, true);
          piece(3, 0, 160, true);  piece(3, 160, 160, true);
          piece(4, 0, 256, true);
          piece(5, 0, 192, true);
          piece(6, 0, 128, true);
        }
        fx_commit(&s_empty[st]);
        if ((t & 3) == 3 || t == T - 1) fx_commit(&s_acc);
      }
    }
  } else {                                              // ---- splitting, draining ---------
    // this thread's column and group of 8 rows, and its column's exponent
    const int sc = tid >> 2, rg = tid & 3;
    const bool col_ok = c0 + sc < N;
    const int se = fx_exp_of_hi(col_ok ? cmax[c0 + sc] : 0u);
    const double *xcol = X + (size_t)(c0 + (col_ok ? sc : 0)) * ldx;
    auto load_v = [&](int t) {
      fx_bulk(smem_u32(base + (t & 1) * kFxStage + kFxXStage),
              V1 + (size_t)(i_begin / 32 + t) * kFxV1Chunk, kFxV1Chunk, &s_full[t & 1]);
    };
    double xv[8];
    const bool even_col = (((uintptr_t)xcol) & 15) == 0;
    auto load_x = [&](int t) {
      const int ib = i_begin + t * 32, i = ib + rg * 2;
      // the registers hold one chunk ahead; L2 gets three (128 bytes per thread pair)
      if (col_ok && (rg & 1) == 0 && ib + 128 <= i_end)
        asm volatile("prefetch.global.L2 [%0];"
                     ::"l"(xcol + k0 + ib + 96 + rg * 8 + (ib + 96 >= nbw ? skip : 0)));
      const bool whole = ib + 32 <= i_end && (ib >= nbw || ib + 32 <= nbw || skip == 0);
      const int off = k0 + i + (ib >= nbw ? skip : 0);
      if (col_ok && whole && even_col && (off & 1) == 0) {
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          const double2 v = *(const double2 *)(xcol + off + k * 4);
          xv[k] = v.x;
          xv[k + 1] = v.y;
        }
      } else if (col_ok && whole) {
#pragma unroll
        for (int k = 0; k < 8; ++k) xv[k] = xcol[off + (k >> 1) * 8 + (k & 1)];
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int ii = ib + fx_row(rg, k);
          xv[k] = (col_ok && ii < i_end) ? xcol[k0 + ii + (ii >= nbw ? skip : 0)] : 0.0;
        }
      }
    };
    int issued = 0;                                     // V copies (thread 0)
    if (tid == 0)
      for (; issued < T && issued < 2; ++issued) load_v(issued);
    load_x(0);
    // drain mapping: TMEM lane = column of X, this thread's 16 reflectors
    const int dq = warp & 3, dh = warp >> 2;
    // Totals in units of 2^ush digit products, ush from the slice's rows: a total
    // is at most ||x|| ||v|| < 2^55 sqrt(RS) sqrt(2) 2^58 of those, 62 bits.
    const int ush = fx_unit(RS);
    long long tot[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) tot[k] = 0;
    auto drain = [&](int b) -> bool {
      if (!fx_wait(&s_acc, b)) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        uint32_t r[kFxOrders][4];
        fx_ld_orders(r, taddr + ((uint32_t)(dq * 32) << 16) + (uint32_t)(dh * 16 + u * 4), 64);
        if (u == 3) {
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          if (lane == 0) fx_arrive(&s_drained);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          // 128 terms: orders 0 and 1 are at most 2^22; of 6 and 7 two units are
          // lost, 2^-63 of the bound; the others are converted
          auto f = [&](int o) { return __uint_as_float(r[o][k]); };
          const long long hi = ((long long)(fx_small(f(0)) * 256 + fx_small(f(1))) << 16) +
                               (long long)__float2int_rn(f(2)) * 256 + __float2int_rn(f(3));
          const long long lo = (long long)__float2int_rn(f(4)) * 65536 +
                               (long long)__float2int_rn(f(5)) * 256 + fx_small_quarter(f(6)) * 4 +
                               (fx_small_quarter(f(7)) >> 6);
          // hi in units of 2^72, lo of 2^48
          tot[u * 4 + k] += (hi << (72 - ush)) + ((lo + (1ll << (ush - 49))) >> (ush - 48));
        }
      }
      return true;
    };
    bool ok = true;
    for (int t = 0; t < T && ok; ++t) {
      const int st = t & 1;
      if (t >= 2) {                                     // the MMAs of chunk t - 2 are done
        ok = fx_wait(&s_empty[st], t / 2 - 1);
        if (!ok) break;
        if (tid == 0) { load_v(t); ++issued; }
      }
      {
        unsigned long long y[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) y[k] = fx_digits(xv[k], se);
        unsigned char *dst = base + st * kFxStage + sc * 64 + ((rg * 16) ^ (((sc >> 1) & 3) << 4));
#pragma unroll
        for (int i = 0; i < kFxD; ++i) *(uint4 *)(dst + i * 8192) = fx_pack8(y, i);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) fx_arrive(&s_xfull[st]);
      if (t + 1 < T) load_x(t + 1);                     // (behind the fence, which waits for loads)
      if (t > 0 && (t & 3) == 0) ok = drain(t / 4 - 1);
    }
    if (ok) ok = drain((T - 1) / 4);
    if (!ok && lane == 0) {
      for (int t = max(0, issued - 2); t < issued; ++t) // let the copies in flight land
        mbar_wait(smem_u32(&s_full[t & 1]), (uint32_t)((t >> 1) & 1));
      atomicCAS(status, 0, SLQR_ETIMEOUT);
    }
    const int c = c0 + dq * 32 + lane;
    if (ok && c < N) {
      const unsigned cm = cmax[c];
      const int e = fx_exp_of_hi(cm);
      double *out = Wp + ((size_t)s * N + c) * 64 + dh * 16;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int f = s_fa[dh * 16 + k];
        // tot 2^ush in units of 2^(e-55) 2^(f-55)
        out[k] = (cm >= 0x7ff00000u || f == kFxNonFinite)
                     ? __longlong_as_double(0x7ff8000000000000ll)
                     : fx_scale((double)tot[k], e + f - 110 + ush);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr));
}

// --------------------------------------------------------------------------
// Gt[j][q] = tau_j G[j][q] (q > j, else 0), row-major, then tau: what the
// substitution of W' = T^T W reads.  One CTA per panel.
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
fx_prep_kernel(const double *__restrict__ wy, int K, int nb, double *__restrict__ out) {
  const int nbw = min(nb, K - (int)blockIdx.x * nb);
  const double *G = wy + (size_t)blockIdx.x * wy_panel_doubles(nb) + nb * nb, *tau = G + nb * nb;
  double *o = out + (size_t)blockIdx.x * kFxGt;
  __shared__ double t[64][65];
  for (int idx = threadIdx.x; idx < nb * nb; idx += 256) t[idx % nb][idx / nb] = G[idx];
  __syncthreads();
  for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
    const int j = idx >> 6, q = idx & 63;
    o[idx] = (q > j && q < nbw) ? tau[j] * t[j][q] : 0.0;
  }
  if (threadIdx.x < 64) o[64 * 64 + threadIdx.x] = threadIdx.x < nbw ? tau[threadIdx.x] : 0.0;
}

// --------------------------------------------------------------------------
// W' = T^T W from the partials by substitution,
//   w'_j = tau_j (w_j - sum_{q<j} G[q,j] w'_q),
// written as the digit image of X -= V W': column c scaled by the largest
// |W'(a, c)| 2^(f_a), f_a the exponent of reflector a.  The entries stay
// unscaled while they are folded in (Gt carries tau), so a step is one shuffle
// and one FMA per 32 rows still to come.  One warp holds CPW columns (two rows
// a lane each).  Bound by the FP64 pipe: 96 FMAs a column and the sum of its
// partials.
// A W entry whose partials' magnitudes add up to less than 2^-kFxLoss |up_a| max |x_c|, as
// does its term of row a, may have lost its digits and is formed again from V and X (the
// columns at the panel's first row).  Without structure that is about 1% of the entries of
// panels of at most 128 rows, which have one partial, and next to none of others.
// W' in FP64 replaces the first partial, for the entries of X -= V W' formed again.
// --------------------------------------------------------------------------
template <int CPW>
__global__ void __launch_bounds__(256, CPW == 1 ? 4 : 3)
fx_tw_kernel(double *__restrict__ Wp, int S, int N, FxPanel p, const double *__restrict__ X, int ldx,
             const unsigned *__restrict__ cmax, const double *__restrict__ Gt,
             unsigned char *__restrict__ Wimg, int *__restrict__ ecol) {
  constexpr int NB = 64, WARPS = CPW == 1 ? 1 : 8;   // (CPW 1: all threads sum one column)
  __shared__ double G[NB * NB];
  __shared__ double part[CPW == 1 ? 4 : 8 * CPW][NB];
  __shared__ float psum[4][NB];
  __shared__ unsigned long long s_low;
  const double *wy = p.Vtop;
  const int nbw = p.nbw;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = (blockIdx.x * WARPS + (CPW == 1 ? 0 : warp)) * CPW;
  {
    double2 gv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) gv[u] = ((const double2 *)Gt)[tid + u * 256];
#pragma unroll
    for (int u = 0; u < 8; ++u) ((double2 *)G)[tid + u * 256] = gv[u];
  }
  const double t0 = Gt[NB * NB + lane], t1 = Gt[NB * NB + lane + 32];
  const double u0 = wy[lane * 65], u1 = wy[(lane + 32) * 65];     // up
  const size_t stride = (size_t)N * NB;
  double r0[CPW], r1[CPW];
  // A partial's magnitude over 2^(exponents of up_a and max |x_c|), by its bits (o: the
  // exponents to take off, in the high word); o of reflector and column.
  auto part_of = [](double v, int o) {
    return __int_as_float(min(max((int)fx_hi(v) - o, 0), 254 << 20) << 3);
  };
  auto off = [](double u, unsigned cm) {
    return min((int)(fx_hi(u) >> 20) + (int)(cm >> 20) - 1023 - 127, 2000) * (1 << 20);
  };
  // whether reflector a's entry, whose partials' magnitudes add up to `sum`, is below the
  // line, and so is the one term up_a x_a
  auto low = [&](int c, int a, float sum, double u) {
    const unsigned cm = cmax[c];
    if (fx_hi(u) == 0 || cm == 0 || cm >= 0x7ff00000u || sum >= 1.f / (1 << kFxLoss)) return false;
    return (int)(fx_hi(X[(size_t)c * ldx + a]) >> 20) < (int)(cm >> 20) - kFxLoss;
  };
  // of few rows every lane forms its own (V of [L^T; C] has its pivots and C's rows)
  auto few = [&](int c, bool low0, bool low1, double &r0, double &r1) {
    if (low0) r0 = fx_dot1(p, X + (size_t)c * ldx, lane);
    if (low1) r1 = fx_dot1(p, X + (size_t)c * ldx, lane + 32);
  };
  if constexpr (CPW == 1) {
    const double *src = Wp + (size_t)c0 * NB + (tid & 63);
    double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    float mg = 0.f;
    const int o = off(wy[(tid & 63) * 65], cmax[c0]);
    auto take = [&](double &a, int s) {
      const double v = src[s * stride];
      mg += part_of(v, o);
      a += v;
    };
    int s = tid >> 6;
    for (; s + 12 < S; s += 16) {
      take(a0, s);
      take(a1, s + 4);
      take(a2, s + 8);
      take(a3, s + 12);
    }
    for (; s < S; s += 4) take(a0, s);
    part[tid >> 6][tid & 63] = (a0 + a1) + (a2 + a3);
    psum[tid >> 6][tid & 63] = mg;
    __syncthreads();
    bool low0 = false, low1 = false;
    if (warp == 0) {
      r0[0] = (part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane]);
      r1[0] = (part[0][lane + 32] + part[1][lane + 32]) + (part[2][lane + 32] + part[3][lane + 32]);
      auto ps = [&](int a) { return psum[0][a] + psum[1][a] + psum[2][a] + psum[3][a]; };
      low0 = low(c0, lane, ps(lane), u0);
      low1 = low(c0, lane + 32, ps(lane + 32), u1);
      if (p.M <= kFxFewRows) {
        few(c0, low0, low1, r0[0], r1[0]);
        low0 = low1 = false;
      }
      const unsigned l0 = __ballot_sync(0xffffffffu, low0), l1 = __ballot_sync(0xffffffffu, low1);
      if (lane == 0) s_low = (unsigned long long)l1 << 32 | l0;
    }
    __syncthreads();
    if (s_low != 0) {                                  // (uniform)
      if ((s_low >> (8 * warp)) & 0xff)
        fx_dots8<1>(p, X + (size_t)c0 * ldx, ldx, 8 * warp, part[0] + 8 * warp);
      __syncthreads();
      if (low0) r0[0] = part[0][lane];
      if (low1) r1[0] = part[0][lane + 32];
    }
    if (warp > 0) return;
  } else {
    float m0[CPW], m1[CPW];                            // sums of the partials' magnitudes
#pragma unroll
    for (int k = 0; k < CPW; ++k) {
      const double *src = Wp + (size_t)min(c0 + k, N - 1) * NB + lane;
      double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
      m0[k] = m1[k] = 0.f;
      const unsigned cm = cmax[min(c0 + k, N - 1)];
      const int o0 = off(u0, cm), o1 = off(u1, cm);
      auto take = [&](double &a, double &b, int s) {
        const double v0 = src[s * stride], v1 = src[s * stride + 32];
        m0[k] += part_of(v0, o0);
        m1[k] += part_of(v1, o1);
        a += v0;
        b += v1;
      };
      int s = 0;
      for (; s + 1 < S; s += 2) {
        take(a0, b0, s);
        take(a1, b1, s + 1);
      }
      if (s < S) take(a0, b0, s);
      r0[k] = a0 + a1;
      r1[k] = b0 + b1;
    }
    __syncthreads();
    if (c0 >= N) return;
    bool low0[CPW], low1[CPW];
    unsigned l0 = 0, l1 = 0;
#pragma unroll
    for (int k = 0; k < CPW; ++k) {
      const bool in = c0 + k < N;
      low0[k] = in && low(c0 + k, lane, m0[k], u0);
      low1[k] = in && low(c0 + k, lane + 32, m1[k], u1);
      if (p.M <= kFxFewRows) {
        few(c0 + k, low0[k], low1[k], r0[k], r1[k]);
        low0[k] = low1[k] = false;
      }
      l0 |= __ballot_sync(0xffffffffu, low0[k]);
      l1 |= __ballot_sync(0xffffffffu, low1[k]);
    }
    if (l0 | l1) {                                     // the warp's columns together
      double *dots = part[warp * CPW];
      for (int g = 0; g < 8; ++g)
        if (((g < 4 ? l0 : l1) >> (8 * (g & 3))) & 0xff)
          fx_dots8<CPW>(p, X + (size_t)c0 * ldx, c0 + CPW <= N ? ldx : 0, 8 * g, dots + 8 * g);
#pragma unroll
      for (int k = 0; k < CPW; ++k) {
        if (low0[k]) r0[k] = dots[k * NB + lane];
        if (low1[k]) r1[k] = dots[k * NB + lane + 32];
      }
    }
  }
  // (on and below the diagonal Gt is zero, but a product with an entry that is
  // not finite would not be)
  for (int j = 0; j < min(nbw, 32); ++j) {
    const double g0 = -G[j * NB + lane], g1 = -G[j * NB + lane + 32];
#pragma unroll
    for (int k = 0; k < CPW; ++k) {
      const double wj = __shfl_sync(0xffffffffu, r0[k], j);
      if (lane > j) r0[k] = fma(g0, wj, r0[k]);
      r1[k] = fma(g1, wj, r1[k]);
    }
  }
  for (int j = 32; j < nbw; ++j) {
    const double g1 = -G[j * NB + lane + 32];
#pragma unroll
    for (int k = 0; k < CPW; ++k) {
      const double wj = __shfl_sync(0xffffffffu, r1[k], j - 32);
      if (lane + 32 > j) r1[k] = fma(g1, wj, r1[k]);
    }
  }
  const int f0 = u0 == 0.0 ? 0 : fx_exp_of_hi(fx_hi(u0));
  const int f1 = u1 == 0.0 ? 0 : fx_exp_of_hi(fx_hi(u1));
#pragma unroll
  for (int k = 0; k < CPW; ++k) {
    const int c = c0 + k;
    if (c >= N) break;
    const double w0 = lane < nbw ? r0[k] * t0 : 0.0, w1 = lane + 32 < nbw ? r1[k] * t1 : 0.0;
    int key = max(fx_key(w0, f0), fx_key(w1, f1));
    key = __reduce_max_sync(0xffffffffu, key);
    const bool bad =
        __any_sync(0xffffffffu, fx_hi(w0) >= 0x7ff00000u || fx_hi(w1) >= 0x7ff00000u);
    const int g = (key == kFxZero) ? kFxZeroExp : fx_exp(key);
    Wp[(size_t)c * NB + lane] = w0;
    Wp[(size_t)c * NB + lane + 32] = w1;
    unsigned char *dst = Wimg + (size_t)(c >> 5) * kFxWTile + (c & 31) * 128;
    const unsigned long long y0 = fx_digits(w0, g - f0), y1 = fx_digits(w1, g - f1);
    const int sw = (c & 7) << 4;
#pragma unroll
    for (int i = 0; i < kFxD; ++i) {
      const int b = 8 * (7 - i);
      const uint32_t v = fx_half2((uint32_t)(y0 >> b) & 0xff, (uint32_t)(y1 >> b) & 0xff, 0);
      *(unsigned short *)(dst + i * 4096 + ((lane * 2) ^ sw)) = (unsigned short)(v & 0xffff);
      *(unsigned short *)(dst + i * 4096 + ((64 + lane * 2) ^ sw)) = (unsigned short)(v >> 16);
    }
    if (lane == 0) ecol[c] = bad ? kFxNonFinite : g;
  }
}

// --------------------------------------------------------------------------
// X(i, c) -= sum_a V(i, a) W'(a, c): a CTA keeps the digits of 128 rows of V
// and goes through `per` tiles of 32 columns.  Warp 16 fetches W' and issues
// the MMAs, a tile ahead of the reassembly (two sets of eight 32-column
// accumulators fill tensor memory); the sixteen worker warps are coupled to it
// by mbarriers only and read X of the next tile before they reassemble this
// one.  A thread owns one row and 8 columns of a tile: TMEM lane = row, so X is
// read and written in 256-byte runs.  The new values' column maxima (rows >= 64,
// those of the next panel) go to cnext.
// An entry is below the line where it and its change are less than 2^-kFxLoss of the
// row's scale times the column's.  By chance that is one entry in 100 of the top rows and
// one in 10^4 of the others (one in 8 of the top rows of [L^T; C]); where rows and columns
// hold their large values in different reflectors it is most entries of a row or of a
// column.  So three of the thread's four columns, or 3/8 of the warp's rows, count as
// lost: those entries are left and formed again from V and W' in FP64 (fx_lost_entries).
// grid: (ceil(M / 128), groups of `per` tiles)
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(kFxThreads, 1)
fx_upd_kernel(double *__restrict__ X, int ldx, int k0, int nbw, int skip, int M, int N, int per,
              const unsigned char *__restrict__ V2, const int *__restrict__ erow,
              const unsigned char *__restrict__ Wimg, const int *__restrict__ ecol, FxPanel p,
              const double *__restrict__ Wf, unsigned *__restrict__ cnext, int *status) {
  extern __shared__ __align__(1024) unsigned char fx_smem_raw[];
  unsigned char *base = (unsigned char *)(((uintptr_t)fx_smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *Ws = base + kFxV2Tile;
  __shared__ uint32_t s_taddr;
  // copies landed; a tile's MMAs done, its accumulators read
  __shared__ __align__(8) uint64_t s_vfull, s_wfull[2], s_mma[2], s_free[2];
  __shared__ int s_ecol[32 * kFxMaxPer];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntiles = (N + 31) / 32;
  const int t_begin = blockIdx.y * per, T = min(ntiles, t_begin + per) - t_begin;
  const int i0 = blockIdx.x * 128;

  for (int idx = tid; idx < 32 * T; idx += kFxThreads)
    s_ecol[idx] = t_begin * 32 + idx < N ? ecol[t_begin * 32 + idx] : kFxZeroExp;
  // entries to be formed again: [column tile][warp][column of 8], a bit a row
  unsigned *lost_rows = (unsigned *)(Ws + 2 * kFxWTile);
  for (int idx = tid; idx < T * kFxLostWords; idx += kFxThreads) lost_rows[idx] = 0;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                 :: "r"(smem_u32(&s_taddr)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    fx_mbar_init(&s_vfull, 1);
    for (int st = 0; st < 2; ++st) {
      fx_mbar_init(&s_wfull[st], 1);
      fx_mbar_init(&s_mma[st], 1);
      fx_mbar_init(&s_free[st], kFxWorkers);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t taddr = s_taddr;

  if (warp == kFxWorkers) {                              // ---- copies and MMAs -------------
    if (lane == 0) {
      int issued = 0;
      auto load_w = [&](int t) {
        fx_bulk(smem_u32(Ws + (t & 1) * kFxWTile), Wimg + (size_t)(t_begin + t) * kFxWTile,
                kFxWTile, &s_wfull[t & 1]);
        ++issued;
      };
      fx_bulk(smem_u32(base), V2 + (size_t)blockIdx.x * kFxV2Tile, kFxV2Tile, &s_vfull);
      load_w(0);
      if (T > 1) load_w(1);
      bool ok = mbar_wait(smem_u32(&s_vfull), 0);
      for (int t = 0; t < T && ok; ++t) {
        const int st = t & 1;
        ok = mbar_wait(smem_u32(&s_wfull[st]), (uint32_t)((t >> 1) & 1));
        if (ok && t >= 2) ok = mbar_wait(smem_u32(&s_free[st]), (uint32_t)((t / 2 - 1) & 1));
        if (!ok) break;                                  // (the workers' waits run out too)
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t va = smem_u32(base), wb = smem_u32(Ws + st * kFxWTile);
        const uint32_t acc0 = taddr + (uint32_t)(st * 256);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          auto piece = [&](int i, int n0, int n, bool ac) {
            fx_mma(acc0 + (uint32_t)(i * 32 + n0), sw128_desc(va + i * 16384 + ks * 32),
                   sw128_desc(wb + n0 * 128 + ks * 32), n, ac);
          };
          piece(0, 0, 224, ks > 0);
          piece(1, 0, 192, true); piece(1, 192, 32, ks > 0);
          piece(2, 0, 192, true);
          piece(3, 0, 160, true);
          piece(4, 0, 128, true);
          piece(5, 0, 96, true);
          piece(6, 0, 64, true);
        }
        fx_commit(&s_mma[st]);
        if (t >= 1 && t + 1 < T) {                       // the stage of tile t - 1 is free
          ok = mbar_wait(smem_u32(&s_mma[st ^ 1]), (uint32_t)(((t - 1) >> 1) & 1));
          if (ok) load_w(t + 1);
        }
      }
      if (!ok) {
        mbar_wait(smem_u32(&s_vfull), 0);                // let the copies in flight land
        for (int t = max(0, issued - 2); t < issued; ++t)
          mbar_wait(smem_u32(&s_wfull[t & 1]), (uint32_t)((t >> 1) & 1));
        atomicCAS(status, 0, SLQR_ETIMEOUT);
      }
    }
  } else {                                               // ---- reassembly ------------------
    // this thread's row of the tile and its 8 columns
    const int q = warp & 3, h = warp >> 2;
    const int i = i0 + q * 32 + lane;
    const bool row_ok = i < M;
    const int ei = erow[i];                              // (defined up to the whole tile)
    const int er = (ei == kFxZeroExp ? 0 : ei) - 56;
    // the line: the scales' product is 2^(sh + 56) or up to two binades less
    const bool live = row_ok && ei != kFxZeroExp;
    const unsigned line = live ? 1u << (23 - kFxLoss) : 0u, line2 = 2 * line;
    const unsigned xline = (unsigned)(er + 1078 - kFxLoss) << 21;
    // (3 of 8 of the rows)
    const int lost_rows_min = 3 * __popc(__ballot_sync(0xffffffffu, live));
    unsigned *lost_mine = lost_rows + warp * 8;
    double *xrow = X + k0 + i + (i >= nbw ? skip : 0) + (size_t)(t_begin * 32 + h * 8) * ldx;
    const bool next_row = row_ok && i >= 64;
    int c = t_begin * 32 + h * 8;
    double xn[8];
    auto load_x = [&]() {
#pragma unroll
      for (int k = 0; k < 8; ++k) xn[k] = (row_ok && c + k < N) ? xrow[(size_t)k * ldx] : 0.0;
    };
    load_x();
    for (int t = 0; t < T; ++t) {
      const int buf = t & 1;
      double x[8];
      double *xw = xrow;
      const int cw = c;
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = xn[k];
      xrow += (size_t)32 * ldx;
      c += 32;
      if (t + 1 < T) load_x();
      const int *g = s_ecol + t * 32 + h * 8;
      if (!fx_wait(&s_mma[buf], t >> 1)) {
        if (lane == 0) atomicCAS(status, 0, SLQR_ETIMEOUT);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t ta = taddr + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + h * 8);
      unsigned mine = 0;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        uint32_t r[kFxOrders][4];
        fx_ld_orders(r, ta + (uint32_t)(u * 4), 32);
        if (u == 1) {
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          if (lane == 0) fx_arrive(&s_free[buf]);
        }
        long long tt[4];
        unsigned low = 0;                                // (of these four: below the line)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int k = u * 4 + kk;
          // Orders in units of 2^(erow + g - 110), kept to 2^54 of those in 63 bits
          // (the leading order sums 64 products).  Orders 0..3 are at most 2^22,
          // 4 and 5 above; of 6 and 7 half a unit is lost, 2^-62 of the bound.
          auto f = [&](int o) { return __uint_as_float(r[o][kk]); };
          tt[kk] =
              fx_join(fx_small(f(0)) * 256 + fx_small(f(1)), fx_small(f(2)) * 256 + fx_small(f(3)),
                      __float2int_rn(f(4)) * 256 + __float2int_rn(f(5)),
                      (fx_small_half(f(6)) * 256 + fx_small_half(f(7))) * 2, 20);
          if ((unsigned)((int)(tt[kk] >> 32) + (int)line) < line2 &&
              (unsigned)__double2hiint(x[k]) * 2u < xline + (unsigned)g[k] * (1u << 21))
            low |= 1u << kk;
        }
        if (__any_sync(0xffffffffu, low != 0)) {
          // (the quick test's exponents wrap, and it takes in columns of zeros, columns that
          // are not finite and the ones past the last)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const int gk = g[u * 4 + kk];
            if (gk == kFxZeroExp || gk == kFxNonFinite ||
                (int)(fx_hi(x[u * 4 + kk]) >> 20) >= er + gk + 1078 - kFxLoss)
              low &= ~(1u << kk);
          }
          unsigned lost = __popc(low) >= min(3, N - cw - u * 4) ? low : 0u;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const unsigned in_col = __ballot_sync(0xffffffffu, low >> kk & 1);
            if (8 * __popc(in_col) >= lost_rows_min) lost |= low & (1u << kk);
            const unsigned rows = __ballot_sync(0xffffffffu, lost >> kk & 1);
            if (lane == kk && rows) lost_mine[t * kFxLostWords + u * 4 + kk] = rows;
            if (lost >> kk & 1) tt[kk] = 0;
          }
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int k = u * 4 + kk;
          const int gk = g[k], sh = er + gk;
          // (uniform: exponents out of the quick form's range are rare)
          if (__all_sync(0xffffffffu, sh >= -1000 && sh <= 900))
            x[k] -= fx_to_double(tt[kk], sh);
          else if (gk == kFxNonFinite)
            x[k] = __longlong_as_double(0x7ff8000000000000ll);
          else if (gk != kFxZeroExp)
            x[k] -= fx_scale_slow((double)tt[kk], sh);
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int k = u * 4 + kk;
          if (row_ok && cw + k < N) xw[(size_t)k * ldx] = x[k];
          const unsigned mx = __reduce_max_sync(0xffffffffu, next_row ? fx_hi(x[k]) : 0u);
          if (lane == k) mine = mx;
        }
      }
      if (cnext && lane < 8 && cw + lane < N && mine) atomicMax(cnext + cw + lane, mine);
    }
    __syncwarp();
    fx_lost_entries(p, Wf, X + k0, ldx, N, i, t_begin * 32 + h * 8, T, lost_mine,
                    cnext);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(taddr));
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
slqr_status init_fx_attrs(slqr_ctx *ctx) {
  cudaError_t e = cudaFuncSetAttribute(fx_vtx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kFxVtxSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fx_upd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kFxUpdSmem);
  if (e != cudaSuccess)
    return fail(ctx, SLQR_ECUDA, "cudaFuncSetAttribute(fp64 tc): %s", cudaGetErrorString(e));
  return SLQR_OK;
}

static int fx_slices(int M, int N, int num_sms, int *RS) {
  // few column tiles: one wave of CTAs (a CTA has an SM to itself); more: about
  // four, so that the last one is a small part
  const int tiles = (N + 127) / 128, blocks = (M + 127) / 128;
  const int want = tiles <= num_sms / 8 ? num_sms / tiles : (4 * num_sms + tiles - 1) / tiles;
  const int S = std::max(1, std::min(blocks, want));
  *RS = (blocks + S - 1) / S * 128;
  return (M + *RS - 1) / *RS;
}

size_t fx_v_bytes(int m) {
  const size_t tiles = ((size_t)m + 127) / 128;
  return tiles * (4 * (size_t)kFxV1Chunk + kFxV2Tile) + align_up(tiles * 128 * sizeof(int), 256);
}

size_t fx_work_bytes(int m, int n, int num_sms) {
  // partials: S N' <= (4 num_sms + tiles') 128 over every width N' <= n, and at
  // most a slice per 128 rows (fx_slices)
  const size_t part = std::min(((size_t)4 * num_sms + 2) * 128 + (size_t)n,
                               ((size_t)m + 127) / 128 * (size_t)n);
  const size_t tiles = ((size_t)n + 31) / 32;
  return align_up(part * 64 * sizeof(double), 256) + tiles * kFxWTile +
         align_up(tiles * 32 * sizeof(int), 256);
}

void fx_split_v(const double *A, int lda, const double *Vtop, int k0, int nbw, int M, int skip,
                void *vbuf, cudaStream_t stream) {
  const size_t tiles = ((size_t)M + 127) / 128;
  unsigned char *V1 = (unsigned char *)vbuf, *V2 = V1 + tiles * 4 * kFxV1Chunk;
  int *erow = (int *)(V2 + tiles * kFxV2Tile);
  fx_vsplit_kernel<<<(unsigned)(tiles * 4), 256, 0, stream>>>(A, lda, Vtop, k0, nbw, M, skip, V1,
                                                              V2, erow);
}

static FxPanel fx_panel(const double *A, int lda, const double *Vtop, int k0, int nbw, int M,
                        int skip) {
  return FxPanel{Vtop, A + (size_t)k0 * lda + k0 + skip, lda, nbw, M, skip};
}

static FxGram fx_gram_args(double *wy_panel, const FxGramBuffers &b, double *Gt, const FxPanel &p,
                           int ctas) {
  FxGram gr;
  gr.sum = (unsigned long long *)b.sums;
  gr.arrived = (unsigned *)(gr.sum + 64 * 64);
  gr.p = p;
  gr.part = b.part;
  gr.G = wy_panel + 64 * 64;
  gr.Gt = Gt;
  const int blocks = (p.M + 127) / 128;
  gr.RS = (blocks + ctas - 1) / ctas * 128;
  gr.slices = (p.M + gr.RS - 1) / gr.RS;
  gr.vtx_slices = 0;
  return gr;
}

void fx_gram(slqr_ctx *ctx, const double *A, int lda, int k0, int nbw, int M, int skip,
             double *wy_panel, const void *vbuf, const FxGramBuffers &gram, double *Gt,
             cudaStream_t stream) {
  const FxGram gr = fx_gram_args(wy_panel, gram, Gt, fx_panel(A, lda, wy_panel, k0, nbw, M, skip),
                                 ctx->num_sms);
  int slot = prof_begin(ctx, stream);
  fx_vtx_kernel<<<dim3(1, gr.slices), kFxThreads, kFxVtxSmem, stream>>>(
      nullptr, 0, 0, nbw, 0, M, 0, 128, (const unsigned char *)vbuf, wy_panel, nullptr, nullptr, gr,
      ctx->d_status);
  prof_end(ctx, stream, slot, kVtx, 0.0);
}

void fx_prep(const double *wy, int K, int nb, double *Gt, cudaStream_t stream) {
  fx_prep_kernel<<<num_panels(K, nb), 256, 0, stream>>>(wy, K, nb, Gt);
}

bool fx_update(slqr_ctx *ctx, const double *A, int lda, int k0, int nbw, int M, int skip,
               const double *wy_panel, const double *Gt, const void *vbuf, double *X, int ldx, int N, const unsigned *cmax,
               unsigned *cnext, void *work, size_t work_bytes, cudaStream_t stream,
               const FxGramBuffers *gram) {
  int RS = 0;
  const int S = fx_slices(M, N, ctx->num_sms, &RS);
  const size_t tiles = ((size_t)M + 127) / 128, wt = ((size_t)N + 31) / 32;
  const size_t part = align_up((size_t)S * N * 64 * sizeof(double), 256);
  if (part + wt * kFxWTile + wt * 32 * sizeof(int) > work_bytes) return false;
  const unsigned char *V1 = (const unsigned char *)vbuf, *V2 = V1 + tiles * 4 * kFxV1Chunk;
  const int *erow = (const int *)(V2 + tiles * kFxV2Tile);
  double *Wp = (double *)work;
  unsigned char *Wimg = (unsigned char *)work + part;
  int *ecol = (int *)(Wimg + wt * kFxWTile);
  const double flops = 2.0 * M * nbw * (double)N;
  int slot = prof_begin(ctx, stream);
  // the panel's Gram terms beside it, on the SMs the products leave (a quarter at least)
  const int vt = (N + 127) / 128;
  const FxPanel p = fx_panel(A, lda, wy_panel, k0, nbw, M, skip);
  FxGram gr = fx_gram_args((double *)wy_panel, gram ? *gram : FxGramBuffers{}, (double *)Gt, p,
                           std::max(ctx->num_sms / 4, ctx->num_sms - vt * S));
  gr.vtx_slices = S;
  fx_vtx_kernel<<<dim3(vt + (gram ? 1 : 0), std::max(S, gram ? gr.slices : 0)), kFxThreads,
                  kFxVtxSmem, stream>>>(X, ldx, k0, nbw, skip, M, N, RS, V1, wy_panel, cmax, Wp, gr,
                                        ctx->d_status);
  prof_end(ctx, stream, slot, kVtx, flops);
  slot = prof_begin(ctx, stream);
  if (N <= 4 * ctx->num_sms)
    fx_tw_kernel<1><<<N, 256, 0, stream>>>(Wp, S, N, p, X + k0, ldx, cmax, Gt, Wimg, ecol);
  else
    fx_tw_kernel<2><<<(N + 15) / 16, 256, 0, stream>>>(Wp, S, N, p, X + k0, ldx, cmax, Gt, Wimg,
                                                       ecol);
  prof_end(ctx, stream, slot, kTw, (double)nbw * nbw * N);
  slot = prof_begin(ctx, stream);
  const int rt = (M + 127) / 128;
  // column tiles per CTA: about four waves of CTAs, at least 4 tiles each (the
  // V tile is 114 KB, as much as 3.5 tiles of X)
  const int groups = std::max(1, (4 * ctx->num_sms + rt - 1) / rt);
  const int per = std::min(
      kFxMaxPer, std::max(rt * (int)wt <= ctx->num_sms ? 1 : 4, ((int)wt + groups - 1) / groups));
  fx_upd_kernel<<<dim3(rt, ((int)wt + per - 1) / per), kFxThreads, kFxUpdSmem, stream>>>(
      X, ldx, k0, nbw, skip, M, N, per, V2, erow, Wimg, ecol, p, Wp, cnext, ctx->d_status);
  prof_end(ctx, stream, slot, kUpd, flops);
  return true;
}

void fx_colmax(const double *X, int ldx, int m, int n, int stacked_top, bool upper, unsigned *cmax,
               int np, int num_sms, cudaStream_t stream) {
  cudaMemsetAsync(cmax, 0, (size_t)np * n * sizeof(unsigned), stream);
  const int r0 = stacked_top;                     // dense: 0; stacked: the rows of C
  if (m > r0) {
    const int sl = std::max(1, std::min((m - r0 + 1023) / 1024, (8 * num_sms + n - 1) / n));
    fx_colmax_kernel<<<dim3(n, sl), 256, 0, stream>>>(X, ldx, r0, m, 0, n, cmax);
  }
  if (stacked_top > 0)
    fx_colmax_diag_kernel<<<dim3((n + 7) / 8, np), 256, 0, stream>>>(X, ldx, n, stacked_top, upper,
                                                                    cmax);
}

}  // namespace slqr
