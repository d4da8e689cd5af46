// qt_vec.cu -- B <- Q^T B for a few right-hand sides (fewer than kFxMinCols) of
// an FP64 factorization with panels of 64 reflectors, in one launch for all
// panels (Section 1 of the paper: the stored reflectors applied again at each
// SLSQP iteration).
//
// The tiled products of factor.cu work on 64 columns whatever their number: one
// right-hand side of a 4096 x 2048 factorization took 166 us a panel, 32
// panels, three launches each.  Here a CTA keeps R rows of the right-hand sides
// in shared memory for all panels and goes through
//   w = V^T b     its rows of V (fetched one panel ahead), eight lanes a column
//   exchange      the CTAs' sums of w: added within a cluster by one of its CTAs
//                 (st.async, mbarrier), the clusters' sums through L2, each slot
//                 polled until it holds a value (as in panel_grid.cu)
//   w' = T^T w    with T formed before (qt_t_kernel), in every CTA
//   b -= V w'
// per panel.  What bounds it is latency: the exchange and 16 clocks of the FP64
// pipe per warp instruction; V is read once.
#include "cluster_common.cuh"

#include <algorithm>

namespace slqr {
using namespace cl;

namespace {

constexpr int kQvThreads = 512;
constexpr int kQvT = 64 * 64;                   // T of a panel
constexpr int kQvPolls = 5;                     // clusters' sums a lane collects (40 clusters)
// An unset slot: all ones, a NaN that no arithmetic returns (published values
// that carry it go out as the canonical NaN).
constexpr unsigned long long kQvUnset = 0xffffffffffffffffull;

__device__ __forceinline__ bool qv_unset(double v) {
  return (unsigned long long)__double_as_longlong(v) == kQvUnset;
}
__device__ __forceinline__ double qv_load(const double *p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double qv_sum8(double v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

}  // namespace

// T of every panel (column-major, zero elsewhere), the inverse of striu(V^T V) +
// diag(1 / tau), by back-substitution with eight lanes to a column (a tau of 0, an
// undefined reflector, gives a zero row and column); grid (panels, column groups).
// In the chain of panels the substitution itself, 64 steps, took 8000 clocks of a
// panel's 22000; the product with T takes 2000 (4096 x 2048, one right-hand side:
// 386 -> 295 us with this launch).
__global__ void __launch_bounds__(128)
qt_t_kernel(const double *__restrict__ wy, int K, int nb, double *__restrict__ out) {
  __shared__ double Gs[64][65];
  __shared__ double ts[64];
  const int tid = threadIdx.x, l = tid & 7, j = blockIdx.y * 16 + (tid >> 3);
  const int nbw = min(nb, K - (int)blockIdx.x * nb), top = blockIdx.y * 16 + 16;
  const double *G = wy + (size_t)blockIdx.x * wy_panel_doubles(nb) + nb * nb, *tau = G + nb * nb;
  double *T = out + (size_t)blockIdx.x * kQvT + (size_t)j * 64;
  if (blockIdx.y * 16 >= nbw) {                // (columns past the panel; uniform)
#pragma unroll
    for (int u = 0; u < 8; ++u) T[l + 8 * u] = 0.0;
    return;
  }
  for (int idx = tid; idx < 64 * top; idx += 128) {
    const int i = idx & 63, c = idx >> 6;
    Gs[i][c] = i < c && c < nbw ? G[i + c * nb] : 0.0;
    if (c == 0) ts[i] = i < nbw ? tau[i] : 0.0;
  }
  __syncthreads();
  double y[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) y[u] = 0.0;
#pragma unroll
  for (int i = 63; i >= 0; --i) {
    if (i >= top) continue;                    // (uniform)
    double t = (i == j && l == 0) ? 1.0 : 0.0;
#pragma unroll
    for (int u = i / 8; u < 8; ++u)            // (y is zero up to row i and past row j)
      if (8 * u < top) t = fma(l + 8 * u <= j ? -Gs[i][l + 8 * u] : 0.0, y[u], t);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    t = t * ts[i];
    if ((i & 7) == l && i <= j) y[i / 8] = t;
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) T[l + 8 * u] = y[u];
}

struct QtVecParams {
  const double *A, *up, *T;
  double *B, *rec;               // rec: [panel][right-hand side][64][clusters], all ones before
  int m, K, nb, lda, ldb, nr, ntop;   // nb: panel width (64, or 32 in 64-column steps)
  int *status;
  unsigned spin;
};

template <int RPL, int NR>
__global__ void __launch_bounds__(kQvThreads, 1)
qt_vec_kernel(QtVecParams p) {
  constexpr int R = 8 * RPL, LD = R + 8;       // (column stride = 64 mod 128 bytes)
  constexpr int CG = kQvThreads / R;           // column groups of the update
  extern __shared__ __align__(16) unsigned char qv_smem[];
  double *Vs = (double *)qv_smem;              // [2][64][LD]
  double *Gs = Vs + 2 * 64 * LD;               // [2][kQvT]: T, column-major
  __shared__ double bs[NR][R];
  __shared__ double s_w[NR][64], s_wt[NR][64]; // w, w'
  __shared__ double s_part[NR][CG][R];
  __shared__ __align__(16) double s_recv[2][8][16 * NR];
  __shared__ __align__(8) unsigned long long s_mbar[2];
  __shared__ int s_reported;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = tid >> 3, l8 = tid & 7;        // column and rows of the dots
  const int rank = cluster_rank(), CS = cluster_ctas();
  const int NC = gridDim.x / CS, cluster = blockIdx.x / CS;
  const int row0 = blockIdx.x * R;
  const int np = (p.K + p.nb - 1) / p.nb;

  // whether the reflectors of panel pnl have entries in this CTA's rows: from the
  // diagonal block down (stacked [L^T; C]: the diagonal block and the rows of C)
  auto takes_part = [&](int pnl) {
    const int k0 = pnl * p.nb;
    return p.ntop > 0 ? row0 + R > p.ntop || (row0 + R > k0 && row0 < k0 + p.nb) : row0 + R > k0;
  };
  // whether a row is one of panel pnl's: only those are read and changed, as in the
  // tiled products (zero times a value that is not finite would reach the others)
  auto panel_row = [&](int pnl, int row) {
    const int k0 = pnl * p.nb;
    return row >= k0 && (p.ntop == 0 || row < min(k0 + p.nb, p.K) || row >= p.ntop);
  };
  // panel pnl's rows of V: the reflector tails, up on the diagonal, zeros above
  // (stacked: the tails are zero down to the rows of C, and not read there)
  auto fetch = [&](int pnl) {
    const int k0 = pnl * p.nb, nbw = min(p.nb, p.K - k0);
    double *dst = Vs + (pnl & 1) * 64 * LD + c * LD;
    const double *col = p.A + (size_t)(k0 + c) * p.lda;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const int r = l8 + 8 * i, row = row0 + r;
      const bool tail = p.ntop > 0 ? row >= p.ntop : row > k0 + c;
      if (c < nbw && row < p.m && tail) cp_async8(dst + r, col + row);
      else dst[r] = (c < nbw && row == k0 + c) ? p.up[k0 + c] : 0.0;
    }
    const double *g = p.T + (size_t)pnl * kQvT;
    double *gd = Gs + (pnl & 1) * kQvT;
    for (int idx = tid; idx < kQvT; idx += kQvThreads) cp_async8(gd + idx, g + idx);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // 16 NR-column pieces of the receive buffer: warps w = rank, rank + CS, ...
  const unsigned bytes = (unsigned)(CS * (16 / CS) * 4 * NR * 8);
  if (tid == 0) {
    mbar_init1(&s_mbar[0]);
    mbar_init1(&s_mbar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect(&s_mbar[0], bytes);
    if (np > 1) mbar_expect(&s_mbar[1], bytes);
    s_reported = 0;
  }
  if (takes_part(0)) fetch(0);
  for (int idx = tid; idx < NR * R; idx += kQvThreads) {
    const int k = idx / R, r = idx - k * R;
    bs[k][r] = (k < p.nr && row0 + r < p.m) ? p.B[SLQR_IDX(row0 + r, k, p.ldb)] : 0.0;
  }
  cluster_sync_all();
  bool dead = false;

  for (int pnl = 0; pnl < np; ++pnl) {
    const int buf = pnl & 1, nbw = min(p.nb, p.K - pnl * p.nb);
    const bool part_of = takes_part(pnl);               // (uniform over the CTA)
    const bool whole = row0 >= (p.ntop > 0 ? p.ntop : pnl * p.nb);   // (all rows are the panel's)
    if (pnl + 1 < np && takes_part(pnl + 1)) {
      fetch(pnl + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const double *V = Vs + buf * 64 * LD;
    // ---- w = V^T b: this CTA's part, to the CTA that adds this warp's columns ---
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      double part = 0.0;
      if (part_of) {
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int i = 0; i < RPL; i += 2) {
          const int r0 = l8 + 8 * i, r1 = r0 + 8;
          if (whole || panel_row(pnl, row0 + r0)) a0 = fma(V[c * LD + r0], bs[k][r0], a0);
          if (whole || panel_row(pnl, row0 + r1)) a1 = fma(V[c * LD + r1], bs[k][r1], a1);
        }
        part = qv_sum8(a0 + a1);
      }
      const int h = lane >> 4;
      double w2[2];
      w2[0] = __shfl_sync(0xffffffffu, part, 16 * h);
      w2[1] = __shfl_sync(0xffffffffu, part, 16 * h + 8);
      if ((lane & 15) == 0)
        st_async16(cluster_addr(&s_recv[buf][rank][((warp / CS) * NR + k) * 4 + 2 * h], warp % CS), w2,
                   cluster_addr(&s_mbar[buf], warp % CS));
    }
    double *rec = p.rec + (size_t)pnl * NR * 64 * NC;
    if (warp % CS == rank) {
      bool reported = s_reported != 0;
      if (!dead && !mbar_wait_bounded(&s_mbar[buf], (unsigned)(pnl >> 1) & 1u, p.spin, p.status,
                                      &reported)) {
        record_status(p.status, SLQR_ETIMEOUT);
        dead = true;
      }
      if (reported && lane == 0) s_reported = 1;
      if (warp + CS >= kQvThreads / 32 && lane == 0 && !dead && pnl + 2 < np)
        mbar_expect(&s_mbar[buf], bytes);
      __syncwarp();
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        double sum =
            qv_sum8(l8 < CS ? s_recv[buf][l8][((warp / CS) * NR + k) * 4 + (lane >> 3)] : 0.0);
        if (qv_unset(sum)) sum = __longlong_as_double(0x7fffffffffffffffll);
        if (l8 == 0)
          asm volatile("st.relaxed.gpu.global.f64 [%0], %1;"
                       ::"l"(rec + ((size_t)k * 64 + c) * NC + cluster), "d"(sum) : "memory");
      }
    }
    // (a CTA without such rows has nothing to update; the waits of the warps above
    // keep it in step with its cluster)
    if (!part_of) {
      __syncthreads();
      continue;
    }
    // ---- the clusters' sums of this thread's column -----------------------------
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const double *src = rec + ((size_t)k * 64 + c) * NC;
      double r[kQvPolls];
#pragma unroll
      for (int u = 0; u < kQvPolls; ++u) r[u] = l8 + 8 * u < NC ? qv_load(src + l8 + 8 * u) : 0.0;
      unsigned it = 0;
      while (!dead) {
        bool miss = false;
#pragma unroll
        for (int u = 0; u < kQvPolls; ++u) miss |= qv_unset(r[u]);
        if (!__any_sync(0xffffffffu, miss)) break;
        if (it == p.spin && lane == 0) record_status(p.status, SLQR_ETIMEOUT);
        if (++it > kSpinLimit) dead = true;
#pragma unroll
        for (int u = 0; u < kQvPolls; ++u)
          if (qv_unset(r[u])) r[u] = qv_load(src + l8 + 8 * u);
      }
      double d = r[0];
#pragma unroll
      for (int u = 1; u < kQvPolls; ++u)
        if (8 * u < NC) d += r[u];
      d = qv_sum8(d);
      if (l8 == 0) s_w[k][c] = d;
    }
    __syncthreads();
    // ---- w' = T^T w: column c of T, entries l8, l8 + 8, .. up to the diagonal ------
    {
      const double *T = Gs + buf * kQvT + c * 64;
      const int last = (4 * warp + 3) >> 3;
      double wt[NR];
#pragma unroll
      for (int k = 0; k < NR; ++k) wt[k] = 0.0;
      for (int u = 0; u <= last; ++u) {
        if (l8 + 8 * u > c) break;             // (T is zero from there on)
        const double t = T[l8 + 8 * u];
#pragma unroll
        for (int k = 0; k < NR; ++k) wt[k] = fma(t, s_w[k][l8 + 8 * u], wt[k]);
      }
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        wt[k] = qv_sum8(wt[k]);
        if (l8 == 0) s_wt[k][c] = wt[k];
      }
    }
    __syncthreads();
    // ---- b -= V w' ----------------------------------------------------------------
    {
      const int r = tid % R, g = tid / R;
      constexpr int CP = 64 / CG;              // columns of a group
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int u = 0; u < CP; u += 2) {
          a0 = fma(V[(g * CP + u) * LD + r], s_wt[k][g * CP + u], a0);
          a1 = fma(V[(g * CP + u + 1) * LD + r], s_wt[k][g * CP + u + 1], a1);
        }
        s_part[k][g][r] = a0 + a1;
      }
    }
    __syncthreads();
    for (int idx = tid; idx < NR * R; idx += kQvThreads) {
      const int k = idx / R, r = idx - k * R;
      double s = s_part[k][0][r];
#pragma unroll
      for (int g = 1; g < CG; ++g) s += s_part[k][g][r];
      if (whole || panel_row(pnl, row0 + r)) bs[k][r] -= s;
    }
  }
  __syncthreads();
  for (int idx = tid; idx < NR * R; idx += kQvThreads) {
    const int k = idx / R, r = idx - k * R;
    if (k < p.nr && row0 + r < p.m) p.B[SLQR_IDX(row0 + r, k, p.ldb)] = bs[k][r];
  }
  cluster_sync_all();                          // (nothing is sent to this CTA any more)
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
// right-hand sides a launch takes: at most 4, 2 with 128 rows per CTA
// (shared memory)
static const void *qt_kernel(int R, int nr) {
  switch (R * 8 + nr) {
    case 32 * 8 + 1: return (const void *)qt_vec_kernel<4, 1>;
    case 32 * 8 + 2: return (const void *)qt_vec_kernel<4, 2>;
    case 32 * 8 + 4: return (const void *)qt_vec_kernel<4, 4>;
    case 64 * 8 + 1: return (const void *)qt_vec_kernel<8, 1>;
    case 64 * 8 + 2: return (const void *)qt_vec_kernel<8, 2>;
    case 64 * 8 + 4: return (const void *)qt_vec_kernel<8, 4>;
    case 128 * 8 + 1: return (const void *)qt_vec_kernel<16, 1>;
    case 128 * 8 + 2: return (const void *)qt_vec_kernel<16, 2>;
    default: return nullptr;
  }
}

static size_t qt_smem(int R) { return (2 * 64 * (size_t)(R + 8) + 2 * kQvT) * sizeof(double); }

slqr_status init_qt_vec_attrs(slqr_ctx *ctx) {
  for (int R : {32, 64, 128})
    for (int nr : {1, 2, 4}) {
      const void *fn = qt_kernel(R, nr);
      if (!fn) continue;
      cudaError_t e =
          cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qt_smem(R));
      if (e != cudaSuccess)
        return fail(ctx, SLQR_ECUDA, "cudaFuncSetAttribute(Q^T b): %s", cudaGetErrorString(e));
    }
  return SLQR_OK;
}

// Rows per CTA: the fewest whose CTAs are at most 64, in clusters of 8 (up to 8
// CTAs: one cluster), beyond that 128 rows and what fits (one CTA per SM, as the
// grid panel); 0: too tall.
static int qt_shape(const slqr_ctx *ctx, int m, int *P, int *cluster) {
  for (int R : {32, 64, 128}) {
    const int ctas = (m + R - 1) / R;
    const int p8 = (ctas + 7) / 8 * 8, p4 = (ctas + 3) / 4 * 4;
    if (p8 <= std::min(ctx->grid_panel_c8, R < 128 ? 64 : 1 << 20)) {
      *P = p8, *cluster = 8;
      return R;
    }
    if (R == 128 && p4 <= ctx->grid_panel_c4) {
      *P = p4, *cluster = 4;
      return R;
    }
  }
  return 0;
}

size_t qt_vec_bytes(const slqr_ctx *ctx, int m, int K, int nb) {
  int P = 0, cluster = 0;
  if (qt_shape(ctx, m, &P, &cluster) == 0) return 0;
  const size_t np = (size_t)num_panels(K, nb);
  return np * (kQvT + 4 * 64 * (size_t)(P / cluster)) * sizeof(double);
}

static int qt_most(int R) { return R == 128 ? 2 : 4; }

int qt_vec_launches(const slqr_ctx *ctx, int m, int nrhs) {
  int P = 0, cluster = 0;
  const int most = qt_most(qt_shape(ctx, m, &P, &cluster));
  return (nrhs + most - 1) / most;
}

slqr_status qt_vec(slqr_ctx *ctx, int m, int K, int nb, const double *A, int lda, const double *up,
                   const double *wy, int nrhs, double *B, int ldb, int ntop, void *work,
                   cudaStream_t stream) {
  const int np = num_panels(K, nb);
  int P = 0, cluster = 0;
  const int R = qt_shape(ctx, m, &P, &cluster);
  double *T = (double *)work;
  int slot = prof_begin(ctx, stream);
  qt_t_kernel<<<dim3(np, 4), 128, 0, stream>>>(wy, K, nb, T);
  prof_end(ctx, stream, slot, kTw, 0.0);
  const int most = qt_most(R);
  for (int k = 0; k < nrhs; k += most) {
    const int nr = std::min(most, nrhs - k), tr = nr == 3 ? 4 : nr;
    QtVecParams p;
    p.A = A; p.up = up; p.T = T; p.B = B + (size_t)k * ldb; p.rec = T + (size_t)np * kQvT;
    p.m = m; p.K = K; p.nb = nb; p.lda = lda; p.ldb = ldb; p.nr = nr; p.ntop = ntop;
    p.status = ctx->d_status; p.spin = ctx->spin_limit;
    cudaError_t e = cudaMemsetAsync(
        p.rec, 0xff, (size_t)np * tr * 64 * (P / cluster) * sizeof(double), stream);
    if (e != cudaSuccess) return fail(ctx, SLQR_ECUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P);
    cfg.blockDim = dim3(kQvThreads);
    cfg.dynamicSmemBytes = qt_smem(R);
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = cluster;
    attrs[0].val.clusterDim.y = 1;
    attrs[0].val.clusterDim.z = 1;
    attrs[1].id = cudaLaunchAttributeCooperative;
    attrs[1].val.cooperative = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = P == cluster ? 1 : 2;     // (a cluster is resident as a whole by itself)
    void *args[] = {&p};
    slot = prof_begin(ctx, stream);
    e = cudaLaunchKernelExC(&cfg, qt_kernel(R, tr), args);
    prof_end(ctx, stream, slot, kVtx, 4.0 * m * K * nr - 2.0 * (double)K * K * nr);
    if (e != cudaSuccess)
      return fail(ctx, SLQR_ECUDA, "Q^T b launch (P=%d, R=%d): %s", P, R, cudaGetErrorString(e));
  }
  return SLQR_OK;
}

}  // namespace slqr
