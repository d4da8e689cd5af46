// panel_grid.cu -- the FP64 panel of 64 columns by thread-block clusters with
// the panel held in registers.
//
// Same arithmetic and outputs as panel_kernel (factor.cu; Alg. 2 of the paper
// on one panel): the scaled norm, the sign rule and up of Alg. 3, the reflector
// applied to the later columns; Vtop, the Gram terms of V^T V and tau for the
// compact-WY update.
//
// What bounds a column step: every FP64 warp instruction holds the SM's FP64
// pipe for 16 clocks, and the step is a chain of two passes over the slice, a
// sum over all CTAs and the pivot's square root and division.  So:
//  * The slice is spread over many CTAs (R = 32 .. 256 rows each) and lives in
//    registers: warp w holds columns 4 w .. 4 w + 3, eight lanes to a column,
//    lane l of them rows l, l + 8, ...  A column's dot needs three butterfly
//    adds (for four columns at once) instead of five per column or a pass
//    through shared memory.
//  * Partial dots go out straight from registers.  Up to 16 CTAs are one
//    cluster: each warp pushes its columns' partials to every CTA (st.async,
//    counted on an mbarrier there).  More CTAs are clusters of 8: the partials
//    of a column go to one CTA of the cluster, which adds the 8 and publishes
//    the sum in L2, and every warp collects the clusters' sums of its own
//    columns.  (Without the first level every CTA reads every CTA's record:
//    128 CTAs spent 3.5 us of a 7.4 us step in those reads.)
//  * The only CTA barriers of a step are the two that hand over the pivot (from
//    the warp of column j) and the next column (through shared memory).
//  * The Gram terms (dots with the finished columns) are formed while the
//    partials travel: the warps of finished columns start once the others have
//    published.
#include "cluster_common.cuh"

#include <algorithm>

namespace slqr {
using namespace cl;

namespace {

constexpr int kGpThreads = 512;
constexpr int kNB = 64;
constexpr int kGpCluster = 8;          // CTAs of a cluster where there are several

// Published sums are exchanged without a barrier: every slot is written once
// per panel, and until then it holds a signalling-NaN pattern that no
// arithmetic result has, so the value is its own message (as in panel_kernel).
constexpr unsigned long long kGpUnset = 0x7ff0dead5a5a5a5aull;

__device__ __forceinline__ bool gp_unset(double v) {
  return (unsigned long long)__double_as_longlong(v) == kGpUnset;
}
__device__ __forceinline__ void gp_publish(double *p, double v) {
  if (gp_unset(v)) v = __longlong_as_double(0x7fffffffffffffffll);
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ double gp_load(const double *p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
// sum over the 8 lanes of a column
__device__ __forceinline__ double gp_sum8(double v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// s = sqrt(S) and rb = 1 / (up cl) for cl = -+s, up = x0 - cl, for S within
// [2^-900, 2^900]: one third-order Householder iteration each from the
// hardware's approximate reciprocal (square root), about 2^-20 relative, then
// one Newton correction of s.  13 dependent FP64 operations; sqrt() and the
// division, with their range checks, are the longest part of a column step
// otherwise (2000 of 9700 clocks at 32 rows per CTA).
__device__ __forceinline__ void gp_pivot(double S, double x0, double *cl, double *up, double *rb) {
  double y, z;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(S));
  const double e = fma(-(S * y), y, 1.0);
  y = fma(fma(e, 0.375, 0.5) * e, y, y);
  double s = S * y;
  s = fma(fma(-s, s, S), 0.5 * y, s);
  const double c = x0 > 0.0 ? -s : s;
  const double u = x0 - c;
  const double b = u * c;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(b));
  const double f = fma(-b, z, 1.0);
  *rb = fma(fma(f, f, f), z, z);
  *cl = c;
  *up = u;
}

}  // namespace

// RPL rows per lane, R = 8 RPL rows per CTA; ONE: the grid is one cluster.
template <int RPL, bool ONE>
__global__ void __launch_bounds__(kGpThreads, 1)
panel_grid_kernel(GridPanelParams p) {
  constexpr int R = 8 * RPL;
  constexpr int SRC = ONE ? kClMaxCtas : kGpCluster;       // senders to a receive buffer
  constexpr int RC = ONE ? kNB : 8;                        // columns of a receive buffer
  extern __shared__ __align__(16) unsigned char gp_smem[];
  double *Gl = (double *)gp_smem;             // [NB][NB] at c + j NB: local Gram terms
  __shared__ __align__(16) double xs[2][R];   // column j's tail by j & 1 (zero elsewhere)
  __shared__ __align__(16) double s_recv[2][SRC][RC];
  __shared__ __align__(16) double s_prow[2][ONE ? kNB : 2];
  __shared__ unsigned s_mx[kNB];
  __shared__ int s_E[kNB];
  __shared__ double s_up[kNB], s_tau[kNB];
  __shared__ double s_piv[2][3];              // cl, up, 1/b by j & 1
  __shared__ int s_def[2];
  __shared__ __align__(8) unsigned long long s_mbar[2];
  __shared__ int s_ok, s_reported;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = warp * 4 + (lane >> 3), l8 = lane & 7;     // this lane's column and rows
  const int cta = blockIdx.x, P = gridDim.x;
  const int rank = cluster_rank();
  const int NC = ONE ? 1 : P / kGpCluster, cluster = ONE ? 0 : cta / kGpCluster;
  const int row0 = cta * R;
  const int nbw = p.nbw;
  const int RO = min(R, p.m - p.k0 - p.skip - row0);       // rows owned (<= 0: none)
  double *A = (double *)p.A;
  double *col = A + (size_t)(p.k0 + c) * p.lda + p.k0;
  auto at = [&](int r) { return row0 + r + (row0 + r >= nbw ? p.skip : 0); };   // (row map)
  auto absent = [&](int r) {
    // (stacked: the strictly lower part of the diagonal block is zero, not read)
    return c >= nbw || r >= RO || (p.stacked && row0 + r < nbw && row0 + r > c);
  };

  double v[RPL];
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = l8 + 8 * i;
    v[i] = absent(r) ? 0.0 : col[at(r)];
  }
  // the slots of this CTA's share back to unset; the barrier below orders this
  // before any publish or poll
  if (!ONE) {
    const int total = nbw * kNB * NC;
    for (int idx = cta * kGpThreads + tid; idx < total; idx += P * kGpThreads)
      p.rec[idx] = __longlong_as_double((long long)kGpUnset);
    if (cta == 0)
      for (int idx = tid; idx < nbw * kNB; idx += kGpThreads)
        p.prow[idx] = __longlong_as_double((long long)kGpUnset);
  }
  for (int idx = tid; idx < kNB * kNB; idx += kGpThreads) Gl[idx] = 0.0;

  // Bytes the receive buffer gets for column j.  ONE: every CTA's partials of
  // the active warps and the pivot row; else the cluster's partials of the
  // active warps among rank and rank + 8 (32 bytes each).
  auto warp_active = [&](int w, int j) { return 4 * w + 3 >= j && 4 * w < nbw; };
  auto step_bytes = [&](int j) -> unsigned {
    if (ONE) return (unsigned)((P + 1) * ((nbw + 3) / 4 - j / 4) * 32);
    return (unsigned)(kGpCluster * 32 * (warp_active(rank, j) + warp_active(rank + 8, j)));
  };
  if (tid == 0) {
    mbar_init1(&s_mbar[0]);
    mbar_init1(&s_mbar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // columns 0 and 1; column j + 2's phase is announced once column j's has
    // completed, before this CTA sends anything for column j + 1
    for (int j = 0; j < 2; ++j)
      if (j < nbw && step_bytes(j) > 0) mbar_expect(&s_mbar[j], step_bytes(j));
    s_ok = 1;
    s_reported = 0;
  }
  // column scales: largest exponent of each column (below its diagonal)
  {
    unsigned mx = 0;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const int r = l8 + 8 * i;
      if (row0 + r >= c) mx = max(mx, (unsigned)__double2hiint(v[i]) & 0x7fffffffu);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (l8 == 0) p.srec[(size_t)cta * kNB + c] = (double)mx;
  }
  if (tid < kNB) s_mx[tid] = 0;
  bool dead = false;                          // a wait ran out completely: no more waits
  if (!ONE) {
    // a barrier over the whole grid.  Past the context's limit it reports and
    // goes on waiting; only when the hard limit runs out does the cluster leave,
    // all CTAs together
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(p.bar, 1u);
      const unsigned target = p.bar_base + (unsigned)P;
      for (unsigned it = 0; ld_acquire_u32(p.bar) < target; ++it) {
        if (it == p.spin) record_status(p.status, SLQR_ETIMEOUT);
        if (it > kSpinLimit) { s_ok = 0; break; }
        if (it > 256) __nanosleep(64);
      }
      __threadfence();
    }
  }
  cluster_sync_all();
  if (!ONE) {
    bool all = true;
    for (int r = 0; r < kGpCluster; ++r) all &= cluster_ld_u32(cluster_addr(&s_ok, r)) != 0;
    cluster_sync_all();
    if (!all) {
      if (tid == 0) record_status(p.status, SLQR_ETIMEOUT);
      return;
    }
  }
  {
    unsigned mx = 0;
    for (int q = tid / kNB; q < P; q += kGpThreads / kNB)
      mx = max(mx, (unsigned)__ldcg(p.srec + (size_t)q * kNB + (tid & (kNB - 1))));
    atomicMax(&s_mx[tid & (kNB - 1)], mx);
  }
  if (c == 0) {                               // column 0's tail
#pragma unroll
    for (int i = 0; i < RPL; ++i) xs[0][l8 + 8 * i] = (row0 + l8 + 8 * i > 0) ? v[i] : 0.0;
  }
  __syncthreads();
  if (tid < kNB) {
    const int E = (int)((s_mx[tid] >> 20) & 0x7ff) - 1023;
    s_E[tid] = min(max(E, -1000), 1022);
  }
  __syncthreads();

  for (int j = 0; j < nbw; ++j) {
    const int buf = j & 1;
    const double *x = xs[buf];
    const bool mine = (j >> 2) == warp;        // this warp holds column j
    // a column of extreme scale squares its scaled entries (uniform)
    const bool extreme = abs(s_E[j]) > 400;
    const double sc = exp2i(-s_E[j]);
    double D = 0.0, pc = 0.0;

    // dot of the tail of x_j with this lane's column (c == j: its norm)
    auto dot = [&]() {
      double a0 = 0.0, a1 = 0.0;
#pragma unroll
      for (int i = 0; i < RPL; i += 2) {
        a0 = fma(x[l8 + 8 * i], v[i], a0);
        a1 = fma(x[l8 + 8 * (i + 1)], v[i + 1], a1);
      }
      if (extreme && mine) {
        double n0 = 0.0;
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          const double t = x[l8 + 8 * i] * sc;
          n0 = fma(t, t, n0);
        }
        if (c == j) a0 = n0, a1 = 0.0;
      }
      return gp_sum8(a0 + a1);
    };

    if (warp_active(warp, j)) {
      const double part = dot();
      // two columns' partials per lane half, 16 bytes to a receiver
      const int h = lane >> 4;
      {
        double w[2];
        w[0] = __shfl_sync(0xffffffffu, part, 16 * h);
        w[1] = __shfl_sync(0xffffffffu, part, 16 * h + 8);
        if (ONE) {
          const int dst = lane & 15;
          if (dst < P)
            st_async16(cluster_addr(&s_recv[buf][rank][warp * 4 + 2 * h], dst), w,
                       cluster_addr(&s_mbar[buf], dst));
        } else if ((lane & 15) == 0) {
          const int dst = warp & (kGpCluster - 1);
          st_async16(cluster_addr(&s_recv[buf][rank][(warp >> 3) * 4 + 2 * h], dst), w,
                     cluster_addr(&s_mbar[buf], dst));
        }
      }
      // the pivot row, by the CTA that holds it
      if (row0 <= j && j < row0 + R) {
        double w = 0.0;
#pragma unroll
        for (int i = 0; i < RPL; ++i) w = (row0 + l8 + 8 * i == j) ? v[i] : w;
        const int l = (j - row0) & 7;
        if (ONE) {
          double ww[2];
          ww[0] = __shfl_sync(0xffffffffu, w, 16 * h + l);
          ww[1] = __shfl_sync(0xffffffffu, w, 16 * h + 8 + l);
          const int dst = lane & 15;
          if (dst < P)
            st_async16(cluster_addr(&s_prow[buf][warp * 4 + 2 * h], dst), ww,
                       cluster_addr(&s_mbar[buf], dst));
        } else if (l8 == l && c >= j && c < nbw) {
          gp_publish(p.prow + (size_t)j * kNB + c, w);
        }
      }
      if (c < j && l8 == 0) Gl[c + j * kNB] = part;
      asm volatile("bar.arrive 1, %0;" ::"n"(kGpThreads) : "memory");
      const bool want = c >= j && c < nbw;
      // the receive buffer of column j (this CTA's columns of the cluster, or all)
      const bool collect = ONE || (warp & (kGpCluster - 1)) == rank;
      if (collect) {
        bool reported = s_reported != 0;
        if (!dead && !mbar_wait_bounded(&s_mbar[buf], (unsigned)(j >> 1) & 1u, p.spin, p.status,
                                        &reported)) {
          record_status(p.status, SLQR_ETIMEOUT);
          dead = true;
        }
        if (reported && lane == 0) s_reported = 1;
        const bool last = ONE ? mine : (warp >= kGpCluster || !warp_active(warp + kGpCluster, j));
        if (last && lane == 0 && !dead && j + 2 < nbw && step_bytes(j + 2) > 0)
          mbar_expect(&s_mbar[buf], step_bytes(j + 2));
        __syncwarp();
        if (ONE) {
          if (want) {
            D = l8 < P ? s_recv[buf][l8][c] : 0.0;
            if (l8 + 8 < P) D += s_recv[buf][l8 + 8][c];
            pc = s_prow[buf][c];
          }
          D = gp_sum8(D);
        } else {
          const double sum = gp_sum8(s_recv[buf][l8][(warp >> 3) * 4 + (lane >> 3)]);
          if (l8 == 0 && want) gp_publish(p.rec + ((size_t)j * kNB + c) * NC + cluster, sum);
        }
      }
      if (!ONE) {
        // the clusters' sums of this lane's column, eight clusters at a time
        const double *rec = p.rec + ((size_t)j * kNB + c) * NC;
        const double *prow = p.prow + (size_t)j * kNB + c;
        unsigned it = 0;
        double r[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int q = l8 + 8 * u;
          r[u] = (want && q < NC) ? gp_load(rec + q) : 0.0;
        }
        pc = want ? gp_load(prow) : 0.0;
        while (!dead) {
          const bool miss = gp_unset(pc) || gp_unset(r[0]) || gp_unset(r[1]) || gp_unset(r[2]);
          if (!__any_sync(0xffffffffu, miss)) break;
          if (it == p.spin && lane == 0) record_status(p.status, SLQR_ETIMEOUT);
          if (++it > kSpinLimit) dead = true;
#pragma unroll
          for (int u = 0; u < 3; ++u)
            if (gp_unset(r[u])) r[u] = gp_load(rec + l8 + 8 * u);
          if (gp_unset(pc)) pc = gp_load(prow);
        }
        D = gp_sum8((r[0] + r[1]) + r[2]);
      }
      if (mine) {
        // the pivot, in every lane of this warp
        const double tail = __shfl_sync(0xffffffffu, D, (j & 3) * 8);
        const double x0 = __shfl_sync(0xffffffffu, pc, (j & 3) * 8);
        const double t0 = extreme ? x0 * sc : x0;
        const double S = fma(t0, t0, tail);
        double cl = 0.0, up = 0.0, rb = 0.0;
        if (!extreme && S > exp2i(-900) && S < exp2i(900)) {
          gp_pivot(S, x0, &cl, &up, &rb);
        } else if (S != 0.0) {
          const double s = extreme ? sqrt(S) * exp2i(s_E[j]) : sqrt(S);
          cl = (x0 > 0.0) ? -s : s;
          up = x0 - cl;
          rb = 1.0 / (up * cl);
        }
        if (lane == 0) {
          s_piv[buf][0] = cl;
          s_piv[buf][1] = up;
          s_piv[buf][2] = rb;
          s_def[buf] = S != 0.0;
          s_up[j] = up;
          s_tau[j] = -rb;
        }
      }
    } else {
      // finished columns: their Gram terms while the partials travel
      asm volatile("bar.sync 1, %0;" ::"n"(kGpThreads) : "memory");
      if (warp * 4 < nbw) {
        const double part = dot();
        if (l8 == 0 && c < nbw) Gl[c + j * kNB] = part;
      }
    }
    __syncthreads();
    const bool defined = s_def[buf] != 0;
    const double cl = s_piv[buf][0], up = s_piv[buf][1], rb = s_piv[buf][2];
    if (defined && c > j && c < nbw) {
      const double sig = fma(up, pc, D) * rb;
      if (row0 <= j) {                         // the CTA with the pivot row (or above it)
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          const int r = l8 + 8 * i;
          v[i] = fma(sig, row0 + r == j ? up : x[r], v[i]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < RPL; ++i) v[i] = fma(sig, x[l8 + 8 * i], v[i]);
      }
    }
    if (c == j + 1) {                          // the next column's tail
#pragma unroll
      for (int i = 0; i < RPL; ++i) xs[buf ^ 1][l8 + 8 * i] = (row0 + l8 + 8 * i > j + 1) ? v[i] : 0.0;
    }
    if (defined && c == j && row0 <= j && j < row0 + R) {
#pragma unroll
      for (int i = 0; i < RPL; ++i) v[i] = (row0 + l8 + 8 * i == j) ? cl : v[i];
    }
    __syncthreads();
  }

  // the slice back to the matrix, Vtop (ld NB: zero above the diagonal, up on
  // it, tails below) from the CTAs of the top rows
  double *Vtop = p.wy;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = l8 + 8 * i, row = row0 + r;
    if (!absent(r)) col[at(r)] = v[i];
    if (row < kNB) {
      double t = 0.0;
      if (c < nbw && row < nbw) {
        if (row == c) t = s_up[c];
        else if (row > c && !absent(r)) t = v[i];
      }
      Vtop[c * kNB + row] = t;
    }
  }
  if (row0 + R < kNB && cta == P - 1) {        // a panel shorter than its width
    for (int idx = tid; idx < kNB * kNB; idx += kGpThreads)
      if (idx % kNB >= row0 + R) Vtop[idx] = 0.0;
  }
  double *G = p.wy + (size_t)kNB * kNB, *tau = p.wy + 2 * (size_t)kNB * kNB;
  if (cta == 0 && tid < kNB) {
    tau[tid] = tid < nbw ? s_tau[tid] : 0.0;
    if (tid < nbw) p.up[p.k0 + tid] = s_up[tid];
  }
  // publish the local Gram terms and reduce them, entry idx by CTA idx % P:
  // G[c, j] = v_c[j] up_j + the sum of the tails' dots
  constexpr int NT = kNB * (kNB - 1) / 2;      // strict upper triangle, packed by column
  {
    double *dst = p.gpart + (size_t)cta * NT;
    for (int idx = tid; idx < kNB * kNB; idx += kGpThreads) {
      const int jj = idx / kNB, cc = idx - jj * kNB;
      if (cc < jj) dst[jj * (jj - 1) / 2 + cc] = Gl[idx];
    }
  }
  cluster_sync_all();                          // (nothing is sent to this CTA any more)
  if (!ONE && !grid_barrier(p.bar, p.bar_base + 2u * (unsigned)P, p.status, &s_ok, p.spin)) return;
  // one warp per entry: the CTAs' terms over its lanes
  for (int idx = cta + warp * P; idx < kNB * kNB; idx += P * (kGpThreads / 32)) {
    const int jj = idx / kNB, cc = idx - jj * kNB;
    double g = 0.0;
    if (cc < jj && jj < nbw) {
      const int pos = jj * (jj - 1) / 2 + cc;
      for (int q = lane; q < P; q += 32) g += __ldcg(p.gpart + (size_t)q * NT + pos);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
      if (lane == 0) g = fma(__ldcg(Vtop + cc * kNB + jj), s_up[jj], g);
    }
    if (lane == 0) G[idx] = g;
  }
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
static const void *grid_kernel(int R, bool one) {
  switch (R) {
    case 32: return one ? (const void *)panel_grid_kernel<4, true> : (const void *)panel_grid_kernel<4, false>;
    case 64: return one ? (const void *)panel_grid_kernel<8, true> : (const void *)panel_grid_kernel<8, false>;
    case 128: return one ? (const void *)panel_grid_kernel<16, true> : (const void *)panel_grid_kernel<16, false>;
    case 256: return one ? nullptr : (const void *)panel_grid_kernel<32, false>;
    default: return nullptr;
  }
}

static void grid_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attrs, int P, bool one,
                        cudaStream_t stream) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(P);
  cfg->blockDim = dim3(kGpThreads);
  cfg->dynamicSmemBytes = kNB * kNB * sizeof(double);
  cfg->stream = stream;
  attrs[0].id = cudaLaunchAttributeClusterDimension;
  attrs[0].val.clusterDim.x = one ? P : kGpCluster;
  attrs[0].val.clusterDim.y = 1;
  attrs[0].val.clusterDim.z = 1;
  attrs[1].id = cudaLaunchAttributeCooperative;
  attrs[1].val.cooperative = 1;
  cfg->attrs = attrs;
  cfg->numAttrs = one ? 1 : 2;       // (a cluster is resident as a whole by itself)
}

slqr_status init_grid_panel_attrs(slqr_ctx *ctx) {
  int clusters = 1 << 30;
  bool one_fits = true;
  for (int R : {32, 64, 128, 256})
    for (int one = 0; one < 2; ++one) {
      const void *fn = grid_kernel(R, one);
      if (!fn) continue;
      cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kNB * kNB * (int)sizeof(double));
      if (e == cudaSuccess && one)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess)
        return fail(ctx, SLQR_ECUDA, "cudaFuncSetAttribute(grid panel): %s", cudaGetErrorString(e));
      cudaLaunchConfig_t cfg;
      cudaLaunchAttribute attrs[2];
      grid_config(&cfg, attrs, one ? kClMaxCtas : kGpCluster, one, nullptr);
      cfg.numAttrs = 1;
      int k = 0;
      if (cudaOccupancyMaxActiveClusters(&k, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        k = 0;
      }
      if (one) one_fits = one_fits && k >= 1;
      else clusters = std::min(clusters, k);
    }
  ctx->grid_panel_ctas = clusters * kGpCluster;
  ctx->grid_panel_one = one_fits ? kClMaxCtas : kGpCluster;
  return SLQR_OK;
}

// One cluster up to 16 CTAs of 64 rows, else several.
int grid_panel_rows(const slqr_ctx *ctx, int M, int rows_min, int *ctas) {
  for (int R : {32, 64, 128, 256}) {
    if (rows_min > 0 && R < rows_min && R < 256) continue;
    int P = (M + R - 1) / R;
    if (P <= ctx->grid_panel_one && R <= 128 && (R <= 64 || rows_min > 0)) {
      *ctas = P;
      return R;
    }
    P = (P + kGpCluster - 1) / kGpCluster * kGpCluster;
    const int most = std::min(ctx->grid_panel_ctas, 24 * kGpCluster);
    if (P <= (rows_min > 0 || R == 256 ? most : std::min(most, 64))) {
      if (R < 64 && rows_min == 0 && (M + 63) / 64 <= ctx->grid_panel_one) continue;
      *ctas = P;
      return R;
    }
  }
  return 0;
}

slqr_status launch_grid_panel(slqr_ctx *ctx, GridPanelParams &p, int R, int P, cudaStream_t stream) {
  const bool one = P <= ctx->grid_panel_one && R <= 128;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attrs[2];
  grid_config(&cfg, attrs, P, one, stream);
  void *args[] = {&p};
  cudaError_t e = cudaLaunchKernelExC(&cfg, grid_kernel(R, one), args);
  if (e != cudaSuccess)
    return fail(ctx, SLQR_ECUDA, "panel launch (P=%d, R=%d): %s", P, R, cudaGetErrorString(e));
  p.bar_base += one ? 0u : 2u * (unsigned)P;
  return SLQR_OK;
}

}  // namespace slqr
