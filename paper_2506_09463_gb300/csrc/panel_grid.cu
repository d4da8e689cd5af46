// panel_grid.cu -- the FP64 panel of 64 columns by thread-block clusters with
// the panel held in registers.
//
// Same arithmetic and outputs as panel_kernel (factor.cu; Alg. 2 of the paper
// on one panel): the scaled norm, the sign rule and up of Alg. 3, the reflector
// applied to the later columns; Vtop and tau for the compact-WY update.  The
// Gram terms of V^T V, a third of the panel's FP64 work there, are formed from
// the digits of V instead (fx_gram_block in tc_fp64.cu).
//
// What bounds a column step: every FP64 warp instruction takes the SM's FP64
// pipe for 16 clocks, the next one of the same warp starts 64 clocks later, and
// the step is a chain of two passes over the slice, a sum over all CTAs and the
// pivot's square root and division.  So:
//  * The slice is spread over many CTAs (R = 32 .. 256 rows each) and lives in
//    registers: warp w holds columns 4 w .. 4 w + 3, eight lanes to a column,
//    lane l of them rows l, l + 8, ...  A column's dot needs three butterfly
//    adds (for four columns at once) instead of five per column or a pass
//    through shared memory.
//  * Partial dots go out straight from registers.  Up to 16 CTAs are one
//    cluster: each warp pushes its columns' partials to every CTA (st.async,
//    counted on an mbarrier there).  More CTAs are clusters of 8 or 4: the
//    partials of a column go to one CTA of the cluster, whose collecting warp
//    adds them and publishes the sum in L2; every CTA polls the clusters' sums.
//    (Without the first level every CTA reads every CTA's record: 128 CTAs spent
//    3.5 us of a 7.4 us step in those reads; norms alone sent that way, around
//    the first level, cost 0.8 us a step on 64 CTAs.)
//  * The sums over all CTAs are taken by four warps, 16 columns each, so that at
//    most five warps share the pipe with the pivot's chain.  (On all sixteen,
//    four columns each, the sums took 1200 clocks of a step and the chain 1700:
//    3.0 us a column at 512 rows against 2.5, 4.4 against 3.6 at 2048.)
//  * A reflector is applied and the next column's dots are taken in one go: the
//    next column's warp hands it over through shared memory and goes on, and one
//    CTA barrier a step, after the multipliers, is left.  In one cluster its
//    partials are counted apart from the others', so that the pivot starts while
//    the other columns' sums are still coming.
// Microseconds a column (with 64 columns): 2.5 at 512 rows, 3.5 at 1100, 3.6 at
// 2048, 4.3 at 4096, 5.7 at 8192, 8.5 at 16384; panel_kernel took 9.8 at 8192.
#include "cluster_common.cuh"
#include "pivot_fp64.cuh"

#include <algorithm>

namespace slqr {
using namespace cl;

namespace {

constexpr int kGpThreads = 512;
constexpr int kNB = 64;
constexpr int kGpPolls = 5;            // clusters' sums a lane collects (40 clusters at most)
constexpr int kGpPivot = 3;            // the warp of the pivot
constexpr int kGpCollector = 5;        // the warp that adds up a cluster's partials

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

}  // namespace

// RPL rows per lane, R = 8 RPL rows per CTA; ONE: the grid is one cluster.
template <int RPL, bool ONE>
__global__ void __launch_bounds__(kGpThreads, 1)
panel_grid_kernel(GridPanelParams p) {
  constexpr int R = 8 * RPL;
  constexpr int SRC = ONE ? kClMaxCtas : 8;                // senders to a receive buffer
  constexpr int RC = ONE ? kNB : 16;                       // columns of a receive buffer
  __shared__ __align__(16) double xs[2][R];   // column j's tail by j & 1 (zero elsewhere)
  __shared__ __align__(16) double s_recv[2][SRC][RC];
  __shared__ __align__(16) double s_prow[2][ONE ? kNB : 2];
  __shared__ unsigned s_mx[kNB];
  __shared__ int s_E[kNB];
  __shared__ double s_up[kNB], s_tau[kNB];
  __shared__ double s_piv[2][3], s_sig[2][kNB];   // cl, up, 1/b; the columns' multipliers, by j & 1
  __shared__ int s_def[2];
  __shared__ __align__(8) unsigned long long s_mbar[2], s_nbar[2];   // sums, column j's warp's
  __shared__ int s_ok, s_reported;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = warp * 4 + (lane >> 3), l8 = lane & 7;     // this lane's column and rows
  const int cta = blockIdx.x, P = gridDim.x;
  const int rank = cluster_rank(), CS = cluster_ctas();
  const int NC = P / CS, cluster = cta / CS;
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

  // Bytes the receive buffer gets for column j.  ONE: every CTA's partials of
  // the active warps and the pivot row, less those of column j's warp, which
  // are counted on s_nbar; else the cluster's partials of the active warps
  // w = rank, rank + CS, ... (32 bytes each).
  auto warp_active = [&](int w, int j) { return 4 * w + 3 >= j && 4 * w < nbw; };
  auto step_bytes = [&](int j) -> unsigned {
    if (ONE) return (unsigned)((P + 1) * ((nbw + 3) / 4 - j / 4 - 1) * 32);
    int act = 0;
    for (int w = rank; w < kGpThreads / 32; w += CS) act += warp_active(w, j);
    return (unsigned)(CS * 32 * act);
  };
  if (tid == 0) {
    mbar_init1(&s_mbar[0]);
    mbar_init1(&s_mbar[1]);
    mbar_init1(&s_nbar[0]);
    mbar_init1(&s_nbar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // columns 0 and 1; column j + 2's phase is announced once column j's has
    // completed, before this CTA sends anything for column j + 1
    for (int j = 0; j < 2; ++j)
      if (j < nbw && step_bytes(j) > 0) mbar_expect(&s_mbar[j], step_bytes(j));
    if (ONE)
      for (int j = 0; j < 2 && j < nbw; ++j) mbar_expect(&s_nbar[j], (unsigned)(P + 1) * 32);
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
    for (int r = 0; r < CS; ++r) all &= cluster_ld_u32(cluster_addr(&s_ok, r)) != 0;
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
  __syncthreads();
  if (tid < kNB) {
    const int E = (int)((s_mx[tid] >> 20) & 0x7ff) - 1023;
    s_E[tid] = min(max(E, -1000), 1022);
  }
  __syncthreads();

  // Who takes the sums over all CTAs: four warps, 16 columns cs and two lanes to
  // a column; the warps whose own columns end first take those that end last.
  // More clusters than two lanes can poll: every warp its own columns.
  const int cshift = ONE || NC <= 2 * kGpPolls ? 4 : 2;
  const int sw = cshift == 2 ? warp : (warp < 3 ? 3 - warp : warp == 7 ? 0 : 16);
  const int cs = (sw << cshift) + (lane & ((1 << cshift) - 1)), sub = lane >> cshift;
  auto wait = [&](unsigned long long *bar, unsigned parity) {
    bool reported = s_reported != 0;
    if (!dead && !mbar_wait_bounded(bar, parity & 1u, p.spin, p.status, &reported, 1u << 16)) {
      record_status(p.status, SLQR_ETIMEOUT);
      dead = true;
    }
    if (reported && lane == 0) s_reported = 1;
    __syncwarp();
  };
  // Named barriers between column j's warp (which does not wait) and the active
  // warps of a quarter of the SM, w = g mod 4
  auto quarter_threads = [&](int g, int j) {
    const int n = (((nbw - 1) >> 2) - g >> 2) - ((j >> 2) - 1 - g >> 2);
    return 32 * (n + (((j >> 2) & 3) != g));
  };
  auto quarter_arrive = [&](int g, int j) {
    const int n = quarter_threads(g, j);
    if (n > 32) asm volatile("bar.arrive %0, %1;" ::"r"(2 + g), "r"(n) : "memory");
  };
  auto quarter_sync = [&](int g, int j) {
    asm volatile("bar.sync %0, %1;" ::"r"(2 + g), "r"(quarter_threads(g, j)) : "memory");
  };
  // reflector k to this lane's column (the multipliers of step k)
  auto apply = [&](int k) {
    const int b = k & 1;
    const double *x = xs[b];
    if (s_def[b] && c > k && c < nbw) {
      const double sig = s_sig[b][c], up = s_piv[b][1];
      if (row0 <= k) {                         // the CTA with the pivot row (or above it)
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          const int r = l8 + 8 * i;
          if (row0 + r >= k) v[i] = fma(sig, row0 + r == k ? up : x[r], v[i]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < RPL; ++i) v[i] = fma(sig, x[l8 + 8 * i], v[i]);
      }
    }
  };
  // the diagonal entry to column k
  auto diagonal = [&](int k) {
    if (s_def[k & 1] && c == k && row0 <= k && k < row0 + R) {
      const double cl = s_piv[k & 1][0];
#pragma unroll
      for (int i = 0; i < RPL; ++i) v[i] = (row0 + l8 + 8 * i == k) ? cl : v[i];
    }
  };

  for (int j = 0; j < nbw; ++j) {
    const int buf = j & 1;
    const unsigned phase = (unsigned)(j >> 1) & 1u;
    const double *x = xs[buf];
    const bool mine = (j >> 2) == warp;        // this warp holds column j
    // a column of extreme scale squares its scaled entries (uniform)
    const bool extreme = abs(s_E[j]) > 400;

    // Reflector j - 1, then the dots with column j.  Its warp does not wait for
    // the others, and those of its quarter let it go first where its norm makes
    // its own way to the pivot.
    if (warp_active(warp, j)) {
      const int quarter = (j >> 2) & 3;
      if (ONE && !mine && (warp & 3) == quarter) quarter_sync(warp & 3, j);
      if (j > 0) apply(j - 1);
      if (mine) {
        if (c == j) {                          // its tail to the other warps
#pragma unroll
          for (int i = 0; i < RPL; ++i)
            xs[buf][l8 + 8 * i] = (row0 + l8 + 8 * i > j) ? v[i] : 0.0;
        }
        __syncwarp();
        for (int g = 0; g < 4; ++g)
          if (!ONE || g != quarter) quarter_arrive(g, j);
      } else if (!ONE || (warp & 3) != quarter) {
        quarter_sync(warp & 3, j);
      }
      // dot of the tail of x_j with this lane's column (c == j: its norm); one
      // chain up to 8 terms: an FP64 operation's latency is the time the pipe
      // takes to issue it
      double part = 0.0, part1 = 0.0;
      if (row0 <= j) {                         // rows up to the pivot's take no part
#pragma unroll
        for (int i = 0; i < RPL; ++i)
          part = fma(x[l8 + 8 * i], row0 + l8 + 8 * i > j ? v[i] : 0.0, part);
      } else {
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          if (RPL > 8 && (i & 1)) part1 = fma(x[l8 + 8 * i], v[i], part1);
          else part = fma(x[l8 + 8 * i], v[i], part);
        }
      }
      if (extreme && mine) {
        const double sc = exp2i(-s_E[j]);
        double n = 0.0;
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          const double t = x[l8 + 8 * i] * sc;
          n = fma(t, t, n);
        }
        if (c == j) part = n, part1 = 0.0;
      }
      if (RPL > 8) part += part1;
      part = gp_sum8(part);
      if (ONE && mine) quarter_arrive(quarter, j);
      // two columns' partials per lane half, 16 bytes to a receiver
      const int h = lane >> 4;
      unsigned long long *bar = mine && ONE ? &s_nbar[buf] : &s_mbar[buf];
      {
        double w[2];
        w[0] = __shfl_sync(0xffffffffu, part, 16 * h);
        w[1] = __shfl_sync(0xffffffffu, part, 16 * h + 8);
        if (ONE) {
          const int dst = lane & 15;
          if (dst < P)
            st_async16(cluster_addr(&s_recv[buf][rank][warp * 4 + 2 * h], dst), w,
                       cluster_addr(bar, dst));
        } else if ((lane & 15) == 0) {
          const int dst = warp % CS;
          st_async16(cluster_addr(&s_recv[buf][rank][(warp / CS) * 4 + 2 * h], dst), w,
                     cluster_addr(bar, dst));
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
                       cluster_addr(bar, dst));
        } else if (l8 == l && c >= j && c < nbw) {
          gp_publish(p.prow + (size_t)j * kNB + c, w);
        }
      }
    }
    if (j > 0 && (j - 1) >> 2 == warp) diagonal(j - 1);
    // the cluster's sums of this CTA's columns: one warp, CS / 2 lanes a column
    if (!ONE && warp == kGpCollector && step_bytes(j) > 0) {
      wait(&s_mbar[buf], phase);
      if (lane == 0 && !dead && j + 2 < nbw && step_bytes(j + 2) > 0)
        mbar_expect(&s_mbar[buf], step_bytes(j + 2));
      __syncwarp();
      const int half = CS / 2, q = CS == 8 ? lane >> 2 : lane >> 1, l = lane & (half - 1);
      double sum = s_recv[buf][l][q] + s_recv[buf][l + half][q];
      for (int o = 1; o < half; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const int cc = ((q >> 2) * CS + rank) * 4 + (q & 3);
      if (l == 0 && cc >= j && cc < nbw)
        gp_publish(p.rec + ((size_t)j * NC + cluster) * kNB + cc, sum);
    }
    // the pivot, in every lane of a warp
    auto pivot = [&](double x0, double tail) {
      const PivotFp64 f = pivot_fp64(x0, tail, extreme, s_E[j]);
      if (lane == 0) {
        s_piv[buf][0] = f.cl;
        s_piv[buf][1] = f.up;
        s_piv[buf][2] = f.rb;
        s_def[buf] = f.defined;
        s_up[j] = f.up;
        s_tau[j] = -f.rb;
      }
    };
    if (ONE && warp == kGpPivot) {
      wait(&s_nbar[buf], phase);
      if (lane == 0 && !dead && j + 2 < nbw) mbar_expect(&s_nbar[buf], (unsigned)(P + 1) * 32);
      __syncwarp();
      double tail = lane < P ? s_recv[buf][lane][j] : 0.0;
      if (P > 8) tail += __shfl_xor_sync(0xffffffffu, tail, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) tail += __shfl_xor_sync(0xffffffffu, tail, o);
      pivot(s_prow[buf][j], __shfl_sync(0xffffffffu, tail, 0));
    }
    // the columns' sums and their multipliers (of the columns after j; in a
    // cluster panel column j's sum is among them, and its warp takes the pivot)
    const int c0 = ONE ? j + 1 : j;
    const int first = c0 >> cshift, last = (nbw - 1) >> cshift;
    const bool summing = c0 < nbw && sw >= first && sw <= last;
    double D = 0.0, pc = 0.0;
    if (summing) {
      if (ONE) {
        wait(&s_nbar[buf], phase);
        if (step_bytes(j) > 0) wait(&s_mbar[buf], phase);
        if (sw == last && lane == 0 && !dead && j + 2 < nbw && step_bytes(j + 2) > 0)
          mbar_expect(&s_mbar[buf], step_bytes(j + 2));
        __syncwarp();
        D = sub < P ? s_recv[buf][sub][cs] : 0.0;
#pragma unroll
        for (int q = 2; q < kClMaxCtas; q += 2) {
          if (q >= P) break;
          D += q + sub < P ? s_recv[buf][q + sub][cs] : 0.0;
        }
        D += __shfl_xor_sync(0xffffffffu, D, 16);
        pc = s_prow[buf][cs];
      } else {
        const bool want = cs >= j && cs < nbw;
        const double *rec = p.rec + ((size_t)j * NC + sub) * kNB + cs;
        const double *prow = p.prow + (size_t)j * kNB + cs;
        const int subs = 32 >> cshift;
        unsigned it = 0;
        double r[kGpPolls];
#pragma unroll
        for (int u = 0; u < kGpPolls; ++u)
          r[u] = (want && sub + u * subs < NC) ? gp_load(rec + (size_t)u * subs * kNB) : 0.0;
        pc = want ? gp_load(prow) : 0.0;
        while (!dead) {
          bool miss = gp_unset(pc);
#pragma unroll
          for (int u = 0; u < kGpPolls; ++u) miss |= gp_unset(r[u]);
          if (!__any_sync(0xffffffffu, miss)) break;
          if (it == p.spin && lane == 0) record_status(p.status, SLQR_ETIMEOUT);
          if (++it > kSpinLimit) dead = true;
#pragma unroll
          for (int u = 0; u < kGpPolls; ++u)
            if (gp_unset(r[u])) r[u] = gp_load(rec + (size_t)u * subs * kNB);
          if (gp_unset(pc)) pc = gp_load(prow);
        }
        // (adds of absent clusters are skipped, uniformly)
        D = r[0];
#pragma unroll
        for (int u = 1; u < kGpPolls; ++u)
          if (u * subs < NC) D += r[u];
        for (int o = 16; o >= 1 << cshift; o >>= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
        if (sw == first) {
          const int l = j & ((1 << cshift) - 1);
          const double x0 = __shfl_sync(0xffffffffu, pc, l);
          pivot(x0, __shfl_sync(0xffffffffu, D, l));
        }
      }
    }
    // the pivot to the summing warps
    if (summing || (ONE && warp == kGpPivot)) {
      const int n = (c0 < nbw ? last - first + 1 : 0) + (ONE ? 1 : 0);
      asm volatile("bar.sync 1, %0;" ::"r"(32 * n) : "memory");
      if (summing && sub == 0) s_sig[buf][cs] = fma(s_piv[buf][1], pc, D) * s_piv[buf][2];
    }
    __syncthreads();
  }
  if (warp == (nbw - 1) >> 2) diagonal(nbw - 1);

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
  double *tau = p.wy + 2 * (size_t)kNB * kNB;
  if (cta == 0 && tid < kNB) {
    tau[tid] = tid < nbw ? s_tau[tid] : 0.0;
    if (tid < nbw) p.up[p.k0 + tid] = s_up[tid];
  }
  cluster_sync_all();                          // (nothing is sent to this CTA any more)
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
constexpr int kGridRows[] = {32, 48, 64, 80, 96, 128, 160, 192, 256};
static const void *grid_kernel(int R, bool one) {
  switch (R) {
    case 32: return one ? (const void *)panel_grid_kernel<4, true> : (const void *)panel_grid_kernel<4, false>;
    case 64: return one ? (const void *)panel_grid_kernel<8, true> : (const void *)panel_grid_kernel<8, false>;
    case 128: return one ? (const void *)panel_grid_kernel<16, true> : (const void *)panel_grid_kernel<16, false>;
    case 48: return one ? (const void *)panel_grid_kernel<6, true> : (const void *)panel_grid_kernel<6, false>;
    case 80: return one ? (const void *)panel_grid_kernel<10, true> : (const void *)panel_grid_kernel<10, false>;
    case 96: return one ? (const void *)panel_grid_kernel<12, true> : (const void *)panel_grid_kernel<12, false>;
    case 160: return one ? nullptr : (const void *)panel_grid_kernel<20, false>;
    case 192: return one ? nullptr : (const void *)panel_grid_kernel<24, false>;
    case 256: return one ? nullptr : (const void *)panel_grid_kernel<32, false>;
    default: return nullptr;
  }
}

static void grid_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attrs, int P, int cluster,
                        cudaStream_t stream) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(P);
  cfg->blockDim = dim3(kGpThreads);
  cfg->stream = stream;
  attrs[0].id = cudaLaunchAttributeClusterDimension;
  attrs[0].val.clusterDim.x = cluster;
  attrs[0].val.clusterDim.y = 1;
  attrs[0].val.clusterDim.z = 1;
  attrs[1].id = cudaLaunchAttributeCooperative;
  attrs[1].val.cooperative = 1;
  cfg->attrs = attrs;
  cfg->numAttrs = P == cluster ? 1 : 2;        // (a cluster is resident as a whole by itself)
}

// CTAs that can be resident at once in clusters of 4, of 8 and as one cluster
slqr_status init_grid_panel_attrs(slqr_ctx *ctx) {
  int c4 = 1 << 20, c8 = 1 << 20;
  bool one_fits = true;
  for (int R : kGridRows)
    for (int one = 0; one < 2; ++one) {
      const void *fn = grid_kernel(R, one);
      if (!fn) continue;
      if (one) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess)
          return fail(ctx, SLQR_ECUDA, "cudaFuncSetAttribute(grid panel): %s", cudaGetErrorString(e));
      }
      auto clusters = [&](int size) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attrs[2];
        grid_config(&cfg, attrs, size, size, nullptr);
        int k = 0;
        if (cudaOccupancyMaxActiveClusters(&k, fn, &cfg) != cudaSuccess) {
          cudaGetLastError();
          k = 0;
        }
        return k;
      };
      if (one) {
        one_fits = one_fits && clusters(kClMaxCtas) >= 1;
      } else {
        c4 = std::min(c4, clusters(4));
        c8 = std::min(c8, clusters(8));
      }
    }
  ctx->grid_panel_c4 = std::min(4 * c4, 4 * 8 * kGpPolls) / 4 * 4;
  ctx->grid_panel_c8 = std::min(8 * c8, 8 * 8 * kGpPolls) / 8 * 8;
  ctx->grid_panel_one = one_fits ? kClMaxCtas : 8;
  return SLQR_OK;
}

// Rows per CTA, smallest first.  One cluster up to 16 CTAs of 80 rows (1100 rows:
// 0.1 us a column less than 35 CTAs of 32 rows in clusters of 8; 1300 rows on CTAs of
// 96: 0.1 more).  Above that clusters of 8, 64 CTAs at most while 256 rows
// each are enough: the sums of more clusters take longer to arrive than the
// shorter slices save (8192 rows: 6.2 us a column on 64 CTAs, 7.6 on 104), and the
// trailing update runs on the other SMs.
GridPanelShape grid_panel_shape(const slqr_ctx *ctx, int M, int rows_min) {
  GridPanelShape s;
  const int one = ctx->grid_panel_one;
  for (int R : kGridRows) {
    const int P = (M + R - 1) / R;
    if (rows_min > 0 && R < rows_min && R < 256) continue;
    if (P <= one && grid_kernel(R, true) && (R <= 80 || rows_min > 0)) {
      s.R = R, s.P = P, s.cluster = P;
      return s;
    }
    if (rows_min == 0 && R < 80 && (M + 79) / 80 <= one) continue;
    const int P8 = (P + 7) / 8 * 8;
    if (P8 <= std::min(ctx->grid_panel_c8, rows_min > 0 || R == 256 ? ctx->grid_panel_c8 : 64) &&
        (P8 > one || !grid_kernel(R, true))) {
      s.R = R, s.P = P8, s.cluster = 8;
      return s;
    }
  }
  const int P4 = ((M + 255) / 256 + 3) / 4 * 4;
  if (P4 <= ctx->grid_panel_c4) s.R = 256, s.P = P4, s.cluster = 4;
  return s;                                    // R = 0: too tall
}

slqr_status launch_grid_panel(slqr_ctx *ctx, GridPanelParams &p, const GridPanelShape &s,
                              cudaStream_t stream) {
  const bool one = s.P == s.cluster && grid_kernel(s.R, true);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attrs[2];
  grid_config(&cfg, attrs, s.P, s.cluster, stream);
  void *args[] = {&p};
  cudaError_t e = cudaLaunchKernelExC(&cfg, grid_kernel(s.R, one), args);
  if (e != cudaSuccess)
    return fail(ctx, SLQR_ECUDA, "panel launch (P=%d, R=%d): %s", s.P, s.R, cudaGetErrorString(e));
  p.bar_base += one ? 0u : (unsigned)s.P;
  return SLQR_OK;
}

}  // namespace slqr
