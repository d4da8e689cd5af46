// batch_fx.cu -- the batched FP64 factorization (slqr_batch_factor, default
// setting) with its products on the tensor cores by exact splitting.
//
// One CTA owns one problem at a time, as in batch_core.cuh (same work queue,
// same outputs).  There every product ran on the FP64 pipe, 16 clocks of the SM
// for a warp instruction, at 82% of that pipe's rate.  Here, panels of 16:
//  * the panel lives in registers (16 rows of one column a thread); a column
//    step hands partial dots, the pivot with every multiplier, and the next
//    column through shared memory, three barriers;
//  * V's digits (fx_digits.cuh, the leading one three bits wider) go to shared
//    memory in FP16, and W = V^T C and C -= V W' are digit products with
//    mma.sync (34 of 49, eight orders summed in FP32 below 2^24, so exactly),
//    put together in integer arithmetic.  A warp forms W for 8 columns over all
//    rows, reading C once and splitting it in registers; the Gram terms of V^T V
//    are two more such column tiles.  Column maxima for the digits come from the
//    update before.
//  * results whose digits may be lost (fx_digits.cuh) are formed again in FP64: W and
//    Gram entries by the sums of |leading digits| formed beside them, entries of
//    C -= V W' by their own size and their change's;
//  * W' = T^T W by substitution, one thread per column, in FP64;
//  * the back-substitution goes in blocks of 32 rows.
// CTAs of 4, 8 or 16 warps hold problems of up to 128, 256 or 512 rows, four,
// two or one to an SM.  What bounds it: the column steps (dots, update and pivot
// on the FP64 pipe), then splitting and reassembly on the integer pipe.
#include "batch_core.cuh"
#include "fx_digits.cuh"
#include "pivot_fp64.cuh"

#include <cuda_fp16.h>

namespace slqr {

namespace {

constexpr int kBfNB = 16;
// The line below which digits count as lost (fx_digits.cuh), two binades lower than in
// tc_fp64.cu: the sums of |products| hold every term here, and V is not scaled by rows
// again for C -= V W', whose entries are known to 2^-56 of the column's scale.
constexpr int kBfLoss = 7;

template <int NW>
struct BfSmem {
  static constexpr int PR = 32 * NW;                 // rows
  static constexpr int CT = 8 * NW;                  // columns of a chunk (a tile per warp)
  static constexpr size_t kVd = 0;                                    // [7][PR][16] FP16
  static constexpr size_t kWd = kVd + (size_t)kFxD * PR * 32;         // [7][CT][16] FP16
  static constexpr size_t kWb = kWd + (size_t)kFxD * CT * 32;         // [16][CT + 1]
  static constexpr size_t kXs = kWb + (size_t)16 * (CT + 1) * 8;      // [2][PR]
  static constexpr size_t kCm = kXs + (size_t)2 * PR * 8;             // [2][PR + 8]
  static constexpr size_t kBytes = kCm + (size_t)2 * (PR + 8) * 4;
};

__device__ __forceinline__ uint32_t bf_smem(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// A 16-byte chunk (8 columns) of V's digit row r: the two chunks of rows 4..7 of
// eight swap places, so that eight rows of one chunk meet all banks once.
__device__ __forceinline__ int bf_vrow(int r, int chunk) {
  return r * 32 + ((chunk ^ ((r >> 2) & 1)) << 4);
}
__device__ __forceinline__ void bf_ldsm4(uint32_t (&a)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void bf_ldsm4t(uint32_t (&a)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void bf_ldsm2t(uint32_t &b0, uint32_t &b1, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(b0), "=r"(b1) : "r"(addr) : "memory");
}
// orders o0 .. o0 + 3 of output k
__device__ __forceinline__ long long bf_four(const float (&acc)[kFxOrders][4], int o0, int k) {
  long long v = __float2int_rn(acc[o0 + 3][k]);
  v += (long long)__float2int_rn(acc[o0 + 2][k]) * 256;
  v += (long long)__float2int_rn(acc[o0 + 1][k]) * 65536;
  v += (long long)__float2int_rn(acc[o0][k]) * 16777216;
  return v;
}
// digit pairs (value 0, value 1) of two biased words, most significant first
__device__ __forceinline__ uint32_t bf_pair(unsigned long long y0, unsigned long long y1, int i) {
  const int byte = 7 - i;
  const uint32_t w0 = byte < 4 ? (uint32_t)y0 : (uint32_t)(y0 >> 32);
  const uint32_t w1 = byte < 4 ? (uint32_t)y1 : (uint32_t)(y1 >> 32);
  return fx_half2(w0, w1, byte & 3);
}
// The panel's V in FP64: reflector a's pivot entry on row a, its tail below (stacked: from
// row nbw on)
struct BfPanel {
  const double *A, *up;                              // A at row k0 of column k0
  int lda, nbw, skip, M;
  bool stacked;
};
__device__ __forceinline__ int bf_row(const BfPanel &p, int r) { return r + (r >= p.nbw ? p.skip : 0); }
__device__ __forceinline__ double bf_v(const BfPanel &p, int r, int a) {
  if (r == a) return p.up[a];
  return r < a || (p.stacked && r < p.nbw) ? 0.0 : p.A[(size_t)a * p.lda + bf_row(p, r)];
}
// out[k] = sum_r V(r, a0 + k) x_r for k < 8 on the FP64 pipe, by a warp; x: a column (at row
// k0), or V's own column c where c >= 0
__device__ __noinline__ void bf_dots8(BfPanel p, const double *x, int c, int a0, double *out) {
  const int lane = threadIdx.x & 31;
  double acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.0;
  for (int r = lane; r < p.M; r += 32) {
    const double xr = c >= 0 ? bf_v(p, r, c) : x[bf_row(p, r)];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (a0 + k < p.nbw) acc[k] = fma(bf_v(p, r, a0 + k), xr, acc[k]);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (lane == 0) out[k] = acc[k];
  }
  __syncwarp();
}
// the same for this thread's reflector a, of a panel [L^T; C] with few rows of C (or of few
// rows at all)
constexpr int kBfFewRows = 32;
__device__ __noinline__ double bf_dot1(BfPanel p, const double *x, int c, int a) {
  auto at = [&](int r) { return c >= 0 ? bf_v(p, r, c) : x[bf_row(p, r)]; };
  double s = p.up[a] * at(a);
  const int r0 = p.stacked ? p.nbw : a + 1;
#pragma unroll 4
  for (int r = r0; r < p.M; ++r) s = fma(bf_v(p, r, a), at(r), s);
  return s;
}
// sum_a V(r, a) W'(a) for this thread's row and column (W'(a) at w[a * ldw])
__device__ __noinline__ double bf_entry(BfPanel p, const double *w, int ldw, int r) {
  double s = 0.0;
#pragma unroll 4
  for (int a = 0; a < p.nbw; ++a) s = fma(bf_v(p, r, a), w[a * ldw], s);
  return s;
}

__device__ __forceinline__ double bf_value(long long t, int sh) {
  if (sh >= -1000 && sh <= 900) return fx_to_double(t, sh);
  return fx_scale_slow((double)t, sh);
}

}  // namespace

// The factorization of one problem (and Q^T b for Bcol), NW warps.
template <int NW>
static __device__ __noinline__ void batch_fx_factor(double *A, int lda, int m, int n, double *up_out,
                                                    double *Bcol, unsigned char *sm, int ntop) {
  using SM = BfSmem<NW>;
  constexpr int NT = 32 * NW, PR = SM::PR, CT = SM::CT, RQ = NW / 4;
  __half *Vd = (__half *)(sm + SM::kVd);
  unsigned char *Wd = sm + SM::kWd;
  double *Wb = (double *)(sm + SM::kWb);
  double *xs = (double *)(sm + SM::kXs);
  unsigned *cm = (unsigned *)(sm + SM::kCm);        // column maxima: this panel's, the next one's
  __shared__ double s_part[RQ][16], s_prow[16], s_sig[16], s_piv[2];
  __shared__ double s_G[16 * 16], s_tau[16], s_up[16];
  __shared__ __align__(16) unsigned s_mx[16][RQ];   // maxima of the panel's columns below the diagonal
  __shared__ int s_f[16], s_def, s_ecol[SM::CT];
  __shared__ double s_dot[NW][8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gid = lane >> 2, tq = lane & 3;         // fragment row and column pair
  const int K = num_reflectors(m, n);
  const int cols = n + (Bcol ? 1 : 0);
  auto col_ptr = [&](int q) { return q < n ? A + (size_t)q * lda : Bcol; };
  for (int k = K + tid; k < n; k += NT) up_out[k] = 0.0;

  // column maxima over the rows of panel 0
  for (int q = warp; q < cols; q += NW) {
    const double *C = col_ptr(q);
    unsigned mx = 0;
    for (int r = lane; r < m; r += 32)
      if (ntop == 0 || r >= ntop || (r < kBfNB && (q >= n || r <= q))) mx = max(mx, fx_hi(C[r]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) cm[q] = mx;
  }
  for (int q = tid; q < PR + 8; q += NT) cm[PR + 8 + q] = 0;
  __syncthreads();

  for (int k0 = 0; k0 < K; k0 += kBfNB) {
    const int nbw = min(kBfNB, K - k0);
    const int skip = ntop > 0 ? ntop - k0 - nbw : 0;
    const int M = m - k0 - skip;
    unsigned *cur = cm + ((k0 / kBfNB) & 1) * (PR + 8), *nxt = cm + (((k0 / kBfNB) & 1) ^ 1) * (PR + 8);
    auto prow = [&](int r) { return k0 + r + (r >= nbw ? skip : 0); };
    // ---- the panel: this thread's column and rows l8 + 8 (rq + RQ i) ---------------
    const int cg = warp / RQ, rq = warp % RQ;
    const int c = cg * 4 + (lane >> 3), r0 = (lane & 7) + 8 * rq;
    const int ni = (M + 8 * RQ - 1) / (8 * RQ);
    double v[16];
    {
      const double *C = A + (size_t)(k0 + min(c, nbw - 1)) * lda;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int r = r0 + 8 * RQ * i;
        v[i] = (c < nbw && r < M && !(ntop > 0 && r < nbw && r > c)) ? C[prow(r)] : 0.0;
      }
    }
    {
      // the column's own rows set its scale: an entry above the diagonal may be larger
      // than the norm by more than its square holds
      unsigned mx = 0;
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (i >= 2 || r0 + 8 * RQ * i >= c) mx = max(mx, fx_hi(v[i]));
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if ((lane & 7) == 0) s_mx[c][rq] = mx;
    }
    if (c == 0) {
#pragma unroll
      for (int i = 0; i < 16; ++i) xs[r0 + 8 * RQ * i] = (r0 + 8 * RQ * i > 0) ? v[i] : 0.0;
    }
    __syncthreads();
    for (int j = 0; j < nbw; ++j) {
      const double *x = xs + (j & 1) * PR;
      // a column of extreme scale squares its scaled entries
      unsigned jmx = s_mx[j][0];
#pragma unroll
      for (int q = 1; q < RQ; ++q) jmx = max(jmx, s_mx[j][q]);
      const int E = min(max((int)((jmx >> 20) & 0x7ff) - 1023, -1000), 1022);
      const bool extreme = abs(E) > 400;
      if (4 * cg + 3 >= j && 4 * cg < nbw) {
        double a = 0.0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          if (i >= ni) break;
          const int r = r0 + 8 * RQ * i;
          a = fma(x[r], i < 2 && r <= j ? 0.0 : v[i], a);   // rows up to the pivot's take no part
        }
        if (extreme) {
          if (cg == (j >> 2)) {
            const double sc = b_pow2(-E);
            double n = 0.0;
            for (int r = r0; r < M; r += 8 * RQ) n = fma(x[r] * sc, x[r] * sc, n);
            if (c == j) a = n;
          }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if ((lane & 7) == 0) s_part[rq][c] = a;
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (r0 + 8 * RQ * i == j) s_prow[c] = v[i];
      }
      __syncthreads();
      if (warp == (j & 3) * RQ) {                        // the pivot and every multiplier
        const int cc = lane & 15;
        double D = s_part[0][cc];
#pragma unroll
        for (int q = 1; q < RQ; ++q) D += s_part[q][cc];
        const double p = s_prow[cc], x0 = s_prow[j];
        const PivotFp64 f = pivot_fp64(x0, __shfl_sync(0xffffffffu, D, j), extreme, E);
        if (lane < 16) s_sig[lane] = fma(f.up, p, D) * f.rb;
        if (lane == 0) {
          s_piv[0] = f.cl;
          s_piv[1] = f.up;
          s_def = f.defined;
          s_up[j] = f.up;
          s_tau[j] = -f.rb;
        }
      }
      __syncthreads();
      const bool defined = s_def != 0;
      if (defined && c > j && c < nbw) {
        const double sig = s_sig[c], up = s_piv[1];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          if (i >= ni) break;
          const int r = r0 + 8 * RQ * i;
          if (i < 2) {
            if (r >= j) v[i] = fma(sig, r == j ? up : x[r], v[i]);
          } else {
            v[i] = fma(sig, x[r], v[i]);
          }
        }
      }
      if (c == j + 1) {
        double *xn = xs + ((j & 1) ^ 1) * PR;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int r = r0 + 8 * RQ * i;
          xn[r] = r > j + 1 ? v[i] : 0.0;
        }
      }
      if (defined && c == j) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (r0 + 8 * RQ * i == j) v[i] = s_piv[0];
      }
      __syncthreads();
    }
    // ---- the panel back to the matrix, V's digits to shared memory ------------------
    {
      double *C = A + (size_t)(k0 + min(c, nbw - 1)) * lda;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int r = r0 + 8 * RQ * i;
        if (c < nbw && r < M && !(ntop > 0 && r < nbw && r > c)) C[prow(r)] = v[i];
      }
    }
    if (tid < nbw) up_out[k0 + tid] = s_up[tid];
    const int NC = cols - (k0 + nbw);                    // trailing columns (b the last)
    if (NC <= 0) break;                                  // (the last panel)
    const int nblk = (M + 15) / 16;
    {
      const double upc = c < nbw ? s_up[c] : 0.0;
      const int f = upc == 0.0 ? 0 : fx_exp_of_hi(fx_hi(upc)) - 3;
      if (rq == 0 && (lane & 7) == 0)
        s_f[c] = fx_hi(upc) >= 0x7ff00000u ? kFxNonFinite : f;
      // two lanes (columns c and c ^ 1) trade rows, so that a store is a pair of
      // columns: even columns keep the even i, odd ones the odd
      const int odd = c & 1, cp = c & ~1;
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        if (i * 8 * RQ >= nblk * 16) break;
        unsigned long long y[2];
        int lead[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = r0 + 8 * RQ * (i + h);
          double t = v[i + h];
          if (i < 2 && r <= c) t = r == c ? upc : 0.0;   // (V: zero above the diagonal)
          y[h] = fx_digits_wide(upc == 0.0 ? 0.0 : t, f, &lead[h]);
        }
        const unsigned long long got = __shfl_xor_sync(0xffffffffu, odd ? y[0] : y[1], 8);
        const int lgot = __shfl_xor_sync(0xffffffffu, odd ? lead[0] : lead[1], 8);
        const unsigned long long ya = odd ? got : y[0], yb = odd ? y[1] : got;
        const int r = r0 + 8 * RQ * (i + odd);
        unsigned char *dst = (unsigned char *)Vd + bf_vrow(r, cp >> 3) + (cp & 7) * 2;
        *(__half2 *)dst = __halves2half2(__int2half_rn(odd ? lgot : lead[0]),
                                         __int2half_rn(odd ? lead[1] : lgot));
#pragma unroll
        for (int d = 1; d < kFxD; ++d) *(uint32_t *)(dst + (size_t)d * PR * 32) = bf_pair(ya, yb, d);
      }
    }
    if (tid >= nbw && tid < 16) s_tau[tid] = 0.0;
    __syncthreads();
    // ---- trailing columns in chunks of a tile per warp; tiles 0 and 1 are V's own ----
    const int tiles = 2 + (NC + 7) / 8;
    const uint32_t vd = bf_smem(Vd);
    for (int t0 = 0; t0 < tiles; t0 += NW) {
      const int T = t0 + warp;
      if (T < tiles) {
        // W[a][q] for the tile's 8 columns: rows in blocks of 16
        const bool gram = T < 2;
        const int q = (T - 2) * 8 + gid;                 // this lane's column of the B fragment
        const bool q_ok = !gram && q < NC;
        const double *C = col_ptr(k0 + nbw + (q_ok ? q : 0));
        const int e = fx_exp_of_hi(q_ok ? cur[k0 + nbw + q] : 0u);
        float acc[kFxOrders][4], mag[4] = {0.f, 0.f, 0.f, 0.f};   // (mag: of |leading digits|)
        long long tot[4] = {0, 0, 0, 0};
#pragma unroll
        for (int o = 0; o < kFxOrders; ++o)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[o][k] = 0.f;
        double xv[4];
        auto load = [&](int rb) {
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const int r = rb * 16 + 2 * tq + (h & 1) + 8 * (h >> 1);
            xv[h] = (q_ok && r < M) ? C[prow(r)] : 0.0;
          }
        };
        if (!gram) load(0);
        for (int rb = 0; rb < nblk; ++rb) {
          uint32_t b[kFxD][2];
          if (gram) {
            const int r = rb * 16 + (lane & 15);
#pragma unroll
            for (int j = 0; j < kFxD; ++j)
              bf_ldsm2t(b[j][0], b[j][1], vd + j * PR * 32 + bf_vrow(r, T));
          } else {
            unsigned long long y[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) y[h] = fx_digits(xv[h], e);
#pragma unroll
            for (int j = 0; j < kFxD; ++j) {
              b[j][0] = bf_pair(y[0], y[1], j);
              b[j][1] = bf_pair(y[2], y[3], j);
            }
            if (rb + 1 < nblk) load(rb + 1);
          }
          const int ar = rb * 16 + (lane & 7) + ((lane >> 4) << 3);
          const uint32_t aa = vd + bf_vrow(ar, (lane >> 3) & 1);
#pragma unroll
          for (int i = 0; i < kFxD; ++i) {
            uint32_t a[4];
            bf_ldsm4t(a, aa + i * PR * 32);
            if (i == 0) {
              const uint32_t m[4] = {fx_abs2(a[0]), fx_abs2(a[1]), fx_abs2(a[2]), fx_abs2(a[3])};
              fx_mma16816(mag, m, fx_abs2(b[0][0]), fx_abs2(b[0][1]));
            }
#pragma unroll
            for (int j = 0; j < kFxD; ++j)
              if (i + j < kFxOrders) fx_mma16816(acc[i + j], a, b[j][0], b[j][1]);
          }
          if ((rb & 7) == 7 || rb == nblk - 1) {         // every 128 rows: still exact
#pragma unroll
            for (int k = 0; k < 4; ++k)
              tot[k] += (bf_four(acc, 0, k) << 16) + ((bf_four(acc, 4, k) + (1 << 15)) >> 16);
#pragma unroll
            for (int o = 0; o < kFxOrders; ++o)
#pragma unroll
              for (int k = 0; k < 4; ++k) acc[o][k] = 0.f;
          }
        }
        // totals in units of 2^56 digit products (at most ||x|| ||v|| = 2^118 of them)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int a = gid + 8 * (k >> 1), cc = 2 * tq + (k & 1);
          const int fa = s_f[a];
          if (a >= nbw || fx_hi(s_up[a]) == 0) mag[k] = 1e30f;       // (no such reflector)
          if (gram) {
            const int fc = s_f[T * 8 + cc];
            s_G[a + (T * 8 + cc) * 16] =
                (fa == kFxNonFinite || fc == kFxNonFinite) ? __longlong_as_double(0x7ff8000000000000ll)
                                                           : bf_value(tot[k], fa + fc - 54);
            if (a >= T * 8 + cc || T * 8 + cc >= nbw || fa == kFxNonFinite || fc == kFxNonFinite)
              mag[k] = 1e30f;
            mag[k] *= 0.25f;                         // (2^20 for |up_a up_c|, and one binade lower)
          } else if ((T - 2) * 8 + cc < NC) {
            const unsigned mx = cur[k0 + nbw + (T - 2) * 8 + cc];
            Wb[a * (CT + 1) + warp * 8 + cc] =
                (fa == kFxNonFinite || mx >= 0x7ff00000u) ? __longlong_as_double(0x7ff8000000000000ll)
                                                          : bf_value(tot[k], fx_exp_of_hi(mx) + fa - 54);
            if (fa == kFxNonFinite || mx >= 0x7ff00000u || mx == 0) mag[k] = 1e30f;
          } else {
            mag[k] = 1e30f;
          }
        }
        // the entries whose |products| add up to less than 2^-kBfLoss of the scales (2^17 in
        // leading digits; 2^-(kBfLoss + 1) for the Gram terms), again in FP64
        unsigned low[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          low[k] = __ballot_sync(0xffffffffu, mag[k] < (float)(1 << (17 - kBfLoss)));
        if (low[0] | low[1] | low[2] | low[3]) {
          const BfPanel p = {A + (size_t)k0 * lda + k0, s_up, lda, nbw, skip, M, ntop > 0};
          const bool few = M <= 8 || (ntop > 0 && M - nbw <= kBfFewRows);
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (!few || !(low[k] >> lane & 1)) continue;
            const int a = gid + 8 * (k >> 1), cc = 2 * tq + (k & 1);
            const double *X = gram ? nullptr : col_ptr(k0 + nbw + (T - 2) * 8 + cc) + k0;
            const double d = bf_dot1(p, X, gram ? T * 8 + cc : -1, a);
            if (gram) s_G[a + (T * 8 + cc) * 16] = d;
            else Wb[a * (CT + 1) + warp * 8 + cc] = d;
          }
          for (int cc = few ? 8 : 0; cc < 8; ++cc)
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const unsigned bits = low[2 * t + (cc & 1)] >> (cc >> 1) & 0x11111111u;
              if (bits == 0) continue;
              const double *X = gram ? nullptr : col_ptr(k0 + nbw + (T - 2) * 8 + cc) + k0;
              bf_dots8(p, X, gram ? T * 8 + cc : -1, 8 * t, s_dot[warp]);
              if (lane < 8 && (bits >> (4 * lane) & 1)) {
                const int a = 8 * t + lane;
                if (gram) s_G[a + (T * 8 + cc) * 16] = s_dot[warp][lane];
                else Wb[a * (CT + 1) + warp * 8 + cc] = s_dot[warp][lane];
              }
              __syncwarp();
            }
        }
      }
      __syncthreads();
      // W' = T^T W and its digits, a thread per column
      if (tid < CT) {
        const int q = (t0 - 2) * 8 + tid;
        if (q >= 0 && q < NC) {
          double w[16];
          int key = kFxZero;
          bool bad = false;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            w[j] = 0.0;
            if (j < nbw) {
              double t = Wb[j * (CT + 1) + tid];
#pragma unroll
              for (int a = 0; a < j; ++a) t = fma(-s_G[a + j * 16], w[a], t);
              w[j] = s_tau[j] * t;
              bad |= fx_hi(w[j]) >= 0x7ff00000u;
              // (s_f carries the three bits of the wide digits)
              key = max(key, fx_key(w[j], s_f[j] + 3));
            }
          }
          const int g = key == kFxZero ? 0 : fx_exp(key);
          unsigned long long y[8];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int k = 0; k < 8; ++k) y[k] = fx_digits(w[8 * h + k], g - (s_f[8 * h + k] + 3));
#pragma unroll
            for (int d = 0; d < kFxD; ++d)
              *(uint4 *)(Wd + ((size_t)d * CT + tid) * 32 + h * 16) = fx_pack8(y, d);
          }
          s_ecol[tid] = bad ? kFxNonFinite : key == kFxZero ? kFxZeroExp : g;
#pragma unroll
          for (int j = 0; j < 16; ++j) Wb[j * (CT + 1) + tid] = w[j];   // (for entries formed again)
        }
      }
      __syncthreads();
      // C -= V W' on 16 x 8 tiles: a warp takes a run of row blocks, tile after
      // tile, and keeps a tile's digits of W', pointers and maxima while it lasts
      const int tile_lo = max(t0, 2), tile_hi = min(tiles, t0 + NW);
      const int tasks = (tile_hi - tile_lo) * nblk;
      int task = (int)((long long)tasks * warp / NW);
      const int task_end = (int)((long long)tasks * (warp + 1) / NW);
      while (task < task_end) {
        const int tl = task / nblk;
        int rb = task - tl * nblk;
        const int rb_end = min(nblk, rb + task_end - task);
        task += rb_end - rb;
        const int slot = (tile_lo - t0 + tl) * 8;        // the tile's columns of this chunk
        const int qb = (tile_lo - 2 + tl) * 8 + 2 * tq;  // this lane's two columns
        double *P[2];
        int g[2];
        bool q_ok[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          q_ok[h] = qb + h < NC;
          P[h] = col_ptr(k0 + nbw + min(qb + h, NC - 1));
          g[h] = q_ok[h] ? s_ecol[slot + 2 * tq + h] : 0;
        }
        uint32_t b[kFxD][2];
#pragma unroll
        for (int j = 0; j < kFxD; ++j) {
          const unsigned char *src = Wd + ((size_t)j * CT + slot + gid) * 32 + tq * 4;
          b[j][0] = *(const uint32_t *)src;
          b[j][1] = *(const uint32_t *)(src + 16);
        }
        double xn[4];
        auto load = [&](int blk) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int r = blk * 16 + gid + 8 * (k >> 1);
            xn[k] = (r < M && q_ok[k & 1]) ? P[k & 1][prow(r)] : 0.0;
          }
        };
        load(rb);
        // a column of extreme scale or not finite: exponents out of the quick form's
        // range (the same branch for the warp, so that it costs nothing otherwise)
        const bool odd_scale = __any_sync(0xffffffffu, abs(g[0]) > 800 || abs(g[1]) > 800);
        unsigned mx[2] = {0, 0};
        for (; rb < rb_end; ++rb) {
          double xv[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) xv[k] = xn[k];
          if (rb + 1 < rb_end) load(rb + 1);
          float acc[kFxOrders][4];
#pragma unroll
          for (int o = 0; o < kFxOrders; ++o)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[o][k] = 0.f;
          const uint32_t aa = vd + bf_vrow(rb * 16 + (lane & 15), lane >> 4);
#pragma unroll
          for (int i = 0; i < kFxD; ++i) {
            uint32_t a[4];
            bf_ldsm4(a, aa + i * PR * 32);
#pragma unroll
            for (int j = 0; j < kFxD; ++j)
              if (i + j < kFxOrders) fx_mma16816(acc[i + j], a, b[j][0], b[j][1]);
          }
          // An entry is below the line where it and its change are less than 2^-kBfLoss of
          // the column's scale; half a row of the tile or 3/8 of a column of it count as lost
          // (as in fx_upd_kernel) and are formed again from V and W' in FP64.
          long long tt[4];
          unsigned low = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int h = k & 1;
            // in units of 2^55 digit products, each 2^(g - 113); an order of 16
            // reflectors is below 2^22 (the leading digits of V count eightfold)
            auto pair = [&](int o) { return fx_small(acc[o][k]) * 256 + fx_small(acc[o + 1][k]); };
            tt[k] = fx_join(pair(0), pair(2), pair(4), pair(6), 19);
            constexpr unsigned kLine = 1u << (25 - kBfLoss);
            if ((unsigned)((int)(tt[k] >> 32) + (int)kLine) < 2 * kLine &&
                (int)(fx_hi(xv[k]) >> 20) < g[h] + 1022 - kBfLoss)
              low |= 1u << k;
          }
          if (__any_sync(0xffffffffu, low != 0)) {
            unsigned in[4], lost = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int r = rb * 16 + gid + 8 * (k >> 1), h = k & 1;
              if (r >= M || !q_ok[h] || g[h] == kFxNonFinite) low &= ~(1u << k);
              in[k] = __ballot_sync(0xffffffffu, low >> k & 1);
            }
            const int cols_here = min(8, NC - (tile_lo - 2 + tl) * 8), rows_here = min(16, M - rb * 16);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int in_row = __popc(in[k & 2] >> (4 * gid) & 0xf) +
                                 __popc(in[(k & 2) + 1] >> (4 * gid) & 0xf);
              const int in_col = __popc((in[k & 1] | in[(k & 1) + 2]) >> tq & 0x11111111u) +
                                 __popc((in[k & 1] & in[(k & 1) + 2]) >> tq & 0x11111111u);
              if (2 * in_row >= cols_here || 8 * in_col >= 3 * rows_here) lost |= low & (1u << k);
            }
            if (__any_sync(0xffffffffu, lost != 0)) {
              const BfPanel p = {A + (size_t)k0 * lda + k0, s_up, lda, nbw, skip, M, ntop > 0};
#pragma unroll
              for (int k = 0; k < 4; ++k)
                if (lost >> k & 1) {
                  xv[k] -= bf_entry(p, Wb + slot + 2 * tq + (k & 1), CT + 1,
                                    rb * 16 + gid + 8 * (k >> 1));
                  tt[k] = 0;
                }
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int r = rb * 16 + gid + 8 * (k >> 1), h = k & 1;
            double x;
            if (!odd_scale) x = xv[k] - fx_to_double(tt[k], g[h] - 58);
            else if (g[h] == kFxNonFinite) x = __longlong_as_double(0x7ff8000000000000ll);
            else if (g[h] == kFxZeroExp) x = xv[k];
            else x = xv[k] - bf_value(tt[k], g[h] - 58);
            if (r < M && q_ok[h]) {
              P[h][prow(r)] = x;
              if (rb > 0) mx[h] = max(mx[h], fx_hi(x));  // (rows of the next panel)
            }
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) mx[h] = max(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], o));
          if (gid == 0 && mx[h]) atomicMax(nxt + k0 + nbw + qb + h, mx[h]);
        }
      }
      __syncthreads();
    }
    // the next panel's maxima are complete but for its diagonal rows (stacked);
    // this panel's array is cleared for the one after
    if (ntop > 0) {
      const int k1 = k0 + nbw;
      for (int q = k1 + tid; q < cols; q += NT) {
        const double *C = col_ptr(q);
        unsigned mx = 0;
        for (int r = k1; r < min(k1 + kBfNB, ntop); ++r)
          if (q >= n || r <= q) mx = max(mx, fx_hi(C[r]));
        nxt[q] = max(nxt[q], mx);
      }
    }
    for (int q = tid; q < PR + 8; q += NT) cur[q] = 0;
    __syncthreads();
  }
  __syncthreads();
}

// R x = b[0:n] in blocks of 32 rows from the bottom: warp 0 solves the diagonal
// block, its rows in the lanes (reciprocals of the diagonal formed beforehand),
// then every thread updates its rows above.  An exact zero R_ii sets x_i = 0.
template <int NW>
static __device__ __noinline__ void batch_fx_solve(const double *A, int lda, int n, double *b,
                                                   double *xv, double *rd, int *status_out) {
  constexpr int NT = 32 * NW;
  const int tid = threadIdx.x, lane = tid & 31;
  __shared__ int s_rank;
  if (tid == 0) s_rank = 0;
  __syncthreads();
  for (int i = tid; i < n; i += NT) {
    const double d = A[(size_t)i * lda + i];
    xv[i] = b[i];
    rd[i] = d != 0.0 ? 1.0 / d : 0.0;
    if (d == 0.0) s_rank = 1;
  }
  __syncthreads();
  for (int i0 = (n - 1) / 32 * 32; i0 >= 0; i0 -= 32) {
    const int w = min(32, n - i0);
    if (tid < 32) {
      double R[32];
#pragma unroll
      for (int k = 0; k < 32; ++k)
        R[k] = (k < w && lane < k) ? A[(size_t)(i0 + k) * lda + i0 + lane] : 0.0;
      double x = lane < w ? xv[i0 + lane] : 0.0;
      const double r = lane < w ? rd[i0 + lane] : 0.0;
#pragma unroll
      for (int k = 31; k >= 0; --k) {
        if (k < w) {
          const double xk = __shfl_sync(0xffffffffu, r != 0.0 ? x * r : 0.0, k);
          if (lane == k) x = xk;
          else if (lane < k) x = fma(-R[k], xk, x);
        }
      }
      if (lane < w) xv[i0 + lane] = x;
    }
    __syncthreads();
    for (int i = tid; i < i0; i += NT) {
      double a0 = 0.0, a1 = 0.0;
      int k = 0;
      for (; k + 1 < w; k += 2) {
        a0 = fma(A[(size_t)(i0 + k) * lda + i], xv[i0 + k], a0);
        a1 = fma(A[(size_t)(i0 + k + 1) * lda + i], xv[i0 + k + 1], a1);
      }
      if (k < w) a0 = fma(A[(size_t)(i0 + k) * lda + i], xv[i0 + k], a0);
      xv[i] -= a0 + a1;
    }
    __syncthreads();
  }
  for (int i = tid; i < n; i += NT) b[i] = xv[i];
  if (tid == 0) *status_out = s_rank ? SLQR_ERANK : SLQR_OK;
  __syncthreads();
}

template <int NW>
__global__ void __launch_bounds__(32 * NW, 16 / NW)
batch_fx_kernel(BatchParams bp) {
  extern __shared__ __align__(16) unsigned char bf_raw[];
  __shared__ int s_item, s_status;
  for (;;) {
    if (threadIdx.x == 0) s_item = (int)atomicAdd(bp.counter, 1u);
    __syncthreads();
    const int item = s_item;
    __syncthreads();
    if (item >= bp.count) break;
    const int p = bp.order[item];
    const BatchProblem pr = bp.probs[p];
    if (threadIdx.x == 0) s_status = SLQR_OK;
    if (pr.n > 0) {
      batch_fx_factor<NW>(pr.A, pr.lda, pr.m, pr.n, pr.up, pr.b, bf_raw, pr.ntop);
      if (pr.b) {
        double *xv = (double *)(bf_raw + BfSmem<NW>::kXs);
        batch_fx_solve<NW>(pr.A, pr.lda, pr.n, pr.b, xv, xv + BfSmem<NW>::PR, &s_status);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0 && bp.status) bp.status[p] = s_status;
  }
}

BatchKernels batch_fx_kernels(int rows) {
  BatchKernels k;
  if (rows <= 128) {
    k.fp64 = (const void *)batch_fx_kernel<4>;
    k.smem_fp64 = BfSmem<4>::kBytes;
    k.threads_fp64 = 128;
  } else if (rows <= 256) {
    k.fp64 = (const void *)batch_fx_kernel<8>;
    k.smem_fp64 = BfSmem<8>::kBytes;
    k.threads_fp64 = 256;
  } else {
    k.fp64 = (const void *)batch_fx_kernel<16>;
    k.smem_fp64 = BfSmem<16>::kBytes;
    k.threads_fp64 = 512;
  }
  return k;
}

}  // namespace slqr
