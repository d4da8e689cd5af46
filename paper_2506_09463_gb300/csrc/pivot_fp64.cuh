// pivot_fp64.cuh -- the pivot of one reflector (sign rule, up, 1/b) in few
// dependent FP64 operations, for the FP64 panel kernels.
#pragma once

#include <cuda_runtime.h>

namespace slqr {

// Whether S lies within [2^-900, 2^900), from its high word: a comparison of
// doubles would take the FP64 pipe for 64 clocks.
__device__ __forceinline__ bool pivot_in_range(double S) {
  return (unsigned)(__double2hiint(S) - ((1023 - 900) << 20)) < (unsigned)(1800 << 20);
}
// x > 0 from the bits (not for NaN)
__device__ __forceinline__ bool bits_positive(double x) { return __double_as_longlong(x) > 0; }

// s = sqrt(S), cl = -+s, up = x0 - cl and rb = 1 / (up cl) = -1 / (S + |x0| s)
// for S in that range: a third-order Householder iteration each from the
// hardware's approximate reciprocal (square root), good to 2^-20 or so, and a
// Newton correction that takes s to half an ulp (its error enters every entry of
// the reflector).  14 FP64 operations, all of one warp and so 64 clocks apart;
// sqrt() and a division with their range checks take 1600 clocks on an idle
// pipe.
__device__ __forceinline__ void pivot_fp64(double S, double x0, double *cl, double *up, double *rb) {
  double y, z;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(S));
  const double ax = fabs(x0);
  const double s0 = S * y;
  const double b0 = fma(ax, s0, S);                      // approximate -b, for the seed
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(b0));
  const double e = fma(-s0, y, 1.0);                     // 1 - S y^2 = 1 - s0^2 / S
  double s = fma(s0 * e, fma(e, 0.375, 0.5), s0);
  const double hy = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));   // y / 2
  s = fma(fma(-s, s, S), hy, s);
  const double b = fma(ax, s, S);
  const double f = fma(-b, z, 1.0);
  *rb = -fma(fma(f, f, f), z, z);
  const double c = bits_positive(x0) ? -s : s;
  *cl = c;
  *up = x0 - c;
}

struct PivotFp64 {
  double cl, up, rb;
  bool defined;                                  // S != 0
};

// Any S = (2^-E x0)^2 + tail, tail of entries scaled alike.  Kept out of line:
// merged into the caller's code as predicated instructions its multiplications,
// square root and division would take the FP64 pipe on every step.
static __device__ __noinline__ PivotFp64 pivot_fp64_general(double x0, double tail, int E) {
  const double t0 = scalbn(x0, -E);
  const double S = fma(t0, t0, tail);
  PivotFp64 r = {0.0, 0.0, 0.0, S != 0.0};
  if (r.defined) {
    const double s = scalbn(sqrt(S), E);
    r.cl = (x0 > 0.0) ? -s : s;
    r.up = x0 - r.cl;
    r.rb = 1.0 / (r.up * r.cl);
  }
  return r;
}

__device__ __forceinline__ PivotFp64 pivot_fp64(double x0, double tail, bool extreme, int E) {
  if (!extreme) {
    const double S = fma(x0, x0, tail);
    if (pivot_in_range(S)) {
      PivotFp64 r;
      r.defined = true;
      pivot_fp64(S, x0, &r.cl, &r.up, &r.rb);
      return r;
    }
  }
  return pivot_fp64_general(x0, tail, extreme ? E : 0);
}

}  // namespace slqr
