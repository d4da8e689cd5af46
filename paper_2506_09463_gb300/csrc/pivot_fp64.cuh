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
// for S in that range, by Newton's iteration from the approximate reciprocal
// square root and reciprocal that PTX has for FP64:
//  * s: x^2 = S with the slope kept at its first value (the simplified Newton or
//    chord iteration; Ortega and Rheinboldt 1970, section 7.1), s <- s + (S - s^2) h
//    with h = y / 2.  From y = (1 + d) / sqrt(S), s = S y has the relative error d,
//    the first step leaves -3/2 d^2 - d^3/2 and the second 3/2 d^3: with |d| below
//    2^-19, 2^-56 of s before the last rounding.
//  * rb: z <- z + z (1 - b z), whose error is squared (Newton).  The first step
//    is on the b of the first s, beside the second step of s; it leaves 2^-37,
//    so the second, on the final b, is exact but for its rounding.
// Eight FP64 operations one after the other, of one warp and so 64 clocks apart;
// sqrt() and a division with their range checks take 1600 clocks on an idle
// pipe.  s is within 0.55 units in the last place and rb within 3 2^-53 of itself,
// the error of sqrt, x0 - cl, a product and a division being up to 5 2^-53
// (tests/test_gpu_pivot.py).
__device__ __forceinline__ void pivot_fp64(double S, double x0, double *cl, double *up, double *rb) {
  double y, z;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(S));
  const double ax = fabs(x0), h = 0.5 * y;
  double s = S * y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(fma(ax, s, S)));
  s = fma(fma(-s, s, S), h, s);
  z = fma(z, fma(-fma(ax, s, S), z, 1.0), z);
  s = fma(fma(-s, s, S), h, s);
  *rb = -fma(z, fma(-fma(ax, s, S), z, 1.0), z);
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
