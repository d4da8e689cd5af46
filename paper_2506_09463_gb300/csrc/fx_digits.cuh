// fx_digits.cuh -- device helpers of the exact splitting of FP64 values into
// balanced base-256 digits (tc_fp64.cu has the scheme): exponents of vector
// maxima, digits, their FP16 form, and the reassembly of order sums.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace slqr {

constexpr int kFxD = 7;                       // digits
constexpr int kFxOrders = 8;                  // accumulated orders i + j
constexpr int kFxNonFinite = 1 << 20;         // exponent that stands for Inf / NaN

// Where the splitting loses digits.  A digit product of two vectors is known to 2^-57
// or so of the product of their largest entries.  An FP64 sum is as accurate as the
// terms it has: where the largest entries of the two meet small ones of the other (rows
// that differ in scale), the sum of |terms| is far below that product and the digits of
// the terms are lost.  So every result is held against a lower bound of its sum of
// |terms|; one whose bound is below 2^-kFxLoss of the product of the scales is formed
// again on the FP64 pipe from the operands in FP64.  At the line the error is 2^-51 of
// the terms, what FP64 leaves of a sum of a hundred.  Row-wise error of the factorization
// of 330 x 270 with the first 100 rows weighted by 2^13 and 2^33, in units of 2^-53: 7600
// and 6e9 without this, 190 and 190 with it, 760 and 330 for the same panels in FP64
// throughout (tests/test_gpu_row_scale.py).  Time: 8192 x 8192 60.0 -> 61.5 ms,
// 16384 x 2048 20.6 -> 20.8, 1203 x 1001 3.68 -> 3.82, [L^T; C] of 4000 + 1000 17.1 -> 17.7.
constexpr int kFxLoss = 5;

// The exponent of a vector of zeros, whose digits are exact.
constexpr int kFxZeroExp = -(1 << 20);

// High word of |x| (sign cleared): ordered as |x|.
__device__ __forceinline__ uint32_t fx_hi(double x) {
  return (uint32_t)__double2hiint(x) & 0x7fffffffu;
}

// Key of a vector maximum: the high word of |x| with the exponent unbiased (a
// denormal counts as its binade), plus a power of two as `shift` exponents;
// kFxZero for a zero.
constexpr int kFxZero = -0x7fffffff;
__device__ __forceinline__ int fx_key_of_hi(uint32_t hi) {
  return (int)(hi < 0x00100000u ? (hi | 0x00100000u) : hi) - (1023 << 20);
}
__device__ __forceinline__ int fx_key(double x, int shift) {
  return x != 0.0 ? fx_key_of_hi(fx_hi(x)) + shift * (1 << 20) : kFxZero;
}

// Exponent e of a vector whose largest entry has this key: every entry is at
// most 1.9883 * 2^(e-1), so that |x| 2^(55-e) stays within the balanced digits
// (127 (256^7 - 1) / 255 = 1.9921 * 2^54).
__device__ __forceinline__ int fx_exp(int key) {
  return (key >> 20) + 1 + ((key & 0xfffff) >= 0xFD000 ? 1 : 0);   // (shift: floor)
}

__device__ __forceinline__ int fx_exp_of_hi(uint32_t hi) { return fx_exp(fx_key_of_hi(hi)); }

// round(x 2^(55-e)) as seven balanced digits, each biased by 128: byte 7 - i of
// the result is d_i + 128, byte 0 what the rounding left.  With t = |x| 2^(63-e)
// (truncated) and its complement for a negative x, adding the biases and half a
// unit does the rounding and the sign at once.
__device__ __forceinline__ unsigned long long fx_digits(double x, int e) {
  const int hi = __double2hiint(x);
  const int Ef = (hi >> 20) & 0x7ff;
  const unsigned mh = (unsigned)hi & 0xfffffu;
  unsigned long long t =
      ((unsigned long long)(Ef ? (mh | 0x100000u) : mh) << 32) | (unsigned)__double2loint(x);
  t <<= 10;
  // (a shift past 63 gives 0)
  asm("shr.u64 %0, %0, %1;" : "+l"(t) : "r"(max(1022 + e - max(Ef, 1), 0)));
  const unsigned long long s = (unsigned long long)(long long)(hi >> 31);
  return 0x8080808080808080ull + (t ^ s);
}

// The same with three bits more for the leading digit (|x| up to 2^3 times the
// bound above): bytes 6 .. 1 the biased digits 1 .. 6, `lead` the signed leading
// one, at most 1024 in magnitude (exact in FP16).
__device__ __forceinline__ unsigned long long fx_digits_wide(double x, int e, int *lead) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int Ef = (int)(b >> 52) & 0x7ff;
  unsigned long long m = b & 0xfffffffffffffull;
  m |= Ef ? (1ull << 52) : 0ull;
  const int rsh = min(max(1022 + e + 3 - max(Ef, 1), 0), 62);
  m = (((m << 6) >> rsh) + 1) >> 1;                       // (m << 5) >> rsh, rounded
  const long long bias = 0x808080808080ll;
  const long long v = (long long)b < 0 ? bias - (long long)m : bias + (long long)m;
  *lead = (int)(v >> 48);
  return (unsigned long long)v << 8;
}

// The digits at byte `byte` of two biased words as two FP16 values (low, high).
__device__ __forceinline__ uint32_t fx_half2(uint32_t w0, uint32_t w1, int byte) {
  // bytes w0[byte], 0x64, w1[byte], 0x64: 1024 + u in each half (exact in FP16)
  const uint32_t r =
      (__byte_perm(w0, w1, byte | ((4 + byte) << 8)) & 0x00ff00ffu) | 0x64006400u;
  uint32_t o;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(o) : "r"(r), "r"(0x64806480u));   // minus 1152
  return o;
}

// Eight values' digits i as 16 bytes (value k in half k).
__device__ __forceinline__ uint4 fx_pack8(const unsigned long long (&y)[8], int i) {
  const int byte = 7 - i;
  uint32_t o[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint32_t w0 = byte < 4 ? (uint32_t)y[2 * p] : (uint32_t)(y[2 * p] >> 32);
    const uint32_t w1 = byte < 4 ? (uint32_t)y[2 * p + 1] : (uint32_t)(y[2 * p + 1] >> 32);
    o[p] = fx_half2(w0, w1, byte & 3);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// t 2^k for any k, apart: inlined, its multiplications would run (predicated off,
// 64 clocks each) wherever the quick forms below are chosen by a branch.
static __device__ __noinline__ double fx_scale_slow(double t, int k) { return scalbn(t, k); }

// t 2^k for any k (the exact power of two in one or more steps)
__device__ __forceinline__ double fx_scale(double t, int k) {
  if (k >= -960 && k <= 1000)
    return t * __longlong_as_double((long long)(k + 1023) << 52);
  return fx_scale_slow(t, k);
}

// t 2^sh rounded to FP64 for sh in [-1000, 900], in integer arithmetic: a
// conversion instruction would hold the FP64 pipe for 16 clocks of the SM.
__device__ __forceinline__ double fx_to_double(long long t, int sh) {
  const unsigned long long a = (unsigned long long)(t < 0 ? -t : t);
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);           // leading bit at 63
  // mantissa rounded half up; its leading bit adds one to the exponent field
  unsigned long long b = ((unsigned long long)(1085 - lz + sh) << 52) + (m >> 11) + ((m >> 10) & 1);
  b = a ? b : 0ull;
  return __longlong_as_double((long long)(b | ((unsigned long long)t & (1ull << 63))));
}

// An order's sum as an integer, |v| <= 2^22: the sum with 1.5 2^23 carries it in
// its low mantissa bits (one FP32 add; a conversion instruction runs at an
// eighth of its rate).
__device__ __forceinline__ int fx_small(float v) {
  return __float_as_int(v + 12582912.f) - 0x4B400000;
}
// half of it, rounded, |v| < 2^23
__device__ __forceinline__ int fx_small_half(float v) {
  return __float_as_int(fmaf(v, 0.5f, 12582912.f)) - 0x4B400000;
}
// a quarter of it, rounded, |v| < 2^24
__device__ __forceinline__ int fx_small_quarter(float v) {
  return __float_as_int(fmaf(v, 0.25f, 12582912.f)) - 0x4B400000;
}
// The eight order sums of one output of X -= V W' put together:
//   p01 2^88 + p23 2^72 + p45 2^56 + p67 2^40  (p = two orders, a 256 + b),
// rounded to units of 2^(74 - up).
__device__ __forceinline__ long long fx_join(int p01, int p23, int p45, int p67, int up) {
  // (up >= 18: the low pair keeps 32 - up bits below the unit)
  long long t = (p67 + (1 << (33 - up))) >> (34 - up);
  t += (long long)p45 * (1 << (up - 18));
  t += (long long)p23 * (1 << (up - 2));
  // p01 2^(up + 14): with up = 20 all in the high word
  return t + (long long)((unsigned long long)(unsigned)p01 << (up + 14));
}

// Orders o0 .. o0 + 3 of one output: sum of acc_o 256^(3 - (o - o0))
__device__ __forceinline__ long long fx_four(const uint32_t (&r)[kFxOrders][4], int o0, int k) {
  long long v = __float2int_rn(__uint_as_float(r[o0 + 3][k]));
  v += (long long)__float2int_rn(__uint_as_float(r[o0 + 2][k])) * 256;
  v += (long long)__float2int_rn(__uint_as_float(r[o0 + 1][k])) * 65536;
  v += (long long)__float2int_rn(__uint_as_float(r[o0][k])) * 16777216;
  return v;
}

// D += A B, 16 x 8 x 16, FP16 in, FP32 out
__device__ __forceinline__ void fx_mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                            uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
               "{%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Magnitudes of two FP16 values
__device__ __forceinline__ uint32_t fx_abs2(uint32_t v) { return v & 0x7fff7fffu; }

// Unit exponent of the totals over slices of RS rows: 56 up to 512 rows, one
// more for every factor of four.
__device__ __forceinline__ int fx_unit(int RS) {
  return 56 + (RS > 512) + (RS > 2048) + (RS > 8192) + (RS > 32768);
}

}  // namespace slqr
