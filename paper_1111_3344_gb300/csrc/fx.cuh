// Exact fixed-point stencils of float64 fields on the integer pipe.
//
// On GB300 a float64 warp instruction holds an SM sub-partition's float64 pipe
// for 64 cycles (1.25 TFLOP/s over 608 sub-partitions), while the integer
// pipe takes one every cycle or two.  The finite-difference stencils -- sums of
// neighbouring values with small whole coefficients, more than half of the
// float64 instructions of a right-hand side -- are therefore summed as 64-bit
// integers, and only their results become float64 again:
//  - the values of one stencil are aligned to the largest exponent E among
//    them: a value becomes its 53-bit significand times 2^FX_BITS (sign
//    applied), shifted right by E minus its own exponent;
//  - the sums of these integers are exact; FX_BITS = 2 leaves the headroom for
//    the largest coefficient sum, 192 (|sum| < 192 2^55 < 2^63);
//  - the result is rounded to float64 once.
// The only other error is the bits shifted out of the values whose magnitude
// is below a quarter of the stencil's largest: at most 2^-54 of that largest
// value each, a quarter of the rounding that one float64 addition at its
// magnitude makes.  Nothing is remembered between stencils or points, so the
// result depends on the stencil's values alone.
//
// Stencils that hold an infinity, a NaN, or only values so small or so large
// that the result's exponent would leave the normal range take the same sums
// in float64 (fx_ok is false); a stencil of zeros is zero.
#pragma once
#include <cuda_runtime.h>

namespace bssn {

constexpr int FX_BITS = 2;

// largest high word (sign cleared) of the values: its top 11 bits are the
// largest biased exponent
template <int N>
__device__ __forceinline__ unsigned fx_top(const double (&v)[N]) {
  unsigned m = 0;
#pragma unroll
  for (int q = 0; q < N; q++) m = max(m, (unsigned)__double2hiint(v[q]) & 0x7fffffffu);
  return m;
}
// whether every value is zero (only asked where fx_ok is false)
template <int N>
__device__ __forceinline__ bool fx_zero(const double (&v)[N]) {
  unsigned m = 0;
#pragma unroll
  for (int q = 0; q < N; q++) m |= ((unsigned)__double2hiint(v[q]) & 0x7fffffffu) | (unsigned)__double2loint(v[q]);
  return m == 0;
}
// biased exponents 128 .. 2026: every value below 2^-64 of the largest shifts
// out whole (so a subnormal's missing leading bit never shows), and no result
// overflows or underflows
__device__ __forceinline__ bool fx_ok(unsigned top) { return (top >> 20) - 128u <= 2026u - 128u; }

// v in units of 2^(E - 1075 - FX_BITS), E the biased exponent of top
__device__ __forceinline__ long long fx_from(double v, int E) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int sh = E - ((hi >> 20) & 0x7ff);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)lo) << FX_BITS;
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(sh));  // shifts of 64 and more give 0
  const long long s = hi >> 31;
  return (long long)((r ^ (unsigned long long)s) - (unsigned long long)s);
}

// s 2^(E - 1075 - FX_BITS + up), rounded to the nearest float64
__device__ __forceinline__ double fx_to(long long s, int E) {
  const int neg = (int)(s >> 63);
  const unsigned long long a = (unsigned long long)((s ^ (long long)neg) - (long long)neg);
  const int n = __clzll((long long)a);
  unsigned long long b;
  asm("shl.b64 %0, %1, %2;" : "=l"(b) : "l"(a), "r"(n));  // leading bit to bit 63 (0 stays 0)
  const unsigned long long r = (b >> 11) + ((b >> 10) & 1ull);
  // exponent of the leading bit: E + 11 - FX_BITS - n; r's own leading bit adds one
  const unsigned ex = (unsigned)(E + 10 - FX_BITS - n) << 20;
  const unsigned hi = a ? ((unsigned)(r >> 32) + ex) | ((unsigned)neg & 0x80000000u) : 0u;
  return __hiloint2double((int)hi, (int)(unsigned)r);
}

}  // namespace bssn
