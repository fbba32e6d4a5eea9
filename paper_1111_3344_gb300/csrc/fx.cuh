// Exact fixed-point stencils of float64 fields on the integer pipe.
//
// On GB300 a float64 warp instruction holds an SM sub-partition's float64 pipe
// for 64 cycles (1.25 TFLOP/s over 608 sub-partitions), while the integer
// pipe takes one every cycle or two.  The finite-difference stencils -- sums of
// neighbouring values with small whole coefficients, more than half of the
// float64 instructions of a right-hand side -- are therefore summed as 64-bit
// integers, and only their results become float64 again:
//  - the values of a derivative along one axis (of a mixed derivative: all
//    sixteen) are aligned to the largest exponent E among them: a value becomes
//    its 53-bit significand times 2^FX_BITS (sign applied), shifted right by E
//    minus its own exponent;
//  - the sums of these integers are exact (an axis' sums that the third
//    neighbours enter are shifted right first where those are larger, and lose a
//    unit of theirs at most); FX_BITS = 2 leaves the headroom for the largest
//    coefficient sum, 192 (|sum| < 192 2^55 < 2^63);
//  - the result is rounded to float64 once.
// The only other error is the bits shifted out of the values whose magnitude
// is below a quarter of the largest: at most 2^-54 of that largest value each, a
// quarter of the rounding that one float64 addition at its magnitude makes.
// (Aligned to the largest value along all three axes, three points away as well,
// a derivative lost the bits by which values that it does not use are larger; a
// right-hand side one point at a time took 1 to 2 % less.)  Nothing is remembered
// between stencils or points, so the result depends on the stencil's values
// alone.  (The stage in tiles, rhs_fx_tile.cuh, aligns a box of a field at once.)
//
// Stencils that hold an infinity, a NaN, or only values so small or so large
// that the result's exponent would leave the normal range take the same sums
// in float64 (fx_ok is false); a stencil of zeros is zero.
#pragma once
#include <cuda_runtime.h>

namespace bssn {

constexpr int FX_BITS = 2;

// Shifts by any count: 64 and more leave 0, or the sign.  (The C++ forms are for
// tests of this header on the host.)
__device__ __forceinline__ unsigned long long fx_shl(unsigned long long v, int n) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return (unsigned)n > 63u ? 0 : v << n;
#endif
}
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long v, int n) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return (unsigned)n > 63u ? 0 : v >> n;
#endif
}
__device__ __forceinline__ long long fx_sar(long long v, int n) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return v >> ((unsigned)n > 63u ? 63 : n);
#endif
}

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
// biased exponents 256 .. 1900: every value below 2^-64 of the largest shifts
// out whole (so a subnormal's missing leading bit never shows), and no result
// overflows or underflows, products with weights (fx_weight) included
__device__ __forceinline__ bool fx_ok(unsigned top) { return (top >> 20) - 256u <= 1900u - 256u; }

// v in units of 2^(E - 1075 - BITS), E the biased exponent of top
template <int BITS = FX_BITS>
__device__ __forceinline__ long long fx_from(double v, int E) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int sh = E - ((hi >> 20) & 0x7ff);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)lo) << BITS;
  const unsigned long long r = fx_shr(m, sh);
  const long long s = hi >> 31;
  return (long long)((r ^ (unsigned long long)s) - (unsigned long long)s);
}

// v in the same units, rounded to the nearest
template <int BITS>
__device__ __forceinline__ long long fx_near(double v, int E) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int sh = E - ((hi >> 20) & 0x7ff);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)lo) << (BITS + 1);
  const unsigned long long r = (fx_shr(m, sh) + 1) >> 1;
  const long long s = hi >> 31;
  return (long long)((r ^ (unsigned long long)s) - (unsigned long long)s);
}

// s 2^(E - 1075 - FX_BITS), rounded to the nearest float64
__device__ __forceinline__ double fx_to(long long s, int E) {
  const int neg = (int)(s >> 63);
  const unsigned long long a = (unsigned long long)((s ^ (long long)neg) - (long long)neg);
  const int n = __clzll((long long)a);
  const unsigned long long b = fx_shl(a, n);  // leading bit to bit 63 (0 stays 0)
  const unsigned long long r = (b >> 11) + ((b >> 10) & 1ull);
  // exponent of the leading bit: E + 11 - FX_BITS - n; r's own leading bit adds one
  const unsigned ex = (unsigned)(E + 10 - FX_BITS - n) << 20;
  const unsigned hi = a ? ((unsigned)(r >> 32) + ex) | ((unsigned)neg & 0x80000000u) : 0u;
  return __hiloint2double((int)hi, (int)(unsigned)r);
}

// Weights of a point for sums of products with stencil results: the significand
// times 2^9 (below 2^62) plus, in the low nine bits, the biased exponent less 831;
// 0 for a weight of zero.  False for exponents outside 895 .. 1123 (2^-128 ..
// 2^100), with which a result could leave the normal range.
__device__ __forceinline__ bool fx_weight(double v, long long& w) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)lo) << 9;
  const long long s = hi >> 31;
  const bool zero = ((hi & 0x7fffffff) | lo) == 0;
  w = zero ? 0 : (long long)((m ^ (unsigned long long)s) - (unsigned long long)s) + (e - 831);
  return zero || (unsigned)(e - 895) <= 228u;
}
// sum_q a[q] w[q], a in units of 2^(E - 1075 - FX_BITS): each a is shifted up to
// its full width, each product aligned to the largest one, and the sum rounded
// once more: off by at most 2^-56 of the largest product, as good as four
// float64 multiply-adds, which would hold the float64 pipe.  (Aligned to the
// largest weight and the largest a instead, a small weight beside a large one
// loses its last bits where only its a is large.)
template <int N>
__device__ __forceinline__ double fx_dot(const long long (&a)[N], int E, const long long (&w)[N]) {
  static_assert(N <= 4, "the sum of |products| stays below 2^63");
  long long p[N];
  int t[N], T = -2048;
#pragma unroll
  for (int q = 0; q < N; q++) {
    const int n = __clzll(a[q] ^ (a[q] >> 63));  // 1 .. 64, 64: a is 0 or -1
    p[q] = __mul64hi((long long)fx_shl((unsigned long long)a[q], n - 1), w[q] & ~511ll);
    t[q] = ((int)w[q] & 511) - n - (a[q] == 0 ? 1024 : 0);  // a zero has no exponent
    T = max(T, t[q]);
  }
  long long s = 0;
#pragma unroll
  for (int q = 0; q < N; q++) s += fx_sar(p[q], T - t[q]);
  return fx_to(s, E + T - 188);
}

// 144 h^2 d_a d_b of the field at p (strides sa, sb; a != b) times 2^up, up 0 or -1.
__device__ __forceinline__ double fx_mixed(const double* p, long long sa, long long sb, int up) {
  double v[16];  // (m, q), m, q in -2, -1, 1, 2
#pragma unroll
  for (int m = 0; m < 4; m++)
#pragma unroll
    for (int q = 0; q < 4; q++) v[4 * m + q] = __ldg(p + (m < 2 ? m - 2 : m - 1) * sa + (q < 2 ? q - 2 : q - 1) * sb);
  const unsigned top = fx_top(v);
  if (fx_ok(top)) {
    const int E = (int)(top >> 20);
    long long l[4];
#pragma unroll
    for (int m = 0; m < 4; m++)
      l[m] = 8 * (fx_from(v[4 * m + 2], E) - fx_from(v[4 * m + 1], E)) - (fx_from(v[4 * m + 3], E) - fx_from(v[4 * m], E));
    // half of 8 (l1 - l-1) - (l2 - l-2): the whole may pass 2^63
    return fx_to(4 * (l[2] - l[1]) - ((l[3] - l[0]) >> 1), E + 1 + up);
  }
  if (fx_zero(v)) return 0.0;
  double l[4];
#pragma unroll
  for (int m = 0; m < 4; m++) l[m] = fma(8.0, v[4 * m + 2] - v[4 * m + 1], -(v[4 * m + 3] - v[4 * m]));
  return (up ? 0.5 : 1.0) * fma(8.0, l[2] - l[1], -(l[3] - l[0]));
}

// The three mixed second derivatives (xy, xz, yz), one copy of the code.
__device__ __forceinline__ void fx_mixed3(const double* p, long long sy, long long sz, int up, double dd[3]) {
  double t[3];
#pragma unroll 1
  for (int m = 0; m < 3; m++) t[m] = fx_mixed(p, m < 2 ? 1 : sy, m == 0 ? sy : sz, up);
  dd[0] = t[0];
  dd[1] = t[1];
  dd[2] = t[2];
}

// 12 h d f along stride s times 2^up.
__device__ __forceinline__ double fx_d1(const double* p, long long s, int up) {
  const double v[4] = {__ldg(p - 2 * s), __ldg(p - s), __ldg(p + s), __ldg(p + 2 * s)};
  const unsigned top = fx_top(v);
  if (fx_ok(top)) {
    const int E = (int)(top >> 20);
    return fx_to(8 * (fx_from(v[2], E) - fx_from(v[1], E)) - (fx_from(v[3], E) - fx_from(v[0], E)), E + up);
  }
  if (fx_zero(v)) return 0.0;
  return (up ? 0.5 : 1.0) * fma(8.0, v[2] - v[1], -(v[3] - v[0]));
}

// 12 h d_d f and, SECOND, 144 h^2 d_d d_d f, d = x, y, z, times 2^up.
template <bool SECOND>
__device__ __forceinline__ void fx_axes(const double* p, long long sy, long long sz, int up, double d1[3],
                                        double d2[3]) {
  double v[13];
  v[0] = SECOND ? __ldg(p) : 0.0;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const long long s = d == 0 ? 1 : (d == 1 ? sy : sz);
    v[1 + 4 * d] = __ldg(p - 2 * s);
    v[2 + 4 * d] = __ldg(p - s);
    v[3 + 4 * d] = __ldg(p + s);
    v[4 + 4 * d] = __ldg(p + 2 * s);
  }
  const unsigned top = fx_top(v);
  if (fx_ok(top)) {
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const double ax[5] = {v[0], v[1 + 4 * d], v[2 + 4 * d], v[3 + 4 * d], v[4 + 4 * d]};
      const int E = max((int)(fx_top(ax) >> 20), 256);
      const long long a = fx_from(ax[1], E), b = fx_from(ax[2], E), c = fx_from(ax[3], E), e = fx_from(ax[4], E);
      d1[d] = fx_to(8 * (c - b) - (e - a), E + up);
      if (SECOND) d2[d] = fx_to(3 * (16 * (c + b) - (e + a) - 30 * fx_from(ax[0], E)), E + 2 + up);
    }
    return;
  }
  const double sc = fx_zero(v) ? 0.0 : (up ? 0.5 : 1.0);
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double a = v[1 + 4 * d], b = v[2 + 4 * d], c = v[3 + 4 * d], e = v[4 + 4 * d];
    d1[d] = sc * fma(8.0, c - b, -(e - a));
    if (SECOND) d2[d] = 12.0 * sc * fma(-30.0, v[0], fma(16.0, c + b, -(e + a)));
  }
}

}  // namespace bssn
