// Float64 BSSN right-hand side of a tile of points: rhs_fx.cuh's arithmetic with
// each field's values brought to shared memory and made integers once per
// block.
//
// One point at a time (rhs_fx.cuh), every stencil aligns its own 19 to 67
// values: some 25,000 integer instructions a point, as long as the float64
// pipe is busy (1114 instructions of 64 cycles for a warp).  Here a block loops
// over the fields:
//  - A tensor load brings the field's box (the tile and three points on every
//    side) into one of two buffers while the other's field is worked on.
//  - Each thread finds the exponents of its share of the points that stencils
//    read, the block their maximum, and each thread turns its share into
//    integers in place, rounded to FX_TILE_BITS bits below the last of the box's
//    largest value.  (Sums: |value| < 2^57; the largest sum of coefficients is
//    64 -- the pure second derivatives without their factor 3, the mixed ones an
//    eighth, half the upwind sum of an axis, a quarter of the axes' KO sum.)
//  - A thread then reads its taps (67 for a twice-differenced field) with fixed
//    offsets and no conversion.  Advection and dissipation are one sum of four
//    products with weights of the point, kept as integers too (fx_weight,
//    fx_dot); the contraction gt^kl d_k d_l is float64: 869 float64
//    instructions a point.
//  - Where the box's largest value is much more than what a thread's star holds,
//    the box's integers have fewer bits than the thread's own values.  That thread
//    takes the field's stencils one point at a time from the register (FX_NEAR,
//    fx_stencils_own), so that every point is as exact as rhs_fx.cuh makes it: a
//    field that falls off steeply inside a tile, a small value beside a large one.
//    On smooth data some percent of the warps or fewer do.  In the first tens of
//    steps of a puncture, whose shift, B^i and Gt^i start from zero and fall off
//    steeply, one to two of a warp's 24 fields at 64^3, 0.16 at 128^3: a step of
//    64^3 takes 2.75 ms then, 2.58 after 150 steps, 2.46 without (the rule's own
//    code and the loop's together exceed the instruction cache).
//  - The algebra runs inside the loop as soon as its fields are there, so that
//    few results wait at a time (33 local slots).
// The stencil code exists once: the instruction cache holds 128 KB, and a
// float64 instruction takes five instruction slots.  Neither part alone fills
// the time (128^3, cycles of an SM sub-partition for a warp's points, with sums
// that took 57 float64 instructions fewer: algebra 58-61 thousand, the loop
// without it 56, together 68; per-point form 88; now 71).
#pragma once
#include "fx.cuh"
#include "fx_algebra.cuh"
#include "rhs_fx.cuh"
#include "tma.cuh"

namespace bssn {

constexpr int FX_TILE_BITS = 4;

// A thread whose star -- the point and those one and two away along each axis: the
// values of its pure derivatives -- reaches no 2^(FX_NEAR - 1) units at the point
// or two away (a sixteenth of the box's largest exponent) takes its own alignment:
// an integer's rounding, half a unit, is then at most 2^-53 of the star's largest
// value, as float64 rounds that value itself.  (Shift and B^i as Gaussians of
// width 1 at h = 0.25, relative error of the shift's right-hand side at each
// point, 90th and 99th percentile: 4e-16 and 2e-15; without this rule 2e-11 and
// 4e-9; float64 stencils 1e-15 and 3e-15.)  A step at 128^3 takes 15.72 -> 15.78 ms
// for it, 75 x 53 x 61 2.58 -> 2.61, 24^3 0.208 -> 0.210: the threads that take
// their own alignment hold up their block.  One bit more 15.82, 2.69 and 0.222,
// for 3e-16 and 9e-16; three threads sharing a point's three axes 16.1, 2.70 and
// 0.218.
constexpr int FX_NEAR = 53;
// a bound on |v|'s high word, whose leading bit is that of |v| (or of |v| - 1)
__device__ __forceinline__ int fx_mag(long long v) {
  const int hi = (int)(v >> 32);
  return hi ^ (hi >> 31);
}

// Tile of TX x TY x TZ interior points, one per thread, and its box: the tile
// plus three points on every side.  TX and the box's x extent are even (tensor
// loads move multiples of 16 bytes).
template <int TX_, int TY_, int TZ_>
struct FxTile {
  static constexpr int TX = TX_, TY = TY_, TZ = TZ_, THREADS = TX * TY * TZ, WARPS = THREADS / 32;
  static constexpr int BX = TX + 2 * GH, BY = TY + 2 * GH, BZ = TZ + 2 * GH, BOX = BX * BY * BZ;
  static constexpr int SY = BX, SZ = BX * BY;                // strides inside the box
  // The box points that stencils read: the tile itself, three layers beyond each
  // face (star), two by two beyond each edge along which two axes mix.
  static constexpr int NX = 6 * TY * TZ, NY = 6 * TX * TZ, NZ = 6 * TX * TY, STAR = NX + NY + NZ;
  static constexpr int MXY = 16 * TZ, MXZ = 16 * TY, MYZ = 16 * TX, MIX = MXY + MXZ + MYZ;
  static constexpr int PS = (STAR + THREADS - 1) / THREADS, PM = (MIX + THREADS - 1) / THREADS;
  static constexpr int PER = 1 + PS + PM;  // points a thread converts: its own, star, mixed
  // box coordinates of point n of the star (n < STAR) or of the mixed edges
  static __device__ __forceinline__ void star(int n, int& x, int& y, int& z) {
    if (n < NX) {
      const int l = n % 6;
      x = l < 3 ? l : TX + l;
      y = GH + n / 6 % TY;
      z = GH + n / (6 * TY);
    } else if (n < NX + NY) {
      n -= NX;
      x = GH + n % TX;
      const int l = n / TX % 6;
      y = l < 3 ? l : TY + l;
      z = GH + n / (6 * TX);
    } else {
      n -= NX + NY;
      x = GH + n % TX;
      y = GH + n / TX % TY;
      const int l = n / (TX * TY);
      z = l < 3 ? l : TZ + l;
    }
  }
  static __device__ __forceinline__ int edge(int l, int t) { return l < 2 ? 1 + l : t + 1 + l; }  // 1, 2, t+3, t+4
  static __device__ __forceinline__ void mixed(int n, int& x, int& y, int& z) {
    if (n < MXY) {
      x = edge(n & 3, TX);
      y = edge(n >> 2 & 3, TY);
      z = GH + (n >> 4);
    } else if (n < MXY + MXZ) {
      n -= MXY;
      x = edge(n & 3, TX);
      z = edge(n >> 2 & 3, TZ);
      y = GH + (n >> 4);
    } else {
      n -= MXY + MXZ;
      x = GH + n % TX;
      y = edge(n / TX & 3, TY);
      z = edge(n / (4 * TX), TZ);
    }
  }
};
// Shared memory of a block: two boxes (one field's values, then integers; the
// next field's on their way) and their barriers, each thread's advection (3)
// and contraction (6) weights, each warp's largest high word.
template <typename Sh>
struct FxShared {
  alignas(128) long long box[2][(Sh::BOX + 15) / 16 * 16];
  unsigned long long bar[2];
  double wt[10][Sh::THREADS];
  unsigned top[Sh::WARPS];
};

// tensor load of field f's box from stored (x, y, z) into a buffer that ordinary
// accesses are done with (one thread, after a barrier of its users)
template <typename Sh>
__device__ __forceinline__ void fx_issue(const void* map, void* box, unsigned bar, int x, int y, int z, int f) {
  fence_async_proxy();
  mbar_expect(bar, Sh::BOX * 8);
  tensor_load_4d(box, map, x, y, z, f, bar);
}

// Box points of thread tid (of Sh::THREADS) as offsets from the box's start, for
// its point (i, j, k) (stored indices, inside the grid) in the tile at (ii0, jj0,
// kk0): into sc[e * Sh::THREADS], e < Sh::PER (a loop: one copy of this code).  In
// a tile that the grid fills partly, points that no point inside the grid reads
// (they may hold anything: the padding of a row, a corner of the ghost zone)
// give way to the thread's own point, which several threads may then convert
// alike.
template <typename Sh>
__device__ __forceinline__ int fx_center(int ii0, int jj0, int kk0, int i, int j, int k) {
  return ((k - kk0) * Sh::BY + j - jj0) * Sh::BX + i - ii0;
}
template <typename Sh>
__device__ __forceinline__ void fx_points(const Grid& g, int tid, int ii0, int jj0, int kk0, int cen, int* sc) {
  const int lx = min(Sh::TX, g.n0 - ii0), ly = min(Sh::TY, g.n1 - jj0), lz = min(Sh::TZ, g.n2 - kk0);
  auto beyond = [](int x, int l) { return max(max(GH - x, x - (GH + l - 1)), 0); };
#pragma unroll 1
  for (int e = 0; e < Sh::PER; e++) {
    int x, y, z;
    if (e == 0) {
      x = GH + tid % Sh::TX;
      y = GH + tid / Sh::TX % Sh::TY;
      z = GH + tid / (Sh::TX * Sh::TY);
    } else if (e <= Sh::PS) {
      Sh::star(min(tid + (e - 1) * Sh::THREADS, Sh::STAR - 1), x, y, z);
    } else {
      Sh::mixed(min(tid + (e - 1 - Sh::PS) * Sh::THREADS, Sh::MIX - 1), x, y, z);
    }
    const int dx = beyond(x, lx), dy = beyond(y, ly), dz = beyond(z, lz), axes = (dx > 0) + (dy > 0) + (dz > 0);
    const bool read = axes < 3 && max(dx, max(dy, dz)) <= (axes == 2 ? 2 : 3);
    sc[e * Sh::THREADS] = read ? z * Sh::SZ + y * Sh::SY + x : cen;
  }
}

// Weights of a point into wt (stride Sh::THREADS): |beta^d| / (24h) 0-2, gt^kl
// doubled off the diagonal 3-8; neg: signs of beta as masks.
template <typename Sh>
__device__ __forceinline__ bool fx_tile_weights(const Grid& g, const double* __restrict__ c0, const FxMetric& M,
                                                double* wt, int neg[3]) {
  bool ok = true;
  long long x;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double b = __ldg(c0 + (F_BETA + d) * g.fstride);
    ok = fx_weight(fabs(b) * (0.5 * g.i12h), x) && ok;
    wt[d * Sh::THREADS] = __longlong_as_double(x);
    neg[d] = __double2hiint(b) >> 31;
  }
  ok = fx_weight(2.0 * g.kos, x) && ok;
  wt[9 * Sh::THREADS] = __longlong_as_double(x);
#pragma unroll
  for (int m = 0; m < 6; m++) wt[(3 + m) * Sh::THREADS] = M.g2u(m);
  return ok;
}

// Fields in the order of the loop, q: gt_ij, Gt^i | phi|W, alpha | beta^i, K,
// At_ij, B^i; the derivatives taken (2: all, 1: first, 0: none) and whether they
// are halved (the metric's and Gt's).
__device__ __forceinline__ int fx_field(int q) {
  if (q < 9) return q < 6 ? F_GT + q : q + (F_GAM - 6);
  if (q < 14) return q == 9 ? (int)F_CHI : q + (F_ALP - 10);
  return q == 14 ? (int)F_TRK : (q < 21 ? q + (F_AT - 15) : q + (F_B - 21));
}
__device__ __forceinline__ int fx_order(int q) { return (q < 6 || (q > 8 && q < 14)) ? 2 : (q < 15 ? 1 : 0); }
__device__ __forceinline__ int fx_up(int q) { return q < 9 ? -1 : 0; }
// Second derivatives of field q into slots: their contraction with gt^kl into
// s0 + 3, those kept after it (all six of phi|W and alpha, q = 9 and 10; the
// three d_k d_a of beta^a, q = 11 + a).
template <typename Sh, typename Slots>
__device__ __forceinline__ void fx_second(const double dd[6], int q, const double* wt, Slots S, int s0) {
  if (q != 9) {  // phi|W's is not used
    double t = 0.0;
#pragma unroll
    for (int m = 0; m < 6; m++) t = fma(wt[(3 + m) * Sh::THREADS], dd[m], t);
    S(s0 + 3) = t;
  }
  if (q > 10) {
    S(s0 + 4) = q == 11 ? dd[0] : (q == 12 ? dd[1] : dd[2]);
    S(s0 + 5) = q == 11 ? dd[1] : (q == 12 ? dd[3] : dd[4]);
    S(s0 + 6) = q == 11 ? dd[2] : (q == 12 ? dd[4] : dd[5]);
  } else if (q > 8) {
#pragma unroll
    for (int m = 0; m < 6; m++) S(s0 + 4 + m) = dd[m];
  }
}

// Field q's stencils at c in a box of integers (units of 2^(E - 1075 - FX_BITS)):
// returns advection and dissipation; its first derivatives into slots s0 ..
// s0 + 2, its contracted second derivative into s0 + 3, those kept after it.
// wt: the thread's weights, stride Sh::THREADS; neg: signs of beta as masks.
// near: the point's value or one two away has FX_NEAR bits or more.
template <typename Sh, typename Slots>
__device__ __forceinline__ double fx_stencils(const long long* c, int q, int order, int up, int E,
                                              const double* wt, const int neg[3], Slots S, int s0, bool& near) {
  constexpr int SY = Sh::SY, SZ = Sh::SZ;
  const long long f0 = c[0];
  long long s2[6], a[4];
  a[3] = 0;
  int big = fx_mag(f0);
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const int s = d == 0 ? 1 : (d == 1 ? SY : SZ);
    long long sp[3], df[3];
#pragma unroll
    for (int m = 0; m < 3; m++) {
      const long long lo = c[-(m + 1) * s], hi = c[(m + 1) * s];
      if (m == 1) big |= fx_mag(lo) | fx_mag(hi);
      sp[m] = hi + lo;
      df[m] = hi - lo;
    }
    if (order >= 1) S(s0 + d) = fx_to(8 * df[0] - df[1], E + up);
    s2[d == 0 ? 0 : (d == 1 ? 3 : 5)] = 16 * sp[0] - sp[1] - 30 * f0;  // 12 h^2 d_d d_d
    const long long kh = (15 * sp[0] - 6 * sp[1] + sp[2] - 20 * f0) >> 1, oh = (21 * df[0] - 6 * df[1] + df[2]) >> 1;
    const long long sg = neg[d];
    a[d] = kh + ((oh ^ sg) - sg);
    a[3] += kh >> 1;
  }
  near = big >> (FX_NEAR - 1 - 32) != 0;
  long long w[4];
#pragma unroll
  for (int m = 0; m < 4; m++) w[m] = __double_as_longlong(wt[(m < 3 ? m : 9) * Sh::THREADS]);
  const double r = fx_dot(a, E + 1, w);
  if (order == 2) {
#pragma unroll
    for (int m = 0; m < 3; m++) {  // xy, xz, yz
      const int sa = m < 2 ? 1 : SY, sb = m == 0 ? SY : SZ;
      long long l[4];
#pragma unroll
      for (int n = 0; n < 4; n++) {
        const long long* p = c + (n < 2 ? n - 2 : n - 1) * sa;
        l[n] = 8 * (p[sb] - p[-sb]) - (p[2 * sb] - p[-2 * sb]);
      }
      // an eighth of 8 (l1 - l-1) - (l2 - l-2): 18 h^2 d_a d_b
      s2[m == 0 ? 1 : 2 * m] = (l[2] - l[1]) - ((l[3] - l[0]) >> 3);
    }
    double dd[6];
#pragma unroll
    for (int m = 0; m < 6; m++) {
      const bool pure = m == 0 || m == 3 || m == 5;  // 12 v = 16 (v - v/4)
      dd[m] = fx_to(pure ? s2[m] - (s2[m] >> 2) : s2[m], E + (pure ? 4 : 3) + up);
    }
    fx_second<Sh>(dd, q, wt, S, s0);
  }
  return r;
}

// The same from the register, each stencil aligned to its own largest value or,
// outside the integers' range, summed in float64 (rhs_fx.cuh), the products in
// float64: also for boxes and weights outside the range.  A call of its own, so
// that its code stays out of the loop's.
template <typename Sh, typename Slots>
__device__ __noinline__ double fx_stencils_own(const double* __restrict__ c0, long long fs, long long sy, long long sz,
                                               double i12h, double kap, int q, int order, int up, const double* wt,
                                               Slots S, int s0) {
  const double* p = c0 + fx_field(q) * fs;
  const FxAdv w = fx_adv(c0, fs, i12h, kap);
  double d1[3], dd[3];
  const double r = fx_axes(p, sy, sz, w, order, up, d1, dd);
  if (order >= 1) {
#pragma unroll
    for (int d = 0; d < 3; d++) S(s0 + d) = d1[d];
  }
  if (order == 2) {
    double dm[3];
    fx_mixed3(p, sy, sz, up, dm);
    const double d6[6] = {dd[0], dm[0], dm[1], dd[1], dm[2], dd[2]};
    fx_second<Sh>(d6, q, wt, S, s0);
  }
  return r;
}

// Test hook (StageArgsT::stall_polls): the round whose copy group grp leaves out, -1
// for none.
template <typename A>
__device__ __forceinline__ int fx_stall_round(const A& a, int grp) {
  if (a.stall_polls <= 0) return -1;
  return a.stall_at < 0 ? 0 : (a.stall_at / 32 == grp ? a.stall_at % 32 : -1);
}

// The right-hand side of all 24 fields at this thread's point (i, j, k) (stored
// indices, inside the grid) of the tile whose first interior point is (ii0,
// jj0, kk0), from the float64 register st, which map describes (its box that
// of Sh); every thread of the block calls it.  False: a wait ran out (at once in
// round stall, after polls, its copy left out).
template <typename Sh>
__device__ __forceinline__ bool rhs_fx_tile(const void* map, const Grid& g, const double* __restrict__ st,
                                            FxShared<Sh>& sm, int tid, int ii0, int jj0, int kk0, int i, int j, int k,
                                            double out[NF], int stall, int polls) {
  const long long fs = g.fstride, id = lin(g, i, j, k);
  const double* c0 = st + id;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  double slots[33];  // results of the stencils, in local memory
  auto S = [&](int n) -> double& { return slots[n]; };

  if (tid == 0) {
    for (int b = 0; b < 2; b++) mbar_init(smem_addr(&sm.bar[b]));
    if (stall != 0) fx_issue<Sh>(map, sm.box[0], smem_addr(&sm.bar[0]), ii0, jj0, kk0, fx_field(0));
  }
  const int cen = fx_center<Sh>(ii0, jj0, kk0, i, j, k);
  // (through the second buffer, which is still free)
  int* sc = reinterpret_cast<int*>(sm.box[1]) + tid;
  static_assert(Sh::PER * Sh::THREADS * sizeof(int) <= sizeof(sm.box[1]), "");
  fx_points<Sh>(g, tid, ii0, jj0, kk0, cen, sc);
  int neg[3];
  FxMetric M;
  fx_metric(g, c0, M);
  const double* wt = &sm.wt[0][tid];
  const bool wok = fx_tile_weights<Sh>(g, c0, M, &sm.wt[0][tid], neg);
  __syncthreads();  // the barriers are initialised
  int at[Sh::PER];
#pragma unroll
  for (int e = 0; e < Sh::PER; e++) at[e] = sc[e * Sh::THREADS];

  double X[6], G2[3][6], V2[3], vj[3], lap = 0.0;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    V2[a] = vj[a] = 0.0;
#pragma unroll
    for (int m = 0; m < 6; m++) G2[a][m] = 0.0;
  }
#pragma unroll
  for (int m = 0; m < 6; m++) X[m] = 0.0;

#pragma unroll 1
  for (int q = 0; q < NF; q++) {
    int order = fx_order(q), up = fx_up(q);
    int s0 = q < 6 ? 4 * q : (q < 9 ? 3 * q + 6 : (q < 11 ? 10 * (q - 9) : (q < 14 ? 7 * (q - 11) : 21)));
    asm volatile("" : "+r"(order), "+r"(up), "+r"(s0));  // one copy of the code below, not one per value
    long long* box = sm.box[q & 1];
    const long long* c = box + cen;
    const bool there = mbar_wait(smem_addr(&sm.bar[q & 1]), (q >> 1) & 1, q == stall ? polls : WAIT_LIMIT);
    double x[Sh::PER];
#pragma unroll
    for (int e = 0; e < Sh::PER; e++) x[e] = __longlong_as_double(box[at[e]]);
    const unsigned wtop = __reduce_max_sync(0xffffffffu, fx_top(x));
    if ((tid & 31) == 0) sm.top[tid >> 5] = wtop;
    // the maxima are there, and the previous field's box is free
    if (!__syncthreads_and(there)) {
      // the one copy in flight lands before the block exits
      if (q != stall) mbar_wait(smem_addr(&sm.bar[q & 1]), (q >> 1) & 1, WAIT_LIMIT);
      return false;
    }
    if (tid == 0 && q + 1 < NF && q + 1 != stall)
      fx_issue<Sh>(map, sm.box[(q + 1) & 1], smem_addr(&sm.bar[(q + 1) & 1]), ii0, jj0, kk0, fx_field(q + 1));
    unsigned top = sm.top[0];
#pragma unroll
    for (int n = 1; n < Sh::WARPS; n++) top = max(top, sm.top[n]);
    // a box of zeros takes any exponent; top does not see low words of subnormals
    bool ok = fx_ok(top);
    if (top == 0) {
      unsigned lo = 0;
#pragma unroll
      for (int e = 0; e < Sh::PER; e++) lo |= (unsigned)__double2loint(x[e]);
      ok = !__syncthreads_or(lo != 0);
    }
    const int E = max((int)(top >> 20), 256) + FX_BITS - FX_TILE_BITS;  // the integers' unit is 2^(E - 1075 - FX_BITS)
    // (points that several threads share: the same value)
    if (ok) {
#pragma unroll
      for (int e = 0; e < Sh::PER; e++) box[at[e]] = fx_near<FX_TILE_BITS>(x[e], E + FX_TILE_BITS - FX_BITS);
    }
    __syncthreads();
    const int f = fx_field(q);
    double r = 0.0;
    bool near = false;
    if (ok) r = fx_stencils<Sh>(c, q, order, up, E, wt, neg, S, s0, near);
    if (!(near && wok) && !(ok && top == 0))
      r = fx_stencils_own<Sh>(c0, fs, g.pitch, g.plane, g.i12h, g.kos, q, order, up, wt, S, s0);
    out[f] = f < nf ? r : 0.0;

    if (q == 8) {
      fx_ricci(g, M, [&](int d, int m) { return S(4 * m + d); }, [&](int m) { return S(4 * m + 3); },
               [&](int a, int d) { return S(24 + 3 * a + d); }, X, G2, V2);
    } else if (q == 10) {
      // slots: d phi|W 0-2, d d phi|W 4-9; d alpha 10-12, gt^kl d_k d_l alpha 13, d d alpha 14-19
      double dchi[3], dalp[3];
#pragma unroll
      for (int a = 0; a < 3; a++) {
        dchi[a] = S(a);
        dalp[a] = S(10 + a);
      }
      fx_lapse(g, M, __ldg(c0 + F_ALP * fs), dchi, dalp, S(13), [&](int m) { return S(4 + m); },
               [&](int m) { return S(14 + m); }, G2, X, lap, vj);
    }
  }

  // slots: 12h d_d beta^a 7 a + d, 144 h^2 gt^kl d_k d_l beta^a 7 a + 3,
  // 144 h^2 d_k d_a beta^a (no sum) 7 a + 4 + k; 12h d_d K 21 + d
  fx_assemble(g, c0, id, i, j, k, M, [&](int a, int d) { return S(7 * a + d); }, [&](int a) { return S(7 * a + 3); },
              [&](int a, int m) { return S(7 * a + 4 + m); }, [&](int d) { return S(21 + d); }, G2, V2, vj, X, lap,
              out);
  return true;
}

}  // namespace bssn
