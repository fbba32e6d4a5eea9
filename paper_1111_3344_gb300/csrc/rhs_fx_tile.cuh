// Float64 BSSN right-hand side of a tile of points: rhs_fx.cuh's arithmetic with
// each field's values brought to shared memory and made integers once per
// block.
//
// One point at a time (rhs_fx.cuh), every stencil aligns its own 19 to 67
// values: some 25,000 integer instructions a point, as long as the float64
// pipe is busy (1016 instructions of 64 cycles for a warp).  Here a block loops
// over the fields:
//  - A tensor load brings the field's box (the tile and three points on every
//    side) into one of two buffers while the other's field is worked on.
//  - Each thread finds the exponents of its share of the points that stencils
//    read, the block their maximum, and each thread turns its share into
//    integers in place, rounded to FX_TILE_BITS bits below the last of the box's
//    largest value: off by at most 2^-57 of it.  (Sums: |value| <= 2^56, the
//    largest coefficient sum 120 -- the pure second derivatives without their
//    factor 3, the mixed ones quartered, half the three axes' KO sum.)
//  - A thread then reads its taps (67 for a twice-differenced field) with fixed
//    offsets and no conversion.  Advection, dissipation and the contraction
//    gt^kl d_k d_l are sums of four and six products with weights of the point,
//    kept as 64-bit integers too (FxWeights: off by at most 2^-60 of the largest
//    product): 860 float64 instructions a point.
//  - The algebra runs inside the loop as soon as its fields are there, so that
//    few results wait at a time (33 local slots).
// The stencil code exists once: the instruction cache holds 128 KB, and a
// float64 instruction takes five instruction slots.  Neither part alone fills
// the time (128^3, cycles of an SM sub-partition for a warp's points: algebra
// 58-61 thousand, the loop without it 56, together 68; per-point form 88).
#pragma once
#include "fx.cuh"
#include "fx_algebra.cuh"
#include "tma.cuh"

namespace bssn {

constexpr int FX_TILE_BITS = 3;

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
// next field's on their way) and their barriers, each thread's advection (4)
// and contraction (6) weights, each warp's largest high word.
template <typename Sh>
struct FxShared {
  alignas(128) long long box[2][(Sh::BOX + 15) / 16 * 16];
  unsigned long long bar[2];
  long long wt[10][Sh::THREADS];
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

// advection and dissipation weights of the point c0: |beta^d| / (24h), eps /
// (64h), and the signs of beta as masks
__device__ __forceinline__ void fx_adv_weights(const Grid& g, const double* __restrict__ c0, double wd[4], int neg[3]) {
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double b = __ldg(c0 + (F_BETA + d) * g.fstride);
    wd[d] = fabs(b) * (0.5 * g.i12h);
    neg[d] = __double2hiint(b) >> 31;
  }
  wd[3] = g.kos;
}

// The float64 forms of a field's stencils at c, for boxes outside the integer
// range (fx_ok): a call of its own, cold code kept out of the loop's
// instructions.  up: the metric's and Gt's derivatives are halved.
static __device__ __noinline__ double fx_field_f64(const double* c, int sy, int sz, const double wd[4], const int neg[3],
                                                   int up, double d1[3], double dd[6]) {
  const double sc = up ? 0.5 : 1.0;
  double r = 0.0;
#pragma unroll 1
  for (int d = 0; d < 3; d++) {
    const int s = d == 0 ? 1 : (d == 1 ? sy : sz), m = d == 0 ? 0 : (d == 1 ? 3 : 5);
    const double a1 = c[-s], b1 = c[s], a2 = c[-2 * s], b2 = c[2 * s], a3 = c[-3 * s], b3 = c[3 * s];
    d1[d] = sc * fma(8.0, b1 - a1, -(b2 - a2));
    dd[m] = 12.0 * sc * fma(-30.0, c[0], fma(16.0, b1 + a1, -(b2 + a2)));
    const double k = fma(15.0, b1 + a1, fma(-6.0, b2 + a2, b3 + a3)) - 20.0 * c[0];
    const double o = fma(21.0, b1 - a1, fma(-6.0, b2 - a2, b3 - a3));
    r = fma(wd[d], neg[d] ? k - o : k + o, r);
    r = fma(wd[3], k, r);
  }
#pragma unroll 1
  for (int m = 0; m < 3; m++) {  // xy, xz, yz
    const int sa = m < 2 ? 1 : sy, sb = m == 0 ? sy : sz;
    double l[4];
#pragma unroll 1
    for (int q = 0; q < 4; q++) {
      const double* p = c + (q < 2 ? q - 2 : q - 1) * sa;
      l[q] = fma(8.0, p[sb] - p[-sb], -(p[2 * sb] - p[-2 * sb]));
    }
    dd[m == 0 ? 1 : 2 * m] = sc * fma(8.0, l[2] - l[1], -(l[3] - l[0]));
  }
  return r;
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

// Fixed-point weights of a point: advection and dissipation (|beta^d| / (24h) and
// eps / (32h), for half the axes' KO sum), and gt^kl, doubled off the diagonal,
// times the 3 that the pure sums leave out on it.
__device__ __forceinline__ FxWeights<4> fx_tile_adv(const Grid& g, const double* __restrict__ c0, int neg[3]) {
  double wd[4];
  fx_adv_weights(g, c0, wd, neg);
  wd[3] *= 2.0;
  return fx_weights(wd);
}
__device__ __forceinline__ FxWeights<6> fx_tile_gu(const FxMetric& M) {
  double v[6];
#pragma unroll
  for (int m = 0; m < 6; m++) v[m] = ((m == 0 || m == 3 || m == 5) ? 3.0 : 2.0) * M.gu[m];
  return fx_weights(v);
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
// component of the m-th second derivative kept of field q: all six of phi|W and
// alpha (q = 9, 10), the three d_k d_a of beta^a (q = 11 + a)
__device__ __forceinline__ int fx_kept(int q, int m) {
  const int a = q - 11;
  return q < 11 ? m : (a == 0 ? m : (m == 0 ? a : (a == 1 ? m + 2 : m + 3)));
}

// Field q's stencils at c in a box of integers (units of 2^(E - 1075 - FX_BITS)):
// returns advection and dissipation; its first derivatives into slots s0 ..
// s0 + 2, its contracted second derivative into s0 + 3, those kept after it.
// wt: the thread's weights, stride Sh::THREADS; neg: signs of beta as masks.
template <typename Sh, typename Slots>
__device__ __forceinline__ double fx_stencils(const long long* c, int q, int order, int up, int E,
                                              const long long* wt_, int wE, int gwE, const int neg[3], Slots S, int s0) {
  constexpr int SY = Sh::SY, SZ = Sh::SZ;
  long long a[4], s2[6];
  a[3] = 0;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const int s = d == 0 ? 1 : (d == 1 ? SY : SZ);
    long long sp[3], df[3];
#pragma unroll
    for (int m = 0; m < 3; m++) {
      const long long lo = c[-(m + 1) * s], hi = c[(m + 1) * s];
      sp[m] = hi + lo;
      df[m] = hi - lo;
    }
    if (order >= 1) S(s0 + d) = fx_to(8 * df[0] - df[1], E + up);
    s2[d == 0 ? 0 : (d == 1 ? 3 : 5)] = 16 * sp[0] - sp[1] - 30 * c[0];  // 12 h^2 d_d d_d
    const long long kd = 15 * sp[0] - 6 * sp[1] + sp[2] - 20 * c[0], o = 21 * df[0] - 6 * df[1] + df[2];
    const long long sg = neg[d];
    a[d] = kd + ((o ^ sg) - sg);
    a[3] += kd >> 1;
  }
  FxWeights<4> wt;
#pragma unroll
  for (int m = 0; m < 4; m++) wt.w[m] = wt_[m * Sh::THREADS];
  wt.E = wE;
  const double r = fx_dot(a, E, wt);
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
      // a quarter of 8 (l1 - l-1) - (l2 - l-2): 36 h^2 d_a d_b
      s2[m == 0 ? 1 : 2 * m] = 2 * (l[2] - l[1]) - ((l[3] - l[0]) >> 2);
    }
    {
      FxWeights<6> t;
#pragma unroll
      for (int m = 0; m < 6; m++) t.w[m] = wt_[(4 + m) * Sh::THREADS];
      t.E = gwE;
      S(s0 + 3) = fx_dot(s2, E + 2 + up, t);
    }
    if (q > 8) {
      const int n = q < 11 ? 6 : 3;
#pragma unroll 1
      for (int m = 0; m < n; m++) {
        const int ab = fx_kept(q, m);
        long long v = s2[0];
#pragma unroll
        for (int t = 1; t < 6; t++) v = ab == t ? s2[t] : v;
        const bool pure = ab == 0 || ab == 3 || ab == 5;  // 12 v = 16 (v - v/4)
        S(s0 + 4 + m) = fx_to(v - (pure ? v >> 2 : 0), E + (pure ? 4 : 2));
      }
    }
  }
  return r;
}

// The same from a box of float64 values (cold).
template <typename Sh, typename Slots>
__device__ __forceinline__ double fx_stencils_f64(const Grid& g, const double* __restrict__ c0, const FxMetric& M,
                                                  const double* c, int q, int order, int up, Slots S, int s0) {
  double d1[3], dd[6], wd[4];
  int neg[3];
  fx_adv_weights(g, c0, wd, neg);
  const double r = fx_field_f64(c, Sh::SY, Sh::SZ, wd, neg, up, d1, dd);
  if (order >= 1) {
#pragma unroll
    for (int d = 0; d < 3; d++) S(s0 + d) = d1[d];
  }
  if (order == 2) {
    double t = 0.0;
#pragma unroll 1
    for (int m = 0; m < 6; m++) {
      double v = M.gu[0];
#pragma unroll
      for (int n = 1; n < 6; n++) v = m == n ? M.g2u(n) : v;
      t = fma(v, dd[m], t);
    }
    S(s0 + 3) = t;
    if (q > 8) {
      const int n = q < 11 ? 6 : 3;
#pragma unroll 1
      for (int m = 0; m < n; m++) S(s0 + 4 + m) = dd[fx_kept(q, m)];
    }
  }
  return r;
}

// The right-hand side of all 24 fields at this thread's point (i, j, k) (stored
// indices, inside the grid) of the tile whose first interior point is (ii0,
// jj0, kk0), from the float64 register st, which map describes (its box that
// of Sh); every thread of the block calls it.  False: a wait ran out.
template <typename Sh>
__device__ __forceinline__ bool rhs_fx_tile(const void* map, const Grid& g, const double* __restrict__ st,
                                            FxShared<Sh>& sm, int tid, int ii0, int jj0, int kk0, int i, int j, int k,
                                            double out[NF]) {
  const long long fs = g.fstride, id = lin(g, i, j, k);
  const double* c0 = st + id;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  double slots[33];  // results of the stencils, in local memory
  auto S = [&](int n) -> double& { return slots[n]; };

  if (tid == 0) {
    for (int b = 0; b < 2; b++) mbar_init(smem_addr(&sm.bar[b]));
    fx_issue<Sh>(map, sm.box[0], smem_addr(&sm.bar[0]), ii0, jj0, kk0, fx_field(0));
  }
  const int cen = fx_center<Sh>(ii0, jj0, kk0, i, j, k);
  // (through the second buffer, which is still free)
  int* sc = reinterpret_cast<int*>(sm.box[1]) + tid;
  static_assert(Sh::PER * Sh::THREADS * sizeof(int) <= sizeof(sm.box[1]), "");
  fx_points<Sh>(g, tid, ii0, jj0, kk0, cen, sc);
  int neg[3];
  const FxWeights<4> aw = fx_tile_adv(g, c0, neg);
  FxMetric M;
  fx_metric(g, c0, M);
  const FxWeights<6> gw = fx_tile_gu(M);
  const bool wok = __syncthreads_and(aw.ok && gw.ok);  // (and the barriers are initialised)
  const int wE = aw.E, gwE = gw.E;
#pragma unroll
  for (int m = 0; m < 4; m++) sm.wt[m][tid] = aw.w[m];
#pragma unroll
  for (int m = 0; m < 6; m++) sm.wt[4 + m][tid] = gw.w[m];
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
    const bool there = mbar_wait(smem_addr(&sm.bar[q & 1]), (q >> 1) & 1, WAIT_LIMIT);
    double x[Sh::PER];
#pragma unroll
    for (int e = 0; e < Sh::PER; e++) x[e] = __longlong_as_double(box[at[e]]);
    const unsigned wtop = __reduce_max_sync(0xffffffffu, fx_top(x));
    if ((tid & 31) == 0) sm.top[tid >> 5] = wtop;
    // the maxima are there, and the previous field's box is free
    if (!__syncthreads_and(there)) {
      mbar_wait(smem_addr(&sm.bar[q & 1]), (q >> 1) & 1, WAIT_LIMIT);  // the one copy in flight lands before the block exits
      return false;
    }
    if (tid == 0 && q + 1 < NF)
      fx_issue<Sh>(map, sm.box[(q + 1) & 1], smem_addr(&sm.bar[(q + 1) & 1]), ii0, jj0, kk0, fx_field(q + 1));
    unsigned top = sm.top[0];
#pragma unroll
    for (int n = 1; n < Sh::WARPS; n++) top = max(top, sm.top[n]);
    // a box of zeros takes any exponent; top does not see low words of subnormals
    bool ok = fx_ok(top) && wok;
    if (top == 0) {
      unsigned lo = 0;
#pragma unroll
      for (int e = 0; e < Sh::PER; e++) lo |= (unsigned)__double2loint(x[e]);
      ok = !__syncthreads_or(lo != 0) && wok;
    }
    const int E = max((int)(top >> 20), 256) + FX_BITS - FX_TILE_BITS;  // the integers' unit is 2^(E - 1075 - FX_BITS)
    // (points that several threads share: the same value)
    if (ok) {
#pragma unroll
      for (int e = 0; e < Sh::PER; e++) box[at[e]] = fx_near<FX_TILE_BITS>(x[e], E + FX_TILE_BITS - FX_BITS);
    }
    __syncthreads();
    const int f = fx_field(q);
    double r;
    if (ok)
      r = fx_stencils<Sh>(c, q, order, up, E, &sm.wt[0][tid], wE, gwE, neg, S, s0);
    else
      r = fx_stencils_f64<Sh>(g, c0, M, reinterpret_cast<const double*>(c), q, order, up, S, s0);
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
