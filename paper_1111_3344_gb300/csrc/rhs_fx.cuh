// Float64 BSSN right-hand side of one point (arXiv:1111.3344, Sec. "Spacetime
// Curvature Evolution"): the equations of rhs_point.cuh with every stencil
// summed exactly in 64-bit integers (fx.cuh) and the algebra arranged for the
// fewest float64 instructions.
//
// Bound: the float64 pipe, 64 cycles of an SM sub-partition for a warp
// instruction.  With the stencils in float64 a point took 1906 of them; here
// the stencils leave 6 per field (advection and dissipation) and none for the
// derivatives, the algebra and the combine about 970.  The integer work, some 25,000
// instructions a point, runs beside the float64 pipe.
//
// Advection: the lopsided stencil is the mean of the KO sum K and the odd sum O =
// 21 (f1 - f-1) - 6 (f2 - f-2) + (f3 - f-3), K + O on the side of positive beta and
// K - O on the other.
#pragma once
#include "bssn_internal.cuh"
#include "fx.cuh"
#include "fx_algebra.cuh"

namespace bssn {

// Advection and dissipation weights of a point: bh = |beta| / (24h), neg the
// signs of beta as masks, kap = eps / (64h).
struct FxAdv {
  double bh[3], kap;
  int neg[3];
};
// of the point c0 of field 0; i12h = 1/(12h), kap = eps / (64h)
__device__ __forceinline__ FxAdv fx_adv(const double* __restrict__ c0, long long fs, double i12h, double kap) {
  FxAdv w;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double b = __ldg(c0 + (F_BETA + d) * fs);
    w.bh[d] = fabs(b) * (0.5 * i12h);
    w.neg[d] = __double2hiint(b) >> 31;
  }
  w.kap = kap;
  return w;
}

// The sums along the three axes of the field at p (strides 1, sy, sz): returns
// sum_d bh[d] (K_d + sign_d O_d) + kap sum_d K_d, upwinded advection plus KO
// dissipation; order >= 1: d1 = 12 h d_d f times 2^up; order == 2: d2 =
// 144 h^2 d_d d_d f times 2^up (up is 0 or -1).
__device__ __forceinline__ double fx_axes(const double* p, long long sy, long long sz, const FxAdv& w, int order,
                                          int up, double d1[3], double d2[3]) {
  double v[19];
  v[0] = __ldg(p);
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const long long s = d == 0 ? 1 : (d == 1 ? sy : sz);
#pragma unroll
    for (int m = 1; m <= 3; m++) {
      v[6 * d + 2 * m - 1] = __ldg(p - m * s);
      v[6 * d + 2 * m] = __ldg(p + m * s);
    }
  }
  const unsigned top = fx_top(v);
  double r = 0.0;
#pragma unroll
  for (int d = 0; d < 3; d++) d1[d] = d2[d] = 0.0;
  if (fx_ok(top)) {
#pragma unroll
    for (int d = 0; d < 3; d++) {
      // the derivatives' five values in units of their own largest, the sums
      // with the third neighbours in units of all seven's
      const double* x = v + 6 * d;
      const double in[5] = {v[0], x[1], x[2], x[3], x[4]}, far[2] = {x[5], x[6]};
      const int Ei = max((int)(fx_top(in) >> 20), 256), E = max((int)(fx_top(far) >> 20), Ei);
      const long long f0 = fx_from(v[0], Ei);
      long long sm[3], df[3];
#pragma unroll
      for (int m = 0; m < 3; m++) {
        const long long a = fx_from(x[2 * m + 1], m < 2 ? Ei : E), b = fx_from(x[2 * m + 2], m < 2 ? Ei : E);
        sm[m] = b + a;
        df[m] = b - a;
      }
      if (order >= 1) d1[d] = fx_to(8 * df[0] - df[1], Ei + up);
      if (order == 2) d2[d] = fx_to(3 * (16 * sm[0] - sm[1] - 30 * f0), Ei + 2 + up);
      const long long k = fx_sar(15 * sm[0] - 6 * sm[1] - 20 * f0, E - Ei) + sm[2];
      const long long o = fx_sar(21 * df[0] - 6 * df[1], E - Ei) + df[2];
      const long long s = w.neg[d];
      r = fma(w.bh[d], fx_to(k + ((o ^ s) - s), E), r);
      r = fma(w.kap, fx_to(k, E), r);
    }
    return r;
  }
  if (fx_zero(v)) return 0.0;
  const double sc = up ? 0.5 : 1.0;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double* x = v + 6 * d;
    d1[d] = sc * fma(8.0, x[2] - x[1], -(x[4] - x[3]));
    d2[d] = 12.0 * sc * fma(-30.0, v[0], fma(16.0, x[2] + x[1], -(x[4] + x[3])));
    const double k = fma(15.0, x[2] + x[1], fma(-6.0, x[4] + x[3], x[6] + x[5])) - 20.0 * v[0];
    const double o = fma(21.0, x[2] - x[1], fma(-6.0, x[4] - x[3], x[6] - x[5]));
    r = fma(w.bh[d], w.neg[d] ? k - o : k + o, r);
    r = fma(w.kap, k, r);
  }
  return r;
}

// The stencils' results at a point, in local memory (indexed by the field loop).
struct FxPoint {
  double d1[15][3];  // 12h d_d of gt_ij (halved), phi|W, alpha, beta^i, K, Gt^i (halved)
  double lap[11];    // 144 h^2 gt^{kl} d_k d_l of gt_ij (halved), -, alpha, beta^i
  double dd[2][6];   // 144 h^2 d_a d_b of phi|W, alpha
  double row[3][3];  // 144 h^2 d_k d_a beta^a (no sum over a)
};

// One loop over the fields, so that the stencil code exists once: at some
// 2,700 instructions the whole right-hand side stays within the instruction
// cache (with one copy per kind of field it was 10 % slower, waiting on
// instruction fetch).  out: advection and dissipation.
__device__ __forceinline__ void fx_fields(const Grid& g, const double* __restrict__ c0, const FxAdv& w,
                                          const double g2u[6], int nf, FxPoint& P, double out[NF]) {
  const long long fs = g.fstride, sy = g.pitch, sz = g.plane;
#pragma unroll 1
  for (int q = 0; q < NF; q++) {
    // q: gt_ij, phi|W, alpha, beta^i | K, Gt^i | At_ij, B^i
    int f, order, up = 0;
    if (q < 11) {
      f = q < 6 ? F_GT + q : (q == 6 ? (int)F_CHI : q + (F_ALP - 7));
      order = 2;
      up = q < 6 ? -1 : 0;
    } else if (q < 15) {
      f = q == 11 ? (int)F_TRK : q + (F_GAM - 12);
      order = 1;
      up = q == 11 ? 0 : -1;
    } else {
      f = q < 21 ? q + (F_AT - 15) : q + (F_B - 21);
      order = 0;
    }
    const double* p = c0 + (long long)f * fs;
    double d1[3], d2[3];
    const double r = fx_axes(p, sy, sz, w, order, up, d1, d2);
    out[f] = f < nf ? r : 0.0;
    if (order == 0) continue;
    P.d1[q][0] = d1[0];
    P.d1[q][1] = d1[1];
    P.d1[q][2] = d1[2];
    if (order == 1) continue;
    double dm[3];
    fx_mixed3(p, sy, sz, up, dm);
    if (q != 6)
      P.lap[q] = fma(g2u[0], d2[0], fma(g2u[3], d2[1], g2u[5] * d2[2])) +
                 fma(g2u[1], dm[0], fma(g2u[2], dm[1], g2u[4] * dm[2]));
    if (q == 6 || q == 7) {
      double* x = P.dd[q - 6];
      x[0] = d2[0];
      x[1] = dm[0];
      x[2] = dm[1];
      x[3] = d2[1];
      x[4] = dm[2];
      x[5] = d2[2];
    } else if (q > 7) {
      double* x = P.row[q - 8];
      x[0] = q == 8 ? d2[0] : (q == 9 ? dm[0] : dm[1]);
      x[1] = q == 8 ? dm[0] : (q == 9 ? d2[1] : dm[2]);
      x[2] = q == 8 ? dm[1] : (q == 9 ? dm[2] : d2[2]);
    }
  }
}

// The right-hand side of all 24 fields at interior point (i, j, k), linear
// index id, from the float64 register st.  out and P are
// indexed by the loop over the fields and live in local memory.
__device__ __forceinline__ void rhs_fx(const Grid& g, const double* __restrict__ st, long long id, int i, int j, int k,
                                       double out[NF]) {
  const long long fs = g.fstride;
  const double* c0 = st + id;
  const double u = g.i12h;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;

  const FxAdv w = fx_adv(c0, fs, u, g.kos);

  FxMetric M;
  fx_metric(g, c0, M);
  double g2u[6];
#pragma unroll
  for (int m = 0; m < 6; m++) g2u[m] = M.g2u(m);

  FxPoint P;
  fx_fields(g, c0, w, g2u, nf, P, out);

  double X[6], G2[3][6], V2[3], vj[3], lap;
  fx_ricci(g, M, [&](int d, int m) { return P.d1[m][d]; }, [&](int m) { return P.lap[m]; },
           [&](int a, int d) { return P.d1[12 + a][d]; }, X, G2, V2);
  double dchi[3], dalp[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    dchi[a] = P.d1[6][a];
    dalp[a] = P.d1[7][a];
  }
  fx_lapse(g, M, __ldg(c0 + F_ALP * fs), dchi, dalp, P.lap[7], [&](int m) { return P.dd[0][m]; },
           [&](int m) { return P.dd[1][m]; }, G2, X, lap, vj);
  fx_assemble(g, c0, id, i, j, k, M, [&](int a, int d) { return P.d1[8 + a][d]; }, [&](int a) { return P.lap[8 + a]; },
              [&](int a, int m) { return P.row[a][m]; }, [&](int d) { return P.d1[11][d]; }, G2, V2, vj, X, lap, out);
}

}  // namespace bssn
