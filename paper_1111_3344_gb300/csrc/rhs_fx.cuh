// Float64 BSSN right-hand side of one point (arXiv:1111.3344, Sec. "Spacetime
// Curvature Evolution"): the equations of rhs_point.cuh with every stencil
// summed exactly in 64-bit integers (fx.cuh) and the algebra arranged for the
// fewest float64 instructions.
//
// Bound: the float64 pipe, 64 cycles of an SM sub-partition for a warp
// instruction.  With the stencils in float64 a point took 1906 of them; here
// the stencils leave 4 per field (advection and dissipation) and none for the
// derivatives, the algebra about 830.  The integer work, some 25,000
// instructions a point, runs beside the float64 pipe.
//
// Arrangement of the algebra (the same equations; identities exact):
//  - Derivatives carry the factor 12h per order (D1 sums as they are, 144 h^2
//    for second derivatives, the pure ones three times their sums and two
//    exponents up); u = 1/(12h) enters once per term of the results.  Metric
//    and Gt derivatives are halved (an exponent), so that Christoffel symbols
//    of the first kind need no factor 1/2.
//  - Only the trace-free part of alpha R_ij - D_i D_j alpha + ... enters, so
//    the terms gt_ij (scalar) of Rphi_ij are left out.
//  - W variant: -2 DD_ij phi + 4 d_i phi d_j phi = DD_ij W / W, the quadratic
//    terms cancelling.
//  - DD_ij alpha appears in the At equation beside DD_ij W with the same
//    Christoffel symbols, contracted once with alpha dW/W - d alpha; the lapse
//    Laplacian uses gt^kl Gt^m_kl.
//  - The trace of d_j beta^k is taken out of its diagonal before contraction.
//  - Advection: the lopsided stencil is the mean of the KO sum K and the odd
//    sum O = 21 (f1 - f-1) - 6 (f2 - f-2) + (f3 - f-3), K + O on the side of
//    positive beta and K - O on the other; the KO sums of the three axes are
//    added as integers and scaled once.
#pragma once
#include "bssn_internal.cuh"
#include "fx.cuh"

namespace bssn {

// Advection and dissipation weights of a point: bh = |beta| / (24h), neg the
// signs of beta as masks, kap = eps / (64h).
struct FxAdv {
  double bh[3], kap;
  int neg[3];
};

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
    const int E = (int)(top >> 20);
    const long long f0 = fx_from(v[0], E);
    long long K = 0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      long long sm[3], df[3];
#pragma unroll
      for (int m = 0; m < 3; m++) {
        const long long a = fx_from(v[6 * d + 2 * m + 1], E), b = fx_from(v[6 * d + 2 * m + 2], E);
        sm[m] = b + a;
        df[m] = b - a;
      }
      if (order >= 1) d1[d] = fx_to(8 * df[0] - df[1], E + up);
      if (order == 2) d2[d] = fx_to(3 * (16 * sm[0] - sm[1] - 30 * f0), E + 2 + up);
      const long long k = 15 * sm[0] - 6 * sm[1] + sm[2] - 20 * f0, o = 21 * df[0] - 6 * df[1] + df[2];
      const long long s = w.neg[d];
      K += k;
      r = fma(w.bh[d], fx_to(k + ((o ^ s) - s), E), r);
    }
    return fma(w.kap, fx_to(K, E), r);
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

  FxAdv w;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double b = __ldg(c0 + (F_BETA + d) * fs);
    w.bh[d] = fabs(b) * (0.5 * u);
    w.neg[d] = __double2hiint(b) >> 31;
  }
  w.kap = g.kos;

  // ---- inverse conformal metric; in the W variant one division gives both
  // 1/det and 1/W (W floored where it divides)
  const double chi = __ldg(c0 + F_CHI * fs);
  double gt[6], gu[6], iW = 0.0;
#pragma unroll
  for (int m = 0; m < 6; m++) gt[m] = __ldg(c0 + (F_GT + m) * fs);
  {
    const double c00 = gt[3] * gt[5] - gt[4] * gt[4];
    const double c01 = gt[2] * gt[4] - gt[1] * gt[5];
    const double c02 = gt[1] * gt[4] - gt[2] * gt[3];
    const double det = gt[0] * c00 + gt[1] * c01 + gt[2] * c02;
    double idet;
    if (g.use_w) {
      const double Wd = chi > g.w_floor ? chi : g.w_floor;
      const double r = 1.0 / (det * Wd);
      idet = Wd * r;
      iW = det * r;
    } else {
      idet = 1.0 / det;
    }
    gu[0] = c00 * idet;
    gu[1] = c01 * idet;
    gu[2] = c02 * idet;
    gu[3] = (gt[0] * gt[5] - gt[2] * gt[2]) * idet;
    gu[4] = (gt[1] * gt[2] - gt[0] * gt[4]) * idet;
    gu[5] = (gt[0] * gt[3] - gt[1] * gt[1]) * idet;
  }
  double g2u[6];  // gt^ab with the off-diagonal entries doubled (symmetric contractions)
#pragma unroll
  for (int m = 0; m < 6; m++) g2u[m] = (m == 0 || m == 3 || m == 5) ? gu[m] : 2.0 * gu[m];

  FxPoint P;
  fx_fields(g, c0, w, g2u, nf, P, out);

  double X[6], G2[3][6], V2[3];
  {
#define HG(d, m) P.d1[m][d]  // 6h d_d gt_m
    // ---- Christoffel symbols; G1[k][ij] and G2[k][ij] are 12h Gt_kij, 12h Gt^k_ij
    double G1[3][6];
#pragma unroll
    for (int kk = 0; kk < 3; kk++)
#pragma unroll
      for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = a; b < 3; b++) {
          double v;
          if (a == b && kk == a)
            v = HG(a, sym(a, a));
          else if (a == b)
            v = fma(2.0, HG(a, sym(kk, a)), -HG(kk, sym(a, a)));
          else if (kk == a)
            v = HG(b, sym(a, a));
          else if (kk == b)
            v = HG(a, sym(b, b));
          else
            v = HG(a, sym(kk, b)) + HG(b, sym(kk, a)) - HG(kk, sym(a, b));
          G1[kk][sym(a, b)] = v;
        }
#pragma unroll
    for (int kk = 0; kk < 3; kk++)
#pragma unroll
      for (int m = 0; m < 6; m++)
        G2[kk][m] = gu[sym(kk, 0)] * G1[0][m] + gu[sym(kk, 1)] * G1[1][m] + gu[sym(kk, 2)] * G1[2][m];
    // V2[k] = -12h d_l gt^{lk} = 2 gt^{kb} gt^{la} (6h d_l gt_ab)
    {
      double Tb[3];
#pragma unroll
      for (int b = 0; b < 3; b++) {
        double s = 0.0;
#pragma unroll
        for (int l = 0; l < 3; l++)
#pragma unroll
          for (int a = 0; a < 3; a++) s = fma(gu[sym(l, a)], HG(l, sym(a, b)), s);
        Tb[b] = 2.0 * s;
      }
#pragma unroll
      for (int kk = 0; kk < 3; kk++) V2[kk] = gu[sym(kk, 0)] * Tb[0] + gu[sym(kk, 1)] * Tb[1] + gu[sym(kk, 2)] * Tb[2];
    }

    // ---- 144 h^2 Rt_ij
    // G1u[j][k][l] = gt^{ls} Gt_jks (first kind, last index raised)
    double G1u[3][3][3];
#pragma unroll
    for (int jj = 0; jj < 3; jj++)
#pragma unroll
      for (int kk = 0; kk < 3; kk++)
#pragma unroll
        for (int l = 0; l < 3; l++)
          G1u[jj][kk][l] = gu[sym(l, 0)] * G1[jj][sym(kk, 0)] + gu[sym(l, 1)] * G1[jj][sym(kk, 1)] +
                           gu[sym(l, 2)] * G1[jj][sym(kk, 2)];
    const double L = g.h12, L2 = 2.0 * g.h12;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = a; b < 3; b++) {
        const int ab = sym(a, b);
        // gt_k(a d_b) Gt^k
        double t = 0.0;
#pragma unroll
        for (int kk = 0; kk < 3; kk++) {
          t = fma(gt[sym(kk, a)], P.d1[12 + kk][b], t);
          if (a != b) t = fma(gt[sym(kk, b)], P.d1[12 + kk][a], t);
        }
        // -1/2 gt^{kl} d_k d_l gt_ab
        double s = fma(a == b ? L2 : L, t, -P.lap[ab]);
        // Gt^k Gt_(ab)k with Gt^k = V2 / 12h, Gt_akb + Gt_bka = d_k gt_ab
#pragma unroll
        for (int kk = 0; kk < 3; kk++) s = fma(HG(kk, ab), V2[kk], s);
        // gt^{lm} (Gt^k_la Gt_bkm + Gt^k_lb Gt_akm + Gt^k_am Gt_klb); the first
        // two coincide on the diagonal
        if (a == b) {
          double q = 0.0;
#pragma unroll
          for (int kk = 0; kk < 3; kk++)
#pragma unroll
            for (int l = 0; l < 3; l++) {
              q = fma(G2[kk][sym(l, a)], G1u[a][kk][l], q);
              s = fma(G2[kk][sym(a, l)], G1u[kk][a][l], s);
            }
          s = fma(2.0, q, s);
        } else {
#pragma unroll
          for (int kk = 0; kk < 3; kk++)
#pragma unroll
            for (int l = 0; l < 3; l++) {
              s = fma(G2[kk][sym(l, a)], G1u[b][kk][l] + G1u[kk][b][l], s);
              s = fma(G2[kk][sym(l, b)], G1u[a][kk][l], s);
            }
        }
        X[ab] = s;
      }
#undef HG
  }

  // ---- phi|W and alpha: first and second derivatives
  const double alp = __ldg(c0 + F_ALP * fs);
  double dalp[3], vj[3], lap;  // 12h d_a alpha, 12h (12 alpha d_a phi - 2 d_a alpha), 144 h^2 (D^i D_i alpha + 2 d_i phi D^i alpha)
  {
    // X_ij: 144 h^2 times alpha R_ij - D_i D_j alpha + 4 d_(i phi d_j) alpha, up
    // to multiples of gt_ij
    double dchi[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
      dchi[a] = P.d1[6][a];
      dalp[a] = P.d1[7][a];
    }
    double cw, cs, r[3], q[3];
    if (g.use_w) {
      cw = alp * iW;  // alpha DD_ij W / W
      cs = -iW;       // 2 d phi = -dW / W
#pragma unroll
      for (int a = 0; a < 3; a++) {
        r[a] = cs * dalp[a];
        vj[a] = fma(-6.0 * cw, dchi[a], -2.0 * dalp[a]);
      }
    } else {
      cw = -2.0 * alp;
      cs = 2.0;
#pragma unroll
      for (int a = 0; a < 3; a++) {
        r[a] = 2.0 * fma(alp, dchi[a], dalp[a]);  // 4 alpha d_i phi d_j phi as well
        vj[a] = fma(-6.0 * cw, dchi[a], -2.0 * dalp[a]);
      }
    }
    lap = P.lap[7];
    double cross = 0.0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
      q[a] = fma(cw, dchi[a], -dalp[a]);
      double c = 0.0;  // gt^kl Gt^a_kl
#pragma unroll
      for (int m = 0; m < 6; m++) c = fma(g2u[m], G2[a][m], c);
      const double ua = gu[sym(a, 0)] * dalp[0] + gu[sym(a, 1)] * dalp[1] + gu[sym(a, 2)] * dalp[2];
      cross = fma(dchi[a], ua, cross);
      lap = fma(-c, dalp[a], lap);
    }
    lap = fma(cs, cross, lap);
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = a; b < 3; b++) {
        const int ab = sym(a, b);
        double t = fma(cw, P.dd[0][ab], -P.dd[1][ab]);
        t = fma(-G2[0][ab], q[0], fma(-G2[1][ab], q[1], fma(-G2[2][ab], q[2], t)));
        X[ab] = fma(alp, X[ab], fma(dchi[a], r[b], fma(dchi[b], r[a], t)));
      }
    double trX = 0.0;
#pragma unroll
    for (int m = 0; m < 6; m++) trX = fma(g2u[m], X[m], trX);
    trX *= 1.0 / 3.0;
#pragma unroll
    for (int m = 0; m < 6; m++) X[m] = fma(-gt[m], trX, X[m]);
  }

  // ---- point values
  const double trK = __ldg(c0 + F_TRK * fs);
  const double em4 = g.use_w ? chi * chi : exp(-4.0 * chi);
  const double em4u = em4 * g.i144h2;
  double At[6], beta[3], Bv[3];
#pragma unroll
  for (int m = 0; m < 6; m++) At[m] = __ldg(c0 + (F_AT + m) * fs);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    beta[a] = __ldg(c0 + (F_BETA + a) * fs);
    Bv[a] = __ldg(c0 + (F_B + a) * fs);
  }

  // ---- At with raised indices
  double Aud[3][3], Auu[6], Auu2[6];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++)
      Aud[a][b] = gu[sym(a, 0)] * At[sym(0, b)] + gu[sym(a, 1)] * At[sym(1, b)] + gu[sym(a, 2)] * At[sym(2, b)];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a; b < 3; b++)
      Auu[sym(a, b)] = Aud[a][0] * gu[sym(0, b)] + Aud[a][1] * gu[sym(1, b)] + Aud[a][2] * gu[sym(2, b)];
#pragma unroll
  for (int m = 0; m < 6; m++) Auu2[m] = (m == 0 || m == 3 || m == 5) ? Auu[m] : 2.0 * Auu[m];
  double AA = 0.0;
#pragma unroll
  for (int m = 0; m < 6; m++) AA = fma(Auu2[m], At[m], AA);

  // ---- shift derivatives db[d][a] = d_d beta^a with a third of the trace
  // taken out of the diagonal
  double db[3][3];
#pragma unroll
  for (int d = 0; d < 3; d++)
#pragma unroll
    for (int a = 0; a < 3; a++) db[d][a] = u * P.d1[8 + a][d];
  const double divb = db[0][0] + db[1][1] + db[2][2];
  const double divb3 = divb * (1.0 / 3.0);
#pragma unroll
  for (int d = 0; d < 3; d++) db[d][d] -= divb3;

  // ---- matter sources, when a stress-energy tensor is given
  double mG[3] = {0.0, 0.0, 0.0};
  if (g.tmunu) {
    double Em, Smi[3], Stf[6];
    matter_at<double>(g, id, alp, beta, Em, Smi, Stf);
    double trs = 0.0;
#pragma unroll
    for (int m = 0; m < 6; m++) trs = fma(g2u[m], Stf[m], trs);
    const double mA = (-8.0 * M_PI) * alp * em4;
#pragma unroll
    for (int m = 0; m < 6; m++)  // [S_ij]^TF (gt_ij gt^kl = gamma_ij gamma^kl)
      out[F_AT + m] = fma(mA, Stf[m] - gt[m] * trs * (1.0 / 3.0), out[F_AT + m]);
    out[F_TRK] += (4.0 * M_PI) * alp * (Em + em4 * trs);
#pragma unroll
    for (int a = 0; a < 3; a++)
      mG[a] = (-16.0 * M_PI) * alp * (gu[sym(a, 0)] * Smi[0] + gu[sym(a, 1)] * Smi[1] + gu[sym(a, 2)] * Smi[2]);
  }

  // ---- assemble onto the advection and dissipation
  const double ak = alp * trK, ma2 = -2.0 * alp;
  out[F_CHI] = g.use_w ? fma(chi * (1.0 / 3.0), ak - divb, out[F_CHI]) : fma(divb - ak, 1.0 / 6.0, out[F_CHI]);
  {
    double M[3][3];  // db[b][k] - 2 alpha At^k_b
#pragma unroll
    for (int kk = 0; kk < 3; kk++)
#pragma unroll
      for (int b = 0; b < 3; b++) M[kk][b] = fma(ma2, Aud[kk][b], db[b][kk]);
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = a; b < 3; b++) {
        const int ab = sym(a, b);
        double sg = fma(ma2, At[ab], out[F_GT + ab]), sa = fma(ak, At[ab], fma(em4u, X[ab], out[F_AT + ab]));
        if (a == b) {
          const double t = gt[sym(0, a)] * db[a][0] + gt[sym(1, a)] * db[a][1] + gt[sym(2, a)] * db[a][2];
          sg = fma(2.0, t, sg);
        } else {
#pragma unroll
          for (int kk = 0; kk < 3; kk++) sg = fma(gt[sym(kk, a)], db[b][kk], fma(gt[sym(kk, b)], db[a][kk], sg));
        }
#pragma unroll
        for (int kk = 0; kk < 3; kk++) sa = fma(At[sym(a, kk)], M[kk][b], fma(At[sym(kk, b)], db[a][kk], sa));
        out[F_GT + ab] = sg;
        out[F_AT + ab] = sa;
      }
  }
  out[F_TRK] = fma(alp, fma(trK * (1.0 / 3.0), trK, AA), fma(-em4u, lap, out[F_TRK]));

  double gam_rhs[3];
  {
    // 12h times: Gt^a_kl At^kl 2 alpha + At^aj (12 alpha d_j phi - 2 d_j alpha)
    // + gt^aj (1/3 d_j d_k beta^k - 4/3 alpha d_j K) + gt^kl d_k d_l beta^a
    // - Gt^j d_j beta^a + 2/3 Gt^a d_k beta^k
    double q[3];
    const double u3 = u * (1.0 / 3.0), ak43 = (-4.0 / 3.0) * alp;
#pragma unroll
    for (int jj = 0; jj < 3; jj++) q[jj] = fma(u3, P.row[0][jj] + P.row[1][jj] + P.row[2][jj], ak43 * P.d1[11][jj]);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      double br = 0.0;
#pragma unroll
      for (int m = 0; m < 6; m++) br = fma(G2[a][m], Auu2[m], br);
      double s = fma(u, P.lap[8 + a], divb3 * V2[a]);
#pragma unroll
      for (int jj = 0; jj < 3; jj++)
        s = fma(gu[sym(a, jj)], q[jj], fma(Auu[sym(a, jj)], vj[jj], fma(-V2[jj], db[jj][a], s)));
      s = u * fma(-ma2, br, s);
      if (g.tmunu) s += mG[a];
      gam_rhs[a] = s;
      out[F_GAM + a] += s;
    }
  }

  if (g.slicing == BSSN_1PLUSLOG)
    out[F_ALP] = fma(-2.0, ak, out[F_ALP]);
  else if (g.slicing == BSSN_HARMONIC)
    out[F_ALP] = fma(-alp, ak, out[F_ALP]);

  if (g.shift == BSSN_SHIFT_FROZEN) {
#pragma unroll
    for (int a = 0; a < 3; a++) out[F_BETA + a] = 0.0;
    return;
  }
  double eq = g.eta;
  if (g.q_R > 0.0 && !isinf(g.q_R)) {
    const double x = g.xmin0 + (i - GH + 0.5) * g.h, y = g.xmin1 + (j - GH + 0.5) * g.h,
                 z = g.xmin2 + (k - GH + 0.5) * g.h;
    const double r = sqrt(x * x + y * y + z * z);
    if (!(r <= g.q_R)) eq *= g.q_R / r;
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    out[F_BETA + a] = fma(0.75, Bv[a], out[F_BETA + a]);
    out[F_B + a] += fma(-eq, Bv[a], gam_rhs[a]);
  }
}

}  // namespace bssn
