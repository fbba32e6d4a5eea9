// The algebra of a point's right-hand side, arranged for the fewest float64
// instructions, in three parts that each follow the stencils they need (the
// per-point right-hand side of rhs_fx.cuh and the tile form of rhs_fx_tile.cuh
// share it).  The stencils' results come through accessors, in units of
// 12h per order of differentiation; u = 1/(12h).
//
// Arrangement (the equations of rhs_point.cuh; identities exact):
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
#pragma once
#include "bssn_internal.cuh"

namespace bssn {

// phi|W, the conformal metric and its inverse at the point c0 of field 0; in
// the W variant one division gives both 1/det and 1/W (W floored where it
// divides)
struct FxMetric {
  double chi, gt[6], gu[6], iW;
  // gt^ab with the off-diagonal entries doubled (symmetric contractions)
  __device__ __forceinline__ double g2u(int m) const { return (m == 0 || m == 3 || m == 5) ? gu[m] : 2.0 * gu[m]; }
};
__device__ __forceinline__ void fx_metric(const Grid& g, const double* __restrict__ c0, FxMetric& M) {
  const long long fs = g.fstride;
  const double chi = M.chi = __ldg(c0 + F_CHI * fs);
  double(&gt)[6] = M.gt, (&gu)[6] = M.gu;
  double& iW = M.iW;
  iW = 0.0;
#pragma unroll
  for (int m = 0; m < 6; m++) gt[m] = __ldg(c0 + (F_GT + m) * fs);
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

// X_ij = 144 h^2 Rt_ij, G2[k][ij] = 12h Gt^k_ij, V2[k] = -12h d_l gt^{lk}.
// HG(d, m) = 6h d_d gt_m, LAP(m) = 72 h^2 gt^{kl} d_k d_l gt_m, DG(a, d) = 6h d_d Gt^a.
template <typename H, typename L_, typename D>
__device__ __forceinline__ void fx_ricci(const Grid& g, const FxMetric& M, H HG, L_ LAP, D DG, double X[6],
                                         double G2[3][6], double V2[3]) {
  const double(&gt)[6] = M.gt, (&gu)[6] = M.gu;
  double hg[3][6];
#pragma unroll
  for (int d = 0; d < 3; d++)
#pragma unroll
    for (int m = 0; m < 6; m++) hg[d][m] = HG(d, m);
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
          v = hg[a][sym(a, a)];
        else if (a == b)
          v = fma(2.0, hg[a][sym(kk, a)], -hg[kk][sym(a, a)]);
        else if (kk == a)
          v = hg[b][sym(a, a)];
        else if (kk == b)
          v = hg[a][sym(b, b)];
        else
          v = hg[a][sym(kk, b)] + hg[b][sym(kk, a)] - hg[kk][sym(a, b)];
        G1[kk][sym(a, b)] = v;
      }
#pragma unroll
  for (int kk = 0; kk < 3; kk++)
#pragma unroll
    for (int m = 0; m < 6; m++)
      G2[kk][m] = gu[sym(kk, 0)] * G1[0][m] + gu[sym(kk, 1)] * G1[1][m] + gu[sym(kk, 2)] * G1[2][m];
  // V2[k] = -12h d_l gt^{lk} = 2 gt^{kb} gt^{la} (6h d_l gt_ab)
  double Tb[3];
#pragma unroll
  for (int b = 0; b < 3; b++) {
    double s = 0.0;
#pragma unroll
    for (int l = 0; l < 3; l++)
#pragma unroll
      for (int a = 0; a < 3; a++) s = fma(gu[sym(l, a)], hg[l][sym(a, b)], s);
    Tb[b] = 2.0 * s;
  }
#pragma unroll
  for (int kk = 0; kk < 3; kk++) V2[kk] = gu[sym(kk, 0)] * Tb[0] + gu[sym(kk, 1)] * Tb[1] + gu[sym(kk, 2)] * Tb[2];

  // ---- X_ij = 144 h^2 Rt_ij
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
        t = fma(gt[sym(kk, a)], DG(kk, b), t);
        if (a != b) t = fma(gt[sym(kk, b)], DG(kk, a), t);
      }
      // -1/2 gt^{kl} d_k d_l gt_ab
      double s = fma(a == b ? L2 : L, t, -LAP(ab));
      // Gt^k Gt_(ab)k with Gt^k = V2 / 12h, Gt_akb + Gt_bka = d_k gt_ab
#pragma unroll
      for (int kk = 0; kk < 3; kk++) s = fma(hg[kk][ab], V2[kk], s);
      // gt^{lm} (Gt^k_la Gt_bkm + Gt^k_lb Gt_akm + Gt^k_am Gt_klb); the first
      // two coincide on the diagonal
      if (a == b) {
        double t2 = 0.0;
#pragma unroll
        for (int kk = 0; kk < 3; kk++)
#pragma unroll
          for (int l = 0; l < 3; l++) {
            t2 = fma(G2[kk][sym(l, a)], G1u[a][kk][l], t2);
            s = fma(G2[kk][sym(a, l)], G1u[kk][a][l], s);
          }
        s = fma(2.0, t2, s);
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
}

// X_ij: 144 h^2 times the trace-free part of alpha R_ij - D_i D_j alpha +
// 4 d_(i phi d_j) alpha; lap: 144 h^2 (D^i D_i alpha + 2 d_i phi D^i alpha); vj:
// 12h (12 alpha d_a phi - 2 d_a alpha).  dchi, dalp: 12h times the derivatives
// of phi|W and alpha; lapA = 144 h^2 gt^kl d_k d_l alpha; DDC(m), DDA(m): 144 h^2
// times the second derivatives of phi|W and alpha.
template <typename C, typename A>
__device__ __forceinline__ void fx_lapse(const Grid& g, const FxMetric& M, double alp, const double dchi[3],
                                         const double dalp[3], double lapA, C DDC, A DDA, const double G2[3][6],
                                         double X[6], double& lap, double vj[3]) {
  const double(&gt)[6] = M.gt, (&gu)[6] = M.gu;
  double cw, cs, r[3], qv[3];
  if (g.use_w) {
    cw = alp * M.iW;  // alpha DD_ij W / W
    cs = -M.iW;       // 2 d phi = -dW / W
#pragma unroll
    for (int a = 0; a < 3; a++) r[a] = cs * dalp[a];
  } else {
    cw = -2.0 * alp;
    cs = 2.0;
#pragma unroll
    for (int a = 0; a < 3; a++) r[a] = 2.0 * fma(alp, dchi[a], dalp[a]);  // 4 alpha d_i phi d_j phi as well
  }
  lap = lapA;
  double cross = 0.0;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    vj[a] = fma(-6.0 * cw, dchi[a], -2.0 * dalp[a]);
    qv[a] = fma(cw, dchi[a], -dalp[a]);
    double t = 0.0;  // gt^kl Gt^a_kl
#pragma unroll
    for (int m = 0; m < 6; m++) t = fma(M.g2u(m), G2[a][m], t);
    const double ua = gu[sym(a, 0)] * dalp[0] + gu[sym(a, 1)] * dalp[1] + gu[sym(a, 2)] * dalp[2];
    cross = fma(dchi[a], ua, cross);
    lap = fma(-t, dalp[a], lap);
  }
  lap = fma(cs, cross, lap);
  double trX = 0.0;
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a; b < 3; b++) {
      const int ab = sym(a, b);
      double t = fma(cw, DDC(ab), -DDA(ab));
      t = fma(-G2[0][ab], qv[0], fma(-G2[1][ab], qv[1], fma(-G2[2][ab], qv[2], t)));
      X[ab] = fma(alp, X[ab], fma(dchi[a], r[b], fma(dchi[b], r[a], t)));
      trX = fma(M.g2u(ab), X[ab], trX);
    }
  trX *= 1.0 / 3.0;
#pragma unroll
  for (int m = 0; m < 6; m++) X[m] = fma(-gt[m], trX, X[m]);
}

// The right-hand sides, added onto out, which holds each field's advection and
// dissipation (zero for a frozen shift).  DB(a, d) = 12h d_d beta^a, LAPB(a) =
// 144 h^2 gt^kl d_k d_l beta^a, ROW(a, k) = 144 h^2 d_k d_a beta^a (no sum), DK(d) =
// 12h d_d K.  (i, j, k), id: the point's stored indices and linear index.
template <typename B_, typename L_, typename R, typename K_, typename Out>
__device__ __forceinline__ void fx_assemble(const Grid& g, const double* __restrict__ c0, long long id, int i, int j,
                                            int k, const FxMetric& M, B_ DB, L_ LAPB, R ROW, K_ DK,
                                            const double G2[3][6], const double V2[3], const double vj[3],
                                            const double X[6], double lap, Out out) {
  const long long fs = g.fstride;
  const double u = g.i12h, chi = M.chi;
  const double(&gt)[6] = M.gt, (&gu)[6] = M.gu;
  // ---- point values
  const double trK = __ldg(c0 + F_TRK * fs), alp = __ldg(c0 + F_ALP * fs);
  const double em4 = g.use_w ? chi * chi : exp(-4.0 * chi);
  const double em4u = em4 * g.i144h2;
  double At[6], Bv[3];
#pragma unroll
  for (int m = 0; m < 6; m++) At[m] = __ldg(c0 + (F_AT + m) * fs);
#pragma unroll
  for (int a = 0; a < 3; a++) Bv[a] = __ldg(c0 + (F_B + a) * fs);

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
    for (int a = 0; a < 3; a++) db[d][a] = u * DB(a, d);
  const double divb = db[0][0] + db[1][1] + db[2][2];
  const double divb3 = divb * (1.0 / 3.0);
#pragma unroll
  for (int d = 0; d < 3; d++) db[d][d] -= divb3;

  // ---- matter sources, when a stress-energy tensor is given
  double mG[3] = {0.0, 0.0, 0.0};
  if (g.tmunu) {
    double Em, Smi[3], Stf[6], beta[3];
#pragma unroll
    for (int a = 0; a < 3; a++) beta[a] = __ldg(c0 + (F_BETA + a) * fs);
    matter_at<double>(g, id, alp, beta, Em, Smi, Stf);
    double trs = 0.0;
#pragma unroll
    for (int m = 0; m < 6; m++) trs = fma(M.g2u(m), Stf[m], trs);
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
    double Q[3][3];  // db[b][k] - 2 alpha At^k_b
#pragma unroll
    for (int kk = 0; kk < 3; kk++)
#pragma unroll
      for (int b = 0; b < 3; b++) Q[kk][b] = fma(ma2, Aud[kk][b], db[b][kk]);
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
        for (int kk = 0; kk < 3; kk++) sa = fma(At[sym(a, kk)], Q[kk][b], fma(At[sym(kk, b)], db[a][kk], sa));
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
    double qv[3];
    const double u3 = u * (1.0 / 3.0), ak43 = (-4.0 / 3.0) * alp;
#pragma unroll
    for (int jj = 0; jj < 3; jj++) qv[jj] = fma(u3, ROW(0, jj) + ROW(1, jj) + ROW(2, jj), ak43 * DK(jj));
#pragma unroll
    for (int a = 0; a < 3; a++) {
      double br = 0.0;
#pragma unroll
      for (int m = 0; m < 6; m++) br = fma(G2[a][m], Auu2[m], br);
      double s = fma(u, LAPB(a), divb3 * V2[a]);
#pragma unroll
      for (int jj = 0; jj < 3; jj++)
        s = fma(gu[sym(a, jj)], qv[jj], fma(Auu[sym(a, jj)], vj[jj], fma(-V2[jj], db[jj][a], s)));
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

  if (g.shift == BSSN_SHIFT_FROZEN) return;  // beta^i and B^i: 0 from the field loop
  double eq = g.eta;
  if (g.q_R > 0.0 && !isinf(g.q_R)) {
    const double px = g.xmin0 + (i - GH + 0.5) * g.h, py = g.xmin1 + (j - GH + 0.5) * g.h,
                 pz = g.xmin2 + (k - GH + 0.5) * g.h;
    const double r = sqrt(px * px + py * py + pz * pz);
    if (!(r <= g.q_R)) eq *= g.q_R / r;
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    out[F_BETA + a] = fma(0.75, Bv[a], out[F_BETA + a]);
    out[F_B + a] += fma(-eq, Bv[a], gam_rhs[a]);
  }
}

}  // namespace bssn
