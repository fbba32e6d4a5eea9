// Weyl scalar Psi4 (arXiv:1111.3344, Sec. "Gravitational Waves", WeylScal4):
// Psi4 = C_abcd n^a mb^b n^c mb^d for the fiducial tetrad n = (u - r)/sqrt2,
// mb = (theta - i phi)/sqrt2, from the projections of the vacuum curvature
// onto the slice (index 0 = along the unit normal u, so n^0 = 1/sqrt2 and
// mb^0 = 0):
//   R_ijkl n mb n mb + 2 n^0 R_0jkl mb n mb + (n^0)^2 R_0j0l mb mb
//   R_ijkl = 3R_ijkl + K_ik K_jl - K_il K_jk,  R_0jkl = D_k K_jl - D_l K_jk,
//   R_0j0l = 3R_jl + K K_jl - K_jm K^m_l.
// The triad starts from r = x^i, phi = (-y, x, 0),
// theta^i = sqrt(det g) g^ik eps_klm phi^l r^m and is made orthonormal in g_ij
// by Gram-Schmidt in the order phi, r, theta; Psi4 = 0 where phi = 0.
//
// Formulation (curv3.cuh): with the Einstein tensor G^mn = -D_mn / det g and, for
// the orthonormal triad, n.n = 1/2, mb.mb = n.mb = 0,
//   R(mb,mb) = G(mb,mb) and 3R(n, mb, n, mb) = R(mb,mb) / 2, so
//   Psi4 = R(mb,mb) + K(n,n) K(mb,mb) - K(n,mb)^2 + (K K(mb,mb) - (K.K)(mb,mb)) / 2
//          - mb^b r^c mb^d (D_c K_bd - D_d K_bc),
// evaluated with the triad's real vectors (mb = (t - i p)/sqrt2, n = -r/sqrt2).
// theta is orthogonal to phi and r from the start, so t_k = sqrt(det g) eps_klm
// p^l r^m from the unit p and r needs no projection and no normalisation; and
// eps_mcd r^c t^d = p_m / sqrt(det g), eps_mcd r^c p^d = -t_m / sqrt(det g) turn
// the last term into C_b^m p_m and C_b^m t_m.  K.K is summed over the triad.
// The ADM fields gamma_ij = e^{4 phi} gt_ij, K_ij = e^{4 phi}(At_ij + gt_ij K/3)
// are formed once per stored point (scratch register) and differenced with the
// 4th-order stencils.  Float64 in every precision mode; one thread per interior
// point.
#include "bssn_internal.cuh"
#include "curv3.cuh"

namespace bssn {

namespace {

constexpr int PB = 128;  // threads per block

__device__ __forceinline__ double dot3(const double a[3], const double b[3]) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}
// T_mn v^n of a symmetric 6-component tensor
__device__ __forceinline__ void sym_mul(const double T[6], const double v[3], double o[3]) {
#pragma unroll
  for (int m = 0; m < 3; m++) o[m] = T[sym(m, 0)] * v[0] + T[sym(m, 1)] * v[1] + T[sym(m, 2)] * v[2];
}

__device__ __forceinline__ void psi4_point(const Grid& g, const double* __restrict__ adm, long long id,
                                           const double x[3], double out[2]) {
  const long long fs = g.fstride, sy = g.pitch, sz = g.plane;
  const double* p = adm + id;
  out[0] = out[1] = 0.0;
  MetricD M;
  double dk[6][3];  // 12h d_d K_m
  metric_stencils(p, fs, sy, sz, M);
#pragma unroll 1
  for (int m = 0; m < 6; m++) {
    double d1[3];
    fx_axes<false>(p + (6 + m) * fs, sy, sz, 0, d1, nullptr);
    dk[m][0] = d1[0];
    dk[m][1] = d1[1];
    dk[m][2] = d1[2];
  }
  double g0[6], k0[6], gu[6], G1[3][6], G2[3][6], D[6], C[3][3];
#pragma unroll
  for (int m = 0; m < 6; m++) {
    g0[m] = __ldg(p + m * fs);
    k0[m] = __ldg(p + (6 + m) * fs);
  }
  const double idet = inverse3(g0, gu);
  christoffel_h(M.hg, gu, G1, G2);
  riemann6(M.hdd, G1, G2, D);
  codazzi3(dk, k0, G2, C);

  // triad p (phi), r, t (theta), upper and lower components
  double pv[3] = {-x[1], x[0], 0.0}, rv[3] = {x[0], x[1], x[2]}, tv[3], pl[3], rl[3], tl[3];
  sym_mul(g0, pv, pl);
  const double pp = dot3(pv, pl);
  if (!(pp > 0.0)) return;  // the z axis: no triad
  const double ip = 1.0 / sqrt(pp);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    pv[a] *= ip;
    pl[a] *= ip;
  }
  const double rp = dot3(rv, pl);
#pragma unroll
  for (int a = 0; a < 3; a++) rv[a] = fma(-rp, pv[a], rv[a]);
  sym_mul(g0, rv, rl);
  const double ir = 1.0 / sqrt(dot3(rv, rl));
#pragma unroll
  for (int a = 0; a < 3; a++) rv[a] *= ir;
  const double isdet = sqrt(idet), sdet = 1.0 / isdet;
  tl[0] = sdet * (pv[1] * rv[2] - pv[2] * rv[1]);
  tl[1] = sdet * (pv[2] * rv[0] - pv[0] * rv[2]);
  tl[2] = sdet * (pv[0] * rv[1] - pv[1] * rv[0]);
  sym_mul(gu, tl, tv);

  // R(mb,mb) from G^mn = -D_mn / det
  double Dt[3], Dp[3];
  sym_mul(D, tl, Dt);
  sym_mul(D, pl, Dp);
  const double gs = -idet * g.i144h2;
  const double Rmm_re = 0.5 * gs * (dot3(tl, Dt) - dot3(pl, Dp)), Rmm_im = -gs * dot3(pl, Dt);
  // forms of K on the triad
  double Kt[3], Kp[3], Kr[3];
  sym_mul(k0, tv, Kt);
  sym_mul(k0, pv, Kp);
  sym_mul(k0, rv, Kr);
  const double Ktt = dot3(tv, Kt), Kpp = dot3(pv, Kp), Ktp = dot3(pv, Kt);
  const double Krr = dot3(rv, Kr), Krt = dot3(rv, Kt), Krp = dot3(rv, Kp);
  const double trK = Ktt + Kpp + Krr;
  const double Kmm_re = 0.5 * (Ktt - Kpp), Kmm_im = -Ktp;                      // K(mb,mb)
  const double KK_re = 0.5 * ((Ktt * Ktt - Kpp * Kpp) + (Krt * Krt - Krp * Krp));  // (K.K)(mb,mb)
  const double KK_im = -(Ktp * (Ktt + Kpp) + Krt * Krp);
  // C_b^m (r x mb)_m with r x t = p_m / sqrt(det), r x p = -t_m / sqrt(det), then mb^b
  double Cp[3], Ct[3];
#pragma unroll
  for (int b = 0; b < 3; b++) {
    Cp[b] = dot3(C[b], pl);
    Ct[b] = dot3(C[b], tl);
  }
  const double cs = 0.5 * isdet * g.i12h;
  const double Cm_re = cs * (dot3(tv, Cp) + dot3(pv, Ct)), Cm_im = -cs * (dot3(pv, Cp) - dot3(tv, Ct));
  // K(n,n) = Krr / 2, K(n,mb) = -(Krt - i Krp) / 2
  out[0] = Rmm_re + 0.5 * Krr * Kmm_re - 0.25 * (Krt * Krt - Krp * Krp) + 0.5 * (trK * Kmm_re - KK_re) - Cm_re;
  out[1] = Rmm_im + 0.5 * Krr * Kmm_im + 0.5 * Krt * Krp + 0.5 * (trK * Kmm_im - KK_im) - Cm_im;
}

__global__ void __launch_bounds__(PB, 4) psi4_kernel(Grid g, const double* __restrict__ adm, double* __restrict__ out) {
  const unsigned npts = (unsigned)g.n0 * g.n1 * g.n2;
  const unsigned t = blockIdx.x * PB + threadIdx.x;
  if (t >= npts) return;
  const unsigned row = t / (unsigned)g.n0;
  const int ii = (int)(t - row * g.n0), kk = (int)(row / (unsigned)g.n1), jj = (int)(row - (unsigned)kk * g.n1);
  const long long id = lin(g, ii + GH, jj + GH, kk + GH);
  const double x[3] = {cell_coord(g.xmin0, ii, g.h), cell_coord(g.xmin1, jj, g.h), cell_coord(g.xmin2, kk, g.h)};
  double o[2];
  psi4_point(g, adm, id, x, o);
  out[id] = o[0];
  out[g.fstride + id] = o[1];
}

}  // namespace

cudaError_t launch_psi4(const Grid& g, const double* y, double* out, cudaStream_t s, double* adm_scratch) {
  const long long npts = (long long)g.n0 * g.n1 * g.n2;
  const unsigned blocks = (unsigned)((npts + PB - 1) / PB);
  const cudaError_t e = launch_adm_fields(g, y, adm_scratch, s);
  if (e != cudaSuccess) return e;
  psi4_kernel<<<blocks, PB, 0, s>>>(g, adm_scratch, out);
  return cudaGetLastError();
}

}  // namespace bssn
