// Curvature of a 3-metric at a point, float64, for the analysis kernels
// (constraints, Psi4, ADM integrals; arXiv:1111.3344, Sec. "Other analysis
// modules", Sec. "Gravitational Waves", Sec. "Masses and Momenta").
//
// Bound: the float64 pipe (a warp instruction holds it for 64 cycles).  The
// stencils are integer sums (fx.cuh) and take none of it.  In three dimensions
// the Riemann tensor has six components, D_mn = R_{pair m, pair n} with pairs
// 0 = (y,z), 1 = (z,x), 2 = (x,y), and fixes all the rest:
//   R = (2 / det g) g_mn D_mn,   G^mn = -D_mn / det g (Einstein tensor),
// so no Ricci tensor is formed (about 60 float64 operations instead of 350).
// At 128^3, before (float64 stencils, Ricci tensor) and now: constraint norms
// 5.60 -> 1.62 ms, Psi4 7.83 -> 1.82 ms, ADM integrals 4.56 -> 2.14 ms.
// Likewise the antisymmetric derivatives of K, C_b^m = D_c K_bd - D_d K_bc with
// (c,d) = pair m, give both the momentum constraint and the magnetic part of
// Psi4; their Gamma^l_cd terms cancel.
//
// Units: first derivatives 12h d, second derivatives 144 h^2 d d; hg and hdd
// are halved (hg[d][m] = 6h d_d g_m, hdd[pq][m] = 72 h^2 d_p d_q g_m), which is
// the 1/2 of the Christoffel symbols and of the Riemann tensor.  Symmetric
// pairs as 6 components (sym()).
#pragma once
#include "bssn_internal.cuh"
#include "fx.cuh"

namespace bssn {

// Stencils of the six metric components at p, p + fs, ...; results in local
// memory (one copy of the code for the six).
struct MetricD {
  double hg[6][3];
  double hdd[6][6];  // [component][pair]
};
__device__ __forceinline__ void metric_stencils(const double* __restrict__ p, long long fs, long long sy, long long sz,
                                                MetricD& M) {
#pragma unroll 1
  for (int m = 0; m < 6; m++) {
    const double* q = p + m * fs;
    double d1[3], d2[3], dm[3];
    fx_axes<true>(q, sy, sz, -1, d1, d2);
    fx_mixed3(q, sy, sz, -1, dm);
#pragma unroll
    for (int d = 0; d < 3; d++) M.hg[m][d] = d1[d];
    M.hdd[m][0] = d2[0];
    M.hdd[m][1] = dm[0];
    M.hdd[m][2] = dm[1];
    M.hdd[m][3] = d2[1];
    M.hdd[m][4] = dm[2];
    M.hdd[m][5] = d2[2];
  }
}

// inverse of a symmetric 3-matrix by cofactors; returns 1 / det
__device__ __forceinline__ double inverse3(const double g[6], double gu[6]) {
  const double c00 = g[3] * g[5] - g[4] * g[4];
  const double c01 = g[2] * g[4] - g[1] * g[5];
  const double c02 = g[1] * g[4] - g[2] * g[3];
  const double idet = 1.0 / (g[0] * c00 + g[1] * c01 + g[2] * c02);
  gu[0] = c00 * idet;
  gu[1] = c01 * idet;
  gu[2] = c02 * idet;
  gu[3] = (g[0] * g[5] - g[2] * g[2]) * idet;
  gu[4] = (g[1] * g[2] - g[0] * g[4]) * idet;
  gu[5] = (g[0] * g[3] - g[1] * g[1]) * idet;
  return idet;
}

// 12h Gamma_kij and 12h Gamma^k_ij
__device__ __forceinline__ void christoffel_h(const double hg[6][3], const double gu[6], double G1[3][6],
                                              double G2[3][6]) {
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = a; b < 3; b++) {
        double v;
        if (a == b && k == a)
          v = hg[sym(a, a)][a];
        else if (a == b)
          v = fma(2.0, hg[sym(k, a)][a], -hg[sym(a, a)][k]);
        else if (k == a)
          v = hg[sym(a, a)][b];
        else if (k == b)
          v = hg[sym(b, b)][a];
        else
          v = hg[sym(k, b)][a] + hg[sym(k, a)][b] - hg[sym(a, b)][k];
        G1[k][sym(a, b)] = v;
      }
#pragma unroll
  for (int k = 0; k < 3; k++)
#pragma unroll
    for (int m = 0; m < 6; m++)
      G2[k][m] = gu[sym(k, 0)] * G1[0][m] + gu[sym(k, 1)] * G1[1][m] + gu[sym(k, 2)] * G1[2][m];
}

// first and second index of pair m: (1,2), (2,0), (0,1)
__host__ __device__ constexpr int pair_a(int m) { return m == 0 ? 1 : (m == 1 ? 2 : 0); }
__host__ __device__ constexpr int pair_b(int m) { return m == 0 ? 2 : (m == 1 ? 0 : 1); }

// 144 h^2 D_mn, six components: R_abcd = 1/2 (d_b d_c g_ad + d_a d_d g_bc
// - d_a d_c g_bd - d_b d_d g_ac) + Gamma_k,bc Gamma^k_ad - Gamma_k,bd Gamma^k_ac
__device__ __forceinline__ void riemann6(const double hdd[6][6], const double G1[3][6], const double G2[3][6],
                                         double D[6]) {
#pragma unroll
  for (int m = 0; m < 3; m++)
#pragma unroll
    for (int n = m; n < 3; n++) {
      const int a = pair_a(m), b = pair_b(m), c = pair_a(n), d = pair_b(n);
      double s;
      if (m == n)
        s = fma(2.0, hdd[sym(a, b)][sym(a, b)], -(hdd[sym(b, b)][sym(a, a)] + hdd[sym(a, a)][sym(b, b)]));
      else
        s = (hdd[sym(a, d)][sym(b, c)] + hdd[sym(b, c)][sym(a, d)]) -
            (hdd[sym(b, d)][sym(a, c)] + hdd[sym(a, c)][sym(b, d)]);
#pragma unroll
      for (int k = 0; k < 3; k++)
        s = fma(G1[k][sym(b, c)], G2[k][sym(a, d)], fma(-G1[k][sym(b, d)], G2[k][sym(a, c)], s));
      D[sym(m, n)] = s;
    }
}

// 12h C[b][m] = 12h (D_c K_bd - D_d K_bc), (c,d) = pair m; dk[j][d] = 12h d_d K_j
__device__ __forceinline__ void codazzi3(const double dk[6][3], const double K[6], const double G2[3][6],
                                         double C[3][3]) {
#pragma unroll
  for (int b = 0; b < 3; b++)
#pragma unroll
    for (int m = 0; m < 3; m++) {
      const int c = pair_a(m), d = pair_b(m);
      double s = dk[sym(b, d)][c] - dk[sym(b, c)][d];
#pragma unroll
      for (int l = 0; l < 3; l++)
        s = fma(G2[l][sym(d, b)], K[sym(l, c)], fma(-G2[l][sym(c, b)], K[sym(l, d)], s));
      C[b][m] = s;
    }
}

// Sum over the warp of N (8 or 16) values per lane: each step halves the
// values a lane keeps, so the sums take N + 1 float64 additions instead of 5 N.
// Lane l returns the sum of value l >> 2 (N = 8) or l >> 1 (N = 16).
template <int N>
__device__ __forceinline__ double warp_sums(double v[N]) {
  static_assert(N == 8 || N == 16, "");
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int n = N / 2; n >= 1; n >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int q = 0; q < n; q++) {
      const double keep = up ? v[n + q] : v[q], give = up ? v[q] : v[n + q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, off);
    }
  }
#pragma unroll
  for (int o = 16 / N; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// Whether (x, y, z) lies farther than r_excise from every puncture.
__device__ __forceinline__ bool outside_punctures(const Punct& pu, double x, double y, double z) {
  bool outside = true;
  for (int a = 0; a < pu.n; a++) {
    const double dx = x - pu.p[a][1], dy = y - pu.p[a][2], dz = z - pu.p[a][3];
    if (sqrt(dx * dx + dy * dy + dz * dz) <= pu.r_ex) outside = false;
  }
  return outside;
}

}  // namespace bssn
