// ADM mass and angular momentum as volume integrals (arXiv:1111.3344, Sec.
// "Masses and Momenta", the ML_ADMQuantities form):
//   M   = 1/(16 pi) int [ e^{5 phi}(16 pi E + At_ij At^ij - (2/3) K^2) - e^{phi} Rt ]
//   J_i = 1/(8 pi) eps_ijk int e^{6 phi} [ At^j_k + (2/3) x^j d_k K
//                                          - (1/2) x^j At_ln d_k gt^{ln} + 8 pi x^j S_k ]
// (E = S_k = 0 unless a stress-energy tensor is given)
// with Rt = gt^ij Rt_ij built from the same pieces as the right-hand side
// (the evolved Gt in gt_k(i d_j) Gt^k, d_l gt^{lk} from the metric stencils
// elsewhere), d_k gt^{ln} = -gt^{la} gt^{nb} d_k gt_ab, so that
// At_ln d_k gt^{ln} = -At^{ab} d_k gt_ab; x^j the grid coordinates;
// e^{phi} = W^{-1/2} (W floored) or exp(phi).  The integrals are midpoint
// sums h^3 sum over interior points, over all of them and over the points
// farther than r_excise from every puncture.  Float64 in every precision mode.
//
// Formulation: only the trace of Rt_ij is formed,
//   Rt = -1/2 gt^ij gt^kl d_k d_l gt_ij + d_k Gt^k - 1/2 gt^ab d_k gt_ab d_l gt^lk
//        + 2 Gt^k_li Gt^i_k^l + Gt_klj Gt^klj,
// with integer-summed stencils (fx.cuh): about 450 float64 operations a point.
//
// One thread per interior point; per block a halving exchange in each warp and
// a serial sum over the warps (fixed order) into 8 partial sums (slot-major),
// then one block per result folds the partials, so the result does not depend
// on scheduling.
#include "curv3.cuh"

namespace bssn {

namespace {

constexpr int AB = 256;  // threads per block
constexpr int NQ = 8;    // M, J_x, J_y, J_z; full then excised

__device__ __forceinline__ void adm_density(const Grid& g, const double* __restrict__ y, long long id,
                                            const double x[3], double out[4]) {
  const long long fs = g.fstride, sy = g.pitch, sz = g.plane;
  const double* p = y + id;
  MetricD M;
  metric_stencils(p + F_GT * fs, fs, sy, sz, M);
  double dK[3];  // 12h d_d K
  fx_axes<false>(p + F_TRK * fs, sy, sz, 0, dK, nullptr);
  double dG = 0.0;  // 12h d_k Gt^k
#pragma unroll 1
  for (int a = 0; a < 3; a++) dG += fx_d1(p + (F_GAM + a) * fs, a == 0 ? 1 : (a == 1 ? sy : sz), 0);
  const double chi = __ldg(p + F_CHI * fs);
  const double trK = __ldg(p + F_TRK * fs);
  double gt[6], At[6], gu[6], g2u[6], G1[3][6], G2[3][6];
#pragma unroll
  for (int m = 0; m < 6; m++) {
    gt[m] = __ldg(p + (F_GT + m) * fs);
    At[m] = __ldg(p + (F_AT + m) * fs);
  }
  inverse3(gt, gu);
#pragma unroll
  for (int m = 0; m < 6; m++) g2u[m] = (m == 0 || m == 3 || m == 5) ? gu[m] : 2.0 * gu[m];
  christoffel_h(M.hg, gu, G1, G2);
  // Rt, times 144 h^2
  double Rtr = 0.0;
  {
    double s = 0.0;  // 72 h^2 gt^ij gt^kl d_k d_l gt_ij
#pragma unroll
    for (int m = 0; m < 6; m++) {
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < 6; q++) t = fma(g2u[q], M.hdd[m][q], t);
      s = fma(g2u[m], t, s);
    }
    Rtr = fma(g.h12, dG, -s);
    // V[k] = 6h gt^{kb} gt^{la} d_l gt_ab = -6h d_l gt^{lk}; tr[k] = 6h gt^ab d_k gt_ab
    double Tb[3];
#pragma unroll
    for (int b = 0; b < 3; b++) {
      double t = 0.0;
#pragma unroll
      for (int l = 0; l < 3; l++)
#pragma unroll
        for (int a = 0; a < 3; a++) t = fma(gu[sym(l, a)], M.hg[sym(a, b)][l], t);
      Tb[b] = t;
    }
    double q3 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double V = gu[sym(k, 0)] * Tb[0] + gu[sym(k, 1)] * Tb[1] + gu[sym(k, 2)] * Tb[2];
      double t = 0.0;
#pragma unroll
      for (int m = 0; m < 6; m++) t = fma(g2u[m], M.hg[m][k], t);
      q3 = fma(t, V, q3);
    }
    Rtr = fma(2.0, q3, Rtr);
    // H[i][k][l] = Gt^i_k^l; 2 Gt^k_li H[i][k][l] + Gt_k,lj Gt^k,lj
    double H[3][3][3];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int k = 0; k < 3; k++)
#pragma unroll
        for (int l = 0; l < 3; l++)
          H[i][k][l] = gu[sym(l, 0)] * G2[i][sym(k, 0)] + gu[sym(l, 1)] * G2[i][sym(k, 1)] + gu[sym(l, 2)] * G2[i][sym(k, 2)];
    double q1 = 0.0, q2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++) {
#pragma unroll
      for (int l = 0; l < 3; l++)
#pragma unroll
        for (int i = 0; i < 3; i++) q1 = fma(G2[k][sym(l, i)], H[i][k][l], q1);
#pragma unroll
      for (int l = 0; l < 3; l++)
#pragma unroll
        for (int j = l; j < 3; j++) {
          const double W = gu[sym(l, 0)] * H[k][0][j] + gu[sym(l, 1)] * H[k][1][j] + gu[sym(l, 2)] * H[k][2][j];
          if (l == j) Rtr = fma(G1[k][sym(l, j)], W, Rtr);
          else q2 = fma(G1[k][sym(l, j)], W, q2);
        }
    }
    Rtr = fma(2.0, q1 + q2, Rtr) * g.i144h2;
  }
  // e^{phi} and its powers
  double ephi;
  if (g.use_w) {
    const double Wd = chi > g.w_floor ? chi : g.w_floor;
    ephi = 1.0 / sqrt(Wd);
  } else {
    ephi = exp(chi);
  }
  const double e2 = ephi * ephi;
  const double e5 = e2 * e2 * ephi;
  const double e6 = e5 * ephi;
  // At^j_k = gt^{jl} At_lk (not symmetric) and At^{ab}
  double Am[3][3], Au[6];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++)
      Am[a][b] = gu[sym(a, 0)] * At[sym(0, b)] + gu[sym(a, 1)] * At[sym(1, b)] + gu[sym(a, 2)] * At[sym(2, b)];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a; b < 3; b++)
      Au[sym(a, b)] = Am[a][0] * gu[sym(0, b)] + Am[a][1] * gu[sym(1, b)] + Am[a][2] * gu[sym(2, b)];
  double Au2[6], AA = 0.0;
#pragma unroll
  for (int m = 0; m < 6; m++) {
    Au2[m] = (m == 0 || m == 3 || m == 5) ? Au[m] : 2.0 * Au[m];
    AA = fma(At[m], Au2[m], AA);
  }
  // matter: E and S_k (zero in vacuum)
  double Em = 0.0, Sk[3] = {0.0, 0.0, 0.0};
  if (g.tmunu) {
    const double alp = __ldg(y + F_ALP * g.fstride + id);
    const double beta[3] = {__ldg(y + F_BETA * g.fstride + id), __ldg(y + (F_BETA + 1) * g.fstride + id),
                            __ldg(y + (F_BETA + 2) * g.fstride + id)};
    double Sij[6];
    matter_at<double>(g, id, alp, beta, Em, Sk, Sij);
  }
  out[0] = (e5 * (16.0 * M_PI * Em + AA - (2.0 / 3.0) * trK * trK) - ephi * Rtr) * (1.0 / (16.0 * M_PI));
  // w[k] = (2/3) d_k K - (1/2) At_ln d_k gt^{ln} + 8 pi S_k, At_ln d_k gt^{ln} = -At^{ab} d_k gt_ab
  double w[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    double t = (2.0 / 3.0) * dK[k];
#pragma unroll
    for (int m = 0; m < 6; m++) t = fma(Au2[m], M.hg[m][k], t);
    w[k] = fma(g.i12h, t, (8.0 * M_PI) * Sk[k]);
  }
  const double c = e6 * (1.0 / (8.0 * M_PI));
#pragma unroll
  for (int i = 0; i < 3; i++) {  // eps_ijk (At^j_k + x^j w_k)
    const int j = (i + 1) % 3, k = (i + 2) % 3;
    out[1 + i] = c * ((Am[j][k] - Am[k][j]) + (x[j] * w[k] - x[k] * w[j]));
  }
}

// three blocks per SM (24 warps, 80 registers): 2.07 ms at 128^3, 2.15 with two
__global__ void __launch_bounds__(AB, 3) adm_integrals_kernel(Grid g, const double* __restrict__ y, Punct pu,
                                                              double* __restrict__ dens,
                                                              double* __restrict__ partials) {
  __shared__ double wsum[NQ][AB / 32];
  const unsigned npts = (unsigned)g.n0 * g.n1 * g.n2;
  const unsigned t = blockIdx.x * AB + threadIdx.x;
  double v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) v[q] = 0.0;
  if (t < npts) {
    const unsigned row = t / (unsigned)g.n0;
    const int ii = (int)(t - row * g.n0), kk = (int)(row / (unsigned)g.n1), jj = (int)(row - (unsigned)kk * g.n1);
    const long long id = lin(g, ii + GH, jj + GH, kk + GH);
    const double x[3] = {cell_coord(g.xmin0, ii, g.h), cell_coord(g.xmin1, jj, g.h), cell_coord(g.xmin2, kk, g.h)};
    double o[4];
    adm_density(g, y, id, x, o);
    if (dens) {
#pragma unroll
      for (int q = 0; q < 4; q++) dens[q * g.fstride + id] = o[q];
    }
    const bool outside = outside_punctures(pu, x[0], x[1], x[2]);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      v[q] = o[q];
      v[4 + q] = outside ? o[q] : 0.0;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double s = warp_sums<NQ>(v);
  if ((lane & 3) == 0) wsum[lane >> 2][warp] = s;
  __syncthreads();
  if (threadIdx.x < NQ) {
    double r = 0.0;
    for (int w = 0; w < AB / 32; w++) r += wsum[threadIdx.x][w];
    partials[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = r;
  }
}

// block q: result q, threads striding over its partials, then a fixed tree
__global__ void __launch_bounds__(AB) adm_integrals_finalize(const double* __restrict__ partials, int nblocks,
                                                             double vol, double* __restrict__ out) {
  __shared__ double a[AB];
  const double* p = partials + (size_t)blockIdx.x * nblocks;
  double v = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += AB) v += p[b];
  a[threadIdx.x] = v;
  for (int w = AB / 2; w > 0; w >>= 1) {
    __syncthreads();
    if (threadIdx.x < w) a[threadIdx.x] += a[threadIdx.x + w];
  }
  if (threadIdx.x == 0) out[blockIdx.x] = a[0] * vol;
}

}  // namespace

int adm_integrals_blocks(const Grid& g) {
  const long long npts = (long long)g.n0 * g.n1 * g.n2;
  return (int)((npts + AB - 1) / AB);
}

cudaError_t launch_adm_integrals(const Grid& g, const double* y, const Punct& pu, double* dens,
                                 double* partials, int nblocks, double* dout8, cudaStream_t s) {
  adm_integrals_kernel<<<nblocks, AB, 0, s>>>(g, y, pu, dens, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  adm_integrals_finalize<<<NQ, AB, 0, s>>>(partials, nblocks, g.h * g.h * g.h, dout8);
  return cudaGetLastError();
}

}  // namespace bssn
