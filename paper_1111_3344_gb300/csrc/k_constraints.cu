// Hamiltonian and momentum constraints with deterministic norm reductions
// (arXiv:1111.3344, Sec. "Other analysis modules"): H = R - K^i_j K^j_i + K^2,
// M_i = nabla_j K_i^j - nabla_i K in vacuum, from the ADM fields
// gamma_ij = e^{4 phi} gt_ij and K_ij = e^{4 phi}(At_ij + gt_ij K / 3), which
// are formed pointwise and then differenced with the same 4th-order stencils as
// the evolution.
//   R_ij = 1/2 gamma^kl (d_k d_j g_il + d_i d_l g_kj - d_k d_l g_ij - d_i d_j g_kl)
//          + gamma^kl (Gamma^m_il Gamma_mkj - Gamma^m_ij Gamma_mkl)
//   M_i  = gamma^jk (d_k K_ij - d_i K_jk) - Gamma^l K_il + Gamma^l_ij K_l^j
// (the Christoffel terms of gamma^jk (nabla_k K_ij - nabla_i K_jk) after the
// symmetric pair cancels).  With a stress-energy tensor, H gets -16 pi E and
// M_i gets -8 pi S_i.  Float64 in every precision mode.
//
// With a scratch register (every context) the ADM fields are formed once per
// stored point and the curvature is curv3.cuh's; without one (norms of a
// caller's state, no allocation) they are formed at every stencil point on the
// fly and R comes from the Ricci tensor (the formulas above).
//
// Reduction: one thread per interior point; per block a halving exchange in
// each warp and a serial sum over the warps, in a fixed order, into per-block
// partials (8 sums of squares, 8 maxima, 2 counts; slot-major), then one block
// per result folds the partials: the result does not depend on scheduling.
// The maxima are taken on the bit patterns of |.|, as integers, where a NaN
// is larger than every number.
#include "bssn_internal.cuh"
#include "curv3.cuh"
#include "ricci3.cuh"

namespace bssn {

constexpr int CB = 256;   // threads per block
constexpr int NPART = 18; // partial values per block

// ADM fields at one stored point, formed from the state.
__device__ __forceinline__ void adm_at(const Grid& g, const double* __restrict__ y, long long id, double gam[6],
                                       double K[6], bool needK) {
  const long long fs = g.fstride;
  const double chi = __ldg(y + F_CHI * fs + id);
  const double e4 = g.use_w ? 1.0 / (chi * chi) : exp(4.0 * chi);
  const double tr3 = needK ? __ldg(y + F_TRK * fs + id) * (1.0 / 3.0) : 0.0;
#pragma unroll
  for (int m = 0; m < 6; m++) {
    const double gt = __ldg(y + (F_GT + m) * fs + id);
    gam[m] = e4 * gt;
    if (needK) K[m] = e4 * (__ldg(y + (F_AT + m) * fs + id) + gt * tr3);
  }
}

// matter terms of the constraints: H -= 16 pi E, M_i -= 8 pi S_i
__device__ __forceinline__ void constraint_sources(const Grid& g, const double* __restrict__ y, long long id,
                                                   double out[4]) {
  if (!g.tmunu) return;
  const long long fs = g.fstride;
  const double alp = __ldg(y + F_ALP * fs + id);
  const double beta[3] = {__ldg(y + F_BETA * fs + id), __ldg(y + (F_BETA + 1) * fs + id),
                          __ldg(y + (F_BETA + 2) * fs + id)};
  double E, Si[3], Sij[6];
  matter_at<double>(g, id, alp, beta, E, Si, Sij);
  out[0] -= 16.0 * M_PI * E;
#pragma unroll
  for (int q = 0; q < 3; q++) out[1 + q] -= 8.0 * M_PI * Si[q];
}

// H and M_i at a point from the ADM fields of a scratch register (12 fields
// gamma_ij, K_ij).
__device__ __forceinline__ void constraints_point_adm(const Grid& g, const double* __restrict__ adm, long long id,
                                                      double out[4]) {
  const long long fs = g.fstride, sy = g.pitch, sz = g.plane;
  const double* p = adm + id;
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
  const double R = fma(2.0, g0[1] * D[1] + g0[2] * D[2] + g0[4] * D[4], g0[0] * D[0] + g0[3] * D[3] + g0[5] * D[5]);
  double Kud[3][3];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++)
      Kud[a][b] = gu[sym(a, 0)] * k0[sym(0, b)] + gu[sym(a, 1)] * k0[sym(1, b)] + gu[sym(a, 2)] * k0[sym(2, b)];
  const double trK = Kud[0][0] + Kud[1][1] + Kud[2][2];
  const double KK = fma(2.0, Kud[0][1] * Kud[1][0] + Kud[0][2] * Kud[2][0] + Kud[1][2] * Kud[2][1],
                        Kud[0][0] * Kud[0][0] + Kud[1][1] * Kud[1][1] + Kud[2][2] * Kud[2][2]);
  out[0] = fma(2.0 * g.i144h2 * idet, R, fma(trK, trK, -KK));
  // M_i = gamma^jk (D_k K_ij - D_i K_jk)
  codazzi3(dk, k0, G2, C);
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const int a = (i + 1) % 3, b = (i + 2) % 3;  // (a, i) is minus pair b, (b, i) pair a
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < 3; j++) s = fma(gu[sym(j, b)], C[j][a], fma(-gu[sym(j, a)], C[j][b], s));
    out[1 + i] = g.i12h * s;
  }
}

__device__ void constraints_point(const Grid& g, const double* __restrict__ y, long long id, double out[4]) {
  const long long sd[3] = {1, g.pitch, g.plane};
  const double i12h = g.i12h;
  const double i12h2 = g.i12h2;
  const double i144h2 = g.i144h2;
  double g0[6], k0[6];
  adm_at(g, y, id, g0, k0, true);
  double dg[3][6], dk[3][6], ddg[6][6];
#pragma unroll
  for (int d = 0; d < 3; d++) {
    double gp1[6], gm1[6], gp2[6], gm2[6], kp1[6], km1[6], kp2[6], km2[6];
    adm_at(g, y, id + sd[d], gp1, kp1, true);
    adm_at(g, y, id - sd[d], gm1, km1, true);
    adm_at(g, y, id + 2 * sd[d], gp2, kp2, true);
    adm_at(g, y, id - 2 * sd[d], gm2, km2, true);
#pragma unroll
    for (int m = 0; m < 6; m++) {
      dg[d][m] = fma(8.0, gp1[m] - gm1[m], -(gp2[m] - gm2[m])) * i12h;
      dk[d][m] = fma(8.0, kp1[m] - km1[m], -(kp2[m] - km2[m])) * i12h;
      ddg[sym(d, d)][m] = fma(-30.0, g0[m], fma(16.0, gp1[m] + gm1[m], -(gp2[m] + gm2[m]))) * i12h2;
    }
  }
  const double c[4] = {1.0, -8.0, 8.0, -1.0};
  const int off[4] = {-2, -1, 1, 2};
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a + 1; b < 3; b++) {
      double acc[6] = {0, 0, 0, 0, 0, 0};
      double dummy[6];
#pragma unroll
      for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) {
          double gv[6];
          adm_at(g, y, id + off[p] * sd[a] + off[q] * sd[b], gv, dummy, false);
          const double w = c[p] * c[q];
#pragma unroll
          for (int m = 0; m < 6; m++) acc[m] = fma(w, gv[m], acc[m]);
        }
#pragma unroll
      for (int m = 0; m < 6; m++) ddg[sym(a, b)][m] = acc[m] * i144h2;
    }

  // inverse metric
  double gu[6];
  {
    const double c00 = g0[3] * g0[5] - g0[4] * g0[4];
    const double c01 = g0[2] * g0[4] - g0[1] * g0[5];
    const double c02 = g0[1] * g0[4] - g0[2] * g0[3];
    const double idet = 1.0 / (g0[0] * c00 + g0[1] * c01 + g0[2] * c02);
    gu[0] = c00 * idet;
    gu[1] = c01 * idet;
    gu[2] = c02 * idet;
    gu[3] = (g0[0] * g0[5] - g0[2] * g0[2]) * idet;
    gu[4] = (g0[1] * g0[2] - g0[0] * g0[4]) * idet;
    gu[5] = (g0[0] * g0[3] - g0[1] * g0[1]) * idet;
  }
  // Christoffel symbols and Ricci tensor (ricci3.cuh); R = g^ij R_ij
  double G1[3][6], G2[3][6], Ric[6];
  christoffel3(gu, dg, G1, G2);
  ricci3(gu, ddg, G1, G2, Ric);
  double R = 0.0;
#pragma unroll
  for (int m = 0; m < 6; m++) R = fma((m == 0 || m == 3 || m == 5) ? gu[m] : 2.0 * gu[m], Ric[m], R);
  double Kud[3][3];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++)
      Kud[a][b] = gu[sym(a, 0)] * k0[sym(0, b)] + gu[sym(a, 1)] * k0[sym(1, b)] +
                  gu[sym(a, 2)] * k0[sym(2, b)];
  const double trK = Kud[0][0] + Kud[1][1] + Kud[2][2];
  double KK = 0.0;
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++) KK = fma(Kud[a][b], Kud[b][a], KK);
  out[0] = R - KK + trK * trK;

  // Gamma^l = gamma^jk Gamma^l_jk
  double Gc[3];
#pragma unroll
  for (int l = 0; l < 3; l++) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
      for (int k = 0; k < 3; k++) s = fma(gu[sym(j, k)], G2[l][sym(j, k)], s);
    Gc[l] = s;
  }
#pragma unroll
  for (int i = 0; i < 3; i++) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
      for (int k = 0; k < 3; k++) s = fma(gu[sym(j, k)], dk[k][sym(i, j)] - dk[i][sym(j, k)], s);
#pragma unroll
    for (int l = 0; l < 3; l++) {
      s = fma(-Gc[l], k0[sym(i, l)], s);
      // Gamma^l_ij K_l^j with K_l^j = Kud[j][l] (K symmetric)
#pragma unroll
      for (int j = 0; j < 3; j++) s = fma(G2[l][sym(i, j)], Kud[j][l], s);
    }
    out[1 + i] = s;
  }
}

// PRE: three blocks per SM (24 warps, 80 registers): 1.44 ms at 128^3 against
// 1.62 with two, 1.44 with four.
template <bool PRE>
__global__ void __launch_bounds__(CB, PRE ? 3 : 1) constraints_kernel(Grid g, const double* __restrict__ y,
                                                            const double* __restrict__ adm, Punct pu,
                                                            double* __restrict__ partials) {
  __shared__ double wsum[8][CB / 32];
  __shared__ long long wmax[8][CB / 32];
  __shared__ int wcnt[2][CB / 32];
  const unsigned npts = (unsigned)g.n0 * g.n1 * g.n2;
  const unsigned t = blockIdx.x * CB + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool in = t < npts;
  double v[8];
  long long m[8];
#pragma unroll
  for (int q = 0; q < 8; q++) {
    v[q] = 0.0;
    m[q] = 0;
  }
  bool outside = false;
  if (in) {
    const unsigned row = t / (unsigned)g.n0;
    const int ii = (int)(t - row * g.n0), kk = (int)(row / (unsigned)g.n1), jj = (int)(row - (unsigned)kk * g.n1);
    const long long id = lin(g, ii + GH, jj + GH, kk + GH);
    double c4[4];
    if constexpr (PRE) constraints_point_adm(g, adm, id, c4);
    else constraints_point(g, y, id, c4);
    constraint_sources(g, y, id, c4);
    outside = outside_punctures(pu, cell_coord(g.xmin0, ii, g.h), cell_coord(g.xmin1, jj, g.h),
                                cell_coord(g.xmin2, kk, g.h));
#pragma unroll
    for (int q = 0; q < 4; q++) {
      v[q] = c4[q] * c4[q];
      m[q] = __double_as_longlong(fabs(c4[q]));
      v[4 + q] = outside ? v[q] : 0.0;
      m[4 + q] = outside ? m[q] : 0;
    }
  }
  const double s = warp_sums<8>(v);
  if ((lane & 3) == 0) wsum[lane >> 2][warp] = s;
#pragma unroll
  for (int q = 0; q < 8; q++) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m[q] = max(m[q], __shfl_xor_sync(0xffffffffu, m[q], off));
    if (lane == 0) wmax[q][warp] = m[q];
  }
  const int n0 = __popc(__ballot_sync(0xffffffffu, in)), n1 = __popc(__ballot_sync(0xffffffffu, outside));
  if (lane == 0) {
    wcnt[0][warp] = n0;
    wcnt[1][warp] = n1;
  }
  __syncthreads();
  // slots: set * 8 + (0..3 sums of squares, 4..7 maxima), then the counts
  const int q = threadIdx.x;
  if (q >= NPART) return;
  double r;
  if (q >= 16) {
    int n = 0;
    for (int w = 0; w < CB / 32; w++) n += wcnt[q - 16][w];
    r = n;
  } else {
    const int src = (q >> 3) * 4 + (q & 3);
    if (q & 4) {
      long long n = 0;
      for (int w = 0; w < CB / 32; w++) n = max(n, wmax[src][w]);
      r = __longlong_as_double(n);
    } else {
      r = 0.0;
      for (int w = 0; w < CB / 32; w++) r += wsum[src][w];
    }
  }
  partials[(size_t)q * gridDim.x + blockIdx.x] = r;
}

// block q: result q from its slot's partials and, for the root mean squares,
// its set's counts; threads stride over the partials, then a fixed tree
__global__ void __launch_bounds__(CB) constraints_finalize(const double* __restrict__ partials, int nblocks,
                                                           double* __restrict__ out) {
  __shared__ double a[CB], c[CB];
  const int q = blockIdx.x;
  const bool mx = q & 4;
  const double* p = partials + (size_t)q * nblocks;
  const double* n = partials + (size_t)(16 + (q >> 3)) * nblocks;
  double v = 0.0, cnt = 0.0;
  long long m = 0;
  for (int b = threadIdx.x; b < nblocks; b += CB) {
    if (mx) {
      m = max(m, __double_as_longlong(p[b]));
    } else {
      v += p[b];
      cnt += n[b];
    }
  }
  a[threadIdx.x] = mx ? __longlong_as_double(m) : v;
  c[threadIdx.x] = cnt;
  for (int w = CB / 2; w > 0; w >>= 1) {
    __syncthreads();
    if (threadIdx.x < w) {
      if (mx) {
        a[threadIdx.x] = __longlong_as_double(
            max(__double_as_longlong(a[threadIdx.x]), __double_as_longlong(a[threadIdx.x + w])));
      } else {
        a[threadIdx.x] += a[threadIdx.x + w];
        c[threadIdx.x] += c[threadIdx.x + w];
      }
    }
  }
  if (threadIdx.x == 0) out[q] = mx ? a[0] : (c[0] > 0.0 ? sqrt(a[0] / c[0]) : 0.0);
}

int constraints_blocks(const Grid& g) {
  const long long npts = (long long)g.n0 * g.n1 * g.n2;
  return (int)((npts + CB - 1) / CB);
}

// gamma_ij = e^{4 phi} gt_ij and K_ij = e^{4 phi}(At_ij + gt_ij K/3) at every
// stored point into adm (12 fields of the register layout).
__global__ void adm_fields_kernel(Grid g, const double* __restrict__ y, double* __restrict__ adm) {
  const long long n = g.fstride;
  for (long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x; id < n;
       id += (long long)gridDim.x * blockDim.x) {
    double gam[6], K[6];
    adm_at(g, y, id, gam, K, true);
#pragma unroll
    for (int m = 0; m < 6; m++) {
      adm[m * n + id] = gam[m];
      adm[(6 + m) * n + id] = K[m];
    }
  }
}

cudaError_t launch_adm_fields(const Grid& g, const double* y, double* adm, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  adm_fields_kernel<<<sms * 8, 256, 0, s>>>(g, y, adm);
  return cudaGetLastError();
}

cudaError_t launch_constraints(const Grid& g, const double* y, const double* punct4, int npunct,
                               double r_excise, double* partials, int nblocks, double* dout16,
                               cudaStream_t s, double* adm_scratch) {
  Punct pu{};
  pu.n = npunct < 8 ? npunct : 8;
  for (int a = 0; a < pu.n; a++)
    for (int q = 0; q < 4; q++) pu.p[a][q] = punct4[4 * a + q];
  pu.r_ex = r_excise;
  cudaError_t e;
  if (adm_scratch) {
    if ((e = launch_adm_fields(g, y, adm_scratch, s)) != cudaSuccess) return e;
    constraints_kernel<true><<<nblocks, CB, 0, s>>>(g, y, adm_scratch, pu, partials);
  } else {
    constraints_kernel<false><<<nblocks, CB, 0, s>>>(g, y, nullptr, pu, partials);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  constraints_finalize<<<16, CB, 0, s>>>(partials, nblocks, dout16);
  return cudaGetLastError();
}

}  // namespace bssn
