// Per-ghost-point outer boundary work (Sommerfeld condition, periodic copy),
// shared by the single-grid kernels (k_boundary.cu) and the batched kernels
// (k_batch.cu).
#pragma once
#include "bssn_internal.cuh"
#include "rhs_point.cuh"
#include "stage_point.cuh"

namespace bssn {

__device__ __forceinline__ double coordv(const Grid& g, int d, int i) {
  const double xm = d == 0 ? g.xmin0 : (d == 1 ? g.xmin1 : g.xmin2);
  return xm + (i - GH + 0.5) * g.h;
}

// Offsets of the two neighbours per axis that the first differences at stored
// point I read: centred where both are stored, else the two inward ones.  Formed
// once per point, so that the fields' loads are under no branch and in flight
// together.
struct RadTaps {
  long long oa[3], ob[3];
  int kind[3];  // 0 centred, 1 one-sided at the last point, -1 at the first
  __device__ __forceinline__ bool edge() const { return (kind[0] | kind[1] | kind[2]) != 0; }
};
__device__ __forceinline__ RadTaps rad_taps(const Grid& g, const int I[3]) {
  const long long sd[3] = {1, g.pitch, g.plane};
  const int dims[3] = {g.sx, g.sy, g.sz};
  RadTaps T;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    T.kind[d] = I[d] >= 1 && I[d] + 1 < dims[d] ? 0 : (I[d] + 1 >= dims[d] ? 1 : -1);
    T.oa[d] = T.kind[d] == 1 ? -sd[d] : sd[d];
    T.ob[d] = T.kind[d] == 0 ? -sd[d] : 2 * T.oa[d];
  }
  return T;
}
// at an interior point
__device__ __forceinline__ RadTaps rad_taps_inside(const Grid& g) {
  return {{1, g.pitch, g.plane}, {-1, -g.pitch, -g.plane}, {0, 0, 0}};
}

// Radiative right-hand side of field f in arithmetic C at the point whose value
// p points at (its taps T); ns = (x / r) / (2h), the normal scaled by the
// difference weight (formed once per point for all fields), ir = 1 / r.
__device__ __forceinline__ bool rad_background(const Grid& g, int f) {
  return f == F_ALP || (f == F_CHI && g.use_w) || f == F_GT + 0 || f == F_GT + 3 || f == F_GT + 5;
}
template <typename C, typename S, bool DEV = false>
__device__ __forceinline__ C rad_at(const Grid& g, const S* __restrict__ p, int f, const RadTaps& T,
                                    const C ns[3], C ir) {
  const C X0 = (DEV || !rad_background(g, f)) ? C(0) : C(1);  // DEV: p holds X - X0 already
  const C v0 = (f == F_ALP || f == F_TRK) ? C(1.4142135623730951) : C(1);
  C s = ((C)p[0] - X0) * ir;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const C va = (C)p[T.oa[d]], vb = (C)p[T.ob[d]];
    C der;
    if (T.kind[d] == 0) {
      der = va - vb;
    } else {
      der = C(3) * (C)p[0] - C(4) * va + vb;
      if (T.kind[d] < 0) der = -der;
    }
    s = fmaT<C>(ns[d], der, s);
  }
  return -v0 * s;
}

// The same in float64 in two halves, for a group of fields: the values, then
// the sum.  One-sided differences become a - b with a = 3 p0 - 4 a, b = -b,
// negated at the first point with the normal's sign: one branch for the group
// (edge), for the float64 pipe bounds that kernel and most points need none.
struct RadVals {
  double p0, a[3], b[3];
  __device__ __forceinline__ void load(const double* __restrict__ p, const RadTaps& T) {
    p0 = p[0];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      a[d] = p[T.oa[d]];
      b[d] = p[T.ob[d]];
    }
  }
  __device__ __forceinline__ void edge(const RadTaps& T) {
#pragma unroll
    for (int d = 0; d < 3; d++)
      if (T.kind[d] != 0) {
        a[d] = 3.0 * p0 - 4.0 * a[d];
        b[d] = -b[d];
      }
  }
  __device__ __forceinline__ double sum(const Grid& g, int f, const RadTaps& T, const double ns[3], double ir) const {
    const double v0 = (f == F_ALP || f == F_TRK) ? 1.4142135623730951 : 1.0;
    double s = (p0 - (rad_background(g, f) ? 1.0 : 0.0)) * ir;
#pragma unroll
    for (int d = 0; d < 3; d++) s = fma(T.kind[d] < 0 ? -ns[d] : ns[d], a[d] - b[d], s);
    return -v0 * s;
  }
};

// Geometry of one ghost point: its anchor and the radial factors.
struct GhostGeo {
  int I[3], A[3];
  long long ib, ia;
  double nb[3], na[3], irb, ira, fac;
  double nbs[3], nas[3];  // nb, na times 1/(2h) (rad_at)
};

__device__ __forceinline__ void ghost_geo(const Grid& g, unsigned q, GhostGeo& G) {
  ghost_decode(g, q, G.I[0], G.I[1], G.I[2]);
  const int n[3] = {g.n0, g.n1, g.n2};
  // walk to the anchor: each step moves one layer inward along the summed normal
#pragma unroll
  for (int d = 0; d < 3; d++) {
    int a = G.I[d];
    if (a < GH) a = GH;
    else if (a >= GH + n[d]) a = GH + n[d] - 1;
    G.A[d] = a;
  }
  double xb[3], xa[3];
#pragma unroll
  for (int d = 0; d < 3; d++) {
    xb[d] = coordv(g, d, G.I[d]);
    xa[d] = coordv(g, d, G.A[d]);
  }
  const double rb = sqrt(xb[0] * xb[0] + xb[1] * xb[1] + xb[2] * xb[2]);
  const double ra = sqrt(xa[0] * xa[0] + xa[1] * xa[1] + xa[2] * xa[2]);
  G.irb = 1.0 / rb;
  G.ira = 1.0 / ra;
  G.fac = (ra * G.irb) * (ra * G.irb);
#pragma unroll
  for (int d = 0; d < 3; d++) {
    G.nb[d] = xb[d] * G.irb;
    G.na[d] = xa[d] * G.ira;
    G.nbs[d] = G.nb[d] * g.i2h;
    G.nas[d] = G.na[d] * g.i2h;
  }
  G.ib = lin(g, G.I[0], G.I[1], G.I[2]);
  G.ia = lin(g, G.A[0], G.A[1], G.A[2]);
}

// Geometry table of the float64 Sommerfeld boundary, one entry per ghost
// point q (formed once per context by ghost_geo, so the same values): the
// stored indices packed in 21 bits each, and nbs[3], irb, fac.
constexpr int GEO_DOUBLES = 5;
__host__ __device__ inline size_t ghost_table_bytes(const Grid& g) {
  return (size_t)ghost_count(g) * (GEO_DOUBLES * sizeof(double) + sizeof(long long));
}
__device__ __forceinline__ void ghost_table_fill(const Grid& g, unsigned q, double* __restrict__ tab,
                                                 long long* __restrict__ itab) {
  GhostGeo G;
  ghost_geo(g, q, G);
  const size_t n = ghost_count(g);
  tab[0 * n + q] = G.nbs[0];
  tab[1 * n + q] = G.nbs[1];
  tab[2 * n + q] = G.nbs[2];
  tab[3 * n + q] = G.irb;
  tab[4 * n + q] = G.fac;
  itab[q] = (long long)G.I[0] | ((long long)G.I[1] << 21) | ((long long)G.I[2] << 42);
}

// The anchor's factors (nas, ira) as ghost_geo forms them.
__device__ __forceinline__ double anchor_geo(const Grid& g, const int A[3], double nas[3]) {
  double xa[3];
#pragma unroll
  for (int d = 0; d < 3; d++) xa[d] = coordv(g, d, A[d]);
  const double ira = 1.0 / sqrt(xa[0] * xa[0] + xa[1] * xa[1] + xa[2] * xa[2]);
#pragma unroll
  for (int d = 0; d < 3; d++) nas[d] = (xa[d] * ira) * g.i2h;
  return ira;
}

// float64 path from the table: ghost point q, fields [F0, F1) (a group of the 24
// per thread, their loads in flight together).  A stage: after the anchor pass,
// from the k - rad that it left in kanchor.  OWN (a right-hand side alone, which
// has no memory but its output to leave anything in): the k of the output, and
// the anchor's radiative term formed here.
template <int F0, int F1, bool OWN = false>
__device__ __forceinline__ void sommerfeld_point_fp64_tab(const Grid& g, const StageArgs& a,
                                                          const double* __restrict__ kanchor,
                                                          const double* __restrict__ tab,
                                                          const long long* __restrict__ itab, unsigned q) {
  const size_t n = ghost_count(g);
  const long long pk = itab[q];
  const int I[3] = {(int)(pk & 0x1fffff), (int)((pk >> 21) & 0x1fffff), (int)((pk >> 42) & 0x1fffff)};
  const int nn[3] = {g.n0, g.n1, g.n2};
  int A[3];
#pragma unroll
  for (int d = 0; d < 3; d++) A[d] = I[d] < GH ? GH : (I[d] >= GH + nn[d] ? GH + nn[d] - 1 : I[d]);
  const double nbs[3] = {tab[q], tab[n + q], tab[2 * n + q]};
  const double irb = tab[3 * n + q], fac = tab[4 * n + q];
  const long long ib = lin(g, I[0], I[1], I[2]), ia = lin(g, A[0], A[1], A[2]);
  const long long fs = g.fstride;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  const RadTaps tb = rad_taps(g, I);
  constexpr int N = F1 - F0;
  long long o[N];
  RadVals v[N];
  double ka[N], rhs[N];
#pragma unroll
  for (int n = 0; n < N; n++) {
    o[n] = (F0 + n) * fs + ib;
    v[n].load(a.src + o[n], tb);
    if (!OWN) ka[n] = kanchor[(F0 + n) * fs + ia];
  }
  if constexpr (OWN) {
    double nas[3];
    const double ira = anchor_geo(g, A, nas);
    const RadTaps ta = rad_taps_inside(g);
#pragma unroll
    for (int n = 0; n < N; n++) {
      const long long oa = (F0 + n) * fs + ia;
      ka[n] = a.rhs[oa] - rad_at<double, double>(g, a.src + oa, F0 + n, ta, nas, ira);
    }
  }
  if (tb.edge()) {
#pragma unroll
    for (int n = 0; n < N; n++) v[n].edge(tb);
  }
#pragma unroll
  for (int n = 0; n < N; n++)
    rhs[n] = F0 + n < nf ? fma(fac, ka[n], v[n].sum(g, F0 + n, tb, nbs, irb)) : 0.0;
  combine_point_fp64(a, o, rhs, false);
}

// float64 path, anchor pass: interior point q of the boundary shell, fields
// [F0, F1): k - rad at the anchor, in place of the k the stage kernel left in
// kanchor (the same operations the ghost points of that anchor would repeat,
// one to three layers and up to eight neighbours over; see sommerfeld_point_fp64).
template <int F0 = 0, int F1 = NF>
__device__ __forceinline__ void sommerfeld_anchor_fp64(const Grid& g, const StageArgs& a,
                                                       double* __restrict__ kanchor, unsigned q) {
  int ii, jj, kk;
  shell_decode(g, q, ii, jj, kk);
  const int A[3] = {ii + GH, jj + GH, kk + GH};
  double nas[3];
  const double ira = anchor_geo(g, A, nas);
  const long long ia = lin(g, A[0], A[1], A[2]);
  const long long fs = g.fstride;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  const RadTaps ta = rad_taps_inside(g);
  double k[F1 - F0];  // every load before the stores
#pragma unroll
  for (int f = F0; f < F1; f++)
    if (f < nf) k[f - F0] = kanchor[f * fs + ia] - rad_at<double, double>(g, a.src + f * fs + ia, f, ta, nas, ira);
#pragma unroll
  for (int f = F0; f < F1; f++)
    if (f < nf) kanchor[f * fs + ia] = k[f - F0];
}

// float64 path: ghost point q, all fields, from the k at the anchors (the batched
// kernel, whose members' anchors no pass of their own has treated).
__device__ __forceinline__ void sommerfeld_point_fp64(const Grid& g, const StageArgs& a,
                                                      const double* __restrict__ kanchor, unsigned q) {
  GhostGeo G;
  ghost_geo(g, q, G);
  const long long fs = g.fstride;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  const RadTaps tb = rad_taps(g, G.I), ta = rad_taps_inside(g);
  for (int f = 0; f < NF; f++) {
    double rhs[1] = {0.0};
    const long long o[1] = {f * fs + G.ib};
    if (f < nf) {
      const double radb = rad_at<double, double>(g, a.src + f * fs + G.ib, f, tb, G.nbs, G.irb);
      const double rada = rad_at<double, double>(g, a.src + f * fs + G.ia, f, ta, G.nas, G.ira);
      rhs[0] = fma(G.fac, kanchor[f * fs + G.ia] - rada, radb);
    }
    combine_fields_fp64(a, o, rhs);
  }
}

// mixed path: ghost point q, field f; float arithmetic, W in float64; RK4
// roles as in the stage kernel.
__device__ __forceinline__ void sommerfeld_point_mixed(const Grid& g, const StageArgsMixed& a,
                                                       const float* __restrict__ kanchor, unsigned q,
                                                       int f) {
  const long long fs = g.fstride;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  int I[3], A[3];
  ghost_decode(g, q, I[0], I[1], I[2]);
  const int n[3] = {g.n0, g.n1, g.n2};
#pragma unroll
  for (int d = 0; d < 3; d++) A[d] = I[d] < GH ? GH : (I[d] >= GH + n[d] ? GH + n[d] - 1 : I[d]);
  const long long ib = lin(g, I[0], I[1], I[2]);
  const long long ia = lin(g, A[0], A[1], A[2]);
  const long long o = f * fs + ib;
  const RadTaps tb = rad_taps(g, I), ta = rad_taps_inside(g);
  if (f == F_CHI) {
    GhostGeo G;
    ghost_geo(g, q, G);
    const double radb = rad_at<double, double>(g, a.srcw + ib, f, tb, G.nbs, G.irb);
    const double rada = rad_at<double, double>(g, a.srcw + ia, f, ta, G.nas, G.ira);
    const double ka = (a.mode == MODE_RHS) ? a.rhs[ia] : (double)kanchor[ia];
    const double rhs = fma(G.fac, ka - rada, radb);
    if (a.mode == MODE_RHS) {
      a.rhs[o] = rhs;
    } else if (a.mode == MODE_LAST) {
      const double v = fma(a.b_dt, a.ksumw[ib] + rhs, a.yn[ib]);
      a.yn[ib] = v;
      a.out0[ib] = (float)(v - background(g, F_CHI));
      a.out0w[ib] = v;
    } else {
      const double v = fma(a.a_dt, rhs, a.src0w[ib]);
      a.out0w[ib] = v;
      a.out0[ib] = (float)(v - background(g, F_CHI));
      a.ksumw[ib] = a.mode == MODE_FIRST ? rhs : fma(2.0, rhs, a.ksumw[ib]);
    }
    return;
  }
  float rhs = 0.0f;
  if (f < nf) {
    float xb[3], xa[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      xb[d] = fmaf((float)(I[d] - GH) + 0.5f, g.hf, g.xminf[d]);
      xa[d] = fmaf((float)(A[d] - GH) + 0.5f, g.hf, g.xminf[d]);
    }
    const float irb = rsqrtf(xb[0] * xb[0] + xb[1] * xb[1] + xb[2] * xb[2]);
    const float ira = rsqrtf(xa[0] * xa[0] + xa[1] * xa[1] + xa[2] * xa[2]);
    const float nbs[3] = {xb[0] * irb * g.i2hf, xb[1] * irb * g.i2hf, xb[2] * irb * g.i2hf};
    const float nas[3] = {xa[0] * ira * g.i2hf, xa[1] * ira * g.i2hf, xa[2] * ira * g.i2hf};
    const float fac = (irb / ira) * (irb / ira);
    const float radb = rad_at<float, float, true>(g, a.src + o, f, tb, nbs, irb);
    const float rada = rad_at<float, float, true>(g, a.src + f * fs + ia, f, ta, nas, ira);
    const float ka = (a.mode == MODE_RHS) ? (float)a.rhs[f * fs + ia] : kanchor[f * fs + ia];
    rhs = fmaf(fac, ka - rada, radb);
  }
  if (a.mode == MODE_RHS) {
    a.rhs[o] = (double)rhs;
  } else if (a.mode == MODE_LAST) {
    const double ks = a.ksum64 ? a.ksum64[o] + (double)rhs : (double)(a.ksum[o] + rhs);
    const double v = fma(a.b_dt, ks, a.yn[o]);
    a.yn[o] = v;
    a.out0[o] = (float)(v - background(g, f));
  } else {
    a.out0[o] = fmaf(a.a_dtf, rhs, a.src0[o]);
    if (a.ksum64)
      a.ksum64[o] = a.mode == MODE_FIRST ? (double)rhs : fma(2.0, (double)rhs, a.ksum64[o]);
    else
      a.ksum[o] = a.mode == MODE_FIRST ? rhs : fmaf(2.0f, rhs, a.ksum[o]);
  }
}

// mixed path, ghost point q, fields [F0, F1): the same per-field arithmetic
// as sommerfeld_point_mixed with the geometry (index decode, anchor,
// coordinates, normals) formed once for the group's float fields; W (field 0,
// when in the group) in float64.  UNROLL: the field loop unrolled, so that the
// group's loads are in flight together.
template <int F0, int F1, bool UNROLL>
__device__ __forceinline__ void sommerfeld_point_mixed_fields(const Grid& g, const StageArgsMixed& a,
                                                              const float* __restrict__ kanchor, unsigned q) {
  if constexpr (F0 == 0) sommerfeld_point_mixed(g, a, kanchor, q, F_CHI);  // W: float64 geometry and arithmetic
  constexpr int FB = F0 == 0 ? 1 : F0;
  const long long fs = g.fstride;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  int I[3], A[3];
  ghost_decode(g, q, I[0], I[1], I[2]);
  const int n[3] = {g.n0, g.n1, g.n2};
#pragma unroll
  for (int d = 0; d < 3; d++) A[d] = I[d] < GH ? GH : (I[d] >= GH + n[d] ? GH + n[d] - 1 : I[d]);
  const long long ib = lin(g, I[0], I[1], I[2]);
  const long long ia = lin(g, A[0], A[1], A[2]);
  float xb[3], xa[3];
#pragma unroll
  for (int d = 0; d < 3; d++) {
    xb[d] = fmaf((float)(I[d] - GH) + 0.5f, g.hf, g.xminf[d]);
    xa[d] = fmaf((float)(A[d] - GH) + 0.5f, g.hf, g.xminf[d]);
  }
  const float irb = rsqrtf(xb[0] * xb[0] + xb[1] * xb[1] + xb[2] * xb[2]);
  const float ira = rsqrtf(xa[0] * xa[0] + xa[1] * xa[1] + xa[2] * xa[2]);
  // normals times 1/(2h) (rad_at)
  const float nbs[3] = {xb[0] * irb * g.i2hf, xb[1] * irb * g.i2hf, xb[2] * irb * g.i2hf};
  const float nas[3] = {xa[0] * ira * g.i2hf, xa[1] * ira * g.i2hf, xa[2] * ira * g.i2hf};
  const float fac = (irb / ira) * (irb / ira);
  const RadTaps tb = rad_taps(g, I), ta = rad_taps_inside(g);
  // groups of N fields, every load of a group before its stores
  constexpr int N = UNROLL && F1 > FB ? F1 - FB : 1;
#pragma unroll 1
  for (int f0 = FB; f0 < F1; f0 += N) {
    float rhs[N], b[N], ks[N];
    double bd[N], kd[N];
#pragma unroll
    for (int m = 0; m < N; m++) {
      const int f = f0 + m;
      rhs[m] = 0.0f;
      if (f < nf) {
        const float radb = rad_at<float, float, true>(g, a.src + f * fs + ib, f, tb, nbs, irb);
        const float rada = rad_at<float, float, true>(g, a.src + f * fs + ia, f, ta, nas, ira);
        const float ka = (a.mode == MODE_RHS) ? (float)a.rhs[f * fs + ia] : kanchor[f * fs + ia];
        rhs[m] = fmaf(fac, ka - rada, radb);
      }
    }
    if (a.mode == MODE_RHS) {
#pragma unroll
      for (int m = 0; m < N; m++) a.rhs[(f0 + m) * fs + ib] = (double)rhs[m];
      continue;
    }
    if (a.mode != MODE_FIRST && a.ksum64) {
#pragma unroll
      for (int m = 0; m < N; m++) kd[m] = a.ksum64[(f0 + m) * fs + ib];
    } else if (a.mode != MODE_FIRST) {
#pragma unroll
      for (int m = 0; m < N; m++) ks[m] = a.ksum[(f0 + m) * fs + ib];
    }
    if (a.mode == MODE_LAST) {
#pragma unroll
      for (int m = 0; m < N; m++) bd[m] = a.yn[(f0 + m) * fs + ib];
#pragma unroll
      for (int m = 0; m < N; m++) {
        const long long o = (f0 + m) * fs + ib;
        const double v = fma(a.b_dt, a.ksum64 ? kd[m] + (double)rhs[m] : (double)(ks[m] + rhs[m]), bd[m]);
        a.yn[o] = v;
        a.out0[o] = (float)(v - background(g, f0 + m));
      }
      continue;
    }
#pragma unroll
    for (int m = 0; m < N; m++) b[m] = a.src0[(f0 + m) * fs + ib];
#pragma unroll
    for (int m = 0; m < N; m++) {
      const long long o = (f0 + m) * fs + ib;
      a.out0[o] = fmaf(a.a_dtf, rhs[m], b[m]);
      if (a.ksum64)
        a.ksum64[o] = a.mode == MODE_FIRST ? (double)rhs[m] : fma(2.0, (double)rhs[m], kd[m]);
      else
        a.ksum[o] = a.mode == MODE_FIRST ? rhs[m] : fmaf(2.0f, rhs[m], ks[m]);
    }
  }
}

// every field in one thread (the batched boundary kernel)
__device__ __forceinline__ void sommerfeld_point_mixed_all(const Grid& g, const StageArgsMixed& a,
                                                           const float* __restrict__ kanchor, unsigned q) {
  sommerfeld_point_mixed_fields<0, NF, false>(g, a, kanchor, q);
}

// Periodic ghosts: copy from the wrapped interior point, all fields (and the
// float64 W array of a mixed stage buffer when w is non-null).
template <typename S>
__device__ __forceinline__ void periodic_point(const Grid& g, S* __restrict__ y,
                                               double* __restrict__ w, unsigned q) {
  int i, j, k;
  ghost_decode(g, q, i, j, k);
  const int si = GH + ((i - GH) % g.n0 + g.n0) % g.n0;
  const int sj = GH + ((j - GH) % g.n1 + g.n1) % g.n1;
  const int sk = GH + ((k - GH) % g.n2 + g.n2) % g.n2;
  const long long d = lin(g, i, j, k), s = lin(g, si, sj, sk);
  // every load of a group before its stores
  constexpr int N = 8;
#pragma unroll
  for (int f0 = 0; f0 < NF; f0 += N) {
    S v[N];
#pragma unroll
    for (int n = 0; n < N; n++) v[n] = y[(f0 + n) * g.fstride + s];
#pragma unroll
    for (int n = 0; n < N; n++) y[(f0 + n) * g.fstride + d] = v[n];
  }
  if (w) w[d] = w[s];
}

}  // namespace bssn
