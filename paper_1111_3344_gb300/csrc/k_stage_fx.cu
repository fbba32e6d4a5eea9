// Float64 fused stage in tiles (rhs_fx_tile.cuh): one block per tile of 8 x 4 x 4
// interior points, one thread per point.
//
// Bound: the float64 pipe (869 instructions of 64 cycles for a warp's
// points), the integer stencils beside it.  Shape and occupancy: six blocks of 128
// threads per SM (80 registers, 33 KB of shared memory each).  A step at 128^3
// 15.8 ms; one point at a time 20, before that with float64 stencils 33.1.
// Found with slightly cheaper sums (a stage then 3.51-3.65 ms): with 4, 5, 7, 8
// blocks 4.1, 3.8, 3.6, 3.7; tiles of 16 x 4 x 2 3.65, 16 x 2 x 4 3.68, 8 x 8 x 2
// 3.60, 8 x 8 x 4 3.95, 32 x 2 x 2 4.4 (a flatter tile converts more box points per
// tile point); one point at a time (k_stage.cu) 4.6.
//
// The waits for the tensor loads are bounded: a block whose wait runs out sets
// the error word (read back by the host as BSSN_ETIMEOUT), waits once more,
// boundedly, for its own copy, and returns without writing results.  (A test hook
// leaves out one copy and polls a given number of times.)
#include "rhs_fx_tile.cuh"
#include "stage_point.cuh"

namespace bssn {

using FxT = FxTile<8, 4, 4>;

__global__ void __launch_bounds__(FxT::THREADS, 6)
    stage_fx_kernel(const __grid_constant__ CUtensorMap map, Grid g, StageArgs a, int* __restrict__ err) {
  __shared__ FxShared<FxT> sm;
  const int tid = threadIdx.x;
  const int ii0 = blockIdx.x * FxT::TX, jj0 = blockIdx.y * FxT::TY, kk0 = blockIdx.z * FxT::TZ;
  const int ii = ii0 + tid % FxT::TX, jj = jj0 + tid / FxT::TX % FxT::TY, kk = kk0 + tid / (FxT::TX * FxT::TY);
  // threads past the grid work on the nearest point inside it; their results are dropped
  const int i = min(ii, g.n0 - 1) + GH, j = min(jj, g.n1 - 1) + GH, k = min(kk, g.n2 - 1) + GH;
  double r[NF];
  if (!rhs_fx_tile<FxT>(&map, g, a.src, sm, tid, ii0, jj0, kk0, i, j, k, r, fx_stall_round(a, 0), a.stall_polls)) {
    if (tid == 0) atomicExch(err, 1);
    return;
  }
  if (ii < g.n0 && jj < g.n1 && kk < g.n2) combine_fp64(g, a, lin(g, i, j, k), ii, jj, kk, r);
}

// ------------------------------------------------------------ few tiles
// With one tile per SM (or a few) a stage takes one block's latency, in which
// each sub-partition has a single warp: some 200 thousand cycles, the float64
// pipe busy for 55 of them.  Here GROUPS groups of threads share the tile's
// fields: each brings and converts its own boxes (barriers of its own), the
// results meet in shared memory, and the first group does the algebra -- the
// Ricci tensor and the lapse terms while the others finish the fields: 108
// thousand cycles.  One block of 512 threads per SM (128 registers, 205 KB of
// shared memory).
constexpr int GROUPS = 4;
template <typename Sh>
struct FxWideShared {
  alignas(128) long long box[GROUPS][2][(Sh::BOX + 15) / 16 * 16];
  unsigned long long bar[GROUPS][2];
  double wt[10][Sh::THREADS];
  double slot[77][Sh::THREADS];  // of fx_stencils: gt_ij 0 (4 each), Gt^i 24 (3), phi|W, alpha 33 (10), beta^i 53 (7), K 74
  double out[NF][Sh::THREADS];
  int neg[Sh::THREADS];  // signs of beta
  unsigned top[GROUPS][Sh::WARPS];
  int fail;
};
// barrier of n threads with the conjunction of p
__device__ __forceinline__ bool group_and(int id, int n, bool p) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred q, %2, %3, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((unsigned)p), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

__global__ void __launch_bounds__(GROUPS * FxT::THREADS, 1)
    stage_fx_wide_kernel(const __grid_constant__ CUtensorMap map, Grid g, StageArgs a, int* __restrict__ err) {
  using Sh = FxT;
  extern __shared__ __align__(128) unsigned char raw[];
  FxWideShared<Sh>& sm = *reinterpret_cast<FxWideShared<Sh>*>(raw);
  constexpr int T = Sh::THREADS;
  const int grp = threadIdx.x / T, tid = threadIdx.x % T;
  const int ii0 = blockIdx.x * Sh::TX, jj0 = blockIdx.y * Sh::TY, kk0 = blockIdx.z * Sh::TZ;
  const int ii = ii0 + tid % Sh::TX, jj = jj0 + tid / Sh::TX % Sh::TY, kk = kk0 + tid / (Sh::TX * Sh::TY);
  const int i = min(ii, g.n0 - 1) + GH, j = min(jj, g.n1 - 1) + GH, k = min(kk, g.n2 - 1) + GH;
  const long long fs = g.fstride, id = lin(g, i, j, k);
  const double* c0 = a.src + id;
  const int nf = g.shift == BSSN_SHIFT_FROZEN ? F_BETA : NF;
  const unsigned bar0 = smem_addr(&sm.bar[grp][0]), bar1 = smem_addr(&sm.bar[grp][1]);
  if (tid == 0) {
    mbar_init(bar0);
    mbar_init(bar1);
    if (grp == 0) sm.fail = 0;
  }
  const int cen = fx_center<Sh>(ii0, jj0, kk0, i, j, k);
  int* sc = reinterpret_cast<int*>(sm.box[grp][1]) + tid;
  fx_points<Sh>(g, tid, ii0, jj0, kk0, cen, sc);
  const int stall = fx_stall_round(a, grp);
  after_previous();
  if (tid == 0 && stall != 0) fx_issue<Sh>(&map, sm.box[grp][0], bar0, ii0, jj0, kk0, fx_field(grp));
  FxMetric M;  // the first group's
  if (grp == 0) {
    int neg[3];
    fx_metric(g, c0, M);
    const bool ok = fx_tile_weights<Sh>(g, c0, M, &sm.wt[0][tid], neg);
    sm.neg[tid] = (neg[0] & 1) | (neg[1] & 2) | (neg[2] & 4) | (ok ? 8 : 0);
  }
  int at[Sh::PER];
#pragma unroll
  for (int e = 0; e < Sh::PER; e++) at[e] = sc[e * T];
  __syncthreads();  // the weights and barriers are there
  const int sg = sm.neg[tid];
  const bool wok = sg & 8;
  const int neg[3] = {-(sg & 1), -(sg >> 1 & 1), -(sg >> 2 & 1)};
  auto S = [&](int n) -> double& { return sm.slot[n][tid]; };
  const double* wt = &sm.wt[0][tid];

  double X[6], G2[3][6], V2[3], vj[3], lap = 0.0;
  // rounds 0-2: fields 0 .. 11, one per group; then the first group does the
  // algebra that these fields allow and the others the remaining 12 fields
#pragma unroll 1
  for (int rd = 0; rd < 7; rd++) {
    if (rd == 3) {
      __syncthreads();
      if (grp == 0) break;
    }
    const int q = rd < 3 ? GROUPS * rd + grp : 11 + grp + (GROUPS - 1) * (rd - 3);
    const int order = fx_order(q), up = fx_up(q);
    const int s0 = q < 6 ? 4 * q : (q < 9 ? 3 * q + 6 : (q < 11 ? 10 * q - 57 : (q < 14 ? 7 * q - 24 : 74)));
    long long* box = sm.box[grp][rd & 1];
    const long long* c = box + cen;
    const unsigned bar = rd & 1 ? bar1 : bar0;
    const bool there = mbar_wait(bar, (rd >> 1) & 1, rd == stall ? a.stall_polls : WAIT_LIMIT);
    double x[Sh::PER];
#pragma unroll
    for (int e = 0; e < Sh::PER; e++) x[e] = __longlong_as_double(box[at[e]]);
    const unsigned wtop = __reduce_max_sync(0xffffffffu, fx_top(x));
    if ((tid & 31) == 0) sm.top[grp][tid >> 5] = wtop;
    if (!group_and(1 + grp, T, there)) {
      // the group's one copy in flight lands before the block exits
      if (rd != stall) mbar_wait(bar, (rd >> 1) & 1, WAIT_LIMIT);
      sm.fail = 1;
      if (rd < 3) __syncthreads();
      break;
    }
    const int next = rd + 1 < 3 ? q + GROUPS : (rd == 2 ? (grp ? 11 + grp : NF) : q + GROUPS - 1);
    if (tid == 0 && next < NF && rd + 1 != stall)
      fx_issue<Sh>(&map, sm.box[grp][(rd + 1) & 1], rd & 1 ? bar0 : bar1, ii0, jj0, kk0, fx_field(next));
    unsigned top = sm.top[grp][0];
#pragma unroll
    for (int n = 1; n < Sh::WARPS; n++) top = max(top, sm.top[grp][n]);
    bool ok = fx_ok(top);
    if (top == 0) {
      unsigned lo = 0;
#pragma unroll
      for (int e = 0; e < Sh::PER; e++) lo |= (unsigned)__double2loint(x[e]);
      ok = group_and(1 + grp, T, lo == 0);
    }
    const int E = max((int)(top >> 20), 256) + FX_BITS - FX_TILE_BITS;
    if (ok) {
#pragma unroll
      for (int e = 0; e < Sh::PER; e++) box[at[e]] = fx_near<FX_TILE_BITS>(x[e], E + FX_TILE_BITS - FX_BITS);
    }
    group_and(1 + grp, T, true);
    const int f = fx_field(q);
    double r = 0.0;
    bool near = false;
    if (ok) r = fx_stencils<Sh>(c, q, order, up, E, wt, neg, S, s0, near);
    if (!(near && wok) && !(ok && top == 0))
      r = fx_stencils_own<Sh>(c0, fs, g.pitch, g.plane, g.i12h, g.kos, q, order, up, wt, S, s0);
    sm.out[f][tid] = f < nf ? r : 0.0;
  }
  if (grp == 0) {
    fx_ricci(g, M, [&](int d, int m) { return S(4 * m + d); }, [&](int m) { return S(4 * m + 3); },
             [&](int a, int d) { return S(24 + 3 * a + d); }, X, G2, V2);
    double dchi[3], dalp[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      dchi[d] = S(33 + d);
      dalp[d] = S(43 + d);
    }
    fx_lapse(g, M, __ldg(c0 + F_ALP * fs), dchi, dalp, S(46), [&](int m) { return S(37 + m); },
             [&](int m) { return S(47 + m); }, G2, X, lap, vj);
  }
  __syncthreads();
  if (sm.fail) {
    if (threadIdx.x == 0) atomicExch(err, 1);
    return;
  }
  struct Out {
    double* p;
    __device__ __forceinline__ double& operator[](int f) const { return p[f * T]; }
  };
  if (grp == 0)
    fx_assemble(g, c0, id, i, j, k, M, [&](int b, int d) { return S(53 + 7 * b + d); },
                [&](int b) { return S(56 + 7 * b); }, [&](int b, int m) { return S(57 + 7 * b + m); },
                [&](int d) { return S(74 + d); }, G2, V2, vj, X, lap, Out{&sm.out[0][tid]});
  __syncthreads();
  if (ii >= g.n0 || jj >= g.n1 || kk >= g.n2) return;
  const bool anchor = a.mode != MODE_RHS && a.kshell && on_shell(g, ii, jj, kk);
  constexpr int N = NF / GROUPS;
  long long o[N];
  double r[N];
#pragma unroll
  for (int n = 0; n < N; n++) {
    o[n] = (n * GROUPS + grp) * fs + id;
    r[n] = sm.out[n * GROUPS + grp][tid];
  }
  combine_point_fp64(a, o, r, anchor);
}

// (and the shared-memory limit of the kernel that may read through the map, so
// that launches under capture need no other call)
cudaError_t make_fx_tensor_map(const Grid& g, const double* base, CUtensorMap* out) {
  static std::atomic<unsigned> done{0};
  const cudaError_t e = smem_optin(stage_fx_wide_kernel, sizeof(FxWideShared<FxT>), done);
  if (e != cudaSuccess) return e;
  return encode_tensor_map(g, base, 8, FxT::BX, FxT::BY, FxT::BZ, out);
}

// Up to three tiles per SM one after another: ms a stage with groups, without:
// 24^3 (108 tiles) 0.053 / 0.100, 32^3 (256) 0.099 / 0.133, 36^3 (405) 0.148 / 0.162,
// 40^3 (500) 0.196 / 0.187.
constexpr long long FX_WIDE_BLOCKS = 3 * 152;
static long long fx_tiles(const Grid& g) {
  return (long long)((g.n0 + FxT::TX - 1) / FxT::TX) * ((g.n1 + FxT::TY - 1) / FxT::TY) *
         ((g.n2 + FxT::TZ - 1) / FxT::TZ);
}
bool fx_launch_early(const Grid& g) { return fx_tiles(g) <= 2 * 152; }

// A tile takes as long with points past the grid as without, 0.75 of the time
// of the same points one at a time (k_stage.cu: blocks of consecutive points, no
// padding).  Measured, ms a stage, tile against point form, with the share of
// threads that have a point: 121^3 0.90 3.18 / 3.71; 73^3 0.84 0.808 / 0.867; 50^3
// 0.83 0.310 / 0.334; 41^3 0.74 0.197 / 0.209; 33^3 0.69 0.157 / 0.145; 9 x 200 x
// 200 0.56 1.11 / 0.97: tiles from 0.72 on.  (On smooth data; while a puncture's
// fields still fall off steeply and many points take their own alignment 3.34,
// 0.889, 0.363, 0.248.)
// With few tiles one block's latency counts, whatever the padding (129 x 5 x 5
// 0.052 / 0.144, 33^3 with groups 0.144 / 0.147).
bool fx_tile_fits(const Grid& g) {
  return fx_tiles(g) <= FX_WIDE_BLOCKS || 100LL * g.n0 * g.n1 * g.n2 >= 72LL * fx_tiles(g) * FxT::THREADS;
}

cudaError_t launch_stage_fx(const Grid& g, const StageArgs& a, const CUtensorMap& map, int* err, cudaStream_t s) {
  const dim3 grid((g.n0 + FxT::TX - 1) / FxT::TX, (g.n1 + FxT::TY - 1) / FxT::TY, (g.n2 + FxT::TZ - 1) / FxT::TZ);
  if (fx_tiles(g) <= FX_WIDE_BLOCKS) {
    return launch_after(stage_fx_wide_kernel, grid, GROUPS * FxT::THREADS, sizeof(FxWideShared<FxT>), s,
                        fx_launch_early(g), map, g, a, err);
  }
  stage_fx_kernel<<<grid, FxT::THREADS, 0, s>>>(map, g, a, err);
  return cudaGetLastError();
}

}  // namespace bssn
