// Float64 fused stage in tiles (rhs_fx_tile.cuh): one block per tile of 8 x 4 x 4
// interior points, one thread per point.
//
// Bound: the float64 pipe (860 instructions of 64 cycles for a warp's points:
// 55 thousand of the 68 thousand cycles a sub-partition takes), the integer
// stencils beside it.  Shape and occupancy: six blocks of 128 threads per SM (80
// registers, 33 KB of shared memory each).  A stage at 128^3: 3.51-3.65 ms (a
// step 15.1; one point at a time 19.7, before that with float64 stencils 33.1);
// with 4, 5, 7, 8 blocks 4.1, 3.8, 3.6, 3.7; tiles of 16 x 4 x 2 3.65, 16 x 2 x 4
// 3.68, 8 x 8 x 2 3.60, 8 x 8 x 4 3.95, 32 x 2 x 2 4.4 (a flatter tile converts
// more box points per tile point); one point at a time (k_stage.cu) 4.6.
//
// The waits for the tensor loads are bounded: a block whose wait runs out sets
// the error word (read back by the host as BSSN_ETIMEOUT), waits once more,
// boundedly, for its own copy, and returns without writing results.
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
  if (!rhs_fx_tile<FxT>(&map, g, a.src, sm, tid, ii0, jj0, kk0, i, j, k, r)) {
    if (tid == 0) atomicExch(err, 1);
    return;
  }
  if (ii < g.n0 && jj < g.n1 && kk < g.n2) combine_fp64(g, a, lin(g, i, j, k), ii, jj, kk, r);
}

cudaError_t make_fx_tensor_map(const Grid& g, const double* base, CUtensorMap* out) {
  return encode_tensor_map(g, base, 8, FxT::BX, FxT::BY, FxT::BZ, out);
}

// A tile takes as long with points past the grid as without, 0.73 of the time
// of the same points one at a time (k_stage.cu: blocks of consecutive points, no
// padding).  Measured, ms a stage, tile against point form, with the share of
// threads that have a point: 121^3 0.90 3.23 / 4.23; 41^3 0.74 0.210 / 0.222;
// 33^3 0.69 0.157 / 0.145; 9 x 200 x 200 0.56 1.11 / 0.97: tiles from 0.72 on.
// Where every block has an SM to itself one block's latency counts, whatever
// the padding: 17^3 0.097 / 0.138, 129 x 5 x 5 0.098 / 0.141.
bool fx_tile_fits(const Grid& g) {
  const long long blocks = (long long)((g.n0 + FxT::TX - 1) / FxT::TX) * ((g.n1 + FxT::TY - 1) / FxT::TY) *
                           ((g.n2 + FxT::TZ - 1) / FxT::TZ);
  return blocks <= 152 || 100LL * g.n0 * g.n1 * g.n2 >= 72LL * blocks * FxT::THREADS;
}

cudaError_t launch_stage_fx(const Grid& g, const StageArgs& a, const CUtensorMap& map, int* err, cudaStream_t s) {
  const dim3 grid((g.n0 + FxT::TX - 1) / FxT::TX, (g.n1 + FxT::TY - 1) / FxT::TY, (g.n2 + FxT::TZ - 1) / FxT::TZ);
  stage_fx_kernel<<<grid, FxT::THREADS, 0, s>>>(map, g, a, err);
  return cudaGetLastError();
}

}  // namespace bssn
