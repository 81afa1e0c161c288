// Double-gyre advection instantiations (2D).
#include "advect_inst.cuh"

#include "capi_internal.cuh"

namespace ftle {

template <int N, bool C>
static void launch_dg_n(bool coord64, const AdvArgs& a, const NodeShape& S, size_t smem, cudaStream_t stream) {
  if constexpr (C) {
    if (coord64)
      k_advect_dg<N, double><<<S.grid, S.block, smem, stream>>>(a);
    else
      k_advect_dg<N, float><<<S.grid, S.block, smem, stream>>>(a);
  } else {
    if (coord64)
      k_advect_dg32<N, double><<<S.grid, S.block, smem, stream>>>(a);
    else
      k_advect_dg32<N, float><<<S.grid, S.block, smem, stream>>>(a);
  }
}

// Measured at T = 15 (1500 steps) on 152 SMs: 64 x 32 and 128 x 64 nodes 170 us with one node per thread
// (two warps a block 178, eight 246), 237-242 with two; 256 x 128: 242 us, one node per thread 248-256;
// 512 x 256: 832 us in two blocks per SM, 925 with one node per thread; 700 x 350: 1467 us in blocks of
// four warps, 1635 of eight; 2048 x 1024: 10.93 ms in blocks of eight, 11.01 of four, 12.07 with one
// node per thread.
int launch_advect_dg_carry(bool coord64, const AdvArgs& a, int block, int blocks_per_sm, cudaStream_t stream) {
  const NodeShape S = node_shape(a.n, block, blocks_per_sm, 49);
  const size_t smem = advect_smem_bytes(FTLE_FLOW_DOUBLE_GYRE, P32C, a.nsteps);
  if (S.two)
    launch_dg_n<2, true>(coord64, a, S, smem, stream);
  else
    launch_dg_n<1, true>(coord64, a, S, smem, stream);
  FTLE_LAUNCH_CHECK("k_advect_dg launch");
  return FTLE_OK;
}

int launch_advect_dg32(bool coord64, const AdvArgs& a, int block, int blocks_per_sm, cudaStream_t stream) {
  const NodeShape S = node_shape(a.n, block, blocks_per_sm, 49);
  const size_t smem = advect_smem_bytes(FTLE_FLOW_DOUBLE_GYRE, P32, a.nsteps);
  if (S.two)
    launch_dg_n<2, false>(coord64, a, S, smem, stream);
  else
    launch_dg_n<1, false>(coord64, a, S, smem, stream);
  FTLE_LAUNCH_CHECK("k_advect_dg32 launch");
  return FTLE_OK;
}

int launch_advect_dg(int prec, int out, bool coord64, const AdvArgs& args, int grid, int block,
                     size_t smem, cudaStream_t stream) {
  return launch_advect_kind<FTLE_FLOW_DOUBLE_GYRE, 2>(prec, out, coord64, args, grid, block, smem, stream);
}
}  // namespace ftle
