// Double-gyre advection instantiations (2D).
#include "advect_inst.cuh"

#include "capi_internal.cuh"

namespace ftle {

template <int N>
static int launch_dg_n(bool coord64, const AdvArgs& a, int grid, int block, size_t smem, cudaStream_t stream) {
  if (coord64)
    k_advect_dg<N, double><<<grid, block, smem, stream>>>(a);
  else
    k_advect_dg<N, float><<<grid, block, smem, stream>>>(a);
  FTLE_LAUNCH_CHECK("k_advect_dg launch");
  return FTLE_OK;
}

// Nodes per thread and launch shape, measured at T = 15 (1500 steps) on 152 SMs:
//   up to one warp per SM sub-partition (19,456 nodes): one node per thread, which has the shorter
//   chain per step (64 x 32 and 128 x 64 nodes: 170 us against 237-242 with two), in blocks of four
//   warps, one on each sub-partition (two warps a block: 178, eight: 246);
//   while two nodes per thread fit at once (16 warps per SM, 155,648 nodes): two blocks per SM of
//   equal size, so that the SMs differ by a warp (256 x 128: 242 us, one node per thread 248-256;
//   512 x 256: 832 us in blocks of eight warps, 925 with one node per thread);
//   beyond that blocks of eight warps, each its own tiles (2048 x 1024: 10.93 ms, one node per
//   thread 12.07); up to three rounds of them, blocks of four warps, which even out the last round
//   (700 x 350: 1467 us against 1635).
int launch_advect_dg_carry(bool coord64, const AdvArgs& a, int block, int blocks_per_sm, cudaStream_t stream) {
  const int64_t sms = device_sm_count() > 0 ? device_sm_count() : 1;
  const size_t smem = advect_smem_bytes(FTLE_FLOW_DOUBLE_GYRE, P32C, a.nsteps);
  const bool two = a.n > sms * 4 * 32;
  const int64_t tile = two ? 64 : 32, tiles = (a.n + tile - 1) / tile;
  int64_t warps = block / 32, cap = blocks_per_sm > 0 ? sms * blocks_per_sm : (int64_t)INT32_MAX;
  if (block == 0) {
    const int64_t per_sm = (tiles + sms - 1) / sms, resident = 8 * kDgBlocks<2>;
    if (!two)
      warps = 4;
    else if (per_sm <= resident)
      warps = (per_sm + kDgBlocks<2> - 1) / kDgBlocks<2>;
    else
      warps = per_sm <= 3 * resident ? 4 : 8;
  }
  const int64_t need = (tiles + warps - 1) / warps;
  const int grid = (int)(need < cap ? need : cap);
  return two ? launch_dg_n<2>(coord64, a, grid, 32 * (int)warps, smem, stream)
             : launch_dg_n<1>(coord64, a, grid, 32 * (int)warps, smem, stream);
}

int launch_advect_dg(int prec, int out, bool coord64, const AdvArgs& args, int grid, int block,
                     size_t smem, cudaStream_t stream) {
  return launch_advect_kind<FTLE_FLOW_DOUBLE_GYRE, 2>(prec, out, coord64, args, grid, block, smem, stream);
}
}  // namespace ftle
