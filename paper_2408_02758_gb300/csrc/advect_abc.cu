// ABC-flow advection instantiations (3D).
#include "advect_inst.cuh"
#include "capi_internal.cuh"

namespace ftle {

template <int N>
static int launch_abc_n(bool coord64, const AdvArgs& a, int grid, int block, cudaStream_t stream) {
  if (coord64)
    k_advect_abc<N, double><<<grid, block, 0, stream>>>(a);
  else
    k_advect_abc<N, float><<<grid, block, 0, stream>>>(a);
  FTLE_LAUNCH_CHECK("k_advect_abc launch");
  return FTLE_OK;
}

// Nodes per thread and launch shape as for the double gyre (launch_advect_dg_carry), 500 steps on 152 SMs:
// one node per thread up to one warp per SM sub-partition (16^3 and 26 x 27 x 25 nodes: 47 us, 74-76 in
// blocks of eight warps); then two (32 x 33 x 34: 68 us against 74), in two blocks per SM of equal size
// while they fit at once (61 x 47 x 53: 240 us, one node per thread 274), beyond that in blocks of four
// warps (96^3: 1350 us, 1410 in blocks of eight; 256^3: 25.2 ms either way, 28.5 with one node per thread).
int launch_advect_abc_carry(bool coord64, const AdvArgs& a, int block, int blocks_per_sm, cudaStream_t stream) {
  const int64_t sms = device_sm_count() > 0 ? device_sm_count() : 1;
  const bool two = a.n > sms * 4 * 32;
  const int64_t tile = two ? 64 : 32, tiles = (a.n + tile - 1) / tile;
  int64_t warps = block / 32, cap = blocks_per_sm > 0 ? sms * blocks_per_sm : (int64_t)INT32_MAX;
  if (block == 0) {
    const int64_t per_sm = (tiles + sms - 1) / sms, resident = 8 * kAbcBlocks<2>;
    if (!two)
      warps = 4;
    else if (per_sm <= resident)
      warps = (per_sm + kAbcBlocks<2> - 1) / kAbcBlocks<2>;
    else
      warps = 4;
  }
  const int64_t need = (tiles + warps - 1) / warps;
  const int grid = (int)(need < cap ? need : cap);
  return two ? launch_abc_n<2>(coord64, a, grid, 32 * (int)warps, stream)
             : launch_abc_n<1>(coord64, a, grid, 32 * (int)warps, stream);
}

int launch_advect_abc(int prec, int out, bool coord64, const AdvArgs& args, int grid, int block,
                      size_t smem, cudaStream_t stream) {
  return launch_advect_kind<FTLE_FLOW_ABC, 3>(prec, out, coord64, args, grid, block, smem, stream);
}
}  // namespace ftle
