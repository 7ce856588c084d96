// Instantiation unit of the tensor-core decode kernel, batched materials / frame: 3 hidden layer(s), FP16 operands.
#include "tc_kernel.cuh"

namespace nbtc {

nbtc_status launch_tc_h3_f16_batch(const TcArgs& p, int W, int slots, int grid, cudaStream_t s) {
  if (W != 4 || slots != 1) return fail(NBTC_ERR_UNSUPPORTED, "the batched decode runs 4 warpgroups x 1 slot");
  return p.mode == kModeFrame ? launch_tc_w<3, kF16, 4, kModeFrame, 1, true>(p, grid, s)
                              : launch_tc_w<3, kF16, 4, kModeBatch, 1, true>(p, grid, s);
}

}  // namespace nbtc
