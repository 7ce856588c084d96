// Instantiation unit of the tensor-core decode kernel: 2 hidden layer(s), split FP16 operands (hi + lo pairs), FP32 output.
#include "tc_kernel.cuh"

namespace nbtc {

nbtc_status launch_tc_h2_f32s(const TcArgs& p, int W, int slots, int grid, cudaStream_t s) {
  if (p.mode == kModeInPlace) return launch_tc_w<2, kF32Split, 4, kModeInPlace, 1, true>(p, grid, s);  // FP32 decodes
  if (p.tmem_a && W == 4 && slots == 1)  // A operands in TMEM
    return launch_tc_w<2, kF32Split, 4, kModeSingle, 1, true>(p, grid, s);
  if (W == 4 && slots == 1) return launch_tc_w<2, kF32Split, 4, kModeSingle, 1>(p, grid, s);
  return fail(NBTC_ERR_UNSUPPORTED, "FP32-output split decode runs 4 warpgroups x 1 slot");
}

}  // namespace nbtc
