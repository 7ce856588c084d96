// FP32 decode: which kernel takes an MLP's shape.
#include "host.h"

namespace nbtc {

nbtc_status launch_decode_fp32_tile(nbtc_context* ctx, const DecodeArgs& a, const nbtc_mlp* mlp, cudaStream_t s);

nbtc_status launch_decode_fp32(nbtc_context* ctx, const DecodeArgs& a, const nbtc_mlp* mlp, bool host_out,
                               cudaStream_t s) {
  // hidden width 64: split operands on the tensor cores (FP32 accuracy); widths 16
  // and 32: the tiled GEMM kernel
  nbtc_status st = launch_decode_fp32_tc(ctx, a, mlp, host_out, s);
  if (st != NBTC_ERR_UNSUPPORTED) return st;
  st = launch_decode_fp32_tile(ctx, a, mlp, s);
  if (st != NBTC_ERR_UNSUPPORTED) return st;
  if (mlp->dims[0] != 12) return fail(NBTC_ERR_UNSUPPORTED, "decode kernels take 12 input features");
  for (int l = 1; l < mlp->num_layers; ++l)
    if (mlp->dims[l] != mlp->dims[1]) return fail(NBTC_ERR_UNSUPPORTED, "hidden layers must share one width");
  return fail(NBTC_ERR_UNSUPPORTED, "no FP32 kernel for this MLP shape");
}

}  // namespace nbtc
