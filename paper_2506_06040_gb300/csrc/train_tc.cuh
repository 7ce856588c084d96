// Tensor-core training kernel (included by train.cu after the shared training
// definitions): the step's MLP products -- forward, backward and weight
// gradients -- on tcgen05 with split FP16 operands (hi + lo, three products
// per GEMM, FP32 accumulation in TMEM), which keeps FP32-level accuracy.
//
// Sixteen warps per CTA.  Warps 0..7 are two warpgroups, one thread per sample of a
// 128-sample tile, whose first warp issues their MMAs; warps 8..11 and 12..15 finish
// the tiles of one warpgroup each (a warp of either owns one lane quarter of TMEM).
// Per tile, six phases (operands in shared memory -> MMAs -> mbarrier):
//   1  X (features + a ones column)    F1: Z1 = X W1^T + b1               (D)
//   2  H1 = relu(Z1)                    F2: Z2 = H1 W2^T + b2              (D)
//   3  H2 = relu(Z2)                    F3: Y  = H2 W3^T + b3              (D)
//   4  G = dL/dy, unscaled (2 r; L1: sign r)
//                                       B1: dH2 = G W3 (D);  G3 += H2^T G
//   5  dZ2 = dH2 [Z2 > 0]  (over H2)    B2: dH1 = dZ2 W2 (D); G2 += dZ2^T H1, G2b += dZ2^T 1
//   6  dZ1 = dH1 [Z1 > 0]  (over H1)    B3: dX = dZ1 W1 (DX); G1 += dZ1^T X
// What bounds the kernel is this chain, two of them an SM (shared memory holds no
// third), so everything that need not be in it is out of it: the next tile's record
// is loaded and split into the other X buffer while B1 runs; a warpgroup hands phase
// 6 over and goes on to its next tile; dX (times the loss scale) is scattered into
// the latent gradients, and the tile's weight gradients are added to the running
// sums, by the finishing warps meanwhile.  A tile took 26.8k cycles with all of it in the
// chain, now 20.8k (shared memory, whose bandwidth MMA operands, tile stores and the
// atomics share, is busy 70% of it); a step at 2^20 samples 612 us,
// now 497 (the small launches around the kernel included in both).
//
// The weight-gradient products reduce over the tile's samples: their operands are
// the same shared-memory tiles read MN-major (the instruction's transpose bits),
// M = 64 (rows in the first 16 lanes of each warp's TMEM quarter).  The G
// accumulators start afresh each tile (a 128-sample sum) and are added to the
// warpgroup's running FP32 sums in the other 16 lanes of each quarter of the same
// columns -- an accumulator chain over all of a warpgroup's samples would lose FP32
// accuracy as it grows.  At the end the running sums are scaled, the two warpgroups
// added (with the rounding error kept as the compensation) and written as the CTA's
// partial sums.  The loss and db3 use compensated per-thread sums (two-sum) and a
// fixed-order CTA reduction.
#pragma once

#include <type_traits>

#include "sm100.cuh"

namespace nbtc {

namespace ttc {

// ---- shared-memory plan (bytes from a 1024-aligned base)
// weight images (K-major unless noted; SW32 = 32-byte rows, SW128 = 128-byte rows)
constexpr int oW1H = 0, oW1L = 2048;          // [64 out][16 in] SW32, hi / lo
constexpr int oBT1 = 4096;                    // [64][16] SW32: column 0 hi(b1), 1 lo(b1)
constexpr int oW3TH = 6144, oW3TL = 8192;     // W3^T [64 hidden][16 channel] SW32
constexpr int oONES = 10240;                  // [128][16] SW32: columns 0 and 1 = 1
constexpr int oBT3 = 14336;                   // [16][16] SW32: b3
constexpr int oBT2 = 15360;                   // [64][16] SW32: b2
constexpr int oW2H = 17408, oW2L = 25600;     // [64 out][64 in] SW128
constexpr int oW3H = 33792, oW3L = 35840;     // [16 channel][64 in] SW128
constexpr int oW1TH = 37888, oW1TL = 39936;   // W1^T [16 feature][64 hidden] SW128
constexpr int oTiles = 41984;
// per warpgroup
constexpr int kTileBytes = 90112;
constexpr int oX = 0, kX = 8192;              // two buffers of [128][16] SW32, hi at 0, lo at 4096
constexpr int oDYH = 16384, oDYL = 20480;     // [128][16] SW32
constexpr int oH1H = 24576, oH1L = 40960, oH2H = 57344, oH2L = 73728;  // [128][64] SW128
constexpr int kWG = 2;
constexpr int kThreads = 512;
constexpr int oBars = oTiles + kWG * kTileBytes;  // D-ready[2], tile-done[2], G-ready[2]
constexpr int oTslot = oBars + 48;
constexpr int kSmem = oTslot + 16 + 1024;
// registers: 512 threads launch with 128 each; 256 x 176 + 256 x 80 is the same total
constexpr int kRegsLaunch = 128, kRegsMain = 176, kRegsFinish = 80;
static_assert(kRegsMain + kRegsFinish == 2 * kRegsLaunch && kThreads * kRegsLaunch == 65536, "register split");
// TMEM columns per warpgroup (base g * 256)
constexpr uint32_t cD = 0, cG2 = 64, cG2b = 128, cG3 = 144, cG1 = 160, cDX = 176;
// Named barriers (0 is __syncthreads), each per warpgroup: its operands are in place,
// and the previous tile's gradients are out of the G accumulators.
__device__ __forceinline__ int bar_a(int g) { return 1 + g; }
__device__ __forceinline__ int bar_folded(int g) { return 3 + g; }

__device__ __forceinline__ uint32_t sw32(int row, int kbyte) {
  return (uint32_t)((row >> 3) * 256 + (row & 7) * 32 + ((((kbyte >> 4) ^ ((row & 7) >> 2)) & 1) << 4) +
                    (kbyte & 15));
}
__device__ __forceinline__ uint32_t sw128(int row, int kbyte) {
  return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((((kbyte >> 4) ^ (row & 7)) & 7) << 4) + (kbyte & 15));
}
__device__ __forceinline__ void st_half(unsigned char* s, uint32_t off, float v) {
  *reinterpret_cast<__half*>(s + off) = __float2half_rn(v);
}
// hi / lo halves of one FP32 value (hi = RN16(v), lo = RN16(v - hi))
__device__ __forceinline__ void put_split(unsigned char* s, uint32_t oh, uint32_t ol, float v) {
  uint32_t h, l;
  sm100::split_f16x2(v, 0.f, h, l);
  *reinterpret_cast<uint16_t*>(s + oh) = (uint16_t)(h & 0xFFFF);
  *reinterpret_cast<uint16_t*>(s + ol) = (uint16_t)(l & 0xFFFF);
}

}  // namespace ttc

// CP: channels the per-channel registers are laid out for (12 for C <= 12, else 16).
template <bool LV, int CP>
__global__ void __launch_bounds__(ttc::kThreads, 1) k_train_tc(TrainDev a) {
  using namespace ttc;
  using namespace sm100;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sb = smem_u32(sm);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid / 32, 0), lane = tid % 32;
  const int C = a.C;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + oTslot);

  // ---- weight images from the FP32 MLP (every CTA builds its own)
  for (int e = tid; e < oTiles / 4; e += blockDim.x) reinterpret_cast<uint32_t*>(sm)[e] = 0u;
  if (warp == 0) {
    tmem_alloc(smem_u32(tslot), 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int g = 0; g < 3 * kWG; ++g) mbar_init(sb + oBars + 8 * g, 1);
    fence_mbar_init();
  }
  __syncthreads();
  {
    const float* W1 = a.W;                // [64][12]
    const float* W2 = a.W + kH * kIn;     // [64][64]
    const float* W3 = W2 + kH * kH;       // [C][64]
    const float* b1 = a.B;
    const float* b2 = a.B + kH;
    const float* b3 = a.B + 2 * kH;
    for (int e = tid; e < kH * kIn; e += blockDim.x) {
      const int n = e / kIn, k = e - n * kIn;
      const float w = W1[e];
      put_split(sm, oW1H + sw32(n, 2 * k), oW1L + sw32(n, 2 * k), w);
      put_split(sm, oW1TH + sw128(k, 2 * n), oW1TL + sw128(k, 2 * n), w);
    }
    for (int e = tid; e < kH * kH; e += blockDim.x) {
      const int n = e / kH, k = e - n * kH;
      const float w = W2[e];
      put_split(sm, oW2H + sw128(n, 2 * k), oW2L + sw128(n, 2 * k), w);
    }
    for (int e = tid; e < C * kH; e += blockDim.x) {
      const int c = e / kH, k = e - c * kH;
      const float w = W3[e];
      put_split(sm, oW3H + sw128(c, 2 * k), oW3L + sw128(c, 2 * k), w);
      put_split(sm, oW3TH + sw32(k, 2 * c), oW3TL + sw32(k, 2 * c), w);
    }
    for (int e = tid; e < kH; e += blockDim.x) {
      put_split(sm, oBT1 + sw32(e, 0), oBT1 + sw32(e, 2), b1[e]);
      put_split(sm, oBT2 + sw32(e, 0), oBT2 + sw32(e, 2), b2[e]);
    }
    for (int e = tid; e < C; e += blockDim.x) put_split(sm, oBT3 + sw32(e, 0), oBT3 + sw32(e, 2), b3[e]);
    for (int r = tid; r < 128; r += blockDim.x) {
      st_half(sm, oONES + sw32(r, 0), 1.f);
      st_half(sm, oONES + sw32(r, 2), 1.f);
    }
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  const int64_t tiles = (a.batch + 127) / 128;
  const int64_t stride = (int64_t)gridDim.x * kWG;
  bool failed = false;

  if (warp >= 4 * kWG) {
    // ------------------------------------------------------------ finishing warps
    // warp wq of group g takes the rows (and TMEM lanes) 32 wq .. 32 wq + 31 of
    // warpgroup g's tiles
    regs_dec<kRegsFinish>();
    const int g = (warp - 4 * kWG) / 4, wq = warp & 3;
    const uint32_t d = tmem + (uint32_t)(g * 256) + ((uint32_t)(32 * wq) << 16);
    const uint32_t ebar = sb + oBars + 8 * (kWG + g);
    const int64_t tile0 = (int64_t)blockIdx.x * kWG + g;
    uint32_t eph = 0;
    for (int64_t tile = tile0; tile < tiles; tile += stride) {
      const int64_t sid = tile * 128 + 32 * wq + lane;
      const bool valid = sid < a.batch;
      const float2 uv = valid ? __ldg(reinterpret_cast<const float2*>(a.uv) + sid) : make_float2(0.f, 0.f);
      if (!mbar_wait_bounded(ebar, eph, kDefaultWaitBudget)) {
        failed = true;
        mbar_wait_bounded(ebar, eph, kDrainBudget);
      }
      eph ^= 1u;
      tc_fence_after();
      uint32_t r[16];
      tmem_ld16_wait(d + cDX, r);
      // this tile's G (lanes 0..15 of the quarter, complete with the last commit)
      // into the running sums (lanes 16..31): lane j + 16 adds lane j's value
#pragma unroll 1
      for (int part = 0; part < 7; ++part) {
        const uint32_t col = part < 4 ? cG2 + 16 * part : part == 4 ? cG2b : part == 5 ? cG3 : cG1;
        uint32_t q[16];
        tmem_ld16_wait(d + col, q);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float v = __shfl_up_sync(0xFFFFFFFFu, __uint_as_float(q[j]), 16);
          if (lane >= 16) q[j] = __float_as_uint(tile == tile0 ? v : __uint_as_float(q[j]) + v);
        }
        tmem_st16(d + col, q);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (tile + stride < tiles) named_bar_arrive(bar_folded(g), 160);
      if (valid) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          Taps Tp = clamp_taps(uv.x, uv.y, a.lw[k], a.lh[k], a.shift[k]);
          check_taps(Tp, (int64_t)a.lw[k] * a.lh[k], a);
          float* G = a.lgrad[k];
          const float g0 = a.scale * __uint_as_float(r[3 * k]), g1 = a.scale * __uint_as_float(r[3 * k + 1]),
                      g2 = a.scale * __uint_as_float(r[3 * k + 2]);
          if constexpr (LV) {
            float4* G4 = reinterpret_cast<float4*>(G);
            atomicAdd(G4 + Tp.i00, make_float4(Tp.w00 * g0, Tp.w00 * g1, Tp.w00 * g2, 0.f));
            atomicAdd(G4 + Tp.i10, make_float4(Tp.w10 * g0, Tp.w10 * g1, Tp.w10 * g2, 0.f));
            atomicAdd(G4 + Tp.i01, make_float4(Tp.w01 * g0, Tp.w01 * g1, Tp.w01 * g2, 0.f));
            atomicAdd(G4 + Tp.i11, make_float4(Tp.w11 * g0, Tp.w11 * g1, Tp.w11 * g2, 0.f));
          } else {
            const float gg[3] = {g0, g1, g2};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              atomicAdd(G + 3 * Tp.i00 + c, Tp.w00 * gg[c]);
              atomicAdd(G + 3 * Tp.i10 + c, Tp.w10 * gg[c]);
              atomicAdd(G + 3 * Tp.i01 + c, Tp.w01 * gg[c]);
              atomicAdd(G + 3 * Tp.i11 + c, Tp.w11 * gg[c]);
            }
          }
        }
      }
    }
    // ---- the warpgroup's gradient sums: G2 (dW2), G2b (db2), G3 (dW3^T), G1 (dW1, db1);
    //      row 16 wq + j of the running sums: lane 16 + j of the quarter; stashed as a
    //      [64][64 + 16 + 16 + 16] float block in its own tile area (its last tile's
    //      MMAs are done)
    const int row = 16 * wq + lane - 16;
    const bool has_tiles = tile0 < tiles;
    float* gs = reinterpret_cast<float*>(sm + oTiles + g * kTileBytes);
    for (int part = 0; part < 7; ++part) {
      // columns: G2 0..63 (4 x 16), G2b 64..79, G3 80..95, G1 96..111
      const uint32_t col = part < 4 ? cG2 + 16 * part : part == 4 ? cG2b : part == 5 ? cG3 : cG1;
      uint32_t r[16];
      tmem_ld16_wait(d + col, r);
      if (lane >= 16) {
#pragma unroll
        for (int j = 0; j < 16; ++j) gs[row * 112 + 16 * part + j] = has_tiles ? __uint_as_float(r[j]) * a.scale : 0.f;
      }
    }
    regs_inc<kRegsLaunch>();
  } else {
    // ------------------------------------------------------------ warpgroups
    regs_inc<kRegsMain>();
    const int g = warp / 4, wq = warp & 3, t = tid & 127;
    const uint32_t d = tmem + (uint32_t)(g * 256) + ((uint32_t)(32 * wq) << 16);
    unsigned char* T = sm + oTiles + g * kTileBytes;
    const uint32_t dbar = sb + oBars + 8 * g, ebar = sb + oBars + 8 * (kWG + g), gbar = sb + oBars + 8 * (2 * kWG + g);
    uint32_t dph = 0, eph = 0, gph = 0;
    // compensated sums of even and odd channels
    float2 loss_s = make_float2(0.f, 0.f), loss_e = loss_s, b3s[CP / 2], b3e[CP / 2];
#pragma unroll
    for (int c = 0; c < CP / 2; ++c) b3s[c] = b3e[c] = make_float2(0.f, 0.f);
    auto wait_bar = [&](uint32_t bar, uint32_t& ph) {
      if (!mbar_wait_bounded(bar, ph, kDefaultWaitBudget)) {
        failed = true;
        mbar_wait_bounded(bar, ph, kDrainBudget);
      }
      ph ^= 1u;
      tc_fence_after();
    };
    auto wait_d = [&]() { wait_bar(dbar, dph); };
    // Phase PH's products, issued by one lane of the warpgroup's first warp once all
    // four have written the operands.  D's products come first and are committed on
    // their own (phases 4, 5: the weight gradients' after them, on gbar; phase 6 as a
    // whole on ebar).
    int n = 0;  // the warpgroup's tile count
    auto issue = [&](auto phase) {
      constexpr int PH = decltype(phase)::value;
      const uint32_t d0 = tmem + (uint32_t)(g * 256), D = d0 + cD;
      const uint32_t T0 = sb + oTiles + g * kTileBytes, XH = T0 + oX + (n & 1) * kX, XL = XH + 4096;
      constexpr uint32_t ID128_64 = idesc(0, 128, 64), ID128_16 = idesc(0, 128, 16);
      constexpr uint32_t ID128_64T = ID128_64 | (1u << 16);  // B MN-major
      constexpr uint32_t IDT64_64 = idesc(0, 64, 64) | (1u << 15) | (1u << 16);
      constexpr uint32_t IDT64_16 = idesc(0, 64, 16) | (1u << 15) | (1u << 16);
      auto k32 = [&](uint32_t addr) { return smem_desc(addr, 16, 256, 6); };                    // SW32 K-major, K = 16
      auto k128 = [&](uint32_t addr, int kk) { return smem_desc(addr + 32 * kk, 16, 1024, 2); };  // SW128 K-major chunk
      auto m128 = [&](uint32_t addr, int kk) { return smem_desc(addr + 2048 * kk, 1024, 1024, 2); };  // SW128 MN-major
      auto m32 = [&](uint32_t addr, int kk) { return smem_desc(addr + 512 * kk, 256, 256, 6); };      // SW32 MN-major
      if constexpr (PH == 4) {  // the G accumulators start afresh below: the finishing warps have the last tile's
        if (elect_one()) {
          tc_fence_after();
          mma_f16(D, k32(T0 + oDYH), k32(sb + oW3TH), ID128_64, 0);
          mma_f16(D, k32(T0 + oDYL), k32(sb + oW3TH), ID128_64, 1);
          mma_f16(D, k32(T0 + oDYH), k32(sb + oW3TL), ID128_64, 1);
          mma_commit(dbar);
        }
        __syncwarp();
        if (n > 0) named_bar_sync(bar_folded(g), 160);
      }
      if (elect_one()) {
        tc_fence_after();
        if constexpr (PH == 1) {
          mma_f16(D, k32(sb + oONES), k32(sb + oBT1), ID128_64, 0);
          mma_f16(D, k32(XH), k32(sb + oW1H), ID128_64, 1);
          mma_f16(D, k32(XL), k32(sb + oW1H), ID128_64, 1);
          mma_f16(D, k32(XH), k32(sb + oW1L), ID128_64, 1);
          mma_commit(dbar);
        } else if constexpr (PH == 2 || PH == 3) {
          const uint32_t AH = T0 + (PH == 2 ? oH1H : oH2H), AL = T0 + (PH == 2 ? oH1L : oH2L);
          const uint32_t BH = sb + (PH == 2 ? oW2H : oW3H), BL = sb + (PH == 2 ? oW2L : oW3L);
          constexpr uint32_t id = PH == 2 ? ID128_64 : ID128_16;
          mma_f16(D, k32(sb + oONES), k32(sb + (PH == 2 ? oBT2 : oBT3)), id, 0);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            mma_f16(D, k128(AH, kk), k128(BH, kk), id, 1);
            mma_f16(D, k128(AL, kk), k128(BH, kk), id, 1);
            mma_f16(D, k128(AH, kk), k128(BL, kk), id, 1);
          }
          mma_commit(dbar);
        } else if constexpr (PH == 4) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            mma_f16(d0 + cG3, m128(T0 + oH2H, kk), m32(T0 + oDYH, kk), IDT64_16, kk == 0 ? 0 : 1);
            mma_f16(d0 + cG3, m128(T0 + oH2L, kk), m32(T0 + oDYH, kk), IDT64_16, 1);
            mma_f16(d0 + cG3, m128(T0 + oH2H, kk), m32(T0 + oDYL, kk), IDT64_16, 1);
          }
          mma_commit(gbar);
        } else if constexpr (PH == 5) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            mma_f16(D, k128(T0 + oH2H, kk), m128(sb + oW2H, kk), ID128_64T, kk > 0);
            mma_f16(D, k128(T0 + oH2L, kk), m128(sb + oW2H, kk), ID128_64T, 1);
            mma_f16(D, k128(T0 + oH2H, kk), m128(sb + oW2L, kk), ID128_64T, 1);
          }
          mma_commit(dbar);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            mma_f16(d0 + cG2, m128(T0 + oH2H, kk), m128(T0 + oH1H, kk), IDT64_64, kk == 0 ? 0 : 1);
            mma_f16(d0 + cG2, m128(T0 + oH2L, kk), m128(T0 + oH1H, kk), IDT64_64, 1);
            mma_f16(d0 + cG2, m128(T0 + oH2H, kk), m128(T0 + oH1L, kk), IDT64_64, 1);
            mma_f16(d0 + cG2b, m128(T0 + oH2H, kk), m32(sb + oONES, kk), IDT64_16, kk == 0 ? 0 : 1);
            mma_f16(d0 + cG2b, m128(T0 + oH2L, kk), m32(sb + oONES, kk), IDT64_16, 1);
          }
          mma_commit(gbar);
        } else {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            mma_f16(d0 + cDX, k128(T0 + oH1H, kk), k128(sb + oW1TH, kk), ID128_16, kk > 0);
            mma_f16(d0 + cDX, k128(T0 + oH1L, kk), k128(sb + oW1TH, kk), ID128_16, 1);
            mma_f16(d0 + cDX, k128(T0 + oH1H, kk), k128(sb + oW1TL, kk), ID128_16, 1);
          }
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            mma_f16(d0 + cG1, m128(T0 + oH1H, kk), m32(XH, kk), IDT64_16, kk == 0 ? 0 : 1);
            mma_f16(d0 + cG1, m128(T0 + oH1L, kk), m32(XH, kk), IDT64_16, 1);
            mma_f16(d0 + cG1, m128(T0 + oH1H, kk), m32(XL, kk), IDT64_16, 1);
          }
          mma_commit(ebar);
        }
      }
      __syncwarp();
    };
    // the warpgroup's operands are written and its accumulator reads done
    auto handoff = [&](auto phase) {
      fence_proxy_async_smem();
      tc_fence_before();
      named_bar_sync(bar_a(g), 128);
      if (wq == 0) issue(phase);
    };
    // split of 32 consecutive accumulator columns (two x16 loads) into a row of a
    // SW128 hi / lo tile pair, through f (ReLU or the derivative mask)
    // (derivatives overwrite activations: once phase 4 / 5's weight-gradient products
    // have read them)
    auto epi64 = [&](uint32_t oh, uint32_t ol, uint32_t mask_lo, uint32_t mask_hi, auto relu_c, uint32_t& m_lo,
                     uint32_t& m_hi) {
      constexpr bool relu = decltype(relu_c)::value;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        uint32_t r[32];
        tmem_ld32_wait(d + cD + 32 * part, r);
        uint32_t mk = 0;
        if (!relu && part == 0) wait_bar(gbar, gph);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t h[4], l[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = 8 * c + 2 * e;
            float v0 = __uint_as_float(r[j]), v1 = __uint_as_float(r[j + 1]);
            if (relu) {
              mk |= (v0 > 0.f ? 1u : 0u) << j;
              mk |= (v1 > 0.f ? 1u : 0u) << (j + 1);
              v0 = fmaxf(v0, 0.f);
              v1 = fmaxf(v1, 0.f);
            } else {
              const uint32_t m = part ? mask_hi : mask_lo;
              if (!((m >> j) & 1u)) v0 = 0.f;
              if (!((m >> (j + 1)) & 1u)) v1 = 0.f;
            }
            split_f16x2(v0, v1, h[e], l[e]);
          }
          const uint32_t o = sw128(t, 16 * (4 * part + c));
          sts128(smem_u32(T + oh + o), h[0], h[1], h[2], h[3]);
          sts128(smem_u32(T + ol + o), l[0], l[1], l[2], l[3]);
        }
        if (part == 0) m_lo = mk;
        else m_hi = mk;
      }
    };
    // A tile's record: the features into x, to be put in place as X (12 features, column
    // 12 = 1 in the hi tile) in buffer b, and the target into tv (rows past the batch
    // and channels past C are zero).
    float4 x[3];
    float4 tv[CP / 4];
#pragma unroll
    for (int q = 0; q < CP / 4; ++q) tv[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_record = [&](int64_t tile) {
      const int64_t sid = tile * 128 + t;
      const bool valid = sid < a.batch;
      const float4* from = reinterpret_cast<const float4*>(a.xt + (valid ? sid : 0) * a.rs);
#pragma unroll
      for (int q = 0; q < 3; ++q) x[q] = valid ? __ldg(from + q) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < CP / 4; ++q)
        if (4 * q < C) tv[q] = valid ? __ldg(from + 3 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
      // the record after that into L2
      const int64_t nsid = sid + stride * 128;
      if (nsid < a.batch) {
        prefetch_l2(a.xt + nsid * a.rs);
        prefetch_l2(a.xt + (nsid + 1) * a.rs - 1);
      }
    };
    auto put_record = [&](int b) {
      unsigned char* X = T + oX + b * kX;
      uint32_t h[8], l[8];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        split_f16x2(x[q].x, x[q].y, h[2 * q], l[2 * q]);
        split_f16x2(x[q].z, x[q].w, h[2 * q + 1], l[2 * q + 1]);
      }
      h[6] = 0x3C00u; l[6] = 0u;  // column 12: 1 (hi) / 0 (lo)
      h[7] = 0u; l[7] = 0u;
      sts128(smem_u32(X + sw32(t, 0)), h[0], h[1], h[2], h[3]);
      sts128(smem_u32(X + sw32(t, 16)), h[4], h[5], h[6], h[7]);
      sts128(smem_u32(X + 4096 + sw32(t, 0)), l[0], l[1], l[2], l[3]);
      sts128(smem_u32(X + 4096 + sw32(t, 16)), l[4], l[5], l[6], l[7]);
    };
    const int64_t tile0 = (int64_t)blockIdx.x * kWG + g;
    if (tile0 < tiles) {
      load_record(tile0);
      put_record(0);
    }
    for (int64_t tile = tile0; tile < tiles; tile += stride, ++n) {
      const bool valid = tile * 128 + t < a.batch;
      // ---- 1: X is in place
      handoff(std::integral_constant<int, 1>{});
      // ---- 2, 3: hidden activations (and their ReLU masks)
      uint32_t m1l, m1h, m2l, m2h;
      wait_d();
      if (n > 0) wait_bar(ebar, eph);  // the tile before: phase 6 has read H1 (and its X buffer)
      epi64(oH1H, oH1L, 0, 0, std::true_type{}, m1l, m1h);
      handoff(std::integral_constant<int, 2>{});
      wait_d();
      epi64(oH2H, oH2L, 0, 0, std::true_type{}, m2l, m2h);
      handoff(std::integral_constant<int, 3>{});
      // ---- 4: y -> loss, unscaled dL/dy
      wait_d();
      {
        uint32_t r[16];
        tmem_ld16_wait(d + cD, r);
        uint32_t h[8], l[8];
#pragma unroll
        for (int i = 0; i < kCMax / 2; ++i) {
          h[i] = l[i] = 0u;
          if (2 * i >= CP || 2 * i >= C) continue;  // uniform
          // y and target are zero past C (zero weights and bias), so an odd count's
          // last pair adds nothing; rows past the batch are masked
          const float4 tq = tv[i / 2];
          const float2 tp = i & 1 ? make_float2(tq.z, tq.w) : make_float2(tq.x, tq.y);
          float2 res = make_float2(__uint_as_float(r[2 * i]) - tp.x, __uint_as_float(r[2 * i + 1]) - tp.y);
          if (!valid) res = make_float2(0.f, 0.f);
          float2 gc;
          if (a.loss_l1) {
            two_sum2(loss_s, loss_e, make_float2(fabsf(res.x), fabsf(res.y)));
            gc = make_float2(res.x > 0.f ? 1.f : (res.x < 0.f ? -1.f : 0.f), res.y > 0.f ? 1.f : (res.y < 0.f ? -1.f : 0.f));
          } else {
            two_sum2(loss_s, loss_e, __fmul2_rn(res, res));
            gc = __fadd2_rn(res, res);
          }
          two_sum2(b3s[i], b3e[i], gc);
          split_f16x2(gc.x, gc.y, h[i], l[i]);
        }
        sts128(smem_u32(T + oDYH + sw32(t, 0)), h[0], h[1], h[2], h[3]);
        sts128(smem_u32(T + oDYH + sw32(t, 16)), h[4], h[5], h[6], h[7]);
        sts128(smem_u32(T + oDYL + sw32(t, 0)), l[0], l[1], l[2], l[3]);
        sts128(smem_u32(T + oDYL + sw32(t, 16)), l[4], l[5], l[6], l[7]);
      }
      const bool more = tile + stride < tiles;
      if (more) load_record(tile + stride);
      handoff(std::integral_constant<int, 4>{});
      // the next tile's X while B1 runs (its buffer was last read by phase 6 of the
      // tile before this one)
      if (more) put_record((n + 1) & 1);
      // ---- 5, 6: dZ2 over H2, dZ1 over H1
      uint32_t dummy0, dummy1;
      wait_d();
      epi64(oH2H, oH2L, m2l, m2h, std::false_type{}, dummy0, dummy1);
      handoff(std::integral_constant<int, 5>{});
      wait_d();
      epi64(oH1H, oH1L, m1l, m1h, std::false_type{}, dummy0, dummy1);
      handoff(std::integral_constant<int, 6>{});
    }
    if (n > 0) wait_bar(ebar, eph);  // the last tile: its shared-memory tiles are free
    // loss and db3: this warpgroup's per-thread compensated sums, reduced in a fixed order
    float* red = reinterpret_cast<float*>(T + 64 * 112 * 4);  // (1 + 16) x 128 threads x 2
    auto put_red = [&](int q, float s0, float e0, float s1, float e1) {
      float s = 0.f, e = e0 + e1;
      neumaier(s, e, s0);
      neumaier(s, e, s1);
      red[(q * 128 + t) * 2] = s;
      red[(q * 128 + t) * 2 + 1] = e;
    };
    put_red(0, loss_s.x, loss_e.x, loss_s.y, loss_e.y);
#pragma unroll
    for (int c = 0; c < CP / 2; ++c) {
      put_red(1 + 2 * c, b3s[c].x * a.scale, b3e[c].x * a.scale, 0.f, 0.f);
      put_red(2 + 2 * c, b3s[c].y * a.scale, b3e[c].y * a.scale, 0.f, 0.f);
    }
    regs_dec<kRegsLaunch>();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // ---- the CTA's partials: warpgroup 0 + warpgroup 1, compensated
  {
    float* part = a.part + (size_t)blockIdx.x * kPart;
    const float* g0 = reinterpret_cast<const float*>(sm + oTiles);
    const float* g1 = reinterpret_cast<const float*>(sm + oTiles + kTileBytes);
    auto put = [&](int slot, float x0, float x1) {
      float s = 0.f, e = 0.f;
      neumaier(s, e, x0);
      neumaier(s, e, x1);
      part[2 * slot] = s;
      part[2 * slot + 1] = e;
    };
    for (int e = tid; e < 64 * 112; e += blockDim.x) {
      const int row = e / 112, col = e - row * 112;
      const float x0 = g0[e], x1 = g1[e];
      if (col < 64) put(kGW2 + row * kH + col, x0, x1);                     // dW2[out = row][in = col]
      else if (col == 64) put(kGB2 + row, x0, x1);                          // db2
      else if (col >= 80 && col < 96) {                                     // dW3[c][in = row]
        const int c = col - 80;
        if (c < kCMax) put(kGW3 + c * kH + row, c < C ? x0 : 0.f, c < C ? x1 : 0.f);
      } else if (col >= 96 && col < 96 + kIn) put(kGW1 + row * kIn + (col - 96), x0, x1);  // dW1
      else if (col == 96 + kIn) put(kGB1 + row, x0, x1);                    // db1 (the ones column of X)
    }
    // warp q: the loss (q = 0) or db3[q - 1], over both warpgroups in a fixed order:
    // lane i takes threads 8 i .. 8 i + 7 of the 256, then a butterfly over the lanes
    for (int q = warp; q <= CP; q += kThreads / 32) {
      const float* r = reinterpret_cast<const float*>(sm + oTiles + (lane >> 4) * kTileBytes + 64 * 112 * 4) +
                       (q * 128 + (lane & 15) * 8) * 2;
      float s = 0.f, e = 0.f;
#pragma unroll
      for (int th = 0; th < 8; ++th) {
        neumaier(s, e, r[2 * th]);
        e += r[2 * th + 1];
      }
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        const float os = __shfl_xor_sync(0xffffffffu, s, off), oe = __shfl_xor_sync(0xffffffffu, e, off);
        neumaier(s, e, os);
        e += oe;
      }
      if (lane == 0) {
        if (q == 0) {
          part[2 * kGN] = s;
          part[2 * kGN + 1] = e;
        } else {
          part[2 * (kGB3 + q - 1)] = s;
          part[2 * (kGB3 + q - 1) + 1] = e;
        }
      }
    }
  }
  if (failed) record_status(a.status, NBTC_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

}  // namespace nbtc
