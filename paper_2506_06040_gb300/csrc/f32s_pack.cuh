// Weight image of the FP32-accurate tensor-core form (kF32Split), built from the
// FP32 MLP by all threads of a CTA: by nbtc_pack_mlp into global memory, or by
// each CTA of an FP32 decode straight into its shared memory.
//
// What a split FP16 product loses against FP32, and what is done about it:
//  - Range.  FP16 holds 2^-24 .. 65504, FP32 networks hold anything.  Scaling a
//    ReLU neuron by a power of two and its outgoing weights by the inverse is
//    exact, so every neuron i of layer l is scaled by 2^a with bound_i 2^a < 2^T_l,
//    bound_i = b_i + sum_k max(w_ik, 0) bound_k >= its largest activation (features
//    lie in [0, 1]), and no scaled weight from a live neuron and no scaled bias
//    beyond 2^15.  So no operand overflows; T_l grows by layer to 15, so the scaled
//    weights of a row sum to 32 and more, which keeps their lo parts out of
//    FP16's subnormals: at unit scale a He-initialised weight's lo part is a
//    multiple of 2^-24, an error of 1e-7 of the weight and the largest of the
//    form.  Output channels are scaled likewise, to a bound that FP16 does not hold
//    (their weights do fit), and multiplied back in FP32, where the bias is added: a
//    bias may be any share of a channel, so it is no FP16 operand.
//  - Operands.  hi + lo hold 22 to 24 bits; the features and layer 1's weights, whose
//    products are few, come in three parts (all 24), and lo.lo is not left out.
//  - Accumulator rounding.  The tensor core's FP32 accumulator truncates: an MMA
//    that leaves a full-size sum takes part of an ulp off it, always toward zero,
//    and more where its products have one sign (they are cut to a common grid
//    first).  The small products are added first, then the bias, then the hi.hi
//    chunks of 16 inputs, which leave the sum at 1/n .. n/n of its final size (on
//    average also for sums of both signs): (n + 1) / 2 times the loss at full size, n
//    the row's chunks that hold a weight.  The row's weights are raised by that.
//    kTruncUlp and kAlignUlp are what took the mean bias off dense and all-positive
//    networks (half an ulp over mantissas in [1, 2) would be 0.35); a lone weight that is
//    a power of two loses nothing and is not raised.
//  - Feature scale.  Texel bytes over 255 are rounded, and by a rounded 1 / 255;
//    the features come as bytes over 64 and 64/255 goes into layer 1's weights.
//
// 2-norm of the error against FP64, over that of FP32 FMAs on the same networks
// (width 64, ten networks of each kind and depth 1 / 2 / 3, 640 x 400 texels):
//   He-initialised                           0.68 / 0.75 / 0.80
//   fitted to a target (800 Adam steps)      0.70 / 0.73 / 0.81
//   He, biases of 0.1 .. 0.9                 0.55 / 0.64 / 0.66
//   all weights positive                     0.43 / 0.42 / 0.43
//   half the weights 0                       0.71 / 0.82 / 0.90
//   nine in ten weights 0                    0.66 / 0.86 / 1.04
//   one weight a row, 1                      0.79 / 0.79 / 0.79
//   one weight a row, any                    0.95 / 1.17 / 1.36
// FP32 FMAs round once per weight that is not 0, a split product once per operand: where
// rows hold one weight or a few the split's error is the larger, 8e-8 to 1.5e-7 in all.
#pragma once

#include "sm100.cuh"
#include "tc.cuh"

namespace nbtc {

struct F32sScratch {
  float bound[2][kHid];
  // 2^a of every neuron's scale and 2^-a: features (0), hidden layers, outputs.  Both 0
  // for a hidden neuron whose bound is 0 (its activation is exactly 0 for any
  // features): that leaves out its weights and its outgoing weights, for which there is
  // no scale (a pruned neuron's may be of any size, and inf * 0 is NaN).
  float up[5][kHid], down[5][kHid];
  float loss[5][kHid];  // mean share of a row's sum that truncation takes
  int bad;              // a weight or bound that is not finite, or beyond 2^100
};

// Mean loss of an MMA that leaves a full-size sum, in 2^-23 of it: of the sum's
// truncation, and of its products' when they all have one sign.
constexpr float kTruncUlp = 0.27f, kAlignUlp = 0.44f;

// Exponent T of the bound of layer l's scaled values (0: features; nhid + 1: outputs).
__host__ __device__ constexpr int f32s_target(int nhid, int l) {
  return l == 0 ? 0 : l > nhid ? 23 : nhid == 1 ? 11 : nhid == 2 ? (l == 1 ? 7 : 15) : 5 * l;
}

// e with x < 2^e, for finite x >= 0 (subnormal ones count as 2^-127).
__device__ __forceinline__ int exponent_above(float x) { return (int)(__float_as_uint(x) >> 23) - 126; }

// 2^a, |a| <= 126.
__device__ __forceinline__ float pow2f(int a) { return __int_as_float((a + 127) << 23); }

// Fills S (in shared memory) but for the bounds.  `t` of `nt` threads (a multiple of
// 32); ends with a barrier.  Out of line, as f32s_pack: inlined they cost the decode
// kernel's main loop registers (4096^2 12-64-64-9: 671 us, 643 so).
static __device__ __noinline__ void f32s_scales(const float* __restrict__ W, const float* __restrict__ B, int nhid,
                                                int hid, int nout, int t, int nt, F32sScratch& S) {
  // every layer waits for the one before: all its weights on their way first
  for (int i = 32 * t; i < 12 * hid + (nhid - 1) * hid * hid + hid * nout; i += 32 * nt) sm100::prefetch_l1(W + i);
  if (32 * t < nhid * hid + nout) sm100::prefetch_l1(B + 32 * t);
  if (t == 0) S.bad = 0;
  if (t < kHid) {
    S.bound[0][t] = 1.f;
    S.up[0][t] = 4.f;  // features come as texel bytes over 64
    S.down[0][t] = 0.25f;
  }
  __syncthreads();
  const float inv_hid = 1.f / (float)hid;
  int off = 0, boff = 0;
  for (int l = 0; l <= nhid; ++l) {
    const int in = l == 0 ? 12 : hid, o = l == nhid ? nout : hid;
    const float* mb = S.bound[l & 1];
    // eight threads a row
    for (int r0 = 0; r0 < o; r0 += nt / 8) {
      const int r = r0 + t / 8;
      float sum = 0.f, sq = 0.f, pos = 0.f;  // of x = |w| bound, of x^2, of x over the positive weights
      float top = 0.f;                       // largest weight once the inputs are scaled
      uint32_t seen = 0;                     // bits 0..3: chunks of 16 inputs, 4: a weight that is no power of two, 8..: weights
      float w[kHid / 8];
      const float b = r < o && l < nhid ? B[boff + r] : 0.f;
#pragma unroll
      for (int j = 0; j < kHid / 8; ++j) {
        const int k = (t & 7) + 8 * j;
        w[j] = r < o && k < in ? W[off + r * in + k] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < kHid / 8; ++j) {
        const int k = (t & 7) + 8 * j;
        if (w[j] == 0.f) continue;
        const float x = fabsf(w[j]) * mb[k];
        sum += x;  // (a weight that is not finite shows here, whatever its input)
        if (mb[k] == 0.f) continue;
        sq = fmaf(x, x, sq);
        pos += w[j] > 0.f ? x : 0.f;
        top = fmaxf(top, fabsf(w[j]) * S.down[l][k]);
        seen = (seen | 1u << (k >> 4) | ((__float_as_uint(w[j]) & 0x7FFFFFu) || l == 0 ? 16u : 0u)) + 256u;
      }
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, d);
        sq += __shfl_xor_sync(0xffffffffu, sq, d);
        pos += __shfl_xor_sync(0xffffffffu, pos, d);
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
        const uint32_t other = __shfl_xor_sync(0xffffffffu, seen, d);
        seen = ((seen | other) & 31u) | ((seen & ~31u) + (other & ~31u));
      }
      if (r < o && (t & 7) == 0) {
        // share of the inputs that carry the row, and how far they have one sign
        const float many = sq > 0.f ? sum * rsqrtf(sq) : 0.f;
        const float one_sign = sum > 0.f ? __fdividef(fabsf(2.f * pos - sum), sum) : 0.f;
        const float coherent = many * many * (l == 0 ? 1.f / 12.f : inv_hid) * one_sign;
        sum += fabsf(b);
        if (!(sum < 1e30f) || !(top < 1e30f)) S.bad = 1;  // (also NaN)
        // the margin covers the FP32 rounding of these sums
        const float bound = l < nhid ? fmaxf(pos + b + 1e-5f * sum, 0.f) : sum;
        int a = 0;
        if (bound > 0.f && sum < 1e30f) {
          a = f32s_target(nhid, l + 1) - exponent_above(1.0001f * bound);
          if (top > 0.f) a = min(a, 15 - exponent_above(top));
          if (b != 0.f) a = min(a, 15 - exponent_above(fabsf(b)));
          a = min(max(a, -120), 120);
        }
        const bool dead = l < nhid && !(bound > 0.f);
        S.bound[(l + 1) & 1][r] = 1.0001f * bound;
        S.up[l + 1][r] = dead ? 0.f : pow2f(a);
        S.down[l + 1][r] = dead ? 0.f : pow2f(-a);
        const int n = l == 0 ? 1 : __popc(seen & 15u);
        const bool lone = (seen >> 8) <= 1 && !(seen & 16u) && b == 0.f;
        S.loss[l + 1][r] = lone ? 0.f : 0.5f * (float)(n + 1) * (kTruncUlp + kAlignUlp * coherent) * 1.1920929e-7f;
      }
    }
    off += in * o;
    boff += o;
    __syncthreads();
  }
}

// The image (see TcLayout; already cleared) from the FP32 MLP and the scales, two
// weights of a row at a time.
static __device__ __noinline__ void f32s_pack(unsigned char* img, const TcLayout L, const float* __restrict__ W,
                                              const float* __restrict__ B, int hid, int nout, int t, int nt,
                                              const F32sScratch& S) {
  const int nhid = L.nhid, R1 = L.w1_row();
  // parts of w + w c, exact to 2^-36 of it
  auto split = [](float w, float c, uint32_t (&part)[3]) {
    const __half h = __float2half_rn(fmaf(w, c, w));
    const float r = fmaf(w, c, w - __half2float(h));  // (the difference is exact)
    const __half lo = __float2half_rn(r);
    part[0] = __half_as_ushort(h);
    part[1] = __half_as_ushort(lo);
    part[2] = __half_as_ushort(__float2half_rn(r - __half2float(lo)));
  };
  auto put = [&](uint32_t at, uint32_t v) { *reinterpret_cast<uint16_t*>(img + at) = (uint16_t)v; };
  auto put2 = [&](uint32_t at, uint32_t v0, uint32_t v1) { *reinterpret_cast<uint32_t*>(img + at) = v0 | v1 << 16; };
  const int sh = hid == 16 ? 3 : hid == 32 ? 4 : 5;  // log2 of a hidden row's pairs
  int off = 0, boff = 0;
  for (int l = 0; l <= nhid; ++l) {
    const int o = l == nhid ? nout : hid;
    if (l == 0) {
      for (int i = t; i < 6 * o; i += nt) {
        const int n = i / 6, k = 2 * (i - 6 * n);
        const float up = S.up[1][n] * S.down[0][0], e = S.loss[1][n], c = 1.f / 255.f + e * (256.f / 255.f);
        uint32_t q[3], q1[3];
        split(W[12 * n + k] * up, c, q);
        split(W[12 * n + k + 1] * up, c, q1);
#pragma unroll
        for (int j = 0; j < 3; ++j) put2(L.off_w1() + off_ilv(n, 2 * (16 * j + k), R1), q[j], q1[j]);
      }
      off += 12 * o;
    } else {
      const int base = l == nhid ? L.off_wo() : L.off_wh(l - 1), part = l == nhid ? L.wo_part() : L.wh_part();
#pragma unroll 4
      for (int i = t; i < o << sh; i += nt) {
        const int n = i >> sh, k = 2 * (i & ((1 << sh) - 1));
        const float* w = W + off + n * hid + k;
        const float up = S.up[l + 1][n], e = S.loss[l + 1][n];
        uint32_t q[3], q1[3];
        split(w[0] * S.down[l][k] * up, e, q);
        split(w[1] * S.down[l][k + 1] * up, e, q1);
        const uint32_t at = base + off_sw128(n, 2 * k);
        put2(at, q[0], q1[0]);
        put2(at + part, q[1], q1[1]);
      }
      off += hid * o;
    }
    for (int i = t; i < o && l < nhid; i += nt) {
      uint32_t q[3];
      split(B[boff + i] * S.up[l + 1][i], S.loss[l + 1][i], q);
      if (l == 0) {
#pragma unroll
        for (int j = 0; j < 3; ++j) put(L.off_w1() + off_ilv(i, 2 * (16 * j + 12), R1), q[j]);
      } else {
        put2(L.off_bth(l - 1) + off_interleave(i, 0), q[0], q[1]);
      }
    }
    boff += o;
  }
  // output biases, then (at nhid kHid) the multipliers of the accumulated products
  float* out = reinterpret_cast<float*>(img + L.off_bias());
  for (int c = t; c < kOutPad; c += nt) {
    out[c] = c < nout ? B[nhid * hid + c] : 0.f;
    out[nhid * kHid + c] = c < nout ? S.down[nhid + 1][c] : 0.f;
  }
}

}  // namespace nbtc
