// Weight image of the FP32-accurate tensor-core form (kF32Split), built from the
// FP32 MLP by all threads of a CTA: by nbtc_pack_mlp into global memory, or by
// each CTA of an FP32 decode straight into its shared memory.
//
// What a split FP16 product loses against FP32, and what is done about it:
//  - Range.  FP16 holds 2^-24 .. 65504, FP32 networks hold anything.  Scaling a
//    ReLU neuron by a power of two and its outgoing weights by the inverse is
//    exact, so every neuron i of layer l is scaled by 2^a with
//    bound_i 2^a < 2^T_l, bound_i = |b_i| + sum_k |w_ik| bound_k >= its largest
//    activation (features lie in [0, 1]).  T_l grows by layer to 15, so neither an
//    activation nor a weight from a live neuron (whose scaled bound is 2^(T_(l-1) - 1)
//    or more) can overflow, and the scaled weights of a row sum to
//    2^(T_l - T_(l-1)) at most (32 or more), which keeps their lo parts out of
//    FP16's subnormals: at unit scale a He-initialised weight's lo part is a
//    multiple of 2^-24, an error of 1e-7 of the weight and the largest of the
//    form.  Output channels are scaled likewise, to a bound that FP16 does not hold
//    (their weights do fit), and multiplied back in FP32, where the bias is added: a
//    bias may be any share of a channel, so it is no FP16 operand.
//  - Accumulator rounding.  The tensor core's FP32 accumulator truncates: each
//    MMA that adds a full-size product loses part of an ulp of the sum, always
//    toward zero.  The hi.lo products are added first, where the sum is 2^-11 of
//    its final size, then the hi.hi chunks of 16 inputs, which leave it at 1/n ..
//    n/n of it (on average also for sums of both signs): c (n + 1) / 2 ulp for n
//    chunks.  Half an ulp over a mantissa in [1, 2) makes c 0.35 to 0.36 of the
//    sum; measured 0.325 (the bias left on 12-64-9, 12-64-64-9 and 12-64-64-64-9
//    decodes is below 1e-8).  The weights are raised by that, into the lo part.
//  - Feature scale.  The kernels multiply texel bytes by RN32(1 / 255), 5.9e-8 too
//    large; layer 1 takes it back the same way.
//
// Against FP64 over 30 networks the form is then as accurate as the FFMA kernels
// at hidden width 64 or better (2-norm of the error 0.89 .. 0.90 of theirs,
// largest error 0.71 .. 0.77), equal at 32 and 1.18 times at 16; before, 2.7 to 3 times.
#pragma once

#include "sm100.cuh"
#include "tc.cuh"

namespace nbtc {

// Instead of an exponent: a hidden neuron whose bound is 0 (no weight from a live
// neuron, no bias).  Its activation is exactly 0, so its outgoing weights are left
// out: no scale fits them (a pruned neuron's may be of any size, and inf * 0 is NaN).
constexpr short kF32sDead = -32768;

struct F32sScratch {
  float bound[2][kHid];
  short a[5][kHid];  // exponent a of every neuron: features (0), hidden layers, outputs; kF32sDead
  int bad;           // a weight or bound that is not finite, or beyond 2^100
};

// Exponent T of the bound of layer l's scaled values (0: features; nhid + 1: outputs).
__host__ __device__ constexpr int f32s_target(int nhid, int l) {
  return l == 0 ? 0 : l > nhid ? 23 : nhid == 1 ? 11 : nhid == 2 ? (l == 1 ? 7 : 15) : 5 * l;
}

// Fills S.a and S.bad.  `t` of `nt` threads (a multiple of 32); ends with a barrier.
__device__ inline void f32s_scales(const float* __restrict__ W, const float* __restrict__ B, int nhid, int hid, int nout,
                                   int t, int nt, F32sScratch& S) {
  if (t == 0) S.bad = 0;
  if (t < kHid) {
    S.bound[0][t] = 1.f;
    S.a[0][t] = 0;
  }
  __syncthreads();
  int off = 0, boff = 0;
  for (int l = 0; l <= nhid; ++l) {
    const int in = l == 0 ? 12 : hid, o = l == nhid ? nout : hid;
    const float* mb = S.bound[l & 1];
    // eight threads a row
    for (int r0 = 0; r0 < o; r0 += nt / 8) {
      const int r = r0 + t / 8;
      float s = 0.f;
      if (r < o)
        for (int k = t & 7; k < in; k += 8) s = fmaf(fabsf(W[off + r * in + k]), mb[k], s);
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      if (r < o && (t & 7) == 0) {
        if (l < nhid) s += fabsf(B[boff + r]);  // an output's bias is added in FP32, unscaled
        s *= 1.0001f;  // FP32 rounding of the sum
        int e = 0;
        if (s < 1e30f) frexpf(s, &e);  // s < 2^e
        else S.bad = 1;                // (also NaN)
        S.bound[(l + 1) & 1][r] = s;
        S.a[l + 1][r] = s > 0.f ? (short)(f32s_target(nhid, l + 1) - e) : l == nhid ? (short)0 : kF32sDead;
      }
    }
    off += in * o;
    boff += o;
    __syncthreads();
  }
}

// The image (see TcLayout; already cleared) from the FP32 MLP and the scales.
__device__ inline void f32s_pack(unsigned char* img, const TcLayout L, const float* __restrict__ W,
                                 const float* __restrict__ B, int hid, int nout, int t, int nt, const F32sScratch& S) {
  const int nhid = L.nhid, R1 = L.w1_row();
  constexpr float kUlp = 0.325f * 1.1920929e-7f;  // mean truncation of a full-size sum
  constexpr double kInv255 = (double)(1.0f / 255.0f);
  const float e1 = kUlp + (float)(1.0 / 255.0 / kInv255 - 1.0);
  const float eh = kUlp * 0.5f * (float)(hid / 16 + 1);
  auto split = [](float w, float e, uint16_t& h, uint16_t& lo) {
    const __half hh = __float2half_rn(w);
    h = __half_as_ushort(hh);
    lo = __half_as_ushort(__float2half_rn(fmaf(w, e, w - __half2float(hh))));
  };
  auto put = [&](uint32_t at, uint16_t v) { *reinterpret_cast<uint16_t*>(img + at) = v; };
  int off = 0, boff = 0;
  for (int l = 0; l <= nhid; ++l) {
    const int in = l == 0 ? 12 : hid, o = l == nhid ? nout : hid;
    const float e = l == 0 ? e1 : eh;
    for (int i = t; i < in * o; i += nt) {
      const int n = i / in, k = i - n * in;
      if (S.a[l + 1][n] == kF32sDead || S.a[l][k] == kF32sDead) continue;  // (the image is cleared)
      uint16_t h, lo;
      split(ldexpf(W[off + i], S.a[l + 1][n] - S.a[l][k]), e, h, lo);
      if (l == 0) {
        put(L.off_w1() + off_ilv(n, 2 * k, R1), h);
        put(L.off_w1() + off_ilv(n, 2 * (16 + k), R1), h);
        put(L.off_w1() + off_ilv(n, 2 * (32 + k), R1), lo);
      } else {
        const int base = l == nhid ? L.off_wo() : L.off_wh(l - 1);
        const int part = l == nhid ? L.wo_part() : L.wh_part();
        put(base + off_sw128(n, 2 * k), h);
        put(base + off_sw128(n, 2 * k) + part, lo);
      }
    }
    for (int i = t; i < o && l < nhid; i += nt) {
      if (S.a[l + 1][i] == kF32sDead) continue;
      uint16_t h, lo;
      split(ldexpf(B[boff + i], S.a[l + 1][i]), l == 0 ? kUlp : e, h, lo);
      if (l == 0) {
        put(L.off_w1() + off_ilv(i, 24, R1), h);
        put(L.off_w1() + off_ilv(i, 2 * (16 + 12), R1), lo);
      } else {
        put(L.off_bth(l - 1) + off_interleave(i, 0), h);
        put(L.off_bth(l - 1) + off_interleave(i, 2), lo);
      }
    }
    off += in * o;
    boff += o;
  }
  // output biases, then (at nhid kHid) the multipliers of the accumulated products
  float* bias = reinterpret_cast<float*>(img + L.off_bias());
  for (int c = t; c < kOutPad; c += nt) {
    bias[c] = c < nout ? B[nhid * hid + c] : 0.f;
    bias[nhid * kHid + c] = c < nout ? ldexpf(1.f, -S.a[nhid + 1][c]) : 0.f;
  }
}

}  // namespace nbtc
