// Feature pass of a frame: the 12 latent features of every pixel, FP16, in
// screen order (24 bytes a pixel), which the tensor-core kernel then reads as
// its tiles' operand rows.
//
// A pixel takes two bilinear samples per level (trilinear), or that many per
// probe of the anisotropic filter: 32 to 512 dependent gathers.  Inside the
// tensor-core kernel, whose 16 warps a SM are set by its registers and tensor
// memory, those gathers were latency-bound; here they run at 36 to 40 warps a SM
// for 24 bytes a pixel written and read back.
#include "features.cuh"
#include "host.h"
#include "sm100.cuh"
#include "tc.cuh"

namespace nbtc {

namespace {

// ---- decoded texels (RGBA8 words, k_frame_texels).  A tap that decodes its BC1
// texel costs ~65 instructions (two endpoints widened, three palette channels
// with a division, three conversions), a tap of a decoded word ~18 with the blend.

// Channel c of an RGBA8 word as 2^23 + value (one byte permute, exact).
__device__ __forceinline__ float byte_magic(uint32_t t, int c) {
  return __uint_as_float(__byte_perm(t, 0x4B000000u, 0x7440u + (uint32_t)c));
}

// One mip's decoded texels.
struct TexelView {
  const uint32_t* t;
  int w, h;
};

__device__ __forceinline__ uint32_t texel_at(const FrameFeatArgs& a, const TexelView& T, int i) {
#ifdef NBTC_CHECKED
  int64_t c = (int64_t)i + a.plant;
  NBTC_CHECK_INDEX(c, (int64_t)T.w * T.h, a.status);
  i = (int)c;
#else
  (void)a;
#endif
  return __ldg(T.t + i);
}

// Bilinear sample in 0..255 units: the horizontal blends of both rows as packed
// FP32 pairs, then the vertical one.
__device__ __forceinline__ float3 sample_texels(const FrameFeatArgs& a, const TexelView& T, float shift, float u, float v,
                                                bool wrap) {
  int x0, x1, y0, y1;
  float fx, fy;
  axis_taps<true>(u, T.w, shift, wrap, x0, x1, fx);
  axis_taps<true>(v, T.h, shift, wrap, y0, y1, fy);
  const int r0 = y0 * T.w, r1 = y1 * T.w;
  const uint32_t t00 = texel_at(a, T, r0 + x0), t10 = texel_at(a, T, r0 + x1);
  const uint32_t t01 = texel_at(a, T, r1 + x0), t11 = texel_at(a, T, r1 + x1);
  float c[3];
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    const float2 l = make_float2(byte_magic(t00, ch), byte_magic(t01, ch));
    const float2 r = make_float2(byte_magic(t10, ch), byte_magic(t11, ch));
    const float2 d = __fadd2_rn(r, make_float2(-l.x, -l.y));                   // exact
    const float2 z = __fadd2_rn(l, make_float2(-8388608.f, -8388608.f));       // exact
    const float2 q = __ffma2_rn(make_float2(fx, fx), d, z);
    c[ch] = fmaf(fy, q.y - q.x, q.x);
  }
  return make_float3(c[0], c[1], c[2]);
}

// The two mips and the blend of a level at lod `lam` (unclamped).
struct MipPair {
  int m0, m1;
  float t;
};
__device__ __forceinline__ MipPair mip_pair(float lam, float last) {
  lam = fminf(fmaxf(lam, 0.f), last);
  const float f = floorf(lam);
  MipPair P;
  P.m0 = (int)f;
  P.m1 = min(P.m0 + 1, (int)last);
  P.t = lam - f;
  return P;
}

// i / n1 correctly rounded for the probe counts (1 <= i < n1 <= 17), r = RN(1 / n1):
// the correction step of gridcoord.h (checked for every pair on the host).
__device__ __forceinline__ float probe_fraction(float i, float n1, float r) {
  const float q = __fmul_rn(i, r);
  return fmaf(fmaf(-q, n1, i), r, q);
}

// Probes of a pixel.  Trilinear: one, at uv.  Anisotropic latent filter (the
// reference formulas of the anisotropic-filtering extension, in
// texture-coordinate units -- the square latents make Pmax / Pmin the same for
// every level): N = min(ceil(Pmax / Pmin), max_aniso) trilinear probes at
// uv + (i / (N + 1) - 1/2) d along the major-axis derivative d, each level at
// lod bias + log2(Pmax W_k / N), averaged.  N is decided with correctly rounded
// FP32 operations in a fixed order (no contraction), so any IEEE implementation
// decides it alike.
struct Probes {
  int n;
  float au, av;
  float lod;
};
__device__ __forceinline__ Probes aniso_probes(float4 d, float bias, int max_aniso) {
  const float px = __fsqrt_rn(__fadd_rn(__fmul_rn(d.x, d.x), __fmul_rn(d.y, d.y)));
  const float py = __fsqrt_rn(__fadd_rn(__fmul_rn(d.z, d.z), __fmul_rn(d.w, d.w)));
  const bool along_x = px >= py;
  const float pmax = along_x ? px : py, pmin = along_x ? py : px;
  Probes P;
  P.n = 1;
  if (pmax > 0.f) P.n = pmin > 0.f ? (int)fminf(ceilf(__fdiv_rn(pmax, pmin)), (float)max_aniso) : max_aniso;
  P.au = along_x ? d.x : d.z;
  P.av = along_x ? d.y : d.w;
  P.lod = bias + log2f(pmax / (float)P.n);  // -inf for a zero footprint: clamps to mip 0
  return P;
}

// One thread per pixel.  TEX: decoded texels; otherwise BC1 at the taps.  The mip
// pair of a level is the same for all probes of a pixel, so levels run outermost.
template <bool ANISO, bool TEX>
__global__ void __launch_bounds__(256) k_frame_features(FrameFeatArgs a) {
  const int64_t px = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (px >= a.pixels) return;
  const int id = __ldg(a.mat_id + px);
  if (id < 0 || id >= a.nmat) return;  // no material: the pixel is not decoded
  const float2 uv = __ldg(reinterpret_cast<const float2*>(a.uv) + px);
  Probes P{1, 0.f, 0.f, __ldg(a.lod + px)};
  if constexpr (ANISO) P = aniso_probes(__ldg(reinterpret_cast<const float4*>(a.duv) + px), P.lod, a.max_aniso);
  const float n1 = (float)(P.n + 1), rn1 = ANISO ? 1.0f / n1 : 0.f;
  const float inv = ANISO ? (TEX ? 1.0f / 255.0f : 1.0f) / (float)P.n : (TEX ? 1.0f / 255.0f : 1.0f);
  float f[12];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    auto probes = [&](float t, bool wrap, auto&& lower, auto&& upper) {
#pragma unroll 1
      for (int i = 1; i <= P.n; ++i) {
        float uu = uv.x, vv = uv.y;
        if constexpr (ANISO) {
          const float off = probe_fraction((float)i, n1, rn1) - 0.5f;
          uu = fmaf(off, P.au, uu);
          vv = fmaf(off, P.av, vv);
        }
        const float2 at = address_uv(uu, vv, wrap);
        const float3 c0 = lower(at.x, at.y), c1 = upper(at.x, at.y);
        s0 += fmaf(t, c1.x - c0.x, c0.x);
        s1 += fmaf(t, c1.y - c0.y, c0.y);
        s2 += fmaf(t, c1.z - c0.z, c0.z);
        if constexpr (!ANISO) break;
      }
    };
    if constexpr (TEX) {
      const FrameLevel* L = a.levels + 4 * id + k;
      const int4 head = __ldg(reinterpret_cast<const int4*>(L));  // base, log2w, shift
      const int2 more = __ldg(reinterpret_cast<const int2*>(L) + 2);  // last, wrap
      const uint32_t* base = L->base;
      const float shift = __int_as_float(head.w);
      const bool wrap = more.y != 0;
      const MipPair Q = mip_pair(P.lod + __int_as_float(head.z), __int_as_float(more.x));
      const int4 g0 = __ldg(reinterpret_cast<const int4*>(L->mip + Q.m0));
      const int4 g1 = __ldg(reinterpret_cast<const int4*>(L->mip + Q.m1));
      const TexelView V0{base + (uint32_t)g0.x, g0.y, g0.z}, V1{base + (uint32_t)g1.x, g1.y, g1.z};
      probes(Q.t, wrap, [&](float uu, float vv) { return sample_texels(a, V0, shift, uu, vv, wrap); },
             [&](float uu, float vv) { return sample_texels(a, V1, shift, uu, vv, wrap); });
    } else {
      const MatDev& M = a.mats[id];
      const bool wrap = M.d.wrap;
      const MipPair Q = mip_pair(P.lod + M.log2w[k], (float)(M.mips[k] - 1));
      probes(Q.t, wrap, [&](float uu, float vv) { return sample_bilinear(mip_view(M, k, Q.m0), uu, vv, wrap); },
             [&](float uu, float vv) { return sample_bilinear(mip_view(M, k, Q.m1), uu, vv, wrap); });
    }
    f[3 * k + 0] = s0 * inv;
    f[3 * k + 1] = s1 * inv;
    f[3 * k + 2] = s2 * inv;
  }
  uint2* o = a.feat + 3 * px;
#pragma unroll
  for (int i = 0; i < 3; ++i)
    o[i] = make_uint2(sm100::cvt_f16x2(f[4 * i], f[4 * i + 1]), sm100::cvt_f16x2(f[4 * i + 2], f[4 * i + 3]));
}

}  // namespace

nbtc_status launch_frame_features(const FrameFeatArgs& a, cudaStream_t s) {
  const unsigned grid = (unsigned)((a.pixels + 255) / 256);
  if (a.duv) {
    if (a.levels) k_frame_features<true, true><<<grid, 256, 0, s>>>(a);
    else k_frame_features<true, false><<<grid, 256, 0, s>>>(a);
  } else {
    if (a.levels) k_frame_features<false, true><<<grid, 256, 0, s>>>(a);
    else k_frame_features<false, false><<<grid, 256, 0, s>>>(a);
  }
  return cuda_check(cudaGetLastError(), "launch k_frame_features");
}

}  // namespace nbtc
