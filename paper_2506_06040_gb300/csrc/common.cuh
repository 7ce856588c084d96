// Shared device-side pieces of the decoder: status reporting, BC1 texel
// decode, bilinear latent sampling.  Host code includes it for the argument
// structs only.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/nbtc.h"
#include "gridcoord.h"

namespace nbtc {

constexpr int kMaxLevels = NBTC_MAX_LEVELS;

// Device-side view of one latent level at one mip.
struct LevelView {
  const uint64_t* blocks;  // row-major 8-byte BC1 blocks of this mip
  int32_t w, h;            // texels
  int32_t wb;              // blocks per row (w / 4)
  float shift;             // texels, both axes
#ifdef NBTC_CHECKED
  int* status;             // checked build: where an index outside the level is recorded
  int32_t plant;           // checked build, tests only: added to every block index (0 otherwise)
#endif
};

// ---------------------------------------------------------------- status word

// First fault wins; later faults leave the recorded code in place.
__device__ __forceinline__ void record_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// ---------------------------------------------------------------- bounds checks
//
// The checked build (compiled with NBTC_CHECKED) tests every gather index the
// kernels form against the extent of the array it indexes: an index outside
// it records NBTC_ERR_BOUNDS in the launch's status word and is replaced by 0,
// a valid element, so no access leaves its array and nothing traps.  The
// default build compiles the checks away.
#ifdef NBTC_CHECKED
__device__ __forceinline__ int64_t checked_index(int64_t i, int64_t n, int* status) {
  if (i < 0 || i >= n) {
    record_status(status, NBTC_ERR_BOUNDS);
    return 0;
  }
  return i;
}
#define NBTC_CHECK_INDEX(i, n, status) ((i) = ::nbtc::checked_index((i), (n), (status)))
#else
#define NBTC_CHECK_INDEX(i, n, status) ((void)0)
#endif

// Index of block (bx, by) of a level view.
__device__ __forceinline__ int64_t block_index(const LevelView& L, int bx, int by) {
  int64_t i = (int64_t)by * L.wb + bx;
#ifdef NBTC_CHECKED
  i += L.plant;
  NBTC_CHECK_INDEX(i, (int64_t)L.wb * (L.h / 4), L.status);
#endif
  return i;
}

// ---------------------------------------------------------------- BC1 decode

// RGB565 -> 8-bit channels by bit replication, as three ints.
__device__ __forceinline__ void expand565(uint32_t c, int& r, int& g, int& b) {
  const int r5 = (c >> 11) & 31, g6 = (c >> 5) & 63, b5 = c & 31;
  r = (r5 << 3) | (r5 >> 2);
  g = (g6 << 2) | (g6 >> 4);
  b = (b5 << 3) | (b5 >> 2);
}

// One palette channel.  Four-colour blocks (c0 > c1) weight the endpoints
// (3,0) (0,3) (2,1) (1,2) for indices 0..3 and divide by 3 after adding 1;
// three-colour blocks weight them (2,0) (0,2) (1,1) and divide by 2 after adding
// 1, index 3 being black.  (3 e + 1) / 3 == e and (2 e + 1) / 2 == e, so the
// endpoints come out unchanged.
__device__ __forceinline__ int palette_channel(int e0, int e1, int a0, int a1, bool four) {
  const int num = a0 * e0 + a1 * e1 + 1;
  return four ? num / 3 : num >> 1;
}

// Decoded RGB8 of texel (tx, ty) of a block, packed r | g << 8 | b << 16.
__device__ __forceinline__ uint32_t bc1_texel(uint64_t blk, int tx, int ty) {
  const uint32_t c0 = (uint32_t)(blk & 0xFFFFu);
  const uint32_t c1 = (uint32_t)((blk >> 16) & 0xFFFFu);
  const int idx = (int)((uint32_t)(blk >> 32) >> (2 * (4 * ty + tx))) & 3;
  const bool four = c0 > c1;
  int r0, g0, b0, r1, g1, b1;
  expand565(c0, r0, g0, b0);
  expand565(c1, r1, g1, b1);
  // endpoint weights per index
  int a0, a1;
  if (four) {
    a0 = (idx == 0) ? 3 : (idx == 1) ? 0 : (idx == 2) ? 2 : 1;
    a1 = 3 - a0;
  } else {
    a0 = (idx == 0) ? 2 : (idx == 1) ? 0 : (idx == 2) ? 1 : 0;
    a1 = (idx == 3) ? 0 : 2 - a0;
  }
  uint32_t r = palette_channel(r0, r1, a0, a1, four);
  uint32_t g = palette_channel(g0, g1, a0, a1, four);
  uint32_t b = palette_channel(b0, b1, a0, a1, four);
  if (!four && idx == 3) r = g = b = 0;
  return r | (g << 8) | (b << 16);
}

__device__ __forceinline__ uint32_t fetch_texel(const LevelView& L, int x, int y) {
  const uint64_t blk = __ldg(L.blocks + block_index(L, x >> 2, y >> 2));
  return bc1_texel(blk, x & 3, y & 3);
}

// ---------------------------------------------------------------- sampling

// A coordinate as the samplers take it: under wrap addressing without its whole
// periods (u - floor(u) is exact), so the texel coordinate keeps its fraction even
// for tiled uv far from [0, 1).
__device__ __forceinline__ float2 address_uv(float u, float v, bool wrap) {
  return wrap ? make_float2(u - floorf(u), v - floorf(v)) : make_float2(u, v);
}

// Integer neighbours and fractional weight along one axis of an address_uv
// coordinate.  The texel coordinate is t = u * n - 0.5 + shift; neighbours
// floor(t) and floor(t) + 1 are clamped to [0, n-1] or wrapped modulo n.
// HALF: the caller knows |shift| <= 1/2.
template <bool HALF = false>
__device__ __forceinline__ void axis_taps(float u, int n, float shift, bool wrap, int& i0, int& i1,
                                          float& f) {
  float t = fmaf(u, (float)n, shift - 0.5f);
  if (!wrap) t = fminf(fmaxf(t, -1.0f), (float)n);  // outside this range clamping decides
  const float fl = floorf(t);
  f = t - fl;  // exact
  const int a = (int)fl;
  if (wrap) {
    // u in [0, 1] and |shift| <= 1/2: a in [-1, n], wrapped by unsigned minima: x + n
    // is the smaller one when x is negative, x - n when x has reached n
    const uint32_t x = __viaddmin_u32((uint32_t)a, (uint32_t)n, (uint32_t)a);
    i0 = (int)__viaddmin_u32(x, (uint32_t)-n, x);
    i1 = (int)__viaddmin_u32((uint32_t)i0 + 1u, (uint32_t)-n, (uint32_t)i0 + 1u);
    if (!HALF && fabsf(shift) > 0.5f) {  // further periods away
      i0 = a % n < 0 ? a % n + n : a % n;
      i1 = i0 + 1 == n ? 0 : i0 + 1;
    }
  } else {
    i0 = min(max(a, 0), n - 1);
    i1 = min(max(a + 1, 0), n - 1);
  }
}

// ---- BC1 texels as FP32, for samples that decode at their taps.  A block's two
// endpoints are widened with all three channels in 10-bit fields of one word; a
// tap's palette numerators a0 e0 + a1 e1 + 1 are then two multiply-adds for the three
// channels, and the rounded division by 3 (or 2) is one FP32 multiply-add each:
// with F = 2^23 + num (the field under the exponent of 2^23),
//   four colours   num = a0 e0 + a1 e1 + 1 <= 766:       RN(F / 3 + 9786709) = 2^23 + 2^22 + num div 3
//   three colours  num = 2 (a0 e0 + a1 e1) + 1 <= 1021:  RN(F / 4 + 10485760) = 2^23 + 2^22 + (num + 1) div 4
// (the second is (a0 e0 + a1 e1 + 1) div 2; both tested for every numerator on the
// host).  ~45 instructions a tap with its share of the
// block, where the integer decode and conversion of bc1_texel took ~65.
struct Bc1Block {
  uint32_t e0, e1;  // endpoints: r | g << 10 | b << 20
  uint32_t bits;    // 16 2-bit indices
  uint32_t wt;      // byte i: endpoint weights a0 | a1 << 4 of index i
  float scale, add;
};

__device__ __forceinline__ uint32_t widen565(uint32_t c) {
  const uint32_t hi = ((c >> 8) & 0xF8u) | ((c << 7) & 0x3F000u) | ((c << 23) & 0xF800000u);
  return hi | ((hi >> 5) & 0x700007u) | ((hi >> 6) & 0xC00u);
}

__device__ __forceinline__ Bc1Block bc1_block(uint64_t blk) {
  const uint32_t lo = (uint32_t)blk, c0 = lo & 0xFFFFu, c1 = lo >> 16;
  const bool four = c0 > c1;
  Bc1Block b;
  b.e0 = widen565(c0);
  b.e1 = widen565(c1);
  b.bits = (uint32_t)(blk >> 32);
  b.wt = four ? 0x21123003u : 0x00224004u;
  b.scale = four ? 1.0f / 3.0f : 0.25f;
  b.add = four ? 9786709.0f : 10485760.0f;
  return b;
}

constexpr float kTexelBase = 12582912.0f;  // 2^23 + 2^22

// Texel (tx, ty) of a block: channels in 0..255 plus kTexelBase, exact.
__device__ __forceinline__ float3 bc1_texel_f(const Bc1Block& b, int tx, int ty) {
  const uint32_t w = b.wt >> (8u * ((b.bits >> (2 * (4 * ty + tx))) & 3u));
  const uint32_t num = (w & 15u) * b.e0 + ((w >> 4) & 15u) * b.e1 + 0x00100401u;
  auto ch = [&](uint32_t f) { return fmaf(__uint_as_float(0x4B000000u | f), b.scale, b.add); };
  return make_float3(ch(num & 0x3FFu), ch((num >> 10) & 0x3FFu), ch(num >> 20));
}

// What a texel byte counts: 1/255, channels in [0, 1], or (P64) 1/64, which is exact,
// for readers that take 64/255 into their weights.
template <bool P64>
__device__ __forceinline__ constexpr float texel_unit() {
  return P64 ? 1.0f / 64.0f : 1.0f / 255.0f;
}

// Bilinear sample of one BC1 level at an address_uv coordinate, FP32: the horizontal
// blends of both rows as packed FP32 pairs, then the vertical one.
template <bool P64 = false>
__device__ __forceinline__ float3 sample_bilinear(const LevelView& L, float u, float v, bool wrap) {
  int x0, x1, y0, y1;
  float fx, fy;
  axis_taps(u, L.w, L.shift, wrap, x0, x1, fx);
  axis_taps(v, L.h, L.shift, wrap, y0, y1, fy);
  const uint64_t b00 = __ldg(L.blocks + block_index(L, x0 >> 2, y0 >> 2)), b10 = __ldg(L.blocks + block_index(L, x1 >> 2, y0 >> 2));
  const uint64_t b01 = __ldg(L.blocks + block_index(L, x0 >> 2, y1 >> 2)), b11 = __ldg(L.blocks + block_index(L, x1 >> 2, y1 >> 2));
  const float3 t00 = bc1_texel_f(bc1_block(b00), x0 & 3, y0 & 3), t10 = bc1_texel_f(bc1_block(b10), x1 & 3, y0 & 3);
  const float3 t01 = bc1_texel_f(bc1_block(b01), x0 & 3, y1 & 3), t11 = bc1_texel_f(bc1_block(b11), x1 & 3, y1 & 3);
  const float s = texel_unit<P64>();
  auto blend = [&](float a0, float a1, float c0, float c1) {  // (top, bottom) left and right taps
    const float2 l = make_float2(a0, a1), r = make_float2(c0, c1);
    const float2 d = __fadd2_rn(r, make_float2(-l.x, -l.y));                    // exact
    const float2 z = __fadd2_rn(l, make_float2(-kTexelBase, -kTexelBase));      // exact
    const float2 q = __ffma2_rn(make_float2(fx, fx), d, z);
    return s * fmaf(fy, q.y - q.x, q.x);
  };
  return make_float3(blend(t00.x, t01.x, t10.x, t11.x), blend(t00.y, t01.y, t10.y, t11.y),
                     blend(t00.z, t01.z, t10.z, t11.z));
}

// Arguments shared by the decode kernels (passed by value).
struct DecodeArgs {
  LevelView lv[4];
  int32_t wrap;
  const float* uv;  // NULL = grid mode
  int64_t n;
  int32_t grid_w, grid_h;  // grid mode: texels per row, rows decoded by this call
  int32_t row0;            // grid mode: first row (of the full grid) decoded by this call
  GridCoord cw, ch;        // grid mode: width and height of the full grid (texel-centre coordinates)
  void* out;
  int* status;
};

// uv of output texel t.
__device__ __forceinline__ float2 texel_uv(const DecodeArgs& a, int64_t t) {
  if (a.uv) return __ldg(reinterpret_cast<const float2*>(a.uv) + t);
  int64_t j, i;
  if (a.n <= 0xFFFFFFFFll) {  // 32-bit division when the grid allows it
    const uint32_t tj = (uint32_t)t / (uint32_t)a.grid_w;
    j = tj;
    i = (uint32_t)t - tj * (uint32_t)a.grid_w;
  } else {
    j = t / a.grid_w;
    i = t - j * a.grid_w;
  }
  return make_float2(grid_coord((float)i, a.cw), grid_coord((float)(j + a.row0), a.ch));
}

}  // namespace nbtc
