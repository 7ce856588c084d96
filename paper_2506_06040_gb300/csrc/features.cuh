// Feature stage shared by the tiled decode kernels: the 12 latent features
// (4 levels x RGB, Sec. 3.1) of a tile of consecutive output texels, computed
// by a group of NT threads (thread t owns texel tile_start + t).
//
// Row-footprint mode (texel-centre grid, tile inside one output row, every
// latent level no wider than the output): the output row samples each level
// at one vertical position, so the group decodes only the latent columns the
// tile touches -- two BC1 texels per column (rows y0, y1), blended vertically
// once -- into shared memory; each texel then blends its two neighbouring
// columns horizontally.  This is the bilinear filter of Sec. 3.1 evaluated in
// separable order, with every BC1 block decoded once per tile instead of once
// per tap.  The tensor-core kernels take it a warp at a time with a column cache over
// rows, the last strip past the row's end (see strip_grid in decode_tc.cu).  Direct
// mode (uv lists, grids too narrow for that, rows that 256 does not divide in the
// FFMA kernel, footprints wider than the group) samples each texel on its own.
#pragma once

#include <climits>

#include "common.cuh"
#include "fastdiv.h"
#include "sm100.cuh"

namespace nbtc {

constexpr int kColCap = 136;  // columns per level per group (>= 128 + 2)

__device__ __forceinline__ int wrap_or_clamp(int x, int n, bool wrap) {
  if (wrap) {
    x %= n;
    return x < 0 ? x + n : x;
  }
  return min(max(x, 0), n - 1);
}

// Texel coordinate along one axis, unwrapped: t = u * n - 0.5 + shift.
__device__ __forceinline__ float texel_coord(float u, int n, float shift) {
  return fmaf(u, (float)n, shift - 0.5f);
}

template <typename T>
__device__ __forceinline__ T pick4(const T (&v)[4], int k) {
  return k == 0 ? v[0] : k == 1 ? v[1] : k == 2 ? v[2] : v[3];
}

// ---- row-footprint feature stage in three steps, so a tile's block loads can
// be issued long before they are decoded:
//   plan      per-level column range of the tile (every thread, identical)
//   prefetch  thread `tid` issues the two block loads of column job `tid`
//   decode    the prefetched (and any further) columns -> colbuf
//   blend     after a group barrier, each texel blends its two columns

struct TilePlan {
  int j, i0;
  int base[4], span[4], pre[4];
  int total;
};

template <int NT>
__device__ __forceinline__ TilePlan plan_tile(const DecodeArgs& a, int64_t tile_start) {
  TilePlan P;
  if (tile_start <= 0xFFFFFFFFll) {
    P.j = (int)((uint32_t)tile_start / (uint32_t)a.grid_w);
    P.i0 = (int)((uint32_t)tile_start - (uint32_t)P.j * (uint32_t)a.grid_w);
  } else {
    P.j = (int)(tile_start / a.grid_w);
    P.i0 = (int)(tile_start - (int64_t)P.j * a.grid_w);
  }
  const float u0 = grid_coord((float)P.i0, a.cw);
  const float u1 = grid_coord((float)(P.i0 + NT - 1), a.cw);
  int total = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int b0 = (int)floorf(texel_coord(u0, a.lv[k].w, a.lv[k].shift));
    const int b1 = (int)floorf(texel_coord(u1, a.lv[k].w, a.lv[k].shift));
    P.base[k] = b0;
    P.pre[k] = total;
    P.span[k] = min(b1 - b0 + 2, kColCap);
    total += P.span[k];
  }
  P.total = total;
  return P;
}

// Texel coordinates of column job `job` (< P.total): level, column slot, the
// two texels (x, y0) and (x, y1) and the vertical weight.
struct ColumnJob {
  int k, rel, x, y0, y1;
  float fy;
};

__device__ __forceinline__ ColumnJob column_job(const DecodeArgs& a, const TilePlan& P, int job) {
  ColumnJob J;
  J.k = (job >= P.pre[1]) + (job >= P.pre[2]) + (job >= P.pre[3]);
  J.rel = job - pick4(P.pre, J.k);
  const LevelView& L = a.lv[J.k];
  const float v = grid_coord((float)(P.j + a.row0), a.ch);
  const float ty = texel_coord(v, L.h, L.shift);
  const float fty = floorf(ty);
  J.fy = ty - fty;
  J.y0 = wrap_or_clamp((int)fty, L.h, a.wrap);
  J.y1 = wrap_or_clamp((int)fty + 1, L.h, a.wrap);
  J.x = wrap_or_clamp(pick4(P.base, J.k) + J.rel, L.w, a.wrap);
  return J;
}

struct BlockPair {
  uint64_t b0, b1;
};

__device__ __forceinline__ BlockPair load_column(const DecodeArgs& a, const ColumnJob& J) {
  const LevelView& L = a.lv[J.k];
  BlockPair B;
  B.b0 = __ldg(L.blocks + block_index(L, J.x >> 2, J.y0 >> 2));
  B.b1 = __ldg(L.blocks + block_index(L, J.x >> 2, J.y1 >> 2));
  return B;
}

__device__ __forceinline__ void store_column(float4* colbuf, const ColumnJob& J, const BlockPair& B) {
  const uint32_t t0 = bc1_texel(B.b0, J.x & 3, J.y0 & 3);
  const uint32_t t1 = bc1_texel(B.b1, J.x & 3, J.y1 & 3);
  const float fy = J.fy;
  float4 c;
  c.x = fmaf(fy, (float)((t1 >> 0) & 255u) - (float)((t0 >> 0) & 255u), (float)((t0 >> 0) & 255u));
  c.y = fmaf(fy, (float)((t1 >> 8) & 255u) - (float)((t0 >> 8) & 255u), (float)((t0 >> 8) & 255u));
  c.z = fmaf(fy, (float)((t1 >> 16) & 255u) - (float)((t0 >> 16) & 255u), (float)((t0 >> 16) & 255u));
  c.w = 0.f;
  colbuf[J.k * kColCap + J.rel] = c;
}

// Issues the loads of column job `tid` (if any); returns them unconsumed.
__device__ __forceinline__ BlockPair prefetch_columns(const DecodeArgs& a, const TilePlan& P, int tid) {
  BlockPair B{0, 0};
  if (tid < P.total) B = load_column(a, column_job(a, P, tid));
  return B;
}

// Decodes column job `tid` from its prefetched blocks, and any further jobs
// (tid + NT, ...) with fresh loads, into colbuf.
template <int NT>
__device__ __forceinline__ void decode_columns(const DecodeArgs& a, const TilePlan& P, int tid, const BlockPair& pf,
                                               float4* colbuf) {
  if (tid < P.total) store_column(colbuf, column_job(a, P, tid), pf);
  for (int job = tid + NT; job < P.total; job += NT) {
    const ColumnJob J = column_job(a, P, job);
    store_column(colbuf, J, load_column(a, J));
  }
}

// Horizontal blend of texel tid from the decoded columns (after a barrier).
template <int NT>
__device__ __forceinline__ void blend_columns(const DecodeArgs& a, const TilePlan& P, int tid, const float4* colbuf,
                                              float (&feat)[12]) {
  const float u = grid_coord((float)(P.i0 + tid), a.cw);
  const float s = 1.0f / 255.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float tx = texel_coord(u, a.lv[k].w, a.lv[k].shift);
    const float ftx = floorf(tx);
    const float fx = tx - ftx;
    // floor is monotone in u, so rel lies in [0, span - 2]; the clamp only guards the buffer
    const int rel = min(max((int)ftx - P.base[k], 0), P.span[k] - 2);
    const float4 A = colbuf[k * kColCap + rel];
    const float4 B = colbuf[k * kColCap + rel + 1];
    feat[3 * k + 0] = s * fmaf(fx, B.x - A.x, A.x);
    feat[3 * k + 1] = s * fmaf(fx, B.y - A.y, A.y);
    feat[3 * k + 2] = s * fmaf(fx, B.z - A.z, A.z);
  }
}

// All three steps back to back (one group barrier): features of texel
// tile_start + tid of a tile lying in one output row.
template <int NT>
__device__ __forceinline__ void footprint_features(const DecodeArgs& a, int64_t tile_start, int tid,
                                                   float4* colbuf, int bar_id, float (&feat)[12]) {
  const TilePlan P = plan_tile<NT>(a, tile_start);
  const BlockPair pf = prefetch_columns(a, P, tid);
  decode_columns<NT>(a, P, tid, pf, colbuf);
  sm100::named_bar_sync(bar_id, NT);
  blend_columns<NT>(a, P, tid, colbuf, feat);
}

// ---- column cache of a warp that decodes vertically consecutive tiles of one column
// strip (the same first column i0, output rows j, j+1, ...).  Across such tiles the
// column plan, each lane's column job and each texel's horizontal taps stay
// fixed, and a latent column's two vertical taps (rows floor(ty), floor(ty)+1)
// change only when ty crosses a texel boundary: every 4th output row for a
// latent at 1/4 of the output side, every 32nd at 1/32.  So each lane keeps
// its job's two decoded texels (as floats) and reloads and decodes the BC1 blocks
// only when floor(ty) changes; per tile it only redoes the vertical blend of its
// column and the horizontal blend of its texel.
struct StripCache {
  int i0;          // first output column of the cached strip (-1: none)
  int total;       // column jobs of the strip
  int job;         // own job: level | column of the level << 2 (-1: none)
  int jx;          // own job: latent column (wrapped or clamped)
  int key;         // floor(ty) of the decoded pair (INT_MIN + 1: none)
  uint32_t rel4;   // own texel: lane that holds its left tap, per level, 8 bits each
  float fx[4];     // own texel: horizontal weight per level
  uint32_t t1;     // own job: RGB8 of texel (jx, y1) -- the next pair's (jx, y0) when the key steps by one
  float c0[3];     // own job: texel (jx, y0), RGB in texel units
  float dc[3];     // own job: texel (jx, y1) minus texel (jx, y0)
  float hf, ys;    // own job: the level's height and shift - 1/2
};

__device__ __forceinline__ void strip_reset(StripCache& C) { C.i0 = -1; }

// ---- row-footprint feature stage of one warp, with the latent columns shared
// between its lanes by shuffles.  The warp's 32 consecutive texels of one
// output row read at most ceil(31 W_k / W_out) + 2 columns of level k: 23 jobs
// over the four levels of the 1/4..1/32 pyramid, 32 for 1/4, 1/4, 1/8, 1/8.
// Lane L owns column job L (the strip cache above, per warp: it keeps its two
// decoded texels across rows and re-decodes only when the vertical tap pair
// moves), blends them vertically once per row, and each texel reads its two
// horizontal neighbours from the lanes that hold them -- no shared memory and
// no barrier across warps.  A footprint of more than 32 jobs (level-to-output
// ratios above ~1/4) samples each texel on its own.
template <bool P64 = false>
__device__ __forceinline__ void direct_features(const DecodeArgs& a, int64_t t, float (&feat)[12]);

template <bool P64>
__device__ __forceinline__ void warp_strip_features(const DecodeArgs& a, int j, int i0w, int lane, StripCache& C,
                                                    float (&feat)[12]) {
  const float s = texel_unit<P64>();
  if (i0w != C.i0) {  // new strip: the warp's column plan, own job, own texel's source lanes
    C.i0 = i0w;
    C.key = INT_MIN + 1;
    const float u0 = grid_coord((float)i0w, a.cw);
    const float u1 = grid_coord((float)(i0w + 31), a.cw);
    const float u = grid_coord((float)(i0w + lane), a.cw);
    int total = 0, job = -1, jx = 0;
    uint32_t src4 = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const LevelView& L = a.lv[k];
      const int b0 = (int)floorf(texel_coord(u0, L.w, L.shift));
      const int b1 = (int)floorf(texel_coord(u1, L.w, L.shift));
      const int span = b1 - b0 + 2;
      if (lane >= total && lane < total + span) {
        job = k | (lane - total) << 2;
        jx = wrap_or_clamp(b0 + lane - total, L.w, a.wrap);
        C.hf = (float)L.h;
        C.ys = L.shift - 0.5f;
      }
      const float tx = texel_coord(u, L.w, L.shift);
      const float ftx = floorf(tx);
      C.fx[k] = tx - ftx;
      // floor is monotone in u, so the left tap's job lies in [0, span - 2]; the clamp only guards the lanes
      src4 |= (uint32_t)min(total + min(max((int)ftx - b0, 0), span - 2), 30) << (8 * k);
      total += span;
    }
    C.total = total;
    C.job = job;
    C.jx = jx;
    C.rel4 = src4;
  }
  if (C.total > 32) {  // warp-uniform: a footprint wider than the warp's lanes
    direct_features<P64>(a, (int64_t)j * a.grid_w + i0w + lane, feat);
    return;
  }
  float cv0 = 0.f, cv1 = 0.f, cv2 = 0.f;
  const float v = grid_coord((float)(j + a.row0), a.ch);
  if (C.job >= 0) {
    const float ty = fmaf(v, C.hf, C.ys);
    const float fty = floorf(ty);
    const float fy = ty - fty;
    const int key = (int)fty;
    if (key != C.key) {
      const LevelView& L = a.lv[C.job & 3];
      uint32_t t0;
      if (key == C.key + 1) {
        t0 = C.t1;
      } else {
        const int y0 = wrap_or_clamp(key, L.h, a.wrap);
        t0 = bc1_texel(__ldg(L.blocks + block_index(L, C.jx >> 2, y0 >> 2)), C.jx & 3, y0 & 3);
      }
      const int y1 = wrap_or_clamp(key + 1, L.h, a.wrap);
      const uint32_t t1 = bc1_texel(__ldg(L.blocks + block_index(L, C.jx >> 2, y1 >> 2)), C.jx & 3, y1 & 3);
      // the next pair's lower texel: its block into L1 now, rows before it is read
      const int y2 = wrap_or_clamp(key + 2, L.h, a.wrap);
      if ((y2 ^ y1) >> 2) sm100::prefetch_l1(L.blocks + block_index(L, C.jx >> 2, y2 >> 2));
      C.key = key;
      C.t1 = t1;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float v0 = (float)((t0 >> (8 * c)) & 255u), v1 = (float)((t1 >> (8 * c)) & 255u);
        C.c0[c] = s * v0;
        C.dc[c] = s * (v1 - v0);
      }
    }
    cv0 = fmaf(fy, C.dc[0], C.c0[0]);
    cv1 = fmaf(fy, C.dc[1], C.c0[1]);
    cv2 = fmaf(fy, C.dc[2], C.c0[2]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int src = (C.rel4 >> (8 * k)) & 255;
    const float a0 = __shfl_sync(0xffffffffu, cv0, src), b0 = __shfl_sync(0xffffffffu, cv0, src + 1);
    const float a1 = __shfl_sync(0xffffffffu, cv1, src), b1 = __shfl_sync(0xffffffffu, cv1, src + 1);
    const float a2 = __shfl_sync(0xffffffffu, cv2, src), b2 = __shfl_sync(0xffffffffu, cv2, src + 1);
    feat[3 * k + 0] = fmaf(C.fx[k], b0 - a0, a0);
    feat[3 * k + 1] = fmaf(C.fx[k], b1 - a1, a1);
    feat[3 * k + 2] = fmaf(C.fx[k], b2 - a2, a2);
  }
}

// Per-material description used by the batched and frame decodes: the level
// views of mip 0 (in `d`) plus every level's mip chain for trilinear sampling.
struct MatDev {
  DecodeArgs d;          // mip-0 views, wrap flag, output grid and buffer of the full decode
  const void* packed;    // FP16 packed MLP
  int nout;
  FastDiv hdiv;          // full decode: division by grid_h (tile number -> column block)
  int64_t tiles;         // full decode: tiles of the grid
  int mips[4];
  float log2w[4];        // log2 of each level's mip-0 width
  int mip_off[4][16];    // block offset of mip m of level k
  // frame: every mip's texels decoded to RGBA8 (k_frame_texels), mip m of level k
  // at texel 16 mip_off[k][m]; NULL when the plan decodes BC1 at the taps
  const uint32_t* tex[4];
};

__device__ __forceinline__ LevelView mip_view(const MatDev& M, int k, int m) {
  LevelView v = M.d.lv[k];
  v.blocks = v.blocks + M.mip_off[k][m];
  v.w = max(4, v.w >> m);
  v.h = max(4, v.h >> m);
  v.wb = v.w / 4;
  return v;
}

// Features of one texel sampled on its own (any uv).
template <bool P64>
__device__ __forceinline__ void direct_features(const DecodeArgs& a, int64_t t, float (&feat)[12]) {
  const float2 tuv = texel_uv(a, t), uv = address_uv(tuv.x, tuv.y, a.wrap);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float3 c = sample_bilinear<P64>(a.lv[k], uv.x, uv.y, a.wrap);
    feat[3 * k + 0] = c.x;
    feat[3 * k + 1] = c.y;
    feat[3 * k + 2] = c.z;
  }
}

}  // namespace nbtc
