// Batched multi-material decode and the frame pipeline of Sec. 4 /
// Algorithm 1, around the persistent tensor-core decode kernel.
//
// Plan: materials' FP16 MLPs packed once, a device table of per-material
// views (MatDev), a cost-sorted list of work chunks (runs of 128-texel tiles of
// one material) for the full decode, and the frame buffers.  The decode kernel
// takes chunks from an atomic counter, so materials of very different sizes
// share the SMs evenly; a CTA reloads an MLP only when its next chunk belongs
// to another material.
//
// Frame: pass A (k_frame_classify) marks each 128-pixel tile uniform or mixed
// and counts, per material, uniform tiles and valid pixels of mixed tiles
// (per-CTA shared-memory histograms, then one global atomic per CTA and material
// -- the paper suggests shared-memory atomics for this, Sec. 6 -- whose old
// value is the CTA's place in the material's list); k_frame_scan turns the counts
// into slot offsets (an exclusive prefix sum; Algorithm 1 reads these offsets but
// does not say how they are made) and into the chunk list, while its other CTAs
// decode the visible materials' latent texels (see frame_texels_rule); pass B
// (k_frame_bin) appends uniform tiles to their material's list and packs
// mixed-tile pixels into their material's 128-slot tiles.  k_frame_features
// (frame_features.cu) leaves every pixel's features, and the decode kernel runs
// over the chunks.  All the launches are captured in one CUDA graph.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "frame_slots.h"
#include "host.h"
#include "tc.cuh"

namespace nbtc {

constexpr int kMaxMaterials = 1024;
// Warpgroups of the batched decode and the frame decode, one TMEM slot each (3 or 4 of
// two shared-memory slots were 10 to 25% behind in every plan timed).
constexpr int kBatchW = 4;
constexpr int kClassifyPerSm = 8;  // the classification's CTAs on each SM, each with a run of tiles

enum TileKind { kTileEmpty = 0, kTileUniform = 1, kTileMixed = 2 };

struct FrameDev {
  const int* mat_id;
  int w, h, tw, th, tiles_x, tiles;
  int nmat;
  int* tkind;
  int* tmat;
  int* ucount;   // uniform tiles per material
  int* pcount;   // valid pixels of mixed tiles per material
  int* ubase;    // [ctas][nmat] place of each CTA's uniform tiles in its material's list
  int* pbase;    // [ctas][nmat] the same for the pixels of mixed tiles
  int* uoff;     // first slot in ulist
  int* poff;     // first packed tile
  int* ulist;
  int* plist;
  WorkChunk* chunks;
  int* nchunks;
  int* counter;  // next chunk of the decode kernel (zeroed by the scan)
  int chunk_cap;
  int decode_ctas;  // CTAs of the decode kernel
  int max_ctas;     // at most so many CTAs of the classification and the binning, each with a run of tiles
  int ctas;         // those of the tile shape
  int per_cta;      // tiles of a run
  int ids16;        // mat_id may be read four pixels at a time
  int* stats;    // [uniform tiles, mixed tiles, packed tiles]
  int64_t ulist_cap, plist_cap;  // slots of ulist and plist (bounds of the checked build)
  int* status;                   // context status word (checked build)
};

// Pixel j (0..127) of screen tile t.
__device__ __forceinline__ int tile_pixel(const FrameDev& F, int t, int j) {
  const int ty = t / F.tiles_x, tx = t - ty * F.tiles_x;
  const int r = j / F.tw;
  return (ty * F.th + r) * F.w + tx * F.tw + (j - r * F.tw);
}

// Material ids of the four pixels px .. px + 3 (one row of a tile; tile widths are
// multiples of 4).  Ids past the table decode as "no material".
__device__ __forceinline__ void tile_ids(const FrameDev& F, int px, int (&ids)[4]) {
  if (F.ids16) {
    const int4 q = __ldg(reinterpret_cast<const int4*>(F.mat_id + px));
    ids[0] = q.x;
    ids[1] = q.y;
    ids[2] = q.z;
    ids[3] = q.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) ids[i] = __ldg(F.mat_id + px + i);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (ids[i] < 0 || ids[i] >= F.nmat) ids[i] = -1;
}

// Pass A: one warp per tile, 4 pixels per lane; a CTA takes a run of tiles and
// touches global memory with one atomic per material it met (one per tile had
// made it a queue at two addresses: 71 us for 65k tiles, 14 us now).
__global__ void __launch_bounds__(256) k_frame_classify(FrameDev F) {
  extern __shared__ int hist[];  // [nmat] uniform tiles, [nmat] pixels of mixed tiles, [2] tiles of each kind
  int* hu = hist;
  int* hp = hist + F.nmat;
  int* hk = hist + 2 * F.nmat;
  for (int m = threadIdx.x; m < 2 * F.nmat + 2; m += blockDim.x) hist[m] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int first = blockIdx.x * F.per_cta, last = min(first + F.per_cta, F.tiles);
  for (int t = first + threadIdx.x / 32; t < last; t += blockDim.x / 32) {
    int ids[4];
    tile_ids(F, tile_pixel(F, t, lane * 4), ids);
    int cnt = 0, mn = 0x7fffffff, mx = -1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (ids[i] >= 0) {
        ++cnt;
        mn = min(mn, ids[i]);
        mx = max(mx, ids[i]);
      }
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    const int kind = cnt == 0 ? kTileEmpty : (mn == mx && 2 * cnt > kTileK ? kTileUniform : kTileMixed);
    if (lane == 0) {
      F.tkind[t] = kind;
      F.tmat[t] = kind == kTileUniform ? mn : -1;
      if (kind == kTileUniform) {
        atomicAdd_block(hu + mn, 1);
        atomicAdd_block(hk + 0, 1);
      }
      if (kind == kTileMixed) atomicAdd_block(hk + 1, 1);
    }
    if (kind == kTileMixed) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (ids[i] >= 0) atomicAdd_block(hp + ids[i], 1);
    }
  }
  __syncthreads();
  for (int m = threadIdx.x; m < F.nmat; m += blockDim.x) {
    if (hu[m]) F.ubase[(size_t)blockIdx.x * F.nmat + m] = atomicAdd(F.ucount + m, hu[m]);
    if (hp[m]) F.pbase[(size_t)blockIdx.x * F.nmat + m] = atomicAdd(F.pcount + m, hp[m]);
  }
  if (threadIdx.x < 2 && hk[threadIdx.x]) atomicAdd(F.stats + threadIdx.x, hk[threadIdx.x]);
}

// Exclusive prefix sum of one value per thread over a 256-thread CTA; `total`
// receives the sum.
__device__ __forceinline__ int block_scan(int x, int& total, int* warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  __syncthreads();  // the previous scan's sums have been read
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  int before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w < warp) before += warp_sums[w];
    sum += warp_sums[w];
  }
  total = sum;
  return before + incl - x;
}

// Offsets (exclusive scans) and the chunk list: per material its uniform-tile
// chunks, then its packed-tile chunks.  One 256-thread CTA, `coff` [nmat + 1].
// Every tile costs the decode kernel the same, and a chunk costs it a
// reload of the MLP (~2 us), so chunks are a quarter of a CTA's share of the frame.
__device__ void frame_scan(const FrameDev& F, int* coff, int* warp_sums) {
  const int t = threadIdx.x;
  int tiles = 0;
  for (int m = t; m < F.nmat; m += blockDim.x) tiles += F.ucount[m] + packed_tiles(F.pcount[m]);
  int all = 0;
  block_scan(tiles, all, warp_sums);
  const int chunk = max(16, (all + 4 * F.decode_ctas - 1) / (4 * F.decode_ctas));
  int su = 0, sp = 0, sc = 0;
  for (int m0 = 0; m0 < F.nmat; m0 += (int)blockDim.x) {
    const int m = m0 + t;
    const int U = m < F.nmat ? F.ucount[m] : 0;
    const int px = m < F.nmat ? F.pcount[m] : 0;
    const int P = packed_tiles(px);
    const int C = (U + chunk - 1) / chunk + (P + chunk - 1) / chunk;
    int tu, tp, tc;
    const int u = su + block_scan(U, tu, warp_sums), q = sp + block_scan(P, tp, warp_sums),
              c = sc + block_scan(C, tc, warp_sums);
    if (m < F.nmat) {
      F.uoff[m] = u;
      F.poff[m] = q;
      coff[m] = c;
      const int64_t end = packed_slot(q + P, 0);
      for (int i = free_slots(px); i > 0; --i) F.plist[end - i] = -1;  // the last packed tile's free slots
    }
    su += tu;
    sp += tp;
    sc += tc;
  }
  if (t == 0) {
    coff[F.nmat] = sc;
    *F.nchunks = min(sc, F.chunk_cap);
    *F.counter = 0;
    F.stats[2] = sp;
  }
  __syncthreads();
  for (int c = t; c < min(sc, F.chunk_cap); c += blockDim.x) {
    int lo = 0, hi = F.nmat - 1;  // the material whose chunks hold c: the last m with coff[m] <= c
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (coff[mid] <= c) lo = mid;
      else hi = mid - 1;
    }
    const int m = lo, U = F.ucount[m], P = packed_tiles(F.pcount[m]);
    const int nu = (U + chunk - 1) / chunk;
    int i = c - coff[m];
    if (i < nu) {
      i *= chunk;
      F.chunks[c] = WorkChunk{m, kChunkUniform, (int64_t)F.uoff[m] + i, min(chunk, U - i), 0};
    } else {
      i = (i - nu) * chunk;
      F.chunks[c] = WorkChunk{m, kChunkPacked, (int64_t)F.poff[m] + i, min(chunk, P - i), 0};
    }
  }
}

// Pass B, over the classification's runs of tiles: uniform tiles -> their
// material's list; mixed-tile pixels -> packed slots of their material.  The
// run's places were taken in pass A, so the cursors are shared-memory ones
// (one atomic per material present in a warp).
__global__ void __launch_bounds__(256) k_frame_bin(FrameDev F) {
  extern __shared__ int cur[];  // [nmat] next slot in ulist, [nmat] next place among the material's packed pixels
  int* cu = cur;
  int* cp = cur + F.nmat;
  for (int m = threadIdx.x; m < F.nmat; m += blockDim.x) {  // places of materials the run does not hold are not used
    cu[m] = F.uoff[m] + F.ubase[(size_t)blockIdx.x * F.nmat + m];
    cp[m] = F.pbase[(size_t)blockIdx.x * F.nmat + m];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int first = blockIdx.x * F.per_cta, last = min(first + F.per_cta, F.tiles);
  for (int t = first + threadIdx.x / 32; t < last; t += blockDim.x / 32) {
    const int kind = F.tkind[t];
    if (kind == kTileUniform) {
      if (lane == 0) {
        int64_t slot = atomicAdd_block(cu + F.tmat[t], 1);
        NBTC_CHECK_INDEX(slot, F.ulist_cap, F.status);
        F.ulist[slot] = t;
      }
    } else if (kind == kTileMixed) {
      const int px = tile_pixel(F, t, lane * 4);
      int ids[4];
      tile_ids(F, px, ids);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int id = ids[i];
        const unsigned peers = __match_any_sync(0xffffffffu, id);
        const int leader = __ffs(peers) - 1;
        int base = 0;
        if (id >= 0 && lane == leader) base = atomicAdd_block(cp + id, __popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (id >= 0) {
          int64_t slot = packed_slot(F.poff[id], base + __popc(peers & lt));
          NBTC_CHECK_INDEX(slot, F.plist_cap, F.status);
          F.plist[slot] = px + i;
        }
      }
    }
  }
}

// ---- decoded latent texels of a frame
//
// A run of consecutive BC1 blocks of one material's level (its mips back to back).
struct TexelRun {
  int mat, level;
  int first, count;  // blocks, count <= kTexelRun
};
constexpr int kTexelRun = 256;

// CTA 0: the offsets and the chunk list.  The others, one thread per block of a
// run: the block's four palette colours, then its 16 texels as RGBA8 words, four
// 16-byte row stores (neighbouring threads write neighbouring 16 bytes of a
// row).  Materials without a pixel in this frame (the counts of pass A) are left
// out.  Bound by its writes, 4 bytes per latent texel: the 7.0 M texels of 64
// materials up to 2048^2 take 11 us, the scan included.
__global__ void __launch_bounds__(kTexelRun) k_frame_scan(const TexelRun* __restrict__ runs,
                                                          const MatDev* __restrict__ mats, FrameDev F) {
  extern __shared__ int coff[];
  __shared__ int warp_sums[8];
  if (blockIdx.x == 0) {
    frame_scan(F, coff, warp_sums);
    return;
  }
  const TexelRun R = runs[blockIdx.x - 1];
  if (F.ucount[R.mat] + F.pcount[R.mat] == 0) return;
  if ((int)threadIdx.x >= R.count) return;
  const MatDev& M = mats[R.mat];
  const int g = R.first + (int)threadIdx.x;  // block of the level, over its mips
  int m = 0;
  while (m + 1 < M.mips[R.level] && g >= M.mip_off[R.level][m + 1]) ++m;
  const LevelView V = mip_view(M, R.level, m);
  const int b = g - M.mip_off[R.level][m];
  const int by = b / V.wb, bx = b - by * V.wb;
  const uint64_t blk = __ldg(V.blocks + block_index(V, bx, by));
  const uint32_t c0 = (uint32_t)(blk & 0xFFFFu), c1 = (uint32_t)((blk >> 16) & 0xFFFFu), bits = (uint32_t)(blk >> 32);
  const bool four = c0 > c1;
  int e0[3], e1[3];
  expand565(c0, e0[0], e0[1], e0[2]);
  expand565(c1, e1[0], e1[1], e1[2]);
  uint32_t p[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    p[0] |= (uint32_t)e0[c] << (8 * c);
    p[1] |= (uint32_t)e1[c] << (8 * c);
    p[2] |= (uint32_t)palette_channel(e0[c], e1[c], four ? 2 : 1, 1, four) << (8 * c);
    if (four) p[3] |= (uint32_t)palette_channel(e0[c], e1[c], 1, 2, true) << (8 * c);  // else black
  }
  uint32_t* out = const_cast<uint32_t*>(M.tex[R.level]) + 16 * (int64_t)M.mip_off[R.level][m] +
                  (int64_t)(4 * by) * V.w + 4 * bx;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    uint32_t t[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const uint32_t i = bits >> (2 * (4 * r + x));
      const uint32_t lo = (i & 1u) ? p[1] : p[0], hi = (i & 1u) ? p[3] : p[2];
      t[x] = (i & 2u) ? hi : lo;
    }
    *reinterpret_cast<uint4*>(out + (int64_t)r * V.w) = make_uint4(t[0], t[1], t[2], t[3]);
  }
}

}  // namespace nbtc

using namespace nbtc;

struct nbtc_batch {
  int device = 0;
  int count = 0;
  int nhid = 0;
  int nout = 0;
  std::vector<nbtc_batch_material> host_mats;
  // device buffers
  MatDev* mats_dev = nullptr;
  unsigned char* packed_dev = nullptr;
  size_t packed_stride = 0;
  WorkChunk* dchunks = nullptr;
  int* dnchunks = nullptr;
  int* dcounter = nullptr;
  int64_t decode_tiles = 0;
  // frame
  bool has_frame = false;
  nbtc_frame frame{};
  FrameDev F{};
  int* frame_block = nullptr;  // all int frame buffers
  WorkChunk* fchunks = nullptr;
  int* fcounter = nullptr;
  size_t plist_ints = 0;
  uint32_t* texels = nullptr;  // decoded texels of every material's levels and mips (NULL: BC1 at the taps)
  TexelRun* truns = nullptr;
  FrameLevel* flevels = nullptr;  // the feature pass's view of them
  uint2* ffeat = nullptr;         // per-pixel features of the frame, 24 bytes each
  int ntruns = 0;
  // tuned configuration and graphs
  int chunk = 32, tw = 16, th = 8;
  cudaStream_t cap = nullptr;
  cudaGraphExec_t g_decode = nullptr, g_render = nullptr;
  nbtc_batch_info info{};
};

namespace nbtc {

static nbtc_status upload(void* dst, const void* src, size_t n, cudaStream_t s) {
  return cuda_check(cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, s), "upload");
}

// Host-built chunk list of the full decode: largest materials first, each
// material's tiles in runs of `chunk` tiles (consecutive column-major tile
// numbers, i.e. neighbouring rows of one 128-texel column block).
static std::vector<WorkChunk> decode_chunks(const nbtc_batch* B, int chunk) {
  std::vector<int> order;
  for (int m = 0; m < B->count; ++m)
    if (B->host_mats[m].out) order.push_back(m);
  auto tiles = [&](int m) { return (int64_t)B->host_mats[m].out_w * B->host_mats[m].out_h / kTile; };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return tiles(a) > tiles(b); });
  std::vector<WorkChunk> v;
  for (int m : order)
    for (int64_t i = 0; i < tiles(m); i += chunk)
      v.push_back(WorkChunk{m, kChunkGrid, i, (int)std::min<int64_t>(chunk, tiles(m) - i), 0});
  return v;
}

static TcArgs base_args(nbtc_context* ctx, const nbtc_batch* B) {
  TcArgs p;
  memset(&p, 0, sizeof(p));
  p.d.status = ctx->status_dev;
  p.budget = ctx->wait_budget > 0 ? ctx->wait_budget : ctx->wait_budget < 0 ? 0 : kDefaultWaitBudget;
  p.mode = kModeBatch;
  p.mats = B->mats_dev;
  return p;
}

static nbtc_status enqueue_decode(nbtc_context* ctx, nbtc_batch* B, cudaStream_t s) {
  nbtc_status st = cuda_check(cudaMemsetAsync(B->dcounter, 0, sizeof(int), s), "reset chunk counter");
  if (st) return st;
  TcArgs p = base_args(ctx, B);
  p.chunks = B->dchunks;
  p.nchunks_dev = B->dnchunks;
  p.chunk_counter = B->dcounter;
  p.tmem_a = 1;
  return launch_tc_args(ctx, p, B->nhid, kF16, kBatchW, 1, ctx->sm_count, s);
}

// Lighting constants of a frame: unit directions and the half vector, in double
// before rounding to FP32.
static LightDev make_light(const nbtc_frame& f) {
  LightDev L;
  auto unit = [](const float* a, double* o) {
    const double n = std::sqrt((double)a[0] * a[0] + (double)a[1] * a[1] + (double)a[2] * a[2]);
    for (int i = 0; i < 3; ++i) o[i] = n > 0 ? a[i] / n : (i == 2 ? 1.0 : 0.0);
  };
  double l[3], v[3], h[3];
  unit(f.light_dir, l);
  unit(f.view_dir, v);
  const double hs[3] = {l[0] + v[0], l[1] + v[1], l[2] + v[2]};
  const double hn = std::sqrt(hs[0] * hs[0] + hs[1] * hs[1] + hs[2] * hs[2]);
  double ldoth = 0;
  for (int i = 0; i < 3; ++i) {
    h[i] = hn > 0 ? hs[i] / hn : (i == 2 ? 1.0 : 0.0);
    ldoth += l[i] * h[i];
  }
  for (int i = 0; i < 3; ++i) {
    L.l[i] = (float)l[i];
    L.v[i] = (float)v[i];
    L.h[i] = (float)h[i];
    L.rgb[i] = f.light_rgb[i];
    L.sky[i] = f.sky[i];
    L.ground[i] = f.ground[i];
  }
  L.ldoth = (float)(ldoth > 0 ? ldoth : 0);
  return L;
}

static nbtc_status enqueue_render(nbtc_context* ctx, nbtc_batch* B, cudaStream_t s) {
  FrameDev& F = B->F;
  nbtc_status st;
  const size_t zero_ints = (size_t)2 * F.nmat + 3;  // ucount, pcount, stats are contiguous
  if ((st = cuda_check(cudaMemsetAsync(F.ucount, 0, zero_ints * sizeof(int), s), "reset frame counts"))) return st;
  k_frame_classify<<<F.ctas, 256, (2 * F.nmat + 2) * sizeof(int), s>>>(F);
  if ((st = cuda_check(cudaGetLastError(), "launch k_frame_classify"))) return st;
  k_frame_scan<<<1 + B->ntruns, kTexelRun, (F.nmat + 1) * sizeof(int), s>>>(B->truns, B->mats_dev, F);
  if ((st = cuda_check(cudaGetLastError(), "launch k_frame_scan"))) return st;
  k_frame_bin<<<F.ctas, 256, 2 * F.nmat * sizeof(int), s>>>(F);
  if ((st = cuda_check(cudaGetLastError(), "launch k_frame_bin"))) return st;
  FrameFeatArgs f;
  f.mat_id = F.mat_id;
  f.uv = B->frame.uv;
  f.lod = B->frame.lod;
  f.duv = B->frame.duv;
  f.max_aniso = B->frame.duv ? B->frame.max_aniso : 1;
  f.nmat = F.nmat;
  f.pixels = (int64_t)F.w * F.h;
  f.levels = B->flevels;
  f.mats = B->mats_dev;
  f.feat = B->ffeat;
  f.status = ctx->status_dev;
  f.plant = ctx->check_plant;
  if ((st = launch_frame_features(f, s))) return st;
  TcArgs p = base_args(ctx, B);
  p.chunks = B->fchunks;
  p.nchunks_dev = F.nchunks;
  p.chunk_counter = B->fcounter;
  p.ulist = F.ulist;
  p.plist = F.plist;
  p.fmat = B->frame.mat_id;
  p.ffeat = B->ffeat;
  p.fshade = B->frame.shaded;
  p.light = make_light(B->frame);
  p.fout = static_cast<uint16_t*>(B->frame.out);
  p.frame_w = F.w;
  {  // the pixels of a tile row of one warp are contiguous in the output: bulk copies of whole 16-byte pieces
    const int seg = std::min(32, F.tw);
    p.fseg = aligned(B->frame.out, 16) && (seg * B->nout * 2) % 16 == 0 && ((int64_t)F.tw * B->nout * 2) % 16 == 0 ? seg : 0;
  }
  p.frame_pixels = (int64_t)F.w * F.h;
  p.tile_w = F.tw;
  p.tile_h = F.th;
  p.tiles_x = F.tiles_x;
  p.mode = kModeFrame;
  p.tmem_a = 1;
  return launch_tc_args(ctx, p, B->nhid, kF16, kBatchW, 1, ctx->sm_count, s);
}

static nbtc_status set_tile_shape(nbtc_batch* B, int tw, int th) {
  FrameDev& F = B->F;
  if (F.w % tw || F.h % th) return fail(NBTC_ERR_UNSUPPORTED, "frame size not a multiple of the tile");
  F.tw = tw;
  F.th = th;
  F.tiles_x = F.w / tw;
  F.tiles = F.tiles_x * (F.h / th);
  F.per_cta = std::max(8, (F.tiles + F.max_ctas - 1) / F.max_ctas);  // at least a tile per warp
  F.ctas = (F.tiles + F.per_cta - 1) / F.per_cta;
  B->tw = tw;
  B->th = th;
  return NBTC_OK;
}

static nbtc_status set_decode_chunk(nbtc_batch* B, int chunk, cudaStream_t s) {
  std::vector<WorkChunk> v = decode_chunks(B, chunk);
  const int n = (int)v.size();
  nbtc_status st;
  if (n && (st = upload(B->dchunks, v.data(), v.size() * sizeof(WorkChunk), s))) return st;
  if ((st = upload(B->dnchunks, &n, sizeof(int), s))) return st;
  B->chunk = chunk;
  return cuda_check(cudaStreamSynchronize(s), "chunk upload");
}

// Mean of `reps` timed runs after one warm-up run (CUDA events on `s`).
template <class F>
static float time_ms(F&& run, cudaStream_t s, int reps, nbtc_status& st) {
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  st = run();
  if (!st) st = cuda_check(cudaStreamSynchronize(s), "tune warm-up");
  float ms = 0.f;
  if (!st) {
    cudaEventRecord(a, s);
    for (int i = 0; i < reps && !st; ++i) st = run();
    cudaEventRecord(b, s);
    cudaEventSynchronize(b);
    cudaEventElapsedTime(&ms, a, b);
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  return ms / reps;
}

static nbtc_status capture(nbtc_context* ctx, nbtc_batch* B, bool render, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  // one uncaptured run first: kernel attributes are set outside the capture
  nbtc_status st = render ? enqueue_render(ctx, B, B->cap) : enqueue_decode(ctx, B, B->cap);
  if (!st) st = cuda_check(cudaStreamSynchronize(B->cap), "pre-capture run");
  if (st) return st;
  st = cuda_check(cudaStreamBeginCapture(B->cap, cudaStreamCaptureModeThreadLocal), "begin capture");
  if (st) return st;
  nbtc_status run = render ? enqueue_render(ctx, B, B->cap) : enqueue_decode(ctx, B, B->cap);
  st = cuda_check(cudaStreamEndCapture(B->cap, &g), "end capture");
  if (run) {
    if (g) cudaGraphDestroy(g);
    return run;
  }
  if (st) return st;
  st = cuda_check(cudaGraphInstantiate(out, g, 0), "instantiate graph");
  cudaGraphDestroy(g);
  return st;
}

// Whether a frame of `pixels` decodes its materials' latents (`texels` of them, all
// levels and mips) once per frame instead of at its taps.  Decoding a texel and
// keeping it in HBM costs 4 bytes of writes, a tap of a BC1 texel ~45 instructions
// more than one of a decoded texel, at 32 taps a pixel and more: up to 16 texels
// a pixel (64 bytes; 0.5 GB for a 3840 x 2160 frame) decoding first is far
// ahead, and the bound keeps a small frame of very many large materials from
// holding, and filling, gigabytes.  The decoded taps wrap a texel index by one
// period, so shifts beyond half a texel stay with the general path.
static bool frame_texels_rule(const std::vector<MatDev>& md, int64_t texels, int64_t pixels) {
  for (const MatDev& d : md)
    for (int k = 0; k < 4; ++k)
      if (!(std::fabs(d.d.lv[k].shift) <= 0.5f) || d.mip_off[k][NBTC_MAX_MIPS - 1] > (1 << 26)) return false;
  return texels <= 16 * pixels;
}

static void free_plan(nbtc_batch* B) {
  if (!B) return;
  cudaSetDevice(B->device);
  cudaDeviceSynchronize();
  if (B->g_decode) cudaGraphExecDestroy(B->g_decode);
  if (B->g_render) cudaGraphExecDestroy(B->g_render);
  if (B->cap) cudaStreamDestroy(B->cap);
  cudaFree(B->mats_dev);
  cudaFree(B->packed_dev);
  cudaFree(B->dchunks);
  cudaFree(B->dnchunks);
  cudaFree(B->dcounter);
  cudaFree(B->frame_block);
  cudaFree(B->texels);
  cudaFree(B->truns);
  cudaFree(B->flevels);
  cudaFree(B->ffeat);
  cudaFree(B->fchunks);
  cudaFree(B->fcounter);
  delete B;
}

}  // namespace nbtc

extern "C" {

nbtc_status nbtc_batch_create(nbtc_context* ctx, const nbtc_batch_material* mats, int32_t count,
                              const nbtc_frame* frame, int32_t flags, nbtc_batch** plan, void* stream) {
  NBTC_RANGE();
  nbtc_status st = enter(ctx);
  if (st) return st;
  if (!plan || !mats || count < 1 || count > kMaxMaterials)
    return fail(NBTC_ERR_INVALID_ARG, "plan/mats NULL or count outside 1..1024");
  *plan = nullptr;
  cudaStream_t s = (cudaStream_t)stream;
  // ---- validate
  int nhid = -1, nout = -1;
  for (int m = 0; m < count; ++m) {
    const nbtc_batch_material& M = mats[m];
    if ((st = check_mlp(&M.mlp))) return st;
    if (M.latents.num_levels != 4) return fail(NBTC_ERR_UNSUPPORTED, "batched materials take 4 latent levels");
    LevelView lv[NBTC_MAX_LEVELS];
    if ((st = make_level_views(&M.latents, 0, lv))) return st;
    if ((st = need_inputs(&M.latents, &M.mlp))) return st;
    size_t pb = 0;
    if ((st = tc_packed_bytes(&M.mlp, NBTC_FP16, &pb))) return st;
    const int h = M.mlp.num_layers - 1, c = M.mlp.dims[M.mlp.num_layers];
    if (nhid < 0) {
      nhid = h;
      nout = c;
    } else if (h != nhid || c != nout) {
      return fail(NBTC_ERR_UNSUPPORTED, "every material needs the same MLP depth and output channels");
    }
    if (M.out) {
      if (M.out_w <= 0 || M.out_h <= 0 || M.out_w % kTile) return fail(NBTC_ERR_INVALID_ARG, "out_w must be a positive multiple of 128");
      if ((int64_t)M.out_w * M.out_h / kTile >= (int64_t)1 << 31) return fail(NBTC_ERR_UNSUPPORTED, "material output too large");
      if (!aligned(M.out, 16)) return fail(NBTC_ERR_INVALID_ARG, "material out not 16-byte aligned");
      if ((st = need_device(M.out, "material out"))) return st;  // written with bulk copies
      for (int k = 0; k < 4; ++k)
        if (M.latents.levels[k].width > M.out_w) return fail(NBTC_ERR_UNSUPPORTED, "latent level wider than the output");
    }
  }
  if (frame) {
    if (frame->width <= 0 || frame->height <= 0 || !frame->mat_id || !frame->uv || !frame->lod || !frame->out)
      return fail(NBTC_ERR_INVALID_ARG, "frame buffers NULL or size <= 0");
    if (!aligned(frame->uv, 8)) return fail(NBTC_ERR_INVALID_ARG, "frame uv not 8-byte aligned");
    if (frame->duv && (!aligned(frame->duv, 16) || frame->max_aniso < 1 || frame->max_aniso > 16))
      return fail(NBTC_ERR_INVALID_ARG, "frame duv not 16-byte aligned or max_aniso outside 1..16");
    if (frame->shaded && !aligned(frame->shaded, 16))
      return fail(NBTC_ERR_INVALID_ARG, "frame shaded output not 16-byte aligned");
    if (frame->shaded && nout < 8) return fail(NBTC_ERR_UNSUPPORTED, "the lighting pass needs at least 8 channels");
    if ((st = need_readable(frame->mat_id, "frame mat_id")) || (st = need_readable(frame->uv, "frame uv")) ||
        (st = need_readable(frame->lod, "frame lod")) || (frame->duv && (st = need_readable(frame->duv, "frame duv"))) ||
        (st = need_device(frame->out, "frame out")) || (frame->shaded && (st = need_device(frame->shaded, "frame shaded"))))
      return st;
    if ((int64_t)frame->width * frame->height >= (int64_t)1 << 31) return fail(NBTC_ERR_UNSUPPORTED, "frame too large");
  }
  nbtc_batch* B = new nbtc_batch();
  B->device = ctx->device;
  B->count = count;
  B->nhid = nhid;
  B->nout = nout;
  B->host_mats.assign(mats, mats + count);
#define NBTC_TRY(x)     \
  do {                  \
    st = (x);           \
    if (st) {           \
      free_plan(B);     \
      return st;        \
    }                   \
  } while (0)
  NBTC_TRY(cuda_check(cudaStreamCreateWithFlags(&B->cap, cudaStreamNonBlocking), "plan stream"));
  // ---- packed MLPs and the material table
  size_t pb = 0;
  tc_packed_bytes(&mats[0].mlp, NBTC_FP16, &pb);
  B->packed_stride = (pb + 255) & ~(size_t)255;
  NBTC_TRY(cuda_check(cudaMalloc(&B->packed_dev, B->packed_stride * count), "plan MLPs"));
  std::vector<MatDev> md(count);
  for (int m = 0; m < count; ++m) {
    const nbtc_batch_material& M = mats[m];
    NBTC_TRY(launch_pack_mlp(ctx, &M.mlp, NBTC_FP16, nullptr, B->packed_dev + B->packed_stride * m, pb, s));
    MatDev& d = md[m];
    memset(&d, 0, sizeof(d));
    make_level_views(&M.latents, 0, d.d.lv);
    attach_checks(ctx, d.d.lv, 4);
    d.d.wrap = M.latents.address == NBTC_WRAP;
    d.d.grid_w = M.out ? M.out_w : 0;
    d.d.grid_h = M.out ? M.out_h : 0;
    d.d.n = M.out ? (int64_t)M.out_w * M.out_h : 0;
    d.d.cw = make_grid_coord(M.out ? M.out_w : 1);
    d.d.ch = make_grid_coord(M.out ? M.out_h : 1);
    d.d.out = M.out;
    d.d.status = ctx->status_dev;
    d.packed = B->packed_dev + B->packed_stride * m;
    d.nout = nout;
    d.hdiv = make_fastdiv(M.out ? (uint32_t)M.out_h : 1u);
    d.tiles = d.d.n / kTile;
    B->decode_tiles += d.tiles;
    for (int k = 0; k < 4; ++k) {
      const nbtc_level& Lv = M.latents.levels[k];
      d.mips[k] = Lv.num_mips;
      d.log2w[k] = (float)std::log2((double)Lv.width);
      int w = Lv.width, h = Lv.height, off = 0;
      for (int mm = 0; mm < NBTC_MAX_MIPS; ++mm) {
        d.mip_off[k][mm] = off;
        off += (w / 4) * (h / 4);
        w = std::max(4, w / 2);
        h = std::max(4, h / 2);
      }
    }
  }
  // ---- frame: decoded texels of every level and its mips, and the runs of blocks that fill them
  if (frame) {
    int64_t texels = 0;
    auto level_blocks = [&](int m, int k) {
      const MatDev& d = md[m];
      const nbtc_level& Lv = mats[m].latents.levels[k];
      const int last = d.mips[k] - 1;
      return d.mip_off[k][last] + (std::max(4, Lv.width >> last) / 4) * (std::max(4, Lv.height >> last) / 4);
    };
    for (int m = 0; m < count; ++m)
      for (int k = 0; k < 4; ++k) texels += 16 * (int64_t)level_blocks(m, k);
    NBTC_TRY(cuda_check(cudaMalloc(&B->ffeat, (size_t)frame->width * frame->height * 3 * sizeof(uint2)), "frame features"));
    if (frame_texels_rule(md, texels, (int64_t)frame->width * frame->height)) {
      const cudaError_t e = cudaMalloc(&B->texels, (size_t)texels * sizeof(uint32_t));
      if (e == cudaErrorMemoryAllocation) {  // no room for them: BC1 at the taps, which needs none
        cudaGetLastError();
        B->texels = nullptr;
      } else {
        NBTC_TRY(cuda_check(e, "frame texels"));
      }
    }
    if (B->texels) {
      std::vector<TexelRun> runs;
      std::vector<FrameLevel> levels((size_t)count * 4);
      int64_t at = 0;
      for (int m = 0; m < count; ++m)
        for (int k = 0; k < 4; ++k) {
          const int n = level_blocks(m, k);
          md[m].tex[k] = B->texels + at;
          for (int i = 0; i < n; i += kTexelRun) runs.push_back(TexelRun{m, k, i, std::min(kTexelRun, n - i)});
          FrameLevel& fl = levels[(size_t)m * 4 + k];
          memset(&fl, 0, sizeof(fl));
          fl.base = md[m].tex[k];
          fl.log2w = md[m].log2w[k];
          fl.shift = md[m].d.lv[k].shift;
          fl.last = (float)(md[m].mips[k] - 1);
          fl.wrap = md[m].d.wrap;
          for (int i = 0; i < md[m].mips[k]; ++i)
            fl.mip[i] = FrameMip{16u * (uint32_t)md[m].mip_off[k][i], std::max(4, md[m].d.lv[k].w >> i),
                                 std::max(4, md[m].d.lv[k].h >> i), 0};
          at += 16 * (int64_t)n;
        }
      B->ntruns = (int)runs.size();
      NBTC_TRY(cuda_check(cudaMalloc(&B->truns, sizeof(TexelRun) * runs.size()), "texel runs"));
      NBTC_TRY(upload(B->truns, runs.data(), sizeof(TexelRun) * runs.size(), s));
      NBTC_TRY(cuda_check(cudaMalloc(&B->flevels, sizeof(FrameLevel) * levels.size()), "frame levels"));
      NBTC_TRY(upload(B->flevels, levels.data(), sizeof(FrameLevel) * levels.size(), s));
    }
  }
  NBTC_TRY(cuda_check(cudaMalloc(&B->mats_dev, sizeof(MatDev) * count), "plan table"));
  NBTC_TRY(upload(B->mats_dev, md.data(), sizeof(MatDev) * count, s));
  // ---- full-decode work list (largest chunk count over the candidate chunk sizes)
  const size_t max_chunks = decode_chunks(B, 8).size() + 1;
  NBTC_TRY(cuda_check(cudaMalloc(&B->dchunks, sizeof(WorkChunk) * max_chunks), "decode chunks"));
  NBTC_TRY(cuda_check(cudaMalloc(&B->dnchunks, sizeof(int)), "decode chunk count"));
  NBTC_TRY(cuda_check(cudaMalloc(&B->dcounter, sizeof(int)), "decode counter"));
  NBTC_TRY(set_decode_chunk(B, 32, s));
  // ---- frame buffers
  if (frame) {
    B->has_frame = true;
    B->frame = *frame;
    FrameDev& F = B->F;
    F.mat_id = frame->mat_id;
    F.w = frame->width;
    F.h = frame->height;
    F.nmat = count;
    F.decode_ctas = ctx->sm_count;
    F.max_ctas = kClassifyPerSm * ctx->sm_count;
    F.ids16 = aligned(frame->mat_id, 16) && frame->width % 4 == 0;
    const int pixels = frame->width * frame->height;
    const int max_tiles = pixels / kTileK + 1;
    B->plist_ints = (size_t)(pixels / kTileK + count + 1) * kTileK;
    const size_t runs = std::min(F.max_ctas, max_tiles / 8 + 1);
    const size_t ints = (size_t)2 * count + 3 /* counts + stats */ + 2 * (size_t)count /* offsets */ +
                        2 * runs * count /* places */ + 2 * (size_t)max_tiles /* kind, mat */ + max_tiles /* ulist */ +
                        B->plist_ints + 1;
    NBTC_TRY(cuda_check(cudaMalloc(&B->frame_block, ints * sizeof(int)), "frame buffers"));
    int* q = B->frame_block;
    F.ucount = q; q += count;
    F.pcount = q; q += count;
    F.stats = q; q += 3;
    F.ubase = q; q += runs * count;
    F.pbase = q; q += runs * count;
    F.uoff = q; q += count;
    F.poff = q; q += count;
    F.tkind = q; q += max_tiles;
    F.tmat = q; q += max_tiles;
    F.ulist = q; q += max_tiles;
    F.nchunks = q; q += 1;
    F.plist = q;
    F.ulist_cap = max_tiles;
    F.plist_cap = (int64_t)B->plist_ints;
    F.status = ctx->status_dev;
    F.chunk_cap = 2 * (max_tiles + count) + 16;
    NBTC_TRY(cuda_check(cudaMalloc(&B->fchunks, sizeof(WorkChunk) * F.chunk_cap), "frame chunks"));
    NBTC_TRY(cuda_check(cudaMalloc(&B->fcounter, sizeof(int)), "frame counter"));
    F.chunks = B->fchunks;
    F.counter = B->fcounter;
    NBTC_TRY(set_tile_shape(B, 16, 8));
  }
  NBTC_TRY(cuda_check(cudaStreamSynchronize(s), "plan set-up"));
  // ---- autotune: chunk size (decode), tile shape (frame)
  if (flags & NBTC_BATCH_AUTOTUNE) {
    if (B->decode_tiles > 0) {
      float best = 1e30f;
      int bc = B->chunk;
      for (int c : {8, 32, 128}) {
        NBTC_TRY(set_decode_chunk(B, c, B->cap));
        const float ms = time_ms([&] { return enqueue_decode(ctx, B, B->cap); }, B->cap, 3, st);
        if (st) {
          free_plan(B);
          return st;
        }
        if (ms < best) {
          best = ms;
          bc = c;
        }
      }
      NBTC_TRY(set_decode_chunk(B, bc, B->cap));
      B->info.tuned_decode_ms = best;
    }
    if (B->has_frame) {
      float bestf = 1e30f;
      int ftw = 16, fth = 8;
      const int shapes[4][2] = {{16, 8}, {32, 4}, {8, 16}, {128, 1}};
      for (auto& sh : shapes) {
        if (set_tile_shape(B, sh[0], sh[1])) continue;
        const float ms = time_ms([&] { return enqueue_render(ctx, B, B->cap); }, B->cap, 3, st);
        if (st) {
          free_plan(B);
          return st;
        }
        if (ms < bestf) {
          bestf = ms;
          ftw = sh[0];
          fth = sh[1];
        }
      }
      NBTC_TRY(set_tile_shape(B, ftw, fth));
      B->info.tuned_render_ms = bestf;
    }
  }
  // ---- graphs
  if (B->decode_tiles > 0) NBTC_TRY(capture(ctx, B, false, &B->g_decode));
  if (B->has_frame) NBTC_TRY(capture(ctx, B, true, &B->g_render));
#undef NBTC_TRY
  B->info.warpgroups = B->info.render_warpgroups = kBatchW;
  B->info.decode_tmem_operands = B->info.render_tmem_operands = 1;
  B->info.chunk_tiles = B->chunk;
  B->info.tile_w = B->tw;
  B->info.tile_h = B->th;
  B->info.decode_tiles = B->decode_tiles;
  *plan = B;
  return NBTC_OK;
}

nbtc_status nbtc_decode_batched(nbtc_context* ctx, nbtc_batch* B, void* stream) {
  NBTC_RANGE();
  nbtc_status st = enter(ctx);
  if (st) return st;
  if (!B) return fail(NBTC_ERR_INVALID_ARG, "plan NULL");
  if (!B->g_decode) return NBTC_OK;  // no material has a full-decode output
  return cuda_check(cudaGraphLaunch(B->g_decode, (cudaStream_t)stream), "launch decode graph");
}

nbtc_status nbtc_render_frame(nbtc_context* ctx, nbtc_batch* B, void* stream) {
  NBTC_RANGE();
  nbtc_status st = enter(ctx);
  if (st) return st;
  if (!B) return fail(NBTC_ERR_INVALID_ARG, "plan NULL");
  if (!B->g_render) return fail(NBTC_ERR_INVALID_ARG, "the plan has no frame");
  return cuda_check(cudaGraphLaunch(B->g_render, (cudaStream_t)stream), "launch render graph");
}

nbtc_status nbtc_batch_info_get(nbtc_batch* B, nbtc_batch_info* info) {
  if (!B || !info) return fail(NBTC_ERR_INVALID_ARG, "NULL argument");
  nbtc_status st = cuda_check(cudaSetDevice(B->device), "cudaSetDevice");
  if (st) return st;
  *info = B->info;
  if (B->has_frame) {
    int stats[3] = {0, 0, 0};
    if ((st = cuda_check(cudaDeviceSynchronize(), "sync")) ||
        (st = cuda_check(cudaMemcpy(stats, B->F.stats, sizeof(stats), cudaMemcpyDeviceToHost), "read stats")))
      return st;
    info->frame_uniform_tiles = stats[0];
    info->frame_mixed_tiles = stats[1];
    info->frame_packed_tiles = stats[2];
  }
  return NBTC_OK;
}

nbtc_status nbtc_batch_destroy(nbtc_batch* B) {
  free_plan(B);
  return NBTC_OK;
}

}  // extern "C"
