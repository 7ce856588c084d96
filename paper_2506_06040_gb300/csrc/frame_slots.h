// Slots of a frame's packed tiles: a material's pixels of mixed tiles, in tiles of
// 128.  Frames hold up to 2^31 - 1 pixels and every material ends in a tile of its
// own, so a slot number needs more than 31 bits where a pixel count does not.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define NBTC_HD __host__ __device__
#else
#define NBTC_HD
#endif

namespace nbtc {

constexpr int kTileK = 128;  // pixels per classification tile

// Tiles of `px` >= 0 pixels.
NBTC_HD inline int packed_tiles(int px) { return px / kTileK + (px % kTileK != 0); }

// Slot `i` of the tiles that begin at tile `first`.
NBTC_HD inline int64_t packed_slot(int first, int i) { return (int64_t)first * kTileK + i; }

// Slots after the last pixel of its tiles.
NBTC_HD inline int free_slots(int px) { return px % kTileK ? kTileK - px % kTileK : 0; }

}  // namespace nbtc
