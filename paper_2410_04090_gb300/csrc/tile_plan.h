// Detection tiles of a batch: how many cells of a level a tile holds (host
// code, no device call).
#pragma once

#include <array>
#include <utility>
#include <vector>

#include "tables.h"

#ifdef __CUDACC__
#define JSLAM_HD __host__ __device__
#else
#define JSLAM_HD
#endif

namespace jslam {

constexpr int kMaxLevels = 8;
// Detection tile: at most this many pixels a side (host picks cells per CTA).
constexpr int kFastMaxTile = 128, kFastThreads = 128, kFastCtasPerSm = 5;
constexpr int kFastMaxCellsPerCta = 2048;  // cells x k per CTA

// The default tile of a tuning stands for what an untuned context does: tile
// heights that follow the batch, and the tiles in order of decreasing work.
constexpr int kDefaultTileW = 128, kDefaultTileH = 64;
constexpr bool default_tile(int w, int h) { return w == kDefaultTileW && h == kDefaultTileH; }
// Tiles the autotuner times, the default first; 128 x 65 gives every batch the
// tall tiles that the default gives large ones.
constexpr int kTuneTiles[][2] = { { kDefaultTileW, kDefaultTileH }, { 128, 65 }, { 128, 32 },
                                  { 128, 128 }, { 64, 64 }, { 64, 128 } };

// Row stride of the bit-planes in 16-byte units for a tile of nch 32-pixel
// chunks: chunks 0..nch (32 bytes each) and a 16-byte pad, an odd count, so
// that the 128-bit loads of two neighbouring rows fall on the two halves of
// the shared-memory banks.
JSLAM_HD inline int bs_row_units(int nch) { return 2 * (nch + 1) + 1; }

// Detection tile box of a level: rows of box_w bytes -- the tile's 32-byte
// chunks and one more, which covers its 4-pixel halo on both sides and up to
// 15 bytes of alignment slack on the left -- and box_h rows (3-row halo above
// and below).
inline void detect_box(int tw, int th, int *box_w, int *box_h)
{
    *box_w = 32 * ((tw + 31) / 32 + 1);
    *box_h = th + 6;
}

// Part of the keys of the tuning cache: raised whenever the detection kernel's
// CTAs or what a tuning's values mean change, so that picks made for others are
// not applied (1: eight warps a CTA and exact tiles; 2: four warps, tiles by
// cost; 3: the default tile stands for the untuned plan).
constexpr int kTuneRevision = 3;

// Cells per tile, horizontally and vertically, of each level of a pair.
using LevelBlocks = std::array<std::pair<int, int>, kMaxLevels>;

// The tiles of every pair of a batch (its geometries); returns how many blocks
// of cells were compared.  A chosen tile size (tile_w x tile_h pixels) is about
// what the tiles get, else the heights follow the batch.
long long detect_blocks(const std::vector<Geometry> &geo, int k, int border, int tile_w, int tile_h, bool chosen,
                        int n_sm, std::vector<LevelBlocks> &blocks);

}  // namespace jslam
