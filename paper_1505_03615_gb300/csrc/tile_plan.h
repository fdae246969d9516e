// tile_plan.h -- plan of the tiled Gauss-Seidel sweep (built by tile_plan.cpp, run by tile.cu).
#pragma once
#include <cstdint>
#include <vector>

#include "hier.h"

namespace lbmg {

constexpr int kTileSteps = 8;        // colour steps of one launch at most
constexpr int kTileParts = 2;        // launches per sweep at most
constexpr int kTileInfo = 16;        // ints per tile in TilePlan::info
constexpr uint16_t kTileNoRow = 0xffff;
constexpr int kTileMinRows = 64;     // rows of a tile on small levels
constexpr int kTileOneRound = 256;   // up to this many rows a tile, one tile per SM; then two, of
constexpr int kTileMaxRows = 800;    // at most this many (with its rim: shared memory; 263 on 152 SMs)
constexpr int kTileTwoParts = 12000; // from this many rows on a sweep takes two launches
constexpr int kTileLevel32 = 80000;  // largest levels whose sweeps are tiled, FP32 and FP64
constexpr int kTileLevel64 = 60000;

// Entries are stored group by group (kTileRows rows of one step, four lanes each): entry k of row l of a
// group at 32 (base + k / 4) + 4 l + k % 4, base the quads of all groups before it, so that lane 4 l + k % 4
// finds its entries at its own place of the group's lines of 32.
constexpr int kTileRows = 8;
struct TilePlan {
    int ntile = 0, nsteps = 0, maxloc = 0, maxcomp = 0, maxgrp = 0, maxquads = 0;   // maxquads: of one group
    int64_t groups = 0, quads = 0;
    // per tile: local rows, computed rows (first), own rows of the steps' colours (first among these), first
    // group, first quad, then the end (from the first group) of every step's groups and of the residual's
    std::vector<int32_t> info;
    std::vector<int32_t> loc;        // [ntile][maxloc] level rows of the local slots, -1 pad
    std::vector<int32_t> cum;        // [ntile][maxgrp + 1] quads before each of the tile's groups
    std::vector<int32_t> row;        // per group: kTileRows level rows (-1: none)
    std::vector<uint16_t> slot;      // per group: their local slots (kTileNoRow: none)
    std::vector<int32_t> qgroup;     // per quad: its group
    std::vector<uint16_t> col;       // per entry: local slot of its column
    std::vector<int32_t> map;        // per entry: stored entry of the level's matrix, -1 pad
};

// Launches per sweep and tiles of a level with that many smoothed rows.
void tile_shape(int rows, int sms, int *parts, int *ntile);
// Tiles as runs of blocks of corners.
struct TileCut {
    std::vector<int64_t> start;      // [ntile + 1] into blocks
    struct Block {
        int32_t at[3], inst;         // block coordinates and mesh
        int32_t first[8], rows[8];   // rows of each colour
        double weight;               // stored entries of all its rows, scaled by its tile's rim
    };
    std::vector<Block> blocks;
};
void cut_tiles(const HostLevel &L, int ntile, TileCut &cut);
// The colour steps seq[0..nsteps) and, when asked, the residual b - A x of the own rows behind them (nsteps =
// 0: of the vector as it is).  False when a tile would need more than 65535 local rows.
bool build_tile_plan(const HostLevel &L, const TileCut &cut, const int *seq, int nsteps, bool residual, TilePlan &out);
// Cuts again, every tile's blocks weighted by the entries the tile processes per own entry in `plan`.
void rebalance_tiles(const TilePlan &plan, TileCut &cut);
// Halves the tiles with more than maxloc local rows in `plan`; false when there is none.
bool split_tiles(const TilePlan &plan, int maxloc, TileCut &cut);

}  // namespace lbmg
