// hd_tile.h -- host-side interface of the tile sweep (hd_tile.cu).
#pragma once

#include <cstddef>
#include <cstdint>

#include "hd_kernels.h"

namespace hd {

// Tiles of one replica: ntx x nty tiles over its cells, tile (x, y) spanning
// half-columns hm x / ntx .. hm (x + 1) / ntx and half-rows likewise, numbered
// row by row from `first` over all replicas.
struct TileGrid {
    int32_t first, ntx, nty;
};

// Largest tile (cells per side) and spill bytes per block.
struct TileLimits {
    int max_x, max_y;
    size_t spill;
};
TileLimits tile_limits(bool fixed);

struct TileCfg {
    const TileGrid* grids;  // device, [R]
    TileGrid grid0;         // replica 0's (one replica: passed by value)
    int64_t total;          // tiles over all replicas
    int blocks;             // blocks resident at once
    uint32_t* sync;         // tile_sync_words(total): ticket, abort word, finished sweeps per tile
    void* spill;            // blocks x TileLimits::spill bytes
    bool stall;             // test hook: ticket 0 is never taken, and waits give up early
};

// Blocks resident at once of the kernel that c selects.
cudaError_t tile_blocks(const LaunchCfg& c, int* blocks);
size_t tile_sync_words(int64_t total);
// nsweeps <= kMaxChunk sweeps of the draw table in one launch, from `from`
// into `to` for the first sweep and alternating after.  Every cell of the
// written generation is written; the other keeps the state before the last
// sweep.
cudaError_t launch_sweeps_tile(const LaunchCfg& c, const TileCfg& t, const Frame* table, int nsweeps, CellBufs from,
                               CellBufs to, unsigned long long* counters, int* err);

// Small boxes (half-side hm <= box_max_hm for every replica): each box kept in
// one block's shared memory over all sweeps of the launch.  hm: the largest
// half-side of the replicas.  spill: R x box_spill bytes.  As launch_sweeps_tile, but the generation not written last
// is left as it was.
int box_max_hm(bool fixed, int R);
size_t box_spill(bool fixed, int hm);
cudaError_t launch_sweeps_box(const LaunchCfg& c, int hm, void* spill, const Frame* table, int nsweeps, CellBufs from,
                              CellBufs to, unsigned long long* counters, int* err);

}  // namespace hd
