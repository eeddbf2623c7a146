// Tiles of a graph's dense corner (hub_tiles.cu): what launch_spmm needs to know of them.
#pragma once
#include "internal.cuh"

namespace mixgcn {

constexpr int HUB_ROWS = 256, HUB_COLS = 128;   // a tile
constexpr int HUB_SLICE = 256;                  // most columns of one product
constexpr int HUB_TILE_MIN = 500;               // entries from which a tile pays: 20 ns to gather them (256 columns), 18 for the tile (1.34 us on one of 74 pairs)
constexpr int64_t HUB_MIN_ENTRIES = 1 << 20;    // graphs below this, and tiles that hold less than a quarter of it, are not worth the launches
struct HubPiece { int32_t begin, end; };       // tiles [begin, end) of one row of tiles

}  // namespace mixgcn

// Tiles of one orientation: rows and columns by rank (descending entry counts: the orders of its schedule and of the transposed one's).
struct HubTiles {
    int row_blocks, kblocks;   // blocks of rows and of columns up to the last ones that hold a tile
    int64_t n_cols;            // hub columns in them
    int n_tiles, n_pieces, clusters;
    int64_t entries;           // stored entries that lie in tiles
    const int32_t* nodes;      // [n_cols] node of a hub column (the transposed schedule's perm)
    int32_t* rank;             // [n] rank of a row that lies in a row of tiles, -1 otherwise
    float *col_scale, *row_scale;
    uint32_t* bits;            // [n_tiles][256 rows][4 words]
    int32_t* tile_cb;          // [n_tiles] column block
    mixgcn::HubPiece* pieces;  // [n_pieces], in the order of the tiles
    int32_t* first_piece;      // [clusters + 1] of a pair of CTAs
    int32_t* piece_first;      // [row_blocks + 1] of a row of tiles
    CsrView rem;               // the matrix without the tiles' entries, all rows, and its schedule
    int64_t rem_nnz;
};

namespace mixgcn {

// the scratch of an aggregation of w columns, where it takes the tiles (t may be null) and there is memory for it
mixgcn_status reserve_tiles_scratch(mixgcn_ctx* ctx, const HubTiles* t, int32_t w);
bool hub_tiles_pay(const HubTiles* t, int32_t w);
// bytes of scratch for w columns: partial rows of ldp floats, images (of at most 256 columns) from *images_at on
int64_t hub_tiles_scratch(const HubTiles* t, int32_t w, int64_t ldp, int64_t* images_at);
// partial rows of the pieces for w <= HUB_SLICE columns: row r of piece q is partial row q * 256 + r, not yet times row_scale
mixgcn_status launch_hub_tiles(mixgcn_ctx* ctx, const HubTiles* t, int phase, int32_t w, const float* Y, int64_t ldy, int64_t y_rows, float* partial, int64_t ldp,
                               uint8_t* images, cudaStream_t s);

}  // namespace mixgcn
