// Scattered coverage by tiles: the visibilities of a call are sorted by the
// tile of their footprint start, and a tile's part of the subgrid (the tile
// and the footprint's reach beyond it) is kept in shared memory while its
// visibilities are summed (tiled_degrid.cu) or gridded (tiled_grid.cu).  A
// footprint then costs 2 KB of shared memory bandwidth instead of 2 KB from
// or to L2, which bounds the kernels that move every footprint by itself
// (gather.cu, scatter.cu).
#pragma once

#include "internal.cuh"

namespace dg {

// Tiles of 2^lx x 2^ly footprint starts (u by v), and the visibilities from
// which a call goes by tiles: min_vis plus min_per_tile for every tile.
struct TileShape {
    int lx, ly;
    int min_vis, min_per_tile;
};

// The tiles of a call.
struct Tiling {
    int lx, ly;
    int nx, ny;             // tiles per row and column of a subgrid
};

inline Tiling tiling_of(const Geometry &g, TileShape t)
{
    return Tiling{t.lx, t.ly, (g.nx - kUV + (1 << t.lx)) >> t.lx, (g.ny - kUV + (1 << t.ly)) >> t.ly};
}

// A visibility as the tile kernels read it.
struct alignas(16) BinRecord {
    unsigned ux, vy;        // GCF row (20 bits) and place in the tile (above), u and v axis
    unsigned fw;            // w row
    unsigned index;         // in the call's lists
};
constexpr int kBinRowBits = 20;     // uv oversampling is at most 2^20

// A piece of work: records [start, start + n) of one tile.
struct alignas(16) BinItem {
    int s, tx, ty;          // subgrid, tile
    int n;
    long long start;
    long long unused;
};

// Device side of a call's bins.
struct Bins {
    Tiling tiling;
    BinRecord *records;
    const BinItem *items;
    const int *n_items;
    int *item_counter;      // claims
};

constexpr int kItemVis = 512;       // records per item at most


}  // namespace dg

// Workspace of a plan's binned calls (bins.cu), grown as needed.
struct dg_bins {
    void *buffer;           // one allocation for the three
    dg::BinRecord *records;
    dg::BinItem *items;
    int *counters;          // [2] items and claims, then [tiles] counts / cursors
    long long cap_records, cap_items, cap_tiles;
};

// Whether a call of n_vis visibilities on n_subgrids subgrids goes by tiles
// of this shape: enough visibilities, and sizes within the records' fields.
bool dg_bins_worth(const degrid_plan *p, dg::TileShape shape, int n_subgrids, long long n_vis);
// Grows the workspace; false when it is too small and cannot grow now (the
// stream is capturing, or no memory is left).
bool dg_bins_reserve(degrid_plan *p, cudaStream_t st, int n_subgrids, long long n_vis);
// Sorts the call's visibilities.  Invalid ones are counted and, with vis_out,
// get their zero; malformed offsets are flagged.
cudaError_t dg_bins_sort(degrid_plan *p, cudaStream_t st, dg::TileShape shape, int n_subgrids,
                         long long n_vis, const double *uvw, const int64_t *vis_offsets, float *vis_out,
                         dg::Bins *out);
void dg_bins_free(degrid_plan *p);

// The tile kernels.  The lines: the sort's kernels cost a call about 30 us
// and a tile 4 ns (degridding: its load) or 7 (gridding: its zeros and its
// add), against 0.06 and 0.11 us saved per thousand visibilities.  Measured
// calls in us, by tiles / footprint by footprint, on subgrids of 512 x 512:
// degridding (complex64) 1 subgrid 100,000 visibilities 38 / 41 and 400,000
// 63 / 75, 16 subgrids 100,000 49 / 42 and 200,000 56 / 59, 64 subgrids
// 200,000 111 / 95 and 400,000 118 / 144; gridding 1 subgrid 50,000 46 / 79,
// 16 subgrids 200,000 160 / 141 and 400,000 135 / 179, 64 subgrids 400,000
// 569 / 386 and 1,600,000 592 / 1,239.
constexpr dg::TileShape kDegridTile{5, 5, 100000, 14}, kGridTile{4, 4, 50000, 11};
cudaError_t dg_launch_tiled_degrid(degrid_plan *p, cudaStream_t st, const dg::Bins &bins, long long max_items,
                                   const void *subgrids, int n_subgrids, const float *scale, float *vis_out);
cudaError_t dg_launch_tiled_grid(degrid_plan *p, cudaStream_t st, const dg::Bins &bins, long long max_items,
                                 int n_subgrids, const float *vis_in, float *sub_out);
