// tiles.cuh -- 2.5-D tiled sweeps of the stencil and assembly kernels.
#pragma once

#include <algorithm>

#include "rf_internal.cuh"

namespace rf {

// Tiled sweeps for the stencil kernels.  A block owns a TX x TY column tile
// and a range of z planes and walks up through them: the x/y neighbours of a
// plane come from shared memory (the plane plus a one-cell halo, double
// buffered so each plane needs one barrier), the z neighbours from registers
// (the planes below and above), and the plane above is loaded while the
// current one is in use.  Blocks loop over (tile, z-range) items; the grid
// never exceeds the reduction's block count.
constexpr int TX = 32, TY = RED_THREADS / 32;
constexpr int HALO = 2 * TY + 2 * TX;   // x- and y-halo cells of a plane (no corners)

struct Tiles {
    int ntx, nty, zc;       // tiles along x, y; planes per item
    int tx, ty;             // tile size
    long long items;
};

inline Tiles make_tiles(const Grid &g, int nblk)
{
    if (g.cap > nblk) nblk = g.cap;
    Tiles t;
    t.tx = TX;
    t.ty = TY;
    t.ntx = (g.nx + TX - 1) / TX;
    t.nty = (g.ny + TY - 1) / TY;
    const long long tiles = (long long)t.ntx * t.nty;
    // split z so that the items fill the grid in one wave when the tiles alone
    // do not (every block then walks the same number of planes)
    const long long want_chunks = nblk / tiles;
    const int chunks = (int)std::min<long long>(std::max<long long>(want_chunks, 1), g.nz);
    t.zc = (g.nz + chunks - 1) / chunks;
    t.items = tiles * ((g.nz + t.zc - 1) / t.zc);
    return t;
}

// Tiles with the z split that minimises (waves of `resident` blocks) x
// (planes per item + the two extra planes an item reads); at most `cap` items
// per wave are launched.
inline Tiles make_tiles_balanced(const Grid &g, int resident, int tile_x, int tile_y = TY)
{
    Tiles t;
    t.tx = tile_x;
    t.ty = tile_y;
    t.ntx = (g.nx + tile_x - 1) / tile_x;
    t.nty = (g.ny + tile_y - 1) / tile_y;
    const long long tiles = (long long)t.ntx * t.nty;
    long long best = -1;
    int best_zc = g.nz;
    for (int ch = 1; ch <= g.nz; ch++) {
        const int zc = (g.nz + ch - 1) / ch;
        const long long items = tiles * ((g.nz + zc - 1) / zc);
        const long long waves = (items + resident - 1) / resident;
        const long long cost = waves * (zc + 2);
        if (best < 0 || cost < best) {
            best = cost;
            best_zc = zc;
        }
    }
    t.zc = best_zc;
    t.items = tiles * ((g.nz + t.zc - 1) / t.zc);
    return t;
}

// Whether a plane of the grid leaves more than three quarters of its tiles
// empty: columns and vertical sections, which a walk plane by plane serves with
// a few threads; they run cell by cell.  us a CG iteration, 600 000 cells, tiled /
// cell by cell: FP64 1 x 1 x 600000 2009 / 23, 600 x 1 x 1000 107 / 26, 600 x 4 x 250
// 42 / 30, 16 x 16 x 2500 39 / 32, 64 x 64 x 150 28 / 30; mixed 1515 / 16, 60 / 18,
// 26 / 21, 19 / 19, 13 / 20.
inline bool narrow_grid(const Grid &g, int tile_x, int tile_y)
{
    const long long tiles = (long long)((g.nx + tile_x - 1) / tile_x) * ((g.ny + tile_y - 1) / tile_y);
    return 4 * g.sxy < tiles * tile_x * tile_y;
}

inline int tile_blocks(const Tiles &t, const Grid &g, int nblk)
{
    return (int)std::min<long long>(t.items, g.cap > nblk ? g.cap : nblk);
}

#ifdef __CUDACC__
struct TileItem {
    int i0, j0, k0, k1;
};

__device__ __forceinline__ TileItem tile_item(const Grid &g, const Tiles &t, long long item)
{
    const long long per_plane = (long long)t.ntx * t.nty;
    const int chunk = (int)(item / per_plane);
    const long long r = item - chunk * per_plane;
    TileItem it;
    it.j0 = (int)(r / t.ntx) * t.ty;
    it.i0 = (int)(r % t.ntx) * t.tx;
    it.k0 = chunk * t.zc;
    it.k1 = min(g.nz, it.k0 + t.zc);
    return it;
}

// Halo cell h (0 <= h < HALO) of a tile, as offsets (hx, hy) from (i0, j0):
// -x column, +x column, -y row, +y row.
__device__ __forceinline__ void halo_cell(int h, int &hx, int &hy)
{
    if (h < TY) { hx = -1; hy = h; }
    else if (h < 2 * TY) { hx = TX; hy = h - TY; }
    else if (h < 2 * TY + TX) { hx = h - 2 * TY; hy = -1; }
    else { hx = h - 2 * TY - TX; hy = TY; }
}
#endif

}  // namespace rf
