// tpfa_tile.h -- shape of the x-y tiles of the FP64-bound kernels (one thread
// per cell).
#pragma once

namespace tpfa {

// Tile of at most `threads` cells that covers a plane with the fewest warps
// (and the shortest rim): on the FP64 pipe a partly filled warp costs as much
// as a full one.  32 x 8 tiles would put 40 % more warps than cells / 32 on a
// 97 x 83 plane, the tile chosen (9 x 28) 5 %.  The widths tried split nx
// evenly.
inline void tile_shape(int nx, int ny, int threads, int& TX, int& TY) {
    double best = 1e300;
    const int first = (nx + 127) / 128, last = nx <= 8 ? 1 : (nx + 7) / 8;
    for (int n = first; n <= last && n < first + 64; ++n) {
        const int x = (nx + n - 1) / n;
        const int ymax = ny < threads / x ? ny : threads / x;
        const int rows = (ny + ymax - 1) / ymax;
        const int y = (ny + rows - 1) / rows;
        const int warps = (x * y + 31) / 32, rim = (2 * (x + 2) + 2 * y + 31) / 32;
        const double cost = (double)((nx + x - 1) / x) * rows * (80.0 * warps + 12.0 * rim);
        if (cost < best) best = cost, TX = x, TY = y;
    }
}

}  // namespace tpfa
