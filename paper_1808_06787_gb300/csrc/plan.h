// How many plain steps one launch takes, and over which parts of the grid: the rules behind
// the passes of tile.cuh.  Plain C++, so that the host can check them.
#pragma once

namespace lbms {

// Tile of a pass over a small grid (tile.cuh) and the most steps it takes; depth 1: single
// steps are faster.
struct TileShape {
    int depth;
    int x, y, z;
};

inline double tile_count(const TileShape& t, int nx, int ny, int nz)
{
    auto cuts = [](int n, int size) { return (double)(n / size + (n % size ? 1 : 0)); };
    return cuts(nx, t.x) * cuts(ny, t.y) * cuts(nz, t.z);
}

// The rule counts tiles, not nodes, against the multiprocessors: a tile has its margins
// formed whole however few of its nodes the grid fills, so a grid one node wide has many
// times the work of a square of as many nodes, and where the tiles make a second wave of
// blocks it takes as long as a full one.  q velocities, s evolved species; fixed: the FP64
// collision runs in fixed point.  us per step at 152 multiprocessors, single -> tiled:
//
// FP32 planes: D2Q5 ternary 48 x 40 1.73 -> 0.77, 128^2 1.77 -> 0.91, 200^2 2.03 -> 1.61,
// 256^2 2.09 -> 1.88, D2Q9 128^2 2.01 -> 1.16, binary 256^2 2.13 -> 1.24; with the tiles of a
// grid of 8192 x 1 (1024 of 8 x 8) it was 1.87 -> 2.37, of 65536 x 1 (4096 of 16 x 16) 2.27 ->
// 17.2, of D2Q9's 4096 x 2 (256 of 16 x 16) 2.07 -> 2.18.  Four species fill an SM with one
// tile of 16 x 16: D2Q9 158 x 186 (120 tiles) 2.64 -> 2.37 and 204^2 (169 tiles) 2.77 -> 3.87.
// FP32 volumes: D3Q7 24 x 16 x 12 1.79 -> 1.33, 28 x 24 x 16 1.95 -> 1.63, 40 x 24 x 24 2.08 -> 2.10
// (single); 7168 x 1 x 1 (1792 tiles of 4^3) 1.97 -> 10.7.
// FP64 in fixed point: binary D2Q5 240 x 40 1.79 -> 1.22, 128^2 1.78 -> 1.44, ternary 64^2 2.84
// -> 2.43, 80^2 2.98 -> 2.68, 100^2 2.97 -> 3.25 (single); 20480 x 1 4.7 -> 6.8.
// FP64 in FP64 arithmetic (frozen mode, wide diffusivities), whose margins cost the pipe that
// bounds the step: two steps, and tiles that fill one wave.  Binary D2Q5 64 x 75 3.11 -> 2.58
// (8 x 4), 96^2 3.06 -> 2.66 (8 x 8); where the single step's blocks of 64 nodes make a third
// layer (more than 128 nodes per multiprocessor) 140^2 4.2 -> 3.9 (12 x 12), D2Q9 6.3 -> 6.35, but
// 135^2 3.5 -> 3.9, 4.5 -> 6.35; ternary 79 x 81 5.21 -> 5.05, D2Q9 7.60 -> 7.75.
// Lines of 100 to 8000 nodes FP64 2.4 -> 1.65, FP32 four species 1.59 -> 0.58; 30000 nodes
// FP64 3.08 -> 3.96 (single).
inline TileShape tile_shape(int dim, int q, int s, bool f64, bool fixed, int nx, int ny, int nz, int sms)
{
    const TileShape none = {1, 0, 0, 0};
    TileShape t = none;
    // takes the shape if its tiles are from `least` to `most` per multiprocessor
    auto take = [&](int depth, int x, int y, int z, double most, double least = 0.0) {
        const TileShape c = {depth, x, y, z};
        const double n = tile_count(c, nx, ny, nz);
        if (n > most * sms || n < least * sms) return false;
        t = c;
        return true;
    };
    const double nodes = (double)nx * ny * nz;
    if (s > 3 || (f64 && s > 2)) return none;
    if (dim == 1) {
        take(8, 16, 1, 1, 3.375);
    } else if (dim == 3) {
        if (f64 || s > 2 || q > 7) return none;
        take(3, 4, 4, 4, 0.75) || take(2, 8, 4, 4, 1.0);
    } else if (!f64) {
        if (take(5, 8, 8, 1, 1.0) || take(4, 16, 8, 1, 1.4)) return t;
        // two waves of the largest tiles cost as much however few nodes they hold
        if (nodes < 128.0 * tile_count({1, 16, 16, 1}, nx, ny, nz)) return none;
        if (s == 2 && q <= 5 && take(2, 16, 16, 1, 1.8, 1.05)) return t;
        take(3, 16, 16, 1, s == 3 ? 1.0 : 1.8);
    } else if (fixed) {
        if (s == 1)
            take(5, 8, 8, 1, 1.0) || take(4, 16, 8, 1, 1.1);
        else
            take(4, 8, 4, 1, 0.9) || take(5, 8, 8, 1, 0.75);
    } else if (s == 1) {
        take(2, 8, 4, 1, 1.0) || take(2, 8, 8, 1, 1.0) || (nodes > 128.0 * sms && take(2, 12, 12, 1, 1.0, 0.9));
    } else {
        take(2, 8, 4, 1, 1.0) || take(2, 8, 8, 1, 0.75);
    }
    return t;
}

}  // namespace lbms
