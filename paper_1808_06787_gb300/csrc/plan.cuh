// How many plain steps one launch takes, and over which parts of the grid: the rules behind
// the passes of tile.cuh and fused.cuh.  Plain C++, so that the host can check them.
#pragma once

#include <initializer_list>

namespace lbms {

// Tile of a pass over a small grid (tile.cuh) and the most steps it takes; depth 1: single
// steps are faster.
struct TileShape {
    int depth;
    int x, y, z;
};

// Nodes of a 2D tile and its margins that a step of its pass forms, on average over the steps.
inline double tile_formed(const TileShape& t)
{
    double sum = 0.0;
    for (int m = 0; m < t.depth; ++m) sum += (double)(t.x + 2 * m) * (t.y + 2 * m);
    return sum / t.depth;
}

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
// Grids of more tiles, flat ones above all, take passes while a step's work, the nodes formed
// times S Q + 4 (about the instructions of a node), is at most 7900 per multiprocessor: binary
// D2Q5 6000 x 4 (4700) 1.97 -> 1.19, 5000 x 13 (6100) 2.06 -> 1.65, ternary 6000 x 4 (7400) 1.97 ->
// 1.81, but D2Q9 4096 x 2 (12100 in tiles of 16 x 16) 2.07 -> 2.18.
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
    if (s > 3 || (f64 && s > 2)) return none;
    if (dim == 1) {
        take(8, 16, 1, 1, 3.375);
    } else if (dim == 3) {
        if (f64 || s > 2 || q > 7) return none;
        take(3, 4, 4, 4, 0.75) || take(2, 8, 4, 4, 1.0);
    } else if (!f64) {
        const double nodes = (double)nx * ny;
        if (take(5, 8, 8, 1, 1.0) || (nodes <= 162.0 * sms && take(4, 16, 8, 1, 1.65))) return t;
        // two waves of the largest tiles cost as much however few nodes they hold
        if (nodes >= 128.0 * tile_count({1, 16, 16, 1}, nx, ny, nz)) {
            if (s == 2 && q <= 5 && take(2, 16, 16, 1, 1.8, 1.12)) return t;
            if (take(3, 16, 16, 1, s == 3 && q > 5 ? 1.0 : 1.8)) return t;
        }
        double least = 7900.0 * sms;
        for (const TileShape& c : {TileShape{5, 8, 8, 1}, TileShape{4, 16, 8, 1}, TileShape{3, 16, 16, 1}}) {
            const double work = tile_count(c, nx, ny, nz) * tile_formed(c) * (s * q + 4);
            if (work > least) continue;
            least = work;
            t = c;
        }
    } else if (fixed) {
        if (s == 1)
            take(5, 8, 8, 1, 1.0) || take(4, 16, 8, 1, 1.1);
        else
            take(4, 8, 4, 1, 0.9) || take(5, 8, 8, 1, 0.75);
    } else if (s == 1) {
        take(2, 8, 4, 1, 1.0) || take(2, 8, 8, 1, 1.0) || ((double)nx * ny > 128.0 * sms && take(2, 12, 12, 1, 1.0, 0.9));
    } else {
        take(2, 8, 4, 1, 1.0) || take(2, 8, 8, 1, 0.75);
    }
    return t;
}

// The passes over rows of large FP32 planes (fused.cuh): q velocities, s evolved species.

// Blocks of 4 warps per SM the row kernels are compiled for.  What bounds them is the
// issue rate (D2Q5 ternary 2048^2: 265 instructions per 32 nodes stored and step, margins
// included, in 78 % of the issue slots, the FP32 pipes 49 % and the ALU 46 % busy; HBM runs at 2.7
// TB/s of its 6.8), so each value is the fewest warps that still keep issuing, with the
// registers that leaves.  Measured, us per step, at
// blocks 2 / 3 / 4 / 5: D2Q5 ternary 4096^2 142 / 138.7 / 142.5 / 143; D2Q9 ternary
// 2048^2 72 / 73 / 57.5 / 67, binary 50 / 50 / 41 / 29.3; D2Q5 with four species 2048^2
// 74.6 / 72 / 57.2 / 59.9; D2Q9 with five species 2048^2 130 / 145 / 179 (single steps:
// 194, 86.6, 47.8, 80.5 and 180.6).  Ratio to the single steps, mean over planes of 1 to 4
// million nodes: D2Q5 with five species 0.89 / 0.83 / 0.84 at 2 / 3 / 4, D2Q4 with five 0.97 / 0.91
// / 0.91, binary D2Q4 0.93 / 0.81 / 0.98 at 3 / 4 / 5, ternary 1.08 / 1.01 / 0.94.
constexpr int row_blocks(int q, int s)
{
    if (q > 5) return s == 1 ? 5 : s == 2 ? 4 : s == 3 ? 3 : 2;
    if (q == 4 && s <= 2) return s == 1 ? 4 : 5;
    return s == 3 ? 4 : 3;
}

// Cuts n rows into parts of at least `least` rows: `wave` parts (per strip) fill the chip
// once.  Warps take different times, so two waves are taken while a part keeps `pair` rows
// and up to four while it keeps `good`; but a part also forms 2 (K - 1) rows for its
// neighbours.  D2Q5 ternary, us per step with one wave -> two: 1448^2 24.4 -> 20.4,
// 2048 x 1100 28.5 -> 22.6, 3474 x 1576 69.5 -> 53.5 (single steps 27.7, 27.6, 65.2);
// D2Q9 ternary 3402 x 1784 93.6 -> 86.4, but 2048^2 (31 rows) 56.5 -> 59.0, and with five
// species, whose parts hold more, 129.9 -> 132.6.
inline void cut(int n, double wave, int pair, int good, int least, int& segments, int& rows)
{
    int waves = (int)((n / good) / wave);
    waves = waves > 4 ? 4 : waves;
    if (waves < 2) waves = n / pair >= 2.0 * wave ? 2 : 1;
    int s = (int)(waves * wave);
    if (s > n / least) s = n / least;
    if (s < 1) s = 1;
    rows = (n + s - 1) / s;
    segments = (n + rows - 1) / rows;
}

// The parts of a pass of `steps` steps.
struct RowPlan {
    int strips, segments, rows;
};
constexpr int row_strip(int steps) { return 32 - 2 * (steps - 1); }  // columns a warp stores
inline double row_slots(int q, int s, int sms) { return (double)sms * row_blocks(q, s) * 4; }  // resident warps
inline RowPlan row_plan(int q, int s, int steps, int nx, int ny, int sms)
{
    RowPlan p;
    p.strips = (nx + row_strip(steps) - 1) / row_strip(steps);
    const int pair = q <= 5 ? 16 : (s <= 2 ? 32 : 80), good = q <= 5 || s <= 2 ? 48 : 80;
    cut(ny, row_slots(q, s, sms) / p.strips, pair, good, 4 * steps, p.segments, p.rows);
    return p;
}

// What a pass costs: nodes formed per node of the grid (margins, idle lanes of the last
// strip), times the warp slots per warp that has a part where the parts leave some idle; whole:
// the slots of the last wave count as well.  At a wall along x a warp reads and selects the wall
// nodes' own populations besides: on D2Q9 (six directions) with four and five species 0.45 and 0.6 of
// a row's work more.
inline double row_cost(int q, int s, int steps, int nx, int ny, bool x_walls, bool whole, int sms)
{
    const RowPlan p = row_plan(q, s, steps, nx, ny, sms);
    const double waves = (double)p.strips * p.segments / row_slots(q, s, sms);
    const double taken = whole || waves < 1.0 ? (double)(long long)(waves + 0.9999) : waves;
    double formed = (double)p.strips * p.segments * 32.0 * (p.rows + 2 * (steps - 1)) / ((double)nx * ny);
    if (x_walls && q > 5 && s >= 3) formed *= 1.0 + 0.15 * s * (p.strips > 1 ? 2.0 / p.strips : 1.0);
    return formed * taken / waves;
}

// Whether passes over rows beat as many single steps.  Sizes (60-step calls, us per step,
// single -> passes): D2Q5 ternary 1448^2 27.6 -> 24.9, 1024^2 14.0 -> 13.7 and 4096 x 300 16.1 ->
// 16.2 (hence the higher line for it), 4096^2 194 -> 138; binary 1024^2 8.4 -> 6.0; D2Q9 ternary
// 1024^2 23.1 -> 18.8, 724^2 11.1 -> 14.5; five species 724^2 24.3 -> 21.2; D2Q4 with four or five
// species at 0.5 to 1 million nodes 1.0 to 1.1 times the single steps' time, at 2 million 0.9.
// Cost: over 900 planes from 56 to 10^5 columns wide the ratio to the single steps grows with it
// from 0.7 at 1.1, and passes 1.00 to 1.05 at the limits below; beyond them it went on to 1.2 to 1.4
// (D2Q4 ternary 64 x 32768 20.3 -> 27.7, D2Q9 with five species 64 x 32768 91 -> 130).  pairs: the
// grid's single steps take two nodes per thread, in three quarters of the time per node, so
// that passes pay up to lower costs only (binary D2Q5 72 x 49498 at 1.46 22.6 -> 23.4, but 113 x
// 18001 at 1.7 16.8 -> 14.8), and short warps feel an incomplete last wave: 66112 x 128 at 1.18 and
// 1.29 waves 51.5 -> 61.5; with five species on D2Q9 36792 x 57 at 1.01 waves 92 -> 113.
inline bool rows_pay(int q, int s, int steps, int nx, int ny, bool x_walls, bool pairs, int sms)
{
    if (s > 4 || nx < 56 || ny < 24) return false;
    const double million = 1 << 20, cells = (double)nx * ny;
    const double least = s >= 3 ? (q == 4 ? (s == 3 ? 1.5 : 1.0) : 0.5) : (s == 2 && q <= 5 ? 1.5 : 1.0);
    if (cells < least * million) return false;
    double limit;
    if (q > 5)
        limit = s == 1 ? 2.0 : s == 2 ? 1.7 : s == 3 ? 1.45 : 1.33;
    else if (s == 1)
        limit = q == 4 ? (pairs ? 1.7 : 2.05) : (pairs ? 1.42 : 1.8);
    else if (s == 2)
        limit = q == 4 ? 1.5 : (pairs ? 1.4 : 1.55);
    else
        limit = s == 3 ? 1.5 : 1.45;
    const bool whole = (s == 1 && pairs) || (q > 5 && s >= 3);
    return row_cost(q, s, steps, nx, ny, x_walls, whole, sms) <= limit;
}

}  // namespace lbms
