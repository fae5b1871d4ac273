// Several time steps in one pass over the populations (FP32 solvers on undivided
// grids without Dirichlet faces).
//
// A plain step reads and writes every population once, so on grids beyond L2 it
// runs at the speed of HBM.  Here a warp marches through its part of the grid
// along the slowest axis and carries K steps with it: the first step gathers
// from memory, and each following one takes the layer its predecessor has just
// formed, one layer behind it, from registers (what is still needed of a layer waits
// in registers; shifts along x come from the neighbouring lanes).  Only the last
// step's populations are stored, so the traffic per step falls by K.  The parts
// overlap: a part forms the K - 1 layers and columns beyond its edges itself.
//
// The node functions, rounding keys and wall rules are those of k_step, so the
// populations are the same bit for bit.
//
// Marching, a part also forms layers that do not exist (beyond a wall) or that nobody
// asks for (before its queues are filled): their loads are clamped into the grid, their
// values are never stored, and at a wall the layer's own populations replace them.
#pragma once

#include <type_traits>

#include "kernels.cuh"
#include "plan.cuh"

namespace lbms {

template <int S>
struct FusedParams {
    const float* __restrict__ fin;
    float* __restrict__ fout;
    int nx, ny;
    uint32_t cells;
    uint32_t noflux;     // bit f set: face f is a no-flux wall
    int relax;           // magic or SRT (frozen solvers take single steps)
    int strips;          // parts along x
    int segments;        // parts along y
    int rows;            // rows of a part (the last one may have fewer)
    const uint32_t* clock_in;
    uint32_t* clock_out;
    Coeffs<float> co;
};

// One collision of a node (or of a packed pair of nodes).
template <int LAT, int S, typename V, typename InvD, typename Key>
__device__ __forceinline__ void fused_node(V (&f)[S][Lattice<LAT>::Q], const InvD& invD, int relax, Key key)
{
    V xi[S + 1], L1[S][S], L2[S][S];
    mole_fractions<LAT, S, V>(f, xi);
    relaxation_matrices<S, V>(xi, invD, (typename Vec<V>::scalar)(1.0 / Lattice<LAT>::cs2()), relax, L1, L2);
    collide<LAT, S, V>(f, xi, L1, L2, key);
}

// Element at a 32-bit byte offset from a base that is the same for the whole grid (a
// uniform register: no 64-bit address arithmetic per load; planes are below 4 GiB).
__device__ __forceinline__ const float& at_bytes(const float* base, uint32_t off)
{
    return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + off);
}
__device__ __forceinline__ float& at_bytes(float* base, uint32_t off)
{
    return *reinterpret_cast<float*>(reinterpret_cast<char*>(base) + off);
}

// The value of the column at x - cx.
__device__ __forceinline__ float from_column(float v, int cx)
{
    return cx == 0 ? v : (cx > 0 ? __shfl_up_sync(0xffffffffu, v, 1) : __shfl_down_sync(0xffffffffu, v, 1));
}

// The source of a gather along the marching axis: the layer below / above, with the
// periodic wrap or the wall (the node's own layer and its opposite populations).
struct March {
    int n;          // layers of the grid
    bool wlo, whi;  // walls at the ends
    __device__ __forceinline__ int place(int r) const  // layer in the grid's range
    {
        if (r >= 0 && r < n) return r;
        if (wlo) return r < 0 ? 0 : n - 1;
        const int m = r % n;
        return m < 0 ? m + n : m;
    }
    __device__ __forceinline__ int below(int y) const { return y == 0 ? (wlo ? 0 : n - 1) : y - 1; }
    __device__ __forceinline__ int above(int y) const { return y == n - 1 ? (whi ? y : 0) : y + 1; }
};

constexpr int kFusedBlock = 128;

// Rows of a plane (2D).  A lane owns one column of its warp's strip of 32 columns, K - 1 of
// them on each side only to feed the later steps (row_plan, plan.cuh).

// The grid a warp marches through: a plane of its own, or one of a batch's (whose nodes
// begin at `base` of a common node space).
struct RowGrid {
    int nx, ny;
    uint32_t noflux;
    uint32_t base;
    uint32_t stride;  // nodes of a population plane
};

struct RowLane {
    uint32_t x0, xl, xr;  // base + the lane's column and its neighbours (wrapped, or clamped at walls)
    bool bl, br;          // the column lies at a wall on its left / right
    bool wall;            // some column of the warp does
};

// The gather of row y for the first step, from memory.  INNER: a row with both neighbours inside the grid.
template <int LAT, int S, bool INNER>
__device__ __forceinline__ void load_row(const float* __restrict__ fin, const RowGrid& g, const RowLane& c, const March& m,
                                         int y, float (&f)[S][Lattice<LAT>::Q])
{
    using L = Lattice<LAT>;
    constexpr int Q = L::Q;
    const bool blo = !INNER && m.wlo && y == 0, bhi = !INNER && m.whi && y == m.n - 1;
    const uint32_t nx = (uint32_t)g.nx, row = (uint32_t)y * nx;
    const uint32_t rdn = INNER ? row - nx : (uint32_t)m.below(y) * nx, rup = INNER ? row + nx : (uint32_t)m.above(y) * nx;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const int cx = L::cx(k), cy = L::cy(k);
        const bool by = (cy > 0 && blo) || (cy < 0 && bhi);  // the source lies across a y wall
        const uint32_t r = cy > 0 ? rdn : (cy < 0 ? rup : row);
        const uint32_t x = (cx == 0 || by) ? c.x0 : (cx > 0 ? c.xl : c.xr);
        const float* plane = fin + (size_t)(by ? opp<LAT>(k) : k) * g.stride;
#pragma unroll
        for (int s = 0; s < S; ++s) f[s][k] = at_bytes(plane + (size_t)(s * Q) * g.stride, (r + x) * 4u);
    }
    if (c.wall) {  // bounce-back at the walls along x: the node's own opposite population
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            if (L::cx(k) == 0) continue;
            if (L::cx(k) > 0 ? c.bl : c.br)
#pragma unroll
                for (int s = 0; s < S; ++s)
                    f[s][k] = at_bytes(fin + (size_t)(s * Q + opp<LAT>(k)) * g.stride, (row + c.x0) * 4u);
        }
    }
}

// What a step after the first holds of its predecessor between two rows: the gather of
// the row it forms next, without the populations that come from the row above it
// (part, c_y >= 0), and that row's upward populations in place (up, c_y > 0).
template <int LAT, int S>
struct RowQueue {
    float part[S][Lattice<LAT>::Q], up[S][Lattice<LAT>::Q];  // (the entries named above)

    // The complete gather of the held row, `above` being the row that follows it; edge:
    // the held row lies at the upper wall.
    template <bool EDGE>
    __device__ __forceinline__ void complete(const float (&above)[S][Lattice<LAT>::Q], const RowLane& c, bool edge,
                                             float (&g)[S][Lattice<LAT>::Q]) const
    {
        using L = Lattice<LAT>;
#pragma unroll
        for (int k = 0; k < L::Q; ++k) {
#pragma unroll
            for (int s = 0; s < S; ++s) {
                if (L::cy(k) >= 0) {
                    g[s][k] = part[s][k];
                    continue;
                }
                float v = from_column(above[s][k], L::cx(k));
                if (EDGE && edge) v = up[s][opp<LAT>(k)];
                g[s][k] = v;
            }
        }
        if (c.wall) {
#pragma unroll
            for (int k = 0; k < L::Q; ++k) {
                const int cx = L::cx(k);
                if (cx == 0 || L::cy(k) >= 0) continue;
                if (cx > 0 ? c.bl : c.br)
#pragma unroll
                    for (int s = 0; s < S; ++s) g[s][k] = up[s][opp<LAT>(k)];
            }
        }
    }

    // Takes the predecessor's next row f; edge: that row lies at the lower wall.
    template <bool EDGE>
    __device__ __forceinline__ void push(const float (&f)[S][Lattice<LAT>::Q], const RowLane& c, bool edge)
    {
        using L = Lattice<LAT>;
#pragma unroll
        for (int k = 0; k < L::Q; ++k) {
            const int cx = L::cx(k), cy = L::cy(k);
            if (cy < 0) continue;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                float v = from_column(cy > 0 ? up[s][k] : f[s][k], cx);
                if (EDGE && cy > 0 && edge) v = f[s][opp<LAT>(k)];
                part[s][k] = v;
                if (cy > 0) up[s][k] = f[s][k];
            }
        }
        if (c.wall) {
#pragma unroll
            for (int k = 0; k < L::Q; ++k) {
                const int cx = L::cx(k);
                if (cx == 0 || L::cy(k) < 0) continue;
                if (cx > 0 ? c.bl : c.br)
#pragma unroll
                    for (int s = 0; s < S; ++s) part[s][k] = f[s][opp<LAT>(k)];
            }
        }
    }
};

template <int LAT, int S>
struct RowOccupancy {
    static constexpr int value = row_blocks(Lattice<LAT>::Q, S);
};

// K steps of the rows [y0, y1) of one strip of W columns, with margins of H (at least K - 1).
template <int LAT, int S, int K, int H, typename InvD>
__device__ __forceinline__ void march_rows(const float* __restrict__ fin, float* __restrict__ fout, const RowGrid& grid,
                                           int strip, int y0, int y1, uint32_t step, int relax, const InvD& invD)
{
    using L = Lattice<LAT>;
    constexpr int Q = L::Q, W = 32 - 2 * H;
    static_assert(L::DIM == 2 && H >= K - 1, "rows march along y");
    const int lane = threadIdx.x & 31;
    const int nx = grid.nx, ny = grid.ny;
    const int X = strip * W - H + lane;  // the lane's column; beyond the grid's edges wrapped or clamped
    RowLane c;
    uint32_t x;
    {
        const bool wl = grid.noflux & 1u, wr = grid.noflux & 2u;
        auto place = [&](int v) -> uint32_t {
            if (wl) return (uint32_t)(v < 0 ? 0 : (v >= nx ? nx - 1 : v));
            const int r = v % nx;
            return (uint32_t)(r < 0 ? r + nx : r);
        };
        x = place(X);
        c.x0 = grid.base + x;
        c.xl = grid.base + place(X - 1);
        c.xr = grid.base + place(X + 1);
        c.bl = wl && X == 0;
        c.br = wr && X == nx - 1;
        c.wall = __any_sync(0xffffffffu, c.bl || c.br);
    }
    const bool mine = lane >= H && lane < 32 - H && X < nx;
    const March m = {ny, (grid.noflux & 4u) != 0, (grid.noflux & 8u) != 0};
    const uint32_t C = 0x27d4eb2du, rowC = (uint32_t)nx * C, key0 = x * C;
    uint32_t hk[K];
#pragma unroll
    for (int l = 0; l < K; ++l) hk[l] = mix32((step + l) * 0x9e3779b9u);
    RowQueue<LAT, S> queue[K - 1];
    float nxt[S][Q];
    // Iteration j: the first step forms row y0 - (K - 1) + j, step l the row l below it.
    // STEADY: all of these rows and their neighbours lie inside the grid.
    auto iteration = [&](int j, auto steady) {
        constexpr bool STEADY = decltype(steady)::value;
        const int r0 = y0 - (K - 1) + j;
        float f[S][Q];
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int k = 0; k < Q; ++k) f[s][k] = nxt[s][k];
        load_row<LAT, S, STEADY>(fin, grid, c, m, STEADY ? r0 + 1 : m.place(r0 + 1), nxt);
#pragma unroll
        for (int l = 0; l < K; ++l) {
            const int r = r0 - l, y = STEADY ? r : m.place(r);
            float g[S][Q];
            if (l == 0) {
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int k = 0; k < Q; ++k) g[s][k] = f[s][k];
            } else {
                queue[l - 1].template complete<!STEADY>(f, c, m.whi && r == ny - 1, g);
                queue[l - 1].template push<!STEADY>(f, c, m.wlo && r + 1 == 0);
            }
            fused_node<LAT, S, float>(g, invD, relax, hk[l] ^ ((uint32_t)y * rowC + key0));
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int k = 0; k < Q; ++k) f[s][k] = g[s][k];
            if (l == K - 1 && mine && (STEADY || (r >= y0 && r < y1))) {
                const uint32_t at = ((uint32_t)y * (uint32_t)nx + c.x0) * 4u;
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int k = 0; k < Q; ++k) at_bytes(fout + (size_t)(s * Q + k) * grid.stride, at) = f[s][k];
            }
        }
    };
    const int count = y1 - y0 + 2 * (K - 1);
    // steady iterations: the last step is under way, its row is at least 1, and the row
    // loaded ahead is at most ny - 2
    const int s0 = y0 > 1 ? 2 * (K - 1) : 2 * K - 1 - y0;
    const int s1 = count - 1 < ny - 4 + K - y0 ? count - 1 : ny - 4 + K - y0;
    load_row<LAT, S, false>(fin, grid, c, m, m.place(y0 - (K - 1)), nxt);
    int j = 0;
    while (j < count) {
        if (j >= s0 && j <= s1) {
#pragma unroll 1
            for (; j <= s1; ++j) iteration(j, std::true_type{});
        } else {
            iteration(j, std::false_type{});
            ++j;
        }
    }
}

template <int LAT, int S, int K>
__global__ void __launch_bounds__(kFusedBlock, RowOccupancy<LAT, S>::value) k_fused_rows(FusedParams<S> p)
{
    await_previous_grid();
    const uint32_t step = *p.clock_in;
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.clock_out = step + K;
    const uint32_t part = blockIdx.x * (kFusedBlock / 32) + (threadIdx.x >> 5);
    const int strip = (int)(part % (uint32_t)p.strips), seg = (int)(part / (uint32_t)p.strips);
    if (seg >= p.segments) return;
    const int y0 = seg * p.rows, y1 = y0 + p.rows < p.ny ? y0 + p.rows : p.ny;  // the part's rows
    const RowGrid grid = {p.nx, p.ny, p.noflux, 0u, p.cells};
    march_rows<LAT, S, K, K - 1>(p.fin, p.fout, grid, strip, y0, y1, step, p.relax, p.co.invD);
}

// Lines (1D): a warp takes kLineBlocks runs of 32 consecutive nodes, a lane one node of
// each, loads its populations once, takes p.depth steps in registers (neighbours by
// shuffles) and stores the nodes that are not within `depth` of its ends.
constexpr int kLineBlocks = 4;
constexpr int kLineNodes = 32 * kLineBlocks;

template <int LAT, int S>
__global__ void __launch_bounds__(kFusedBlock, 4) k_fused_line(FusedParams<S> p, int depth)
{
    using L = Lattice<LAT>;
    constexpr int Q = L::Q, NP = kLineBlocks / 2;
    static_assert(L::DIM == 1, "lines are one-dimensional");
    await_previous_grid();
    const uint32_t step = *p.clock_in;
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.clock_out = step + depth;
    const int part = (int)(blockIdx.x * (kFusedBlock / 32) + (threadIdx.x >> 5));
    if (part >= p.strips) return;
    const int lane = threadIdx.x & 31, nx = p.nx;
    const int W = kLineNodes - 2 * depth;
    const int first = part * W, end = first + W < nx ? first + W : nx;  // nodes stored
    const bool wl = p.noflux & 1u, wr = p.noflux & 2u;
    uint32_t at[kLineBlocks];
    bool bl[kLineBlocks], br[kLineBlocks], any = false;
#pragma unroll
    for (int b = 0; b < kLineBlocks; ++b) {
        const int X = first - depth + 32 * b + lane;
        int m = X;
        if (wl) {
            m = X < 0 ? 0 : (X >= nx ? nx - 1 : X);
        } else if (X < 0 || X >= nx) {
            m = X % nx;
            if (m < 0) m += nx;
        }
        at[b] = (uint32_t)m;
        bl[b] = wl && X == 0;
        br[b] = wr && X == nx - 1;
        any |= bl[b] || br[b];
    }
    const bool wall = __any_sync(0xffffffffu, any);
    f2 f[NP][S][Q];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const float* base = p.fin + (size_t)(s * Q + k) * p.cells;
#pragma unroll
            for (int q = 0; q < NP; ++q) f[q][s][k] = pack2(base[at[2 * q]], base[at[2 * q + 1]]);
        }
    for (int l = 0; l < depth; ++l) {
        f2 g[NP][S][Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const int cx = L::cx(k);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                if (cx == 0) {
#pragma unroll
                    for (int q = 0; q < NP; ++q) g[q][s][k] = f[q][s][k];
                    continue;
                }
                // rotate every run by one lane; the lane that wrapped takes the next run's
                float t[kLineBlocks], v[kLineBlocks];
                const int from = (cx > 0 ? lane + 31 : lane + 1) & 31;
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    t[2 * q] = __shfl_sync(0xffffffffu, lo(f[q][s][k]), from);
                    t[2 * q + 1] = __shfl_sync(0xffffffffu, hi(f[q][s][k]), from);
                }
#pragma unroll
                for (int b = 0; b < kLineBlocks; ++b) {
                    v[b] = t[b];
                    if (cx > 0 && b > 0) v[b] = lane == 0 ? t[b - 1] : t[b];
                    if (cx < 0 && b + 1 < kLineBlocks) v[b] = lane == 31 ? t[b + 1] : t[b];
                }
                if (wall) {
                    const int o = opp<LAT>(k);
#pragma unroll
                    for (int b = 0; b < kLineBlocks; ++b)
                        if (cx > 0 ? bl[b] : br[b]) v[b] = (b & 1) ? hi(f[b / 2][s][o]) : lo(f[b / 2][s][o]);
                }
#pragma unroll
                for (int q = 0; q < NP; ++q) g[q][s][k] = pack2(v[2 * q], v[2 * q + 1]);
            }
        }
        const uint32_t hk = mix32((step + l) * 0x9e3779b9u);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const Key2 key = {hk ^ (at[2 * q] * 0x27d4eb2du), hk ^ (at[2 * q + 1] * 0x27d4eb2du)};
            fused_node<LAT, S, f2>(g[q], p.co.invD, p.relax, key);
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int k = 0; k < Q; ++k) f[q][s][k] = g[q][s][k];
        }
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            float* out = p.fout + (size_t)(s * Q + k) * p.cells;
#pragma unroll
            for (int b = 0; b < kLineBlocks; ++b) {
                const int X = first - depth + 32 * b + lane;
                if (X >= first && X < end) out[X] = (b & 1) ? hi(f[b / 2][s][k]) : lo(f[b / 2][s][k]);
            }
        }
}

// Steps one fused pass may take for a solver, or 1 where none applies.  Planes: three
// (D2Q5 ternary 4096^2: 152 us per step at two, 138 at three, 143 at four); with four or
// five species two (their queues fill the registers).  Lines: eight (10^7 nodes: 56, 50, 47.8
// and 45.7 us per step at two, three, four and eight; single steps 87).  The 3D lattices keep
// single steps: a marching pass of two steps over 32 x 10 columns with shared-memory
// exchange took 247 us per step on D3Q7 256^3 (265), but lost on grids below 200^3 (c. 62
// against 53 at 161 x 127 x 143), for a quarter of its work is redundant there.
template <int LAT, int S>
constexpr int fused_limit()
{
    return Lattice<LAT>::DIM == 1 ? (S <= 2 ? 8 : 1) : (Lattice<LAT>::DIM == 2 && S <= 4 ? (S <= 2 ? 3 : 2) : 1);
}

template <int LAT, int S, int K>
cudaError_t launch_rows(FusedParams<S>& p, const KArgs& a)
{
    const RowPlan plan = row_plan(Lattice<LAT>::Q, S, K, a.nx, a.ny, a.sms);
    p.strips = plan.strips;
    p.segments = plan.segments;
    p.rows = plan.rows;
    const uint32_t parts = (uint32_t)p.strips * (uint32_t)p.segments;
    return launch_chained(k_fused_rows<LAT, S, K>, (parts + 3) / 4, kFusedBlock, a.stream, p);
}

// p.steps steps (2 .. fused_limit) in one pass.
template <int LAT, int S>
cudaError_t launch_fused(const KArgs& a)
{
    constexpr int DIM = Lattice<LAT>::DIM;
    FusedParams<S> p;
    p.fin = static_cast<const float*>(a.fin);
    p.fout = static_cast<float*>(a.fout);
    p.nx = a.nx; p.ny = a.ny;
    p.cells = a.cells;
    p.noflux = a.noflux;
    p.relax = a.relax;
    p.clock_in = a.clock_in;
    p.clock_out = a.clock_out;
    p.co = make_coeffs<float>(a, 0.5);
    p.segments = 1;
    p.rows = 1;
    if constexpr (fused_limit<LAT, S>() < 2) {
        return cudaErrorInvalidValue;
    } else if constexpr (DIM == 1) {
        const int W = kLineNodes - 2 * a.steps;
        p.strips = (a.nx + W - 1) / W;
        return launch_chained(k_fused_line<LAT, S>, (uint32_t)(p.strips + 3) / 4, kFusedBlock, a.stream, p, a.steps);
    } else {
        switch (a.steps) {
            case 2: return launch_rows<LAT, S, 2>(p, a);
            case 3:
                if constexpr (fused_limit<LAT, S>() >= 3) return launch_rows<LAT, S, 3>(p, a);
            default: return cudaErrorInvalidValue;
        }
    }
}

}  // namespace lbms
