// Several time steps in one pass on grids too small to fill the chip.
//
// A step of a small grid is a wait: the launch, the loads from L2 and the dependent
// arithmetic of one node take 1.7 us (FP32) however few nodes there are.  Here a block
// takes a tile of the grid with a margin of K - 1 nodes around it, one node per thread,
// and advances it K steps: the first gathers from memory, the others from shared memory,
// each on a region one node narrower, and the last one's tile is stored.  The margins are
// formed by several blocks at once, which costs nothing while SMs are idle.
//
// The node functions, faces (Dirichlet ones included) and rounding keys are those of
// k_step, so the populations are the same bit for bit.
#pragma once

#include "kernels.cuh"

namespace lbms {

// Collision of one node (k_step's arithmetic; FIXED as there).
template <int LAT, int S, typename T, bool FIXED>
__device__ __forceinline__ void advance_node(T (&f)[S][Lattice<LAT>::Q], const StepParams<T>& p, uint32_t key)
{
    using L = Lattice<LAT>;
    if constexpr (FIXED) {
        if (collide_fixed<L, S>(f, p.fixed.table)) return;
    }
    T xi[S + 1], xl[S + 1], L1[S][S], L2[S][S];
    mole_fractions<LAT, S, T>(f, xi);
    lambda_composition<S, T>(xi, p.co, p.relax, xl);
    relaxation_matrices<S, T>(xl, p.co.invD, T(1.0 / L::cs2()), p.relax, L1, L2);
    collide<LAT, S, T>(f, xi, L1, L2, key);
}

template <int LAT, int S, typename T, bool FIXED>
__global__ void __launch_bounds__(kTileThreads) k_step_tile(StepParams<T> p, Tiles t)
{
    using L = Lattice<LAT>;
    constexpr int Q = L::Q, DIM = L::DIM;
    extern __shared__ __align__(16) unsigned char raw[];
    T* const shared = reinterpret_cast<T*>(raw);
    // the thread's node: its place in the region, in the grid (wrapped along periodic axes)
    // and the first step on which it lies outside the region
    const int i = (int)threadIdx.x, region = t.rx * t.ry * t.rz, m = t.depth - 1;
    const int lx = i % t.rx, ly = DIM > 1 ? i / t.rx % t.ry : 0, lz = DIM > 2 ? i / (t.rx * t.ry) : 0;
    const int bx = (int)blockIdx.x % t.nx, by = (int)blockIdx.x / t.nx % t.ny, bz = (int)blockIdx.x / (t.nx * t.ny);
    const int vx = bx * t.tx + lx - m, vy = DIM > 1 ? by * t.ty + ly - m : 0, vz = DIM > 2 ? bz * t.tz + lz - m : 0;
    bool inside = i < region;
    auto place = [&](int v, int n, bool wall) {  // inside: not beyond a wall
        if (wall) {
            inside &= v >= 0 && v < n;
            return v;
        }
        const int r = v % n;
        return r < 0 ? r + n : r;
    };
    const int x = place(vx, p.g.nx, p.g.noflux & 1u), y = place(vy, p.g.ny, p.g.noflux & 4u);
    const int z = place(vz, p.g.nz, p.g.noflux & 16u);
    int edge = lx < t.rx - 1 - lx ? lx : t.rx - 1 - lx;  // distance from the region's edge
    if (DIM > 1) edge = min(edge, min(ly, t.ry - 1 - ly));
    if (DIM > 2) edge = min(edge, min(lz, t.rz - 1 - lz));
    const uint32_t cell = inside ? (uint32_t)((z * p.g.ny + y) * p.g.nx + x) : 0u;
    Neighbourhood h = neighbourhood<DIM, false>(p.g, cell);
    await_previous_grid();
    const uint32_t step = *p.clock_in;
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.clock_out = step + (uint32_t)t.depth;
    T f[S][Q];
    if (inside) {
        pull<LAT, S, T>(p.fin, p.g, cell, h, f, p.xb);
        advance_node<LAT, S, T, FIXED>(f, p, mix32(step * 0x9e3779b9u) ^ (cell * 0x27d4eb2du));
    }
    // within the region neighbours lie next to each other whatever the grid's wraps
    h.ox[0] = -1;
    h.ox[1] = 1;
    h.oy[0] = -t.rx;
    h.oy[1] = t.rx;
    h.oz[0] = -t.rx * t.ry;
    h.oz[1] = t.rx * t.ry;
    Geom g = p.g;
    g.cells = (uint32_t)region;  // plane stride of the shared copies
    for (int l = 1; l < t.depth; ++l) {
        T* const now = shared + (t.depth > 2 ? l & 1 : 0) * (size_t)region * (S * Q);
        if (inside && edge >= l - 1) {
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int k = 0; k < Q; ++k) now[(s * Q + k) * region + i] = f[s][k];
        }
        __syncthreads();
        if (inside && edge >= l) {
            pull<LAT, S, T>(now, g, (uint32_t)i, h, f, p.xb);
            advance_node<LAT, S, T, FIXED>(f, p, mix32((step + l) * 0x9e3779b9u) ^ (cell * 0x27d4eb2du));
        }
    }
    // the tile's own nodes (those beyond a ragged end belong to nobody, or wrapped to others)
    if (inside && edge >= m && vx < p.g.nx && vy < p.g.ny && vz < p.g.nz) {
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int k = 0; k < Q; ++k) p.fout[(size_t)(s * Q + k) * p.g.cells + cell] = f[s][k];
    }
}

template <int LAT, int S, typename T, bool FIXED>
cudaError_t launch_tile_of(const KArgs& a)
{
    const Tiles& t = a.tiles;
    const int region = t.rx * t.ry * t.rz;
    const size_t shared = (size_t)(t.depth > 2 ? 2 : 1) * region * S * Lattice<LAT>::Q * sizeof(T);
    // The limit belongs to the kernel, not to a launch, and other threads launch it too: every
    // one of them sets the same, the most a pass of it can take.
    constexpr size_t most = size_t(2) * kTileThreads * S * Lattice<LAT>::Q * sizeof(T);
    static_assert(most <= size_t(227) << 10, "more than a block has");
    if (shared > size_t(48) << 10) {
        cudaError_t e = cudaFuncSetAttribute(k_step_tile<LAT, S, T, FIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return e;
    }
    const uint32_t blocks = (uint32_t)t.nx * (uint32_t)t.ny * (uint32_t)((a.nz + t.tz - 1) / t.tz);
    return launch_chained_shared(k_step_tile<LAT, S, T, FIXED>, blocks, (uint32_t)(region + 31) / 32 * 32, shared, a.stream,
                                 make_step_params<T>(a), t);
}

template <int LAT, int S, typename T>
cudaError_t launch_tile(const KArgs& a)
{
    if constexpr (sizeof(T) == 8) {
        if (a.fixed.on) return launch_tile_of<LAT, S, T, true>(a);
    }
    return launch_tile_of<LAT, S, T, false>(a);
}

template <int LAT, typename T>
cudaError_t launch_tile_species(const KArgs& a)
{
    switch (a.n_species) {
        case 2: return launch_tile<LAT, 1, T>(a);
        case 3: return launch_tile<LAT, 2, T>(a);
        case 4:
            if constexpr (sizeof(T) == 4 && Lattice<LAT>::DIM < 3) return launch_tile<LAT, 3, T>(a);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbms
