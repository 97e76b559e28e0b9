// fp_grid.cuh -- the count grid in two launches: sums of its coarser levels, and
// what a second pass needs to know about the rest of the grid.
//
// The 8^g cells are cut into tiles of 4096 consecutive ones, which are the cells
// of one level-(g - 4) node (g >= 4) or the whole grid.  k_grid_tiles, one block
// per tile, sums the four levels above the cells (eight cells a half thread, 64
// four lanes, 512 a warp, 4096 a block).  The second kernel of each user
// (k_merge_write, k_cells_open) is one block per tile too: the at most 512 tile
// sums are all it reads of the rest of the grid, and every block derives the
// levels above the tiles and the prefixes over the earlier tiles from them by
// itself -- no scan launches, no wait between blocks.  (The level-by-level sums,
// marks and three-launch scans took 16 launches in the merge and 13 in the
// octree stage; each launch costs about 2 us of host time and 2 - 5 us on the
// device, more than the 8 MB grid's reads and writes.)
#pragma once
#include "fp_internal.cuh"

namespace fp {

constexpr int kGtNT = 256;
constexpr int kGtPer = 16;                        // cells per thread
constexpr int kGtCells = kGtNT * kGtPer;          // 4096
constexpr int kGtMaxTiles = 512;                  // g = 7

inline int grid_tiles(int g) { return g <= 4 ? 1 : 1 << (3 * (g - 4)); }

FP_DEV uint32_t pyr_off(int l) { return ((1u << (3 * l)) - 1u) / 7u; }   // level l < g in the pyramid

// cells [base, base + 16) of the grid (0 beyond it)
FP_DEV void grid_load16(const uint32_t* p, uint32_t base, uint32_t cells, uint32_t v[kGtPer])
{
    if (base + kGtPer <= cells && (reinterpret_cast<uintptr_t>(p + base) & 15) == 0) {
#pragma unroll
        for (int q = 0; q < kGtPer / 4; ++q) {
            const uint4 x = *reinterpret_cast<const uint4*>(p + base + 4 * q);
            v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < kGtPer; ++q) v[q] = base + q < cells ? p[base + q] : 0u;
    }
}

// the four levels above this thread's cells
struct GridSums {
    uint32_t s1[2];   // its two runs of 8 cells (level g - 1)
    uint32_t s2;      // 64 cells: four lanes (level g - 2)
    uint32_t s3;      // 512 cells: the warp (level g - 3)
    uint32_t s4;      // 4096 cells: the block (level g - 4)
};

FP_DEV GridSums grid_sums(const uint32_t v[kGtPer], uint32_t* smem_warp /* 8 words */)
{
    GridSums s;
    s.s1[0] = s.s1[1] = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) { s.s1[0] += v[q]; s.s1[1] += v[8 + q]; }
    uint32_t x = s.s1[0] + s.s1[1];
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 1);
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 2);
    s.s2 = x;
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 4);
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 8);
    x += __shfl_xor_sync(0xFFFFFFFFu, x, 16);
    s.s3 = x;
    if ((threadIdx.x & 31) == 0) smem_warp[threadIdx.x >> 5] = x;
    __syncthreads();
    s.s4 = 0;
#pragma unroll
    for (int w = 0; w < kGtNT / 32; ++w) s.s4 += smem_warp[w];
    __syncthreads();
    return s;
}

// Chunk starts among this thread's cells (bit q: cell q starts a chunk) in a
// tile whose own node holds more than T points: of every cell the largest node
// with at most T points around it, or the cell, counted at the node's first cell.
FP_DEV uint32_t chunk_starts(const uint32_t v[kGtPer], const GridSums& s, uint64_t T)
{
    if (s.s3 <= T) return (threadIdx.x & 31) == 0 && s.s3 ? 1u : 0u;
    if (s.s2 <= T) return (threadIdx.x & 3) == 0 && s.s2 ? 1u : 0u;
    uint32_t f = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (s.s1[h] <= T) {
            f |= (s.s1[h] ? 1u : 0u) << (8 * h);
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) f |= (v[8 * h + q] ? 1u : 0u) << (8 * h + q);
        }
    }
    return f;
}

// Levels g - 1 .. g - 4 of the pyramid of `counts`; with `rcounts` (which may be
// another grid, of records) every tile's sum of it to rsum; with `starts` every
// tile's chunk starts under threshold T (of tiles above T; see chunk_starts).
// Also clears `zero` (nzero words) for the kernels behind.
static __global__ void __launch_bounds__(kGtNT) k_grid_tiles(const uint32_t* __restrict__ counts, int g,
                                                             uint32_t* __restrict__ pyr,
                                                             const uint32_t* __restrict__ rcounts, uint32_t* rsum,
                                                             uint32_t* starts, uint64_t T, uint32_t* zero, int nzero)
{
    __shared__ uint32_t s_warp[kGtNT / 32];
    const uint32_t cells = 1u << (3 * g), tile = blockIdx.x, base = tile * kGtCells + threadIdx.x * kGtPer;
    uint32_t v[kGtPer];
    grid_load16(counts, base, cells, v);
    const GridSums s = grid_sums(v, s_warp);
    if (base < cells) {
        const uint32_t i1 = base >> 3;
        pyr[pyr_off(g - 1) + i1] = s.s1[0];
        if (i1 + 1 < cells >> 3) pyr[pyr_off(g - 1) + i1 + 1] = s.s1[1];
        if (g >= 2 && (threadIdx.x & 3) == 0) pyr[pyr_off(g - 2) + (base >> 6)] = s.s2;
        if (g >= 3 && (threadIdx.x & 31) == 0) pyr[pyr_off(g - 3) + (base >> 9)] = s.s3;
        if (g >= 4 && threadIdx.x == 0) pyr[pyr_off(g - 4) + tile] = s.s4;
    }
    if (starts) {
        const uint32_t n = __reduce_add_sync(0xFFFFFFFFu, s.s4 > T ? __popc(chunk_starts(v, s, T)) : 0u);
        if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = n;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (int w = 0; w < kGtNT / 32; ++w) t += s_warp[w];
            starts[tile] = t;
        }
    }
    if (rsum) {
        uint32_t t = s.s4;
        if (rcounts != counts) {
            grid_load16(rcounts, base, cells, v);
            __syncthreads();
            t = grid_sums(v, s_warp).s4;
        }
        if (threadIdx.x == 0) rsum[tile] = t;
    }
    for (int q = tile * kGtNT + threadIdx.x; q < nzero; q += gridDim.x * kGtNT) zero[q] = 0;
}

// The levels above the tiles, in shared memory: t[0] the tiles' own counts, t[a]
// (a <= up) the nodes a levels above them.
struct GridTop {
    uint32_t t0[kGtMaxTiles], t1[kGtMaxTiles / 8], t2[kGtMaxTiles / 64], t3[1];
    // count of the node a levels above tile i
    FP_DEV uint32_t at(int a, uint32_t i) const
    {
        return a == 0 ? t0[i] : (a == 1 ? t1[i >> 3] : (a == 2 ? t2[i >> 6] : t3[0]));
    }
};

// fills G from the pyramid (g >= 4; else the one tile's sum `own`); returns the levels above the tiles
FP_DEV int grid_top(GridTop& G, const uint32_t* pyr, int g, uint32_t own)
{
    const int up = g > 4 ? g - 4 : 0;
    const uint32_t nt = 1u << (3 * up);
    for (uint32_t i = threadIdx.x; i < nt; i += kGtNT) G.t0[i] = up ? pyr[pyr_off(g - 4) + i] : own;
    __syncthreads();
    auto fold = [&](const uint32_t* from, uint32_t* to, uint32_t n) {
        for (uint32_t i = threadIdx.x; i < n; i += kGtNT) {
            uint32_t s = 0;
            for (int q = 0; q < 8; ++q) s += from[8 * i + q];
            to[i] = s;
        }
        __syncthreads();
    };
    if (up >= 1) fold(G.t0, G.t1, nt >> 3);
    if (up >= 2) fold(G.t1, G.t2, nt >> 6);
    if (up >= 3) fold(G.t2, G.t3, 1);
    return up;
}

template <typename T>
FP_DEV T block_sum(T v, T* smem_warp /* kGtNT / 32 words */)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0) smem_warp[threadIdx.x >> 5] = v;
    __syncthreads();
    T t = 0;
    for (int w = 0; w < kGtNT / 32; ++w) t += smem_warp[w];
    __syncthreads();
    return t;
}

}  // namespace fp
