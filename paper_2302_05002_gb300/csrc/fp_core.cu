// fp_core.cu -- bounds, preview decimation, count grid and chunk merge.
//
//   k_bounds_bulk      one pass over the cloud: per-axis min/max (Sec. 4.4) and,
//                      optionally, the preview compaction (Sec. 3 / Sec. 4.2):
//                      index i is kept iff splitmix64(first + i) % m == 0.  Kept
//                      points keep ascending index order through a single-pass
//                      scan with decoupled look-back across tiles.  Each tile
//                      arrives in shared memory by one bulk copy issued when the
//                      tile is claimed, in flight during the ranking and look-back.
//   k_keep, k_keep_write   the previews without extents: the uniform one, and
//                      the spatial one (with k_cell_min_hash before them).
//   k_count            count grid: one level-g Morton key per point, warp-
//                      aggregated atomics into an L2-resident 8^g histogram.
//   k_merge_write      with k_grid_tiles' sums of the grid: the chunk rule of
//                      Fig. "octree" (maximal nodes with 0 < count <= T, plus
//                      overflowing finest cells), listed in Morton preorder.
#include "fp_cluster.cuh"
#include "fp_grid.cuh"

namespace fp {

// ----------------------------------------------------------------- bounds
constexpr int kBdNT = 256;
constexpr int kBdIPT = 8;
constexpr int kBdTile = kBdNT * kBdIPT;   // 2048 points per tile

// The previews that need no extents, without a look-back.  Keep rule: the index
// hash is a multiple of the modulus (the uniform preview), or it is the smallest
// of the point's cell (the spatial one, whose keep bits k_cell_mark sets first).
// Only the kept points are read.  A block takes a segment of consecutive tiles; a
// warp takes ROWS rows of 32 points, lane r holds row r's keep bits.  When every
// block has counted its segment, a tile's output starts at the totals of the earlier
// segments plus its place in its own.
//   k_keep_all: both halves in one cooperative launch, the keep bits in shared
//     memory across the barrier (the uniform rule, up to kKeepTiles tiles a block);
//   k_keep, k_keep_write: in two launches (the spatial rule, and larger pieces,
//     whose bits are computed again).
// The hash takes 10 us of integer instructions for 8M points; the two launches of the
// uniform rule compute it twice.  (In one launch with a look-back, all tiles of a wave publish
// at about the same time and the last walks back over all of them: 38 us for 8M
// points, 25 us now.)
constexpr int kKeepSegs = 2048;
constexpr int kKeepRows = 32, kKeepRowsSmall = 8;   // rows per warp and tile

struct KeepScratch {
    uint32_t* words;      // spatial rule: keep bits, bit i & 31 of word i / 32 for point i
    uint32_t* before;     // per tile: kept points of its segment before it
    uint32_t* seg;        // per segment: kept points
    uint64_t ntiles, per; // tiles, tiles per segment
};

// uniform rule: keep bits of ROWS rows of 32 indices from i (this lane's in the first), row r's in lane r
template <int ROWS>
FP_DEV uint32_t keep_word(uint64_t i, uint64_t n, uint64_t first, const KeepMultiple& mult)
{
    uint32_t word = 0;
    const uint32_t left = (uint32_t)min(n - min(n, i), (uint64_t)(32 * ROWS));   // rows reach n at 32 r >= left
    const uint64_t v = first + i;
#pragma unroll 8
    for (int r = 0; r < ROWS; ++r) {
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, mult(v + 32 * r) && 32u * r < left);
        if ((int)(threadIdx.x & 31) == r) word = bal;
    }
    return word;
}

template <bool BITS, int ROWS>
__global__ void __launch_bounds__(kBdNT) k_keep(uint64_t n, uint64_t first, KeepMultiple mult, KeepScratch s)
{
    constexpr int kWarps = kBdNT / 32;
    __shared__ uint32_t s_tot[2][kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t t0 = blockIdx.x * s.per, t1 = min(s.ntiles, t0 + s.per);
    uint32_t run = 0;
    for (uint64_t tile = t0; tile < t1; ++tile) {
        const uint64_t w0 = (tile * kWarps + warp) * ROWS;
        const uint32_t word = BITS ? (lane < ROWS ? s.words[w0 + lane] : 0u)
                                   : keep_word<ROWS>(w0 * 32 + lane, n, first, mult);
        const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, __popc(word));
        uint32_t* tot = s_tot[(tile - t0) & 1];   // (two sets: one barrier a tile)
        if (lane == 0) tot[warp] = total;
        __syncthreads();
        if (threadIdx.x == 0) s.before[tile] = run;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) run += tot[w];
    }
    if (threadIdx.x == 0) s.seg[blockIdx.x] = run;
}

template <bool BITS, int ROWS>
__global__ void __launch_bounds__(kBdNT) k_keep_write(const fp_point* __restrict__ pts, uint64_t n, uint64_t first,
                                                      KeepMultiple mult, KeepScratch s, uint32_t nseg,
                                                      fp_point* __restrict__ out, uint64_t out_cap,
                                                      uint64_t* __restrict__ out_count, uint32_t* err)
{
    constexpr int kWarps = kBdNT / 32;
    __shared__ uint64_t s_sum[kWarps], s_all[kWarps];
    __shared__ uint32_t s_tot[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t tile = blockIdx.x;
    const uint32_t g = (uint32_t)(tile / s.per);
    const uint64_t w0 = (tile * kWarps + warp) * ROWS;
    const uint32_t word = BITS ? (lane < ROWS ? s.words[w0 + lane] : 0u)
                               : keep_word<ROWS>(w0 * 32 + lane, n, first, mult);
    uint64_t sum = 0, rest = 0;
    for (uint32_t q = threadIdx.x; q < nseg; q += kBdNT) {
        const uint32_t v = s.seg[q];
        if (q < g) sum += v;
        else rest += v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        rest += __shfl_xor_sync(0xFFFFFFFFu, rest, o);
    }
    uint32_t inc = __popc(word);
#pragma unroll
    for (int o = 1; o < ROWS; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 0) { s_sum[warp] = sum; s_all[warp] = sum + rest; }
    if (lane == ROWS - 1) s_tot[warp] = inc;
    __syncthreads();
    uint64_t at = s.before[tile], all = 0;
    for (int w = 0; w < kWarps; ++w) {
        at += s_sum[w];
        all += s_all[w];
        if (w < warp) at += s_tot[w];
    }
    if (tile == 0 && threadIdx.x == 0) {
        *out_count = all;
        if (all > out_cap) raise(err, FP_ERR_CAPACITY, 0);
    }
    const uint32_t ex = inc - __popc(word);   // of row `lane`
#pragma unroll 8
    for (int r = 0; r < ROWS; ++r) {
        const uint32_t bal = __shfl_sync(0xFFFFFFFFu, word, r);
        const uint32_t rx = __shfl_sync(0xFFFFFFFFu, ex, r);
        if ((bal >> lane) & 1u) {
            const uint64_t pos = at + rx + __popc(bal & lanemask_lt());
            if (pos < out_cap) st_point(out, pos, ld_point(pts, (w0 + r) * 32 + lane));
        }
    }
}

__global__ void __launch_bounds__(256) k_bounds_final(const int32_t* partial, int nblocks, uint64_t n,
                                                      fp_cube* cube)
{
    __shared__ int32_t s_red[6][8];
    int32_t lo[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, hi[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            lo[a] = min(lo[a], partial[b * 6 + a]);
            hi[a] = max(hi[a], partial[b * 6 + 3 + a]);
        }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int a = 0; a < 3; ++a) {
        lo[a] = __reduce_min_sync(0xFFFFFFFFu, lo[a]);
        hi[a] = __reduce_max_sync(0xFFFFFFFFu, hi[a]);
        if (lane == 0) { s_red[a][warp] = lo[a]; s_red[3 + a][warp] = hi[a]; }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    fp_cube c;
    for (int a = 0; a < 3; ++a) { c.o[a] = 0; c.mx[a] = 0; }
    c.S = 0;
    if (n > 0) {
        uint64_t ext = 0;
        for (int a = 0; a < 3; ++a) {
            int32_t l = s_red[a][0], h = s_red[3 + a][0];
            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) { l = min(l, s_red[a][w]); h = max(h, s_red[3 + a][w]); }
            c.o[a] = l;
            c.mx[a] = h;
            uint64_t e = (uint64_t)((int64_t)h - (int64_t)l);
            ext = e > ext ? e : ext;
        }
        c.S = ext + 1;
    }
    *cube = c;
}

__global__ void k_zero_count(uint64_t* out_count) { *out_count = 0; }

// ----------------------------------------------------------------- count
// Each block also keeps a small direct-mapped table of cells in shared memory:
// the first cell to reach a slot owns it for the block's lifetime and its hits
// are added there, flushed to the grid at the end.  Clouds with dense spots
// (scanner surroundings) send most of their hits to a few cells; those end up
// in the tables and stop contending for the same global counters.
constexpr int kCountSlots = 1024;

// cells (nullable): the level-g Morton cell of every point, for fp_distribute_cells
__global__ void __launch_bounds__(256) k_count(const fp_point* __restrict__ pts, uint64_t n,
                                               const fp_cube* __restrict__ cube, int g, uint32_t* __restrict__ counts,
                                               uint32_t* __restrict__ cells)
{
    __shared__ uint32_t s_tag[kCountSlots], s_cnt[kCountSlots];
    for (int q = threadIdx.x; q < kCountSlots; q += blockDim.x) { s_tag[q] = kNone; s_cnt[q] = 0; }
    __syncthreads();
    const CubeDev c = load_cube(cube);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x; i0 < n; i0 += stride * 4) {
        uint32_t key[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint64_t i = i0 + u * stride + threadIdx.x;
            key[u] = kNone;
            if (i < n) {
                int4 p = ld_point_cs(pts, i);
                key[u] = key_cell(p.x, p.y, p.z, c, g);
                if (cells) cells[i] = key[u];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            // a warp whose neighbouring lanes never share a cell (spread-out
            // points) adds directly; otherwise its equal cells are merged first
            const uint32_t knext = __shfl_down_sync(0xFFFFFFFFu, key[u], 1);   // (lane 31: its own)
            const bool twin = lane < 31 && key[u] != kNone && key[u] == knext;
            if (__any_sync(0xFFFFFFFFu, twin)) {
                uint32_t peers = __match_any_sync(0xFFFFFFFFu, key[u]);
                if (key[u] != kNone && lane == __ffs(peers) - 1) {
                    const uint32_t slot = (key[u] * 2654435761u) >> 22;   // 10-bit multiplicative hash
                    uint32_t t = s_tag[slot];
                    if (t == kNone) t = atomicCAS(&s_tag[slot], kNone, key[u]) == kNone ? key[u] : s_tag[slot];
                    if (t == key[u]) atomicAdd(&s_cnt[slot], (uint32_t)__popc(peers));
                    else atomicAdd(&counts[key[u]], (uint32_t)__popc(peers));
                }
            } else if (key[u] != kNone) {
                atomicAdd(&counts[key[u]], 1u);
            }
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < kCountSlots; q += blockDim.x)
        if (s_cnt[q]) atomicAdd(&counts[s_tag[q]], s_cnt[q]);
}

// Large clouds: one block per SM with a table of 32768 cells (128 KB).  A scan's
// points lie in some 10^5 cells and half of them in a few thousand, whose global
// counters queue up at their L2 slices (10^8 LiDAR points: 59 * 10^9 adds a second,
// uniform ones 143 * 10^9): most of their hits stay on chip instead.  A slot is one
// word, found by a bijective hash of the cell: its upper bits are the slot, its
// lower ones tell which of the slot's cells owns it (bits 24 .. 30, with a bit that
// says that one does; the count below), the first cell that comes.  A block tries
// the table with its first points and goes past it when less than an eighth of them
// brought an add that it took, which is where neighbouring lanes share cells (points
// in cell order: few adds, to cells that no other block is at), unless one cell alone
// holds an eighth: then every block is at the same few counters.  The next points are
// loaded while these are counted.  With the cells written: 10^8 LiDAR points in random
// order 1562 -> 518 us, scan by scan 1761 -> 934 us; 10^7 168 -> 87 and 127 -> 95 us;
// uniform, 10^8 710 -> 692 us (707 past the table), 4 * 10^6 32 -> 42 us (half the warps
// in flight and the trial), so smaller clouds keep the 1024-slot table of k_count.  In
// cell order, 10^8: 666 -> 469 us (518 with the table); 5 * 10^7 points in one cell 336 ->
// 264 us (1280 past the table), 95 in 100 of them 334 -> 276 us.
constexpr uint64_t kCountTable = 1ull << 23;             // from this many points on
constexpr int kCtNT = 1024, kCtIPT = 4;
constexpr int kCtBits = 15, kCtSlots = 1 << kCtBits;
constexpr int kCtLow = 21 - kCtBits;                    // bits of the hash below the slot
constexpr uint32_t kCtMul = 0x9E3779B1u & 0x1FFFFFu;    // odd: a bijection of 21 bits
constexpr int kCtProbe = 2;                             // rounds of kCtNT * kCtIPT points before the table is kept or given up
constexpr uint32_t kCtTrial = kCtProbe * kCtNT * kCtIPT / 8;   // an eighth of these points
constexpr uint64_t kCtMost = 1ull << 23;                // most points a block takes, so that counts stay below 2^24

constexpr uint32_t inverse21(uint32_t d)
{
    uint32_t x = d;
    for (int i = 0; i < 4; ++i) x *= 2 - d * x;
    return x & 0x1FFFFFu;
}

__global__ void __launch_bounds__(kCtNT, 1) k_count_table(const fp_point* __restrict__ pts, uint64_t n,
                                                          const fp_cube* __restrict__ cube, int g,
                                                          uint32_t* __restrict__ counts, uint32_t* __restrict__ cells)
{
    extern __shared__ uint32_t s_slot[];
    __shared__ uint32_t s_hits, s_hot;
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x; q < kCtSlots; q += kCtNT) s_slot[q] = 0;
    if (threadIdx.x == 0) s_hits = s_hot = 0;
    __syncthreads();
    const CubeDev c = load_cube(cube);
    auto flush = [&]() {
        __syncthreads();
        for (int q = threadIdx.x; q < kCtSlots; q += kCtNT) {
            const uint32_t w = s_slot[q];
            if (w & 0xFFFFFFu) {
                const uint32_t h = ((uint32_t)q << kCtLow) | ((w >> 24) & ((1u << kCtLow) - 1));
                atomicAdd(&counts[(h * inverse21(kCtMul)) & 0x1FFFFFu], w & 0xFFFFFFu);
                if ((w & 0xFFFFFFu) >= kCtTrial) s_hot = 1;
                s_slot[q] = w & 0xFF000000u;
            }
        }
        __syncthreads();
    };
    const uint64_t stride = (uint64_t)gridDim.x * kCtNT;
    bool table = true;
    uint32_t round = 0, hits = 0;
    int4 p[kCtIPT];   // the next round's points, on their way while this one is counted
    auto load = [&](uint64_t i0) {
#pragma unroll
        for (int u = 0; u < kCtIPT; ++u) {
            const uint64_t i = i0 + u * stride + threadIdx.x;
            if (i < n) p[u] = ld_point_cs(pts, i);
        }
    };
    load((uint64_t)blockIdx.x * kCtNT);
    for (uint64_t i0 = (uint64_t)blockIdx.x * kCtNT; i0 < n; i0 += stride * kCtIPT, ++round) {
        uint32_t key[kCtIPT];
#pragma unroll
        for (int u = 0; u < kCtIPT; ++u) {
            const uint64_t i = i0 + u * stride + threadIdx.x;
            key[u] = kNone;
            if (i < n) {
                key[u] = key_cell(p[u].x, p[u].y, p[u].z, c, g);
                if (cells) cells[i] = key[u];
            }
        }
        load(i0 + stride * kCtIPT);
#pragma unroll
        for (int u = 0; u < kCtIPT; ++u) {
            // neighbouring lanes that share a cell: equal cells are merged first
            uint32_t add = key[u] != kNone ? 1u : 0u;
            const uint32_t knext = __shfl_down_sync(0xFFFFFFFFu, key[u], 1);   // (lane 31: its own)
            if (__any_sync(0xFFFFFFFFu, lane < 31 && add && key[u] == knext)) {
                const uint32_t peers = __match_any_sync(0xFFFFFFFFu, key[u]);
                add = add && lane == __ffs(peers) - 1 ? __popc(peers) : 0u;
            }
            if (!add) continue;
            if (table) {
                const uint32_t h = (key[u] * kCtMul) & 0x1FFFFFu, tag = (h & ((1u << kCtLow) - 1)) | (1u << 6);
                uint32_t* w = &s_slot[h >> kCtLow];
                uint32_t has = *(volatile uint32_t*)w;
                if (has == 0) has = atomicCAS(w, 0u, tag << 24) == 0u ? tag << 24 : *(volatile uint32_t*)w;
                if (has >> 24 == tag) {
                    atomicAdd(w, add);
                    ++hits;
                    continue;
                }
            }
            atomicAdd(&counts[key[u]], add);
        }
        if (round == kCtProbe - 1) {
            hits = __reduce_add_sync(0xFFFFFFFFu, hits);
            if (lane == 0) atomicAdd(&s_hits, hits);
            flush();   // (its barriers publish the sum)
            table = s_hits >= kCtTrial || s_hot;
        }
    }
    flush();
}

// ----------------------------------------------------------------- merge
// One block per tile of the grid.  The chunks before the tile, and the points
// before it, are sums over the earlier tiles: of k_grid_tiles' starts where the
// tile's node holds more than T points, else 1 for the first tile of the largest
// node of at most T points around it.  10^9 points, 512 chunks: 0.10 -> 0.02 ms
// (16 launches -> 2).
__global__ void __launch_bounds__(kGtNT) k_merge_write(const uint32_t* __restrict__ counts, int g, uint64_t T,
                                                       const uint32_t* __restrict__ pyr,
                                                       const uint32_t* __restrict__ starts,
                                                       fp_chunk* __restrict__ chunks, uint32_t* num_chunks,
                                                       uint32_t* __restrict__ lut, uint64_t* __restrict__ offsets)
{
    __shared__ GridTop top;
    __shared__ uint32_t s_warp[kGtNT / 32];
    __shared__ uint64_t s_warp64[kGtNT / 32];
    const uint32_t cells = 1u << (3 * g), tile = blockIdx.x, base = tile * kGtCells + threadIdx.x * kGtPer;
    uint32_t v[kGtPer];
    grid_load16(counts, base, cells, v);
    const GridSums s = grid_sums(v, s_warp);
    const int up = grid_top(top, pyr, g, s.s4);
    // levels above a tile of at most T points up to its chunk's node
    auto height = [&](uint32_t i) {
        int h = 0;
        for (int a = 1; a <= up; ++a)
            if (top.at(a, i) <= T) h = a;
        return h;
    };
    uint32_t before = 0;
    uint64_t pts_before = 0;
    for (uint32_t i = threadIdx.x; i < tile; i += kGtNT) {
        pts_before += top.t0[i];
        if (top.t0[i] > T) {
            before += starts[i];
        } else {
            const int h = height(i);
            before += (i & ((1u << (3 * h)) - 1)) == 0 && top.at(h, i) ? 1u : 0u;
        }
    }
    before = block_sum(before, s_warp);
    pts_before = block_sum(pts_before, s_warp64);

    // this thread's chunk starts, and the level and count of the node around each
    uint32_t f;
    int h = 0;
    if (s.s4 > T) {
        f = chunk_starts(v, s, T);
    } else {
        h = height(tile);
        f = threadIdx.x == 0 && (tile & ((1u << (3 * h)) - 1)) == 0 && top.at(h, tile) ? 1u : 0u;
    }
    uint32_t total;
    uint32_t id = before + block_exclusive_scan<kGtNT, uint32_t>(__popc(f), s_warp, total);
    uint64_t ptotal;
    uint64_t at = pts_before + block_exclusive_scan<kGtNT, uint64_t>((uint64_t)s.s1[0] + s.s1[1], s_warp64, ptotal);
    if (tile == gridDim.x - 1 && threadIdx.x == 0) {
        *num_chunks = before + total;
        offsets[before + total] = pts_before + ptotal;
    }
    if (base >= cells) return;
    uint32_t l16[kGtPer];
#pragma unroll
    for (int q = 0; q < kGtPer; ++q) {
        if ((f >> q) & 1u) {
            int lev = g;   // (a grid of fewer than 4096 cells has no levels below 0)
            uint32_t cnt = v[q];
            if (s.s4 <= T) { lev = g - 4 - h; cnt = top.at(h, tile); }
            else if (s.s3 <= T) { lev = g - 3; cnt = s.s3; }
            else if (s.s2 <= T) { lev = g - 2; cnt = s.s2; }
            else if (s.s1[q >> 3] <= T) { lev = g - 1; cnt = s.s1[q >> 3]; }
            lev = max(lev, 0);
            fp_chunk ch;
            ch.key = (base + q) >> (3 * (g - lev));
            ch.count = cnt;
            ch.level = (uint32_t)lev;
            chunks[id] = ch;
            offsets[id] = at;
            ++id;
        }
        at += v[q];
        l16[q] = v[q] ? id - 1 : kNone;
    }
    if (base + kGtPer <= cells && (reinterpret_cast<uintptr_t>(lut + base) & 15) == 0) {
#pragma unroll
        for (int q = 0; q < kGtPer; q += 4)
            *reinterpret_cast<uint4*>(lut + base + q) = make_uint4(l16[q], l16[q + 1], l16[q + 2], l16[q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < kGtPer; ++q)
            if (base + q < cells) lut[base + q] = l16[q];
    }
}

// The bounds + preview pass of the main path: the tile's 32 KB of points are
// brought into shared memory by one bulk copy (cp.async.bulk, completion on an
// mbarrier) issued when the tile is claimed, so the copy is in flight while the
// keep flags are ranked and the tile's output offset is found by decoupled
// look-back; extents and kept points are then read from shared memory.  Few
// registers and 32 KB of shared memory per block: six blocks per SM, each with
// a whole tile in flight (2048-point tiles measured faster than 4096 and 1024).
// A second buffer per block, with the next tile claimed ahead, is slower: the
// claimed tile publishes its keep count only when its block reaches it, and
// every later tile's look-back waits for that.  Waits are bounded
// (FP_ERR_TIMEOUT).
constexpr size_t kBdBulkSmem = sizeof(int4) * kBdTile;

template <bool DECIM>
__global__ void __launch_bounds__(kBdNT) k_bounds_bulk(const fp_point* __restrict__ pts, uint64_t n, uint64_t first,
                                                       KeepMultiple mult, fp_point* __restrict__ out, uint64_t out_cap,
                                                       uint64_t* __restrict__ out_count, int32_t* __restrict__ partial,
                                                       uint64_t* tile_status, uint32_t* tile_counter, uint64_t ntiles,
                                                       uint32_t* err)
{
    extern __shared__ __align__(128) int4 s_pts[];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_cnt[kBdIPT][kBdNT / 32];
    __shared__ uint64_t s_base;
    __shared__ int32_t s_red[6][kBdNT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t lo[3] = {INT32_MAX, INT32_MAX, INT32_MAX};
    int32_t hi[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
    if (threadIdx.x == 0) mbar_init(&s_bar, 1);
    uint32_t nwait = 0;
    for (;;) {
        __syncthreads();   // the previous tile's reads of s_pts are done
        if (threadIdx.x == 0) {
            const uint32_t t = atomicAdd(tile_counter, 1u);
            s_tile = t;
            if (t < ntiles) {
                const uint64_t b = (uint64_t)t * kBdTile;
                const uint32_t bytes = (uint32_t)(sizeof(int4) * min((uint64_t)kBdTile, n - b));
                fence_async_smem();
                mbar_expect_tx(&s_bar, bytes);
                bulk_g2s(s_pts, reinterpret_cast<const int4*>(pts) + b, bytes, &s_bar);
            }
        }
        __syncthreads();
        const uint64_t tile = s_tile;
        if (tile >= ntiles) break;
        const uint64_t base = tile * kBdTile;

        uint32_t keepmask = 0;
        if (DECIM) {
#pragma unroll
            for (int r = 0; r < kBdIPT; ++r) {
                const uint64_t i = base + (uint64_t)r * kBdNT + threadIdx.x;
                const bool k = i < n && mult(first + i);
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, k);
                if (lane == 0) s_cnt[r][warp] = __popc(bal);
                keepmask |= (uint32_t)k << r;
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                constexpr int per = kBdIPT * (kBdNT / 32) / 32;
                uint32_t v[per];
                uint32_t s = 0;
#pragma unroll
                for (int q = 0; q < per; ++q) {
                    const int e = lane * per + q;
                    v[q] = s_cnt[e / (kBdNT / 32)][e % (kBdNT / 32)];
                    s += v[q];
                }
                uint32_t x = s;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                    if (lane >= o) x += y;
                }
                const uint32_t total = __shfl_sync(0xFFFFFFFFu, x, 31);
                uint32_t ex = x - s;
#pragma unroll
                for (int q = 0; q < per; ++q) {
                    const int e = lane * per + q;
                    s_cnt[e / (kBdNT / 32)][e % (kBdNT / 32)] = ex;
                    ex += v[q];
                }
                const uint64_t excl = preview_base(tile_status, tile, ntiles, total, out_cap, out_count, err);
                if (lane == 0) s_base = excl;
            }
        }
        // the tile's points have landed (bounded wait; on a time-out the copy is
        // given a second bounded wait to land before the block leaves)
        const bool ok = mbar_wait(&s_bar, nwait & 1);
        ++nwait;
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) raise(err, FP_ERR_TIMEOUT);
            mbar_wait(&s_bar, (nwait - 1) & 1);
            break;
        }
#pragma unroll 4
        for (int r = 0; r < kBdIPT; ++r) {
            const uint64_t i = base + (uint64_t)r * kBdNT + threadIdx.x;
            if (i < n) {
                const int4 p = s_pts[r * kBdNT + threadIdx.x];
                lo[0] = min(lo[0], p.x); hi[0] = max(hi[0], p.x);
                lo[1] = min(lo[1], p.y); hi[1] = max(hi[1], p.y);
                lo[2] = min(lo[2], p.z); hi[2] = max(hi[2], p.z);
            }
        }
        if (DECIM) {
#pragma unroll 4
            for (int r = 0; r < kBdIPT; ++r) {
                const bool kept = (keepmask >> r) & 1u;
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, kept);
                if (kept) {
                    const uint64_t pos = s_base + s_cnt[r][warp] + __popc(bal & lanemask_lt());
                    if (pos < out_cap) st_point(out, pos, s_pts[r * kBdNT + threadIdx.x]);
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = __reduce_min_sync(0xFFFFFFFFu, lo[a]);
        hi[a] = __reduce_max_sync(0xFFFFFFFFu, hi[a]);
    }
    if (lane == 0)
        for (int a = 0; a < 3; ++a) { s_red[a][warp] = lo[a]; s_red[3 + a][warp] = hi[a]; }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int a = threadIdx.x;
        int32_t v = s_red[a][0];
        for (int w = 1; w < kBdNT / 32; ++w) v = a < 3 ? min(v, s_red[a][w]) : max(v, s_red[a][w]);
        partial[blockIdx.x * 6 + a] = v;
    }
}

// ----------------------------------------------------------------- host side
// the carve of the preview passes: block partials (grid <= 8 per SM), one
// look-back word per tile and the tile counter behind them (cleared together)
struct BoundsScratch {
    int32_t* partial;
    uint64_t* status;      // [ntiles], then the counter
    uint32_t* counter;
    uint64_t ntiles;       // of kBdTile points (the previews' larger tiles use fewer words)
};

static BoundsScratch bounds_carve(const Workspace& ws, uint64_t n, int num_sms)
{
    BoundsScratch b;
    b.ntiles = (n + kBdTile - 1) / kBdTile;
    b.partial = ws.take<int32_t>(6 * (size_t)num_sms * 8);
    b.status = ws.take<uint64_t>(b.ntiles + 1);
    b.counter = reinterpret_cast<uint32_t*>(b.status + b.ntiles);
    return b;
}

size_t bounds_ws_bytes(uint64_t n, int num_sms)   // (the uniform preview's tile counts take less)
{
    Workspace dry;
    bounds_carve(dry, n, num_sms);
    return dry.used;
}

constexpr int kKeepTiles = 24;   // 1 KB of keep bits a tile, eight blocks per SM

__global__ void __launch_bounds__(kBdNT, 8) k_keep_all(const fp_point* __restrict__ pts, uint64_t n, uint64_t first,
                                                       KeepMultiple mult, KeepScratch s, uint32_t* bar,
                                                       fp_point* __restrict__ out, uint64_t out_cap,
                                                       uint64_t* __restrict__ out_count, uint32_t* err)
{
    constexpr int kWarps = kBdNT / 32, ROWS = kKeepRows;
    extern __shared__ uint32_t s_words[];   // [tiles of the block][kWarps][32]
    __shared__ uint32_t s_tot[kKeepTiles][kWarps];
    __shared__ uint64_t s_sum[kWarps], s_all[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t t0 = blockIdx.x * s.per, t1 = min(s.ntiles, t0 + s.per);
    const int nt = (int)(t1 - t0);
    for (int t = 0; t < nt; ++t) {
        const uint32_t word = keep_word<ROWS>(((t0 + t) * kWarps + warp) * (32 * ROWS) + lane, n, first, mult);
        s_words[(t * kWarps + warp) * 32 + lane] = word;
        const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, __popc(word));
        if (lane == 0) s_tot[t][warp] = total;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int t = 0; t < nt; ++t)
            for (int w = 0; w < kWarps; ++w) {   // kept points of the segment before the tile's warp
                const uint32_t v = s_tot[t][w];
                s_tot[t][w] = run;
                run += v;
            }
        s.seg[blockIdx.x] = run;
    }
    if (!grid_barrier(bar, 1, err)) return;
    uint64_t sum = 0, rest = 0;
    for (uint32_t q = threadIdx.x; q < gridDim.x; q += kBdNT) {
        const uint32_t v = s.seg[q];
        if (q < blockIdx.x) sum += v;
        else rest += v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        rest += __shfl_xor_sync(0xFFFFFFFFu, rest, o);
    }
    if (lane == 0) { s_sum[warp] = sum; s_all[warp] = sum + rest; }
    __syncthreads();
    uint64_t base = 0, all = 0;
    for (int w = 0; w < kWarps; ++w) { base += s_sum[w]; all += s_all[w]; }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *out_count = all;
        if (all > out_cap) raise(err, FP_ERR_CAPACITY, 0);
    }
    for (int t = 0; t < nt; ++t) {
        const uint32_t word = s_words[(t * kWarps + warp) * 32 + lane];
        uint32_t inc = __popc(word);
#pragma unroll
        for (int o = 1; o < ROWS; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        const uint64_t at = base + s_tot[t][warp];
        const uint32_t ex = inc - __popc(word);
        const uint64_t i0 = ((t0 + t) * kWarps + warp) * (32 * ROWS) + lane;
#pragma unroll 8
        for (int r = 0; r < ROWS; ++r) {
            const uint32_t bal = __shfl_sync(0xFFFFFFFFu, word, r);
            const uint32_t rx = __shfl_sync(0xFFFFFFFFu, ex, r);
            if ((bal >> lane) & 1u) {
                const uint64_t pos = at + rx + __popc(bal & lanemask_lt());
                if (pos < out_cap) st_point(out, pos, ld_point(pts, i0 + 32 * r));
            }
        }
    }
}

// the carve of the previews without extents
static KeepScratch keep_carve(const Workspace& ws, uint64_t n, int rows, bool bits)
{
    KeepScratch s;
    const uint64_t tile = (uint64_t)kBdNT * rows;
    s.ntiles = (n + tile - 1) / tile;
    s.per = std::max<uint64_t>(1, (s.ntiles + kKeepSegs - 1) / kKeepSegs);
    s.words = bits ? ws.take<uint32_t>(s.ntiles * (tile / 32)) : nullptr;
    s.before = ws.take<uint32_t>(s.ntiles);
    s.seg = ws.take<uint32_t>(kKeepSegs);
    return s;
}

static size_t keep_bytes(uint64_t n, int rows, bool bits)
{
    Workspace dry;
    keep_carve(dry, n, rows, bits);
    return dry.used;
}

template <bool BITS, int ROWS>
static void keep_launch(const KeepScratch& s, const fp_point* pts, uint64_t n, uint64_t first, uint32_t modulus,
                        fp_point* out, uint64_t out_cap, uint64_t* out_count, const Workspace& ws, cudaStream_t st)
{
    const uint32_t nseg = (uint32_t)((s.ntiles + s.per - 1) / s.per);
    k_keep<BITS, ROWS><<<nseg, kBdNT, 0, st>>>(n, first, KeepMultiple::of(modulus), s);
    k_keep_write<BITS, ROWS><<<(unsigned)s.ntiles, kBdNT, 0, st>>>(pts, n, first, KeepMultiple::of(modulus), s, nseg, out,
                                                                   out_cap, out_count, ws.err);
}

cudaError_t launch_bounds_decimate(const fp_point* pts, uint64_t n, fp_cube* cube, bool bounds, bool decim,
                                   uint64_t first, uint32_t modulus, fp_point* out, uint64_t out_cap,
                                   uint64_t* out_count, const Workspace& ws, cudaStream_t st)
{
    cudaError_t e;
    if (decim && n == 0) k_zero_count<<<1, 1, 0, st>>>(out_count);
    if (!bounds) {
        KTimerScope kt(FP_KERNEL_BOUNDS_DECIMATE, st);
        if (n == 0) return cudaGetLastError();
        // tiles of 2048 points in two launches while fewer than four tiles of 8192 an SM would leave most of the GPU
        // without work; those, as many blocks as are resident, in one launch up to kKeepTiles a block, else in two
        constexpr uint64_t kTile = (uint64_t)kBdNT * kKeepRows;
        if ((n + kTile - 1) / kTile < (uint64_t)ws.num_sms * 4) {
            keep_launch<false, kKeepRowsSmall>(keep_carve(ws, n, kKeepRowsSmall, false), pts, n, first, modulus, out,
                                               out_cap, out_count, ws, st);
            return cudaGetLastError();
        }
        const KeepScratch two = keep_carve(ws, n, kKeepRows, false);
        uint32_t* bar = ws.take<uint32_t>(1);
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_keep_all, kBdNT, kKeepTiles * kBdNT * 4)))
            return e;
        const uint64_t blocks = std::min<uint64_t>((uint64_t)std::max(per_sm, 1) * ws.num_sms, kKeepSegs);
        KeepScratch s = two;
        s.per = (s.ntiles + blocks - 1) / blocks;
        if (s.per > (uint64_t)kKeepTiles) {
            keep_launch<false, kKeepRows>(two, pts, n, first, modulus, out, out_cap, out_count, ws, st);
            return cudaGetLastError();
        }
        if ((e = cudaMemsetAsync(bar, 0, sizeof(uint32_t), st))) return e;
        return coop_launch(k_keep_all, (unsigned)((s.ntiles + s.per - 1) / s.per), kBdNT, s.per * kBdNT * 4, st, pts, n,
                           first, KeepMultiple::of(modulus), s, bar, out, out_cap, out_count, ws.err);
    }
    const BoundsScratch b = bounds_carve(ws, n, ws.num_sms);
    const int grid = (int)std::min<uint64_t>(b.ntiles ? b.ntiles : 1, (uint64_t)ws.num_sms * 8);
    if (n) {
        if (decim) e = cudaMemsetAsync(b.status, 0, (b.ntiles + 1) * sizeof(uint64_t), st);
        else e = cudaMemsetAsync(b.counter, 0, sizeof(uint32_t), st);
        if (e) return e;
        KTimerScope kt(FP_KERNEL_BOUNDS_DECIMATE, st);
        auto kern = decim ? k_bounds_bulk<true> : k_bounds_bulk<false>;   // points by bulk copy into shared memory
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBdBulkSmem))) return e;
        kern<<<grid, kBdNT, kBdBulkSmem, st>>>(pts, n, first, KeepMultiple::of(decim ? modulus : 1), out, out_cap, out_count,
                                               b.partial, b.status, b.counter, b.ntiles, ws.err);
    }
    k_bounds_final<<<1, 256, 0, st>>>(b.partial, n ? grid : 0, n, cube);
    return cudaGetLastError();
}

// ----------------------------------------------------- spatial preview
// Spatially constrained random sampler (the alternative preview the paper
// proposes for clouds whose file order makes the uniform one uneven, Sec. 6):
// of the points of every occupied cell of the 2^level grid, the one with the
// smallest splitmix64(first + i) is kept (a uniformly random point of the cell,
// the same on every run).  One pass over the points takes each cell's smallest
// hash; the hash is a bijection, so the index of the point it is from follows from
// it, and the points of all cells are compacted in index order as the uniform
// preview's are.  (A second pass over the points, comparing each one's hash with
// its cell's smallest: 10^8 points, 800 us; 75 us now.)  The cube is the caller's and
// may be another cloud's: points outside it fall into the cells that repeat there.
constexpr int kMinIPT = 4, kMinCtas = 5;

__global__ void __launch_bounds__(256, kMinCtas) k_cell_min_hash(const fp_point* __restrict__ pts, uint64_t n,
                                                                 uint64_t first, const fp_cube* cube_p, int level,
                                                                 unsigned long long* cell_min)
{
    const CubeDev cube = load_cube(cube_p);
    // a cell's running minimum only falls: a hash not below any value read for
    // it (however stale) cannot be the minimum, and the atomic is skipped --
    // in a cell of c points in random order about ln c atomics remain.  (Read
    // through L1: an SM's own atomics drop its stale line; 0.62 -> 0.54 ms at 10^8.)
    // Bound by instructions: without a test per point and with no more blocks than
    // are resident 0.54 -> 0.45 ms, the same at 2 to 8 points and 3 to 8 blocks an SM;
    // 0.43 ms with the shorter cell arithmetic (0.42 without the masks of points outside).
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i0 + (kMinIPT - 1) * stride < n; i0 += stride * kMinIPT) {
        int4 q[kMinIPT];
#pragma unroll
        for (int u = 0; u < kMinIPT; ++u) q[u] = ld_point_cs(pts, i0 + u * stride);   // points, then minima, in flight together
        uint32_t cell[kMinIPT];
        unsigned long long seen[kMinIPT];
#pragma unroll
        for (int u = 0; u < kMinIPT; ++u) {
            cell[u] = key_cell_any(q[u].x, q[u].y, q[u].z, cube, level);
            seen[u] = cell_min[cell[u]];
        }
#pragma unroll
        for (int u = 0; u < kMinIPT; ++u) {
            const unsigned long long h = splitmix64(first + i0 + u * stride);
            if (h < seen[u]) atomicMin(cell_min + cell[u], h);
        }
    }
    for (; i0 < n; i0 += stride) {
        const int4 q = ld_point_cs(pts, i0);
        unsigned long long* slot = cell_min + key_cell_any(q.x, q.y, q.z, cube, level);
        const unsigned long long h = splitmix64(first + i0);
        if (h < *slot) atomicMin(slot, h);
    }
}

size_t spatial_ws_bytes(uint64_t n, int level, int num_sms)
{
    (void)num_sms;
    return Workspace::bytes_for({sizeof(uint64_t) << (3 * level)}) + keep_bytes(n, kKeepRows, true);
}

constexpr uint64_t inverse64(uint64_t d)   // d odd, modulo 2^64: three bits right, doubled by every step
{
    uint64_t x = d;
    for (int i = 0; i < 5; ++i) x *= 2 - d * x;
    return x;
}

// the v with splitmix64(v) = z: every step of the hash undone
FP_DEV uint64_t splitmix64_inverse(uint64_t z)
{
    constexpr uint64_t m1 = inverse64(0xBF58476D1CE4E5B9ull), m2 = inverse64(0x94D049BB133111EBull);
    z = (z ^ (z >> 31) ^ (z >> 62)) * m2;
    z = (z ^ (z >> 27) ^ (z >> 54)) * m1;
    return (z ^ (z >> 30) ^ (z >> 60)) - 0x9E3779B97F4A7C15ull;
}

// keep bits of the points whose hashes the cells' smallest are.  A cell of ~0 is
// empty, or holds only the one point whose hash that is: thread 0 looks at it.
__global__ void __launch_bounds__(256) k_cell_mark(const uint64_t* __restrict__ cell_min, uint32_t cells,
                                                   const fp_point* pts, uint64_t n, uint64_t first,
                                                   const fp_cube* cube_p, int level, uint32_t* words)
{
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= cells) return;
    const uint64_t h = cell_min[m], i = splitmix64_inverse(h) - first;
    if (h != ~0ull && i < n) atomicOr(&words[i >> 5], 1u << (i & 31));
    if (m == 0) {
        const uint64_t last = splitmix64_inverse(~0ull) - first;
        if (last < n) {
            const CubeDev cube = load_cube(cube_p);
            const int4 p = ld_point(pts, last);
            if (cell_min[key_cell_any(p.x, p.y, p.z, cube, level)] == ~0ull)
                atomicOr(&words[last >> 5], 1u << (last & 31));
        }
    }
}

cudaError_t launch_preview_spatial(const fp_point* pts, uint64_t n, const fp_cube* cube, int level, uint64_t first,
                                   fp_point* out, uint64_t out_cap, uint64_t* out_count, const Workspace& ws,
                                   cudaStream_t st)
{
    const uint64_t cells = 1ull << (3 * level);
    uint64_t* cell_min = ws.take<uint64_t>(cells);
    cudaError_t e;
    if (n == 0) {
        k_zero_count<<<1, 1, 0, st>>>(out_count);
        return cudaGetLastError();
    }
    if ((e = cudaMemsetAsync(cell_min, 0xFF, cells * sizeof(uint64_t), st))) return e;
    const int gm = (int)std::min<uint64_t>((n + 255) / 256, (uint64_t)ws.num_sms * kMinCtas);
    k_cell_min_hash<<<gm, 256, 0, st>>>(pts, n, first, cube, level, reinterpret_cast<unsigned long long*>(cell_min));
    const KeepScratch s = keep_carve(ws, n, kKeepRows, true);
    if ((e = cudaMemsetAsync(s.words, 0, s.ntiles * kBdNT * kKeepRows / 8, st))) return e;
    k_cell_mark<<<(unsigned)((cells + 255) / 256), 256, 0, st>>>(cell_min, (uint32_t)cells, pts, n, first, cube, level,
                                                                 s.words);
    keep_launch<true, kKeepRows>(s, pts, n, first, 1, out, out_cap, out_count, ws, st);
    return cudaGetLastError();
}

cudaError_t launch_count(const fp_point* pts, uint64_t n, const fp_cube* cube, int g, uint32_t* counts,
                         bool accumulate, uint32_t* cells, const Workspace& ws, cudaStream_t st)
{
    const uint64_t ncell = 1ull << (3 * g);
    if (!accumulate) {
        cudaError_t e = cudaMemsetAsync(counts, 0, ncell * sizeof(uint32_t), st);
        if (e) return e;
    }
    if (n == 0) return cudaSuccess;
    uint64_t want = (n + 1023) / 1024;
    int grid = (int)std::min<uint64_t>(want, (uint64_t)ws.num_sms * 8);
    KTimerScope kt(FP_KERNEL_COUNT, st);
    if (n >= kCountTable) {
        const int smem = kCtSlots * (int)sizeof(uint32_t);
        cudaError_t e = cudaFuncSetAttribute(k_count_table, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e) return e;
        const unsigned blocks = (unsigned)std::max<uint64_t>(ws.num_sms, n / kCtMost + 1);   // (n < 2^30: 152 are enough)
        k_count_table<<<blocks, kCtNT, smem, st>>>(pts, n, cube, g, counts, cells);
        return cudaGetLastError();
    }
    k_count<<<grid, 256, 0, st>>>(pts, n, cube, g, counts, cells);
    return cudaGetLastError();
}

// the carve of launch_merge: the pyramid, one word of chunk starts per tile
size_t merge_ws_bytes(int g)
{
    const uint64_t npyr = ((1ull << (3 * g)) - 1) / 7;
    return Workspace::bytes_for({(npyr ? npyr : 1) * 4, (size_t)grid_tiles(g) * 4});
}

cudaError_t launch_merge(const uint32_t* counts, int g, uint64_t T, fp_chunk* chunks, uint32_t* num_chunks,
                         uint32_t* lut, uint64_t* offsets, const Workspace& ws, cudaStream_t st)
{
    const uint64_t npyr = ((1ull << (3 * g)) - 1) / 7;
    uint32_t* pyr = ws.take<uint32_t>(npyr ? npyr : 1);
    const int nt = grid_tiles(g);
    uint32_t* starts = ws.take<uint32_t>(nt);
    k_grid_tiles<<<nt, kGtNT, 0, st>>>(counts, g, pyr, nullptr, nullptr, starts, T, nullptr, 0);
    k_merge_write<<<nt, kGtNT, 0, st>>>(counts, g, T, pyr, starts, chunks, num_chunks, lut, offsets);
    return cudaGetLastError();
}

}  // namespace fp
