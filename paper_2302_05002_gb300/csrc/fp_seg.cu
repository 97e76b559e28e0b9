// fp_seg.cu -- setup and launch of the chunk-segmented scatter (fp_seg.cuh).
#include "fp_cluster.cuh"
#include "fp_seg.cuh"

namespace fp {

// Node id of (key, level) in a preorder node table, kNone if absent.  Preorder
// is lexicographic in (key << 3 (21 - level), level): a node's cell starts at
// its first descendant's, and the ancestor comes first.
FP_DEV uint32_t find_node(const fp_node* nodes, uint32_t M, uint64_t key, uint32_t level)
{
    const uint64_t K = key << (3 * (kKeyLevels - level));
    uint32_t a = 0, b = M;
    while (a < b) {
        const uint32_t m = (a + b) >> 1;
        const uint32_t lm = nodes[m].level;
        const uint64_t km = nodes[m].key << (3 * (kKeyLevels - lm));
        if (km < K || (km == K && lm < level)) a = m + 1;
        else b = m;
    }
    if (a < M && nodes[a].level == level && nodes[a].key == key) return a;
    return kNone;
}

// What the segmented scatter needs before its passes, in three steps:
//   A (owner layout): first point of every node (prefix of the owned counts),
//     the scratch words cleared;
//   B: per chunk its node, digits and tiles, and the flags of the nodes inside
//     chunk subtrees; the look-back words of tiles that others will read cleared;
//   C (owner layout): the nodes outside every chunk subtree ranked in order, and
//     where each one's staged points start.
// Three launches: A's sums of segments of the node table (k_seg_nodes); B, with A's
// prefixes (k_seg_chunks), both on the whole GPU; C by one cluster (k_seg_plan), which
// reads five bytes a node.  One cluster also does all of A where nothing else is asked
// for (clouds of up to 2^21 points).  (A by one cluster everywhere: the plan of 2.4 *
// 10^6 nodes 840 us, 320 us now; of 2257, 25 and 23 us.)
constexpr uint32_t kSegNodes = 512;   // segments of the node table
struct SegPlan {
    int owner;               // 1: owner layout, 0: leaf grouping
    int step_c;              // k_seg_plan: 0: A, 1: C
    fp_node* nodes;
    const uint32_t* num_nodes;
    uint32_t node_cap;
    const fp_chunk* chunks;
    const uint32_t* num_chunks;
    const uint64_t* offsets;
    uint64_t kmax, n, tiles_max;
    uint32_t *seg_lo, *seg_nb;
    SegTile* tiles[2];
    uint32_t* status[2];
    uint32_t* cnt;           // SegScratch::cnt
    uint8_t* inside;
    uint64_t* part;
    // owner layout
    uint32_t* nown;
    uint64_t* first;
    uint32_t *rank, *list, *nrank, *soff, *nm, *nstaged;
    uint32_t *hist, *hist2;  // the sorts' histograms, cleared in A
    uint32_t* err;
};

// A's scratch words (thread t of nt)
FP_DEV void seg_clear(const SegPlan& a, uint32_t t, uint32_t nt, uint32_t M)
{
    for (uint32_t q = t; q < 8; q += nt) a.cnt[q] = 0;
    for (uint32_t q = t; q < (uint32_t)kSortHistWords; q += nt) {
        a.hist[q] = 0;
        if (a.hist2) a.hist2[q] = 0;
    }
    if (a.owner && t == 0) { *a.nm = M; *a.nstaged = 0; }
}

// nodes of a segment: a multiple of 256, so that its words can be read as vectors
FP_DEV uint32_t seg_nodes_per(uint32_t M) { return ((M + kSegNodes - 1) / kSegNodes + 255) & ~255u; }

// step A, first half: scratch words, owned counts, and their sum per segment
__global__ void __launch_bounds__(256) k_seg_nodes(SegPlan a)
{
    __shared__ uint64_t s_warp[8];
    const uint32_t M = min(*a.num_nodes, a.node_cap);
    seg_clear(a, blockIdx.x * 256 + threadIdx.x, gridDim.x * 256, M);
    if (!a.owner) return;
    const uint32_t per = seg_nodes_per(M), lo = min((uint64_t)M, (uint64_t)blockIdx.x * per), hi = min(M, lo + per);
    uint64_t sum = 0, total;
#pragma unroll 8
    for (uint32_t i = lo + threadIdx.x; i < hi; i += 256) {
        const uint32_t v = a.nodes[i].n_own;
        a.nown[i] = v;
        a.inside[i] = 0;
        sum += v;
    }
    block_exclusive_scan<256, uint64_t>(sum, s_warp, total);
    if (threadIdx.x == 0) a.part[blockIdx.x] = total;
}

// second half: the first points of the nodes of segment q
FP_DEV void seg_first(const SegPlan& a, uint32_t q, uint32_t M, uint64_t* smem /* 8 */)
{
    const uint32_t per = seg_nodes_per(M), lo = min((uint64_t)M, (uint64_t)q * per), hi = min(M, lo + per);
    if (lo >= hi) return;   // (the same for the block)
    uint64_t before = 0, run;
    for (uint32_t i = threadIdx.x; i < q; i += 256) before += a.part[i];
    block_exclusive_scan<256, uint64_t>(before, smem, run);
    for (uint32_t i0 = lo; i0 < hi; i0 += 1024) {
        const uint32_t i = i0 + 4 * threadIdx.x;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (i < hi) v = *reinterpret_cast<const uint4*>(a.nown + i);   // (hi is rounded up within the array)
        const uint32_t w[4] = {v.x, i + 1 < hi ? v.y : 0u, i + 2 < hi ? v.z : 0u, i + 3 < hi ? v.w : 0u};
        uint64_t total;
        uint64_t ex = run + block_exclusive_scan<256, uint64_t>((uint64_t)w[0] + w[1] + w[2] + w[3], smem, total);
        run += total;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i + u < hi) {
                a.first[i + u] = ex;
                a.nodes[i + u].first = ex;
            }
            ex += w[u];
        }
    }
}

// chunk c's node and digits; false: it does not fit the scatter
FP_DEV bool seg_digits(const SegPlan& a, uint64_t c, uint32_t M, uint32_t& id, uint32_t& nb)
{
    const fp_chunk ch = a.chunks[c];
    id = find_node(a.nodes, M, ch.key, ch.level);
    if (id == kNone) return false;   // not in the table
    const uint32_t nd = a.nodes[id].n_desc;
    const uint64_t b = (uint64_t)nd + (a.owner ? 2 : 1);
    nb = (uint32_t)b;
    return (uint64_t)id + nd < M && b <= (1u << kSegMaxBits);
}

FP_DEV int seg_variant(uint32_t nb) { return nb <= (1u << kSegSmallBits) ? 0 : 1; }

// step B for the chunk of this lane (c < K): its node, digits and tiles; all 32
// lanes of the warp take part.  Callers spread the chunks over the warps first (a
// few large chunks: one each).
FP_DEV void seg_chunk(const SegPlan& a, uint64_t c, uint64_t K, uint32_t M)
{
    const int lane = threadIdx.x & 31;
    uint32_t id = 0, ntl = 0, at = 0, nb = 1;
    if (c < K) {
        const uint64_t beg = a.offsets[c], end = a.offsets[c + 1], cn = end - beg;
        bool ok = end <= a.n && end >= beg;   // else: offsets not a partition of [0, n)
        if (ok && cn) {
            ok = seg_digits(a, c, M, id, nb);
            if (ok) {
                ntl = (uint32_t)((cn + kSortTile - 1) / kSortTile);
                at = atomicAdd(&a.cnt[seg_variant(nb)], ntl);
                if ((uint64_t)at + ntl > a.tiles_max) {
                    raise(a.err, FP_ERR_CAPACITY, 12);
                    ok = false;
                }
            }
        }
        if (!ok) {   // the whole-array path runs
            atomicOr(&a.cnt[2], 1u);
            id = 0; nb = 1; ntl = 0;
        }
        a.seg_lo[c] = id;
        a.seg_nb[c] = nb;
    }
    // the lists of every lane's chunk, by the whole warp
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, ntl != 0); todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        const uint32_t nt = __shfl_sync(0xFFFFFFFFu, ntl, l), t0 = __shfl_sync(0xFFFFFFFFu, at, l);
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, nb, l), x0 = __shfl_sync(0xFFFFFFFFu, id, l);
        const uint32_t cc = __shfl_sync(0xFFFFFFFFu, (uint32_t)c, l);
        SegTile* tl = a.tiles[seg_variant(b)];
        for (uint32_t i = lane; i < nt; i += 32) tl[t0 + i] = SegTile{cc, i};
        if (a.owner)
            for (uint32_t x = lane; x < b - 1; x += 32) a.inside[x0 + x] = 1;   // the chunk's node and n_desc below it
    }
}

// step B: the look-back words of rows r0 + lane (lane < per) cleared, by the whole
// warp.  A row is written and read back where it holds the start of a tile that is
// not its chunk's last: of the last chunk that starts in or before the row.
FP_DEV void seg_rows(const SegPlan& a, uint64_t r0, uint32_t per, uint64_t rows, uint64_t K, uint32_t M)
{
    const int lane = threadIdx.x & 31;
    const uint64_t r = r0 + lane;
    uint32_t nb = 0;
    if (lane < (int)per && r < rows) {
        const uint64_t last = (r + 1) * kSortTile - 1;
        uint64_t x = 0, y = K;   // chunks that start at or before `last`
        while (x < y) {
            const uint64_t m = (x + y) >> 1;
            if (a.offsets[m] <= last) x = m + 1;
            else y = m;
        }
        if (x) {
            const uint64_t beg = a.offsets[x - 1], base = beg + (last - beg) / kSortTile * kSortTile;
            uint32_t id;
            if (base + kSortTile < a.offsets[x] && !seg_digits(a, x - 1, M, id, nb)) nb = 0;
        }
    }
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, nb != 0); todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, nb, l);
        const int v = seg_variant(b);
        uint32_t* row = a.status[v] + ((r0 + l) << (v ? kSegMaxBits : kSegSmallBits));
        for (uint32_t d = lane; d < b; d += 32) row[d] = 0;
    }
}

// The chunks go over the warps from the first one, the rows from the last.  (The rows
// of a chunk cleared by the chunk's warp: subsample of 10^8 points in one chunk, 133 MB
// of look-back words, 8.5 instead of 2.9 ms.)
__global__ void __launch_bounds__(256) k_seg_chunks(SegPlan a)
{
    __shared__ uint64_t s_warp[8];
    const uint64_t K = min((uint64_t)*a.num_chunks, a.kmax);
    const uint32_t M = min(*a.num_nodes, a.node_cap);
    if (blockIdx.x == 0 && threadIdx.x == 0 && (*a.num_chunks > a.kmax || a.offsets[K] != a.n)) atomicOr(&a.cnt[2], 1u);
    if (blockIdx.x == 0 && a.owner) {   // more owned points than there are: step C counts them in 32 bits
        uint64_t sum = 0, total;
        for (uint32_t q = threadIdx.x; q < kSegNodes; q += 256) sum += a.part[q];
        block_exclusive_scan<256, uint64_t>(sum, s_warp, total);
        if (threadIdx.x == 0 && total > a.n) {
            raise(a.err, FP_ERR_CAPACITY, 15);
            atomicOr(&a.cnt[2], 1u);
        }
    }
    // lane l of warp w: chunks w + l * nwarps, + 32 * nwarps, ...
    const uint64_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint64_t c0 = warp; c0 < K; c0 += 32 * nwarps) seg_chunk(a, c0 + (threadIdx.x & 31) * nwarps, K, M);
    const uint64_t rows = a.n / kSortTile + 1, per = min((uint64_t)32, (rows + nwarps - 1) / nwarps);
    for (uint64_t r0 = (nwarps - 1 - warp) * per; r0 < rows; r0 += nwarps * per) seg_rows(a, r0, (uint32_t)per, rows, K, M);
    if (a.owner)   // (from the blocks in the middle on)
        for (uint32_t q = (blockIdx.x + gridDim.x / 2) % gridDim.x; q < kSegNodes; q += gridDim.x) seg_first(a, q, M, s_warp);
}

__global__ void __launch_bounds__(kClNT, 1) k_seg_plan(SegPlan a)
{
    __shared__ ClScanSmem s_scan;
    const uint32_t t = cl_rank() * kClNT + threadIdx.x;
    const uint32_t M = min(*a.num_nodes, a.node_cap);
    if (!a.step_c) {
        seg_clear(a, t, kClThreads, M);
#pragma unroll 8
        for (uint32_t i = t; i < M; i += kClThreads) a.nown[i] = a.nodes[i].n_own;
        cl_sync();
        cl_scan(M, a.part, s_scan, [&](uint32_t i) -> uint64_t { return a.nown[i]; },
                [&](uint32_t i, uint64_t ex) {
                    a.first[i] = ex;
                    a.nodes[i].first = ex;
                });
        return;
    }
    if (a.cnt[2]) {   // the whole-array path runs, without ranks
        if (t == 0) *a.nrank = 0;
        return;
    }
    const uint64_t all = cl_scan(
        M, a.part, s_scan,
        [&](uint32_t i) -> uint64_t { return a.inside[i] ? 0ull : (1ull << 32) | a.nown[i]; },
        [&](uint32_t i, uint64_t ex) {
            a.soff[i] = (uint32_t)ex;
            a.rank[i] = (uint32_t)(ex >> 32);
            if (!a.inside[i]) a.list[ex >> 32] = i;
        });
    if (t == 0) *a.nrank = (uint32_t)(all >> 32);
}

SegScratch take_seg_scratch(const Workspace& ws, uint64_t n, uint64_t kmax, uint64_t node_cap)
{
    SegScratch s;
    s.kmax = kmax ? kmax : 1;
    s.rows = n / kSortTile + 1;
    s.tiles_max = n / kSortTile + s.kmax + 1;
    s.node_cap = node_cap ? node_cap : 1;
    s.lo = ws.take<uint32_t>(s.kmax);
    s.nb = ws.take<uint32_t>(s.kmax);
    s.tiles[0] = ws.take<SegTile>(s.tiles_max);
    s.tiles[1] = ws.take<SegTile>(s.tiles_max);
    s.status[0] = ws.take<uint32_t>(s.rows << kSegSmallBits);
    s.status[1] = ws.take<uint32_t>(s.rows << kSegMaxBits);
    s.cnt = ws.take<uint32_t>(8);
    s.inside = ws.take<uint8_t>(s.node_cap);
    s.part = ws.take<uint64_t>(std::max<int>(kClCtas, kSegNodes));
    return s;
}

template <bool CPT, int MAXB>
static cudaError_t seg_launch(SegArgs a, const SegScratch& sc, int v, int num_sms, cudaStream_t st)
{
    using SM = SegSmem<CPT, MAXB>;
    auto kern = k_seg_pass<CPT, MAXB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::total);
    if (e) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSortNT, SM::total))) return e;
    if (per_sm < 1) per_sm = 1;
    a.tiles = sc.tiles[v];
    a.d_ntiles = sc.cnt + v;
    a.ntiles_max = sc.tiles_max;
    a.status = sc.status[v];
    a.counter = sc.cnt + 3 + v;
    const int grid = (int)std::min<uint64_t>(sc.tiles_max, (uint64_t)num_sms * per_sm);
    kern<<<grid, kSortNT, SM::total, st>>>(a);
    return cudaGetLastError();
}

// ---- the distribution into up to 4096 chunks, in four launches and without any
// wait between blocks (the sweep with per-warp histograms for up to 512 chunks,
// the one that sorts each tile for 513 .. 4096; chosen on the device):
//   k_dist_table: per node of level L = min(g, 5), its chunk when every
//     occupied cell of the node lies in that one chunk (else none) -- a 64 KB
//     table that spares most points the gather of the cell -> chunk table;
//   k_dist_count: one block per group of consecutive tiles writes every point's
//     chunk (from its cell, given or computed), and per tile the points of each
//     chunk in the group's earlier tiles, and per group its totals;
//   k_dist_colscan: per chunk, the exclusive prefix of the group totals plus the
//     chunk's offset -- each group's output start in every chunk;
//   k_dist_sweep: two CTAs of 512 threads per SM; tiles taken in order from a
//     counter.  A tile stages only (tile position, chunk) per output slot, and
//     its write phase reads every point from the tile's copy.  A tile's run of
//     chunk d starts at its group's start in d plus the points of d in the
//     group's earlier tiles.
constexpr int kDistNT = 512;                     // two CTAs an SM
constexpr int kDistIPT = kSortTile / kDistNT;
constexpr int kDistWarps = kDistNT / 32;
constexpr int kDistBits = 9;
constexpr int kDistDig = 1 << kDistBits;
constexpr int kDistWideBits = 12;               // the wide sweep: 513 .. 4096 chunks
constexpr int kDistWideDig = 1 << kDistWideBits;
constexpr int kDistGroup = 64;                  // most tiles per block of k_dist_count
constexpr int kDistSpread = 608;                // small clouds: about this many blocks (4 per SM) instead
constexpr int kDistCountNT = 512;               // thread d of k_dist_count owns chunks d, d + 512, ...
constexpr int kDistCountIPT = kSortTile / kDistCountNT;
constexpr int kDistTabLevel = 5;                // level of the node -> chunk table
constexpr uint16_t kDistSplit = 0xFFFFu;        // the node's points lie in several chunks

struct DistSweepArgs {
    const int4* pts;
    const uint32_t* cells;      // nullable: level-g cell of every point (else computed from the point)
    const fp_cube* cube;
    const uint32_t* lut;        // cell -> chunk (kNone: empty cell)
    const uint64_t* offsets;    // chunk c = output positions [offsets[c], offsets[c + 1])
    int4* out;
    uint32_t* perm;             // nullable
    uint16_t* tab;              // [8^tl]: chunk of a level-tl node, or kDistSplit
    uint16_t* chunk;            // chunk of every point, 16-byte aligned
    uint32_t group;             // consecutive tiles of one k_dist_count block
    uint32_t* before;           // [tile][DIG]: points of the chunk in the group's earlier tiles
    uint32_t* gstart;           // [group][DIG]: group totals, then the group's start in the chunk
    uint32_t* counter;          // the sweep's tile counter
    uint64_t ntiles;
    const uint32_t* num_chunks; // more than kDistWideDig: the radix passes run instead
    uint32_t* run_sort;         // set to 1 then, else 0
    uint32_t* hist;             // the radix passes' histogram, cleared here
    uint64_t n;
    uint32_t ncell;             // cells of the grid (bound of a cell id)
    int g, tl;                  // grid level, table level (tl <= g)
    uint32_t* err;
};

FP_DEV uint32_t dist_chunks(const DistSweepArgs& a)   // 0: not this path
{
    const uint32_t K = *a.num_chunks;
    return K <= (uint32_t)kDistWideDig ? K : 0u;
}

// one warp per level-tl node: the chunks of its occupied cells
__global__ void __launch_bounds__(256) k_dist_table(DistSweepArgs a)
{
    const uint32_t nb = dist_chunks(a);
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) {
        *a.counter = 0;
        *a.run_sort = nb ? 0u : 1u;
    }
    if (!nb)
        for (uint32_t q = t; q < (uint32_t)kSortHistWords; q += gridDim.x * blockDim.x) a.hist[q] = 0;
    const int lane = threadIdx.x & 31;
    const uint32_t k = t >> 5;
    if (!nb || k >= (1u << (3 * a.tl))) return;
    const uint32_t span = 1u << (3 * (a.g - a.tl)), lo = k * span;
    uint32_t cmin = kNone, cmax = 0;
    for (uint32_t q = lane; q < span; q += 32) {
        const uint32_t c = __ldg(a.lut + lo + q);
        if (c != kNone) { cmin = min(cmin, c); cmax = max(cmax, c); }
    }
    cmin = __reduce_min_sync(0xFFFFFFFFu, cmin);
    cmax = __reduce_max_sync(0xFFFFFFFFu, cmax);
    if (lane == 0) a.tab[k] = (cmin == cmax && cmin < (uint32_t)kDistWideDig) ? (uint16_t)cmin : kDistSplit;
}

template <int DIG, bool CELLS>
FP_DEV void dist_count(const DistSweepArgs& a, uint32_t nb, const uint16_t* dist_tab, uint32_t* h)
{
    constexpr int kOwn = DIG / kDistCountNT;   // chunks per thread
    const uint64_t ngroups = (a.ntiles + a.group - 1) / a.group;
    const uint32_t d = threadIdx.x;
    const int tsh = 3 * (a.g - a.tl);
    CubeDev cube;
    if (!CELLS) {
        cube = load_cube(a.cube);
    }
    for (uint64_t gi = blockIdx.x; gi < ngroups; gi += gridDim.x) {
        const uint64_t t0 = gi * a.group, t1 = min(a.ntiles, t0 + a.group);
        uint32_t run[kOwn];
#pragma unroll
        for (int o = 0; o < kOwn; ++o) { run[o] = 0; h[d + o * kDistCountNT] = 0; }
        // given cells: those of the next tile are loaded while the current one is counted
        uint32_t c[kDistCountIPT];
        auto load = [&](uint64_t t) {
            const uint64_t base = t * kSortTile;
            if (CELLS) {
#pragma unroll
                for (int r = 0; r < kDistCountIPT; ++r) {
                    const uint64_t i = base + (uint64_t)r * kDistCountNT + d;
                    c[r] = i < a.n ? __ldg(a.cells + i) : kNone;
                }
            } else {
                int4 p[kDistCountIPT];
#pragma unroll
                for (int r = 0; r < kDistCountIPT; ++r) {   // all loads in flight together
                    const uint64_t i = base + (uint64_t)r * kDistCountNT + d;
                    p[r] = i < a.n ? __ldg(a.pts + i) : make_int4(cube.o[0], cube.o[1], cube.o[2], 0);
                }
#pragma unroll
                for (int r = 0; r < kDistCountIPT; ++r)
                    c[r] = base + (uint64_t)r * kDistCountNT + d < a.n ? key_cell(p[r].x, p[r].y, p[r].z, cube, a.g)
                                                                      : kNone;
            }
        };
        load(t0);
        __syncthreads();   // (also: the table is in shared memory)
        for (uint64_t t = t0; t < t1; ++t) {
            uint32_t k[kDistCountIPT];
#pragma unroll
            for (int r = 0; r < kDistCountIPT; ++r) {
                k[r] = c[r];
                if (k[r] != kNone && k[r] >= a.ncell) { raise(a.err, FP_ERR_CAPACITY, 19); k[r] = 0; }
            }
            if (t + 1 < t1) load(t + 1);
#pragma unroll
            for (int r = 0; r < kDistCountIPT; ++r)   // the table, else the gather
                if (k[r] != kNone) {
                    const uint16_t v = dist_tab[k[r] >> tsh];
                    k[r] = v != kDistSplit ? (uint32_t)v : __ldg(a.lut + k[r]);
                }
            const uint64_t base = t * kSortTile;
#pragma unroll
            for (int r = 0; r < kDistCountIPT; ++r) {
                const uint64_t i = base + (uint64_t)r * kDistCountNT + d;
                if (i < a.n) {
                    if (k[r] >= nb) { raise(a.err, FP_ERR_CAPACITY, 13); k[r] = nb - 1; }   // not a chunk
                    a.chunk[i] = (uint16_t)k[r];
                    atomicAdd(&h[k[r]], 1u);
                }
            }
            __syncthreads();
#pragma unroll
            for (int o = 0; o < kOwn; ++o) {
                const uint32_t cd = d + o * kDistCountNT;
                if (cd < nb) {
                    a.before[t * DIG + cd] = run[o];
                    run[o] += h[cd];
                }
                h[cd] = 0;
            }
            __syncthreads();
        }
#pragma unroll
        for (int o = 0; o < kOwn; ++o)
            if (d + o * kDistCountNT < nb) a.gstart[gi * DIG + d + o * kDistCountNT] = run[o];
    }
}

template <bool CELLS>
__global__ void __launch_bounds__(kDistCountNT) k_dist_count(DistSweepArgs a)
{
    extern __shared__ __align__(16) uint16_t dist_tab[];   // 8^tl entries
    __shared__ uint32_t h[kDistWideDig];
    const uint32_t nb = dist_chunks(a);
    if (!nb) return;
    const uint32_t nt4 = (1u << (3 * a.tl)) / 8;   // uint4 words of the table (8^tl >= 8: tl >= 1)
    for (uint32_t q = threadIdx.x; q < nt4; q += kDistCountNT)
        reinterpret_cast<uint4*>(dist_tab)[q] = __ldg(reinterpret_cast<const uint4*>(a.tab) + q);
    if (nb <= (uint32_t)kDistDig) dist_count<kDistDig, CELLS>(a, nb, dist_tab, h);
    else dist_count<kDistWideDig, CELLS>(a, nb, dist_tab, h);
}

// one warp per chunk: exclusive prefix of the group totals, plus the chunk's offset
__global__ void __launch_bounds__(256) k_dist_colscan(DistSweepArgs a)
{
    const uint64_t ngroups = (a.ntiles + a.group - 1) / a.group;
    const uint32_t nb = dist_chunks(a);
    const uint32_t dig = nb <= (uint32_t)kDistDig ? kDistDig : kDistWideDig;
    const int lane = threadIdx.x & 31;
    const uint32_t d = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (d >= nb) return;
    uint32_t run = (uint32_t)a.offsets[d];
    for (uint64_t g0 = 0; g0 < ngroups; g0 += 32) {
        const uint64_t gi = g0 + lane;
        const uint32_t v = gi < ngroups ? a.gstart[gi * dig + d] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (gi < ngroups) a.gstart[gi * dig + d] = run + x - v;
        run += __shfl_sync(0xFFFFFFFFu, x, 31);
    }
}

// The sweeps take tiles in order from a counter.  A tile's points arrive by one bulk
// copy while its chunks, in registers, are ranked; the next tile's are on their way
// to L2.  Two CTAs of 512 threads an SM: one ranks (latency of shared memory and
// barriers) while the other writes.  (One CTA of 1024 threads with two buffers: 10^8
// LiDAR points, 3057 chunks, 1.97 ms, 1.70 now; 10^8 uniform, 512 chunks, 1.12 ms,
// 0.86 now; 10^6 points, a tile a CTA, +- 3 us.)
struct TileSmem {
    int4 raw[kSortTile];   // the tile's points, as stored
    uint64_t bar;
    uint32_t tile;         // the tile to work on
    uint32_t scan[kDistWarps];
};

struct TileFeed {
    const DistSweepArgs& a;
    TileSmem& S;
    uint32_t phase = 0, dig;
    uint32_t nx = 0;       // thread 0: the tile after this one

    FP_DEV TileFeed(const DistSweepArgs& args, TileSmem& smem, uint32_t d) : a(args), S(smem), dig(d) {}
    FP_DEV bool full(uint64_t t) const { return (t + 1) * kSortTile <= a.n; }
    FP_DEV void open()
    {
        if (threadIdx.x == 0) {
            mbar_init(&S.bar, 1);
            nx = atomicAdd(a.counter, 1u);
        }
    }
    // the next tile (ntiles or more: none left), its copy under way; all threads
    FP_DEV uint64_t next()
    {
        if (threadIdx.x == 0) {
            S.tile = nx;
            if (nx < a.ntiles && full(nx)) {
                fence_async_smem();
                mbar_expect_tx(&S.bar, kSortTile * (uint32_t)sizeof(int4));
                bulk_g2s(S.raw, a.pts + (uint64_t)nx * kSortTile, kSortTile * (uint32_t)sizeof(int4), &S.bar);
            }
        }
        __syncthreads();
        const uint64_t t = S.tile;
        if (t < a.ntiles && !full(t))
            for (uint64_t i = t * kSortTile + threadIdx.x; i < a.n; i += kDistNT) S.raw[i - t * kSortTile] = __ldg(a.pts + i);
        if (threadIdx.x == 0 && t < a.ntiles) nx = atomicAdd(a.counter, 1u);
        return t;
    }
    FP_DEV void prefetch()   // once the claim's round trip is over
    {
        if (threadIdx.x == 0 && nx < a.ntiles && full(nx)) {
            bulk_prefetch_l2(a.pts + (uint64_t)nx * kSortTile, kSortTile * (uint32_t)sizeof(int4));
            bulk_prefetch_l2(a.before + (uint64_t)nx * dig, dig * (uint32_t)sizeof(uint32_t));
            bulk_prefetch_l2(a.chunk + (uint64_t)nx * kSortTile, kSortTile * (uint32_t)sizeof(uint16_t));
        }
    }
    FP_DEV void arrived(uint64_t t)   // (a partial tile's points: a barrier later)
    {
        if (!full(t)) return;
        if (!mbar_wait(&S.bar, phase & 1u)) {
            raise(a.err, FP_ERR_TIMEOUT);
            mbar_wait(&S.bar, phase & 1u);   // the copy in flight, once more (bounded)
        }
        ++phase;
    }
};

struct DistSmem : TileSmem {
    uint32_t slot[kSortTile];               // by output slot: tile position | chunk << 16
    uint16_t whist[kDistWarps][kDistDig];   // per-warp counts, then exclusive prefixes over the warps
    uint32_t gbase[kDistDig];               // output position of slot 0 of every chunk's run
    uint32_t cnt[kDistDig];
};

FP_DEV void dist_sweep(const DistSweepArgs& a, DistSmem& S, int nb)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t n = a.n;
    TileFeed feed(a, S, kDistDig);
    feed.open();
    for (;;) {
        const uint64_t tile = feed.next();
        if (tile >= a.ntiles) break;
        // this tile's chunks, and its start in every chunk, in flight together
        const uint64_t base = tile * kSortTile;
        const int tn = (int)(n - base < (uint64_t)kSortTile ? n - base : (uint64_t)kSortTile);
        uint32_t pack[kDistIPT];
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r) {
            const int p = warp * (kDistIPT * 32) + r * 32 + lane;
            pack[r] = p < tn ? (uint32_t)__ldg(a.chunk + base + p) : 0xFFFFu;
        }
        uint32_t start = 0;
        if (threadIdx.x < (unsigned)nb)
            start = __ldg(a.gstart + (tile / a.group) * kDistDig + threadIdx.x) +
                    __ldg(a.before + tile * kDistDig + threadIdx.x);
        for (int q = threadIdx.x; q < kDistWarps * kDistDig / 8; q += kDistNT)
            reinterpret_cast<uint4*>(&S.whist[0][0])[q] = make_uint4(0, 0, 0, 0);
        __syncthreads();

        // ---- in-warp stable ranks of the chunks (checked below nb by k_dist_count)
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r) {
            uint32_t d = pack[r];
            if (d != 0xFFFFu && d >= (uint32_t)nb) d = (uint32_t)(nb - 1);
            const uint32_t peers = match_bits<kDistBits>(d, d != 0xFFFFu);
            const int leader = __ffs(peers) - 1;
            uint32_t old = 0;
            if (lane == leader && d != 0xFFFFu) {
                old = S.whist[warp][d];
                S.whist[warp][d] = (uint16_t)(old + __popc(peers));
            }
            old = __shfl_sync(0xFFFFFFFFu, old, leader);
            pack[r] = d | ((old + __popc(peers & lanemask_lt())) << 16);
            __syncwarp();
        }
        feed.prefetch();
        __syncthreads();
        // ---- per-chunk totals and per-warp exclusive prefixes; first slot of every chunk's run, and the output
        // position of its slot 0
        uint32_t c = 0;
        if (threadIdx.x < (unsigned)nb) {
#pragma unroll
            for (int w = 0; w < kDistWarps; ++w) {
                const uint32_t v = S.whist[w][threadIdx.x];
                S.whist[w][threadIdx.x] = (uint16_t)c;
                c += v;
            }
        }
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<kDistNT, uint32_t>(c, S.scan, tot);
        if (threadIdx.x < (unsigned)nb) {
            S.gbase[threadIdx.x] = start - ex;
            S.cnt[threadIdx.x] = ex;
        }
        __syncthreads();
        // ---- staging entries
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r) {
            const int p = warp * (kDistIPT * 32) + r * 32 + lane;
            if (p < tn) {
                const uint32_t d = pack[r] & 0xFFFFu;
                S.slot[S.cnt[d] + S.whist[warp][d] + (pack[r] >> 16)] = (uint32_t)p | (d << 16);
            }
        }
        feed.arrived(tile);
        __syncthreads();
        // ---- coalesced writes of every chunk's run
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r) {
            const int q = r * kDistNT + threadIdx.x;
            if (q >= tn) continue;
            const uint32_t v = S.slot[q];
            const uint32_t p = v & 0xFFFFu;
            const uint64_t o = (uint32_t)(S.gbase[v >> 16] + (uint32_t)q);   // positions are below 2^30
            if (o >= n) { raise(a.err, FP_ERR_CAPACITY, 15); continue; }   // offsets not those of these points
            a.out[o] = S.raw[p];
            if (a.perm) a.perm[o] = (uint32_t)(base + p);
        }
        __syncthreads();
    }
}

// The wide sweep: 513 .. 4096 chunks, 12-bit chunk ids.  Per-warp histograms of
// 4096 chunks would not fit beside the tile, so a tile ranks its
// points by a stable two-pass sort of (chunk, position) in shared memory (6-bit
// digits, ballot-matched per warp); every chunk present takes its output start
// once (its group's start plus the points of the chunk in the group's earlier
// tiles) and each point the start plus its place in the chunk's run.
constexpr int kWideRadix = 6;
constexpr int kWideBins = 1 << kWideRadix;

struct WideSmem : TileSmem {
    uint32_t s0[kSortTile];                  // chunk << 12 | position, after the first pass; then, by chunk
                                             // present, the output position of its first point
    uint32_t s1[kSortTile];                  // the same, sorted by chunk (then position)
    uint16_t whist[kDistWarps][kWideBins];   // per-warp digit counts, then their prefixes
    uint32_t off[kWideBins];                 // first slot of every digit
    uint16_t rstart[kDistWideDig];           // first slot of every chunk present
};
static_assert(kDistWideDig <= kSortTile, "a start per chunk fits s0");

// one stable pass of the tile's (chunk << 12 | position) words by 6 chunk bits at `shift`;
// pass 0 builds the words from the chunks `chk`, the other reads `src`
FP_DEV void wide_pass(WideSmem& S, const uint16_t* chk, const uint32_t* src, uint32_t* dst, int tn, int shift)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < kDistWarps * kWideBins / 2; q += kDistNT)
        reinterpret_cast<uint32_t*>(&S.whist[0][0])[q] = 0u;
    uint32_t v[kDistIPT], pack[kDistIPT];
#pragma unroll
    for (int r = 0; r < kDistIPT; ++r) {   // all loads in flight together
        const int p = warp * (kDistIPT * 32) + r * 32 + lane;
        v[r] = 0;
        if (p < tn) v[r] = chk ? ((uint32_t)__ldg(chk + p) << 12) | (uint32_t)p : src[p];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kDistIPT; ++r) {
        const bool valid = warp * (kDistIPT * 32) + r * 32 + lane < tn;
        const uint32_t d = valid ? (v[r] >> (12 + shift)) & (kWideBins - 1) : 0u;
        const uint32_t peers = match_bits<kWideRadix>(d, valid);
        const int leader = __ffs(peers) - 1;
        uint32_t old = 0;
        if (lane == leader && valid) {
            old = S.whist[warp][d];
            S.whist[warp][d] = (uint16_t)(old + __popc(peers));
        }
        old = __shfl_sync(0xFFFFFFFFu, old, leader < 0 ? 0 : leader);
        pack[r] = valid ? (d | ((old + __popc(peers & lanemask_lt())) << 16)) : 0xFFFFFFFFu;
        __syncwarp();
    }
    __syncthreads();
    uint32_t tot_d = 0;
    if (threadIdx.x < kWideBins) {   // prefix over the warps of every digit
        for (int w = 0; w < kDistWarps; ++w) {
            const uint32_t x = S.whist[w][threadIdx.x];
            S.whist[w][threadIdx.x] = (uint16_t)tot_d;
            tot_d += x;
        }
    }
    uint32_t tot;
    const uint32_t ex = block_exclusive_scan<kDistNT, uint32_t>(threadIdx.x < kWideBins ? tot_d : 0u, S.scan, tot);
    if (threadIdx.x < kWideBins) S.off[threadIdx.x] = ex;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kDistIPT; ++r) {
        if (pack[r] == 0xFFFFFFFFu) continue;
        const uint32_t d = pack[r] & 0xFFFFu;
        dst[S.off[d] + S.whist[warp][d] + (pack[r] >> 16)] = v[r];
    }
    __syncthreads();
}

FP_DEV void dist_sweep_wide(const DistSweepArgs& a, WideSmem& S, uint32_t nb)
{
    const uint64_t n = a.n;
    uint32_t* const startv = S.s0;
    TileFeed feed(a, S, kDistWideDig);
    feed.open();
    for (;;) {
        const uint64_t tile = feed.next();
        if (tile >= a.ntiles) break;
        const uint64_t base = tile * kSortTile;
        const int tn = (int)(n - base < (uint64_t)kSortTile ? n - base : (uint64_t)kSortTile);
        wide_pass(S, a.chunk + base, nullptr, S.s0, tn, 0);
        feed.prefetch();
        wide_pass(S, nullptr, S.s0, S.s1, tn, kWideRadix);
        // ---- every chunk present: its first slot and its output start (all loads in flight together)
        const uint32_t* gs = a.gstart + (tile / a.group) * kDistWideDig;
        const uint32_t* bf = a.before + tile * kDistWideDig;
        uint32_t at[kDistIPT], ch[kDistIPT];
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r) {
            const int q = r * kDistNT + threadIdx.x;
            ch[r] = kNone;
            at[r] = 0;
            if (q >= tn) continue;
            const uint32_t c = S.s1[q] >> 12;
            if (q != 0 && (S.s1[q - 1] >> 12) == c) continue;
            if (c >= nb) { raise(a.err, FP_ERR_CAPACITY, 13); continue; }   // not a chunk
            ch[r] = c;
            at[r] = __ldg(gs + c) + __ldg(bf + c);
        }
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r)
            if (ch[r] != kNone) {
                S.rstart[ch[r]] = (uint16_t)(r * kDistNT + threadIdx.x);
                startv[ch[r]] = at[r];
            }
        feed.arrived(tile);
        __syncthreads();
        // ---- writes: every chunk's run in position order
#pragma unroll
        for (int r = 0; r < kDistIPT; ++r) {
            const int q = r * kDistNT + threadIdx.x;
            if (q >= tn) continue;
            const uint32_t v = S.s1[q];
            const uint32_t c = v >> 12, p = v & 0xFFFu;
            if (c >= nb) continue;
            const uint64_t o = (uint64_t)startv[c] + (uint64_t)(q - S.rstart[c]);
            if (o >= n) { raise(a.err, FP_ERR_CAPACITY, 15); continue; }   // offsets not those of these points
            a.out[o] = S.raw[p];
            if (a.perm) a.perm[o] = (uint32_t)(base + p);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kDistNT, 2) k_dist_sweep(DistSweepArgs a)
{
    extern __shared__ __align__(128) unsigned char dist_smem[];
    const uint32_t nb = dist_chunks(a);
    if (!nb) return;
    if (nb <= (uint32_t)kDistDig) dist_sweep(a, *reinterpret_cast<DistSmem*>(dist_smem), (int)nb);
    else dist_sweep_wide(a, *reinterpret_cast<WideSmem*>(dist_smem), nb);
}

struct DistScratch {
    uint32_t *counter, *before, *gstart;
    uint16_t* tab;
    uint64_t ntiles, group;
};

static DistScratch dist_carve(const Workspace& ws, uint64_t n)
{
    DistScratch d;
    d.ntiles = (n + kSortTile - 1) / kSortTile;
    const uint64_t T = d.ntiles ? d.ntiles : 1;
    d.group = std::max<uint64_t>(1, std::min<uint64_t>(kDistGroup, T / kDistSpread));
    d.counter = ws.take<uint32_t>(1);
    d.before = ws.take<uint32_t>(T << kDistWideBits);
    d.gstart = ws.take<uint32_t>(((T + d.group - 1) / d.group) << kDistWideBits);
    d.tab = ws.take<uint16_t>(1u << (3 * kDistTabLevel));
    return d;
}

size_t dist_wide_bytes(uint64_t n)
{
    Workspace dry;
    dist_carve(dry, n);
    return dry.used;
}

// Small clouds: the whole distribution in one launch of one cluster, any number of
// chunks: every point's chunk, stable sort by it, points and indices moved once.
// Bound by the latency of its phases; 20,000 points: 43 -> 21 us, nine launches
// before (the sweep's four kernels on 5 blocks, and the radix passes not taken).
struct DistClusterArgs {
    const int4* pts;
    const uint32_t* cells;      // nullable
    const fp_cube* cube;
    const uint32_t* lut;
    const uint64_t* offsets;
    const uint32_t* num_chunks;
    int4* out;
    uint32_t* perm;             // nullable
    uint32_t *key[2], *val[2];  // n each
    uint32_t* hist;             // [kClCtas * 256]
    uint32_t n, ncell;
    int g;
    uint32_t* err;
};

__global__ void __launch_bounds__(kClNT, 1) k_dist_cluster(DistClusterArgs a)
{
    __shared__ ClSortSmem s_sort;
    const uint32_t t = cl_rank() * kClNT + threadIdx.x;
    const uint32_t K = *a.num_chunks;
    const CubeDev cube = load_cube(a.cube);
    for (uint32_t i = t; i < a.n; i += kClThreads) {
        uint32_t m;
        if (a.cells) {
            m = __ldg(a.cells + i);
        } else {
            const int4 p = __ldg(a.pts + i);
            m = key_cell(p.x, p.y, p.z, cube, a.g);
        }
        if (m >= a.ncell) { raise(a.err, FP_ERR_CAPACITY, 19); m = 0; }   // not a cell of the grid
        uint32_t c = __ldg(a.lut + m);
        if (c >= K) { raise(a.err, FP_ERR_CAPACITY, 13); c = K ? K - 1 : 0; }   // not a chunk
        a.key[0][i] = c;
        a.val[0][i] = i;
    }
    cl_sync();
    int cur = 0;
    for (uint32_t sh = 0; sh < 32 && (K ? K - 1 : 0u) >> sh; sh += 8) {
        const uint32_t *kin = a.key[cur], *vin = a.val[cur];
        uint32_t *kout = a.key[cur ^ 1], *vout = a.val[cur ^ 1];
        cl_sort_pass(
            a.n, s_sort, a.hist, [&](uint32_t i) -> uint32_t { return (kin[i] >> sh) & 255u; },
            [&](uint32_t i, uint32_t at) {
                kout[at] = kin[i];
                vout[at] = vin[i];
            });
        cur ^= 1;
    }
    const uint32_t* key = a.key[cur];
    for (uint32_t q = t; q < a.n; q += kClThreads) {
        const uint32_t c = key[q], j = a.val[cur][q];
        if (c >= K) continue;   // (no chunks)
        const uint64_t start = a.offsets[c];
        uint64_t o = q;
        // starts in chunk order are the sorted places; else place q - (the chunk's first) behind the start
        if (start > q || key[start] != c || (start && key[start - 1] == c)) {
            uint32_t x = 0, y = q;
            while (x < y) {
                const uint32_t m = (x + y) >> 1;
                if (key[m] < c) x = m + 1;
                else y = m;
            }
            o = start + (q - x);
        }
        if (o >= a.n) { raise(a.err, FP_ERR_CAPACITY, 15); continue; }   // offsets not those of these points
        a.out[o] = __ldg(a.pts + j);
        if (a.perm) a.perm[o] = j;
    }
}

cudaError_t dist_cluster(const int4* pts, uint64_t n, const fp_cube* cube, int g, const uint32_t* lut,
                         const uint64_t* offsets, const uint32_t* num_chunks, int4* out, uint32_t* perm,
                         const uint32_t* cells, uint32_t* const tmp[4], uint32_t* hist, uint32_t* err, cudaStream_t st)
{
    DistClusterArgs a{};
    a.pts = pts; a.cells = cells; a.cube = cube; a.lut = lut; a.offsets = offsets; a.num_chunks = num_chunks;
    a.out = out; a.perm = perm;
    a.key[0] = tmp[0]; a.key[1] = tmp[1]; a.val[0] = tmp[2]; a.val[1] = tmp[3];
    a.hist = hist; a.n = (uint32_t)n; a.ncell = 1u << (3 * g); a.g = g; a.err = err;
    return cl_launch(k_dist_cluster, a, st);
}

cudaError_t dist_wide(const int4* pts, uint64_t n, const fp_cube* cube, int g, const uint32_t* lut,
                      const uint64_t* offsets, const uint32_t* num_chunks, int4* out, uint32_t* perm,
                      uint32_t* run_sort, uint32_t* hist, const Workspace& ws, cudaStream_t st, const uint32_t* cells,
                      uint16_t* chunk_tmp)
{
    const DistScratch d = dist_carve(ws, n);
    DistSweepArgs b{};
    b.pts = pts; b.cells = cells; b.cube = cube; b.lut = lut; b.offsets = offsets;
    b.out = out; b.perm = perm; b.tab = d.tab; b.chunk = chunk_tmp;
    b.group = (uint32_t)d.group; b.before = d.before; b.gstart = d.gstart;
    b.counter = d.counter; b.ntiles = d.ntiles;
    b.num_chunks = num_chunks; b.run_sort = run_sort; b.hist = hist;
    b.n = n; b.ncell = 1u << (3 * g); b.g = g; b.tl = std::min(g, kDistTabLevel); b.err = ws.err;
    const uint32_t nodes = 1u << (3 * b.tl);
    k_dist_table<<<(nodes * 32 + 255) / 256, 256, 0, st>>>(b);
    const uint64_t ngroups = (d.ntiles + d.group - 1) / d.group;
    const int tsm = (int)(nodes * sizeof(uint16_t));
    const int gc = (int)std::max<uint64_t>(1, std::min<uint64_t>(ngroups, (uint64_t)ws.num_sms * 2));
    const int grid = (int)std::max<uint64_t>(1, std::min<uint64_t>(d.ntiles, (uint64_t)ws.num_sms * 2));
    cudaError_t e;
    auto kcount = cells ? k_dist_count<true> : k_dist_count<false>;
    if ((e = cudaFuncSetAttribute(kcount, cudaFuncAttributeMaxDynamicSharedMemorySize, tsm))) return e;
    kcount<<<gc, kDistCountNT, tsm, st>>>(b);
    k_dist_colscan<<<kDistWideDig * 32 / 256, 256, 0, st>>>(b);
    const int smem = (int)std::max(sizeof(DistSmem), sizeof(WideSmem));
    if ((e = cudaFuncSetAttribute(k_dist_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return e;
    k_dist_sweep<<<grid, kDistNT, smem, st>>>(b);
    return cudaGetLastError();
}

static SegPlan seg_plan(const SegScratch& sc, const SegCall& c, const Workspace& ws)
{
    SegPlan p{};
    p.owner = c.mode == SEG_OWNER;
    p.nodes = c.nodes; p.num_nodes = c.num_nodes; p.node_cap = c.node_cap;
    p.chunks = c.chunks; p.num_chunks = c.num_chunks; p.offsets = c.offsets;
    p.kmax = sc.kmax; p.n = c.n; p.tiles_max = sc.tiles_max;
    p.seg_lo = sc.lo; p.seg_nb = sc.nb;
    for (int v = 0; v < 2; ++v) { p.tiles[v] = sc.tiles[v]; p.status[v] = sc.status[v]; }
    p.cnt = sc.cnt; p.inside = sc.inside; p.part = sc.part;
    p.nown = c.nown; p.first = c.first_out;
    p.rank = c.st_rank; p.list = c.st_list; p.nrank = c.st_nrank; p.soff = c.st_soff; p.nm = c.nm; p.nstaged = c.st_count;
    p.hist = c.hist; p.hist2 = c.hist2;
    p.err = ws.err;
    return p;
}

cudaError_t seg_node_starts(const SegScratch& sc, const SegCall& c, const Workspace& ws, cudaStream_t st)
{
    const SegPlan p = seg_plan(sc, c, ws);
    return cl_launch(k_seg_plan, p, st);
}

cudaError_t seg_scatter(const SegScratch& sc, const SegCall& c, const Workspace& ws, cudaStream_t st)
{
    cudaError_t e;
    const bool owner = c.mode == SEG_OWNER;
    SegPlan p = seg_plan(sc, c, ws);
    k_seg_nodes<<<owner ? kSegNodes : 1, 256, 0, st>>>(p);
    const int gk = (int)std::min<uint64_t>(std::max<uint64_t>((sc.kmax + 255) / 256, (sc.rows + 7) / 8),
                                           (uint64_t)ws.num_sms * 8);   // (a thread a chunk, a warp a row)
    k_seg_chunks<<<gk, 256, 0, st>>>(p);
    p.step_c = 1;
    if (owner && (e = cl_launch(k_seg_plan, p, st))) return e;
    SegArgs a{};
    a.pt_in = c.pt_in; a.pt_out = c.pt_out;
    a.val_in = c.val_in; a.val_out = c.val_out;
    a.id_in = c.id_in;
    a.offsets = c.offsets;
    a.seg_lo = sc.lo; a.seg_nb = sc.nb;
    a.first = c.first; a.first_stride = c.first_stride;
    a.stitch = owner ? 1 : 0;
    a.st_key = c.st_key; a.st_src = c.st_src; a.st_count = c.st_count; a.st_cap = c.n; a.st_shift = c.st_shift;
    a.st_rank = c.st_rank;
    a.st_nrank = c.st_nrank; a.st_code = c.st_code; a.st_inv = c.st_inv;
    a.n = c.n;
    a.d_fail = sc.cnt + 2;
    a.err = ws.err;
    const bool cpt = c.pt_in && c.pt_out;
    if (cpt) {
        if ((e = seg_launch<true, kSegSmallBits>(a, sc, 0, ws.num_sms, st))) return e;
        return seg_launch<true, kSegMaxBits>(a, sc, 1, ws.num_sms, st);
    }
    if ((e = seg_launch<false, kSegSmallBits>(a, sc, 0, ws.num_sms, st))) return e;
    return seg_launch<false, kSegMaxBits>(a, sc, 1, ws.num_sms, st);
}

}  // namespace fp
