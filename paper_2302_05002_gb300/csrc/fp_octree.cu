// fp_octree.cu -- local octrees of the chunks, the stitch above them and the
// level-of-detail selection (paper Sec. 4.4, Fig. "octree"; "shallow octree",
// Abstract).
//
// Definitions (exact-integer reading):
//   * node (L, k) exists iff it holds a point and (L == 0 or its parent holds
//     more than C points and lies above max_level); it is a leaf iff it holds
//     at most C points or L == max_level;
//   * an inner node at level L keeps, per occupied level-(L+s) cell among its
//     children's remaining points, the smallest original index (deepest first).
// Closed form used here: with lambda(p) the shallowest level at which p has the
// smallest index of its cell, p is kept by its ancestor at level
// min(max(0, lambda(p) - s), leaf level of p).  Every cell at a level >= s >= g
// lies inside one level-g cell, hence inside one chunk, so lambda is decided
// per level-g cell.  Inside a chunk the distributed order is index order.
//
// Steps:
//   1. group the distributed points by level-g cell (records (key21, j) with j
//      the position in the chunk array, i.e. index order; any order inside a
//      cell);
//   2. cells with more than kPieceMax points are cut into node-aligned pieces of at
//      most kPieceMax points, three levels a round (split tree, k_rounds); the split
//      tree also gives the nodes between level g and the pieces, and which piece
//      minimum is the minimum of which coarser node;
//   3. lambda piece by piece, by its size and depth: pairs of points, tables of the
//      smallest index per occupied cell, or a sort by key and nearest smaller
//      indices; the nodes inside pieces whose node is split further; each point gets
//      its owner level and leaf level;
//   4. node records (levels <= g from the count pyramid, deeper ones from steps
//      2-3) are sorted into preorder; ids are resolved per point;
//   5. the points are scattered stably by leaf id (leaf-grouped output) and,
//      in fp_subsample, by owner id (final output); owner segments of nodes
//      above the chunks (the stitch) are re-sorted by original index.
#include "fp_cluster.cuh"
#include "fp_grid.cuh"
#include "fp_seg.cuh"

namespace fp {

constexpr int kPieceMax = 1024;                 // largest piece handled in shared memory
constexpr int kRoundLevels = 3;                 // levels a split round groups the open nodes' records by
constexpr uint8_t kInner = 0xFF;                // hierarchy still inner at this level
constexpr uint8_t kEmpty = 0xFE;

struct NodeRec {   // a node before preorder numbering
    uint64_t key;
    uint32_t count, leaf_first;
    uint8_t level, is_leaf, pad[6];
};
static_assert(sizeof(NodeRec) == 24, "NodeRec layout");

struct Piece {
    uint32_t begin, count;   // record range in the cell-grouped arrays
    uint8_t q, hier, A;      // level, leaf level or kInner, first-min level of its minimum
    uint8_t srt;             // its records are in key order down to this level
    uint8_t buf;             // record buffer that holds them (OctCtx::recs)
    uint8_t pad[3];
};
static_assert(sizeof(Piece) == 16, "Piece layout");

struct OpenNode {
    uint64_t key;
    uint32_t begin, count;
    uint8_t q, hier, A, buf;
    uint32_t tile0;       // large nodes of a round: first tile
    uint32_t pad2, pad3;
};
static_assert(sizeof(OpenNode) == 32, "OpenNode layout");

// A record of the cell-grouped arrays in one 16-byte word, so that a record is
// moved by one load and one store: Morton key (level 21) in x | y << 32, its
// position j in the chunk array in z; w is the counting slot in the split
// rounds' copy and 0 elsewhere.
FP_DEV uint4 rec_make(uint64_t key, uint32_t j, uint32_t w)
{
    return make_uint4((uint32_t)key, (uint32_t)(key >> 32), j, w);
}
FP_DEV uint64_t rec_key(const uint4& r) { return (uint64_t)r.x | ((uint64_t)r.y << 32); }

struct OctCtx {   // device pointers of one fp_build_chunk_octree call
    const uint32_t* counts;    // points per level-g cell: the hierarchy
    const uint32_t* rcounts;   // records per level-g cell: the points at hand (a chunk group's, or all)
    uint32_t leaf_base;        // position of the first record in the whole distributed array
    const uint32_t* cstart;
    const uint32_t* cursor;    // ends of the cells as k_cell_scatter left them (cursor_slot)
    uint8_t* cell_leaf;
    uint4* recs[2];       // cell-grouped records (rec_key, rec_j), and the split rounds' second buffer
    uint64_t nrec_max;    // records
    Piece* list[4];       // the pieces by the way their lambda is found (PieceList), any order
    uint32_t* n[4];       // their numbers
    uint32_t* tab_claim;  // table pieces taken
    uint32_t piece_cap;   // of each list
    NodeRec* nrec;
    uint32_t* nnode;
    uint32_t node_cap_ws;
    uint32_t* codes;      // per record position j: code_make(LOD owner level, leaf level, level-g cell)
    int g, s, lmax, dl;
    uint64_t C;
    uint32_t* err;
};

// record i of the cell-grouped array, checked against the record count (a zero
// record beyond it: an inconsistent grouping must not turn into a stray access)
FP_DEV uint4 get_rec(const OctCtx& c, int buf, uint64_t i)
{
    if (i < c.nrec_max) return c.recs[buf][i];
    raise(c.err, FP_ERR_CAPACITY, 18);
    return make_uint4(0u, 0u, 0u, 0u);
}

FP_DEV void put_node(const OctCtx& c, uint32_t id, uint64_t key, int level, uint32_t count, uint32_t leaf_first,
                     bool leaf)
{
    if (id >= c.node_cap_ws) { raise(c.err, FP_ERR_CAPACITY, 1); return; }
    NodeRec r;
    r.key = key;
    r.count = count;
    r.leaf_first = leaf_first + c.leaf_base;
    r.level = (uint8_t)level;
    r.is_leaf = leaf ? 1 : 0;
    for (int q = 0; q < 6; ++q) r.pad[q] = 0;
    c.nrec[id] = r;
}

// levels below a piece of level q (leaf level hier, not inner) that can decide
// lambda: an owner at level hier or deeper is the leaf itself
FP_DEV int piece_depth(const OctCtx& c, int q, int hier) { return max(0, min(kKeyLevels, c.s + hier - 1) - q); }

constexpr int kSmallMax = 32;   // largest piece done by pairs of points
constexpr int kHashMaxD = 10;   // deepest piece on the tables: 3 * 10 cell bits beside a 30-bit index in 64 bits

enum PieceList : uint8_t { LIST_TAB = 0, LIST_SMALL = 1, LIST_GEN = 2, LIST_DUP = 3 };

FP_DEV PieceList piece_list(const OctCtx& c, uint32_t count, int q, uint8_t hier)
{
    if (count > (uint32_t)kPieceMax) return LIST_DUP;
    if (count <= (uint32_t)kSmallMax) return LIST_SMALL;
    if (hier == kInner) return LIST_GEN;
    return piece_depth(c, q, hier) > kHashMaxD ? LIST_GEN : LIST_TAB;
}

FP_DEV Piece make_piece(uint32_t begin, uint32_t count, int q, uint8_t hier, uint8_t A, int srt, int buf)
{
    Piece p;
    p.begin = begin;
    p.count = count;
    p.q = (uint8_t)q;
    p.hier = hier;
    p.A = A;
    p.srt = (uint8_t)srt;
    p.buf = (uint8_t)buf;
    p.pad[0] = p.pad[1] = p.pad[2] = 0;
    return p;
}

FP_DEV void put_piece(const OctCtx& c, PieceList l, uint32_t id, const Piece& p)
{
    if (id >= c.piece_cap) { raise(c.err, FP_ERR_CAPACITY, 2); return; }
    c.list[l][id] = p;
}

// ---------------------------------------------------------------- cells
// Records (key21, j) grouped by level-g cell, j = position in the chunk array:
// cell m's records fill [cstart[m], cstart[m] + rcounts[m]) in any order --
// every later step is independent of the order inside a cell (minima are
// reductions, keys are sorted where their order matters).  One pass over the
// points; the lanes of a warp that share a cell take their slots with one
// atomic on the cell's cursor, which starts at cstart[m].  The points arrive
// chunk by chunk, so the cells in use at any time are consecutive: the cursors of
// 8 cells share a sector, and the sectors sit at bit-reversed places, which
// spreads those atomics over the whole array (and every L2 slice) while the
// passes over all cells still write and read whole sectors.  A cursor that does not end at cstart[m + 1] means the
// count grid was not the grid of these points (reported by k_small_pieces).
FP_DEV uint32_t cursor_slot(uint32_t m, int g)
{
    return g == 1 ? m : ((__brev(m >> 3) >> (35 - 3 * g)) << 3) | (m & 7u);
}

__global__ void __launch_bounds__(256) k_cell_scatter(const int4* __restrict__ pts, uint64_t n, const fp_cube* cube_p,
                                                      uint32_t* cursor, uint4* __restrict__ rec, int g,
                                                      uint32_t* err)
{
    const CubeDev cube = load_cube(cube_p);
    const int lane = threadIdx.x & 31;
    const int sh = 3 * (kKeyLevels - g);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x; i0 < n; i0 += stride) {   // warp-uniform trip count
        const uint64_t i = i0 + threadIdx.x;
        uint64_t k = 0;
        uint32_t m = kNone;
        if (i < n) {
            const int4 q = __ldg(pts + i);
            k = key21(q.x, q.y, q.z, cube);
            m = (uint32_t)(k >> sh);
        }
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, m);
        const int leader = __ffs(peers) - 1;
        uint32_t at = 0;
        if (lane == leader && m != kNone) at = atomicAdd(&cursor[cursor_slot(m, g)], (uint32_t)__popc(peers));
        at = __shfl_sync(0xFFFFFFFFu, at, leader) + (uint32_t)__popc(peers & lanemask_lt());
        if (m != kNone) {
            if (at >= n) { raise(err, FP_ERR_CAPACITY, 3); continue; }   // a count grid of other points
            rec[at] = rec_make(k, (uint32_t)i, 0u);
        }
    }
}

// ------------------------------------------------- big cells: split rounds
// Cells of more than kPieceMax records are split into node-aligned pieces, three
// levels a round, all rounds in one cooperative launch (70 launches before: most
// clouds have few open nodes or none, and then the launches were all there was).
// The records of an open node are grouped by their cell three levels down, which
// puts them in key order down to that depth, and the nodes of those levels follow
// from the 512 counts and smallest indices:
//   * nodes of at most kRoundTile records by one block each, records in
//     registers, counted, ranked (any order inside a cell) and put back in place
//     with shared-memory atomics: 16 bytes read and written per record, no
//     global atomic;
//   * larger nodes in tiles of kRoundTile records by all blocks: counts and
//     minima per tile into the node's column (phase 1), columns into starts (2),
//     every tile's records to the other record buffer at slots taken once per
//     tile and cell (3), one block per node for the split (4), with a barrier of
//     the grid between the phases.
// (Copying every open node's records out, counting per record with global
// atomics, and scattering them back moved 64 bytes per record and round: 4.1 ms
// of 10^8 LiDAR points, 1.5 ms now.)
constexpr int kRoundNT = 512;
constexpr int kRoundIPT = 8;
constexpr int kRoundTile = kRoundNT * kRoundIPT;   // 4096
static_assert(kRoundNT == 1 << (3 * kRoundLevels), "one thread per cell of a round");

struct RoundCnt {          // open nodes of one round
    unsigned long long big;    // nodes of more than kRoundTile records << 32 | their tiles
    uint32_t small, pad;
};
constexpr int kMaxRounds = (kKeyLevels + kRoundLevels - 1) / kRoundLevels;

struct RoundArgs {
    OctCtx c;
    OpenNode *small[2], *big[2];   // open nodes of even and odd rounds
    RoundCnt* cnt;                 // [kMaxRounds + 1], zeroed
    uint32_t small_cap, big_cap;
    uint32_t *slots, *smin;        // [512][big_cap]: counts, then starts, then ends; smallest index
    uint32_t* bar;                 // barrier word, zeroed
};

FP_DEV void open_node(const RoundArgs& a, int round, const OpenNode& node)
{
    OpenNode o = node;
    if (o.count <= (uint32_t)kRoundTile) {
        const uint32_t id = atomicAdd(&a.cnt[round].small, 1u);
        if (id >= a.small_cap) { raise(a.c.err, FP_ERR_CAPACITY, 7); return; }
        a.small[round & 1][id] = o;
    } else {
        const uint32_t nt = (o.count + kRoundTile - 1) / kRoundTile;
        const unsigned long long at = atomicAdd(&a.cnt[round].big, (1ull << 32) | nt);
        const uint32_t id = (uint32_t)(at >> 32);
        if (id >= a.big_cap) { raise(a.c.err, FP_ERR_CAPACITY, 7); return; }
        o.tile0 = (uint32_t)at;   // (ids and first tiles grow together)
        a.big[round & 1][id] = o;
    }
}

struct RoundSmem {
    uint32_t h[kRoundNT], st[kRoundNT], mn[kRoundNT];   // per cell three levels down: count, start, smallest index
    uint32_t c2[64], m2[64], m1[8];
    uint64_t warp[kRoundNT / 32];
    uint32_t warp32[kRoundNT / 32];
    uint32_t base[3], tile[2];
};

// The nodes of the three levels below open node o (level q), thread d the cell d
// three levels down: children of more than kPieceMax records stay open down to
// the round's end, the others become pieces; inner nodes' children are nodes.
FP_DEV void split_node(const RoundArgs& a, RoundSmem& S, const OpenNode& o, int round, int buf)
{
    const OctCtx& c = a.c;
    const int d = threadIdx.x, q = o.q;
    const uint32_t begin = S.st[d];
    uint32_t cn[4], mn[4];   // by levels below o
    cn[3] = S.h[d];
    mn[3] = S.mn[d];
    cn[2] = cn[3]; mn[2] = mn[3];
#pragma unroll
    for (int x = 1; x < 8; x <<= 1) {
        cn[2] += __shfl_xor_sync(0xFFFFFFFFu, cn[2], x);
        mn[2] = min(mn[2], __shfl_xor_sync(0xFFFFFFFFu, mn[2], x));
    }
    if ((d & 7) == 0) { S.c2[d >> 3] = cn[2]; S.m2[d >> 3] = mn[2]; }
    __syncthreads();
    cn[1] = 0; mn[1] = kNone;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        cn[1] += S.c2[(d >> 6) * 8 + x];
        mn[1] = min(mn[1], S.m2[(d >> 6) * 8 + x]);
    }
    if ((d & 63) == 0) S.m1[d >> 6] = mn[1];
    __syncthreads();
    mn[0] = kNone;
#pragma unroll
    for (int x = 0; x < 8; ++x) mn[0] = min(mn[0], S.m1[x]);

    // per level: is this thread the child's first cell, the child's hierarchy and first-min level
    bool node[4] = {false, false, false, false}, piece[4] = {false, false, false, false};
    uint8_t hier[4], A[4];
    hier[0] = o.hier;
    A[0] = o.A;
    bool open = true;
#pragma unroll
    for (int t = 1; t <= 3; ++t) {
        const int lev = q + t;
        hier[t] = hier[t - 1] != kInner ? hier[t - 1] : ((cn[t] <= c.C || lev == c.lmax) ? (uint8_t)lev : kInner);
        // the child's minimum is the parent's minimum: it keeps the parent's first-min level
        A[t] = mn[t] == mn[t - 1] ? A[t - 1] : (uint8_t)lev;
        const bool here = open && cn[t] && (d & ((1 << (3 * (3 - t))) - 1)) == 0;
        open = open && cn[t] > (uint32_t)kPieceMax && lev < c.dl;
        if (here) {
            node[t] = hier[t - 1] == kInner;
            if (!open) {
                piece[t] = true;
            } else if (t == 3) {
                OpenNode ch;
                ch.key = (o.key << 9) | (uint64_t)d;
                ch.begin = begin;
                ch.count = cn[3];
                ch.q = (uint8_t)lev;
                ch.hier = hier[3];
                ch.A = A[3];
                ch.buf = (uint8_t)buf;
                ch.tile0 = ch.pad2 = ch.pad3 = 0;
                open_node(a, round + 1, ch);
            }
        }
    }
    // appends of table pieces, small pieces and nodes: one scan, one atomic each
    const int srt = min(q + kRoundLevels, kKeyLevels);
    uint64_t want = 0;
    PieceList list[4];
#pragma unroll
    for (int t = 1; t <= 3; ++t) {
        list[t] = piece_list(c, cn[t], q + t, hier[t]);
        if (piece[t] && list[t] == LIST_TAB) want += 1;
        if (piece[t] && list[t] == LIST_SMALL) want += 1ull << 21;
        if (node[t]) want += 1ull << 42;
    }
    uint64_t total;
    const uint64_t ex = block_exclusive_scan<kRoundNT, uint64_t>(want, S.warp, total);
    constexpr uint32_t kF = (1u << 21) - 1;
    if (d < 3) {
        const uint32_t n = (uint32_t)(total >> (21 * d)) & kF;
        uint32_t* ctr = d == 0 ? c.n[LIST_TAB] : (d == 1 ? c.n[LIST_SMALL] : c.nnode);
        S.base[d] = n ? atomicAdd(ctr, n) : 0u;
    }
    __syncthreads();
    uint32_t ti = S.base[0] + ((uint32_t)ex & kF), si = S.base[1] + ((uint32_t)(ex >> 21) & kF),
             ni = S.base[2] + (uint32_t)(ex >> 42);
#pragma unroll
    for (int t = 1; t <= 3; ++t) {
        if (node[t])
            put_node(c, ni++, (o.key << (3 * t)) | (uint64_t)(d >> (3 * (3 - t))), q + t, cn[t], begin, hier[t] != kInner);
        if (piece[t]) {
            const Piece p = make_piece(begin, cn[t], q + t, hier[t], A[t], srt, buf);
            if (list[t] == LIST_TAB) put_piece(c, LIST_TAB, ti++, p);
            else if (list[t] == LIST_SMALL) put_piece(c, LIST_SMALL, si++, p);
            else put_piece(c, list[t], atomicAdd(c.n[list[t]], 1u), p);
        }
    }
    __syncthreads();   // the arrays are free for the next node
}

__global__ void __launch_bounds__(kRoundNT, 2) k_rounds(RoundArgs a)
{
    __shared__ RoundSmem S;
    const OctCtx& c = a.c;
    const int tid = threadIdx.x, lane = tid & 31;
    uint32_t nbar = 0;
    for (int round = 0, q = c.g; q < c.dl; ++round, q += kRoundLevels) {
        const uint32_t ns = min(ld_volatile(&a.cnt[round].small), a.small_cap);
        const uint64_t bp = ld_volatile64(reinterpret_cast<const uint64_t*>(&a.cnt[round].big));
        const uint32_t nb = min((uint32_t)(bp >> 32), a.big_cap), ntile = nb ? (uint32_t)bp : 0u;
        if (ns == 0 && nb == 0) return;   // (the same in every block)
        const OpenNode* small = a.small[round & 1];
        const OpenNode* big = a.big[round & 1];
        // the record's cell three levels below q (beyond the key's last level: zeros)
        const int sh = 3 * (kKeyLevels - q - kRoundLevels);
        auto digit = [&](const uint4& r) {
            const uint64_t k = rec_key(r);
            return (uint32_t)(sh >= 0 ? k >> sh : k << -sh) & (kRoundNT - 1);
        };
        if (nb) {
            for (uint64_t x = (uint64_t)blockIdx.x * kRoundNT + tid; x < (uint64_t)nb * kRoundNT;
                 x += (uint64_t)gridDim.x * kRoundNT) {
                const uint64_t slot = (x / nb) * a.big_cap + x % nb;
                a.slots[slot] = 0;
                a.smin[slot] = kNone;
            }
            if (!grid_barrier(a.bar, ++nbar, c.err)) return;
        }
        // loads a run of at most kRoundTile records, counts them per cell; returns each one's cell | rank << 16
        uint4 rec[kRoundIPT];
        uint32_t pk[kRoundIPT];
        auto count_run = [&](const uint4* src, uint32_t n, bool minima) {
            S.h[tid] = 0;
            S.mn[tid] = kNone;
            __syncthreads();
#pragma unroll
            for (int r = 0; r < kRoundIPT; ++r)
                if (r * kRoundNT + tid < n) rec[r] = src[r * kRoundNT + tid];
#pragma unroll
            for (int r = 0; r < kRoundIPT; ++r)
                if (r * kRoundNT + tid < n) {
                    const uint32_t d = digit(rec[r]);
                    pk[r] = d | (atomicAdd(&S.h[d], 1u) << 16);
                    if (minima && S.mn[d] > rec[r].z) atomicMin(&S.mn[d], rec[r].z);
                }
            __syncthreads();
        };
        for (uint32_t i = blockIdx.x; i < ns; i += gridDim.x) {
            const OpenNode o = small[i];
            if ((uint64_t)o.begin + o.count > c.nrec_max) { raise(c.err, FP_ERR_CAPACITY, 6); continue; }
            uint4* buf = c.recs[o.buf];
            count_run(buf + o.begin, o.count, true);
            uint32_t tot;
            const uint32_t ex = block_exclusive_scan<kRoundNT, uint32_t>(S.h[tid], S.warp32, tot);
            S.st[tid] = o.begin + ex;
            __syncthreads();
#pragma unroll
            for (int r = 0; r < kRoundIPT; ++r)
                if (r * kRoundNT + tid < o.count) buf[S.st[pk[r] & 0xFFFFu] + (pk[r] >> 16)] = rec[r];
            split_node(a, S, o, round, o.buf);
        }
        // tile t of the large nodes: its node and its first record
        auto tile_of = [&](uint32_t t) {
            if (tid == 0) {
                uint32_t x = 0, y = nb;
                while (y - x > 1) {
                    const uint32_t m = (x + y) >> 1;
                    if (big[m].tile0 <= t) x = m;
                    else y = m;
                }
                S.tile[0] = x;
                S.tile[1] = (t - big[x].tile0) * kRoundTile;
            }
            __syncthreads();
        };
        for (uint32_t t = blockIdx.x; t < ntile; t += gridDim.x) {
            tile_of(t);
            const uint32_t b = S.tile[0], off = S.tile[1];
            const OpenNode o = big[b];
            const bool ok = off < o.count && (uint64_t)o.begin + o.count <= c.nrec_max;
            if (!ok && tid == 0) raise(c.err, FP_ERR_CAPACITY, 6);
            count_run(c.recs[o.buf] + o.begin + off, ok ? min((uint32_t)kRoundTile, o.count - off) : 0u, true);
            if (S.h[tid]) {
                atomicAdd(&a.slots[(uint64_t)tid * a.big_cap + b], S.h[tid]);
                atomicMin(&a.smin[(uint64_t)tid * a.big_cap + b], S.mn[tid]);
            }
            __syncthreads();
        }
        if (nb) {
            if (!grid_barrier(a.bar, ++nbar, c.err)) return;
            // counts -> starts, one warp per node
            const uint32_t warp = (blockIdx.x * kRoundNT + tid) >> 5, nwarps = (gridDim.x * kRoundNT) >> 5;
            for (uint32_t b = warp; b < nb; b += nwarps) {
                uint32_t v[kRoundNT / 32], sum = 0;
#pragma unroll
                for (int x = 0; x < kRoundNT / 32; ++x) {
                    v[x] = a.slots[(uint64_t)(lane * (kRoundNT / 32) + x) * a.big_cap + b];
                    sum += v[x];
                }
                uint32_t inc = sum;
                for (int s = 1; s < 32; s <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, s);
                    if (lane >= s) inc += y;
                }
                uint32_t run = big[b].begin + inc - sum;
#pragma unroll
                for (int x = 0; x < kRoundNT / 32; ++x) {
                    a.slots[(uint64_t)(lane * (kRoundNT / 32) + x) * a.big_cap + b] = run;
                    run += v[x];
                }
            }
            if (!grid_barrier(a.bar, ++nbar, c.err)) return;
            for (uint32_t t = blockIdx.x; t < ntile; t += gridDim.x) {
                tile_of(t);
                const uint32_t b = S.tile[0], off = S.tile[1];
                const OpenNode o = big[b];
                const uint32_t n = off < o.count && (uint64_t)o.begin + o.count <= c.nrec_max
                                       ? min((uint32_t)kRoundTile, o.count - off) : 0u;
                count_run(c.recs[o.buf] + o.begin + off, n, false);
                S.st[tid] = S.h[tid] ? atomicAdd(&a.slots[(uint64_t)tid * a.big_cap + b], S.h[tid]) : 0u;
                __syncthreads();
                uint4* dst = c.recs[o.buf ^ 1];
#pragma unroll
                for (int r = 0; r < kRoundIPT; ++r)
                    if (r * kRoundNT + tid < n) {
                        const uint64_t at = (uint64_t)S.st[pk[r] & 0xFFFFu] + (pk[r] >> 16);
                        if (at < c.nrec_max) dst[at] = rec[r];
                        else raise(c.err, FP_ERR_CAPACITY, 6);
                    }
                __syncthreads();
            }
            if (!grid_barrier(a.bar, ++nbar, c.err)) return;
            for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {   // slots hold the cells' ends now
                const OpenNode o = big[b];
                const uint32_t end = a.slots[(uint64_t)tid * a.big_cap + b];
                S.mn[tid] = a.smin[(uint64_t)tid * a.big_cap + b];
                S.h[tid] = end;
                __syncthreads();
                const uint32_t from = tid ? S.h[tid - 1] : o.begin;
                __syncthreads();
                S.st[tid] = from;
                S.h[tid] = end - from;
                __syncthreads();
                split_node(a, S, o, round, o.buf ^ 1);
            }
        }
        if (!grid_barrier(a.bar, ++nbar, c.err)) return;
    }
}

// One block per tile of the grid (k_grid_tiles before it).  With `cells`: every
// cell's start among the records and its cursor; its leaf level when the
// hierarchy ends at or above g, kInner if the cell's node is inner, kEmpty
// without a record.  Cells with at most kPieceMax records become pieces
// (k_small_pieces finds the smallest by itself); larger ones open the split
// tree.  With `upper`: the nodes at levels <= g.  The tile's counts, starts and
// coarser sums go through shared memory, and the cells are taken 1024 at a time,
// four neighbours per thread, in one rolled loop each for the decisions and the
// appends (unrolled over a thread's 16 cells the code overran the instruction
// cache).  The decisions are selects over the counts around the four cells, read
// together, and the four starts, cursors and leaf levels are stored as one vector
// each: bound by instructions (120 a cell of its own at one cell per thread and
// round; as a chain of branches a round took 900 cycles of latency on top, and the
// few tiles that hold a small cloud's points kept the whole kernel waiting).  The
// 2^21 cells of 10^6 points: 29 -> 21 -> 15 us, of 20,000 points: 24 -> 14 us.
// Pieces for the tables, nearly all of them on large clouds, and nodes are appended
// with one atomic per tile, the pieces in cell order: those in work at one time
// then lie in one or two tiles, and their scattered codes stay in L2 (appended one
// by one as the atomics fell, k_tab_pieces took 15.5 instead of 13.0 ms for
// 5 * 10^8 uniform points, before it took its pieces in order).
constexpr int kOpenRounds = kGtPer / 4;

struct __align__(16) OpenSmem {
    uint32_t v[kGtCells], st[kGtCells + 4];   // points (hierarchy) and start of every cell; the end
    uint32_t s1[kGtCells / 8], s2[kGtCells / 64], s3[kGtCells / 512];
    uint32_t at[kOpenRounds][kGtNT / 32]; // appends before a warp's 128 cells: pieces | nodes << 16
    GridTop top;
    uint32_t warp[kGtNT / 32], base[2];
};

__global__ void __launch_bounds__(kGtNT, 4) k_cells_open(RoundArgs ra, const uint32_t* __restrict__ pyr,
                                                         const uint32_t* __restrict__ rsum, int cells, int upper,
                                                         uint32_t* __restrict__ cstart, uint32_t* __restrict__ cursor)
{
    __shared__ OpenSmem S;
    const OctCtx& c = ra.c;
    const int g = c.g, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t ncell = 1u << (3 * g), tile = blockIdx.x, base = tile * kGtCells + tid * kGtPer;
    const bool same = c.rcounts == c.counts;
    uint32_t before = 0;
    uint32_t s4;
    {
        uint32_t v[kGtPer];
        grid_load16(c.counts, base, ncell, v);
        const GridSums s = grid_sums(v, S.warp);
        s4 = s.s4;
#pragma unroll
        for (int q = 0; q < kGtPer; q += 4)
            *reinterpret_cast<uint4*>(&S.v[tid * kGtPer + q]) = make_uint4(v[q], v[q + 1], v[q + 2], v[q + 3]);
        S.s1[2 * tid] = s.s1[0];
        S.s1[2 * tid + 1] = s.s1[1];
        if ((tid & 3) == 0) S.s2[tid >> 2] = s.s2;
        if (lane == 0) S.s3[warp] = s.s3;
        for (uint32_t i = tid; i < tile; i += kGtNT) before += rsum[i];
        before = block_sum(before, S.warp);
        if (!same) grid_load16(c.rcounts, base, ncell, v);
        uint32_t mine = 0;
#pragma unroll
        for (int q = 0; q < kGtPer; ++q) mine += v[q];
        uint32_t total;
        uint32_t at = before + block_exclusive_scan<kGtNT, uint32_t>(mine, S.warp, total);
#pragma unroll
        for (int q = 0; q < kGtPer; q += 4) {
            const uint4 w = make_uint4(at, at + v[q], at + v[q] + v[q + 1], at + v[q] + v[q + 1] + v[q + 2]);
            *reinterpret_cast<uint4*>(&S.st[tid * kGtPer + q]) = w;
            at = w.w + v[q + 3];
        }
        if (tid == kGtNT - 1) S.st[kGtCells] = at;
        if (cells && tile == gridDim.x - 1 && tid == 0) cstart[ncell] = before + total;
    }
    const int up = grid_top(S.top, pyr, g, s4);   // (its barriers publish the arrays above)
    int ht = 255;                                 // leaf level at or above the tile's node
    for (int a = 0; a <= up; ++a)
        if (S.top.at(a, tile) <= c.C) ht = max(g - 4 - a, 0);   // (a grid of fewer than 4096 cells: its root)
    const uint32_t C = (uint32_t)min((unsigned long long)c.C, 0xFFFFFFFFull);
    const bool lowest = g == c.lmax;
    uint32_t topf = 0;                            // nodes at levels <= g - 4 whose first cell is the tile's first
    if (tid == 0)
        for (int a = 0; a <= up; ++a)
            if (g - 4 - a >= 0 && (tile & ((1u << (3 * a)) - 1)) == 0 && S.top.at(a, tile) &&
                (g - 4 - a == 0 || (a < up && S.top.at(a + 1, tile) > C)))
                topf |= 16u << a;
    const bool tab_g = piece_depth(c, g, (uint8_t)g) <= kHashMaxD;   // table pieces whose leaf is the cell
    // Cells i .. i + 3 of the tile (i a multiple of 4): their starts and the end, their leaf levels or kInner, the
    // ones that are table pieces, and the nodes whose first cell is one of them: bit k < 8 for level g - k at cell
    // i, bits 8 .. 10 for level g at the others.  A node exists when it holds points and is the root or its parent
    // holds more than C.
    struct Look {
        uint4 v, st;
        uint32_t end, hier, tab, f;   // hier: a byte per cell
    };
    auto look = [&](uint32_t i) {
        const uint32_t a1 = S.s1[i >> 3], a2 = S.s2[i >> 6], a3 = S.s3[i >> 9];
        Look o;
        o.v = *reinterpret_cast<const uint4*>(&S.v[i]);
        o.st = *reinterpret_cast<const uint4*>(&S.st[i]);
        o.end = S.st[i + 4];
        int h = -1;   // leaf level above the cells
        h = a1 <= C ? max(g - 1, 0) : h;
        h = a2 <= C ? max(g - 2, 0) : h;
        h = a3 <= C ? max(g - 3, 0) : h;
        h = ht != 255 ? ht : h;
        const bool tab_h = h >= 0 && piece_depth(c, g, (uint8_t)h) <= kHashMaxD;
        o.hier = o.tab = o.f = 0;
        auto cell = [&](int q, uint32_t v, uint32_t n) {
            const bool own = v <= C || lowest;   // (h < 0) the cell is a leaf
            const uint32_t hq = h >= 0 ? (uint32_t)h : (own ? (uint32_t)g : (uint32_t)kInner);
            o.hier |= (n ? hq : (uint32_t)kEmpty) << (8 * q);
            if (n > (uint32_t)kSmallMax && n <= (uint32_t)kPieceMax && (h >= 0 ? tab_h : own && tab_g)) o.tab |= 1u << q;
            if (v && a1 > C) o.f |= q ? 128u << q : 1u;
        };
        cell(0, o.v.x, o.st.y - o.st.x);
        cell(1, o.v.y, o.st.z - o.st.y);
        cell(2, o.v.z, o.st.w - o.st.z);
        cell(3, o.v.w, o.end - o.st.w);
        o.f |= (i & 7) == 0 && a1 && (g == 1 || a2 > C) ? 2u : 0u;
        o.f |= (i & 63) == 0 && g >= 2 && a2 && (g == 2 || a3 > C) ? 4u : 0u;
        o.f |= (i & 511) == 0 && g >= 3 && a3 && (g == 3 || s4 > C) ? 8u : 0u;
        o.f |= i == 0 ? topf : 0u;
        o.f = upper ? o.f : 0u;
        o.tab = cells ? o.tab : 0u;
        return o;
    };
    auto start_of = [](const Look& o, int q) { return q == 0 ? o.st.x : (q == 1 ? o.st.y : (q == 2 ? o.st.z : o.st.w)); };
    auto end_of = [](const Look& o, int q) { return q == 0 ? o.st.y : (q == 1 ? o.st.z : (q == 2 ? o.st.w : o.end)); };
    auto hier_of = [](const Look& o, int q) { return (uint8_t)(o.hier >> (8 * q)); };
    // 64 cells without a point that no node of a coarser level starts with either:
    // nothing to decide (LiDAR clouds fill a few percent of the cells)
    auto idle = [&](uint32_t i) {
        return i >= 64 && S.s2[i >> 6] == 0 && ((i & 511) >= 64 || S.s3[i >> 9] == 0);
    };
    const uint32_t in_tile = min((uint32_t)kGtCells, ncell);
    uint32_t busy = 0;   // bit r (the same for the warp): the warp's cells of round r append pieces or nodes
#pragma unroll 1
    for (int r = 0; r < kOpenRounds; ++r) {
        const uint32_t i = (r * kGtNT + tid) * 4, m = tile * kGtCells + i;
        const bool write = cells && i < in_tile;
        uint32_t sum = 0;
        if (__all_sync(0xFFFFFFFFu, idle(i))) {
            if (write) {
                const uint4 st = *reinterpret_cast<const uint4*>(&S.st[i]);
                *reinterpret_cast<uint4*>(cstart + m) = st;
                *reinterpret_cast<uint4*>(cursor + cursor_slot(m, g)) = st;
                *reinterpret_cast<uint32_t*>(c.cell_leaf + m) = kEmpty * 0x01010101u;
            }
        } else {
            const Look o = look(i);
            if (write) {
                *reinterpret_cast<uint4*>(cstart + m) = o.st;
                *reinterpret_cast<uint4*>(cursor + cursor_slot(m, g)) = o.st;
                *reinterpret_cast<uint32_t*>(c.cell_leaf + m) = o.hier;
#pragma unroll 1
                for (int q = 0; q < 4; ++q) {   // what is neither empty, small nor for the tables
                    const uint32_t at = start_of(o, q), n = end_of(o, q) - at;
                    const uint8_t h = hier_of(o, q);
                    if (n <= (uint32_t)kSmallMax || ((o.tab >> q) & 1u)) continue;
                    if (n <= (uint32_t)kPieceMax) {
                        put_piece(c, LIST_GEN, atomicAdd(c.n[LIST_GEN], 1u), make_piece(at, n, g, h, (uint8_t)g, g, 0));
                    } else {
                        OpenNode b;
                        b.key = m + q;
                        b.begin = at;
                        b.count = n;
                        b.q = (uint8_t)g;
                        b.hier = h;
                        b.A = (uint8_t)g;
                        b.buf = 0;
                        b.tile0 = b.pad2 = b.pad3 = 0;
                        open_node(ra, 0, b);
                    }
                }
            }
            sum = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(o.tab) | ((uint32_t)__popc(o.f) << 16));
            if (sum) busy |= 1u << r;
        }
        if (lane == 0) S.at[r][warp] = sum;
    }
    __syncthreads();
    {   // the 32 runs of 128 cells in order; one atomic each for the tile's pieces and nodes
        uint32_t* at = &S.at[0][0];
        const uint32_t v = tid < kOpenRounds * (kGtNT / 32) ? at[tid] : 0u;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan<kGtNT, uint32_t>(v, S.warp, total);
        if (tid < kOpenRounds * (kGtNT / 32)) at[tid] = ex;
        if (tid == 0) {
            S.base[0] = (total & 0xFFFFu) ? atomicAdd(c.n[LIST_TAB], total & 0xFFFFu) : 0u;
            S.base[1] = (total >> 16) ? atomicAdd(c.nnode, total >> 16) : 0u;
        }
        __syncthreads();
        if (total == 0) return;
    }
#pragma unroll 1
    for (; busy; busy &= busy - 1) {
        const int r = __ffs(busy) - 1;
        const uint32_t i = (r * kGtNT + tid) * 4, m = tile * kGtCells + i;
        const Look o = look(i);
        const uint32_t mine = (uint32_t)__popc(o.tab) | ((uint32_t)__popc(o.f) << 16);
        uint32_t inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        const uint32_t ex = S.at[r][warp] + inc - mine;
        uint32_t pi = S.base[0] + (ex & 0xFFFFu), ni = S.base[1] + (ex >> 16);
#pragma unroll 1
        for (uint32_t todo = o.tab; todo; todo &= todo - 1) {
            const int q = __ffs(todo) - 1;
            const uint32_t at = start_of(o, q);
            put_piece(c, LIST_TAB, pi++, make_piece(at, end_of(o, q) - at, g, hier_of(o, q), (uint8_t)g, g, 0));
        }
#pragma unroll 1
        for (uint32_t todo = o.f; todo; todo &= todo - 1) {
            const int b = __ffs(todo) - 1;
            const int k = b < 8 ? b : 0, q = b < 8 ? 0 : b - 7;   // levels above the cell, and which of the four
            const int lev = g - k;
            const uint32_t cnt =
                k == 0 ? (q == 0 ? o.v.x : (q == 1 ? o.v.y : (q == 2 ? o.v.z : o.v.w)))
                       : (k == 1 ? S.s1[i >> 3] : (k == 2 ? S.s2[i >> 6] : (k == 3 ? S.s3[i >> 9] : S.top.at(k - 4, tile))));
            put_node(c, ni++, (m + q) >> (3 * k), lev, cnt, start_of(o, q), cnt <= C || lev == c.lmax);
        }
    }
}

// ------------------------------------------------------------ pieces
// Lambda of every record, by the size and depth of its piece:
//   * at most kSmallMax points: k_small_pieces, one lane per point, cells straight
//     from the count grid (no piece is listed);
//   * pieces whose node is not inner, at most kHashMaxD levels deep: k_tab_pieces,
//     one block per piece, smallest index per occupied cell in tables (on large
//     clouds the small shallow ones by one warp each, k_warp_pieces);
//   * larger inner pieces, and deeper ones: k_general_pieces, one block per piece, sort
//     and nearest-smaller search, which also finds the nodes inside the piece;
//   * more than kPieceMax equal keys: k_general_pieces too, by a minimum.
// A piece is worked on by itself, so nothing about a record (its piece, the
// levels that decide it) is looked up per record, the lists need no order, and
// blocks wait on nothing but themselves.  (Windows of 1024 records with all of
// their pieces in one 512-thread block, and the pieces sorted into record order
// first, spent 950 instructions per point at 238 points per cell, where the
// fourth and fifth table of a window did not fit its shared memory: 26.1 ms for
// 5 * 10^8 uniform points, 5.3 ms now at about 300 instructions per point.)
constexpr int kTabNT = 128;
constexpr int kTabRun = 8;                    // pieces taken at a time
constexpr int kTabCtas = 10;                  // blocks per SM (20 KB of tables each)
constexpr int kTabDirect = 4;                 // levels in direct-mapped tables
constexpr int kTabWords = 4680;               // 8 + 64 + 512 + 4096 entries
constexpr uint64_t kHashEmpty = ~0ull;
constexpr int kHashSlots = kPieceMax + kPieceMax / 2;
constexpr int kTabBytes = sizeof(uint64_t) * (kPieceMax + kHashSlots);   // records and hash table
static_assert(kTabWords * sizeof(uint32_t) <= kTabBytes, "the direct tables overlay the hash path's arrays");

// owner level of a record with first-minimum level lambda, and its code
FP_DEV void put_lambda(const OctCtx& c, uint32_t jj, int lambda, int leafl, uint32_t cell)
{
    int K = lambda - c.s;
    K = K < 0 ? 0 : (K > leafl ? leafl : K);
    if (jj < c.nrec_max) c.codes[jj] = code_make(K, leafl, cell);
    else raise(c.err, FP_ERR_CAPACITY, 17);
}

// The points of up to 64 small pieces, two neighbouring ones per lane (cnt 0:
// none), spread over the lanes of the warp one record each: lambda is one more
// than the deepest level shared with any point of smaller index in the piece
// (every pair of the piece; its records are a few consecutive words, read
// through L1).
struct SmallPiece {
    uint32_t begin, cnt, what;   // what: record buffer | leaf level << 8 | first-min level << 16
};

FP_DEV void small_warp(const OctCtx& c, SmallPiece a, SmallPiece b)
{
    const int lane = threadIdx.x & 31;
    if ((uint64_t)a.begin + a.cnt > c.nrec_max || (uint64_t)b.begin + b.cnt > c.nrec_max) {
        raise(c.err, FP_ERR_CAPACITY, 18);
        a.cnt = b.cnt = 0;
    }
    uint32_t inc = a.cnt + b.cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, inc, 31);
    const uint32_t counts = a.cnt | (b.cnt << 16);
    for (uint32_t r0 = 0; r0 < total; r0 += 32) {
        const uint32_t r = r0 + lane;
        int o = 0;   // lanes whose pieces end at or before r
#pragma unroll
        for (int s = 16; s > 0; s >>= 1)
            if (__shfl_sync(0xFFFFFFFFu, inc, (o + s - 1) & 31) <= r) o += s;
        o &= 31;
        const uint32_t cc = __shfl_sync(0xFFFFFFFFu, counts, o);
        const uint32_t ca = cc & 0xFFFFu, cb = cc >> 16;
        const uint32_t k0 = r - (__shfl_sync(0xFFFFFFFFu, inc, o) - ca - cb);   // place in the lane's two pieces
        const bool second = k0 >= ca;
        const uint32_t ba = __shfl_sync(0xFFFFFFFFu, a.begin, o), bb = __shfl_sync(0xFFFFFFFFu, b.begin, o);
        const uint32_t wa = __shfl_sync(0xFFFFFFFFu, a.what, o), wb = __shfl_sync(0xFFFFFFFFu, b.what, o);
        if (r >= total) continue;   // (no shuffle below)
        const uint32_t w = second ? wb : wa, cn = second ? cb : ca;
        const uint4* rec = c.recs[w & 1u] + (second ? bb : ba);
        const uint4 me = rec[second ? k0 - ca : k0];
        const uint64_t k = rec_key(me);
        uint64_t near = ~0ull;   // smallest key difference to a smaller index: the deepest shared level
        for (uint32_t t = 0; t < cn; t += 4) {   // four loads in flight (the last record again beyond the end)
            uint4 other[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) other[u] = rec[min(t + u, cn - 1)];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t x = rec_key(other[u]) ^ k;
                if (other[u].z < me.z && x < near) near = x;
            }
        }
        int lambda = (int)(w >> 16);   // the piece minimum: from the split tree
        if (near != ~0ull) lambda = (near == 0 ? kKeyLevels : (__clzll((long long)near) - 1) / 3) + 1;
        put_lambda(c, me.z, lambda, (int)((w >> 8) & 255u), (uint32_t)(k >> (3 * (kKeyLevels - c.g))));
    }
}

// An inner piece of up to 32 points, one a lane: sorted by key (15 exchanges), so that
// every cell's points are neighbouring lanes; lambda by all pairs, as above; the nodes
// below the piece's level by level, those of a level appended with one atomic.  (One
// block per piece, as larger inner ones: 2 * 10^6 uniform points at capacity 1, an
// octree of 2.9 * 10^6 nodes, 12.4 instead of 1.2 ms.)
FP_DEV void inner_warp(const OctCtx& c, uint32_t begin, uint32_t cnt, int q, int A, int buf)
{
    const int lane = threadIdx.x & 31;
    if (cnt > 32u || (uint64_t)begin + cnt > c.nrec_max) {   // (the same for the warp)
        if (lane == 0) raise(c.err, FP_ERR_CAPACITY, 18);
        return;
    }
    const bool here = lane < (int)cnt;
    uint64_t k = ~0ull;   // (beyond the points: last)
    uint32_t j = kNone;
    if (here) {
        const uint4 r = c.recs[buf][begin + lane];
        k = rec_key(r);
        j = r.z;
    }
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int d = size >> 1; d > 0; d >>= 1) {
            const uint64_t ok = __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)k, d);
            const uint32_t oj = __shfl_xor_sync(0xFFFFFFFFu, j, d);
            const bool low = ((lane & d) == 0) == ((lane & size) == 0);   // this lane keeps the smaller pair
            const bool less = ok < k || (ok == k && oj < j);
            if (low == less) { k = ok; j = oj; }
        }
    }
    uint64_t near = ~0ull;   // smallest key difference to a smaller index: the deepest shared level
    for (uint32_t t = 0; t < cnt; ++t) {
        const uint64_t x = __shfl_sync(0xFFFFFFFFu, (unsigned long long)k, t) ^ k;
        if (__shfl_sync(0xFFFFFFFFu, j, t) < j && x < near) near = x;
    }
    int leafl = c.lmax;
    bool open = here;   // this point's node is inner down to the level before
    for (int L = q + 1; L <= c.lmax && __any_sync(0xFFFFFFFFu, open); ++L) {
        const int sh = 3 * (kKeyLevels - L);
        const uint64_t up = __shfl_up_sync(0xFFFFFFFFu, (unsigned long long)k, 1);
        const bool head = here && (lane == 0 || (up ^ k) >> sh != 0);
        const uint32_t heads = __ballot_sync(0xFFFFFFFFu, head);
        const uint32_t later = heads & ~((2u << lane) - 1u);
        const int first = 31 - __clz(heads & ((2u << lane) - 1u));   // (cnt >= 1: lane 0 is one)
        const uint32_t n = (later ? (uint32_t)__ffs(later) - 1u : cnt) - (uint32_t)first;
        const bool leaf = n <= c.C || L == c.lmax;
        const uint32_t put = __ballot_sync(0xFFFFFFFFu, head && open);
        uint32_t id = 0;
        if (lane == 0 && put) id = atomicAdd(c.nnode, (uint32_t)__popc(put));
        id = __shfl_sync(0xFFFFFFFFu, id, 0);
        if (head && open)
            put_node(c, id + (uint32_t)__popc(put & lanemask_lt()), k >> sh, L, n, begin + (uint32_t)lane, leaf);
        if (open && leaf) {
            leafl = L;
            open = false;
        }
    }
    if (here) {
        const int lambda = near == ~0ull ? A : (near == 0 ? kKeyLevels : (__clzll((long long)near) - 1) / 3) + 1;
        put_lambda(c, j, lambda, leafl, (uint32_t)(k >> (3 * (kKeyLevels - c.g))));
    }
}

// level-g cells of 1 .. kSmallMax points, then the small pieces of the
// split rounds.  The cells in groups of 64, two per lane: a lane reads the counts
// of 32 groups (grid level g - 2) first and only those that hold points are
// opened; the four words of a group's cells arrive together.  Bound by the latency
// of these reads.  (Reading every cell's count first: 10^7 LiDAR points 36 -> 30 us,
// 20,000 points 12 -> 10 us; 10^6 uniform points, where every group holds some, 18 ->
// 19 us.)
__global__ void __launch_bounds__(256) k_small_pieces(OctCtx c, const uint32_t* __restrict__ pyr)
{
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t cells = 1u << (3 * c.g);   // (a multiple of 8)
    if (warp == 0 && lane == 0 && c.cstart[cells] != c.nrec_max) raise(c.err, FP_ERR_CAPACITY, 4);
    const uint32_t groups = max(cells / 64, 1u);
    const uint32_t* held = c.g >= 2 ? pyr + pyr_off(c.g - 2) : nullptr;   // points of every group
    struct Words {   // of two cells: cursors' ends, starts, the next start, leaf levels
        uint2 end, st;
        uint32_t to, leaf;
    };
    auto load = [&](uint32_t m) {
        Words w{make_uint2(0u, 0u), make_uint2(0u, 0u), 0u, 0u};
        if (m < cells) {
            w.end = *reinterpret_cast<const uint2*>(c.cursor + cursor_slot(m, c.g));
            w.st = *reinterpret_cast<const uint2*>(c.cstart + m);
            w.to = c.cstart[m + 2];
            w.leaf = *reinterpret_cast<const uint16_t*>(c.cell_leaf + m);
        }
        return w;
    };
    for (uint64_t g0 = warp; g0 < groups; g0 += 32ull * nwarps) {
        const uint64_t mine = g0 + (uint64_t)lane * nwarps;
        uint32_t todo = __ballot_sync(0xFFFFFFFFu, mine < groups && (!held || __ldg(held + mine) != 0));
        if (!todo) continue;
        auto cell = [&](uint32_t left) {   // this lane's first cell of the next group (cells: none)
            const uint64_t m = left ? (g0 + (uint64_t)(__ffs(left) - 1) * nwarps) * 64 + 2 * lane : (uint64_t)cells;
            return (uint32_t)min(m, (uint64_t)cells);
        };
        Words ahead = load(cell(todo));
        for (; todo; todo &= todo - 1) {   // the next group's words are on their way while this one is worked on
            const Words w = ahead;
            ahead = load(cell(todo & (todo - 1)));
            SmallPiece a{0u, 0u, 0u}, b{0u, 0u, 0u};
            const uint32_t na = w.st.y - w.st.x, nb = w.to - w.st.y;
            // a cell's cursor that does not end at the next one's start: a count grid of other points (points
            // in a cell without any by the grid make another one come up short, or the totals differ)
            if ((na && w.end.x != w.st.y) || (nb && w.end.y != w.to)) raise(c.err, FP_ERR_CAPACITY, 4);
            const uint32_t la = w.leaf & 255u, lb = w.leaf >> 8;
            if (na <= (uint32_t)kSmallMax && la != kInner) a = SmallPiece{w.st.x, na, (la << 8) | ((uint32_t)c.g << 16)};
            if (nb <= (uint32_t)kSmallMax && lb != kInner) b = SmallPiece{w.st.y, nb, (lb << 8) | ((uint32_t)c.g << 16)};
            if (__any_sync(0xFFFFFFFFu, (a.cnt | b.cnt) != 0)) small_warp(c, a, b);
            // the inner ones, one after the other
            uint32_t ia = __ballot_sync(0xFFFFFFFFu, na && na <= (uint32_t)kSmallMax && la == kInner);
            uint32_t ib = __ballot_sync(0xFFFFFFFFu, nb && nb <= (uint32_t)kSmallMax && lb == kInner);
            for (; ia; ia &= ia - 1) {
                const int l = __ffs(ia) - 1;
                inner_warp(c, __shfl_sync(0xFFFFFFFFu, w.st.x, l), __shfl_sync(0xFFFFFFFFu, na, l), c.g, c.g, 0);
            }
            for (; ib; ib &= ib - 1) {
                const int l = __ffs(ib) - 1;
                inner_warp(c, __shfl_sync(0xFFFFFFFFu, w.st.y, l), __shfl_sync(0xFFFFFFFFu, nb, l), c.g, c.g, 0);
            }
        }
    }
    const uint32_t ns = min(*c.n[LIST_SMALL], c.piece_cap);
    // spread over the warps (32 pieces in a row kept a few warps busy for 40 us after the others)
    for (uint64_t p0 = warp; p0 < ns; p0 += 32ull * nwarps) {
        SmallPiece a{0u, 0u, 0u};
        const uint64_t at = p0 + (uint64_t)lane * nwarps;
        Piece p{};
        if (at < ns) {
            p = c.list[LIST_SMALL][at];
            if (p.hier != kInner)
                a = SmallPiece{p.begin, p.count, (uint32_t)p.buf | ((uint32_t)p.hier << 8) | ((uint32_t)p.A << 16)};
        }
        if (__any_sync(0xFFFFFFFFu, a.cnt != 0)) small_warp(c, a, SmallPiece{0u, 0u, 0u});
        for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, at < ns && p.hier == kInner); todo; todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            const uint32_t what = __shfl_sync(0xFFFFFFFFu, (uint32_t)p.q | ((uint32_t)p.A << 8) | ((uint32_t)p.buf << 16), l);
            inner_warp(c, __shfl_sync(0xFFFFFFFFu, p.begin, l), __shfl_sync(0xFFFFFFFFu, p.count, l), (int)(what & 255u),
                       (int)((what >> 8) & 255u), (int)(what >> 16));
        }
    }
}

// A record that is not the smallest index of its cell at some level is not at
// any coarser one either, so levels are taken deepest first and a record stops
// at the first level it loses; lambda is the last level it held.

// A piece of at most R * kTabNT records and kTabDirect levels: a direct-mapped
// table of 8^d entries per level, the whole chain entered first and read back
// after one barrier.
template <int R>
FP_DEV void direct_piece(const OctCtx& c, const Piece& p, int D, uint32_t* tab, uint32_t* s_min)
{
    const int tid = threadIdx.x;
    const int n = (int)p.count, leafl = p.hier, q = p.q;
    const int sh = 3 * (kKeyLevels - q - D);
    const uint32_t cmask = (1u << (3 * D)) - 1u;
    uint32_t kk[R], j[R], cell = 0;
    {
        uint4 rec[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            rec[r] = make_uint4(0u, 0u, 0u, 0u);
            if (r * kTabNT + tid < n) rec[r] = get_rec(c, p.buf, (uint64_t)p.begin + r * kTabNT + tid);
        }
        // clear the tables while the records arrive
        const int words4 = (int)((((1u << (3 * (D + 1))) - 8u) / 7u + 3u) / 4u);
        for (int x = tid; x < words4; x += kTabNT)
            reinterpret_cast<uint4*>(tab)[x] = make_uint4(kNone, kNone, kNone, kNone);
        if (tid == 0) *s_min = kNone;
        cell = (uint32_t)(rec_key(rec[0]) >> (3 * (kKeyLevels - c.g)));   // the piece lies in one level-g cell
#pragma unroll
        for (int r = 0; r < R; ++r) {
            kk[r] = (uint32_t)(rec_key(rec[r]) >> sh) & cmask;
            j[r] = rec[r].z;
        }
    }
    __syncthreads();
    int lost[R];   // level at which the record met a smaller index (0: none)
#pragma unroll
    for (int r = 0; r < R; ++r) {
        lost[r] = 0;
        if (r * kTabNT + tid >= n) continue;
        const uint32_t jv = j[r];
        bool least = true;
#pragma unroll
        for (int d = kTabDirect; d >= 1; --d) {
            if (d <= D && least) {
                uint32_t* t = &tab[((1u << (3 * d)) - 8u) / 7u + (kk[r] >> (3 * (D - d)))];
                if (*t < jv) { least = false; lost[r] = d; }
                else atomicMin(t, jv);
            }
        }
        if (least && *s_min > jv) atomicMin(s_min, jv);
    }
    __syncthreads();
    const uint32_t jmin = *s_min;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r * kTabNT + tid >= n) continue;
        int top = kKeyLevels + 1 - q;   // never its cell's minimum down to the piece's depth
        bool held = true;
#pragma unroll
        for (int d = kTabDirect; d >= 1; --d) {
            if (d <= D && held) {
                held = d > lost[r] && tab[((1u << (3 * d)) - 8u) / 7u + (kk[r] >> (3 * (D - d)))] == j[r];
                if (held) top = d;
            }
        }
        put_lambda(c, j[r], j[r] == jmin ? (int)p.A : q + top, leafl, cell);   // (the minimum: from the split tree)
    }
    __syncthreads();   // the tables are free for the next piece
}

// A deeper piece: level by level, one hash table of (cell << 30 | index) words,
// entered by the records still holding; loops instead of registers, since few
// records hold on at the coarser levels and unrolled code overran the
// instruction cache (the top stall).
FP_DEV void hash_piece(const OctCtx& c, const Piece& p, int D, uint64_t* mine /* kPieceMax */,
                       unsigned long long* ht /* kHashSlots */, uint32_t* s_min)
{
    const int tid = threadIdx.x;
    const int n = (int)p.count, leafl = p.hier, q = p.q;
    const int sh = 3 * (kKeyLevels - q - D);
    const uint32_t cmask = (uint32_t)((1ull << (3 * D)) - 1);
    const uint32_t cell = (uint32_t)(rec_key(get_rec(c, p.buf, p.begin)) >> (3 * (kKeyLevels - c.g)));
    const uint32_t slots = (uint32_t)(n + (n >> 1)) & ~1u;   // even; at most two thirds are taken
    if (tid == 0) *s_min = kNone;
#pragma unroll 4
    for (int r = tid; r < n; r += kTabNT) {
        const uint4 rec = get_rec(c, p.buf, (uint64_t)p.begin + r);
        mine[r] = ((uint64_t)((uint32_t)(rec_key(rec) >> sh) & cmask) << 30) | rec.z;
    }
    constexpr uint32_t kJMask = (1u << 30) - 1u;
    for (int d = D; d >= 1; --d) {
        for (uint32_t x = tid; x < slots / 2; x += kTabNT)
            reinterpret_cast<uint4*>(ht)[x] = make_uint4(kNone, kNone, kNone, kNone);
        __syncthreads();
        const int lambda = d == D ? kKeyLevels + 1 : q + d + 1;   // of a record that loses level d
        for (int r = tid; r < n; r += kTabNT) {
            const uint64_t m0 = mine[r];
            if (m0 == kHashEmpty) continue;   // lost before
            const uint32_t key = (uint32_t)(m0 >> 30) >> (3 * (D - d));
            const unsigned long long m = ((unsigned long long)key << 30) | (m0 & kJMask);
            uint32_t h = __umulhi(key * 2654435761u, slots);
            for (;;) {   // fewer cells than slots: an empty one is reached
                unsigned long long e = ht[h];
                if (e == kHashEmpty && (e = atomicCAS(&ht[h], kHashEmpty, m)) == kHashEmpty) break;
                if ((uint32_t)(e >> 30) == key) {
                    if (e > m) e = atomicMin(&ht[h], m);   // (words of one cell differ by the index)
                    if (e < m) {
                        mine[r] = kHashEmpty;
                        put_lambda(c, (uint32_t)m & kJMask, lambda, leafl, cell);
                    }
                    break;
                }
                h = h + 1 == slots ? 0 : h + 1;
            }
        }
        __syncthreads();
        for (int r = tid; r < n; r += kTabNT) {
            const uint64_t m0 = mine[r];
            if (m0 == kHashEmpty) continue;
            const uint32_t key = (uint32_t)(m0 >> 30) >> (3 * (D - d)), jv = (uint32_t)m0 & kJMask;
            uint32_t h = __umulhi(key * 2654435761u, slots);
            unsigned long long e = ht[h];
            while ((uint32_t)(e >> 30) != key) {   // the record's cell is in the table
                h = h + 1 == slots ? 0 : h + 1;
                e = ht[h];
            }
            if (((uint32_t)e & kJMask) != jv) {
                mine[r] = kHashEmpty;
                put_lambda(c, jv, lambda, leafl, cell);
            } else if (d == 1) {
                atomicMin(s_min, jv);
            }
        }
        __syncthreads();
    }
    const uint32_t jmin = *s_min;
    for (int r = tid; r < n; r += kTabNT)
        if (mine[r] != kHashEmpty) {
            const uint32_t jv = (uint32_t)mine[r] & kJMask;
            put_lambda(c, jv, jv == jmin ? (int)p.A : q + 1, leafl, cell);
        }
    __syncthreads();
}

__global__ void __launch_bounds__(kTabNT, kTabCtas) k_tab_pieces(OctCtx c)
{
    __shared__ __align__(16) unsigned char buf[kTabBytes];
    __shared__ uint32_t s_min;
    __shared__ uint32_t s_next;
    const uint32_t nt = min(*c.n[LIST_TAB], c.piece_cap);
    // runs of up to kTabRun pieces (fewer when that would leave blocks without
    // work: 10^7 points, 0.23 against 0.29 ms) are taken in order from a counter: with a fixed share
    // per block the blocks drifted apart over a large cloud until their scattered
    // codes no longer met in L2 (5 * 10^8 points: 19.4 GB read and 12.5 GB
    // written instead of 8 and 2, 13.0 instead of 6.1 ms)
    const uint32_t run = max(1u, min((uint32_t)kTabRun, nt / (gridDim.x * 16)));
    if (threadIdx.x == 0) s_next = atomicAdd(c.tab_claim, run);
    __syncthreads();
    uint32_t k = s_next, k1 = k + run;
    __syncthreads();   // every warp has read s_next before thread 0 writes it (at once, where run is 1)
    Piece next{};
    if (k < nt) next = c.list[LIST_TAB][k];
    while (k < nt) {
        const Piece p = next;
        if (k + 1 == k1) {   // (a barrier before this write, the piece's own ones before the read below)
            if (threadIdx.x == 0) s_next = atomicAdd(c.tab_claim, run);
        } else if (k + 1 < nt) {   // the next piece's records on their way to L2 during this one's work
            next = c.list[LIST_TAB][k + 1];
            const uint32_t line = threadIdx.x * 8;   // 128 bytes a thread
            if (line < next.count && (uint64_t)next.begin + line < c.nrec_max)
                prefetch_l2(c.recs[next.buf] + next.begin + line);
        }
        const int D = piece_depth(c, p.q, p.hier);
        uint32_t* tab = reinterpret_cast<uint32_t*>(buf);
        if (D > kTabDirect)
            hash_piece(c, p, D, reinterpret_cast<uint64_t*>(buf),
                       reinterpret_cast<unsigned long long*>(buf + sizeof(uint64_t) * kPieceMax), &s_min);
        else if (p.count <= 2 * kTabNT) direct_piece<2>(c, p, D, tab, &s_min);
        else if (p.count <= 4 * kTabNT) direct_piece<4>(c, p, D, tab, &s_min);
        else direct_piece<kPieceMax / kTabNT>(c, p, D, tab, &s_min);
        if (++k == k1) {
            k = s_next;
            k1 = k + run;
            if (k < nt) next = c.list[LIST_TAB][k];
            __syncthreads();   // s_next is read before it is written again
        }
    }
}

// Large clouds: table pieces of up to kWarpMax points and kWarpDepth levels take one
// warp each, with a table of its own and no block barrier (k_warp_pieces); a block
// takes the other ones of the same list, a run's in order (k_tab_pieces_split).  A
// block of 128 threads per piece spent its time on barriers and half-empty rows.
// Octree stage of uniform points: 6.4 * 10^7 (31 a cell) 3.9 -> 3.0 ms, 10^8 6.6 -> 5.3,
// 2 * 10^8 9.2 -> 7.8; pieces of 5 * 10^8 (238 a cell) 6.6 -> 5.3 ms, of 10^8 LiDAR points
// 2.0 -> 1.9 ms; of 10^7 LiDAR points, mostly deep pieces, 0.235 -> 0.265 ms: hence
// the line at kTabSplit points.
constexpr uint64_t kTabSplit = 1ull << 25;
constexpr int kWarpMax = 128, kWarpDepth = 3;
constexpr int kWarpWords = 592;   // 8 + 64 + 512 entries, 16-byte rows

FP_DEV bool warp_kind(const OctCtx& c, const Piece& p)
{
    return p.count <= (uint32_t)kWarpMax && piece_depth(c, p.q, p.hier) <= kWarpDepth;
}

__global__ void __launch_bounds__(kTabNT, kTabCtas) k_tab_pieces_split(OctCtx c)
{
    __shared__ __align__(16) unsigned char buf[kTabBytes];
    __shared__ Piece s_piece[kTabNT];
    __shared__ uint32_t s_min;
    __shared__ uint32_t s_next;
    __shared__ uint32_t s_warp[kTabNT / 32];
    const uint32_t nt = min(*c.n[LIST_TAB], c.piece_cap);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // (runs as above; while one holds nothing but pieces for single warps, the next is twice as long)
    const uint32_t run0 = max(1u, min((uint32_t)kTabRun, nt / (gridDim.x * 16)));
    uint32_t run = run0;
    if (threadIdx.x == 0) s_next = atomicAdd(c.tab_claim, run);
    __syncthreads();
    uint32_t k = s_next;
    while (k < nt) {
        // the run's pieces for a block, in order
        Piece mine{};
        const bool in = threadIdx.x < run && k + threadIdx.x < nt;
        if (in) mine = c.list[LIST_TAB][k + threadIdx.x];
        const bool take = in && !warp_kind(c, mine);
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, take);
        if (lane == 0) s_warp[warp] = __popc(bal);
        __syncthreads();   // (also: s_next is read)
        uint32_t before = 0, m = 0;
#pragma unroll
        for (int x = 0; x < kTabNT / 32; ++x) {
            if (x < warp) before += s_warp[x];
            m += s_warp[x];
        }
        if (take) s_piece[before + __popc(bal & lanemask_lt())] = mine;
        run = m ? run0 : min(2 * run, (uint32_t)kTabNT);
        if (threadIdx.x == 0) s_next = atomicAdd(c.tab_claim, run);
        __syncthreads();
        for (uint32_t i = 0; i < m; ++i) {
            const Piece p = s_piece[i];
            if (i + 1 < m) {   // the next piece's records on their way to L2 during this one's work
                const Piece next = s_piece[i + 1];
                const uint32_t line = threadIdx.x * 8;   // 128 bytes a thread
                if (line < next.count && (uint64_t)next.begin + line < c.nrec_max)
                    prefetch_l2(c.recs[next.buf] + next.begin + line);
            }
            const int D = piece_depth(c, p.q, p.hier);
            uint32_t* tab = reinterpret_cast<uint32_t*>(buf);
            if (D > kTabDirect)
                hash_piece(c, p, D, reinterpret_cast<uint64_t*>(buf),
                           reinterpret_cast<unsigned long long*>(buf + sizeof(uint64_t) * kPieceMax), &s_min);
            else if (p.count <= 2 * kTabNT) direct_piece<2>(c, p, D, tab, &s_min);
            else if (p.count <= 4 * kTabNT) direct_piece<4>(c, p, D, tab, &s_min);
            else direct_piece<kPieceMax / kTabNT>(c, p, D, tab, &s_min);
        }
        k = s_next;   // (written before the barrier above)
    }
}

constexpr int kWarpNT = 256;

__global__ void __launch_bounds__(kWarpNT, 6) k_warp_pieces(OctCtx c)
{
    __shared__ __align__(16) uint32_t s_tab[kWarpNT / 32][kWarpWords];
    const int lane = threadIdx.x & 31;
    uint32_t* tab = s_tab[threadIdx.x >> 5];
    const uint32_t nt = min(*c.n[LIST_TAB], c.piece_cap);
    const uint32_t w = (blockIdx.x * kWarpNT + threadIdx.x) >> 5, nwarps = gridDim.x * (kWarpNT / 32);
    constexpr uint32_t kRun = 8;   // pieces a warp looks at together; the warps side by side
    for (uint64_t k0 = (uint64_t)w * kRun; k0 < nt; k0 += (uint64_t)nwarps * kRun) {
        Piece mine{};
        const bool in = lane < (int)kRun && k0 + lane < nt;
        if (in) mine = c.list[LIST_TAB][k0 + lane];
        uint32_t todo = __ballot_sync(0xFFFFFFFFu, in && warp_kind(c, mine));
        for (; todo; todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            Piece p;
            p.begin = __shfl_sync(0xFFFFFFFFu, mine.begin, l);
            const uint32_t n = __shfl_sync(0xFFFFFFFFu, mine.count, l);
            const uint32_t what = __shfl_sync(
                0xFFFFFFFFu, (uint32_t)mine.q | ((uint32_t)mine.hier << 8) | ((uint32_t)mine.A << 16) | ((uint32_t)mine.buf << 24), l);
            const int q = (int)(what & 255u), leafl = (int)((what >> 8) & 255u), A = (int)((what >> 16) & 255u);
            const int bufi = (int)(what >> 24);
            const int D = piece_depth(c, q, leafl);
            const int sh = 3 * (kKeyLevels - q - D);
            const uint32_t cmask = (1u << (3 * D)) - 1u;
            constexpr int R = kWarpMax / 32;
            uint32_t kk[R], j[R], cell = 0;
            {
                uint4 rec[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    rec[r] = make_uint4(0u, 0u, 0u, 0u);
                    if (r * 32u + lane < n) rec[r] = get_rec(c, bufi, (uint64_t)p.begin + r * 32 + lane);
                }
                const int words4 = (int)((((1u << (3 * (D + 1))) - 8u) / 7u + 3u) / 4u);
                for (int x = lane; x < words4; x += 32)
                    reinterpret_cast<uint4*>(tab)[x] = make_uint4(kNone, kNone, kNone, kNone);
                cell = (uint32_t)(rec_key(rec[0]) >> (3 * (kKeyLevels - c.g)));   // the piece lies in one level-g cell
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    kk[r] = (uint32_t)(rec_key(rec[r]) >> sh) & cmask;
                    j[r] = rec[r].z;
                }
            }
            __syncwarp();
            uint32_t least_j = kNone;
            int lost[R];   // level at which the record met a smaller index (0: none)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                lost[r] = 0;
                if (r * 32u + lane >= n) continue;
                const uint32_t jv = j[r];
                least_j = min(least_j, jv);
                bool least = true;
#pragma unroll
                for (int d = kWarpDepth; d >= 1; --d) {
                    if (d <= D && least) {
                        uint32_t* t = &tab[((1u << (3 * d)) - 8u) / 7u + (kk[r] >> (3 * (D - d)))];
                        if (*(volatile uint32_t*)t < jv) { least = false; lost[r] = d; }
                        else atomicMin(t, jv);
                    }
                }
            }
            const uint32_t jmin = __reduce_min_sync(0xFFFFFFFFu, least_j);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r * 32u + lane >= n) continue;
                int top = kKeyLevels + 1 - q;   // never its cell's minimum down to the piece's depth
                bool held = true;
#pragma unroll
                for (int d = kWarpDepth; d >= 1; --d) {
                    if (d <= D && held) {
                        held = d > lost[r] &&
                               *(volatile uint32_t*)&tab[((1u << (3 * d)) - 8u) / 7u + (kk[r] >> (3 * (D - d)))] == j[r];
                        if (held) top = d;
                    }
                }
                put_lambda(c, j[r], j[r] == jmin ? A : q + top, leafl, cell);   // (the minimum: from the split tree)
            }
            __syncwarp();   // the table is free for the next piece
        }
    }
}

// ---- general pieces
constexpr int kGenNT = 256;
constexpr int kGenWarps = kGenNT / 32;
struct GenSmem {
    uint64_t key[kPieceMax];
    uint64_t key2[kPieceMax];
    uint32_t j[kPieceMax];       // by load order
    uint32_t mt[kPieceMax];      // min-tree over hj: internal nodes 1..P-1 (the leaves are hj itself)
    uint32_t hj[kPieceMax];      // by run: smallest index of the run
    uint16_t v[kPieceMax];       // load position by sorted position
    uint16_t v2[kPieceMax];
    uint16_t hid[kPieceMax];     // by sorted position: run number
    uint8_t cl[kPieceMax];       // by run: common level with the nearest smaller index on the left (255: none)
    uint8_t cr[kPieceMax];       // ... on the right
    uint8_t leaf[kPieceMax];     // leaf level by sorted position (inner pieces)
    uint16_t whist[kGenWarps][256];
    uint32_t scan[64];
    uint64_t wmin[kGenWarps], wmax[kGenWarps];
    unsigned long long kmin, kmax;
    uint32_t nh, base;
};

// stable LSD pass over the piece's records by 8 key bits at `shift`
FP_DEV void gen_sort_pass(GenSmem& S, const uint64_t* kin, const uint16_t* vin, uint64_t* kout, uint16_t* vout,
                          int cnt, int shift)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int per_warp = kPieceMax / kGenWarps;   // records per warp
    for (int q = threadIdx.x; q < kGenWarps * 256; q += kGenNT) (&S.whist[0][0])[q] = 0;
    __syncthreads();
    uint32_t pack[per_warp / 32];
#pragma unroll
    for (int r = 0; r < per_warp / 32; ++r) {
        int p = warp * per_warp + r * 32 + lane;
        uint32_t d = p < cnt ? (uint32_t)(kin[p] >> shift) & 255u : 0xFFFFu;
        uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        int leader = __ffs(peers) - 1;
        uint32_t old = 0;
        if (lane == leader && d != 0xFFFFu) {
            old = S.whist[warp][d];
            S.whist[warp][d] = (uint16_t)(old + __popc(peers));
        }
        old = __shfl_sync(0xFFFFFFFFu, old, leader);
        pack[r] = d | ((old + __popc(peers & lanemask_lt())) << 16);
        __syncwarp();
    }
    __syncthreads();
    // exclusive prefix over (digit, warp): each thread owns one digit
    uint32_t tot_d = 0;
    for (int w = 0; w < kGenWarps; ++w) {
        uint32_t v = S.whist[w][threadIdx.x];
        S.whist[w][threadIdx.x] = (uint16_t)tot_d;
        tot_d += v;
    }
    uint32_t tot;
    uint32_t ex = block_exclusive_scan<kGenNT, uint32_t>(tot_d, S.scan, tot);
    for (int w = 0; w < kGenWarps; ++w) S.whist[w][threadIdx.x] = (uint16_t)(S.whist[w][threadIdx.x] + ex);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < per_warp / 32; ++r) {
        int p = warp * per_warp + r * 32 + lane;
        if (p < cnt) {
            uint32_t d = pack[r] & 0xFFFFu;
            uint32_t pos = S.whist[warp][d] + (pack[r] >> 16);
            kout[pos] = kin[p];
            vout[pos] = vin[p];
        }
    }
    __syncthreads();
}
static_assert(kGenNT == 256, "gen_sort_pass: one thread per digit");

// One piece per block: sort the records by key (stable, 8-bit LSD passes in
// shared memory); nearest smaller index on each side along the key order
// (min-tree walks over one representative per run of equal keys).  The deeper
// of the levels shared with those two neighbours, plus one, is lambda unless
// the record is the minimum of its piece, whose lambda comes from the split
// tree.  The nodes of inner pieces follow from the sorted keys too.
FP_DEV void general_piece(const OctCtx& c, GenSmem& S, const Piece& pc)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cnt = (int)pc.count;
    const int dl = pc.hier == kInner ? c.dl : min(kKeyLevels, c.s + (int)pc.hier - 1);
    {
        uint64_t mn = ~0ull, mx = 0;
        constexpr int kPer = kPieceMax / kGenNT;   // records per thread
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int r = threadIdx.x + q * kGenNT;
            if (r < cnt) {
                const uint4 rec = get_rec(c, pc.buf, (uint64_t)pc.begin + r);
                const uint64_t k = rec_key(rec);
                S.key[r] = k;
                S.j[r] = rec.z;
                S.v[r] = (uint16_t)r;
                mn = min(mn, k);
                mx = max(mx, k);
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            mn = min(mn, (uint64_t)__shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)mn, o));
            mx = max(mx, (uint64_t)__shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)mx, o));
        }
        if (lane == 0) { S.wmin[warp] = mn; S.wmax[warp] = mx; }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 0; w < kGenWarps; ++w) { mn = min(mn, S.wmin[w]); mx = max(mx, S.wmax[w]); }
            S.kmin = mn;
            S.kmax = mx;
        }
    }
    __syncthreads();
    const int clev = common_level(S.kmin, S.kmax);
    const int lo_bit = 3 * (kKeyLevels - max(dl, clev));
    {
        // records already in key order down to the needed depth need no sort
        const int hi_bit = (int)pc.srt >= max(dl, clev) ? 0 : 3 * (kKeyLevels - clev);
        bool in_key = true;
        for (int sh = lo_bit; sh < hi_bit; sh += 8) {
            if (in_key) gen_sort_pass(S, S.key, S.v, S.key2, S.v2, cnt, sh);
            else gen_sort_pass(S, S.key2, S.v2, S.key, S.v, cnt, sh);
            in_key = !in_key;
        }
        if (!in_key) {
            for (int r = threadIdx.x; r < cnt; r += kGenNT) { S.key[r] = S.key2[r]; S.v[r] = S.v2[r]; }
        }
    }
    __syncthreads();
    // ---- runs: records equal down to the sorted depth share every cell down
    // to that depth, so only the smallest index of a run can be the minimum of
    // any of those cells and the others inherit "never" (lambda beyond the
    // depth).  The search below runs over one representative per run: the
    // run's smallest index, with the run's key.
    {
        constexpr int per_h = kPieceMax / kGenNT;   // records per thread, contiguous
        const int h0 = threadIdx.x * per_h;
        uint32_t flags = 0, cntf = 0;
        for (int q = 0; q < per_h; ++q) {
            const int r = h0 + q;
            bool head = false;
            if (r < cnt) head = r == 0 || ((S.key[r] ^ S.key[r - 1]) >> lo_bit) != 0;
            flags |= (uint32_t)head << q;
            cntf += head;
        }
        uint32_t tot;
        const uint32_t ex0 = block_exclusive_scan<kGenNT, uint32_t>(cntf, S.scan, tot);
        for (uint32_t x = threadIdx.x; x < tot; x += kGenNT) S.hj[x] = 0xFFFFFFFFu;
        __syncthreads();
        int run = (int)ex0 - 1;   // run of the record before this thread's block
        uint32_t mn = 0xFFFFFFFFu;
        for (int q = 0; q < per_h; ++q) {
            const int r = h0 + q;
            if (r >= cnt) break;
            if ((flags >> q) & 1u) {
                if (run >= 0 && mn != 0xFFFFFFFFu) atomicMin(&S.hj[run], mn);
                ++run;
                mn = 0xFFFFFFFFu;
                S.key2[run] = S.key[r];
            }
            S.hid[r] = (uint16_t)run;
            mn = min(mn, S.j[S.v[r]]);
        }
        if (run >= 0 && mn != 0xFFFFFFFFu) atomicMin(&S.hj[run], mn);
        if (threadIdx.x == 0) S.nh = tot;
    }
    __syncthreads();
    const int nh = (int)S.nh;
    // ---- nearest smaller index on each side of every representative, by a
    // min-tree over hj (the leaves are hj itself, padded to a power of two
    // P >= 32): climb to the first sibling subtree that holds a smaller
    // index, then descend into it towards the near side.  The five levels
    // above the leaves are built per warp with shuffles, the rest by one
    // warp.  The level shared with that neighbour is the deepest level at
    // which the representative is not its cell's minimum on that side (keys
    // are sorted, so nearer records share at least as many levels).
    int P = 32;
    while (P < nh) P <<= 1;
    for (int b = warp; b < (P >> 5); b += kGenWarps) {
        const int i = (b << 5) + lane;
        uint32_t v = i < nh ? S.hj[i] : 0xFFFFFFFFu;
#pragma unroll
        for (int t = 1; t <= 5; ++t) {
            v = min(v, __shfl_xor_sync(0xFFFFFFFFu, v, 1 << (t - 1)));
            if ((lane & ((1 << t) - 1)) == 0) S.mt[(P + i) >> t] = v;
        }
    }
    __syncthreads();
    if (warp == 0) {
        for (int m = P >> 6; m >= 1; m >>= 1) {
            for (int k = m + lane; k < 2 * m; k += 32) S.mt[k] = min(S.mt[2 * k], S.mt[2 * k + 1]);
            __syncwarp();
        }
    }
    __syncthreads();
    auto tv = [&](int k) -> uint32_t {
        return k >= P ? (k - P < nh ? S.hj[k - P] : 0xFFFFFFFFu) : S.mt[k];
    };
    for (int r = threadIdx.x; r < nh; r += kGenNT) {
        const uint32_t jr = S.hj[r];
        const uint64_t kr = S.key2[r];
        int left = -1, right = -1;
        for (int k = P + r; k > 1; k >>= 1) {
            if ((k & 1) && tv(k - 1) < jr) {
                k = k - 1;
                while (k < P) k = tv(2 * k + 1) < jr ? 2 * k + 1 : 2 * k;
                left = k - P;
                break;
            }
        }
        for (int k = P + r; k > 1; k >>= 1) {
            if (!(k & 1) && tv(k + 1) < jr) {
                k = k + 1;
                while (k < P) k = tv(2 * k) < jr ? 2 * k : 2 * k + 1;
                right = k - P;
                break;
            }
        }
        S.cl[r] = left >= 0 ? (uint8_t)common_level(kr, S.key2[left]) : (uint8_t)255;
        S.cr[r] = right >= 0 ? (uint8_t)common_level(kr, S.key2[right]) : (uint8_t)255;
    }
    // ---- the nodes of a piece whose node is still inner.  A cell holds more than C of
    // the sorted records where two of them C apart share it: a record is in an inner
    // node down to the deepest level shared by the ends of any C + 1 neighbours it is
    // one of, a sliding maximum (by doubling), and starts the nodes from below the level
    // it shares with the record before it down to its leaf.  (The children of one node
    // after the other, by one warp of the block, was the longest part of such pieces: 5 *
    // 10^6 LiDAR points at capacity 2, 5.4 * 10^6 nodes, octree stage 12.0 -> 2.55 ms.)
    if (pc.hier == kInner) {
        const int C = (int)min((uint64_t)c.C, (uint64_t)cnt - 1), W = C + 1;   // (an inner node holds more than C)
        uint8_t *m = reinterpret_cast<uint8_t*>(S.mt), *m2 = m + 2 * kPieceMax;
        __syncthreads();   // (the min-tree is read)
        for (int x = threadIdx.x; x < cnt + C; x += kGenNT) {   // entry x: records x - C and x
            m[x] = x >= C && x < cnt ? (uint8_t)common_level(S.key[x - C], S.key[x]) : (uint8_t)0;
        }
        __syncthreads();
        int p = 1;
        for (; 2 * p <= W; p *= 2) {
            for (int x = threadIdx.x; x < cnt + C; x += kGenNT) m2[x] = max(m[x], x + p < cnt + C ? m[x + p] : (uint8_t)0);
            uint8_t* const o = m;
            m = m2;
            m2 = o;
            __syncthreads();
        }
        constexpr int kPer = kPieceMax / kGenNT;
        int from[kPer];
        uint32_t ne = 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int r = threadIdx.x + u * kGenNT;
            from[u] = 0;
            if (r >= cnt) continue;
            const int leafl = min(c.lmax, 1 + (int)max(m[r], m[r + W - p]));
            S.leaf[r] = (uint8_t)leafl;
            from[u] = max((int)pc.q, r ? common_level(S.key[r - 1], S.key[r]) : 0) + 1;
            ne += (uint32_t)max(0, leafl + 1 - from[u]);
        }
        uint32_t total;
        uint32_t id = block_exclusive_scan<kGenNT, uint32_t>(ne, S.scan, total);
        if (threadIdx.x == 0) S.base = atomicAdd(c.nnode, total);
        __syncthreads();
        id += S.base;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int r = threadIdx.x + u * kGenNT;
            if (r >= cnt) continue;
            const int leafl = S.leaf[r];
            int end = cnt;   // the next cell's first record, by levels
            for (int L = from[u]; L <= leafl; ++L) {
                const int sh = 3 * (kKeyLevels - L);
                const uint64_t cell = S.key[r] >> sh;
                int x = r + 1, y = end;
                while (x < y) {
                    const int mid = (x + y) >> 1;
                    if (S.key[mid] >> sh == cell) x = mid + 1;
                    else y = mid;
                }
                end = x;
                put_node(c, id++, cell, L, (uint32_t)(end - r), pc.begin + (uint32_t)r, L == leafl);
            }
        }
    }
    __syncthreads();
    // ---- owner level and leaf level of every record
    for (int r = threadIdx.x; r < cnt; r += kGenNT) {
        const int vv = S.v[r];
        const int h = S.hid[r];
        int lm = kKeyLevels;   // not its run's minimum: shares the sorted depth with a smaller index
        if (S.j[vv] == S.hj[h]) {
            const int ql = S.cl[h] == 255 ? -1 : (int)S.cl[h];
            const int qr = S.cr[h] == 255 ? -1 : (int)S.cr[h];
            lm = max(ql, qr);
        }
        const int lambda = lm < (int)pc.q ? (int)pc.A : lm + 1;   // the piece minimum: from the split tree
        const int leafl = pc.hier == kInner ? (int)S.leaf[r] : (int)pc.hier;
        put_lambda(c, S.j[vv], lambda, leafl, (uint32_t)(S.key[r] >> (3 * (kKeyLevels - c.g))));
    }
    __syncthreads();
}

// the general pieces, then the oversized ones (more than kPieceMax identical keys
// down to the deepest needed level): only their smallest index can be a minimum
__global__ void __launch_bounds__(kGenNT) k_general_pieces(OctCtx c)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GenSmem& S = *reinterpret_cast<GenSmem*>(smem_raw);
    const uint32_t ng = min(*c.n[LIST_GEN], c.piece_cap);
    for (uint32_t k = blockIdx.x; k < ng; k += gridDim.x) general_piece(c, S, c.list[LIST_GEN][k]);
    const uint32_t nd = min(*c.n[LIST_DUP], c.piece_cap);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t k = blockIdx.x; k < nd; k += gridDim.x) {
        const Piece p = c.list[LIST_DUP][k];
        const int leafl = p.hier == kInner ? c.lmax : (int)p.hier;
        uint32_t mn = kNone;
        for (uint32_t r = threadIdx.x; r < p.count; r += kGenNT) mn = min(mn, get_rec(c, p.buf, (uint64_t)p.begin + r).z);
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        if (lane == 0) S.scan[warp] = mn;
        __syncthreads();
        mn = S.scan[0];
        for (int w = 1; w < kGenWarps; ++w) mn = min(mn, S.scan[w]);
        for (uint32_t r = threadIdx.x; r < p.count; r += kGenNT) {
            const uint4 rr = get_rec(c, p.buf, (uint64_t)p.begin + r);
            put_lambda(c, rr.z, rr.z == mn ? (int)p.A : kKeyLevels + 1, leafl,
                       (uint32_t)(rec_key(rr) >> (3 * (kKeyLevels - c.g))));
        }
        __syncthreads();
    }
}

__global__ void k_clamp(uint32_t* v, uint32_t cap)
{
    if (*v > cap) *v = cap;
}

// ------------------------------------------------------------ node table
__global__ void k_node_keys(const NodeRec* nrec, const uint32_t* nnode, uint64_t* start, uint32_t* level, int lmax)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= *nnode) return;
    NodeRec r = nrec[i];
    start[i] = r.key << (3 * (lmax - r.level));
    level[i] = r.level;
}

// preorder id of node (level, start); kNone when absent
FP_DEV uint32_t node_lookup(const uint64_t* sorted_start, const uint8_t* sorted_level, uint32_t M, uint64_t start,
                            int level)
{
    uint32_t a = 0, b = M;
    while (a < b) {
        uint32_t m = (a + b) >> 1;
        if (sorted_start[m] < start) a = m + 1;
        else b = m;
    }
    if (a >= M || sorted_start[a] != start || (int)sorted_level[a] > level) return kNone;
    uint32_t id = a + (uint32_t)(level - (int)sorted_level[a]);
    if (id >= M || sorted_start[id] != start || (int)sorted_level[id] != level) return kNone;
    return id;
}

// fp_node records in preorder; lookup structures for the id resolution
__global__ void k_node_write(const NodeRec* nrec, const uint32_t* nnode, const uint32_t* order,
                             const uint64_t* sorted_start, uint8_t* sorted_level, fp_node* nodes, uint32_t node_cap,
                             uint32_t* num_nodes, uint32_t* idxtab, uint32_t* leafw, int g, int lmax, uint32_t* err)
{
    const uint32_t M = *nnode;
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        *num_nodes = M;
        if (M > node_cap) raise(err, FP_ERR_CAPACITY, 8);
    }
    if (i >= M) return;
    NodeRec r = nrec[order[i]];
    sorted_level[i] = r.level;
    leafw[i] = r.is_leaf ? r.count : 0;
    if (r.level <= g) idxtab[((1ull << (3 * r.level)) - 1) / 7 + r.key] = i;
}

__global__ void k_node_fill(const NodeRec* nrec, const uint32_t* nnode, const uint32_t* order,
                            const uint64_t* sorted_start, const uint8_t* sorted_level, fp_node* nodes,
                            uint32_t node_cap, uint32_t* ndesc, int lmax)
{
    const uint32_t M = *nnode;
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    NodeRec r = nrec[order[i]];
    fp_node o;
    o.key = r.key;
    o.first = 0;
    o.leaf_first = r.leaf_first;
    o.count = r.count;
    o.n_own = 0;
    uint64_t end = (r.key + 1) << (3 * (lmax - r.level));
    uint32_t a = i + 1, b = M;
    while (a < b) {
        uint32_t m = (a + b) >> 1;
        if (sorted_start[m] < end) a = m + 1;
        else b = m;
    }
    o.n_desc = a - i - 1;
    o.level = r.level;
    o.child_mask = 0;
    o.is_leaf = r.is_leaf;
    o.pad = 0;
    ndesc[i] = o.n_desc;
    if (i < node_cap) nodes[i] = o;
}

__global__ void k_node_children(const uint32_t* nnode, const uint64_t* sorted_start, const uint8_t* sorted_level,
                                fp_node* nodes, uint32_t node_cap, int lmax)
{
    const uint32_t M = *nnode;
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M || i >= node_cap || sorted_level[i] == 0) return;
    const int L = sorted_level[i];
    const uint64_t key = sorted_start[i] >> (3 * (lmax - L));
    uint32_t p = node_lookup(sorted_start, sorted_level, M, (key >> 3) << (3 * (lmax - L + 1)), L - 1);
    if (p != kNone && p < node_cap) {
        // child_mask is byte 37 of the 40-byte record
        unsigned char* rec = reinterpret_cast<unsigned char*>(nodes + p);
        uint32_t* word = reinterpret_cast<uint32_t*>(rec + 36);
        atomicOr(word, (1u << (key & 7)) << 8);
    }
}

// The node table in one launch of one cluster, for at most kNodeClusterMax nodes
// by the host's bound (18 launches otherwise; 1M points: about 110 -> 19 us).  Stable
// least-significant-digit-first passes over (level, start); a pass in which all
// records share the digit is left out (without nodes below the count grid: all bits
// below level g).  Octree stage with the cluster and with the grid's sorts: 122 nodes
// 129 and 242 us, 9478 nodes 1.85 and 1.96 ms, 18,295 nodes 215 and 285 us, 60,387
// nodes 362 and 318 us.  Only the bound is known here, 20 times too high for a usual
// tree (9018 nodes, bound 2 * 10^5), so the line lies where such trees do; clusters of
// points made to reach it (137,885 nodes) take 0.26 ms longer than by the sorts.
constexpr uint64_t kNodeClusterMax = 1ull << 18;

struct NodeClusterArgs {
    const NodeRec* rec;
    uint32_t* nnode;
    uint32_t ncap;
    uint64_t *key[2];
    uint32_t *val[2];
    uint32_t* hist;        // [kClCtas][256]
    uint64_t* part;        // [kClCtas]
    uint64_t* starts;      // (not one of key[])
    uint8_t* slevel;
    uint32_t *ndesc, *idxtab, *leafw;
    fp_node* nodes;
    uint32_t node_cap;
    uint32_t* num_nodes;
    int g, lmax;
    uint32_t* err;
};

__global__ void __launch_bounds__(kClNT, 1) k_node_cluster(NodeClusterArgs a)
{
    __shared__ ClSortSmem s_sort;
    __shared__ unsigned long long s_mask;
    const uint32_t rank = cl_rank(), tid = threadIdx.x, lane = tid & 31;
    const uint32_t M = min(*a.nnode, a.ncap);
    const int lmax = a.lmax;
    if (rank == 0 && tid == 0) {
        *a.num_nodes = M;
        if (M > a.node_cap) raise(a.err, FP_ERR_CAPACITY, 8);
    }
    // starts, and the bits in which any two of them differ
    if (tid == 0) s_mask = 0;
    __syncthreads();
    uint64_t diff = 0;
    const uint64_t s0 = M ? a.rec[0].key << (3 * (lmax - a.rec[0].level)) : 0;
    for (uint32_t i = rank * kClNT + tid; i < M; i += kClThreads) {
        const uint64_t s = a.rec[i].key << (3 * (lmax - a.rec[i].level));
        a.key[0][i] = s;
        a.val[0][i] = i;
        diff |= s ^ s0;
    }
    diff |= __shfl_xor_sync(0xFFFFFFFFu, diff, 16);
    diff |= __shfl_xor_sync(0xFFFFFFFFu, diff, 8);
    diff |= __shfl_xor_sync(0xFFFFFFFFu, diff, 4);
    diff |= __shfl_xor_sync(0xFFFFFFFFu, diff, 2);
    diff |= __shfl_xor_sync(0xFFFFFFFFu, diff, 1);
    if (lane == 0) atomicOr(&s_mask, (unsigned long long)diff);
    __syncthreads();
    if (tid == 0) a.part[rank] = s_mask;
    cl_sync();
    uint64_t mask = 0;
    for (int r = 0; r < kClCtas; ++r) mask |= *(volatile const uint64_t*)(a.part + r);

    int cur = 0;
    for (int pass = -1; pass < 8; ++pass) {   // -1: the level
        if (pass >= 0 && !((mask >> (8 * pass)) & 255u)) continue;
        const uint64_t* kin = a.key[cur];
        const uint32_t* vin = a.val[cur];
        uint64_t* kout = a.key[cur ^ 1];
        uint32_t* vout = a.val[cur ^ 1];
        cl_sort_pass(
            M, s_sort, a.hist,
            [&](uint32_t i) -> uint32_t {
                return pass < 0 ? a.rec[vin[i]].level : (uint32_t)(kin[i] >> (8 * pass)) & 255u;
            },
            [&](uint32_t i, uint32_t at) {
                kout[at] = kin[i];
                vout[at] = vin[i];
            });
        cur ^= 1;
    }
    // records in preorder and the lookups
    const uint64_t* ks = a.key[cur];
    const uint32_t* vs = a.val[cur];
    for (uint32_t i = rank * kClNT + tid; i < M; i += kClThreads) {
        const NodeRec r = a.rec[vs[i]];
        const uint64_t end = (r.key + 1) << (3 * (lmax - r.level));
        uint32_t b0 = i + 1, b1 = M;
        while (b0 < b1) {
            const uint32_t m = (b0 + b1) >> 1;
            if (ks[m] < end) b0 = m + 1;
            else b1 = m;
        }
        fp_node o;
        o.key = r.key;
        o.first = 0;
        o.leaf_first = r.leaf_first;
        o.count = r.count;
        o.n_own = 0;
        o.n_desc = b0 - i - 1;
        o.level = r.level;
        o.child_mask = 0;
        o.is_leaf = r.is_leaf;
        o.pad = 0;
        if (i < a.node_cap) a.nodes[i] = o;
        a.starts[i] = ks[i];
        a.slevel[i] = r.level;
        a.ndesc[i] = o.n_desc;
        a.leafw[i] = r.is_leaf ? r.count : 0;
        if (r.level <= a.g) a.idxtab[((1ull << (3 * r.level)) - 1) / 7 + r.key] = i;
    }
    cl_sync();
    for (uint32_t i = rank * kClNT + tid; i < M; i += kClThreads) {
        const NodeRec r = a.rec[vs[i]];
        if (r.level == 0 || r.key >> (3 * r.level)) continue;   // (a key beyond its level: not a record of these points)
        uint32_t p;
        if (r.level - 1 <= a.g) p = a.idxtab[((1ull << (3 * (r.level - 1))) - 1) / 7 + (r.key >> 3)];
        else p = node_lookup(ks, a.slevel, M, (r.key >> 3) << (3 * (lmax - r.level + 1)), r.level - 1);
        if (p < M && p < a.node_cap)   // child_mask is byte 37 of the 40-byte record
            atomicOr(reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(a.nodes + p) + 36),
                     (1u << (r.key & 7)) << 8);
    }
    if (rank == 0 && tid == 0 && *a.nnode > M) *a.nnode = M;   // (every CTA has read it: barriers above)
}

// The layouts of small clouds in one launch of one cluster: the points sorted
// stably by node id, from the chunk order (leaf grouping) or from the original
// order (final layout: every node's points in ascending index, the stitch
// included), then moved once.  Bound by the latency of its phases: 20,000 points,
// 157 nodes (one pass): subsample 107 -> 25 us, the leaf grouping 40 -> 15 us; the
// chain of plan, scatters, sort passes and placement was 15 launches.  Two passes
// of 65,000 points take 66 us here and 57 us as one grid-wide sort (below); one
// pass takes 37 us in both.
constexpr uint64_t kLayoutCluster = 1ull << 15;

struct LayoutArgs {
    fp_node* nodes;              // original order: `first` is filled too
    const uint32_t* num_nodes;
    uint32_t node_cap, n;
    int original;                // 1: original order, 0: chunk order
    const int4* pts;
    const uint32_t *perm, *id;   // by chunk position
    uint32_t *key[2], *val[2];   // n each
    uint32_t* hist;              // [kClCtas * 256]
    uint64_t* part;              // [kClCtas]
    int4* out;                   // nullable
    uint32_t* out_perm;          // nullable
    uint32_t* err;
};

__global__ void __launch_bounds__(kClNT, 1) k_layout_cluster(LayoutArgs a)
{
    __shared__ ClSortSmem s_sort;
    __shared__ ClScanSmem s_scan;
    const uint32_t t = cl_rank() * kClNT + threadIdx.x;
    const uint32_t M = min(*a.num_nodes, a.node_cap);
    if (a.original)
        cl_scan(M, a.part, s_scan, [&](uint32_t i) -> uint64_t { return a.nodes[i].n_own; },
                [&](uint32_t i, uint64_t ex) { a.nodes[i].first = ex; });
    for (uint32_t j = t; j < a.n; j += kClThreads) {
        uint32_t i = a.original ? a.perm[j] : j;
        uint32_t id = a.id[j];
        if (i >= a.n) { raise(a.err, FP_ERR_CAPACITY, 11); i = j; }
        if (id >= M) { raise(a.err, FP_ERR_CAPACITY, 15); id = 0; }   // not a node of the table
        a.key[0][i] = id;
        a.val[0][i] = j;
    }
    cl_sync();
    int cur = 0;
    for (uint32_t sh = 0; sh < 32 && (M ? M - 1 : 0u) >> sh; sh += 8) {
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
    const uint32_t* v = a.val[cur];
    for (uint32_t q = t; q < a.n; q += kClThreads) {
        const uint32_t j = v[q];
        if (j >= a.n) continue;   // (a slot that no point claimed: perm holds repeats)
        if (a.original) {         // the node's own range, as its record says
            const uint32_t id = a.id[j];
            if (id >= M || q < a.nodes[id].first || q - a.nodes[id].first >= a.nodes[id].n_own)
                raise(a.err, FP_ERR_CAPACITY, 15);
        }
        if (a.out) a.out[q] = __ldg(a.pts + j);
        if (a.out_perm) a.out_perm[q] = a.perm[j];
    }
}

// Above, up to kLayoutWhole points: one sort by node id of the whole array, a pass
// per 8 bits of the node count, over arrays that stay in L2.  It moves the points
// once or twice more than the chunk-wise scatter but is a third of its launches:
// 1M points, subsample 133 -> 55 us (195 nodes), 167 -> 71 us (7192 nodes), the
// leaf grouping 57 -> 46 us; at 4M points 217 -> 240 us and 98 -> 125 us.
constexpr uint64_t kLayoutWhole = 1ull << 21;

// owner and leaf ids of every distributed point; owned counts per node.
// A node at a level <= g is found from the level-g cell in the point's code
// (the id table of levels <= g); a node deeper than g lies in the subtree of its
// level-g ancestor, whose ids are consecutive in preorder: the search runs over
// that subtree only, with the point's key at max_level (32-bit for max_level
// <= 10) -- only then is the point itself read.  leafid (nullable): the leaf id.
// Owned counts are summed per tile of consecutive points in a
// shared-memory table keyed by node id (open addressing, bounded probes; a point
// that finds no slot adds to the global count directly), then flushed with one
// global atomic per node of the tile: consecutive points lie in one chunk, whose
// owners are few, and the nodes above the chunks (the root owns a point of every
// occupied level-s cell) are not hit by an atomic per point.
// Tiles of 4096 points, of 1024 for clouds of up to kResolveSmall points, whose few
// large tiles left most SMs idle: 20,000 points 11 -> 6 us (5 blocks before); 500,000 points 9 -> 6 us.
constexpr int kResolveNT = 256;
constexpr int kResolveIPT = 16, kResolveIPTSmall = 4;
constexpr uint64_t kResolveSmall = 1ull << 19;
constexpr int kOwnSlots = 1024;   // power of two
constexpr int kOwnProbes = 32;
constexpr int kResolveTabLevel = 4;   // node ids of the levels 0..4 in shared memory
constexpr int kResolveTab = ((1 << (3 * (kResolveTabLevel + 1))) - 1) / 7;

struct OwnCounts {   // the owned count of node id < cap: word id * stride
    uint32_t* n_own;
    uint32_t stride, cap;
    FP_DEV void add(uint32_t id, uint32_t v) const
    {
        if (id < cap) atomicAdd(&n_own[(uint64_t)id * stride], v);
    }
};

FP_DEV void own_add(uint32_t* keys, uint32_t* cnt, const OwnCounts& own, uint32_t id, uint32_t v)
{
    uint32_t h = (id * 2654435761u) & (kOwnSlots - 1);
    for (int q = 0; q < kOwnProbes; ++q) {
        uint32_t k = keys[h];
        if (k == kNone) {
            k = atomicCAS(&keys[h], kNone, id);
            if (k == kNone) k = id;
        }
        if (k == id) { atomicAdd(&cnt[h], v); return; }
        h = (h + 1) & (kOwnSlots - 1);
    }
    own.add(id, v);   // the table is crowded: straight to the global count
}

// id of the node at level L > g holding distributed point j (kNone when absent):
// by binary search among the descendants of its level-g cell's node, on the
// point's key at max_level
template <bool SMALL>
__device__ __noinline__ uint32_t deep_id(const fp_point* __restrict__ pts, uint64_t j, const CubeDev& cb,
                                         uint32_t cell, int L, const uint32_t* idxtab, const uint64_t* sorted_start,
                                         const uint8_t* sorted_level, const uint32_t* ndesc, uint32_t M, int g, int lmax)
{
    const uint32_t c0 = idxtab[((1ull << (3 * g)) - 1) / 7 + cell];
    if (L > lmax || c0 >= M) return kNone;
    const int4 p = ld_point(pts, j);
    const uint64_t kl = SMALL ? (uint64_t)key_small(p.x, p.y, p.z, cb, lmax)
                              : key21(p.x, p.y, p.z, cb) >> (3 * (kKeyLevels - lmax));
    const uint64_t k = kl >> (3 * (lmax - L));
    const uint32_t rr =
        node_lookup(sorted_start + c0, sorted_level + c0, min(ndesc[c0] + 1, M - c0), k << (3 * (lmax - L)), L);
    return rr != kNone ? c0 + rr : kNone;
}

template <bool SMALL, int kResolveIPT>
__global__ void __launch_bounds__(kResolveNT) k_resolve(const fp_point* __restrict__ pts, uint64_t n,
                                                        const fp_cube* cube, const uint32_t* codes,
                                                        const uint32_t* idxtab, const uint64_t* sorted_start,
                                                        const uint8_t* sorted_level, const uint32_t* ndesc,
                                                        const uint32_t* nnode, uint32_t* owner, uint32_t* leafid,
                                                        OwnCounts own, int g, int lmax, uint32_t* err)
{
    __shared__ uint32_t s_key[kOwnSlots], s_cnt[kOwnSlots];
    __shared__ uint32_t s_idx[kResolveTab];   // the node ids of the coarse levels' cells
    const CubeDev cb = load_cube(cube);
    const int tl = min(g, kResolveTabLevel);
    const uint32_t ntab = ((1u << (3 * (tl + 1))) - 1) / 7;
    for (uint32_t q = threadIdx.x; q < ntab; q += kResolveNT) s_idx[q] = idxtab[q];
    const uint32_t M = *nnode;
    const int nt = leafid ? 2 : 1;
    constexpr uint64_t kResolveTile = (uint64_t)kResolveNT * kResolveIPT;
    const uint64_t ntiles = (n + kResolveTile - 1) / kResolveTile;
    for (int q = threadIdx.x; q < kOwnSlots; q += kResolveNT) { s_key[q] = kNone; s_cnt[q] = 0; }
    for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        __syncthreads();   // the table is clear
        const uint64_t base = t * kResolveTile;
        uint32_t cw[kResolveIPT];
#pragma unroll
        for (int r = 0; r < kResolveIPT; ++r) {   // all loads in flight together
            const uint64_t j = base + (uint64_t)r * kResolveNT + threadIdx.x;
            cw[r] = j < n ? codes[j] : 0u;
        }
#pragma unroll 4
        for (int r = 0; r < kResolveIPT; ++r) {
            const uint64_t j = base + (uint64_t)r * kResolveNT + threadIdx.x;
            uint32_t oid = kNone;
            if (j < n) {
                // (the mask: a point that no piece held, of a count grid of other points, has any code)
                const uint32_t cell = code_cell(cw[r]) & ((1u << (3 * g)) - 1u);
                const int ks[2] = {code_own(cw[r]), code_leaf(cw[r])};
                uint32_t ids[2] = {0u, 0u};
                for (int u = 0; u < nt; ++u) {
                    const int L = ks[u];
                    if (L <= tl)
                        ids[u] = s_idx[((1u << (3 * L)) - 1) / 7 + (cell >> (3 * (g - L)))];
                    else if (L <= g)
                        ids[u] = idxtab[((1ull << (3 * L)) - 1) / 7 + (cell >> (3 * (g - L)))];
                    else   // (kept out of the unrolled loop: its code is large and rarely run)
                        ids[u] = deep_id<SMALL>(pts, j, cb, cell, L, idxtab, sorted_start, sorted_level,
                                                ndesc, M, g, lmax);
                }
                if (ids[0] >= M || ids[1] >= M) {   // never for a consistent tree
                    raise(err, FP_ERR_CAPACITY, 9);
                    ids[0] = ids[1] = 0;
                }
                owner[j] = ids[0];
                if (leafid) leafid[j] = ids[1];
                oid = ids[0];
            }
            if (oid != kNone) own_add(s_key, s_cnt, own, oid, 1u);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < kOwnSlots; q += kResolveNT) {   // flush, and clear for the next tile
            const uint32_t k = s_key[q];
            if (k != kNone) {
                own.add(k, s_cnt[q]);
                s_key[q] = kNone;
                s_cnt[q] = 0;
            }
        }
    }
}

typedef void (*ResolveKernel)(const fp_point*, uint64_t, const fp_cube*, const uint32_t*, const uint32_t*,
                              const uint64_t*, const uint8_t*, const uint32_t*, const uint32_t*, uint32_t*, uint32_t*,
                              OwnCounts, int, int, uint32_t*);

// the variant for n points, and its grid
static ResolveKernel resolve_kernel(uint64_t n, int lmax, int num_sms, int& grid)
{
    const bool few = n <= kResolveSmall;
    const uint64_t tile = (uint64_t)kResolveNT * (few ? kResolveIPTSmall : kResolveIPT);
    grid = (int)std::max<uint64_t>(1, std::min<uint64_t>((n + tile - 1) / tile, (uint64_t)num_sms * 8));
    if (lmax <= 10) return few ? k_resolve<true, kResolveIPTSmall> : k_resolve<true, kResolveIPT>;
    return few ? k_resolve<false, kResolveIPTSmall> : k_resolve<false, kResolveIPT>;
}

__global__ void k_write_nown(fp_node* nodes, const uint32_t* nnode, uint32_t node_cap, const uint32_t* n_own)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < *nnode && i < node_cap) nodes[i].n_own = n_own[i];
}

__global__ void k_set_u32(uint32_t* p, uint32_t v) { *p = v; }

__global__ void k_level_keys(const uint32_t* level, const uint32_t* nnode, uint64_t* keys)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < *nnode) keys[i] = level[i];
}

__global__ void k_gather_u64(const uint64_t* src, const uint32_t* idx, const uint32_t* nn, uint64_t* dst)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < *nn) dst[i] = src[idx[i]];
}

// ------------------------------------------------------------ host: octree
struct OctLayout {
    uint64_t cells, npyr, piece_cap, open_cap, big_cap, node_cap;
};

static OctLayout oct_layout(uint64_t n, const fp_params& p)
{
    OctLayout L;
    L.cells = 1ull << (3 * p.grid_log2);
    L.npyr = (L.cells - 1) / 7;
    L.piece_cap = L.cells + 16 * (n / kPieceMax) + 4096;
    L.open_cap = n / kPieceMax + 1;   // open nodes are disjoint, of more than kPieceMax records each
    L.big_cap = n / kRoundTile + 1;
    const uint64_t upper = (L.cells * 8 - 1) / 7;
    const uint64_t C = p.node_capacity ? p.node_capacity : 1;
    // every deep node is a child of an inner node, and an inner node holds more than C points:
    // at most n / C inner nodes per level, 8 children each
    uint64_t deep = 8 * (n / C + 1) * (uint64_t)(p.max_level - p.grid_log2 + 1) + 4096;
    if (deep > 2 * n + 4096) deep = 2 * n + 4096;
    L.node_cap = upper + deep;
    if (L.node_cap > 0xFFFFFFF0ull) L.node_cap = 0xFFFFFFF0ull;
    return L;
}

uint64_t node_capacity_bound(uint64_t n, const fp_params& p) { return oct_layout(n, p).node_cap; }

// nodes of a cloud of n points: every node but the root is the child of an inner
// node, and the inner nodes of a level hold more than C points each
static uint64_t node_bound(uint64_t n, const fp_params& p)
{
    const uint64_t inner = n > p.node_capacity ? n / (p.node_capacity + 1) : 0;   // (a capacity of 2^64 - 1 is one)
    uint64_t b = 1;
    for (uint32_t l = 0; l < p.max_level; ++l) b += 8 * std::min<uint64_t>(l < 20 ? 1ull << (3 * l) : ~0ull, inner);
    return b;
}

struct OctBufs {
    SortScratch sc;
    uint32_t* rcnt;        // counting slots of a split round: 8^3 per large open node
    uint32_t* rmin;        // the smallest index of every slot
    uint4* trec;           // split rounds: the second record buffer
    int4* lt_pt;
    uint32_t *lt_val, *lt_k32;
    uint32_t *pyr, *rsum, *cstart, *cursor;
    uint8_t* cell_leaf;
    uint4* rec;           // cell-grouped records (rec_key, rec_j)
    Piece* pieces[4];     // table, small, general, oversized
    uint32_t* counters;   // [0..3] their numbers, [4] node records, [5] table pieces taken, [6] barrier of the rounds
    RoundCnt* rounds;
    OpenNode *open[2], *big[2];
    NodeRec* nrec;
    uint64_t *nk, *nk2, *nk3, *nk4;
    uint32_t *nl, *nv2, *nv3;
    uint8_t* slevel;
    uint32_t *idxtab, *leafw;
    uint32_t* codes;
    uint32_t* leafid;
    uint32_t* ndesc;
    SegScratch seg;
};

constexpr int kOctCounters = 8 + (kMaxRounds + 1) * (int)(sizeof(RoundCnt) / sizeof(uint32_t));   // words, zeroed

// one carve-up serves both the size query (base == nullptr) and the launch
static OctBufs oct_carve(const Workspace& ws, uint64_t n, const OctLayout& Ly)
{
    OctBufs B;
    const uint64_t N = n ? n : 1;
    B.sc = take_sort_scratch(ws, std::max<uint64_t>(N, Ly.node_cap));
    B.rcnt = ws.take<uint32_t>(Ly.big_cap << (3 * kRoundLevels));
    B.rmin = ws.take<uint32_t>(Ly.big_cap << (3 * kRoundLevels));
    // aliased phase region: grouping temporaries, later the leaf scatter temporaries
    const size_t phase_base = ws.used;
    B.trec = ws.take<uint4>(N);
    const size_t phase_end = ws.used;
    ws.used = phase_base;
    B.lt_pt = ws.take<int4>(N); B.lt_val = ws.take<uint32_t>(N); B.lt_k32 = ws.take<uint32_t>(N);
    ws.used = std::max(phase_end, ws.used);
    B.pyr = ws.take<uint32_t>(Ly.npyr ? Ly.npyr : 1);
    B.rsum = ws.take<uint32_t>(kGtMaxTiles);
    B.cstart = ws.take<uint32_t>(Ly.cells + 1);
    B.cursor = ws.take<uint32_t>(Ly.cells);
    B.cell_leaf = ws.take<uint8_t>(Ly.cells);
    B.rec = ws.take<uint4>(N);
    for (Piece*& p : B.pieces) p = ws.take<Piece>(Ly.piece_cap);
    B.counters = ws.take<uint32_t>(kOctCounters);
    B.rounds = reinterpret_cast<RoundCnt*>(B.counters + 8);
    B.open[0] = ws.take<OpenNode>(Ly.open_cap); B.open[1] = ws.take<OpenNode>(Ly.open_cap);
    B.big[0] = ws.take<OpenNode>(Ly.big_cap); B.big[1] = ws.take<OpenNode>(Ly.big_cap);
    B.nrec = ws.take<NodeRec>(Ly.node_cap);
    B.nk = ws.take<uint64_t>(Ly.node_cap); B.nk2 = ws.take<uint64_t>(Ly.node_cap);
    B.nk3 = ws.take<uint64_t>(Ly.node_cap); B.nk4 = ws.take<uint64_t>(Ly.node_cap);
    B.nl = ws.take<uint32_t>(Ly.node_cap); B.nv2 = ws.take<uint32_t>(Ly.node_cap);
    B.nv3 = ws.take<uint32_t>(Ly.node_cap);
    B.slevel = ws.take<uint8_t>(Ly.node_cap);
    B.idxtab = ws.take<uint32_t>(Ly.cells * 8 / 7 + 8);
    B.leafw = ws.take<uint32_t>(std::max<uint64_t>(Ly.node_cap, kScanMaxTiles));
    B.codes = ws.take<uint32_t>(N);
    B.leafid = ws.take<uint32_t>(N);
    B.ndesc = ws.take<uint32_t>(Ly.node_cap);
    B.seg = take_seg_scratch(ws, N, Ly.cells, 1);
    return B;
}

size_t octree_ws_bytes(uint64_t n, const fp_params& p)
{
    Workspace dry;
    oct_carve(dry, n, oct_layout(n, p));
    return dry.used;
}

// node records -> fp_node table in preorder, the level-g id table, sorted starts,
// levels and subtree sizes (the lookups of the id resolution)
struct NodeSortBufs {
    uint64_t *nk, *nk2, *nk3, *nk4;
    uint32_t *nl, *nv2, *nv3;
    uint8_t* slevel;
    uint32_t *idxtab, *leafw, *ndesc;
};

static cudaError_t node_table(const SortScratch& sc, const NodeRec* nrec, uint32_t* nnode, uint32_t ncap,
                              uint64_t bound, const NodeSortBufs& B, fp_node* nodes, uint32_t node_cap,
                              uint32_t* num_nodes, int g, int lmax, const Workspace& ws, cudaStream_t st)
{
    cudaError_t e;
    if (bound <= kNodeClusterMax) {
        NodeClusterArgs a{};
        a.rec = nrec; a.nnode = nnode; a.ncap = ncap;
        a.key[0] = B.nk2; a.key[1] = B.nk3; a.val[0] = B.nl; a.val[1] = B.nv2;
        a.hist = sc.hist; a.part = B.nk4;
        a.starts = B.nk; a.slevel = B.slevel; a.ndesc = B.ndesc; a.idxtab = B.idxtab; a.leafw = B.leafw;
        a.nodes = nodes; a.node_cap = node_cap; a.num_nodes = num_nodes;
        a.g = g; a.lmax = lmax; a.err = ws.err;
        return cl_launch(k_node_cluster, a, st);
    }
    const unsigned gn = (ncap + 255) / 256;
    k_clamp<<<1, 1, 0, st>>>(nnode, ncap);
    k_node_keys<<<gn, 256, 0, st>>>(nrec, nnode, B.nk, B.nl, lmax);
    k_level_keys<<<gn, 256, 0, st>>>(B.nl, nnode, B.nk3);
    SortArgs a{};
    a.b.k64_src = B.nk3; a.b.k64_tmp = B.nk2; a.b.k64_dst = B.nk4;
    a.b.val_src = nullptr; a.b.val_tmp = B.nv2; a.b.val_dst = B.nv3;
    a.n = ncap; a.d_n = nnode; a.err = ws.err;
    if ((e = sort_plan_keys(sc, a, 0, 5, nullptr, false, ws.num_sms, st))) return e;
    if ((e = sort_run<DIG_K64, false, true, false>(a, sort_passes(5), ws.num_sms, st))) return e;
    k_gather_u64<<<gn, 256, 0, st>>>(B.nk, B.nv3, nnode, B.nk3);
    SortArgs b2{};
    b2.b.k64_src = B.nk3; b2.b.k64_tmp = B.nk2; b2.b.k64_dst = B.nk;   // nk <- sorted starts
    b2.b.val_src = B.nv3; b2.b.val_tmp = B.nv2; b2.b.val_dst = B.nl;   // nl <- record of preorder position
    b2.n = ncap; b2.d_n = nnode; b2.err = ws.err;
    if ((e = sort_plan_keys(sc, b2, 0, (uint32_t)std::max(1, 3 * lmax), nullptr, false, ws.num_sms, st))) return e;
    if ((e = sort_run<DIG_K64, false, true, false>(b2, sort_passes(3 * lmax), ws.num_sms, st))) return e;
    k_node_write<<<gn, 256, 0, st>>>(nrec, nnode, B.nl, B.nk, B.slevel, nodes, node_cap, num_nodes, B.idxtab, B.leafw,
                                     g, lmax, ws.err);
    k_node_fill<<<gn, 256, 0, st>>>(nrec, nnode, B.nl, B.nk, B.slevel, nodes, node_cap, B.ndesc, lmax);
    k_node_children<<<gn, 256, 0, st>>>(nnode, B.nk, B.slevel, nodes, node_cap, lmax);
    return cudaGetLastError();
}

// append the node records of a chunk group to the caller's array
__global__ void k_append_nodes(const NodeRec* rec, const uint32_t* nrec, uint32_t cap_ws, NodeRec* out,
                               uint32_t* nout, uint32_t out_cap, uint32_t* err)
{
    const uint32_t M = min(*nrec, cap_ws), base = *nout;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += stride) {
        if (base + i < out_cap) out[base + i] = rec[i];
        else raise(err, FP_ERR_CAPACITY, 10);
    }
}

__global__ void k_add_u32(uint32_t* a, const uint32_t* b, uint32_t cap_b) { *a += min(*b, cap_b); }

cudaError_t launch_octree(const fp_point* sorted, const uint32_t* perm, uint64_t n, const fp_cube* cube,
                          const fp_chunk* chunks, const uint32_t* num_chunks, const uint64_t* offsets,
                          const uint32_t* counts, const fp_params& prm, fp_node* nodes, uint32_t node_cap,
                          uint32_t* num_nodes, fp_point* leaf_pts, uint32_t* leaf_perm, uint32_t* owner,
                          const Workspace& ws, cudaStream_t st)
{
    return launch_octree_impl(sorted, perm, n, cube, chunks, num_chunks, offsets, counts, prm, nodes, node_cap,
                              num_nodes, leaf_pts, leaf_perm, owner, nullptr, ws, st);
}

cudaError_t launch_octree_impl(const fp_point* sorted, const uint32_t* perm, uint64_t n, const fp_cube* cube,
                               const fp_chunk* chunks, const uint32_t* num_chunks, const uint64_t* offsets,
                               const uint32_t* counts, const fp_params& prm, fp_node* nodes, uint32_t node_cap,
                               uint32_t* num_nodes, fp_point* leaf_pts, uint32_t* leaf_perm, uint32_t* owner,
                               const OctGroup* grp, const Workspace& ws, cudaStream_t st)
{
    cudaError_t e;
    if (n == 0) {
        if (!grp) k_set_u32<<<1, 1, 0, st>>>(num_nodes, 0);
        return cudaGetLastError();
    }
    const uint32_t* rcounts = grp ? grp->rec_counts : counts;
    const int g = (int)prm.grid_log2, s = (int)prm.sub_log2, lmax = (int)prm.max_level;
    const int dl = std::min(kKeyLevels, std::max(s + lmax - 1, g + 1));
    const OctLayout Ly = oct_layout(n, prm);
    const uint64_t N = n;
    const OctBufs B = oct_carve(ws, n, Ly);
    const SortScratch& sc = B.sc;
    uint32_t* nnode = B.counters + 4;
    OctCtx c;
    c.counts = counts; c.rcounts = rcounts; c.leaf_base = grp ? grp->leaf_base : 0u;
    c.cstart = B.cstart; c.cursor = B.cursor; c.cell_leaf = B.cell_leaf;
    c.recs[0] = B.rec; c.recs[1] = B.trec; c.nrec_max = N; c.piece_cap = (uint32_t)Ly.piece_cap;
    for (int l = 0; l < 4; ++l) { c.list[l] = B.pieces[l]; c.n[l] = B.counters + l; }
    c.tab_claim = B.counters + 5;
    c.nrec = B.nrec; c.nnode = nnode; c.node_cap_ws = (uint32_t)Ly.node_cap;
    c.codes = grp ? grp->codes : B.codes;
    c.g = g; c.s = s; c.lmax = lmax; c.dl = dl; c.C = prm.node_capacity; c.err = ws.err;
    RoundArgs ra{};
    ra.c = c;
    for (int l = 0; l < 2; ++l) { ra.small[l] = B.open[l]; ra.big[l] = B.big[l]; }
    ra.cnt = B.rounds; ra.small_cap = (uint32_t)Ly.open_cap; ra.big_cap = (uint32_t)Ly.big_cap;
    ra.slots = B.rcnt; ra.smin = B.rmin; ra.bar = B.counters + 6;

    // 1. the grid's levels, every cell's start, leaf level and piece, the nodes at
    // levels <= g (a chunk group leaves those to the whole-cloud node table)
    const int ntile = grid_tiles(g);
    k_grid_tiles<<<ntile, kGtNT, 0, st>>>(counts, g, B.pyr, rcounts, B.rsum, nullptr, 0, B.counters, kOctCounters);
    k_cells_open<<<ntile, kGtNT, 0, st>>>(ra, B.pyr, B.rsum, 1, grp ? 0 : 1, B.cstart, B.cursor);
    // 2. group by level-g cell: (key21, j) scattered by cell id
    {
        const int gs = (int)std::max<uint64_t>(1, std::min<uint64_t>((N + 255) / 256, (uint64_t)ws.num_sms * 8));
        KTimerScope kt(FP_KERNEL_CELL_GROUP, st);
        k_cell_scatter<<<gs, 256, 0, st>>>(reinterpret_cast<const int4*>(sorted), N, cube, B.cursor, B.rec, g,
                                           ws.err);
    }
    // 3. big cells split into pieces
    if (N > (uint64_t)kPieceMax) {
        KTimerScope kt(FP_KERNEL_SPLIT_ROUNDS, st);
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rounds, kRoundNT, 0))) return e;
        const unsigned grid = (unsigned)std::min<uint64_t>((N + kRoundTile - 1) / kRoundTile,
                                                           (uint64_t)ws.num_sms * std::max(per_sm, 1));
        if ((e = coop_launch(k_rounds, grid, kRoundNT, 0, st, ra))) return e;
    }
    // 4. lambda of every record: owner level and leaf level
    {
        KTimerScope kt(FP_KERNEL_UNITS, st);
        const uint64_t blk = N / (kSmallMax + 1) + 1;   // at most that many table pieces
        const int gt = (int)std::min<uint64_t>(blk, (uint64_t)ws.num_sms * kTabCtas);
        if (N >= kTabSplit) {
            k_tab_pieces_split<<<gt, kTabNT, 0, st>>>(c);
            k_warp_pieces<<<(int)std::min<uint64_t>(blk / (kWarpNT / 4) + 1, (uint64_t)ws.num_sms * 6), kWarpNT, 0, st>>>(c);
        } else {
            k_tab_pieces<<<gt, kTabNT, 0, st>>>(c);
        }
        k_small_pieces<<<(int)std::max<uint64_t>(1, std::min<uint64_t>(Ly.cells / 256, ws.num_sms * 8ull)), 256, 0,
                         st>>>(c, B.pyr);
        const size_t smem = sizeof(GenSmem);
        if ((e = cudaFuncSetAttribute(k_general_pieces, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
            return e;
        k_general_pieces<<<(int)std::min<uint64_t>(blk, ws.num_sms * 4ull), kGenNT, smem, st>>>(c);
    }
    if (grp) {   // a chunk group: its nodes below level g are appended to the caller's list
        const unsigned ga = (unsigned)std::max(1, std::min(ws.num_sms * 8, (int)((Ly.node_cap + 255) / 256)));
        k_append_nodes<<<ga, 256, 0, st>>>(B.nrec, nnode, (uint32_t)Ly.node_cap, grp->deep, grp->num_deep,
                                           grp->deep_cap, ws.err);
        k_add_u32<<<1, 1, 0, st>>>(grp->num_deep, nnode, (uint32_t)Ly.node_cap);
        return cudaGetLastError();
    }
    // 5. node table in preorder: stable sort by level, then by start at max_level resolution
    {
        NodeSortBufs nb{B.nk, B.nk2, B.nk3, B.nk4, B.nl, B.nv2, B.nv3, B.slevel, B.idxtab, B.leafw, B.ndesc};
        KTimerScope kt(FP_KERNEL_NODE_TABLE, st);
        if ((e = node_table(sc, B.nrec, nnode, (uint32_t)Ly.node_cap, node_bound(N, prm), nb, nodes, node_cap,
                            num_nodes, g, lmax, ws, st)))
            return e;
    }
    // 6. owner and leaf ids per distributed point, owned counts
    {
        int grid;
        const ResolveKernel kres = resolve_kernel(N, lmax, ws.num_sms, grid);
        // counted in the node records (zeroed with the table)
        const OwnCounts own{reinterpret_cast<uint32_t*>(nodes) + offsetof(fp_node, n_own) / sizeof(uint32_t),
                            sizeof(fp_node) / sizeof(uint32_t), node_cap};
        KTimerScope kt(FP_KERNEL_RESOLVE, st);
        kres<<<grid, kResolveNT, 0, st>>>(sorted, N, cube, B.codes, B.idxtab, B.nk, B.slevel, B.ndesc, nnode, owner,
                                   (leaf_pts || leaf_perm) ? B.leafid : nullptr,
                                   own, g, lmax, ws.err);
    }
    // 7. leaf-grouped points: stable scatter by leaf id, chunk by chunk (every
    // leaf lies in the subtree of its points' chunk); the whole-array sort by
    // leaf id runs instead, gated on the device, when a chunk does not fit
    if (leaf_pts || leaf_perm) {
        KTimerScope kt(FP_KERNEL_LEAF_SCATTER, st);
        if (N <= kLayoutCluster) {
            LayoutArgs a{};
            a.nodes = nodes; a.num_nodes = nnode; a.node_cap = (uint32_t)Ly.node_cap; a.n = (uint32_t)N;
            a.pts = reinterpret_cast<const int4*>(sorted); a.perm = perm; a.id = B.leafid;
            a.key[0] = B.leafid; a.key[1] = B.lt_k32; a.val[0] = B.lt_val; a.val[1] = B.codes;
            a.hist = sc.hist; a.part = B.seg.part;
            a.out = reinterpret_cast<int4*>(leaf_pts); a.out_perm = leaf_perm; a.err = ws.err;
            return cl_launch(k_layout_cluster, a, st);
        }
        SegCall sg{};
        sg.mode = SEG_LEAF;
        sg.nodes = nodes; sg.num_nodes = num_nodes; sg.node_cap = node_cap;
        sg.chunks = chunks; sg.num_chunks = num_chunks; sg.offsets = offsets;
        sg.pt_in = leaf_pts ? reinterpret_cast<const int4*>(sorted) : nullptr;
        sg.pt_out = reinterpret_cast<int4*>(leaf_pts);
        sg.val_in = perm; sg.val_out = leaf_perm;
        sg.id_in = B.leafid;
        sg.n = N;
        sg.first = reinterpret_cast<const uint64_t*>(nodes) + offsetof(fp_node, leaf_first) / sizeof(uint64_t);
        sg.first_stride = sizeof(fp_node) / sizeof(uint64_t);
        sg.hist = sc.hist;
        const bool all = N <= kLayoutWhole;   // the one sort by leaf id
        if (all) e = cudaMemsetAsync(sc.hist, 0, sizeof(uint32_t) * kSortHistWords, st);
        else e = seg_scatter(B.seg, sg, ws, st);
        if (e) return e;
        SortArgs a{};
        a.b.pt_src = reinterpret_cast<const int4*>(sorted);
        a.b.pt_tmp = B.lt_pt;
        a.b.pt_dst = reinterpret_cast<int4*>(leaf_pts);
        a.b.val_src = perm; a.b.val_tmp = B.lt_val; a.b.val_dst = leaf_perm;
        // (three passes read the ids back from dst; the codes are not needed any more)
        a.b.k32_src = B.leafid; a.b.k32_tmp = B.lt_k32; a.b.k32_dst = B.codes;
        a.n = N; a.run_if = all ? nullptr : B.seg.cnt + 2; a.err = ws.err;
        if ((e = sort_plan_weights(sc, a, B.leafw, nullptr, nnode, Ly.node_cap, true, ws.num_sms, st))) return e;
        const int np = sort_passes(count_bits(Ly.node_cap));   // leaf ids below node_cap
        if (leaf_pts) e = sort_run<DIG_K32, true, false, true>(a, np, ws.num_sms, st);
        else e = sort_run<DIG_K32, false, false, true>(a, np, ws.num_sms, st);
        if (e) return e;
    }
    return cudaGetLastError();
}

// ------------------------------------------- whole-cloud tables (chunk groups)
__global__ void k_copy_u32(uint32_t* dst, const uint32_t* src) { *dst = *src; }

struct NodesBufs {
    SortScratch sc;
    uint32_t *pyr, *rsum;
    NodeSortBufs nb;
};

static NodesBufs nodes_carve(const Workspace& ws, const fp_params& p, uint64_t rec_cap)
{
    NodesBufs B;
    const uint64_t cells = 1ull << (3 * p.grid_log2);
    const uint64_t R = rec_cap ? rec_cap : 1;
    B.sc = take_sort_scratch(ws, R);
    B.pyr = ws.take<uint32_t>((cells - 1) / 7 ? (cells - 1) / 7 : 1);
    B.rsum = ws.take<uint32_t>(kGtMaxTiles);
    B.nb.nk2 = ws.take<uint64_t>(R); B.nb.nk3 = ws.take<uint64_t>(R); B.nb.nk4 = ws.take<uint64_t>(R);
    B.nb.nl = ws.take<uint32_t>(R); B.nb.nv2 = ws.take<uint32_t>(R); B.nb.nv3 = ws.take<uint32_t>(R);
    return B;
}

size_t nodes_ws_bytes(const fp_params& p, uint64_t rec_cap)
{
    Workspace dry;
    nodes_carve(dry, p, rec_cap);
    return dry.used;
}

cudaError_t launch_octree_nodes(const uint32_t* counts, uint64_t n, const fp_params& prm, NodeRec* recs, uint64_t rec_cap,
                                const uint32_t* num_deep, fp_node* nodes, uint32_t node_cap, uint32_t* num_nodes,
                                const NodeTables& T, const Workspace& ws, cudaStream_t st)
{
    cudaError_t e;
    const int g = (int)prm.grid_log2, lmax = (int)prm.max_level;
    const NodesBufs B = nodes_carve(ws, prm, rec_cap);
    k_copy_u32<<<1, 1, 0, st>>>(T.nnode, num_deep);
    OctCtx c{};
    c.counts = counts; c.rcounts = counts; c.leaf_base = 0;
    c.nrec = recs; c.nnode = T.nnode; c.node_cap_ws = (uint32_t)rec_cap;
    c.g = g; c.s = (int)prm.sub_log2; c.lmax = lmax; c.C = prm.node_capacity; c.err = ws.err;
    k_grid_tiles<<<grid_tiles(g), kGtNT, 0, st>>>(counts, g, B.pyr, counts, B.rsum, nullptr, 0, nullptr, 0);
    RoundArgs ra{};
    ra.c = c;
    k_cells_open<<<grid_tiles(g), kGtNT, 0, st>>>(ra, B.pyr, B.rsum, 0, 1, nullptr, nullptr);
    NodeSortBufs nb = B.nb;
    nb.nk = T.starts; nb.slevel = T.slevel; nb.idxtab = T.idxtab; nb.ndesc = T.ndesc;
    nb.leafw = T.nown;   // (nobody reads the leaf sizes; cleared below)
    if ((e = node_table(B.sc, recs, T.nnode, (uint32_t)rec_cap, n ? node_bound(n, prm) : rec_cap, nb, nodes, node_cap,
                        num_nodes, g, lmax, ws, st)))
        return e;
    return cudaMemsetAsync(T.nown, 0, rec_cap * sizeof(uint32_t), st);
}

cudaError_t launch_octree_resolve(const fp_point* pts, uint64_t n, const fp_cube* cube, const uint32_t* codes,
                                  const NodeTables& T, const fp_params& prm,
                                  uint32_t* owner, const Workspace& ws, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    int grid;
    const ResolveKernel kres = resolve_kernel(n, (int)prm.max_level, ws.num_sms, grid);
    kres<<<grid, kResolveNT, 0, st>>>(pts, n, cube, codes, T.idxtab, T.starts, T.slevel, T.ndesc, T.nnode, owner, nullptr,
                               OwnCounts{T.nown, 1u, 0xFFFFFFFFu}, (int)prm.grid_log2, (int)prm.max_level, ws.err);
    return cudaGetLastError();
}

// n_own of every node from the owned counts, then first = exclusive prefix of n_own
cudaError_t launch_node_first(fp_node* nodes, const uint32_t* num_nodes, uint32_t node_cap, const uint32_t* nown,
                              uint64_t* first, uint32_t* nm, uint64_t* tiles64, cudaStream_t st);

// ------------------------------------------------------------ subsample
__global__ void k_first_out(fp_node* nodes, const uint32_t* num_nodes, uint32_t node_cap, const uint64_t* first)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t M = *num_nodes < node_cap ? *num_nodes : node_cap;
    if (i < M) nodes[i].first = first[i];
}

__global__ void k_clamp_copy(const uint32_t* v, uint32_t cap, uint32_t* out) { *out = *v < cap ? *v : cap; }

// The stitch for up to kStitchRanks nodes outside every chunk subtree (a hundred or
// so are usual: the levels above the chunks).  The segmented scatter has marked
// their points by original index, a byte with the node's rank and the point's
// position; in that order each node's points only have to be told apart:
//   k_stitch_count: points of every node per tile of 8192 indices;
//   k_stitch_scan: per node, the exclusive prefix over the tiles;
//   k_stitch_move: ranks in the tile (as a sort pass has them), points fetched and
//     written in runs.
// Bound by the marks (a random byte and word a point) and the fetches, so only
// while the marks stay in L2.  Whole subsample against the radix passes over (node,
// index): 10^7 LiDAR points 374 -> 336 us, uniform 756 -> 434; 4 * 10^6 uniform 348 ->
// 236; 3.3 * 10^7 966 -> 913 and 2053 -> 1742; 10^8 2367 -> 2447 and 5460 -> 6100: the
// line lies at kStitchMarked points.
constexpr uint64_t kStitchMarked = 1ull << 25;
constexpr int kStNT = 512, kStIPT = 16;
constexpr int kStTile = kStNT * kStIPT;
constexpr int kStWarps = kStNT / 32;
constexpr int kStDig = 256;

struct StitchArgs {
    const uint32_t *nrank, *fail;   // other than 1 .. kStitchRanks nodes, or a failed scatter: nothing to do
    const uint8_t* code;            // rank + 1, 0: not staged
    const uint32_t* inv;            // position among the distributed points
    uint32_t* cnt;                  // [rank][ntiles]
    const uint32_t* list;           // node of a rank
    const uint64_t* first;
    const int4* pts;
    int4* fin;
    uint32_t* fperm;
    uint64_t n;
    uint32_t ntiles;
    uint32_t* err;
};

FP_DEV uint32_t stitch_ranks(const StitchArgs& a)
{
    const uint32_t R = *a.nrank;
    return *a.fail || R > kStitchRanks ? 0u : R;
}

__global__ void __launch_bounds__(kStNT) k_stitch_count(StitchArgs a)
{
    __shared__ uint32_t s_cnt[kStDig];
    const uint32_t R = stitch_ranks(a);
    if (!R) return;
    for (uint32_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        if (threadIdx.x < kStDig) s_cnt[threadIdx.x] = 0;
        __syncthreads();
        const uint64_t i0 = (uint64_t)tile * kStTile + threadIdx.x * 16;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (i0 + 16 <= a.n) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(a.code + i0));
            w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
        } else {
            for (int b = 0; b < 16; ++b)
                if (i0 + b < a.n) w[b >> 2] |= (uint32_t)a.code[i0 + b] << (8 * (b & 3));
        }
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const uint32_t c = (w[b >> 2] >> (8 * (b & 3))) & 255u;
            if (c) atomicAdd(&s_cnt[c - 1], 1u);
        }
        __syncthreads();
        if (threadIdx.x < R) a.cnt[(uint64_t)threadIdx.x * a.ntiles + tile] = s_cnt[threadIdx.x];
        __syncthreads();
    }
}

// one block per rank
__global__ void __launch_bounds__(kStNT) k_stitch_scan(StitchArgs a)
{
    __shared__ uint32_t s_warp[kStWarps];
    const uint32_t R = stitch_ranks(a);
    if (blockIdx.x >= R) return;
    uint32_t* row = a.cnt + (uint64_t)blockIdx.x * a.ntiles;
    uint32_t run = 0;
    constexpr int kPer = 8;
    for (uint32_t t0 = 0; t0 < a.ntiles; t0 += kStNT * kPer) {
        uint32_t v[kPer], sum = 0, tot;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const uint32_t t = t0 + threadIdx.x * kPer + q;
            v[q] = t < a.ntiles ? row[t] : 0u;
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) sum += v[q];
        uint32_t ex = run + block_exclusive_scan<kStNT, uint32_t>(sum, s_warp, tot);
        run += tot;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const uint32_t t = t0 + threadIdx.x * kPer + q;
            if (t < a.ntiles) row[t] = ex;
            ex += v[q];
        }
    }
}

__global__ void __launch_bounds__(kStNT, 2) k_stitch_move(StitchArgs a)
{
    __shared__ uint16_t s_whist[kStWarps][kStDig];
    __shared__ uint32_t s_off[kStDig], s_warp[kStWarps];
    __shared__ uint64_t s_base[kStDig];
    __shared__ uint16_t s_idx[kStTile];
    __shared__ uint8_t s_dig[kStTile];
    const uint32_t R = stitch_ranks(a);
    if (!R) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        const uint64_t base = (uint64_t)tile * kStTile;
        for (int q = threadIdx.x; q < kStWarps * kStDig / 8; q += kStNT)
            reinterpret_cast<uint4*>(&s_whist[0][0])[q] = make_uint4(0u, 0u, 0u, 0u);
        uint32_t w[kStIPT / 4] = {};   // the codes of this lane, one per row of 32
#pragma unroll
        for (int r = 0; r < kStIPT; ++r) {
            const uint64_t i = base + warp * (kStIPT * 32) + r * 32 + lane;
            if (i < a.n) w[r >> 2] |= (uint32_t)__ldg(a.code + i) << (8 * (r & 3));
        }
        // (the first run position of every rank, on its way)
        uint32_t before = 0;
        uint64_t first = 0;
        if (threadIdx.x < R) {
            before = __ldg(a.cnt + (uint64_t)threadIdx.x * a.ntiles + tile);
            first = __ldg(a.first + __ldg(a.list + threadIdx.x));
        }
        __syncthreads();
        uint16_t place[kStIPT];   // place among the warp's points of the same node
#pragma unroll
        for (int r = 0; r < kStIPT; ++r) {
            const uint32_t c = (w[r >> 2] >> (8 * (r & 3))) & 255u;
            place[r] = 0;
            if (!__any_sync(0xFFFFFFFFu, c != 0)) continue;
            const uint32_t d = c - 1;
            const uint32_t peers = match_bits<8>(d, c != 0);
            const int leader = peers ? __ffs(peers) - 1 : 0;
            uint32_t old = 0;
            if (c && lane == leader) {
                old = s_whist[warp][d];
                s_whist[warp][d] = (uint16_t)(old + __popc(peers));
            }
            old = __shfl_sync(0xFFFFFFFFu, old, leader);
            place[r] = (uint16_t)(old + __popc(peers & lanemask_lt()));
            __syncwarp();
        }
        __syncthreads();
        uint32_t c = 0, total;
        if (threadIdx.x < kStDig) {
#pragma unroll
            for (int x = 0; x < kStWarps; ++x) {
                const uint32_t v = s_whist[x][threadIdx.x];
                s_whist[x][threadIdx.x] = (uint16_t)c;
                c += v;
            }
        }
        const uint32_t ex = block_exclusive_scan<kStNT, uint32_t>(c, s_warp, total);
        if (threadIdx.x < kStDig) {
            s_off[threadIdx.x] = ex;
            s_base[threadIdx.x] = threadIdx.x < R ? first + before - ex : ~0ull >> 1;   // (no node: out of range)
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kStIPT; ++r) {
            const uint32_t cc = (w[r >> 2] >> (8 * (r & 3))) & 255u;
            if (!cc) continue;
            const uint32_t lp = s_off[cc - 1] + s_whist[warp][cc - 1] + place[r];
            s_idx[lp] = (uint16_t)(warp * (kStIPT * 32) + r * 32 + lane);
            s_dig[lp] = (uint8_t)(cc - 1);
        }
        __syncthreads();
        for (uint32_t q0 = threadIdx.x; q0 < total; q0 += 4 * kStNT) {   // four fetches in flight
            uint32_t j[4];
            uint64_t f[4];
            int4 p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t q = q0 + u * kStNT;
                j[u] = kNone;
                if (q < total) {
                    j[u] = __ldg(a.inv + base + s_idx[q]);
                    f[u] = s_base[s_dig[q]] + q;
                    if (f[u] >= a.n || j[u] >= a.n) { raise(a.err, FP_ERR_CAPACITY, 11); j[u] = kNone; }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j[u] != kNone) p[u] = __ldg(a.pts + j[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j[u] != kNone) {
                    a.fin[f[u]] = p[u];
                    a.fperm[f[u]] = (uint32_t)(base + s_idx[q0 + u * kStNT]);
                }
        }
        __syncthreads();
    }
}

// sorted staging record t = (rank of node X, original index): final position
// first[X] + rank inside X
__global__ void k_stitch_place(const uint32_t* nstaged, const uint64_t* key, const uint32_t* src, int shift,
                               const uint32_t* list, const uint32_t* nlist, const uint32_t* nm, const uint32_t* soff,
                               const uint64_t* first, const int4* pts, const uint32_t* perm, uint64_t n, int4* fin,
                               uint32_t* fperm, uint32_t* err)
{
    const uint32_t S = *nstaged, M = *nm, R = *nlist;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < S; t += gridDim.x * blockDim.x) {
        const uint32_t r = (uint32_t)(key[t] >> shift);
        const uint32_t X = r < R ? list[r] : M;
        const uint32_t j = src[t];
        const uint64_t f = X < M ? first[X] + (t - soff[X]) : n;
        if (f >= n || j >= n) { raise(err, FP_ERR_CAPACITY, 11); continue; }
        fin[f] = __ldg(pts + j);
        fperm[f] = perm[j];
    }
}

cudaError_t launch_node_first(fp_node* nodes, const uint32_t* num_nodes, uint32_t node_cap, const uint32_t* nown,
                              uint64_t* first, uint32_t* nm, uint64_t* tiles64, cudaStream_t st)
{
    const unsigned gM = (node_cap + 255) / 256;
    k_write_nown<<<gM, 256, 0, st>>>(nodes, num_nodes, node_cap, nown);
    k_clamp_copy<<<1, 1, 0, st>>>(num_nodes, node_cap, nm);
    cudaError_t e = scan_exclusive<uint32_t, uint64_t>(nown, first, node_cap, nm, tiles64, (uint64_t*)nullptr,
                                                       (uint64_t*)nullptr, st);
    if (e) return e;
    k_first_out<<<gM, 256, 0, st>>>(nodes, num_nodes, node_cap, first);
    return cudaGetLastError();
}

// Whole-array path: the points and owners in original order, from which one
// stable sort by owner gives the final layout.  For clouds of up to kLayoutWhole
// points, and where a chunk holds more nodes than the segmented scatter takes.
__global__ void __launch_bounds__(256) k_original_order(const uint32_t* gate, const int4* pts, const uint32_t* perm,
                                                        const uint32_t* owner, uint64_t n, int4* opts,
                                                        uint32_t* oowner, uint32_t* err)
{
    if (gate && !*gate) return;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t i = perm[j];
        if (i >= n) { raise(err, FP_ERR_CAPACITY, 11); continue; }
        opts[i] = __ldg(pts + j);
        oowner[i] = owner[j];
    }
}

constexpr uint64_t kMaxNodes = 1ull << 23;   // node_cap of a subsample call

struct SubBufs {
    SortScratch sc;
    uint32_t* hist2;           // histogram of the whole-array sort
    uint32_t *nown, *soff, *cnt;
    uint32_t *srank, *slist;   // rank of a node outside every chunk subtree, and back
    uint64_t* first;
    int4 *o_pt, *t_pt;
    uint32_t *o_own, *o_own2, *t_val, *t_k32;
    uint64_t *s_key, *s_key2, *s_key3;
    uint32_t *s_val, *s_val2, *s_val3;
    SegScratch seg;
};

// chunks of a cloud of n points: at most n, and at most 8^7 count-grid cells
static uint64_t chunk_bound(uint64_t n) { return std::min<uint64_t>(n ? n : 1, 1ull << 21); }

static SubBufs sub_carve(const Workspace& ws, uint64_t n, uint64_t M)
{
    SubBufs B;
    const uint64_t N = n ? n : 1;
    B.sc = take_sort_scratch(ws, N);
    B.hist2 = ws.take<uint32_t>(kSortHistWords);
    B.nown = ws.take<uint32_t>(M); B.first = ws.take<uint64_t>(M + 1);
    B.soff = ws.take<uint32_t>(M + 1); B.cnt = ws.take<uint32_t>(8);
    B.srank = ws.take<uint32_t>(M); B.slist = ws.take<uint32_t>(M);
    // One region serves two sets of per-point buffers that are never live
    // together: the whole-array path's, and the staged records and their sort's.
    const size_t region = ws.used;
    B.o_pt = ws.take<int4>(N); B.o_own = ws.take<uint32_t>(N); B.o_own2 = ws.take<uint32_t>(N);
    B.t_pt = ws.take<int4>(N); B.t_val = ws.take<uint32_t>(N); B.t_k32 = ws.take<uint32_t>(N);
    const size_t end_t = ws.used;
    ws.used = region;
    B.s_key = ws.take<uint64_t>(N); B.s_val = ws.take<uint32_t>(N);
    B.s_key2 = ws.take<uint64_t>(N); B.s_val2 = ws.take<uint32_t>(N);
    B.s_key3 = ws.take<uint64_t>(N); B.s_val3 = ws.take<uint32_t>(N);
    ws.used = std::max(end_t, ws.used);
    B.seg = take_seg_scratch(ws, N, chunk_bound(n), M);
    return B;
}

size_t subsample_ws_bytes(uint64_t n, uint64_t node_cap)
{
    Workspace dry;
    sub_carve(dry, n, std::max<uint64_t>(node_cap, 1));
    return dry.used;
}

cudaError_t launch_subsample(fp_node* nodes, const uint32_t* num_nodes, uint32_t node_cap, const fp_point* sorted,
                             const uint32_t* perm, const uint32_t* owner, uint64_t n, const fp_chunk* chunks,
                             const uint32_t* num_chunks, const uint64_t* offsets, fp_point* final_pts,
                             uint32_t* final_perm, const Workspace& ws, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    if (node_cap > kMaxNodes) return cudaErrorInvalidValue;
    cudaError_t e;
    const uint64_t N = n;
    const uint32_t M = node_cap;
    const SubBufs B = sub_carve(ws, n, M);
    const SortScratch& sc = B.sc;
    uint32_t* nm = B.cnt + 2;   // node count clamped to the capacity
    uint32_t* nstaged = B.cnt + 3;
    uint32_t* nrank = B.cnt + 4;   // nodes outside every chunk subtree
    const unsigned gN = (unsigned)std::min<uint64_t>((N + 255) / 256, (uint64_t)ws.num_sms * 16);

    if (N <= kLayoutCluster) {
        LayoutArgs a{};
        a.nodes = nodes; a.num_nodes = num_nodes; a.node_cap = node_cap; a.n = (uint32_t)N;
        a.original = 1;
        a.pts = reinterpret_cast<const int4*>(sorted); a.perm = perm; a.id = owner;
        a.key[0] = B.o_own; a.key[1] = B.o_own2; a.val[0] = B.t_val; a.val[1] = B.t_k32;
        a.hist = sc.hist; a.part = B.seg.part;
        a.out = reinterpret_cast<int4*>(final_pts); a.out_perm = final_perm; a.err = ws.err;
        KTimerScope kt(FP_KERNEL_OWNER_SCATTER, st);
        return cl_launch(k_layout_cluster, a, st);
    }
    // the sort by owner of the points in original order, gated or not
    auto whole = [&](const uint32_t* gate) -> cudaError_t {
        k_original_order<<<gN, 256, 0, st>>>(gate, reinterpret_cast<const int4*>(sorted), perm, owner, N, B.o_pt,
                                             B.o_own, ws.err);
        SortArgs a{};
        a.b.pt_src = B.o_pt; a.b.pt_tmp = B.t_pt; a.b.pt_dst = reinterpret_cast<int4*>(final_pts);
        a.b.val_src = nullptr; a.b.val_tmp = B.t_val; a.b.val_dst = final_perm;   // the original index
        a.b.k32_src = B.o_own; a.b.k32_tmp = B.t_k32; a.b.k32_dst = B.o_own2;
        a.n = N; a.run_if = gate; a.err = ws.err;
        const SortScratch sc2{B.hist2, {sc.status[0], sc.status[1]}};
        cudaError_t x = sort_plan_weights(sc2, a, B.nown, nullptr, nm, M, true, ws.num_sms, st);
        if (x) return x;
        return sort_run<DIG_K32, true, false, true>(a, sort_passes(count_bits(M)), ws.num_sms, st);
    };

    // 1. stable scatter by owner id, chunk by chunk; owners above the chunk are staged
    int pbits = 1;
    while ((1ull << pbits) < N) ++pbits;   // original indices are below 2^pbits
    SegCall sg{};
    sg.mode = SEG_OWNER;
    sg.nodes = nodes; sg.num_nodes = num_nodes; sg.node_cap = node_cap;
    sg.chunks = chunks; sg.num_chunks = num_chunks; sg.offsets = offsets;
    sg.pt_in = reinterpret_cast<const int4*>(sorted); sg.pt_out = reinterpret_cast<int4*>(final_pts);
    sg.val_in = perm; sg.val_out = final_perm;
    sg.id_in = owner;
    sg.n = N;
    sg.first = B.first; sg.first_stride = 1;
    sg.hist = sc.hist; sg.hist2 = B.hist2;
    sg.nown = B.nown; sg.first_out = B.first; sg.nm = nm;
    sg.st_key = B.s_key; sg.st_src = B.s_val; sg.st_count = nstaged; sg.st_shift = pbits;
    sg.st_rank = B.srank; sg.st_list = B.slist; sg.st_nrank = nrank; sg.st_soff = B.soff;
    const bool marks = N <= kStitchMarked;
    if (marks) {   // where the staged records and their sort would be (it is one or the other)
        sg.st_code = reinterpret_cast<uint8_t*>(B.s_key2);
        sg.st_inv = B.s_val;
    }
    if (N <= kLayoutWhole) {
        KTimerScope kt(FP_KERNEL_OWNER_SCATTER, st);
        if ((e = seg_node_starts(B.seg, sg, ws, st))) return e;
        return whole(nullptr);
    }
    {
        KTimerScope kt(FP_KERNEL_OWNER_SCATTER, st);
        if (marks && (e = cudaMemsetAsync(sg.st_code, 0, N, st))) return e;
        if ((e = seg_scatter(B.seg, sg, ws, st))) return e;
    }
    // 2. the stitch: marked points moved in index order; or staged records sorted by
    // (node, original index), then placed
    {
        KTimerScope kt(FP_KERNEL_STITCH, st);
        if (marks) {
            StitchArgs t{};
            t.nrank = nrank; t.fail = B.seg.cnt + 2; t.code = sg.st_code; t.inv = sg.st_inv;
            t.cnt = reinterpret_cast<uint32_t*>(B.s_key3);
            t.list = B.slist; t.first = B.first; t.pts = reinterpret_cast<const int4*>(sorted);
            t.fin = reinterpret_cast<int4*>(final_pts); t.fperm = final_perm;
            t.n = N; t.ntiles = (uint32_t)((N + kStTile - 1) / kStTile); t.err = ws.err;
            const unsigned gt = (unsigned)std::min<uint64_t>(t.ntiles, (uint64_t)ws.num_sms * 2);
            k_stitch_count<<<(unsigned)std::min<uint64_t>(t.ntiles, (uint64_t)ws.num_sms * 4), kStNT, 0, st>>>(t);
            k_stitch_scan<<<kStitchRanks, kStNT, 0, st>>>(t);
            k_stitch_move<<<gt, kStNT, 0, st>>>(t);
        }
        SortArgs b{};
        b.b.k64_src = B.s_key; b.b.k64_tmp = B.s_key2; b.b.k64_dst = B.s_key3;
        b.b.val_src = B.s_val; b.b.val_tmp = B.s_val2; b.b.val_dst = B.s_val3;
        b.n = N; b.d_n = nstaged; b.err = ws.err;
        if ((e = sort_plan_keys(sc, b, 0, (uint32_t)pbits, nrank, true, ws.num_sms, st))) return e;
        // a node outside every chunk subtree lies above the count grid's cells: at most 8^0 + .. + 8^6 of them
        const uint64_t above = std::min<uint64_t>(M, 299593);
        if ((e = sort_run<DIG_K64, false, true, false>(b, sort_passes(pbits + count_bits(above)), ws.num_sms, st)))
            return e;
        k_stitch_place<<<gN, 256, 0, st>>>(nstaged, B.s_key3, B.s_val3, pbits, B.slist, nrank, nm, B.soff, B.first,
                                           reinterpret_cast<const int4*>(sorted), perm, N,
                                           reinterpret_cast<int4*>(final_pts), final_perm, ws.err);
    }
    // a chunk did not fit: all of it again
    return whole(B.seg.cnt + 2);
}

}  // namespace fp
