// fp_seg.cuh -- single-pass stable scatter of the chunk array by node id, chunk
// by chunk: the leaf grouping of fp_build_chunk_octree and the owner layout of
// fp_subsample (Sec. 4.4: every chunk's local octree is a subtree of the global
// one).
//
// Inside a chunk the distributed order is index order, and every leaf of a
// chunk's points, and every owner below the chunk, lies in the subtree of the
// chunk's node, whose ids are consecutive in preorder.  So the scatter runs
// chunk by chunk with digit = node id - id of the chunk's node: tiles never
// straddle chunks, the decoupled look-back stops at the chunk's first tile, and
// the bucket bases come from the node table -- no histogram or plan passes.
// Points owned by a node above their chunk (the stitch, owner layout only) take
// the last digit and go to a staging area, merged across chunks afterwards.
//
// Two widths: chunks of at most 256 digits run on the 8-bit variant (two CTAs
// per SM), chunks of up to 2048 on the 11-bit one; a chunk with more sets the
// fail word and the caller's whole-array sort runs instead.
#pragma once
#include <cstddef>
#include "fp_sort.cuh"

namespace fp {

static_assert(sizeof(fp_node) == 40 && offsetof(fp_node, leaf_first) % 8 == 0, "fp_node layout");

constexpr int kSegSmallBits = 8;
// earlier tiles' words one look-back round trip reads per digit
constexpr int kSegLookBatch = 8;
constexpr int kSegMaxBits = 11;

struct SegTile {
    uint32_t chunk, index;   // chunk, and tile number inside the chunk
};

struct SegArgs {
    const int4* pt_in;                    // nullable: points not carried
    int4* pt_out;
    const uint32_t* val_in;               // original index of every record
    uint32_t* val_out;                    // nullable
    const uint32_t* id_in;                // node id of every record
    const uint64_t* offsets;              // chunk c = records [offsets[c], offsets[c + 1])
    const uint32_t* seg_lo;               // id of the chunk's node
    const uint32_t* seg_nb;               // digits of the chunk
    const SegTile* tiles;                 // this variant's tiles, each chunk's in order
    const uint32_t* d_ntiles;
    uint64_t ntiles_max;
    const uint64_t* first;                // output start of node id: first[id * first_stride]
    uint32_t first_stride;
    uint32_t* status;                     // [row][1 << MAXB], row = tile start / kSortTile
    uint32_t* counter;
    int stitch;                           // nonzero: the chunk's last digit is the staging digit
    uint64_t* st_key;                     // (st_rank[node] << st_shift) | original index
    const uint32_t* st_rank;              // rank of a node among those outside every chunk subtree (stitch)
    uint32_t* st_src;                     // position in the chunk array
    uint32_t* st_count;
    uint64_t st_cap;
    int st_shift;
    uint64_t n;                           // bound of the output positions

    const uint32_t* d_fail;
    // up to kStitchRanks nodes outside every chunk subtree: staged points marked by
    // original index instead (rank + 1, and the position they are at)
    const uint32_t* st_nrank;
    uint8_t* st_code;
    uint32_t* st_inv;
    uint32_t* err;
};
constexpr uint32_t kStitchRanks = 254;   // (rank + 1 in a byte, for an inconsistent table's ranks too)

template <bool CPT, int MAXB>
struct SegSmem {
    using dig_t = typename std::conditional<(MAXB <= 8), uint8_t, uint16_t>::type;
    static constexpr size_t pt = CPT ? sizeof(int4) * kSortTile : 0;
    static constexpr size_t gbase = sizeof(uint64_t) * (1 << MAXB);
    static constexpr size_t val = sizeof(uint32_t) * kSortTile;
    static constexpr size_t cnt = sizeof(uint32_t) * (1 << MAXB);
    static constexpr size_t off = sizeof(uint32_t) * (1 << MAXB);
    static constexpr size_t pos = sizeof(uint16_t) * kSortTile;   // tile position of a staged record
    static constexpr size_t dig = sizeof(dig_t) * kSortTile;
    static constexpr size_t whist = sizeof(uint16_t) * kSortWarps * (1 << MAXB);
    static constexpr size_t misc = 4 * (1 + kSortWarps + 15);
    static constexpr size_t tiles = 4 * 2;   // current and next tile id
    static constexpr size_t total = pt + gbase + val + cnt + off + pos + dig + whist + misc + tiles;
};

// two CTAs per SM while the shared memory allows it (8-bit digits)
template <bool CPT, int MAXB>
constexpr int seg_ctas() { return SegSmem<CPT, MAXB>::total <= 113 * 1024 ? 2 : 1; }

template <bool CPT, int MAXB>
__global__ void __launch_bounds__(kSortNT, (seg_ctas<CPT, MAXB>())) k_seg_pass(SegArgs a)
{
    if (*a.d_fail) return;
    using SM = SegSmem<CPT, MAXB>;
    using dig_t = typename SM::dig_t;
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char* sp = smem;
    int4* s_pt = reinterpret_cast<int4*>(sp); sp += SM::pt;
    uint64_t* s_gbase = reinterpret_cast<uint64_t*>(sp); sp += SM::gbase;
    uint32_t* s_val = reinterpret_cast<uint32_t*>(sp); sp += SM::val;
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(sp); sp += SM::cnt;
    uint32_t* s_off = reinterpret_cast<uint32_t*>(sp); sp += SM::off;
    uint16_t* s_pos = reinterpret_cast<uint16_t*>(sp); sp += SM::pos;
    dig_t* s_dig = reinterpret_cast<dig_t*>(sp); sp += SM::dig;
    uint16_t* s_whist = reinterpret_cast<uint16_t*>(sp); sp += SM::whist;
    uint32_t* s_misc = reinterpret_cast<uint32_t*>(sp); sp += SM::misc;
    uint32_t* s_tile = reinterpret_cast<uint32_t*>(sp);

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t ntiles = min((uint64_t)*a.d_ntiles, a.ntiles_max);
    constexpr int kStride = 1 << MAXB;
    const bool marked = a.stitch && a.st_code && *a.st_nrank <= kStitchRanks;

    // the next tile is claimed while the current one is worked on (tiles only
    // wait on earlier tiles of their chunk, so a reserved tile cannot deadlock)
    if (threadIdx.x == 0) s_tile[0] = atomicAdd(a.counter, 1u);
    for (int it = 0;; ++it) {
        __syncthreads();
        const uint64_t tile = s_tile[it & 1];
        if (tile >= ntiles) break;
        if (threadIdx.x == 0) s_tile[(it + 1) & 1] = atomicAdd(a.counter, 1u);
        const SegTile td = a.tiles[tile];
        const uint32_t lo = a.seg_lo[td.chunk];
        const int nb = (int)a.seg_nb[td.chunk];   // 1 .. 1 << MAXB (checked by the setup)
        const uint64_t cend = a.offsets[td.chunk + 1];
        const uint64_t base = a.offsets[td.chunk] + (uint64_t)td.index * kSortTile;
        const int tn = (int)(cend - base < (uint64_t)kSortTile ? cend - base : (uint64_t)kSortTile);
        const bool last = base + (uint64_t)tn >= cend;   // no later tile of the chunk reads this one
        const uint64_t row = base / kSortTile;            // tiles that are not last are full: rows are distinct
        const int sdig = a.stitch ? nb - 1 : nb;          // staging digit (nb: none)
        for (int q = threadIdx.x; q < kSortWarps * nb; q += kSortNT) s_whist[q] = 0;
        __syncthreads();
        uint16_t* wh = s_whist + warp * nb;

        // ---- digits (all loads issued first), then in-warp stable ranks
        uint32_t dg[kSortIPT];
#pragma unroll
        for (int r = 0; r < kSortIPT; ++r) {
            const int p = warp * (kSortIPT * 32) + r * 32 + lane;
            dg[r] = p < tn ? a.id_in[base + p] - lo : 0xFFFFFFFFu;
        }
        uint32_t pack[kSortIPT];
#pragma unroll
        for (int r = 0; r < kSortIPT; ++r) {
            const int p = warp * (kSortIPT * 32) + r * 32 + lane;
            uint32_t d = 0xFFFFu;
            if (p < tn) {
                d = dg[r];
                if (d >= (uint32_t)sdig) {
                    if (!a.stitch) raise(a.err, FP_ERR_CAPACITY, 13);   // a leaf outside the chunk's subtree
                    d = (uint32_t)(nb - 1);
                }
            }
            uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
            int leader = __ffs(peers) - 1;
            uint32_t old = 0;
            if (lane == leader && d != 0xFFFFu) {
                old = wh[d];
                wh[d] = (uint16_t)(old + __popc(peers));
            }
            old = __shfl_sync(0xFFFFFFFFu, old, leader);
            pack[r] = d | ((old + __popc(peers & lanemask_lt())) << 16);
            __syncwarp();
        }
        __syncthreads();
        // ---- per-digit totals, per-warp exclusive prefixes; publish aggregates
        for (int d = threadIdx.x; d < nb; d += kSortNT) {
            uint32_t s = 0;
#pragma unroll
            for (int w = 0; w < kSortWarps; ++w) {
                uint32_t v = s_whist[w * nb + d];
                s_whist[w * nb + d] = (uint16_t)s;
                s += v;
            }
            s_cnt[d] = s;
            if (!last && d != sdig) a.status[row * kStride + d] = (td.index == 0 ? kStFlagInc : kStFlagAgg) | s;
        }
        __syncthreads();
        {
            const int per = (nb + kSortNT - 1) / kSortNT;
            const int d0 = threadIdx.x * per;
            uint32_t s = 0;
            for (int q = 0; q < per; ++q)
                if (d0 + q < nb) s += s_cnt[d0 + q];
            uint32_t tot;
            uint32_t ex = block_exclusive_scan<kSortNT, uint32_t>(s, s_misc + 1, tot);
            for (int q = 0; q < per; ++q)
                if (d0 + q < nb) { s_off[d0 + q] = ex; ex += s_cnt[d0 + q]; }
        }
        __syncthreads();
        // ---- stage the records in digit order
#pragma unroll
        for (int r = 0; r < kSortIPT; ++r) {
            const int p = warp * (kSortIPT * 32) + r * 32 + lane;
            if (p < tn) {
                const uint32_t d = pack[r] & 0xFFFFu;
                const uint32_t lp = s_off[d] + s_whist[warp * nb + d] + (pack[r] >> 16);
                const uint64_t i = base + p;
                if (CPT) s_pt[lp] = __ldg(a.pt_in + i);
                s_val[lp] = a.val_in[i];
                s_pos[lp] = (uint16_t)p;
                s_dig[lp] = (dig_t)d;
            }
        }
        // ---- look-back over the chunk's earlier tiles; staging slots for the stitch digit
        for (int d = threadIdx.x; d < nb; d += kSortNT) {
            if (d == sdig) {
                const uint32_t k = s_cnt[d];
                const uint32_t at = k && !marked ? atomicAdd(a.st_count, k) : 0u;
                s_gbase[d] = (uint64_t)at - s_off[d];
                continue;
            }
            uint32_t excl = 0;
            if (td.index > 0) {
                auto word = [&](int64_t t) { return &a.status[(uint64_t)t * kStride + d]; };
                excl = look_back<decltype(word), kSegLookBatch>(word, (int64_t)row - 1,
                                                                (int64_t)row - (int64_t)td.index, a.err);
                if (!last) atomicExch(&a.status[row * kStride + d], kStFlagInc | (excl + s_cnt[d]));
            }
            s_gbase[d] = a.first[(uint64_t)(lo + d) * a.first_stride] + excl - s_off[d];
        }
        __syncthreads();
        // ---- coalesced writes of each digit run
        for (int q = threadIdx.x; q < tn; q += kSortNT) {
            const int d = s_dig[q];
            const uint64_t o = s_gbase[d] + q;
            if (d == sdig) {
                const uint64_t src = base + s_pos[q];
                const uint32_t id = a.id_in[src];
                if (marked) {
                    const uint32_t i = s_val[q];
                    if (i >= a.n) { raise(a.err, FP_ERR_CAPACITY, 14); continue; }
                    a.st_code[i] = (uint8_t)(a.st_rank[id] + 1);
                    a.st_inv[i] = (uint32_t)src;
                    continue;
                }
                if (o >= a.st_cap) { raise(a.err, FP_ERR_CAPACITY, 14); continue; }
                a.st_key[o] = ((uint64_t)a.st_rank[id] << a.st_shift) | s_val[q];
                a.st_src[o] = (uint32_t)src;
            } else {
                if (o >= a.n) { raise(a.err, FP_ERR_CAPACITY, 15); continue; }   // inconsistent node table
                if (CPT) a.pt_out[o] = s_pt[q];
                if (a.val_out) a.val_out[o] = s_val[q];
            }
        }
        __syncthreads();
    }
}

// ---- host side
struct SegScratch {
    uint32_t* lo;          // [kmax]
    uint32_t* nb;          // [kmax]
    SegTile* tiles[2];     // [tiles_max] per variant
    uint32_t* status[2];   // [rows][256] and [rows][2048]
    uint32_t* cnt;         // [0..1] tiles per variant, [2] fail, [3..4] tile counters
    uint8_t* inside;       // [node_cap] owner layout: node lies in a chunk's subtree
    uint64_t* part;        // cluster scan scratch
    uint64_t kmax, tiles_max, rows, node_cap;
};
SegScratch take_seg_scratch(const Workspace& ws, uint64_t n, uint64_t kmax, uint64_t node_cap);

enum SegMode { SEG_LEAF = 0, SEG_OWNER = 1 };

struct SegCall {
    SegMode mode;
    fp_node* nodes; const uint32_t* num_nodes; uint32_t node_cap;
    const fp_chunk* chunks; const uint32_t* num_chunks; const uint64_t* offsets;
    const int4* pt_in; int4* pt_out;
    const uint32_t* val_in; uint32_t* val_out;
    const uint32_t* id_in;
    uint64_t n;
    const uint64_t* first; uint32_t first_stride;
    uint32_t *hist, *hist2;   // sort histograms to clear (kSortHistWords each; hist2 nullable)
    // owner layout: owned counts and starts of the nodes (written, also into the node records)
    uint32_t* nown; uint64_t* first_out; uint32_t* nm;
    // owner layout: staging, keyed by rank among the nodes outside every chunk
    // subtree (in node order, so the sorted order is that of node ids):
    // st_rank[node] (node_cap), st_list[rank] = node, *st_nrank = their number,
    // st_soff[node] = staged points of the nodes before it
    uint64_t* st_key; uint32_t* st_src; uint32_t* st_count; int st_shift;
    uint32_t *st_rank, *st_list, *st_nrank, *st_soff;
    uint8_t* st_code;         // n bytes, zero, and n words: marks of up to kStitchRanks nodes' points instead
    uint32_t* st_inv;
};

// distribution of up to kDistCluster points in one launch (tmp: n words each;
// hist: kClCtas * 256 words).  At 32,768 points 27 us and 45 us by the sweep with 37
// chunks (one pass), 38 and 51 us with 1268 (two); its time grows with the points,
// 1 us per 2000, and would meet the sweep's near 65,000.
constexpr uint64_t kDistCluster = 1ull << 15;
cudaError_t dist_cluster(const int4* pts, uint64_t n, const fp_cube* cube, int g, const uint32_t* lut,
                         const uint64_t* offsets, const uint32_t* num_chunks, int4* out, uint32_t* perm,
                         const uint32_t* cells, uint32_t* const tmp[4], uint32_t* hist, uint32_t* err, cudaStream_t st);

// Distribution of n points into up to 4096 chunks by the counting pass and the sweep
// (fp_seg.cu); the points' cells given or computed.
// chunk_tmp: n chunk ids, 16-byte aligned.  *run_sort is set to 1, and hist
// (kSortHistWords) cleared, when there are more chunks (the radix passes run
// instead), else 0.
size_t dist_wide_bytes(uint64_t n);
cudaError_t dist_wide(const int4* pts, uint64_t n, const fp_cube* cube, int g, const uint32_t* lut,
                      const uint64_t* offsets, const uint32_t* num_chunks, int4* out, uint32_t* perm,
                      uint32_t* run_sort, uint32_t* hist, const Workspace& ws, cudaStream_t st, const uint32_t* cells,
                      uint16_t* chunk_tmp);

// The plan (k_seg_plan) and both pass variants.
// Afterwards cnt[2] != 0 means a chunk did not fit: the caller's whole-array
// path, gated on it, must run.
cudaError_t seg_scatter(const SegScratch& sc, const SegCall& call, const Workspace& ws, cudaStream_t st);

// Only the plan's first step (owner layout): owned counts and first points of the
// nodes, the sorts' histograms cleared.
cudaError_t seg_node_starts(const SegScratch& sc, const SegCall& call, const Workspace& ws, cudaStream_t st);

}  // namespace fp
