// fp_render.cu -- the renderer's side of the octree, headless (Sec. 4.5):
// which nodes a camera draws, and the points of those nodes rasterised into a
// device framebuffer.
//
// Selection: a node is drawn when its box is not outside the view frustum and
// every ancestor was refined; a node is refined when it is drawn, is not a
// leaf, and its box covers more than min_node_px pixels on screen (a box that
// reaches behind the camera plane counts as infinitely large).  So each drawn
// node contributes its own level-of-detail sample, and finer nodes are drawn
// only where the coarser ones are large on screen.  In preorder a node's
// subtree is the range [i, i + n_desc]: a node that is not refined excludes
// that range (difference array + scan), then the drawn nodes are compacted.
// One cooperative launch over all of it, whose blocks own consecutive nodes: as
// 14 launches (flags, mark, write and three scans of three) a selection among
// 5,628 nodes took about 40 us of a frame, 17 us now.
//
// Rasterisation: each point of a drawn node is projected by the 4x4 matrix;
// the nearest one per pixel wins through a 64-bit atomicMin on
// (depth bits << 32 | colour), depth = clip z / w in [0, 1].  One cooperative
// launch clears the framebuffer, finds the drawn nodes' point starts and draws.
//
// All floating point is fp32 with the fused multiply-adds, divisions and
// roundings spelled out, so that the CPU restatement reproduces every
// projection, pixel and visibility decision bit for bit.
#include "fp_cluster.cuh"
#include "fp_internal.cuh"

namespace fp {

namespace {

struct CamDev {
    float m[16];
    float W, H, minpx;
    uint32_t w, h;
};

CamDev cam_dev(const fp_camera& c)
{
    CamDev d;
    for (int i = 0; i < 16; ++i) d.m[i] = c.m[i];
    d.W = (float)c.width;
    d.H = (float)c.height;
    d.minpx = c.min_node_px;
    d.w = c.width;
    d.h = c.height;
    return d;
}

struct Clip {
    float x, y, z, w;
};

// clip = m * (x, y, z, 1), each row as fma(m0, x, fma(m1, y, fma(m2, z, m3)))
FP_DEV Clip clip_of(const CamDev& c, float x, float y, float z)
{
    Clip r;
    r.x = __fmaf_rn(c.m[0], x, __fmaf_rn(c.m[1], y, __fmaf_rn(c.m[2], z, c.m[3])));
    r.y = __fmaf_rn(c.m[4], x, __fmaf_rn(c.m[5], y, __fmaf_rn(c.m[6], z, c.m[7])));
    r.z = __fmaf_rn(c.m[8], x, __fmaf_rn(c.m[9], y, __fmaf_rn(c.m[10], z, c.m[11])));
    r.w = __fmaf_rn(c.m[12], x, __fmaf_rn(c.m[13], y, __fmaf_rn(c.m[14], z, c.m[15])));
    return r;
}

// screen x (or y) of a normalised device coordinate: fma(n, 0.5, 0.5) * W
FP_DEV float screen(float n, float W) { return __fmul_rn(__fmaf_rn(n, 0.5f, 0.5f), W); }

// integer bounds of the points of node (level, key): lo_a = o_a + ceil(c S / 2^L),
// hi_a = o_a + ceil((c + 1) S / 2^L) - 1, exact in 64 bits (c S < 2^53)
FP_DEV void node_box(const fp_cube& cb, int L, uint64_t key, float lo[3], float hi[3])
{
    uint64_t c[3] = {0, 0, 0};
    for (int b = 0; b < L; ++b) {
        c[0] |= ((key >> (3 * b + 2)) & 1ull) << b;
        c[1] |= ((key >> (3 * b + 1)) & 1ull) << b;
        c[2] |= ((key >> (3 * b)) & 1ull) << b;
    }
    const uint64_t r = (1ull << L) - 1;
    for (int a = 0; a < 3; ++a) {
        const int64_t l = (int64_t)cb.o[a] + (int64_t)((c[a] * cb.S + r) >> L);
        const int64_t h = (int64_t)cb.o[a] + (int64_t)(((c[a] + 1) * cb.S + r) >> L) - 1;
        lo[a] = __ll2float_rn(l);
        hi[a] = __ll2float_rn(h);
    }
}

constexpr int kRenderNT = 256;
constexpr uint32_t kRenderBlocks = 640;   // most blocks of a launch
static_assert(3 * kRenderBlocks <= kScanMaxTiles, "the blocks' words fit the scratch");

// sum over the blocks before this one, and over all, of part[block] (any
// block's threads; part published before the last grid barrier)
struct BlockPrefix {
    uint64_t before, all;
};
FP_DEV BlockPrefix block_prefix(const uint64_t* part, uint64_t* smem /* 2 */)
{
    if (threadIdx.x < 2) smem[threadIdx.x] = 0;
    __syncthreads();
    uint64_t before = 0, all = 0;
    for (uint32_t b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
        const uint64_t v = *(const volatile uint64_t*)(part + b);
        if (b < blockIdx.x) before += v;
        all += v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
        all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd((unsigned long long*)&smem[0], (unsigned long long)before);
        atomicAdd((unsigned long long*)&smem[1], (unsigned long long)all);
    }
    __syncthreads();
    const BlockPrefix r{smem[0], smem[1]};
    __syncthreads();
    return r;
}

struct SelectArgs {
    const fp_node* nodes;
    const uint32_t* num_nodes;
    uint32_t cap;
    const fp_cube* cube;
    CamDev cam;
    uint8_t* vis;        // cap
    uint32_t* diff;      // cap + 1
    uint64_t* part;      // three words per block
    uint32_t* ids;
    uint32_t* num_sel;
    uint64_t* num_points;
    uint32_t* bar;       // 0
    uint32_t* err;
};

// bit 0: node i is not outside the frustum; bit 1: its subtree is not drawn
FP_DEV uint32_t render_flags(const SelectArgs& a, const fp_cube& cb, uint32_t i, fp_node& nd)
{
    const CamDev& cam = a.cam;
    nd = a.nodes[i];
    float lo[3], hi[3];
    node_box(cb, nd.level, nd.key, lo, hi);
    bool all_l = true, all_r = true, all_b = true, all_t = true, all_n = true, all_f = true, behind = false;
    bool any = false;
    float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
    for (int k = 0; k < 8; ++k) {
        const Clip c = clip_of(cam, (k & 4) ? hi[0] : lo[0], (k & 2) ? hi[1] : lo[1], (k & 1) ? hi[2] : lo[2]);
        all_l &= c.x < -c.w;
        all_r &= c.x > c.w;
        all_b &= c.y < -c.w;
        all_t &= c.y > c.w;
        all_n &= c.z < 0.f;
        all_f &= c.z > c.w;
        if (c.w <= 0.f) {
            behind = true;
        } else {
            const float sx = screen(__fdiv_rn(c.x, c.w), cam.W), sy = screen(__fdiv_rn(c.y, c.w), cam.H);
            if (!any || sx < x0) x0 = sx;
            if (!any || sx > x1) x1 = sx;
            if (!any || sy < y0) y0 = sy;
            if (!any || sy > y1) y1 = sy;
            any = true;
        }
    }
    const bool visible = !(all_l || all_r || all_b || all_t || all_n || all_f);
    const float ex = __fsub_rn(x1, x0), ey = __fsub_rn(y1, y0);
    const float size = ex > ey ? ex : ey;
    const bool refine = visible && !nd.is_leaf && (behind || size > cam.minpx);
    return (visible ? 1u : 0u) | (refine ? 0u : 2u);
}

// Four grid barriers: differences cleared | flags and differences | every block's
// sum of them | every block's drawn nodes and points | ids.
__global__ void __launch_bounds__(kRenderNT, 4) k_select(SelectArgs a)
{
    __shared__ uint32_t s_warp[kRenderNT / 32];
    __shared__ uint64_t s_pre[2];
    const uint32_t M = min(*a.num_nodes, a.cap), tid = threadIdx.x;
    const uint32_t per = (M + gridDim.x - 1) / gridDim.x;
    const uint32_t lo = min((uint64_t)M, (uint64_t)blockIdx.x * per), hi = min((uint64_t)M, (uint64_t)lo + per);
    const fp_cube cb = *a.cube;
    for (uint32_t i = lo + tid; i < hi; i += kRenderNT) a.diff[i] = 0;
    if (blockIdx.x == 0 && tid == 0) a.diff[M] = 0;
    if (!grid_barrier(a.bar, 1, a.err)) return;
    for (uint32_t i = lo + tid; i < hi; i += kRenderNT) {
        fp_node nd;
        const uint32_t f = render_flags(a, cb, i, nd);
        a.vis[i] = (uint8_t)(f & 1u);
        if ((f & 2u) && nd.n_desc && nd.n_desc < M - i) {   // the subtree below is not drawn
            atomicAdd(&a.diff[i + 1], 1u);
            atomicAdd(&a.diff[i + nd.n_desc + 1], 0xFFFFFFFFu);
        }
    }
    if (!grid_barrier(a.bar, 2, a.err)) return;
    uint32_t sum = 0, total;
    for (uint32_t i = lo + tid; i < hi; i += kRenderNT) sum += ld_volatile(a.diff + i);
    block_exclusive_scan<kRenderNT, uint32_t>(sum, s_warp, total);
    if (tid == 0) a.part[blockIdx.x] = total;
    if (!grid_barrier(a.bar, 3, a.err)) return;
    uint32_t run = (uint32_t)block_prefix(a.part, s_pre).before;   // (differences are taken modulo 2^32)
    uint64_t points = 0;
    uint32_t drawn = 0;
    for (uint32_t i0 = lo; i0 < hi; i0 += kRenderNT) {
        const uint32_t i = i0 + tid;
        const uint32_t d = i < hi ? ld_volatile(a.diff + i) : 0u;
        const uint32_t in = run + block_exclusive_scan<kRenderNT, uint32_t>(d, s_warp, total) + d;
        run += total;
        if (i < hi) {
            const bool sel = a.vis[i] && in == 0;
            a.vis[i] = sel ? 1 : 0;   // (read back by this thread only)
            if (sel) { ++drawn; points += a.nodes[i].n_own; }
        }
    }
    for (int o = 16; o > 0; o >>= 1) points += __shfl_xor_sync(0xFFFFFFFFu, points, o);
    drawn = __reduce_add_sync(0xFFFFFFFFu, drawn);
    if (tid < 2) s_pre[tid] = 0;
    __syncthreads();
    if ((tid & 31) == 0) {
        atomicAdd((unsigned long long*)&s_pre[0], (unsigned long long)drawn);
        atomicAdd((unsigned long long*)&s_pre[1], (unsigned long long)points);
    }
    __syncthreads();
    if (tid == 0) {
        a.part[kRenderBlocks + blockIdx.x] = s_pre[0];
        a.part[2 * kRenderBlocks + blockIdx.x] = s_pre[1];
    }
    if (!grid_barrier(a.bar, 4, a.err)) return;
    const BlockPrefix pre = block_prefix(a.part + kRenderBlocks, s_pre);
    if (blockIdx.x == 0) {
        const uint64_t all = block_prefix(a.part + 2 * kRenderBlocks, s_pre).all;
        if (tid == 0) { *a.num_sel = (uint32_t)pre.all; *a.num_points = all; }
    }
    uint32_t at = (uint32_t)pre.before;
    for (uint32_t i0 = lo; i0 < hi; i0 += kRenderNT) {
        const uint32_t i = i0 + tid, sel = i < hi ? a.vis[i] : 0u;
        const uint32_t q = at + block_exclusive_scan<kRenderNT, uint32_t>(sel, s_warp, total);
        at += total;
        if (sel) a.ids[q] = i;
    }
}

struct RasterArgs {
    const fp_node* nodes;
    const uint32_t *ids, *num_sel;
    uint32_t cap;
    uint64_t* pstart;    // cap: first drawn point of every drawn node
    uint64_t* pshift;    // cap: its place among the points, less pstart
    uint64_t* part;      // one word per block
    const int4* fin;
    uint64_t n;
    CamDev cam;
    unsigned long long* fb;
    uint32_t* bar;       // 0
    uint32_t* err;
};

// Each block draws a run of consecutive points of the drawn nodes, its warps 128
// of them in turn: four loads and four projections a lane in flight.  A warp
// follows the node it is in and holds the starts of the next 32 and where their
// points are, one a lane; 128 points that span more nodes are searched among those
// nodes, and a node further ahead is found by 32 probes at a time.  (Nodes of a few
// points: with a search of all drawn nodes a chunk, and of each point where they are
// many, 3 * 10^6 points of 176,581 nodes took 142 us, 86 now.)
//
// A node's points fall on few pixels, in random order, about 30 of them on each:
// a direct-mapped table in shared memory (32 x 32 pixels, pixel and depth in one
// word) remembers depths drawn before, and a point behind its entry is done.  An
// entry is a depth that some point of the block offers to the pixel, so what is
// skipped could not have won; an entry lost to another pixel or to a race costs a
// read of the framebuffer.
//
// Bound by instructions (about 140 a point) and latency at 32 warps an SM.  A frame
// of 30M points, 26.6M drawn, selection included: one point in flight a lane, each
// searched among all drawn nodes, 385 us; runs and four in flight 278 us; with the
// table 203 us; the next points on their way to L2 196, also across nodes 188 us.  Two points a lane and
// five blocks an SM drew in 200 us instead of 182, three and five in 208.
constexpr int kRasterPer = 4, kRasterCtas = 4;
constexpr int kRasterTabX = 32, kRasterTabY = 32;   // powers of two
constexpr int kRasterTab = kRasterTabX * kRasterTabY;

__global__ void __launch_bounds__(kRenderNT, kRasterCtas) k_raster(RasterArgs a)
{
    __shared__ uint64_t s_warp[kRenderNT / 32], s_pre[2];
    __shared__ unsigned long long s_tab[kRasterTab];   // pixel << 32 | depth
    const uint32_t S = min(*a.num_sel, a.cap), tid = threadIdx.x;
    for (int q = tid; q < kRasterTab; q += kRenderNT) s_tab[q] = ~0ull;
    const int lane = tid & 31;
    const CamDev& cam = a.cam;
    {   // the framebuffer cleared (16 bytes a store; its last pixel by itself where the count is odd)
        const uint64_t px = (uint64_t)cam.w * cam.h, t = (uint64_t)blockIdx.x * kRenderNT + tid;
        const bool aligned = (reinterpret_cast<uintptr_t>(a.fb) & 15u) == 0;
        const uint64_t pairs = aligned ? px / 2 : 0, stride = (uint64_t)gridDim.x * kRenderNT;
        for (uint64_t q = t; q < pairs; q += stride)
            reinterpret_cast<ulonglong2*>(a.fb)[q] = make_ulonglong2(~0ull, ~0ull);
        for (uint64_t q = 2 * pairs + t; q < px; q += stride) a.fb[q] = ~0ull;
    }
    const uint32_t per = (S + gridDim.x - 1) / gridDim.x;
    const uint32_t lo = min((uint64_t)S, (uint64_t)blockIdx.x * per), hi = min((uint64_t)S, (uint64_t)lo + per);
    uint64_t sum = 0, total;
    for (uint32_t k = lo + tid; k < hi; k += kRenderNT) sum += a.nodes[a.ids[k]].n_own;
    block_exclusive_scan<kRenderNT, uint64_t>(sum, s_warp, total);
    if (tid == 0) a.part[blockIdx.x] = total;
    if (!grid_barrier(a.bar, 1, a.err)) return;
    const BlockPrefix pre = block_prefix(a.part, s_pre);
    uint64_t run = pre.before;
    for (uint32_t k0 = lo; k0 < hi; k0 += kRenderNT) {
        const uint32_t k = k0 + tid;
        const fp_node* nd = k < hi ? a.nodes + a.ids[k] : nullptr;
        const uint64_t v = nd ? nd->n_own : 0, first = nd ? nd->first : 0;
        const uint64_t ex = run + block_exclusive_scan<kRenderNT, uint64_t>(v, s_warp, total);
        run += total;
        if (k < hi) {
            a.pstart[k] = ex;
            a.pshift[k] = first - ex;
        }
    }
    if (!grid_barrier(a.bar, 2, a.err)) return;

    const uint64_t P = pre.all;
    constexpr uint32_t kChunk = 32 * kRasterPer, kStep = kChunk * (kRenderNT / 32);
    const uint64_t len = (P + (uint64_t)gridDim.x * kStep - 1) / ((uint64_t)gridDim.x * kStep) * kStep;
    const uint64_t p1 = min(P, ((uint64_t)blockIdx.x + 1) * len);
    uint64_t c = (uint64_t)blockIdx.x * len + (tid >> 5) * kChunk;
    if (c >= p1) return;
    const uint64_t *ps = a.pstart, *psh = a.pshift;
    // last start <= p (nodes without points share starts), from x on, by the whole warp:
    // two reads a lane where it is among the next 1024 nodes, then 32 probes of the rest
    // at a time
    auto node_ahead = [&](uint64_t p, uint32_t x) {
        uint32_t y = min((uint64_t)S, (uint64_t)x + 1024);
        while (x < y) {
            const uint32_t step = (y - x + 31) >> 5, i = x + lane * step;
            const uint32_t n = __popc(__ballot_sync(0xFFFFFFFFu, i < y && __ldcg(ps + i) <= p));
            if (!n) break;
            const uint32_t lo = x + (n - 1) * step, hi = min(y, lo + step);
            y = hi == y ? (y < S ? S : y) : hi;   // (past the window: the rest)
            x = lo + 1;
        }
        return x - 1;
    };
    uint32_t k = node_ahead(c, 0);
    uint64_t shift, nxt, nsh;   // of node k; start and shift of node k + 1 + lane
    auto enter = [&]() {
        const bool in = k + 1 + lane < S;
        shift = __ldcg(psh + k);
        nxt = in ? __ldcg(ps + k + 1 + lane) : ~0ull;
        nsh = in ? __ldcg(psh + k + 1 + lane) : 0ull;
    };
    enter();
    for (; c < p1; c += kStep) {
        if (const int past = __popc(__ballot_sync(0xFFFFFFFFu, nxt <= c))) {   // this chunk starts in a later node
            k = past < 32 ? k + past : node_ahead(c, k + 1);
            enter();
        }
        const uint64_t ce = min(p1, c + kChunk);
        // the next chunk's lines on their way to L2 (8 points a line; drawn nodes mostly follow one another)
        if (lane < kChunk / 8 && c + shift + kStep + 8 * lane < a.n) prefetch_l2(a.fin + c + shift + kStep + 8 * lane);
        int4 q[kRasterPer];
        uint32_t ok = 0;   // bit r: point r is there
        if (__shfl_sync(0xFFFFFFFFu, nxt, 0) >= ce) {   // all in one node
            const uint64_t at = c + shift;
            const uint32_t left = at < a.n ? (uint32_t)min(ce - c, a.n - at) : 0u;   // (a node table of another
            const int4* src = a.fin + at;                                            // point array may pass n)
#pragma unroll
            for (int r = 0; r < kRasterPer; ++r) {
                q[r] = make_int4(0, 0, 0, 0);
                if (r * 32 + lane < left) {
                    q[r] = __ldg(src + r * 32 + lane);
                    ok |= 1u << r;
                }
            }
        } else {
            const bool held = __shfl_sync(0xFFFFFFFFu, nxt, 31) >= ce;   // the 32 starts reach beyond the chunk
            uint64_t at[kRasterPer];
            if (held) {
#pragma unroll
                for (int r = 0; r < kRasterPer; ++r) {
                    const uint64_t p = c + r * 32 + lane;
                    int o = 0;   // nodes of the 32 that start at or before p
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1)
                        if (__shfl_sync(0xFFFFFFFFu, nxt, (o + d - 1) & 31) <= p) o += d;
                    const uint64_t f = __shfl_sync(0xFFFFFFFFu, nsh, (o + 31) & 31);
                    at[r] = p + (o ? f : shift);
                }
            } else {   // a search each, all in step, among the nodes of the chunk
                const uint32_t last = node_ahead(ce - 1, k + 1);
                uint32_t x[kRasterPer];
#pragma unroll
                for (int r = 0; r < kRasterPer; ++r) x[r] = k;
                for (uint32_t bit = 0x80000000u >> __clz(last - k); bit; bit >>= 1)
#pragma unroll
                    for (int r = 0; r < kRasterPer; ++r)
                        if (x[r] + bit <= last && __ldcg(ps + x[r] + bit) <= c + r * 32 + lane) x[r] += bit;
#pragma unroll
                for (int r = 0; r < kRasterPer; ++r) at[r] = c + r * 32 + lane + __ldcg(psh + x[r]);
            }
#pragma unroll
            for (int r = 0; r < kRasterPer; ++r) {
                q[r] = make_int4(0, 0, 0, 0);
                if (c + r * 32 + lane < ce && at[r] < a.n) {
                    q[r] = __ldg(a.fin + at[r]);
                    ok |= 1u << r;
                }
            }
        }
        uint32_t px[kRasterPer];
        unsigned long long v[kRasterPer];
#pragma unroll
        for (int r = 0; r < kRasterPer; ++r) {
            px[r] = kNone;
            const Clip t = clip_of(cam, __int2float_rn(q[r].x), __int2float_rn(q[r].y), __int2float_rn(q[r].z));
            if (!((ok >> r) & 1u) || !(t.w > 0.f) || fabsf(t.x) > t.w || fabsf(t.y) > t.w || t.z < 0.f || t.z > t.w)
                continue;
            const float sx = screen(__fdiv_rn(t.x, t.w), cam.W), sy = screen(__fdiv_rn(t.y, t.w), cam.H);
            const uint32_t x = min(__float2uint_rd(sx), cam.w - 1), y = min(__float2uint_rd(sy), cam.h - 1);
            const float depth = __fadd_rn(__fdiv_rn(t.z, t.w), 0.f);   // -0 -> +0
            v[r] = ((unsigned long long)__float_as_uint(depth) << 32) | (uint32_t)q[r].w;
            px[r] = y * cam.w + x;
            unsigned long long* e = &s_tab[(y & (kRasterTabY - 1u)) * kRasterTabX + (x & (kRasterTabX - 1u))];
            const unsigned long long had = *(volatile unsigned long long*)e;
            const bool same = (uint32_t)(had >> 32) == px[r];
            const uint32_t d = (uint32_t)(v[r] >> 32);
            if (same && d > (uint32_t)had) px[r] = kNone;
            else if (!same || d < (uint32_t)had) *(volatile unsigned long long*)e = ((unsigned long long)px[r] << 32) | d;
        }
        unsigned long long old[kRasterPer];
#pragma unroll
        for (int r = 0; r < kRasterPer; ++r) old[r] = px[r] != kNone ? __ldcg(a.fb + px[r]) : 0;
#pragma unroll
        for (int r = 0; r < kRasterPer; ++r)   // a pixel's value only falls: skip the hopeless
            if (px[r] != kNone && v[r] < old[r]) atomicMin(a.fb + px[r], v[r]);
    }
}

}  // namespace

struct RenderBufs {
    uint8_t* vis;
    uint32_t *diff, *num;
    uint64_t *pstart, *pshift, *tiles64;
};

static RenderBufs render_carve(const Workspace& ws, uint32_t cap)
{
    RenderBufs B;
    const uint64_t M = cap ? cap : 1;
    B.vis = ws.take<uint8_t>(M);
    B.diff = ws.take<uint32_t>(M + 1);
    B.num = ws.take<uint32_t>(2);
    B.pstart = ws.take<uint64_t>(M);
    B.pshift = ws.take<uint64_t>(M);
    B.tiles64 = ws.take<uint64_t>(kScanMaxTiles);
    return B;
}

size_t render_ws_bytes(uint32_t cap)
{
    Workspace dry;
    render_carve(dry, cap);
    return dry.used;
}

cudaError_t launch_select_nodes(const fp_node* nodes, const uint32_t* num_nodes, uint32_t cap, const fp_cube* cube,
                                const fp_camera& cam, uint32_t* ids, uint32_t* num_sel, uint64_t* num_points,
                                const Workspace& ws, cudaStream_t st)
{
    const RenderBufs B = render_carve(ws, cap);
    cudaError_t e;
    if ((e = cudaMemsetAsync(B.num, 0, 2 * sizeof(uint32_t), st))) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_select, kRenderNT, 0))) return e;
    SelectArgs a{};
    a.nodes = nodes; a.num_nodes = num_nodes; a.cap = cap; a.cube = cube; a.cam = cam_dev(cam);
    a.vis = B.vis; a.diff = B.diff; a.part = B.tiles64;
    a.ids = ids; a.num_sel = num_sel; a.num_points = num_points; a.bar = B.num; a.err = ws.err;
    const uint64_t most = std::min<uint64_t>(kRenderBlocks, (uint64_t)ws.num_sms * std::min(std::max(per_sm, 1), 4));
    const unsigned grid = (unsigned)std::min<uint64_t>(((uint64_t)cap + kRenderNT - 1) / kRenderNT + 1, most);
    return coop_launch(k_select, grid, kRenderNT, 0, st, a);
}

cudaError_t launch_rasterize(const fp_node* nodes, const uint32_t* ids, const uint32_t* num_sel, uint32_t cap,
                             const fp_point* fin, uint64_t n, const fp_camera& cam, unsigned long long* fb,
                             const Workspace& ws, int num_sms, cudaStream_t st)
{
    const RenderBufs B = render_carve(ws, cap);
    cudaError_t e;
    if ((e = cudaMemsetAsync(B.num, 0, 2 * sizeof(uint32_t), st))) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_raster, kRenderNT, 0))) return e;
    RasterArgs a{};
    a.nodes = nodes; a.ids = ids; a.num_sel = num_sel; a.cap = cap; a.pstart = B.pstart; a.pshift = B.pshift; a.part = B.tiles64;
    a.fin = reinterpret_cast<const int4*>(fin); a.n = n; a.cam = cam_dev(cam); a.fb = fb; a.bar = B.num;
    a.err = ws.err;
    const unsigned grid = (unsigned)std::min<uint64_t>(kScanMaxTiles, (uint64_t)num_sms * std::min(std::max(per_sm, 1), kRasterCtas));
    return coop_launch(k_raster, grid, kRenderNT, 0, st, a);
}

}  // namespace fp
