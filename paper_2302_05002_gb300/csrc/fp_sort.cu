// fp_sort.cu -- plans of the stable bucket-scatter passes and fp_distribute.
//
// fp_distribute (Sec. 4.4: the cloud is "sorted into a number of chunks", each
// a node of the global tree, Fig. "octree") is a stable scatter of the points by
// chunk id, looked up from the point's level-g cell (lut).  Up to 4096 chunks the
// count and sweep of fp_seg.cu; more take two or three least-significant-digit-
// first passes, chosen on the device.  Small clouds take one launch (k_dist_cluster).
#include "fp_seg.cuh"

namespace fp {

// the first pass's look-back words of the tiles of n records
FP_DEV void zero_status(uint32_t* status, uint64_t n, uint32_t bits)
{
    const uint64_t words = ((n + kSortTile - 1) / kSortTile) << bits;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (uint64_t i = t; i < words / 4; i += stride) reinterpret_cast<uint4*>(status)[i] = make_uint4(0, 0, 0, 0);
    for (uint64_t i = words / 4 * 4 + t; i < words; i += stride) status[i] = 0;
}

__global__ void __launch_bounds__(1024) k_plan_hist_weights(SortSpec p, uint32_t* status, uint64_t n,
                                                            const uint32_t* d_n, const uint32_t* run_if,
                                                            const uint32_t* weights, const uint64_t* offsets)
{
    if (run_if && !*run_if) return;
    if (d_n && *d_n < n) n = *d_n;
    if (n == 0) return;
    __shared__ uint32_t sh[kSortMaxPass << kSortMaxBits];
    const uint64_t nw = p.d_nw ? *p.d_nw : p.nw_max;
    uint32_t npass, bits;
    sort_shape(p, npass, bits);
    zero_status(status, n, bits);
    const uint32_t mask = (1u << bits) - 1;
    for (int q = threadIdx.x; q < (kSortMaxPass << kSortMaxBits); q += blockDim.x) sh[q] = 0;
    __syncthreads();
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t id = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; id < nw; id += stride) {
        uint32_t w = weights ? weights[id] : (uint32_t)(offsets[id + 1] - offsets[id]);
        if (!w) continue;
        for (uint32_t k = 0; k < npass; ++k)
            atomicAdd(&sh[(k << kSortMaxBits) + ((id >> (k * bits)) & mask)], w);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < (kSortMaxPass << kSortMaxBits); q += blockDim.x)
        if (sh[q]) atomicAdd(&p.hist[q], sh[q]);
}

__global__ void __launch_bounds__(1024) k_plan_hist_keys(SortSpec p, uint32_t* status, const uint64_t* keys,
                                                         uint64_t n, const uint32_t* d_n, const uint32_t* run_if)
{
    if (run_if && !*run_if) return;
    if (d_n && *d_n < n) n = *d_n;
    if ((uint64_t)blockIdx.x * blockDim.x >= n) return;   // (a block with keys is there for every tile's words)
    __shared__ uint32_t sh[kSortMaxPass << kSortMaxBits];
    uint32_t npass, bits;
    sort_shape(p, npass, bits);
    {   // the words of the tiles whose records this block counts first
        const uint64_t words = ((n + kSortTile - 1) / kSortTile) << bits;
        const uint64_t used = min((uint64_t)gridDim.x, (n + blockDim.x - 1) / blockDim.x);   // blocks with keys
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += used * blockDim.x) status[i] = 0;
    }
    const uint32_t mask = (1u << bits) - 1;
    for (int q = threadIdx.x; q < (kSortMaxPass << kSortMaxBits); q += blockDim.x) sh[q] = 0;
    __syncthreads();
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        uint64_t k = keys[i] >> p.shift0;
        for (uint32_t q = 0; q < npass; ++q) atomicAdd(&sh[(q << kSortMaxBits) + ((k >> (q * bits)) & mask)], 1u);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < (kSortMaxPass << kSortMaxBits); q += blockDim.x)
        if (sh[q]) atomicAdd(&p.hist[q], sh[q]);
}

size_t sort_status_bytes(uint64_t n)
{
    return Workspace::round((sizeof(uint32_t) * std::max<uint64_t>(1, (n + kSortTile - 1) / kSortTile)) << kSortMaxBits);
}

// (the histogram first: callers clear it together with what lies before it)
size_t sort_scratch_bytes(uint64_t n)
{
    Workspace dry;
    take_sort_scratch(dry, n);
    return dry.used;
}

SortScratch take_sort_scratch(const Workspace& ws, uint64_t n, const Workspace* second)
{
    const size_t words = sort_status_bytes(n) / sizeof(uint32_t);
    SortScratch s;
    s.hist = ws.take<uint32_t>(kSortHistWords);
    s.status[0] = ws.take<uint32_t>(words);
    s.status[1] = (second ? *second : ws).take<uint32_t>(words);
    return s;
}

static void set_plan(const SortScratch& sc, SortArgs& a)
{
    a.spec.hist = sc.hist;
    a.status[0] = sc.status[0];
    a.status[1] = sc.status[1];
}

cudaError_t sort_plan_weights(const SortScratch& sc, SortArgs& a, const uint32_t* weights, const uint64_t* offsets,
                              const uint32_t* d_nw, uint64_t nw_max, bool zeroed, int num_sms, cudaStream_t st)
{
    a.spec = SortSpec{d_nw, nw_max, 0u, nullptr, 0u, nullptr};
    set_plan(sc, a);
    cudaError_t e;
    if (!zeroed && (e = cudaMemsetAsync(sc.hist, 0, sizeof(uint32_t) * kSortHistWords, st))) return e;
    const int grid = (int)std::min<uint64_t>(std::max<uint64_t>((nw_max + 1023) / 1024, a.n / 65536 + 1), num_sms * 2ull);
    k_plan_hist_weights<<<grid, 1024, 0, st>>>(a.spec, sc.status[0], a.n, a.d_n, a.run_if, weights, offsets);
    return cudaGetLastError();
}

cudaError_t sort_plan_keys(const SortScratch& sc, SortArgs& a, uint32_t shift0, uint32_t total_bits,
                           const uint32_t* d_rank_n, bool zeroed, int num_sms, cudaStream_t st)
{
    a.spec = SortSpec{nullptr, 0u, total_bits, d_rank_n, shift0, nullptr};
    set_plan(sc, a);
    cudaError_t e;
    if (!zeroed && (e = cudaMemsetAsync(sc.hist, 0, sizeof(uint32_t) * kSortHistWords, st))) return e;
    const int grid = (int)std::max<uint64_t>(1, std::min<uint64_t>((a.n + 4095) / 4096, num_sms * 2ull));
    k_plan_hist_keys<<<grid, 1024, 0, st>>>(a.spec, sc.status[0], a.b.k64_src, a.n, a.d_n, a.run_if);
    return cudaGetLastError();
}

// ------------------------------------------------------------- distribute
// The tables of the sweep lie where the radix passes' second point buffer does: one
// or the other runs.
struct DistBufs {
    SortScratch sc;
    int4* pt_tmp;
    uint32_t *val_tmp, *run_sort;
    Workspace sweep;   // dist_wide's
};

static DistBufs dist_bufs(const Workspace& ws, uint64_t n)
{
    DistBufs B;
    B.sc = take_sort_scratch(ws, n);
    B.sweep = ws;
    B.pt_tmp = ws.take<int4>(n);
    ws.used = std::max(ws.used, B.sweep.used + dist_wide_bytes(n));
    B.val_tmp = ws.take<uint32_t>(n);
    B.run_sort = ws.take<uint32_t>(1);
    return B;
}

size_t distribute_ws_bytes(uint64_t n, int g)
{
    (void)g;
    Workspace dry;
    dist_bufs(dry, n);
    return dry.used;
}

cudaError_t launch_distribute(const fp_point* pts, uint64_t n, const fp_cube* cube, int g, const uint32_t* lut,
                              const uint64_t* offsets, const uint32_t* num_chunks, fp_point* out, uint32_t* perm,
                              const Workspace& ws, cudaStream_t st, const uint32_t* cells)
{
    if (n == 0) return cudaSuccess;
    const DistBufs B = dist_bufs(ws, n);
    const SortScratch& sc = B.sc;
    int4* const pt_tmp = B.pt_tmp;
    uint32_t *const val_tmp = B.val_tmp, *const run_sort = B.run_sort;
    KTimerScope kt(FP_KERNEL_DISTRIBUTE, st);
    if (n <= kDistCluster) {
        uint32_t* const w = reinterpret_cast<uint32_t*>(pt_tmp);   // four words a point
        uint32_t* const tmp[4] = {w, w + n, w + 2 * n, w + 3 * n};
        return dist_cluster(reinterpret_cast<const int4*>(pts), n, cube, g, lut, offsets, num_chunks,
                            reinterpret_cast<int4*>(out), perm, cells, tmp, sc.hist, ws.err, st);
    }
    // Up to 4096 chunks: the count, scan and sweep (every point's chunk kept in
    // val_tmp, which the radix passes below then do not use), from
    // the cells or from the points.  More: the radix passes, which compute the
    // cells from the points.
    cudaError_t e = dist_wide(reinterpret_cast<const int4*>(pts), n, cube, g, lut, offsets, num_chunks,
                              reinterpret_cast<int4*>(out), perm, run_sort, sc.hist, B.sweep, st, cells,
                              reinterpret_cast<uint16_t*>(val_tmp));
    if (e) return e;
    SortArgs a{};
    a.b.pt_src = reinterpret_cast<const int4*>(pts);
    a.b.pt_tmp = pt_tmp;
    a.b.pt_dst = reinterpret_cast<int4*>(out);
    a.b.val_src = nullptr;   // value = original index
    a.b.val_tmp = perm ? val_tmp : nullptr;
    a.b.val_dst = perm;
    a.n = n;
    a.cube = cube;
    a.lut = lut;
    a.g = g;
    a.err = ws.err;
    a.run_if = run_sort;
    // bucket weights = chunk counts (offsets[c+1] - offsets[c])
    if ((e = sort_plan_weights(sc, a, nullptr, offsets, num_chunks, 1ull << (3 * g), true, ws.num_sms, st))) return e;
    return sort_run<DIG_CHUNK, true, false, false>(a, sort_passes(count_bits(1ull << (3 * g))), ws.num_sms, st);
}

}  // namespace fp
