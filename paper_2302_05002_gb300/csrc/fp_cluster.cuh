// fp_cluster.cuh -- several phases in one launch, by a barrier of the whole grid
// (cooperative launch) or of one cluster.
//
// Steps over a few thousand nodes or chunks: a
// cluster of 8 CTAs of 1024 threads whose phases are separated by the hardware
// cluster barrier.  Such a step used to be a chain of grid launches (scans of
// three, sorts of two per pass); at these sizes a launch costs more, on the host
// (about 2 us) and on the device (2 - 5 us), than the work between two barriers.
#pragma once
#include "fp_internal.cuh"

namespace fp {

constexpr int kClCtas = 8;        // portable cluster size
constexpr int kClNT = 1024;
constexpr int kClThreads = kClCtas * kClNT;

FP_DEV uint32_t cl_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// barrier of the cluster; orders global memory between its CTAs (release, acquire)
FP_DEV void cl_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Exclusive prefix sums over i in [0, n) of value(i) (a pair packed into 64
// bits, each half below 2^32 in all), handed to store(i, prefix); returns the
// total.  part: kClCtas words of global memory.  All threads of the cluster.
// Rows of 1024 values, eight in flight a thread: with more than some 10^4 values
// the time is the latency of these loads on 8 SMs (one in flight: 1.5 times as long).
constexpr int kClRows = 8;
struct ClScanSmem {
    uint64_t row[kClRows][kClNT / 32], total, warp[kClNT / 32];
};

template <typename Value, typename Store>
FP_DEV uint64_t cl_scan(uint32_t n, uint64_t* part, ClScanSmem& S, Value value, Store store)
{
    constexpr int kWarps = kClNT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t per = (n + kClCtas - 1) / kClCtas, lo = min(n, cl_rank() * per), hi = min(n, lo + per);
    uint64_t s = 0;
#pragma unroll 8
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kClNT) s += value(i);
    uint64_t tot;
    block_exclusive_scan<kClNT, uint64_t>(s, S.warp, tot);
    if (threadIdx.x == 0) part[cl_rank()] = tot;
    cl_sync();
    uint64_t run = 0, all = 0;
    for (int r = 0; r < kClCtas; ++r) {
        const uint64_t v = *(volatile const uint64_t*)(part + r);
        if (r < (int)cl_rank()) run += v;
        all += v;
    }
    for (uint32_t i0 = lo; i0 < hi; i0 += kClNT * kClRows) {
        uint64_t v[kClRows], ex[kClRows];
#pragma unroll
        for (int u = 0; u < kClRows; ++u) {
            const uint32_t i = i0 + u * kClNT + threadIdx.x;
            v[u] = i < hi ? value(i) : 0;
        }
#pragma unroll
        for (int u = 0; u < kClRows; ++u) {
            uint64_t x = v[u];
            if (i0 + u * kClNT < hi)   // (a small table has one row; the same for the block)
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                    if (lane >= o) x += y;
                }
            if (lane == 31) S.row[u][warp] = x;
            ex[u] = x - v[u];
        }
        __syncthreads();
        if (warp == 0) {   // the rows' warps in order, eight of them a lane
            constexpr int kPer = kClRows * kWarps / 32;
            uint64_t* w = &S.row[0][0] + lane * kPer;
            uint64_t sum = 0, x;
#pragma unroll
            for (int q = 0; q < kPer; ++q) sum += w[q];
            x = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) S.total = x;
            x -= sum;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const uint64_t y = w[q];
                w[q] = x;
                x += y;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kClRows; ++u) {
            const uint32_t i = i0 + u * kClNT + threadIdx.x;
            if (i < hi) store(i, run + S.row[u][warp] + ex[u]);
        }
        run += S.total;
        __syncthreads();
    }
    cl_sync();   // (part may be written again)
    return all;
}

// barrier number `k` (from 1) of the grid, every block of which is resident
// (cooperative launch); false when the bounded wait ran out
FP_DEV bool grid_barrier(uint32_t* word, uint32_t k, uint32_t* err)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(word, 1u);
        const uint32_t target = k * gridDim.x;
        uint32_t spins = 0;
        s_ok = 1;
        while (ld_volatile(word) < target) {
            if (++spins > (1u << 22)) { raise(err, FP_ERR_TIMEOUT); s_ok = 0; break; }
            __nanosleep(64);
        }
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

// One pass of a stable sort of n records by an 8-bit digit: digit(i) of record i,
// put(i, at) moves it to place `at`.  Every CTA counts the digits of its slice,
// all CTAs' counts (hist: kClCtas * 256 words) give every digit's base, and each
// tile of 1024 records is ranked by ballots.  All threads of the cluster.
struct ClSortSmem {
    uint32_t whist[kClNT / 32][256];
    uint32_t cnt[256], base[256], warp[32];
};

template <typename Digit, typename Put>
FP_DEV void cl_sort_pass(uint32_t n, ClSortSmem& S, uint32_t* hist, Digit digit, Put put)
{
    const uint32_t rank = cl_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t per = (n + kClCtas - 1) / kClCtas, lo = min(n, rank * per), hi = min(n, lo + per);
    if (tid < 256) S.cnt[tid] = 0;
    __syncthreads();
    for (uint32_t i0 = lo; i0 < hi; i0 += kClNT) {
        const uint32_t i = i0 + tid;
        const uint32_t d = i < hi ? digit(i) : 0u;
        const uint32_t peers = match_bits<8>(d, i < hi);
        if (i < hi && lane == (uint32_t)__ffs(peers) - 1) atomicAdd(&S.cnt[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
    if (tid < 256) hist[rank * 256 + tid] = S.cnt[tid];
    cl_sync();
    {
        uint32_t before = 0, total = 0;
        if (tid < 256)
            for (int r = 0; r < kClCtas; ++r) {
                const uint32_t v = ld_volatile(hist + r * 256 + tid);
                if (r < (int)rank) before += v;
                total += v;
            }
        uint32_t all;
        const uint32_t ex = block_exclusive_scan<kClNT, uint32_t>(total, S.warp, all);
        if (tid < 256) S.base[tid] = ex + before;
    }
    for (uint32_t i0 = lo; i0 < hi; i0 += kClNT) {
        for (uint32_t q = tid; q < (kClNT / 32) * 256 / 4; q += kClNT)
            reinterpret_cast<uint4*>(&S.whist[0][0])[q] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        const uint32_t i = i0 + tid;
        const bool valid = i < hi;
        const uint32_t d = valid ? digit(i) : 0u;
        const uint32_t peers = match_bits<8>(d, valid);
        if (valid && lane == (uint32_t)__ffs(peers) - 1) S.whist[warp][d] = __popc(peers);
        __syncthreads();
        if (tid < 256) {
            uint32_t run = S.base[tid];
            for (int w = 0; w < kClNT / 32; ++w) {
                const uint32_t c = S.whist[w][tid];
                S.whist[w][tid] = run;
                run += c;
            }
            S.base[tid] = run;
        }
        __syncthreads();
        if (valid) put(i, S.whist[warp][d] + __popc(peers & lanemask_lt()));
        __syncthreads();
    }
    cl_sync();
}

// cooperative launch (all blocks resident, so that they may wait for one another)
template <typename... Params, typename... Args>
inline cudaError_t coop_launch(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                               Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// launch of kernel(args) as one cluster
template <typename Args>
inline cudaError_t cl_launch(void (*kernel)(Args), const Args& args, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kClCtas);
    cfg.blockDim = dim3(kClNT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kClCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args);
}

}  // namespace fp
