// fp_common.cuh -- device helpers shared by the kernels of libfastpoints.
//
// Cell arithmetic (paper Sec. 4.4; exact-integer reading): for axis a,
//   c_a(l) = floor((p_a - o_a) * 2^l / S),   0 <= p_a - o_a < S <= 2^32,  S >= 1.
// (floor of a floor: c(l) = c(21) >> (21 - l), so the deepest level in use is
// enough).  With R = floor(2^a / S), a = 31 + ceil(log2 S), so 2^31 <= R < 2^32:
// the truncated product (d R) >> (a - l) is the cell or one less, because
// d R / 2^(a-l) falls short of d 2^l / S by less than 2^l S / 2^a <= 2^(l-31);
// one test of the remainder, which is below 2 S, corrects it.  For S <= 2^31 the
// remainder fits 32 bits and the whole takes about eight integer instructions
// (which run at half rate, and bound the passes that compute cells); the one
// binade above takes 64-bit steps.  (An fp32 estimate corrected both ways in 64
// bits took about three times as many.)
// The Morton key interleaves one bit per axis per level with the x bit most
// significant inside every 3-bit digit.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "../../include/fastpoints.h"

#define FP_DEV __device__ __forceinline__

namespace fp {

constexpr int kKeyLevels = 21;          // deepest level of the 63-bit key
constexpr uint32_t kNone = 0xFFFFFFFFu;

// Sticky per-device error word (passed to every kernel); bit (1u << fp_status)
// marks each kind of fault.
// err[0]: status bits (1 << status); err[1]: the check sites that fired (one
// bit per site, for diagnosing which capacity or consistency check failed)
FP_DEV void raise(uint32_t* err, fp_status s, int site = -1)
{
    atomicOr(err, 1u << (unsigned)s);
    if (site >= 0) atomicOr(err + 1, 1u << (unsigned)site);
}

// ------------------------------------------------------------------ cube
struct CubeDev {
    int32_t o[3];
    uint64_t S;
    uint32_t R;      // floor(2^a / S)
    int32_t a;       // 31 + ceil(log2 S)
};

FP_DEV CubeDev load_cube(const fp_cube* c)
{
    CubeDev d;
    d.o[0] = c->o[0]; d.o[1] = c->o[1]; d.o[2] = c->o[2];
    d.S = c->S;
    d.a = 31 + (d.S > 1 ? 64 - __clzll((long long)(d.S - 1)) : 0);
    // floor(2^a / S) with a <= 63: 2^a - 1 has the same quotient unless S divides 2^a (S a power of two)
    d.R = d.S ? ((d.S & (d.S - 1)) ? (uint32_t)(((1ull << d.a) - 1) / d.S) : 0x80000000u) : 0u;
    return d;
}

// floor(d * 2^l / S) for d = p - o, 0 <= d < S, l <= 21
FP_DEV uint32_t cell_at(int32_t p, int32_t o, const CubeDev& c, int l)
{
    const uint32_t d = (uint32_t)p - (uint32_t)o;
    const int sh = c.a - l;   // 10 .. 62
    const uint32_t hi = __umulhi(d, c.R);
    uint32_t q = sh >= 32 ? hi >> (sh - 32) : __funnelshift_r(d * c.R, hi, sh);
    if (c.S <= 0x80000000ull) {
        const uint32_t S = (uint32_t)c.S;
        q += (d << l) - q * S >= S ? 1u : 0u;
    } else {
        q += ((uint64_t)d << l) - (uint64_t)q * c.S >= c.S ? 1u : 0u;
    }
    return q;
}

FP_DEV uint32_t spread3_10(uint32_t x)   // 10 bits -> bits 0, 3, ..., 27
{
    x &= 0x3FFu;
    x = (x | (x << 16)) & 0x030000FFu;
    x = (x | (x << 8)) & 0x0300F00Fu;
    x = (x | (x << 4)) & 0x030C30C3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

FP_DEV uint64_t spread3(uint32_t v)   // 21 bits -> bits 0, 3, ..., 60
{
    return (uint64_t)spread3_10(v) | ((uint64_t)spread3_10(v >> 10) << 30) | ((uint64_t)((v >> 20) & 1u) << 60);
}

// 63-bit Morton key of the level-21 cell of a point
FP_DEV uint64_t key21(int32_t x, int32_t y, int32_t z, const CubeDev& c)
{
    uint32_t cx = cell_at(x, c.o[0], c, kKeyLevels);
    uint32_t cy = cell_at(y, c.o[1], c, kKeyLevels);
    uint32_t cz = cell_at(z, c.o[2], c, kKeyLevels);
    return (spread3(cx) << 2) | (spread3(cy) << 1) | spread3(cz);
}

// Morton key of the level-l cell of a point, l <= 10 (equal to key21 >> 3 (21 - l))
FP_DEV uint32_t key_small(int32_t x, int32_t y, int32_t z, const CubeDev& c, int l)
{
    return (spread3_10(cell_at(x, c.o[0], c, l)) << 2) | (spread3_10(cell_at(y, c.o[1], c, l)) << 1) |
           spread3_10(cell_at(z, c.o[2], c, l));
}

// The same for l <= 8 (the grids): one spreading step less per axis, and the axes
// joined by shifts with addition.  The passes that compute a cell per point are bound
// by these instructions: count of 10^8 LiDAR points 546 -> 518 us, smallest hash per
// cell 447 -> 418 us, chunks of 10^7 points 65 -> 62 us.
FP_DEV uint32_t spread3_8(uint32_t x)   // 8 bits -> bits 0, 3, ..., 21
{
    x = (x | (x << 8)) & 0x0300F00Fu;
    x = (x | (x << 4)) & 0x030C30C3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}
FP_DEV uint32_t key_cell(int32_t x, int32_t y, int32_t z, const CubeDev& c, int l)
{
    return spread3_8(cell_at(x, c.o[0], c, l)) * 4u + spread3_8(cell_at(y, c.o[1], c, l)) * 2u +
           spread3_8(cell_at(z, c.o[2], c, l));
}

// key_cell of a point that may lie outside the cube, whose cells repeat there with
// the cube's side: always below 8^l (exact up to 2^(31 - l) sides away)
FP_DEV uint32_t key_cell_any(int32_t x, int32_t y, int32_t z, const CubeDev& c, int l)
{
    const uint32_t m = (1u << l) - 1u;
    return spread3_8(cell_at(x, c.o[0], c, l) & m) * 4u + spread3_8(cell_at(y, c.o[1], c, l) & m) * 2u +
           spread3_8(cell_at(z, c.o[2], c, l) & m);
}

// per-point code of the octree stage: LOD owner level (5 bits), leaf level (5
// bits) and the Morton key of the point's level-g cell (3 g <= 21 bits)
FP_DEV uint32_t code_make(int own, int leaf, uint32_t cell)
{
    return (uint32_t)own | ((uint32_t)leaf << 5) | (cell << 10);
}
FP_DEV int code_own(uint32_t c) { return (int)(c & 31u); }
FP_DEV int code_leaf(uint32_t c) { return (int)((c >> 5) & 31u); }
FP_DEV uint32_t code_cell(uint32_t c) { return c >> 10; }

// level of the deepest cell two level-21 keys share (-1: not even the root? no: >= 0)
FP_DEV int common_level(uint64_t a, uint64_t b)
{
    uint64_t x = a ^ b;
    if (x == 0) return kKeyLevels;
    int lz = __clzll((long long)x) - 1;   // bit 63 is always 0
    return lz / 3;
}

// ------------------------------------------------------------------ hash
// first output of a splitmix64 generator seeded with v (Steele, Lea, Flood 2014)
FP_DEV uint64_t splitmix64(uint64_t v)
{
    uint64_t z = v + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Keep rule of the uniform preview: splitmix64(v) is a multiple of m >= 1.
// m a power of two: the hash's low bits, for which its last step needs 32 bits
// only.  Else by one multiplication: with m = 2^k d, d odd, x is a multiple of m
// iff x times the inverse of d modulo 2^64, rotated right by k, is at most
// floor((2^64 - 1) / m) (Granlund and Montgomery 1994; Hacker's Delight, "test for
// zero remainder").  The previews are as much bound by these integer instructions
// as by memory: 51M points at modulus 52 took 307 us with a 64-bit remainder and
// 199 us now.
struct KeepMultiple {
    uint64_t inv, lim;
    uint32_t k, mask, pow2;
    static KeepMultiple of(uint32_t m)
    {
        KeepMultiple r;
        r.k = 0;
        r.mask = m - 1;
        r.pow2 = (m & (m - 1)) == 0;
        uint64_t d = m;
        while (!(d & 1)) { d >>= 1; ++r.k; }
        uint64_t x = d;   // d * d = 1 mod 8: three bits right, doubled by every step
        for (int i = 0; i < 5; ++i) x *= 2 - d * x;
        r.inv = x;
        r.lim = ~0ull / m;
        return r;
    }
    FP_DEV bool operator()(uint64_t v) const
    {
        uint64_t z = v + 0x9E3779B97F4A7C15ull;   // splitmix64 up to its last step
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        if (pow2) return (((uint32_t)z ^ (uint32_t)(z >> 31)) & mask) == 0;
        const uint64_t q = (z ^ (z >> 31)) * inv;
        const uint32_t lo = (uint32_t)q, hi = (uint32_t)(q >> 32);   // k < 32
        const uint64_t rot = (uint64_t)__funnelshift_r(lo, hi, k) | ((uint64_t)__funnelshift_r(hi, lo, k) << 32);
        return rot <= lim;
    }
};

// ------------------------------------------------------------------ memory
FP_DEV int4 ld_point(const fp_point* p, uint64_t i) { return __ldg(reinterpret_cast<const int4*>(p) + i); }
FP_DEV int4 ld_point_cs(const fp_point* p, uint64_t i)
{
    return __ldcs(reinterpret_cast<const int4*>(p) + i);
}
FP_DEV void st_point(fp_point* p, uint64_t i, int4 v) { reinterpret_cast<int4*>(p)[i] = v; }

FP_DEV uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Lanes of the warp holding the same BITS-bit value v as this lane, among the
// lanes with `valid` set (one ballot per bit: the cost does not grow with the
// number of distinct values in the warp).  All 32 lanes take part.
template <int BITS>
FP_DEV uint32_t match_bits(uint32_t v, bool valid)
{
    uint32_t peers = __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
        const bool bit = (v >> b) & 1u;
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// the line at p on its way to L2
FP_DEV void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// size bytes at p (16-byte aligned, size a multiple of 16) on their way to L2
FP_DEV void bulk_prefetch_l2(const void* p, uint32_t size)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(size) : "memory");
}

// volatile load for inter-block flags
FP_DEV uint32_t ld_volatile(const uint32_t* p) { return *(const volatile uint32_t*)p; }

// ---- bulk copies global -> shared memory completing on an mbarrier (TMA,
// one-dimensional form: 16-byte aligned addresses, size a multiple of 16)
FP_DEV uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
FP_DEV void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// orders this CTA's earlier shared-memory accesses before later bulk copies into it
FP_DEV void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
FP_DEV void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
FP_DEV void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
FP_DEV bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}
constexpr uint32_t kWaitLimit = 1u << 22;   // try_wait rounds before a wait counts as timed out
FP_DEV bool mbar_wait(uint64_t* bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kWaitLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
FP_DEV uint64_t ld_volatile64(const uint64_t* p) { return *(const volatile uint64_t*)p; }

// ------------------------------------------------------------------ block scan
// Exclusive scan of one value per thread over a block of NT threads (NT % 32 == 0).
template <int NT, typename T>
FP_DEV T block_exclusive_scan(T v, T* smem_warp /* NT/32 entries */, T& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < NT / 32 ? smem_warp[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xFFFFFFFFu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < NT / 32) smem_warp[lane] = w;
    }
    __syncthreads();
    total = smem_warp[NT / 32 - 1];
    T before = warp ? smem_warp[warp - 1] : T(0);
    __syncthreads();
    return before + x - v;
}

// Bounded spin: number of polls before an inter-block wait gives up.
constexpr uint32_t kSpinLimit = 1u << 24;

// Look-back words of the preview: state in the top two bits, sum below.
constexpr uint64_t kFlagAgg = 1ull << 62;
constexpr uint64_t kFlagInc = 2ull << 62;
constexpr uint64_t kValMask = (1ull << 62) - 1;

// The tile's output offset by decoupled look-back, by one warp: 32 earlier
// tiles' words per round trip; the sum runs back to the nearest inclusive
// prefix, and stops (and reads again) at the nearest word not yet published.
// Publishes the tile's own words; the last tile writes the total.  (By the whole
// block, 256 words a trip, the polling slowed the publishing: 0.21 -> 0.27 ms at
// 51M points.)
FP_DEV uint64_t preview_base(uint64_t* tile_status, uint64_t tile, uint64_t ntiles, uint32_t total, uint64_t out_cap,
                             uint64_t* out_count, uint32_t* err)
{
    const int lane = threadIdx.x & 31;
    uint64_t excl = 0;
    if (tile == 0) {
        if (lane == 0) atomicExch((unsigned long long*)&tile_status[0], (unsigned long long)(kFlagInc | total));
    } else {
        if (lane == 0) atomicExch((unsigned long long*)&tile_status[tile], (unsigned long long)(kFlagAgg | total));
        int64_t t = (int64_t)tile - 1;
        uint32_t spins = 0;
        while (t >= 0) {
            const int64_t q = t - lane;
            const uint64_t w = q >= 0 ? ld_volatile64(&tile_status[q]) : kFlagInc;
            const uint32_t inc = __ballot_sync(0xFFFFFFFFu, (w >> 62) == 2);
            const uint32_t none = __ballot_sync(0xFFFFFFFFu, (w >> 62) == 0);
            const int fi = inc ? __ffs(inc) - 1 : 32, fn = none ? __ffs(none) - 1 : 32;
            // lanes [0, take) are summed: up to the first unpublished word, or
            // through the first inclusive prefix, or all 32 aggregates
            const int take = fn < fi ? fn : (fi < 32 ? fi + 1 : 32);
            uint64_t v = lane < take ? (w & kValMask) : 0;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
            excl += v;
            if (fi < fn) break;   // reached an inclusive prefix
            if (take == 0 && ++spins > kSpinLimit) {
                if (lane == 0) raise(err, FP_ERR_TIMEOUT);
                break;
            }
            t -= take;
        }
        if (lane == 0)
            atomicExch((unsigned long long*)&tile_status[tile], (unsigned long long)(kFlagInc | (excl + total)));
    }
    if (lane == 0 && tile == ntiles - 1) {
        *out_count = excl + total;
        if (excl + total > out_cap) raise(err, FP_ERR_CAPACITY, 0);
    }
    return excl;
}

}  // namespace fp
