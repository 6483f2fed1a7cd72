// Device-wide scan and stable LSD radix passes, the building blocks of the
// block-sorting transform (Method 3).
//
//  - scan: exclusive or inclusive prefix sum of u32 in three launches (tile
//    sums; one CTA scans the tile sums and writes the total; every tile adds
//    its offset), tiles of 4096 elements.
//  - radix pass: stable scatter of (u64 key, u32 value) pairs by the 8-bit
//    digit (key >> shift) & 255, in three launches: per-tile digit counts
//    stored digit-major (see RadixSpan), their exclusive scan (which
//    is then each tile's first output slot per digit, tiles in order within
//    a digit: stability across tiles), and the scatter.  The scatter ranks
//    equal digits inside a tile in element order with a ballot per digit bit
//    and per-warp running counts, sorts the tile in shared memory and writes
//    it out digit run by digit run, so consecutive threads write consecutive
//    slots.
// The kernels are launched behind one another (see launch_chained).  All loops
// are bounded by the element count; nothing waits on another CTA.
#pragma once

#include "huff_internal.cuh"

namespace huff {
namespace srt {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr uint32_t kScanTile = kScanThreads * kScanItems;  // 4096
constexpr int kRadixThreads = 512;
constexpr int kRadixItems = 8;
constexpr uint32_t kRadixTile = kRadixThreads * kRadixItems;  // 4096
constexpr int kRadixWarps = kRadixThreads / 32;

__host__ __device__ inline uint32_t div_up(uint64_t a, uint32_t b) { return (uint32_t)((a + b - 1) / b); }

// ---- scan -----------------------------------------------------------------
// block-wide exclusive scan of one value per thread (kScanThreads threads);
// returns the exclusive prefix, *total gets the sum
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *warp_sums, uint32_t &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d)
            x += y;
    }
    if (lane == 31)
        warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < kScanThreads / 32 ? warp_sums[lane] : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d)
                s += y;
        }
        if (lane < kScanThreads / 32)
            warp_sums[lane] = s;  // inclusive warp prefix
    }
    __syncthreads();
    total = warp_sums[kScanThreads / 32 - 1];
    const uint32_t before = w > 0 ? warp_sums[w - 1] : 0u;
    __syncthreads();  // warp_sums reusable after return
    return before + x - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(const uint32_t *in, uint32_t count,
                                                             uint32_t *part)
{
    chain_wait();
    chain_next();
    __shared__ uint32_t ws[kScanThreads / 32];
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        if (base + j < count)
            s += in[base + j];
    uint32_t total;
    block_excl_scan(s, ws, total);
    if (threadIdx.x == 0)
        part[blockIdx.x] = total;
}

// one CTA: exclusive scan of the tile sums in place, the total to *total
__global__ void __launch_bounds__(kScanThreads) k_scan_parts(uint32_t *part, uint32_t tiles,
                                                             uint32_t *total)
{
    chain_wait();
    chain_next();
    __shared__ uint32_t ws[kScanThreads / 32];
    uint32_t carry = 0;
    for (uint32_t b = 0; b < tiles; b += kScanThreads) {
        const uint32_t i = b + threadIdx.x;
        const uint32_t v = i < tiles ? part[i] : 0u;
        uint32_t t;
        const uint32_t x = block_excl_scan(v, ws, t);
        if (i < tiles)
            part[i] = carry + x;
        carry += t;
    }
    if (threadIdx.x == 0 && total)
        *total = carry;
}

template <bool kInclusive>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const uint32_t *in, uint32_t count,
                                                             const uint32_t *part, uint32_t *out)
{
    chain_wait();
    chain_next();
    __shared__ uint32_t ws[kScanThreads / 32];
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        v[j] = base + j < count ? in[base + j] : 0u;
        s += v[j];
    }
    uint32_t total;
    uint32_t run = part[blockIdx.x] + block_excl_scan(s, ws, total);
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        if (base + j < count)
            out[base + j] = kInclusive ? run + v[j] : run;
        run += v[j];
    }
}

inline uint64_t scan_parts_bytes(uint64_t count) { return 4ull * div_up(count, kScanTile) + 16; }

// out[i] = sum of in[0, i) (or [0, i]); *d_total = sum of all (if given).
// `part` holds scan_parts_bytes(count).  in == out is allowed.
inline cudaError_t scan_u32(const uint32_t *in, uint32_t *out, uint32_t count, bool inclusive,
                            uint32_t *part, uint32_t *d_total, cudaStream_t s)
{
    const uint32_t tiles = div_up(count, kScanTile);
    cudaError_t e = cudaSuccess;
    if (tiles > 0)
        e = launch_chained(k_scan_tiles, tiles, kScanThreads, 0, s, in, count, part);
    if (e == cudaSuccess)
        e = launch_chained(k_scan_parts, 1, kScanThreads, 0, s, part, tiles, d_total);
    if (e == cudaSuccess && tiles > 0)
        e = launch_chained(inclusive ? k_scan_apply<true> : k_scan_apply<false>, tiles, kScanThreads, 0, s,
                           in, count, part, out);
    return e;
}

// ---- radix pass -----------------------------------------------------------
__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
__device__ __forceinline__ uint32_t lanemask_le()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
    return m;
}

// The lanes whose 8-bit digit equals this lane's, of those with `ok`: a ballot
// per bit.  (__match_any_sync takes a step per distinct digit: on diverse
// digits it made a pass over 64 M elements 0.43 + 0.52 ms, counting and
// scattering, against 0.10 + 0.36 ms on a digit of few values.)
__device__ __forceinline__ uint32_t same_digit(uint32_t d, bool ok)
{
    uint32_t mask = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const uint32_t set = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        mask &= ((d >> b) & 1u) ? set : ~set;
    }
    return mask;
}

// The elements of a sort: all of them, or blocks of `block` elements that are
// sorted each by itself, with `per` tiles (the last one ragged) to a block.
// Digit d of tile t of block b is counted at [(b * 256 + d) * per + t]: the
// exclusive sum of these counts is its first place in the output.
struct RadixSpan {
    uint32_t count, block, per;
    // this CTA's tile: its elements [lo, hi), and its first counter
    __device__ __forceinline__ void tile(uint64_t &lo, uint64_t &hi, uint64_t &first) const
    {
        const uint32_t b = blockIdx.x / per, t = blockIdx.x - b * per;
        const uint64_t s = (uint64_t)b * block, end = s + block < count ? s + block : count;
        lo = s + (uint64_t)t * kRadixTile;
        hi = lo + kRadixTile < end ? lo + kRadixTile : end;
        if (hi < lo)
            hi = lo;
        first = (uint64_t)b * 256 * per + t;
    }
};

__global__ void __launch_bounds__(kRadixThreads) k_radix_count(const uint64_t *keys, RadixSpan sp,
                                                               uint32_t shift, uint32_t *hist)
{
    chain_wait();
    chain_next();
    __shared__ uint32_t c[256];
    if (threadIdx.x < 256)
        c[threadIdx.x] = 0;
    __syncthreads();
    uint64_t base, end, first;
    sp.tile(base, end, first);
    const int lane = threadIdx.x & 31;
    uint32_t dig[kRadixItems];
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {  // every load in flight before the first use
        const uint64_t e = base + (uint64_t)j * kRadixThreads + threadIdx.x;
        dig[j] = e < end ? (uint32_t)(keys[e] >> shift) & 255u : 256u;
    }
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {
        const uint32_t d = dig[j];
        // a warp of one digit adds once, else lane by lane (equal digits
        // then meet in a bank, but a run of them is rare)
        if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
            if (lane == 0 && d < 256u)
                atomicAdd(&c[d], 32u);
        } else if (d < 256u) {
            atomicAdd(&c[d], 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x < 256)
        hist[first + (uint64_t)threadIdx.x * sp.per] = c[threadIdx.x];
}

// shared memory of the scatter: the tile in sorted order, the digits' counts
// per warp (then their first places in the tile), and what a place in the tile
// lacks to the one in the output, per digit
struct RadixShared {
    uint64_t key[kRadixTile];
    uint32_t val[kRadixTile];
    uint32_t cnt[kRadixWarps][256];
    uint32_t to_out[256];
    uint32_t ws[8];
};

// Bound by the ALU pipe (62%), the shared-memory pipe (62%) and the barriers of
// two CTAs per SM (64 registers; 94 where a warp's counters are read once, or
// spilled to fit, are slower). 64 M elements in 0.49 ms (24 bytes each, 3.3
// TB/s); with the digits' first places in the tile and in the output looked up
// per element, not folded into the counters, a 64 MiB transform of text took
// 7.57 ms instead of 7.46.
__global__ void __launch_bounds__(kRadixThreads) k_radix_scatter(
    const uint64_t *kin, const uint32_t *vin, uint64_t *kout, uint32_t *vout, RadixSpan sp,
    uint32_t shift, const uint32_t *offs)
{
    chain_wait();
    chain_next();
    extern __shared__ __align__(16) unsigned char radix_sm[];
    RadixShared &sh = *reinterpret_cast<RadixShared *>(radix_sm);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // warp w owns the tile's elements [w * 256, (w + 1) * 256), taken 32 at
    // a time in order, so ranks follow element order
    uint64_t tb, end, first;
    sp.tile(tb, end, first);
    const uint64_t base = tb + (uint64_t)w * (kRadixItems * 32);
    uint64_t key[kRadixItems];
    uint32_t val[kRadixItems], rank[kRadixItems];
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {  // every load in flight before the first use
        const uint64_t e = base + (uint64_t)j * 32 + lane;
        const bool ok = e < end;
        key[j] = ok ? kin[e] : 0ull;
        val[j] = !ok ? 0u : vin ? vin[e] : (uint32_t)e;
    }
    uint32_t *const cnt = sh.cnt[w];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        cnt[j * 32 + lane] = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {
        const bool ok = base + (uint64_t)j * 32 + lane < end;
        const uint32_t d = (uint32_t)(key[j] >> shift) & 255u;
        const uint32_t mask = same_digit(d, ok);
        rank[j] = ok ? cnt[d] + __popc(mask & lanemask_lt()) : 0u;
        __syncwarp();
        if (ok && lane == __ffs(mask) - 1)
            cnt[d] += __popc(mask);
        __syncwarp();
    }
    __syncthreads();
    // per digit: the place in the tile of each warp's first element with it, and
    // the way from a place in the tile to one in the output
    uint32_t of[kRadixWarps], run = 0, x = 0, g = 0;
    if (tid < 256) {
        g = offs[first + (uint64_t)tid * sp.per];
#pragma unroll
        for (int ww = 0; ww < kRadixWarps; ++ww) {
            of[ww] = sh.cnt[ww][tid];
            run += of[ww];
        }
        // scan of the 256 digit totals (8 warps)
        x = run;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, s);
            if (lane >= s)
                x += y;
        }
        if (lane == 31)
            sh.ws[w] = x;
    }
    __syncthreads();
    if (tid < 256) {
        uint32_t at = x - run;
        for (int ww = 0; ww < w; ++ww)
            at += sh.ws[ww];
        sh.to_out[tid] = g - at;
#pragma unroll
        for (int ww = 0; ww < kRadixWarps; ++ww) {
            sh.cnt[ww][tid] = at;
            at += of[ww];
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {
        if (base + (uint64_t)j * 32 + lane < end) {
            const uint32_t q = cnt[(uint32_t)(key[j] >> shift) & 255u] + rank[j];
            sh.key[q] = key[j];
            sh.val[q] = val[j];
        }
    }
    __syncthreads();
    const uint32_t n_here = (uint32_t)(end - tb);
#pragma unroll 4
    for (uint32_t q = tid; q < n_here; q += kRadixThreads) {
        const uint64_t k = sh.key[q];
        const uint32_t dst = q + sh.to_out[(uint32_t)(k >> shift) & 255u];
        kout[dst] = k;
        vout[dst] = sh.val[q];
    }
}

// scratch of one radix pass over so many tiles: the digit counts (scanned in
// place) and the scan's tile sums
inline uint64_t radix_tiles_bytes(uint64_t tiles)
{
    const uint64_t hist = 256ull * tiles;
    return ((4 * hist + 255) & ~255ull) + scan_parts_bytes(hist);
}
inline uint64_t radix_scratch_bytes(uint64_t count) { return radix_tiles_bytes(div_up(count, kRadixTile)); }

// Stable sort of (k, v)[0, count) by the key bits [lo, hi) in passes of 8
// bits, ping-ponging between (k0, v0) and (k1, v1); with a block size, of each
// block by itself (div_up(count, block) * div_up(block, kRadixTile) tiles).
// `indices`: v0 holds nothing yet, element i's value is i.  Returns in `flip`
// whether the result ended in (k1, v1).
inline cudaError_t radix_sort_bits(uint64_t *k0, uint32_t *v0, uint64_t *k1, uint32_t *v1,
                                   uint32_t count, uint32_t lo, uint32_t hi, void *scratch,
                                   cudaStream_t s, bool &flip, uint32_t block = 0, bool indices = false)
{
    flip = false;
    if (count <= 1)
        return indices && count ? cudaMemsetAsync(v0, 0, sizeof(uint32_t), s) : cudaSuccess;
    static KernelSetup setup;
    int per_sm = 0;
    const cudaError_t err = kernel_setup(setup, (const void *)k_radix_scatter, kRadixThreads,
                                         sizeof(RadixShared), &per_sm);
    if (err != cudaSuccess)
        return err;
    if (block == 0)
        block = count;
    const RadixSpan sp = {count, block, div_up(block, kRadixTile)};
    const uint32_t tiles = div_up(count, block) * sp.per;
    uint32_t *hist = static_cast<uint32_t *>(scratch);
    const uint64_t hist_n = 256ull * tiles;
    uint32_t *part = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(scratch) +
                                                  ((4 * hist_n + 255) & ~255ull));
    for (uint32_t sh = lo; sh < hi; sh += 8) {
        uint64_t *ki = flip ? k1 : k0;
        uint32_t *vi = flip ? v1 : v0;
        uint64_t *ko = flip ? k0 : k1;
        uint32_t *vo = flip ? v0 : v1;
        cudaError_t e = launch_chained(k_radix_count, tiles, kRadixThreads, 0, s, ki, sp, sh, hist);
        if (e != cudaSuccess)
            return e;
        e = scan_u32(hist, hist, (uint32_t)hist_n, false, part, nullptr, s);
        if (e != cudaSuccess)
            return e;
        e = launch_chained(k_radix_scatter, tiles, kRadixThreads, sizeof(RadixShared), s, ki,
                           indices && sh == lo ? nullptr : vi, ko, vo, sp, sh, hist);
        if (e != cudaSuccess)
            return e;
        flip = !flip;
    }
    return cudaSuccess;
}

}  // namespace srt
}  // namespace huff
