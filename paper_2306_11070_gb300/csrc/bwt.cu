// Method 3 (Section III-A): the block-sorting (Burrows-Wheeler) transform of
// every block before Method 2's coder, its inverse, and the Method 3
// container.
//
// Forward: the rotations of all blocks are sorted at once by prefix
// doubling.  Every position i carries a rank RK[i] = the first sorted slot
// of its group (the rotations that agree on the prefix compared so far);
// slots of block b are [b * block, b * block + m_b), so ranks are global.
//   round 0: sort all positions by (block, first q bytes of the rotation),
//            the bytes as digits of a number in base sigma, the number of byte
//            values that occur (q = 11 on text; see first_key);
//   round r: with h = q * 2^(r-1), the still-unresolved positions (groups of
//            more than one) are sorted by (group, RK[i + h within the block])
//            and their groups split where that second rank changes;
// until no group has two members or the compared prefix covers the longest
// block (then the remaining groups are equal rotations, already in start
// order since every pass is stable and the first order is by position).
// The sorts are stable LSD radix passes over only the key bits in use.  In
// rounds r >= 1 the active list is already in group order, so only each
// group's members need sorting: groups that fit one CTA's window (most of
// them on text) are sorted in shared memory in place, and only the members
// of the larger groups go through the global radix passes.
//
// Inverse: LF[p] = the slot of row p's last byte in a stable sort of the
// last column by (block, byte), which is the byte's first slot in the block
// plus the rank of row p among the block's rows with that byte: counted per
// tile and scanned, so LF is written in row order.  The block is the walk
// p -> LF[p] from the primary row, emitted backwards.  The walk is cut at
// sample rows (every 32nd or 64th row and the primary rows): each sample walks to the
// next sample, keeping the bytes it passes, list ranking by pointer jumping
// over the samples gives each sample's distance from the primary row, and its
// bytes are copied to their place.  A periodic block's walk returns to the
// primary row after one period c; the rest of the block repeats it.
#include <cmath>

#include "api_trace.h"
#include "batch_internal.cuh"
#include "sort_impl.cuh"

namespace huff {
namespace {

using namespace srt;

constexpr int kEw = 256;               // threads of the elementwise kernels
// Rows between regular samples of the inverse: 32 for blocks whose samples
// are ranked in one CTA's shared memory (k_rank), 64 for others.  The longest
// of the walks, ln(samples) gaps, and the cached part of LF that the walks in
// flight read both shrink with the gap: 64 MiB of text in 1 MiB blocks, walk
// 0.72 -> 0.57 ms.
constexpr uint32_t kRankMin = 4096, kRankMax = 1u << 20;  // such blocks, bytes
__host__ __device__ __forceinline__ uint32_t sample_gap(uint64_t most)
{
    return most >= kRankMin && most <= kRankMax ? 32u : 64u;
}
constexpr uint32_t kNil = 0xffffffffu;

unsigned ew_grid(uint64_t count)
{
    const uint64_t cap = (uint64_t)device_sm_count() * 16;
    uint64_t g = (count + kEw - 1) / kEw;
    if (g > cap)
        g = cap;
    return (unsigned)(g < 1 ? 1 : g);
}

uint32_t bit_width(uint64_t v)
{
    uint32_t b = 0;
    while (v) {
        ++b;
        v >>= 1;
    }
    return b;
}

__device__ __forceinline__ void block_span(uint32_t i, uint32_t block, uint32_t n, uint32_t &s,
                                           uint32_t &m)
{
    s = (i / block) * block;
    m = n - s < block ? n - s : block;
}

// ---- forward --------------------------------------------------------------
// Round 0's key: q bytes as base-sigma digits below the block id.
struct FirstKey {
    uint32_t q, sigma;
    uint32_t bits;      // of the digits' number
    bool by_block;      // the blocks are sorted each by itself
    uint64_t top;       // sigma^(q - 1), the first digit's weight
    uint8_t code[256];  // a byte value's digit
};
constexpr uint32_t kInitTile = 2048;
constexpr uint32_t kMaxFirst = 16;  // most bytes in a first key

// Round 0 keys: (block id, the digits of the rotation's first q bytes).  A
// thread makes the keys of eight consecutive rotations, each from the one
// before (less its first digit, and one more), and the keys leave through
// shared memory in order: 64 MiB of text take 204 us, digit by digit 421.
// The rotations' indices need no array: the first radix pass makes them.
__global__ void __launch_bounds__(kEw) k_bwt_init(const uint8_t *x, uint32_t n, uint32_t block,
                                                  const __grid_constant__ FirstKey f, uint64_t *key)
{
    constexpr uint32_t kPer = kInitTile / kEw;  // 8
    __shared__ uint64_t out[kInitTile + kInitTile / kPer];  // a gap per thread: no bank conflicts
    __shared__ uint8_t code[256], tile[kInitTile + kMaxFirst];
    static_assert(kEw == 256, "a thread per byte value");
    code[threadIdx.x] = f.code[threadIdx.x];
    for (uint64_t t0 = (uint64_t)blockIdx.x * kInitTile; t0 < n; t0 += (uint64_t)gridDim.x * kInitTile) {
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < kInitTile + kMaxFirst; j += kEw)
            tile[j] = t0 + j < n ? code[x[t0 + j]] : 0;
        __syncthreads();
        const uint32_t j0 = threadIdx.x * kPer;
        uint64_t *const o = out + threadIdx.x * (kPer + 1);
        if (t0 + j0 < n) {
            const uint32_t i0 = (uint32_t)t0 + j0;
            uint32_t s, m;
            block_span(i0, block, n, s, m);
            if ((uint64_t)(i0 - s) + kPer + f.q <= m) {
                const uint64_t id = f.bits < 64 ? (uint64_t)(i0 / block) << f.bits : 0;
                uint64_t k = 0;
                for (uint32_t t = 0; t < f.q; ++t)
                    k = k * f.sigma + tile[j0 + t];
                o[0] = id | k;
#pragma unroll
                for (uint32_t j = 1; j < kPer; ++j) {
                    k = (k - tile[j0 + j - 1] * f.top) * f.sigma + tile[j0 + j + f.q - 1];
                    o[j] = id | k;
                }
            } else {  // a rotation goes on at its block's start, or blocks end here
                for (uint32_t j = 0; j < kPer && t0 + j0 + j < n; ++j) {
                    const uint32_t i = i0 + j;
                    block_span(i, block, n, s, m);
                    uint64_t k = 0;
                    for (uint32_t t = 0; t < f.q; ++t)
                        k = k * f.sigma + code[x[s + (uint32_t)(((uint64_t)(i - s) + t) % m)]];
                    o[j] = f.bits < 64 ? ((uint64_t)(i / block) << f.bits) | k : k;
                }
            }
        }
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < kInitTile && t0 + j < n; j += kEw)
            key[t0 + j] = out[j + j / kPer];
    }
}

// the counts of the bytes before the first 16-byte boundary
__global__ void k_count_head(const uint8_t *x, uint32_t count, unsigned long long *hist)
{
    if (threadIdx.x < count)
        atomicAdd(hist + x[threadIdx.x], 1ull);
}

// round r keys: (group, rank of the rotation h bytes on, relative to the
// block), packed so that the passes cover only the bits in use
__global__ void k_bwt_round_keys(const uint32_t *sa, const uint32_t *rk, const uint32_t *act,
                                 const uint32_t *grp, uint32_t count, uint32_t n, uint32_t block,
                                 uint64_t h, uint32_t lo_bits, uint64_t *key, uint32_t *val)
{
    chain_wait();
    chain_next();
    for (uint32_t k = blockIdx.x * kEw + threadIdx.x; k < count; k += gridDim.x * kEw) {
        const uint32_t i = sa[act[k]];
        uint32_t s, m;
        block_span(i, block, n, s, m);
        const uint32_t j = s + (uint32_t)(((uint64_t)(i - s) + h) % m);
        key[k] = ((uint64_t)grp[k] << lo_bits) | (rk[j] - s);
        val[k] = i;
    }
}

// ---- sorting the small groups of a round in shared memory ------------------
// The active list of round r >= 1 is in group order (its keys' high bits, the
// group number, never decrease), so sorting it means sorting every group's
// members by the low bits.  CTA t takes the groups that start in the window
// [t W, (t+1) W) of the list; they end before the first group start of the
// next window, so its range [a, b) is at most 2 W long, unless the last group
// starting in the window runs past the next one: such a group (more than W
// members) is left out (range [a, L)) and marked uncovered for the global
// passes.  Sorting within groups keeps every key's group bits at its index,
// so the start tests of neighbouring CTAs read the same groups whether or
// not a range beside them has been rewritten; ranges are disjoint and each is
// read into registers before it is written back.  In shared memory a key is
// (group index within the range, low bits): group numbers skip the groups
// already resolved, so the range's own numbering keeps the key to 32 bits
// (else the range is left to the global passes).  Stable 8-bit passes rank
// like the global scatter (warps own consecutive elements, equal digits in
// order by __match_any_sync and per-warp running counts); the group bits
// written back are those already at each index.
constexpr int kSegThreads = 512;
constexpr int kSegWarps = kSegThreads / 32;
constexpr uint32_t kSegWin = 2048;
constexpr uint32_t kSegCap = 2 * kSegWin;
constexpr uint32_t kSegSteps = kSegCap / kSegWarps / 32;  // at most 8 warp steps per pass
constexpr size_t kSegSmem = (5 * (size_t)kSegCap + (size_t)kSegWarps * 256 + 256) * 4;

__global__ void __launch_bounds__(kSegThreads) k_seg_sort(uint64_t *key, uint32_t *val, uint32_t count,
                                                          uint32_t lo_bits, uint32_t *cov)
{
    chain_wait();
    chain_next();
    extern __shared__ __align__(16) uint32_t seg_sm[];
    uint32_t *sk = seg_sm;                      // [2][kSegCap] range keys
    uint32_t *sv = sk + 2 * kSegCap;            // [2][kSegCap] values
    uint32_t *sg = sv + 2 * kSegCap;            // [kSegCap] group numbers of [w0, w2)
    uint32_t *wcnt = sg + kSegCap;              // [kSegWarps][256]
    uint32_t *dstart = wcnt + kSegWarps * 256;  // [256]
    __shared__ uint32_t s_a, s_b, s_l, s_gprev, s_ws[kSegWarps];
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint64_t w0 = (uint64_t)blockIdx.x * kSegWin;
    const uint64_t w1 = w0 + kSegWin < count ? w0 + kSegWin : count;
    const uint64_t w2 = w0 + kSegCap < count ? w0 + kSegCap : count;
    const uint32_t span = (uint32_t)(w2 - w0), win = (uint32_t)(w1 - w0);
    const uint64_t lo_mask = (1ull << lo_bits) - 1;
    // [w0, w2) into shared memory, coalesced: group numbers (they fit 32 bits:
    // fewer than count) and low bits (in the second key buffer for now)
    for (uint32_t i = tid; i < span; i += kSegThreads) {
        const uint64_t k = key[w0 + i];
        sg[i] = (uint32_t)(k >> lo_bits);
        sk[kSegCap + i] = (uint32_t)(k & lo_mask);
    }
    if (tid == 0) {
        s_a = kNil;
        s_b = kNil;
        s_l = 0;
        s_gprev = w0 > 0 ? (uint32_t)(key[w0 - 1] >> lo_bits) : kNil;
    }
    __syncthreads();
    {  // group starts in [w0, w2), one atomic per warp
        uint32_t a = kNil, l = 0, b = kNil;
        for (uint32_t i = tid; i < span; i += kSegThreads) {
            const bool st = i == 0 ? (w0 == 0 || sg[0] != s_gprev) : sg[i] != sg[i - 1];
            if (st) {
                if (i < win) {
                    a = i < a ? i : a;
                    l = i > l ? i : l;
                } else {
                    b = i < b ? i : b;
                }
            }
        }
        a = __reduce_min_sync(0xffffffffu, a);
        b = __reduce_min_sync(0xffffffffu, b);
        l = __reduce_max_sync(0xffffffffu, l);
        if (lane == 0) {
            atomicMin(&s_a, a);
            atomicMin(&s_b, b);
            atomicMax(&s_l, l);
        }
    }
    __syncthreads();
    const uint32_t a = s_a;
    if (a == kNil)
        return;  // no group starts in this window
    const uint32_t b = s_b != kNil ? s_b : (w2 == count ? span : s_l);
    if (b <= a)
        return;
    const uint32_t m = b - a;
    // warp w ranks the elements [w * steps * 32, (w + 1) * steps * 32) of the
    // range in every pass: an equal share each, in element order
    const uint32_t steps = (m + kSegThreads - 1) / kSegThreads;
    // each element's group index within the range: starts counted by ballots
    // over the warp's elements, then across the warps
    uint32_t mine = 0;
    for (uint32_t j = 0; j < steps; ++j) {
        const uint32_t i = (w * steps + j) * 32 + lane;
        const bool st = i > 0 && i < m && sg[a + i] != sg[a + i - 1];
        mine += __popc(__ballot_sync(0xffffffffu, st));
    }
    uint32_t groups;
    const uint32_t wbefore = srt::block_excl_scan(lane == 0 ? mine : 0u, s_ws, groups);
    const uint32_t wbase = __shfl_sync(0xffffffffu, wbefore, 0);
    if (((uint64_t)(groups + 1) << lo_bits) - 1 > 0xffffffffull)
        return;  // keys of this range wider than 32 bits: global passes
    const uint32_t bits = 64 - __clzll((long long)((((uint64_t)groups + 1) << lo_bits) - 1));
    {
        uint32_t run = wbase;
        for (uint32_t j = 0; j < steps; ++j) {
            const uint32_t i = (w * steps + j) * 32 + lane;
            const bool st = i > 0 && i < m && sg[a + i] != sg[a + i - 1];
            const uint32_t mask = __ballot_sync(0xffffffffu, st);
            if (i < m)
                sk[i] = ((run + __popc(mask & srt::lanemask_le())) << lo_bits) | sk[kSegCap + a + i];
            run += __popc(mask);
        }
    }
    for (uint32_t i = tid; i < m; i += kSegThreads)
        sv[i] = val[w0 + a + i];
    __syncthreads();
    uint32_t cur = 0;
    for (uint32_t shift = 0; shift < bits; shift += 8) {
        for (uint32_t i = tid; i < kSegWarps * 256; i += kSegThreads)
            wcnt[i] = 0;
        __syncthreads();
        const uint32_t *ck = sk + cur * kSegCap, *cv = sv + cur * kSegCap;
        uint32_t rank[kSegSteps], dg[kSegSteps];
#pragma unroll
        for (uint32_t j = 0; j < kSegSteps; ++j) {
            if (j >= steps)
                break;
            const uint32_t e = (w * steps + j) * 32 + lane;
            const uint32_t d = e < m ? (ck[e] >> shift) & 255u : 256u;
            const uint32_t mask = __match_any_sync(0xffffffffu, d);
            rank[j] = d < 256u ? wcnt[w * 256 + d] + __popc(mask & srt::lanemask_lt()) : 0u;
            __syncwarp();
            if (d < 256u && lane == (uint32_t)__ffs(mask) - 1)
                wcnt[w * 256 + d] += __popc(mask);
            __syncwarp();
            dg[j] = d;
        }
        __syncthreads();
        // per digit: exclusive prefix over the warps, then over the digits
        uint32_t run = 0, x = 0;
        if (tid < 256) {
#pragma unroll
            for (int ww = 0; ww < kSegWarps; ++ww) {
                const uint32_t t = wcnt[ww * 256 + tid];
                wcnt[ww * 256 + tid] = run;
                run += t;
            }
            x = run;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= (uint32_t)d)
                    x += y;
            }
            if (lane == 31)
                s_ws[w] = x;
        }
        __syncthreads();
        if (tid < 256) {
            uint32_t pre = 0;
            for (uint32_t ww = 0; ww < w; ++ww)
                pre += s_ws[ww];
            dstart[tid] = pre + x - run;
        }
        __syncthreads();
        uint32_t *nk = sk + (cur ^ 1) * kSegCap, *nv = sv + (cur ^ 1) * kSegCap;
#pragma unroll
        for (uint32_t j = 0; j < kSegSteps; ++j) {
            if (j >= steps)
                break;
            const uint32_t e = (w * steps + j) * 32 + lane;
            if (dg[j] < 256u) {
                const uint32_t q = dstart[dg[j]] + wcnt[w * 256 + dg[j]] + rank[j];
                nk[q] = ck[e];
                nv[q] = cv[e];
            }
        }
        __syncthreads();
        cur ^= 1;
    }
    const uint32_t *ck = sk + cur * kSegCap, *cv = sv + cur * kSegCap;
    for (uint32_t i = tid; i < m; i += kSegThreads) {
        key[w0 + a + i] = ((uint64_t)sg[a + i] << lo_bits) | ((uint64_t)ck[i] & lo_mask);
        val[w0 + a + i] = cv[i];
        cov[w0 + a + i] = 1u;
    }
}

// flags[k] = 1 - cov[k]: the members of groups left to the global passes
__global__ void k_uncovered(uint32_t *cov, uint32_t count)
{
    chain_wait();
    chain_next();
    for (uint32_t k = blockIdx.x * kEw + threadIdx.x; k < count; k += gridDim.x * kEw)
        cov[k] = 1u - cov[k];
}

// gather the uncovered elements (inclusive scan of their flags in incl) in
// list order, with their list indices
__global__ void k_gather_uncovered(const uint64_t *key, const uint32_t *val, const uint32_t *incl,
                                   uint32_t count, uint64_t *gk, uint32_t *gv, uint32_t *idx)
{
    for (uint32_t k = blockIdx.x * kEw + threadIdx.x; k < count; k += gridDim.x * kEw) {
        const uint32_t c = incl[k];
        if (c != (k ? incl[k - 1] : 0u)) {
            gk[c - 1] = key[k];
            gv[c - 1] = val[k];
            idx[c - 1] = k;
        }
    }
}

// the sorted uncovered elements back to their list indices: each large group
// owns the same indices before and after, so list order is kept
__global__ void k_scatter_uncovered(const uint64_t *gk, const uint32_t *gv, const uint32_t *idx,
                                    uint32_t count, uint64_t *key, uint32_t *val)
{
    for (uint32_t j = blockIdx.x * kEw + threadIdx.x; j < count; j += gridDim.x * kEw) {
        key[idx[j]] = gk[j];
        val[idx[j]] = gv[j];
    }
}

// ---- refining the groups of a sorted active list ---------------------------
// Element k of the sorted list starts a group when its key differs from
// k-1's (head), and its group has two members or more unless it is a head
// whose successor is a head too (flag).  One scan over the list gives, per
// element, the number of heads up to it (its group's number + 1), the number
// of flagged elements before it (its place in the next active list) and the
// largest head slot up to it (its group's first slot: slots increase along
// the list, so the last head wins), the three carried together.  From round 1
// on, a head that also starts a group of the round before (the key's group
// bits change there) carries a mark in the slot's low bit: elements whose
// last head is marked keep the first slot they had, so their rank is not
// written again.
constexpr int kRfThreads = 512;
constexpr int kRfItems = 8;
constexpr uint32_t kRfTile = kRfThreads * kRfItems;

struct AddOp {
    __device__ __forceinline__ uint32_t operator()(uint32_t a, uint32_t b) const { return a + b; }
};
struct MaxOp {
    __device__ __forceinline__ uint32_t operator()(uint32_t a, uint32_t b) const { return a > b ? a : b; }
};

// block-wide exclusive scan under op (kRfThreads threads), *total the
// reduction of all
template <class Op>
__device__ __forceinline__ uint32_t rf_block_scan(uint32_t v, uint32_t *ws, uint32_t &total, Op op,
                                                  uint32_t id)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d)
            x = op(x, y);
    }
    if (lane == 31)
        ws[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t t = lane < kRfThreads / 32 ? ws[lane] : id;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, d);
            if (lane >= d)
                t = op(t, y);
        }
        if (lane < kRfThreads / 32)
            ws[lane] = t;
    }
    __syncthreads();
    total = ws[kRfThreads / 32 - 1];
    const uint32_t before = w > 0 ? ws[w - 1] : id;
    uint32_t xe = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0)
        xe = id;
    __syncthreads();
    return op(before, xe);
}

struct RfItems {
    uint32_t head[kRfItems], flag[kRfItems], slot[kRfItems];
};

// A tile's keys and slots staged in shared memory with coalesced loads, so
// that each thread then reads its kRfItems consecutive elements from there.
// Index t is stored at t + t / 8: a thread's 8 consecutive words and a warp's
// consecutive fills then fall in distinct banks.
__device__ __forceinline__ uint32_t rf_pad(uint32_t t) { return t + (t >> 3); }
constexpr uint32_t kRfKeyWords = kRfTile + 2 + (kRfTile + 2) / 8 + 1;  // keys of [t0 - 1, t0 + kRfTile + 1)
constexpr uint32_t kRfIdxWords = kRfTile + kRfTile / 8;
constexpr size_t kRfTilesSmem = 8 * (size_t)kRfKeyWords + 4 * (size_t)kRfIdxWords;
constexpr size_t kRfApplySmem = kRfTilesSmem + 4 * (size_t)kRfIdxWords;

__device__ __forceinline__ void rf_stage(const uint64_t *key, const uint32_t *act, const uint32_t *val,
                                         uint32_t count, uint64_t t0, uint64_t *skey, uint32_t *sact,
                                         uint32_t *sval)
{
    for (uint32_t t = threadIdx.x; t < kRfTile + 2; t += kRfThreads) {
        const uint64_t k = t0 + t;  // element k - 1
        skey[rf_pad(t)] = (k >= 1 && k - 1 < count) ? key[k - 1] : 0ull;
    }
    for (uint32_t t = threadIdx.x; t < kRfTile; t += kRfThreads) {
        const uint64_t k = t0 + t;
        sact[rf_pad(t)] = k < count ? (act ? act[k] : (uint32_t)k) : 0u;
        if (val)
            sval[rf_pad(t)] = k < count ? val[k] : 0u;
    }
    __syncthreads();
}

// the values of this thread's kRfItems consecutive elements (from the stage)
__device__ __forceinline__ RfItems rf_items(const uint64_t *skey, const uint32_t *sact, uint32_t count,
                                            uint64_t t0, uint32_t gbits)
{
    const uint32_t t = threadIdx.x * kRfItems;
    const uint64_t base = t0 + t;
    uint64_t kk[kRfItems + 2];
#pragma unroll
    for (int j = 0; j < kRfItems + 2; ++j)
        kk[j] = skey[rf_pad(t + j)];  // element base + j - 1
    RfItems r;
#pragma unroll
    for (int j = 0; j < kRfItems; ++j) {
        const uint64_t k = base + j;
        const bool ok = k < count;
        const bool hd = ok && (k == 0 || kk[j + 1] != kk[j]);
        const bool nh = k + 1 >= count || kk[j + 2] != kk[j + 1];
        // gbits < 64: the key's bits from gbits up are the previous round's group
        const bool old = gbits < 64 && hd && (k == 0 || (kk[j + 1] >> gbits) != (kk[j] >> gbits));
        r.head[j] = hd ? 1u : 0u;
        r.flag[j] = (ok && !(hd && nh)) ? 1u : 0u;
        r.slot[j] = hd ? (sact[rf_pad(t + j)] << 1) | (old ? 1u : 0u) : 0u;
    }
    return r;
}

__global__ void __launch_bounds__(kRfThreads) k_refine_tiles(const uint64_t *key, const uint32_t *act,
                                                             uint32_t count, uint32_t gbits,
                                                             uint32_t *ph, uint32_t *pf, uint32_t *pm)
{
    chain_wait();
    chain_next();
    extern __shared__ __align__(16) uint64_t rf_sm[];
    uint64_t *skey = rf_sm;
    uint32_t *sact = reinterpret_cast<uint32_t *>(rf_sm + kRfKeyWords);
    __shared__ uint32_t ws[kRfThreads / 32];
    const uint64_t t0 = (uint64_t)blockIdx.x * kRfTile;
    rf_stage(key, act, nullptr, count, t0, skey, sact, nullptr);
    const RfItems r = rf_items(skey, sact, count, t0, gbits);
    uint32_t h = 0, f = 0, m = 0;
#pragma unroll
    for (int j = 0; j < kRfItems; ++j) {
        h += r.head[j];
        f += r.flag[j];
        m = r.slot[j] > m ? r.slot[j] : m;
    }
    uint32_t th, tf, tm;
    rf_block_scan(h, ws, th, AddOp(), 0u);
    rf_block_scan(f, ws, tf, AddOp(), 0u);
    rf_block_scan(m, ws, tm, MaxOp(), 0u);
    if (threadIdx.x == 0) {
        ph[blockIdx.x] = th;
        pf[blockIdx.x] = tf;
        pm[blockIdx.x] = tm;
    }
}

// one CTA: exclusive scans of the tile aggregates in place; the totals of
// heads (groups) and flags (next active count) to tot[0], tot[1]
__global__ void __launch_bounds__(kRfThreads) k_refine_parts(uint32_t *ph, uint32_t *pf, uint32_t *pm,
                                                             uint32_t tiles, uint32_t *tot)
{
    chain_wait();
    chain_next();
    __shared__ uint32_t ws[kRfThreads / 32];
    constexpr int kPer = 8;  // tiles per thread and step: a step is three scans (103 -> 54 us at 1)
    uint32_t ch = 0, cf = 0, cm = 0;
    for (uint32_t b = 0; b < tiles; b += kRfThreads * kPer) {
        const uint32_t i0 = b + threadIdx.x * kPer;
        uint32_t h[kPer], f[kPer], m[kPer], sh = 0, sf = 0, sm = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const bool ok = i0 + j < tiles;
            h[j] = ok ? ph[i0 + j] : 0u;
            f[j] = ok ? pf[i0 + j] : 0u;
            m[j] = ok ? pm[i0 + j] : 0u;
            sh += h[j];
            sf += f[j];
            sm = m[j] > sm ? m[j] : sm;
        }
        uint32_t th, tf, tm;
        uint32_t xh = ch + rf_block_scan(sh, ws, th, AddOp(), 0u);
        uint32_t xf = cf + rf_block_scan(sf, ws, tf, AddOp(), 0u);
        uint32_t xm = rf_block_scan(sm, ws, tm, MaxOp(), 0u);
        xm = xm > cm ? xm : cm;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            if (i0 + j < tiles) {
                ph[i0 + j] = xh;
                pf[i0 + j] = xf;
                pm[i0 + j] = xm;
            }
            xh += h[j];
            xf += f[j];
            xm = m[j] > xm ? m[j] : xm;
        }
        ch += th;
        cf += tf;
        cm = tm > cm ? tm : cm;
    }
    if (threadIdx.x == 0) {
        tot[0] = ch;
        tot[1] = cf;
    }
}

// sorted slots back into SA, new ranks scattered to the positions, and the
// elements of groups still unresolved appended to the next active list with
// their group numbers (staged in shared memory, where the keys were, and
// written out coalesced)
__global__ void __launch_bounds__(kRfThreads) k_refine_apply(
    const uint64_t *key, const uint32_t *val, const uint32_t *act, uint32_t count, uint32_t gbits,
    const uint32_t *ph, const uint32_t *pf, const uint32_t *pm, uint32_t *sa, uint32_t *rk,
    uint32_t *act2, uint32_t *grp2)
{
    chain_wait();
    chain_next();
    extern __shared__ __align__(16) uint64_t rf_sm[];
    uint64_t *skey = rf_sm;
    uint32_t *sact = reinterpret_cast<uint32_t *>(rf_sm + kRfKeyWords);
    uint32_t *sval = sact + kRfIdxWords;
    uint32_t *so_act = reinterpret_cast<uint32_t *>(rf_sm);  // after the keys are read
    uint32_t *so_grp = so_act + kRfIdxWords;
    __shared__ uint32_t ws[kRfThreads / 32];
    const uint64_t t0 = (uint64_t)blockIdx.x * kRfTile;
    rf_stage(key, act, val, count, t0, skey, sact, sval);
    if (act)  // (the first list's values are the slots already)
        for (uint32_t t = threadIdx.x; t < kRfTile && t0 + t < count; t += kRfThreads)
            sa[sact[rf_pad(t)]] = sval[rf_pad(t)];
    const RfItems r = rf_items(skey, sact, count, t0, gbits);
    uint32_t h = 0, f = 0, m = 0;
#pragma unroll
    for (int j = 0; j < kRfItems; ++j) {
        h += r.head[j];
        f += r.flag[j];
        m = r.slot[j] > m ? r.slot[j] : m;
    }
    uint32_t th, tf, tm;
    uint32_t gh = ph[blockIdx.x] + rf_block_scan(h, ws, th, AddOp(), 0u);
    uint32_t lf = rf_block_scan(f, ws, tf, AddOp(), 0u);  // flagged before, within the tile
    const uint32_t xm = rf_block_scan(m, ws, tm, MaxOp(), 0u);  // (its barriers: keys all read)
    const uint32_t pmb = pm[blockIdx.x];
    uint32_t gm = xm > pmb ? xm : pmb;
    const uint32_t t = threadIdx.x * kRfItems;
#pragma unroll
    for (int j = 0; j < kRfItems; ++j) {
        if (t0 + t + j >= count)
            break;
        gh += r.head[j];
        gm = r.slot[j] > gm ? r.slot[j] : gm;
        if (!(gm & 1u))  // else the group's first slot is unchanged
            rk[sval[rf_pad(t + j)]] = gm >> 1;
        if (r.flag[j]) {
            so_act[rf_pad(lf)] = sact[rf_pad(t + j)];
            so_grp[rf_pad(lf)] = gh - 1;
        }
        lf += r.flag[j];
    }
    __syncthreads();
    const uint32_t pfb = pf[blockIdx.x];
    for (uint32_t i = threadIdx.x; i < tf; i += kRfThreads) {
        act2[pfb + i] = so_act[rf_pad(i)];
        grp2[pfb + i] = so_grp[rf_pad(i)];
    }
}

__global__ void k_bwt_output(const uint8_t *x, const uint32_t *sa, uint32_t n, uint32_t block,
                             uint8_t *last, uint32_t *primary)
{
    chain_wait();
    chain_next();
    for (uint32_t p = blockIdx.x * kEw + threadIdx.x; p < n; p += gridDim.x * kEw) {
        const uint32_t i = sa[p];
        uint32_t s, m;
        block_span(p, block, n, s, m);
        last[p] = x[i == s ? s + m - 1 : i - 1];
        if (i == s)
            primary[p / block] = p - s;
    }
}

struct FwdWs {
    uint32_t *sa, *rk, *act, *act2, *grp, *grp2, *part, *scal;
    uint64_t *k0, *k1;
    uint32_t *v0, *v1;
    void *radix;
    uint64_t bytes;
};

template <class T>
T *carve(uint8_t *base, uint64_t &off, uint64_t bytes)
{
    T *p = reinterpret_cast<T *>(base ? base + off : nullptr);
    off += (bytes + 255) & ~255ull;
    return p;
}

FwdWs fwd_layout(uint8_t *base, uint64_t n)
{
    FwdWs w;
    uint64_t off = 0;
    w.sa = carve<uint32_t>(base, off, 4 * n);
    w.rk = carve<uint32_t>(base, off, 4 * n);
    w.act = carve<uint32_t>(base, off, 4 * n);
    w.act2 = carve<uint32_t>(base, off, 4 * n);
    w.grp = carve<uint32_t>(base, off, 4 * n);
    w.grp2 = carve<uint32_t>(base, off, 4 * n);
    w.part = carve<uint32_t>(base, off, 3 * 4 * (uint64_t)div_up(n, kRfTile) + 16);
    w.scal = carve<uint32_t>(base, off, 16);
    w.k0 = carve<uint64_t>(base, off, 8 * n);
    w.k1 = carve<uint64_t>(base, off, 8 * n);
    w.v0 = carve<uint32_t>(base, off, 4 * n);
    w.v1 = carve<uint32_t>(base, off, 4 * n);
    w.radix = carve<uint8_t>(base, off, radix_scratch_bytes(n));
    w.bytes = off;
    return w;
}

// stable LSD over the key bits [0, bits)
cudaError_t sort_keys(FwdWs &w, uint32_t count, uint32_t bits, cudaStream_t s, uint64_t *&ks,
                      uint32_t *&vs)
{
    bool f = false;
    const cudaError_t e = radix_sort_bits(w.k0, w.v0, w.k1, w.v1, count, 0, bits, w.radix, s, f);
    ks = f ? w.k1 : w.k0;
    vs = f ? w.v1 : w.v0;
    return e;
}

// sort a round's active list (keys in k0/v0, already in group order) by its
// key bits [0, bits): small groups in shared memory in place, the members of
// the others gathered into k1/v1 (the second half as the ping-pong buffer),
// sorted by the global passes and put back.  If they are more than half the
// list, the whole list takes the global passes.  act2 / grp2 are free until
// the refinement and hold the indices and flags.
cudaError_t sort_groups(FwdWs &w, uint32_t count, uint32_t lo_bits, uint32_t bits, cudaStream_t s,
                        uint64_t *&ks, uint32_t *&vs)
{
    static KernelSetup setup;
    int per_sm = 0;
    cudaError_t e = kernel_setup(setup, (const void *)k_seg_sort, kSegThreads, kSegSmem, &per_sm);
    if (e != cudaSuccess)
        return e;
    uint32_t *cov = w.grp2, *idx = w.act2;
    if ((e = cudaMemsetAsync(cov, 0, 4ull * count, s)) != cudaSuccess)
        return e;
    if ((e = launch_chained(k_seg_sort, div_up(count, kSegWin), kSegThreads, kSegSmem, s, w.k0, w.v0, count,
                            lo_bits, cov)) != cudaSuccess ||
        (e = launch_chained(k_uncovered, ew_grid(count), kEw, 0, s, cov, count)) != cudaSuccess)
        return e;
    if ((e = scan_u32(cov, cov, count, true, w.part, w.scal + 2, s)) != cudaSuccess)
        return e;
    uint32_t big = 0;
    if ((e = cudaMemcpyAsync(&big, w.scal + 2, sizeof(big), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return e;
    ks = w.k0;
    vs = w.v0;
    if (big == 0)
        return cudaSuccess;
    if (2ull * big > count)
        return sort_keys(w, count, bits, s, ks, vs);
    k_gather_uncovered<<<ew_grid(count), kEw, 0, s>>>(w.k0, w.v0, cov, count, w.k1, w.v1, idx);
    bool f = false;
    if ((e = radix_sort_bits(w.k1, w.v1, w.k1 + big, w.v1 + big, big, 0, bits, w.radix, s, f)) !=
        cudaSuccess)
        return e;
    k_scatter_uncovered<<<ew_grid(big), kEw, 0, s>>>(f ? w.k1 + big : w.k1, f ? w.v1 + big : w.v1,
                                                      idx, big, w.k0, w.v0);
    return cudaGetLastError();
}

// split the groups of the sorted active list; returns the number still
// unresolved and the number of groups of the list (host values)
cudaError_t refine(FwdWs &w, const uint64_t *ks, const uint32_t *vs, uint32_t count,
                   uint32_t gbits, cudaStream_t s, uint32_t &n_act, uint32_t &groups)
{
    const uint32_t tiles = div_up(count, kRfTile);
    uint32_t *ph = w.part, *pf = w.part + tiles, *pm = w.part + 2 * tiles;
    static KernelSetup setup_tiles, setup_apply;
    int per_sm = 0;
    cudaError_t e;
    if ((e = kernel_setup(setup_tiles, (const void *)k_refine_tiles, kRfThreads, kRfTilesSmem,
                          &per_sm)) != cudaSuccess ||
        (e = kernel_setup(setup_apply, (const void *)k_refine_apply, kRfThreads, kRfApplySmem,
                          &per_sm)) != cudaSuccess)
        return e;
    // the first list is every slot in order
    const uint32_t *act = gbits < 64 ? w.act : nullptr;
    if ((e = launch_chained(k_refine_tiles, tiles, kRfThreads, kRfTilesSmem, s, ks, act, count, gbits, ph, pf,
                            pm)) != cudaSuccess ||
        (e = launch_chained(k_refine_parts, 1, kRfThreads, 0, s, ph, pf, pm, tiles, w.scal)) != cudaSuccess ||
        (e = launch_chained(k_refine_apply, tiles, kRfThreads, kRfApplySmem, s, ks, vs, act, count, gbits, ph,
                            pf, pm, w.sa, w.rk, w.act2, w.grp2)) != cudaSuccess)
        return e;
    uint32_t h[2];
    if ((e = cudaMemcpyAsync(h, w.scal, sizeof(h), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return e;
    groups = h[0];
    n_act = h[1];
    uint32_t *t = w.act;
    w.act = w.act2;
    w.act2 = t;
    t = w.grp;
    w.grp = w.grp2;
    w.grp2 = t;
    return cudaSuccess;
}

// The first key of an input with these byte counts: as many bytes as make most
// rotations of a block of m bytes differ, then as many more as the last pass
// has room for.  On the synthetic text (34 byte values, order-0 entropy 4.3
// bits, 1 MiB blocks) 96% of the positions are left in groups after 4 bytes,
// 42% after 8 and a quarter after 11, and a position left costs as much as
// about eight passes over it, so text wants 2.4 log2 m bits of order-0 entropy;
// bytes close to random differ after 1.5 log2 m.  Forward transform of 64 MiB
// in 1 MiB blocks against keys of four bytes always (and a radix pass that
// ranked with match.any): text 13.1 -> 8.2 ms, Zipf bytes 8.8 -> 7.0, uniform
// bytes 7.0 -> 4.9, the bitstream stand-in 47.3 -> 45.5; with blocks sorted each
// by itself and rolling keys 7.6, 6.3, 4.4 and 46.
FirstKey first_key(const unsigned long long *hist, uint64_t n, uint64_t blocks, uint64_t m)
{
    FirstKey f;
    f.sigma = 0;
    double entropy = 0;
    for (int b = 0; b < 256; ++b) {
        f.code[b] = (uint8_t)f.sigma;
        if (hist[b]) {
            ++f.sigma;
            const double p = (double)hist[b] / (double)n;
            entropy -= p * std::log2(p);
        }
    }
    if (f.sigma < 2)
        f.sigma = 2;
    // The block id need not be sorted by where the passes can take each block by
    // itself: blocks that fill their tiles, so that a pass costs no more (64 MiB
    // of text in 1 MiB blocks: 7 passes instead of 8, each 0.55 ms).  The pass
    // counters then lie in the ranks, which the first refinement writes.
    const uint64_t per = div_up(m, kRadixTile), tiles = blocks * per;
    const bool can = blocks > 1 && per * kRadixTile <= m + m / 8 && radix_tiles_bytes(tiles) <= 4 * n;
    const uint32_t room = 64 - bit_width(blocks - 1);
    const double want = (entropy > 7.5 ? 1.5 : 2.4) * bit_width(m - 1);
    f.q = f.bits = 0;
    for (uint64_t v = 1; f.q < kMaxFirst;) {  // v = sigma^q
        if (v > ~0ull / f.sigma)
            break;
        v *= f.sigma;
        const uint32_t bits = bit_width(v - 1);
        if (bits > room)
            break;
        const uint32_t used = can ? 0 : 64 - room;
        if (f.q >= 4 && f.q * entropy >= want && (bits + used + 7) / 8 > (f.bits + used + 7) / 8)
            break;  // enough, and one more byte would take another pass
        ++f.q;
        f.bits = bits;
    }
    f.top = 1;
    for (uint32_t t = 1; t < f.q; ++t)
        f.top *= f.sigma;
    f.by_block = can && (f.bits + 7) / 8 < (f.bits + (64 - room) + 7) / 8;
    return f;
}

// ---- inverse --------------------------------------------------------------
__global__ void k_lf_keys(const uint8_t *last, uint32_t n, uint32_t block, uint64_t *key,
                          uint32_t *val)
{
    for (uint32_t p = blockIdx.x * kEw + threadIdx.x; p < n; p += gridDim.x * kEw) {
        key[p] = ((uint64_t)(p / block) << 8) | last[p];
        val[p] = p;
    }
}

// A row's LF within its block and its byte in one word, so that a step of a
// walk is one load: 32 bits for blocks of up to 16 MiB, else 64.
template <class T>
__device__ __forceinline__ T lf_word(uint32_t lf, uint32_t byte)
{
    return (T)lf << 8 | byte;
}
constexpr uint32_t kMaxBlock32 = 1u << 24;

// blocks of less than a tile: from the sorted (block, byte) keys
__global__ void k_lf_scatter(const uint64_t *ks, const uint32_t *vs, uint32_t n, uint32_t block,
                             uint32_t *lf)
{
    for (uint32_t q = blockIdx.x * kEw + threadIdx.x; q < n; q += gridDim.x * kEw)
        lf[vs[q]] = lf_word<uint32_t>(q % block, (uint32_t)ks[q] & 255u);
}

// Other blocks: tiles of 4096 rows that do not cross blocks, `per` of them to a
// block; byte counts at [(block * 256 + byte) * per + tile], whose exclusive
// sum is a tile's first slot for each byte.
constexpr int kLfThreads = 512;
constexpr int kLfItems = 8;
constexpr int kLfWarps = kLfThreads / 32;
constexpr uint32_t kLfTile = kLfThreads * kLfItems;

// a warp's rows of the tile in order, 32 at a time
__device__ __forceinline__ void lf_tile(uint32_t n, uint32_t block, uint32_t per, uint32_t &s,
                                        uint32_t &t, uint32_t &row, uint32_t &left)
{
    const uint32_t b = blockIdx.x / per;
    t = blockIdx.x - b * per;
    s = b * block;
    const uint32_t m = n - s < block ? n - s : block;
    row = t * kLfTile + (threadIdx.x >> 5) * (kLfItems * 32);  // within the block
    left = row < m ? (m - row < kLfItems * 32 ? m - row : kLfItems * 32) : 0u;
}

// same_digit for a transformed column: where a warp's 32 rows hold few runs
// they hold few distinct bytes, which match.any takes one by one faster than
// eight ballots
__device__ __forceinline__ uint32_t same_byte(uint32_t d, bool ok)
{
    const uint32_t key = ok ? d : 256u;
    const uint32_t before = __shfl_up_sync(0xffffffffu, key, 1);
    if (__popc(__ballot_sync(0xffffffffu, key != before)) <= 6)
        return __match_any_sync(0xffffffffu, key);
    return same_digit(d, ok);
}

__global__ void __launch_bounds__(kLfThreads) k_lf_count(const uint8_t *last, uint32_t n,
                                                         uint32_t block, uint32_t per,
                                                         uint32_t *hist)
{
    __shared__ uint32_t c[256];
    if (threadIdx.x < 256)
        c[threadIdx.x] = 0;
    __syncthreads();
    uint32_t s, t, row, left;
    lf_tile(n, block, per, s, t, row, left);
    const uint32_t lane = threadIdx.x & 31;
    uint32_t d[kLfItems];
#pragma unroll
    for (int j = 0; j < kLfItems; ++j)
        d[j] = j * 32 + lane < left ? last[s + row + j * 32 + lane] : 0u;
#pragma unroll
    for (int j = 0; j < kLfItems; ++j) {
        // the last row of each run adds the run (a transformed column is runs)
        const bool ok = j * 32 + lane < left;
        const uint32_t key = ok ? d[j] : 256u;
        const uint32_t after = __shfl_down_sync(0xffffffffu, key, 1);
        const bool end = lane == 31 || after != key;
        const uint32_t before = __ballot_sync(0xffffffffu, end) & lanemask_lt();
        if (ok && end)
            atomicAdd(&c[d[j]], lane + 1 - (before ? 32 - __clz(before) : 0));
    }
    __syncthreads();
    if (threadIdx.x < 256)
        hist[((uint64_t)(blockIdx.x / per) * 256 + threadIdx.x) * per + t] = c[threadIdx.x];
}

template <class T>
__global__ void __launch_bounds__(kLfThreads) k_lf_rank(const uint8_t *last, uint32_t n,
                                                        uint32_t block, uint32_t per,
                                                        const uint32_t *offs, T *lf)
{
    __shared__ uint32_t cnts[kLfWarps][256];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t s, t, row, left;
    lf_tile(n, block, per, s, t, row, left);
    uint32_t *const cnt = cnts[w];
    uint32_t d[kLfItems], rank[kLfItems];
#pragma unroll
    for (int j = 0; j < kLfItems; ++j)
        d[j] = j * 32 + lane < left ? last[s + row + j * 32 + lane] : 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        cnt[j * 32 + lane] = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kLfItems; ++j) {
        const bool ok = j * 32 + lane < left;
        const uint32_t mask = same_byte(d[j], ok);
        rank[j] = cnt[d[j]] + __popc(mask & lanemask_lt());
        __syncwarp();
        if (ok && lane == (uint32_t)__ffs(mask) - 1)
            cnt[d[j]] += __popc(mask);
        __syncwarp();
    }
    __syncthreads();
    // per byte: the tile's first slot in the block, then the warps before
    if (threadIdx.x < 256) {
        uint32_t run =
            offs[((uint64_t)(blockIdx.x / per) * 256 + threadIdx.x) * per + t] - s;
#pragma unroll
        for (int ww = 0; ww < kLfWarps; ++ww) {
            const uint32_t x = cnts[ww][threadIdx.x];
            cnts[ww][threadIdx.x] = run;
            run += x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kLfItems; ++j)
        if (j * 32 + lane < left)
            lf[s + row + j * 32 + lane] = lf_word<T>(cnt[d[j]] + rank[j], d[j]);
}

__global__ void k_check_primary(const uint32_t *primary, uint32_t n, uint32_t block,
                                uint32_t blocks, int32_t *status)
{
    for (uint32_t b = blockIdx.x * kEw + threadIdx.x; b < blocks; b += gridDim.x * kEw) {
        const uint32_t s = b * block;
        const uint32_t m = n - s < block ? n - s : block;
        if (primary[b] >= m)
            set_status(status, HUFF_ERR_CORRUPT_STREAM);
    }
}

struct Samples {
    uint32_t n, block, regular, gap;  // regular samples: rows 0, gap, 2 gap, ...
    const uint32_t *primary;  // a primary row is its block's extra sample (id regular + block)
    // row of sample id, or kNil for a regular sample that is a primary row
    __device__ __forceinline__ uint32_t row_of(uint32_t id) const
    {
        if (id >= regular)
            return (id - regular) * block + primary[id - regular];
        const uint32_t p = id * gap;
        const uint32_t b = p / block;
        return p - b * block == primary[b] ? kNil : p;
    }
};

// The inverse of 64 MiB of text in 1 MiB blocks takes 1.21 ms (4.32 ms with LF
// from two radix passes and a scatter, bytes read in a second walk and global
// pointer jumping): LF 0.38, walk 0.57, rank 0.06, emit 0.13.  The walk is bound
// by its random reads of LF, 64 M sectors of L2 (half of them in it).
//
// Every sample walks to the next sample: link, length and the first `cap`
// bytes on the way (kept[id * cap]).  The link into a block's primary sample
// is cut (kNil), which turns the primary's cycle into a list headed by the
// primary.
template <class T>
__global__ void k_walk(const T *lf, Samples S, uint32_t count, uint32_t cap, uint32_t *nxt,
                       uint32_t *len, uint8_t *kept, int32_t *status)
{
    if (chain_failed(status))
        return;
    for (uint32_t id = blockIdx.x * kEw + threadIdx.x; id < count; id += gridDim.x * kEw) {
        const uint32_t p0 = S.row_of(id);
        uint32_t t = 0, to = kNil;
        if (p0 != kNil) {
            const uint32_t b = p0 / S.block, s = b * S.block;
            const uint32_t m = S.n - s < S.block ? S.n - s : S.block;
            const uint32_t prim = S.primary[b];
            uint64_t acc = 0;
            uint2 *const out = reinterpret_cast<uint2 *>(kept + (uint64_t)id * cap);
            uint32_t r = p0 - s;
            bool more = true;
            do {  // ends on p0 at the latest: LF is a permutation of the block
                const T v = lf[s + r];
                r = (uint32_t)(v >> 8);
                acc |= (uint64_t)((uint32_t)v & 255u) << (8 * (t & 7u));
                ++t;
                more = r != prim && ((s + r) & (S.gap - 1)) != 0 && t < m;
                if ((t & 7u) == 0 || !more) {
                    if (t <= cap)  // a multiple of 8
                        out[(t - 1) >> 3] = make_uint2((uint32_t)acc, (uint32_t)(acc >> 32));
                    acc = 0;
                }
            } while (more);
            if (r != prim) {
                to = (s + r) / S.gap;
                if (((s + r) & (S.gap - 1)) != 0) {  // cannot happen for a sorted column
                    set_status(status, HUFF_ERR_CORRUPT_STREAM);
                    to = kNil;
                    t = 0;
                }
            }
        }
        nxt[id] = to;
        len[id] = t;
    }
}

// one pointer-jumping step: sum[id] = stretch lengths from id to the list's
// end after enough steps
__global__ void k_jump(const uint32_t *nx_in, const uint32_t *sum_in, uint32_t count,
                       uint32_t *nx_out, uint32_t *sum_out, const int32_t *status)
{
    if (chain_failed(status))
        return;
    for (uint32_t id = blockIdx.x * kEw + threadIdx.x; id < count; id += gridDim.x * kEw) {
        const uint32_t x = nx_in[id];
        if (x == kNil) {
            nx_out[id] = kNil;
            sum_out[id] = sum_in[id];
        } else {
            nx_out[id] = nx_in[x];
            sum_out[id] = sum_in[id] + sum_in[x];
        }
    }
}

// The same for one block per CTA, in shared memory: sum[id] = stretch lengths
// from id to the end of its list, nx_out[id] = kNil where the list ends (all of
// them, but for lists that close in a cycle, which keep a link).  Up to
// kRankThreads - 1 evenly spaced samples and the primary split the lists; each
// walks its piece (about 32 links at 1 MiB, a chain of shared loads), pointer
// jumping ranks the pieces, and each walks its piece again to hand out the
// sums (and to mark its samples as ended).  A block's one list that ends is
// headed by the primary, so its pieces hold all of it.  For 64 blocks of 1 MiB 64
// us, against 209 us in 16 launches of global jumps at half the samples.
constexpr int kRankThreads = 1024;
constexpr uint32_t kRankCap = kRankMax / 32 + 3;  // samples of a block
constexpr uint32_t kRankEnd = 0xffffu;            // no link
struct RankShared {
    uint32_t len[kRankCap];  // a stretch's length, then its sum
    uint16_t nxt[kRankCap];
    uint32_t sum[2][kRankThreads];  // of the pieces
    uint16_t to[2][kRankThreads];   // the splitter a piece ends at
};

__global__ void __launch_bounds__(kRankThreads) k_rank(const uint32_t *nxt, const uint32_t *len,
                                                       Samples S, uint32_t *nx_out, uint32_t *sum_out,
                                                       const int32_t *status)
{
    extern __shared__ __align__(16) unsigned char rank_sm[];
    RankShared &sh = *reinterpret_cast<RankShared *>(rank_sm);
    if (chain_failed(status))
        return;
    const uint32_t tid = threadIdx.x, b = blockIdx.x;
    const uint32_t s = b * S.block, m = S.n - s < S.block ? S.n - s : S.block;
    // the block's regular samples, then its primary's
    const uint32_t first = (s + S.gap - 1) / S.gap;
    const uint32_t regs = (s + m + S.gap - 1) / S.gap - first, count = regs + 1;
    for (uint32_t i = tid; i < count; i += kRankThreads) {
        const uint32_t id = i < regs ? first + i : S.regular + b;
        const uint32_t to = nxt[id];
        sh.len[i] = len[id];
        sh.nxt[i] = (uint16_t)(to == kNil ? kRankEnd : to - first);  // a primary is never linked to
    }
    __syncthreads();
    // splitters: the samples step, 2 step, ... and the primary (the last piece)
    uint32_t step = 32;
    while (regs && (regs - 1) / step + 1 > (uint32_t)kRankThreads)
        step <<= 1;
    const uint32_t pieces = (regs ? (regs - 1) / step : 0u) + 1;
    const uint32_t own = tid + 1 < pieces ? (tid + 1) * step : regs;
    auto split = [&](uint32_t i) { return i == regs || (i && (i & (step - 1)) == 0); };
    uint32_t total = 0, at = own;
    if (tid < pieces) {
        uint32_t left = count;
        do {
            total += sh.len[at];
            at = sh.nxt[at];
        } while (at != kRankEnd && !split(at) && --left);
        sh.sum[0][tid] = total;
        sh.to[0][tid] = (uint16_t)(at == kRankEnd ? kRankEnd : at == regs ? pieces - 1 : at / step - 1);
    }
    __syncthreads();
    uint32_t cur = 0;
    for (uint32_t d = 1; d < pieces; d <<= 1, cur ^= 1) {
        if (tid < pieces) {
            const uint32_t t = sh.to[cur][tid];
            sh.sum[cur ^ 1][tid] = sh.sum[cur][tid] + (t != kRankEnd ? sh.sum[cur][t] : 0u);
            sh.to[cur ^ 1][tid] = t != kRankEnd ? sh.to[cur][t] : (uint16_t)kRankEnd;
        }
        __syncthreads();
    }
    // sums handed out along each piece of a list that ends
    if (tid < pieces && sh.to[cur][tid] == kRankEnd) {
        uint32_t rest = sh.sum[cur][tid], i = own;
        do {
            const uint32_t l = sh.len[i], j = sh.nxt[i];
            sh.len[i] = rest;
            rest -= l;
            sh.nxt[i] = (uint16_t)kRankEnd;
            i = j;
        } while (i != kRankEnd && !split(i));
    }
    __syncthreads();
    for (uint32_t i = tid; i < count; i += kRankThreads) {
        const uint32_t id = i < regs ? first + i : S.regular + b;
        nx_out[id] = sh.nxt[i] == kRankEnd ? kNil : 0u;
        sum_out[id] = sh.len[i];
    }
}

// Samples on their block's primary list put their bytes in place, last first:
// the primary's sum is the cycle length c, a sample's distance from the
// primary is c - its own sum.  A warp takes 32 samples, a lane each for their
// numbers and all lanes for each one's bytes; a stretch longer than `cap` is
// walked again.
template <class T>
__global__ void k_emit(const T *lf, Samples S, uint32_t count, uint32_t cap, const uint32_t *len,
                       const uint32_t *nx, const uint32_t *sum, const uint8_t *kept, uint8_t *out,
                       int32_t *status)
{
    if (chain_failed(status))
        return;
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t i0 = (blockIdx.x * kEw + threadIdx.x) & ~31u; i0 < count; i0 += gridDim.x * kEw) {
        const uint32_t id = i0 + lane;
        uint32_t L = id < count ? len[id] : 0u;
        if (L && nx[id] != kNil)
            L = 0;  // not on the primary's cycle
        uint32_t end = 0;  // the place of the first byte
        if (L) {
            const uint32_t p = S.row_of(id);
            uint32_t s, m;
            block_span(p, S.block, S.n, s, m);
            const uint32_t c = sum[S.regular + p / S.block];
            const uint32_t d = c - sum[id];
            if (c > m || d + L > c) {
                set_status(status, HUFF_ERR_CORRUPT_STREAM);
                L = 0;
            } else {
                end = s + m - 1 - d;
                if (L > cap) {
                    uint32_t r = p - s;
                    for (uint32_t t = 0; t < L; ++t) {
                        const T v = lf[s + r];
                        if (t >= cap)
                            out[end - t] = (uint8_t)v;
                        r = (uint32_t)(v >> 8);
                    }
                    L = cap;
                }
            }
        }
        __syncwarp();
        for (int j = 0; j < 32; j += 4) {  // four at a time: their loads in flight together
            uint32_t Lj[4], ej[4], a[4], b[4];
            const uint8_t *src[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                Lj[q] = __shfl_sync(0xffffffffu, L, j + q);
                ej[q] = __shfl_sync(0xffffffffu, end, j + q);
                src[q] = kept + (uint64_t)(i0 + j + q) * cap + lane;
                a[q] = lane < Lj[q] ? src[q][0] : 0u;
                b[q] = lane + 32 < Lj[q] ? src[q][32] : 0u;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (lane < Lj[q])
                    out[ej[q] - lane] = (uint8_t)a[q];
                if (lane + 32 < Lj[q])
                    out[ej[q] - lane - 32] = (uint8_t)b[q];
                for (uint32_t t = 64; t + lane < Lj[q]; t += 32)
                    out[ej[q] - lane - t] = src[q][t];
            }
        }
    }
}

// A block whose walk closed after c < m rows repeats its last c bytes: a warp per
// piece of a block, `per` of them to one (a CTA per block took 158 us for one
// of 1 MiB, and as much longer as the block).
constexpr uint32_t kFillPiece = 4096;
__global__ void k_periodic_fill(uint8_t *out, uint32_t n, uint32_t block, uint32_t blocks, uint32_t per,
                                uint32_t regular, const uint32_t *sum, const int32_t *status)
{
    if (chain_failed(status))
        return;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t pieces = (uint64_t)blocks * per, warps = (uint64_t)gridDim.x * (kEw / 32);
    for (uint64_t i = (uint64_t)blockIdx.x * (kEw / 32) + (threadIdx.x >> 5); i < pieces; i += warps) {
        const uint32_t b = (uint32_t)(i / per), t0 = (uint32_t)(i - (uint64_t)b * per) * kFillPiece;
        const uint32_t s = b * block, m = n - s < block ? n - s : block;
        const uint32_t c = sum[regular + b];
        const uint32_t end = m < t0 || m - t0 < kFillPiece ? m : t0 + kFillPiece;
        uint32_t t = (t0 > c ? t0 : c) + lane;  // walk steps past the cycle
        uint32_t r = t % c;
        const uint32_t step = 32 % c;
        for (; t < end; t += 32) {
            out[s + m - 1 - t] = out[s + m - 1 - r];
            r += step;
            r = r >= c ? r - c : r;
        }
    }
}

struct InvWs {
    uint32_t *lf, *nxt, *len, *nx2, *sum, *sum2;
    uint64_t *k0, *k1;
    uint32_t *v0, *v1;
    void *radix;
    uint64_t bytes;
};

uint32_t sample_count(uint64_t n, uint32_t block)
{
    const uint32_t gap = sample_gap(n < block ? n : block);
    return (uint32_t)((n + gap - 1) / gap + (n + block - 1) / block);
}

InvWs inv_layout(uint8_t *base, uint64_t n, uint32_t block)
{
    InvWs w;
    uint64_t off = 0;
    const uint64_t S = sample_count(n, block);
    w.lf = carve<uint32_t>(base, off, 4 * n);
    w.nxt = carve<uint32_t>(base, off, 4 * S);
    w.len = carve<uint32_t>(base, off, 4 * S);
    w.nx2 = carve<uint32_t>(base, off, 4 * S);
    w.sum = carve<uint32_t>(base, off, 4 * S);
    w.sum2 = carve<uint32_t>(base, off, 4 * S);
    w.k0 = carve<uint64_t>(base, off, 8 * n);
    w.k1 = carve<uint64_t>(base, off, 8 * n);
    w.v0 = carve<uint32_t>(base, off, 4 * n);
    w.v1 = carve<uint32_t>(base, off, 4 * n);
    w.radix = carve<uint8_t>(base, off, radix_scratch_bytes(n));
    w.bytes = off;
    return w;
}

// The inverse after the primary rows are checked, with LF words in `lf` (w.lf,
// or w.k1 where they are 64 bits wide).  The bytes kept by the walks, at most
// `cap` a sample (a multiple of 8 no larger than a block needs), lie from w.k0
// on: S * cap bytes for the S samples, with a gap of 32 at most 16 n + 512
// blocks of 4 KiB and more, with 64 at most 9 n + 1 KiB (24 n from w.k0 to the
// end of w.v1), with 64-bit words 4 n + 256 blocks (8 n from w.k0 to w.k1).
constexpr uint32_t kKept = 512;

template <class T>
bool invert(InvWs &w, const uint8_t *last, uint32_t n, uint32_t block, uint32_t blocks,
            const uint32_t *d_primary, uint8_t *d_out, int32_t *d_status, T *lf, uint32_t cap,
            cudaStream_t s)
{
    const uint32_t most = n < block ? n : block;  // of a block
    if (most >= kLfTile) {
        const uint32_t per = div_up(most, kLfTile);
        const uint64_t tiles = (uint64_t)blocks * per;
        uint32_t *hist = reinterpret_cast<uint32_t *>(w.k0);  // 1 KiB per tile: at most n / 2 and a block's
        k_lf_count<<<(unsigned)tiles, kLfThreads, 0, s>>>(last, n, block, per, hist);
        if (scan_u32(hist, hist, (uint32_t)(256 * tiles), false, w.v0, nullptr, s) != cudaSuccess)
            return false;
        k_lf_rank<T><<<(unsigned)tiles, kLfThreads, 0, s>>>(last, n, block, per, hist, lf);
    } else {
        k_lf_keys<<<ew_grid(n), kEw, 0, s>>>(last, n, block, w.k0, w.v0);
        bool flip = false;
        if (radix_sort_bits(w.k0, w.v0, w.k1, w.v1, n, 0, 8 + bit_width(blocks - 1), w.radix, s,
                            flip) != cudaSuccess)
            return false;
        k_lf_scatter<<<ew_grid(n), kEw, 0, s>>>(flip ? w.k1 : w.k0, flip ? w.v1 : w.v0, n, block,
                                                w.lf);  // (blocks this short have 32-bit words)
    }
    if (cap > ((most + 7) & ~7u))
        cap = (most + 7) & ~7u;
    uint8_t *const kept = reinterpret_cast<uint8_t *>(w.k0);
    Samples S;
    S.n = n;
    S.block = block;
    S.gap = sample_gap(most);
    S.regular = (uint32_t)(((uint64_t)n + S.gap - 1) / S.gap);
    S.primary = d_primary;
    const uint32_t count = sample_count(n, block);
    k_walk<T><<<ew_grid(count), kEw, 0, s>>>(lf, S, count, cap, w.nxt, w.len, kept, d_status);
    uint32_t *nx = w.nxt, *sm = w.len;
    if (S.gap == 32) {
        static KernelSetup setup;
        int per_sm = 0;
        if (kernel_setup(setup, (const void *)k_rank, kRankThreads, sizeof(RankShared), &per_sm) !=
            cudaSuccess)
            return false;
        k_rank<<<blocks, kRankThreads, sizeof(RankShared), s>>>(w.nxt, w.len, S, w.nx2, w.sum,
                                                                d_status);
        nx = w.nx2;
        sm = w.sum;
    } else {
        // the longest list is one block's samples
        const uint64_t per_block = (uint64_t)most / S.gap + 2;
        const uint32_t rounds = bit_width(per_block) + 1;
        uint32_t *nx_o = w.nx2, *sm_o = w.sum;
        for (uint32_t r = 0; r < rounds; ++r) {
            k_jump<<<ew_grid(count), kEw, 0, s>>>(nx, sm, count, nx_o, sm_o, d_status);
            if (r == 0) {  // len stays; later steps ping-pong between sum and sum2
                nx = nx_o;
                sm = sm_o;
                nx_o = w.nxt;
                sm_o = w.sum2;
            } else {
                uint32_t *t = nx;
                nx = nx_o;
                nx_o = t;
                t = sm;
                sm = sm_o;
                sm_o = t;
            }
        }
    }
    k_emit<T><<<ew_grid(count), kEw, 0, s>>>(lf, S, count, cap, w.len, nx, sm, kept, d_out, d_status);
    const uint32_t per = div_up(most, kFillPiece);
    k_periodic_fill<<<ew_grid((uint64_t)blocks * per * 32), kEw, 0, s>>>(d_out, n, block, blocks, per,
                                                                         S.regular, sm, d_status);
    return true;
}

bool bwt_args_ok(uint64_t n, uint32_t block)
{
    return block >= 1 && n <= HUFF_BWT_MAX_N;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

__global__ void k_m3_header(uint8_t *out, uint64_t n, uint32_t block, uint32_t count,
                            uint32_t stages, uint32_t head)
{
    for (uint32_t i = threadIdx.x; i < head; i += blockDim.x) {
        if (i < 8)
            out[i] = (uint8_t)(n >> (8 * i));
        else if (i < 12)
            out[i] = (uint8_t)(block >> (8 * (i - 8)));
        else if (i < 16)
            out[i] = (uint8_t)(count >> (8 * (i - 12)));
        else if (i < 20)
            out[i] = (uint8_t)(stages >> (8 * (i - 16)));
        else if (i >= 20 + 4 * count)
            out[i] = 0;
    }
}

__global__ void k_add_u64(unsigned long long *p, uint64_t v, const int32_t *status)
{
    if (!chain_failed(status))
        *p += v;
}

uint32_t m3_head_bytes(uint64_t count) { return (uint32_t)((20 + 4 * count + 15) & ~15ull); }

uint64_t max3(uint64_t a, uint64_t b, uint64_t c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }

}  // namespace
}  // namespace huff

using namespace huff;

extern "C" {

uint64_t huff_bwt_workspace_size(uint64_t n, uint32_t block)
{
    if (!bwt_args_ok(n, block))
        return 0;
    const uint64_t f = fwd_layout(nullptr, n).bytes;
    const uint64_t i = inv_layout(nullptr, n, block).bytes;
    return f > i ? f : i;
}

huff_status_t huff_bwt_forward(const uint8_t *d_in, uint64_t n, uint32_t block, uint8_t *d_last,
                               uint32_t *d_primary, void *d_ws, uint64_t ws_bytes,
                               int32_t *d_status, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_bwt_forward");
    if (!bwt_args_ok(n, block) || !d_status || (n && (!d_in || !d_last || !d_primary || !d_ws)) ||
        (n && ws_bytes < huff_bwt_workspace_size(n, block)) || (d_ws && !aligned16(d_ws)))
        return HUFF_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess)
        return HUFF_ERR_CUDA;
    if (n == 0)
        return HUFF_OK;
    const uint32_t N = (uint32_t)n;
    FwdWs w = fwd_layout(static_cast<uint8_t *>(d_ws), n);
    const uint64_t blocks = (n + block - 1) / block;
    const uint64_t mmax = n < block ? n : block;
    // byte counts (in the workspace's first 2 KiB, not in use yet)
    auto *hist = static_cast<unsigned long long *>(d_ws);
    const uint32_t lead = (uint32_t)(0u - reinterpret_cast<uintptr_t>(d_in)) & 15u;
    const uint32_t head = lead < N ? lead : N;
    unsigned long long h_hist[256];
    if (launch_histogram(d_in + head, n - head, hist, nullptr, s) != cudaSuccess)
        return HUFF_ERR_CUDA;
    if (head)
        k_count_head<<<1, 32, 0, s>>>(d_in, head, hist);
    if (cudaMemcpyAsync(h_hist, hist, sizeof(h_hist), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return HUFF_ERR_CUDA;
    const FirstKey f = first_key(h_hist, n, blocks, mmax);
    k_bwt_init<<<ew_grid((n + 7) / 8), kEw, 0, s>>>(d_in, N, block, f, w.k0);
    bool flip = false;
    if (radix_sort_bits(w.k0, w.v0, w.k1, w.v1, N, 0, f.by_block ? f.bits : f.bits + bit_width(blocks - 1),
                        f.by_block ? w.rk : w.radix, s, flip, f.by_block ? block : 0, true) != cudaSuccess)
        return HUFF_ERR_CUDA;
    uint64_t *ks = flip ? w.k1 : w.k0;
    uint32_t *vs = flip ? w.v1 : w.v0;
    // the sorted indices are the first SA: the arrays change places
    (flip ? w.v1 : w.v0) = w.sa;
    w.sa = vs;
    uint32_t n_act = 0, groups = 0;
    if (refine(w, ks, vs, N, 64, s, n_act, groups) != cudaSuccess)
        return HUFF_ERR_CUDA;
    for (uint64_t h = f.q; n_act > 0 && h < mmax; h *= 2) {
        const uint32_t lo_bits = bit_width(mmax - 1);
        if (launch_chained(k_bwt_round_keys, ew_grid(n_act), kEw, 0, s, w.sa, w.rk, w.act, w.grp, n_act, N,
                           block, h, lo_bits, w.k0, w.v0) != cudaSuccess)
            return HUFF_ERR_CUDA;
        if (sort_groups(w, n_act, lo_bits, lo_bits + bit_width(groups - 1), s, ks, vs) != cudaSuccess)
            return HUFF_ERR_CUDA;
        if (refine(w, ks, vs, n_act, lo_bits, s, n_act, groups) != cudaSuccess)
            return HUFF_ERR_CUDA;
    }
    if (launch_chained(k_bwt_output, ew_grid(n), kEw, 0, s, d_in, w.sa, N, block, d_last, d_primary) !=
        cudaSuccess)
        return HUFF_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

huff_status_t huff_bwt_inverse(const uint8_t *d_last, uint64_t n, uint32_t block,
                               const uint32_t *d_primary, uint8_t *d_out, void *d_ws,
                               uint64_t ws_bytes, int32_t *d_status, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_bwt_inverse");
    if (!bwt_args_ok(n, block) || !d_status || (n && (!d_last || !d_primary || !d_out || !d_ws)) ||
        (n && ws_bytes < huff_bwt_workspace_size(n, block)) || (d_ws && !aligned16(d_ws)))
        return HUFF_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess)
        return HUFF_ERR_CUDA;
    if (n == 0)
        return HUFF_OK;
    const uint32_t N = (uint32_t)n;
    InvWs w = inv_layout(static_cast<uint8_t *>(d_ws), n, block);
    const uint32_t blocks = (uint32_t)((n + block - 1) / block);
    k_check_primary<<<ew_grid(blocks), kEw, 0, s>>>(d_primary, N, block, blocks, d_status);
    const bool wide = block > kMaxBlock32 && n > kMaxBlock32;
    const bool ok = wide ? invert(w, d_last, N, block, blocks, d_primary, d_out, d_status,
                                  reinterpret_cast<uint64_t *>(w.k1), kKept / 2, s)
                         : invert(w, d_last, N, block, blocks, d_primary, d_out, d_status, w.lf, kKept,
                                  s);
    if (!ok)
        return HUFF_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

uint64_t huff_m3_max_size(uint64_t n, uint32_t block, uint64_t segment_bytes,
                          uint32_t chunk_symbols)
{
    if (!bwt_args_ok(n, block))
        return 0;
    const uint64_t seg = huff_segmented_max_size(n, segment_bytes, chunk_symbols);
    return seg ? m3_head_bytes((n + block - 1) / block) + seg : 0;
}

uint64_t huff_m3_workspace_size(uint64_t n, uint32_t block, uint64_t segment_bytes,
                                uint32_t chunk_symbols)
{
    if (!bwt_args_ok(n, block))
        return 0;
    const uint64_t seg = huff_segmented_workspace_size(n, segment_bytes, chunk_symbols);
    if (!seg)
        return 0;
    return ((n + 255) & ~255ull) +
           max3(huff_bwt_workspace_size(n, block), seg, huff_mtf_workspace_size(n, block));
}

huff_status_t huff_m3_compress(const uint8_t *d_in, uint64_t n, uint32_t block,
                               uint64_t segment_bytes, uint32_t chunk_symbols, uint32_t stages,
                               uint8_t *d_out, uint64_t out_cap, uint64_t *d_out_bytes,
                               void *d_ws, uint64_t ws_bytes, int32_t *d_status,
                               huff_stream_t stream)
{
    HUFF_API_RANGE("huff_m3_compress");
    const uint64_t need = huff_m3_workspace_size(n, block, segment_bytes, chunk_symbols);
    const uint64_t count = block ? (n + block - 1) / block : 0;
    const uint32_t head = m3_head_bytes(count);
    if (!need || !d_out || !d_out_bytes || !d_status || !d_ws || ws_bytes < need ||
        out_cap < head || (n && !d_in) || !aligned16(d_out) || !aligned16(d_ws) ||
        (stages & ~HUFF_M3_MTF))
        return HUFF_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    uint8_t *ws = static_cast<uint8_t *>(d_ws);
    uint8_t *last = ws;
    uint8_t *rest = ws + ((n + 255) & ~255ull);
    const uint64_t rest_bytes = ws_bytes - (uint64_t)(rest - ws);
    huff_status_t st = huff_bwt_forward(d_in, n, block, last,
                                        reinterpret_cast<uint32_t *>(d_out + 20), rest, rest_bytes,
                                        d_status, stream);
    if (st == HUFF_OK && (stages & HUFF_M3_MTF))
        st = huff_mtf_forward(last, n, block, last, rest, rest_bytes, stream);
    if (st != HUFF_OK)
        return st;
    k_m3_header<<<1, 256, 0, s>>>(d_out, n, block, (uint32_t)count, stages, head);
    if (cudaGetLastError() != cudaSuccess)
        return HUFF_ERR_CUDA;
    // the transform's workspace is free again: what the coder's leaves of it
    // holds the batch's block, so that nothing is allocated
    const uint64_t seg_ws =
        (huff_segmented_workspace_size(n, segment_bytes, chunk_symbols) + 255) & ~255ull;
    st = segmented_compress(last, n, segment_bytes, chunk_symbols, d_out + head, out_cap - head,
                            d_out_bytes, rest, rest_bytes, d_status, s,
                            seg_ws < rest_bytes ? rest + seg_ws : nullptr,
                            seg_ws < rest_bytes ? rest_bytes - seg_ws : 0);
    if (st != HUFF_OK)
        return st;
    k_add_u64<<<1, 1, 0, s>>>(reinterpret_cast<unsigned long long *>(d_out_bytes), head, d_status);
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

uint64_t huff_m3_decompress_workspace_size(uint64_t n, uint32_t block)
{
    if (!bwt_args_ok(n, block))
        return 0;
    const uint64_t b = huff_bwt_workspace_size(n, block), m = huff_mtf_workspace_size(n, block);
    return ((n + 255) & ~255ull) + (b > m ? b : m);
}

huff_status_t huff_m3_decompress(const uint8_t *d_in, uint64_t in_bytes, uint8_t *d_out,
                                 uint64_t out_cap, uint64_t *d_n, void *d_ws, uint64_t ws_bytes,
                                 int32_t *d_status, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_m3_decompress");
    if (!d_in || !d_n || !d_status || !aligned16(d_in) || (d_ws && !aligned16(d_ws)))
        return HUFF_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess)
        return HUFF_ERR_CUDA;
    uint8_t h[20];
    uint64_t n = 0;
    uint32_t block = 0, count = 0, stages = 0;
    bool ok = in_bytes >= 20;
    if (ok) {
        if (cudaMemcpyAsync(h, d_in, 20, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return HUFF_ERR_CUDA;
        for (int i = 7; i >= 0; --i)
            n = (n << 8) | h[i];
        for (int i = 11; i >= 8; --i)
            block = (block << 8) | h[i];
        for (int i = 15; i >= 12; --i)
            count = (count << 8) | h[i];
        for (int i = 19; i >= 16; --i)
            stages = (stages << 8) | h[i];
        ok = block >= 1 && n <= HUFF_BWT_MAX_N && count == (n + block - 1) / block &&
             (stages & ~HUFF_M3_MTF) == 0 && 20 + 4ull * count <= in_bytes &&
             m3_head_bytes(count) <= in_bytes;
    }
    if (!ok) {
        static const int32_t corrupt = HUFF_ERR_CORRUPT_STREAM;
        if (cudaMemcpyAsync(d_status, &corrupt, 4, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return HUFF_ERR_CUDA;
        return HUFF_OK;
    }
    if (n > out_cap) {
        static const int32_t cap = HUFF_ERR_CAPACITY;
        if (cudaMemcpyAsync(d_status, &cap, 4, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return HUFF_ERR_CUDA;
        return HUFF_OK;
    }
    if (!d_out || !d_ws || ws_bytes < huff_m3_decompress_workspace_size(n, block))
        return HUFF_ERR_INVALID_ARG;
    const uint32_t head = m3_head_bytes(count);
    uint8_t *ws = static_cast<uint8_t *>(d_ws);
    uint8_t *last = ws;
    uint8_t *rest = ws + ((n + 255) & ~255ull);
    const uint64_t rest_bytes = ws_bytes - (uint64_t)(rest - ws);
    huff_status_t st = segmented_decompress(d_in + head, in_bytes - head, last, n, d_n, d_status, s,
                                            rest, rest_bytes);
    if (st != HUFF_OK)
        return st;
    // the segmented container must hold exactly n bytes
    uint64_t got = 0;
    int32_t sst = 0;
    if (cudaMemcpyAsync(&got, d_n, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(&sst, d_status, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return HUFF_ERR_CUDA;
    if (sst != 0)
        return HUFF_OK;  // the segment error stays in *d_status
    if (got != n) {
        static const int32_t corrupt = HUFF_ERR_CORRUPT_STREAM;
        if (cudaMemcpyAsync(d_status, &corrupt, 4, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return HUFF_ERR_CUDA;
        return HUFF_OK;
    }
    if (stages & HUFF_M3_MTF) {
        st = huff_mtf_inverse(last, n, block, last, rest, rest_bytes, stream);
        if (st != HUFF_OK)
            return st;
    }
    return huff_bwt_inverse(last, n, block, reinterpret_cast<const uint32_t *>(d_in + 20), d_out,
                            rest, rest_bytes, d_status, stream);
}

}  // extern "C"
