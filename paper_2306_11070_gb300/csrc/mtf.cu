// Move-to-front coding per block: the optional second stage of Method 3
// (Section III-A; Burrows and Wheeler 1994, Section 4).  Every block starts
// from the list 0..255; a byte is coded as its position in the list and then
// moved to the front.
//
// Blocks are cut into 1 KiB segments, and the list a segment starts from is
// found without running the blocks serially:
//  - forward: the list at the end of a segment is the segment's distinct
//    bytes, latest occurrence first, followed by the rest of the list it
//    started from in their old order.  k_mtf_distinct (a warp per segment)
//    writes every segment's distinct bytes; the list kernels chain them into
//    every segment's starting list (256 bytes per segment); k_mtf_encode
//    codes each segment, a thread each, from its own starting list.
//  - inverse: decoding a segment from the identity list gives, for every
//    position, the index of its byte in the real starting list, and the
//    final list as a permutation of the starting one.  k_mtf_decode_rel does
//    that per segment; the list kernels compose the permutations into every
//    segment's starting list; k_mtf_map replaces each relative byte by the
//    real one.
// Chaining is associative, so blocks of more than kSuper segments chain in
// three steps: every run of kSuper segments by itself (its result kept in the
// list slot of its last segment, which the third step fills last), then the
// runs of a block (the list each run starts from, into the slot of its first
// segment), then every run's segments from there.
// A coding thread keeps the first 16 entries of its list in registers, four
// to a word, and the others in a shared-memory column of words ([word][thread]):
// a byte is found by a zero-byte test of each word, and moved to the front by
// shifting words by a byte under a mask, so the lanes of a warp run the same
// straight line unless a byte lies beyond the 16th entry.
#include "api_trace.h"
#include "huff_internal.cuh"

namespace huff {
namespace {

constexpr uint32_t kSeg = 1024;    // bytes per segment
constexpr int kMtfThreads = 128;   // threads (segments) per CTA of the coding kernels
constexpr int kListWarps = 4;      // warps per CTA of the warp-wide kernels
constexpr uint32_t kSuper = 32;    // segments chained by one warp
constexpr uint32_t kFull = 0xffffffffu;

struct Segs {
    uint64_t n;
    uint32_t block;
    uint32_t per_block;  // segments of a whole block
    uint64_t count;      // segments in all
    __host__ __device__ uint64_t start(uint64_t g) const
    {
        return (g / per_block) * block + (g % per_block) * (uint64_t)kSeg;
    }
    // bytes of segment g (0 past the end of a short last block)
    __host__ __device__ uint32_t len(uint64_t g) const
    {
        const uint64_t bs = (g / per_block) * block;
        const uint64_t be = bs + block < n ? bs + block : n;
        const uint64_t s = start(g);
        if (s >= be)
            return 0;
        return (uint32_t)(be - s < kSeg ? be - s : kSeg);
    }
};

Segs make_segs(uint64_t n, uint32_t block)
{
    Segs S;
    S.n = n;
    S.block = block;
    S.per_block = (block + kSeg - 1) / kSeg;
    const uint64_t blocks = (n + block - 1) / block;
    S.count = blocks * S.per_block;
    return S;
}

// The distinct bytes of every segment, latest occurrence first: one warp per
// segment notes the last position of every byte value (only ends of runs
// compete for a value), then walks the positions backwards and keeps those.
__global__ void __launch_bounds__(kListWarps * 32) k_mtf_distinct(const uint8_t *in, Segs S,
                                                                  uint8_t *dist, uint32_t *dcount)
{
    __shared__ uint32_t last_of[kListWarps][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t *last = last_of[w];
    for (uint64_t g = (uint64_t)blockIdx.x * kListWarps + w; g < S.count;
         g += (uint64_t)gridDim.x * kListWarps) {
        const uint8_t *x = in + S.start(g);
        const uint32_t L = S.len(g);
        for (int i = lane; i < 256; i += 32)
            last[i] = 0;
        __syncwarp();
        for (uint32_t i = lane; i < L; i += 32) {
            const uint32_t c = x[i];
            if (i + 1 == L || x[i + 1] != c)
                atomicMax(last + c, i + 1);
        }
        __syncwarp();
        uint32_t k = 0;
        for (uint32_t top = L; top > 0; top -= top < 32 ? top : 32) {
            const bool in_range = (uint32_t)lane < top;
            const uint32_t i = top - 1 - lane;
            const uint32_t c = in_range ? x[i] : 0u;
            const bool keep = in_range && last[c] == i + 1;
            const uint32_t b = __ballot_sync(kFull, keep);
            if (keep)
                dist[g * 256 + k + __popc(b & ((1u << lane) - 1u))] = (uint8_t)c;
            k += __popc(b);
        }
        if (lane == 0)
            dcount[g] = k;
        __syncwarp();
    }
}

// One warp's list with room for the next one; entries in order.
struct ListPair {
    uint8_t lst[2][256];
    uint32_t stamp[256];  // the step that last met a byte value
};

// lst[cur ^ 1] = the k bytes of `d`, then the other bytes of lst[cur] in
// their order.  e0, e1: d[lane], d[lane + 32], loaded ahead.  `step` differs
// between calls and is never 0.
__device__ __forceinline__ void push_front(ListPair &P, int &cur, const uint8_t *d, uint32_t k,
                                           uint32_t e0, uint32_t e1, uint32_t step, int lane)
{
    uint8_t *const now = P.lst[cur], *const nxt = P.lst[cur ^ 1];
    reinterpret_cast<uint2 *>(nxt)[lane] = reinterpret_cast<const uint2 *>(now)[lane];
    for (uint32_t i = lane; i < k; i += 32)
        P.stamp[i < 32 ? e0 : i < 64 ? e1 : d[i]] = step;
    __syncwarp();
    for (uint32_t i = lane; i < k; i += 32)
        nxt[i] = (uint8_t)(i < 32 ? e0 : i < 64 ? e1 : d[i]);
    // entries past the last one taken stay where they are
    uint32_t at = k, taken = 0;
    for (uint32_t i = lane; taken < k && i < 256; i += 32) {
        const uint32_t c = now[i];
        const uint32_t b = __ballot_sync(kFull, P.stamp[c] != step);
        if ((b >> lane) & 1u)
            nxt[at + __popc(b & ((1u << lane) - 1u))] = (uint8_t)c;
        at += __popc(b);
        taken += 32 - __popc(b);
    }
    __syncwarp();
    cur ^= 1;
}

// Forward step 1: the distinct bytes of every kSuper segments, latest first,
// into the list slot of the last of them; the entries past their number
// repeat the first.
__global__ void __launch_bounds__(kListWarps * 32)
    k_mtf_supers(const uint8_t *dist, const uint32_t *dcount, Segs S, uint32_t supers,
                 uint64_t total, uint8_t *lists)
{
    __shared__ __align__(16) uint8_t acc[kListWarps][256];
    __shared__ __align__(16) uint8_t seen[kListWarps][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t v = (uint64_t)blockIdx.x * kListWarps + w;
    if (v >= total)
        return;
    const uint64_t first = (v / supers) * S.per_block + (v % supers) * kSuper;
    const uint64_t left = S.per_block - (v % supers) * kSuper;
    const uint32_t cnt = left < kSuper ? (uint32_t)left : kSuper;
    reinterpret_cast<uint2 *>(seen[w])[lane] = make_uint2(0, 0);
    __syncwarp();
    uint32_t k = 0;
    uint32_t nk = dcount[first + cnt - 1];
    for (uint32_t j = cnt; j-- > 0;) {
        const uint64_t g = first + j;
        const uint32_t dk = nk;
        if (j)
            nk = dcount[g - 1];
        for (uint32_t i0 = 0; i0 < dk; i0 += 32) {
            const bool has = i0 + lane < dk;
            const uint32_t c = has ? dist[g * 256 + i0 + lane] : 0u;
            const bool add = has && !seen[w][c];
            const uint32_t b = __ballot_sync(kFull, add);
            if (add) {
                acc[w][k + __popc(b & ((1u << lane) - 1u))] = (uint8_t)c;
                seen[w][c] = 1;
            }
            k += __popc(b);
            __syncwarp();
        }
    }
    if (k == 0)  // past the end of a short last block
        return;
    for (uint32_t i = k + lane; i < 256; i += 32)
        acc[w][i] = acc[w][0];
    __syncwarp();
    reinterpret_cast<uint2 *>(lists + (first + cnt - 1) * 256)[lane] =
        reinterpret_cast<const uint2 *>(acc[w])[lane];
}

// Forward step 2, one warp per block: the list each run of kSuper segments
// starts from, into the slot of its first segment.  L_0 = 0..255.
__global__ void __launch_bounds__(kListWarps * 32)
    k_mtf_chain_supers(Segs S, uint32_t supers, uint64_t blocks, uint8_t *lists)
{
    __shared__ __align__(16) ListPair pair[kListWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t b = (uint64_t)blockIdx.x * kListWarps + w;
    if (b >= blocks)
        return;
    ListPair &P = pair[w];
    for (int i = lane; i < 256; i += 32) {
        P.lst[0][i] = (uint8_t)i;
        P.stamp[i] = 0;
    }
    int cur = 0;
    __syncwarp();
    for (uint32_t v = 0; v < supers; ++v) {
        const uint64_t first = b * S.per_block + (uint64_t)v * kSuper;
        const uint64_t end = v + 1 < supers ? first + kSuper : (b + 1) * S.per_block;
        const uint8_t *d = lists + (end - 1) * 256;
        const bool any = S.len(first) != 0;
        uint32_t k = 0, e0 = 0, e1 = 0;
        if (any && v + 1 < supers) {  // their number: up to where the first repeats
            e0 = d[lane];
            e1 = d[lane + 32];
            const uint32_t f = __shfl_sync(kFull, e0, 0);
            k = 256;
            for (uint32_t i = lane; i < 256; i += 32) {
                const uint32_t c = i < 32 ? e0 : i < 64 ? e1 : d[i];
                const uint32_t same = __ballot_sync(kFull, c == f && i > 0);
                if (same) {
                    k = (i & ~31u) + __ffs(same) - 1;
                    break;
                }
            }
        }
        reinterpret_cast<uint2 *>(lists + first * 256)[lane] =
            reinterpret_cast<const uint2 *>(P.lst[cur])[lane];
        if (k)
            push_front(P, cur, d, k, e0, e1, v + 1, lane);
    }
}

// Forward step 3, one warp per run of kSuper segments: the list every segment
// starts from.  from_slot: the run's own starting list is in the slot of its
// first segment (else it is 0..255).
__global__ void __launch_bounds__(kListWarps * 32)
    k_mtf_lists(const uint8_t *dist, const uint32_t *dcount, Segs S, uint32_t supers, uint64_t total,
                bool from_slot, uint8_t *lists)
{
    __shared__ __align__(16) ListPair pair[kListWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t v = (uint64_t)blockIdx.x * kListWarps + w;
    if (v >= total)
        return;
    ListPair &P = pair[w];
    const uint64_t first = (v / supers) * S.per_block + (v % supers) * kSuper;
    const uint64_t left = S.per_block - (v % supers) * kSuper;
    const uint32_t cnt = left < kSuper ? (uint32_t)left : kSuper;
    for (int i = lane; i < 256; i += 32) {
        P.lst[0][i] = from_slot ? lists[first * 256 + i] : (uint8_t)i;
        P.stamp[i] = 0;
    }
    int cur = 0;
    uint32_t k = dcount[first], e0 = dist[first * 256 + lane], e1 = dist[first * 256 + 32 + lane];
    __syncwarp();
    for (uint32_t j = 0; j < cnt; ++j) {
        const uint64_t g = first + j;
        reinterpret_cast<uint2 *>(lists + g * 256)[lane] =
            reinterpret_cast<const uint2 *>(P.lst[cur])[lane];
        if (j + 1 == cnt)
            break;
        const uint32_t k0 = k, a0 = e0, a1 = e1;
        k = dcount[g + 1];  // the next segment's, loaded ahead
        e0 = dist[(g + 1) * 256 + lane];
        e1 = dist[(g + 1) * 256 + 32 + lane];
        if (k0)
            push_front(P, cur, dist + g * 256, k0, a0, a1, j + 1, lane);
    }
}

constexpr int kRegWords = 4;  // list words in registers

// A thread's list: words 0..3 in registers, word i >= 4 at col[i * kMtfThreads].
struct List {
    uint32_t w[kRegWords];
    uint32_t *col;
};

__device__ __forceinline__ uint32_t splat(uint32_t c) { return __byte_perm(c, 0u, 0u); }
// the top bit of the lowest zero byte of x (and perhaps of bytes above it); 0
// when no byte is zero
__device__ __forceinline__ uint32_t zero_byte(uint32_t x)
{
    return (x - 0x01010101u) & ~x & 0x80808080u;
}

// The position of byte c in the list, and c moved to the front.
__device__ __forceinline__ uint32_t find_and_move(List &l, uint32_t c)
{
    const uint32_t c4 = splat(c);
    uint32_t in = c << 24, j = 0;  // in: the byte shifted into the next word, on top
    bool found = false;
#pragma unroll
    for (int i = 0; i < kRegWords; ++i) {
        const uint32_t v = l.w[i], z = zero_byte(v ^ c4);
        // the bytes up to c's, all of a word without it, none after it
        const uint32_t m = found ? 0u : z ^ (z - 1u);
        if (!found && z)
            j = 4 * i + ((uint32_t)(__ffs(z) - 1) >> 3);
        found = found || z;
        l.w[i] = (v & ~m) | (__funnelshift_l(in, v, 8) & m);
        in = v;
    }
    if (!found) {
        for (uint32_t i = kRegWords; i < 64; ++i) {
            const uint32_t v = l.col[i * kMtfThreads], z = zero_byte(v ^ c4);
            const uint32_t m = z ^ (z - 1u);
            l.col[i * kMtfThreads] = (v & ~m) | (__funnelshift_l(in, v, 8) & m);
            in = v;
            if (z) {
                j = 4 * i + ((uint32_t)(__ffs(z) - 1) >> 3);
                break;
            }
        }
    }
    return j;
}

// The byte at position j of the list, and it moved to the front.
__device__ __forceinline__ uint32_t take_and_move(List &l, uint32_t j)
{
    const uint32_t at = j >> 2;
    uint32_t word = at == 0 ? l.w[0] : at == 1 ? l.w[1] : at == 2 ? l.w[2] : l.w[3];
    if (at >= kRegWords)
        word = l.col[at * kMtfThreads];
    const uint32_t c = (word >> (8 * (j & 3u))) & 0xffu;
    const int bits = 8 * (int)(j + 1);
    uint32_t in = c << 24;
#pragma unroll
    for (int i = 0; i < kRegWords; ++i) {
        const uint32_t v = l.w[i];
        const int s = bits - 32 * i;
        const uint32_t m = __funnelshift_lc(kFull, 0u, s > 0 ? (uint32_t)s : 0u);  // low s bits
        l.w[i] = (v & ~m) | (__funnelshift_l(in, v, 8) & m);
        in = v;
    }
    for (uint32_t i = kRegWords; i <= at; ++i) {
        const uint32_t v = l.col[i * kMtfThreads];
        const uint32_t m = __funnelshift_lc(kFull, 0u, (uint32_t)bits - 32 * i);
        l.col[i * kMtfThreads] = (v & ~m) | (__funnelshift_l(in, v, 8) & m);
        in = v;
    }
    return c;
}

// Run f over the bytes of one segment, 16 at a time where `vec` says that
// they are aligned; out may be in.
template <class F>
__device__ __forceinline__ void map_bytes(const uint8_t *x, uint8_t *y, uint32_t L, bool vec, F f)
{
    uint32_t i = 0;
    if (vec) {
        uint4 next = L >= 16 ? *reinterpret_cast<const uint4 *>(x) : make_uint4(0, 0, 0, 0);
        for (; i + 16 <= L; i += 16) {
            const uint4 v = next;
            if (i + 32 <= L)
                next = *reinterpret_cast<const uint4 *>(x + i + 16);
            uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                uint32_t r = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    r |= f((q[a] >> (8 * b)) & 0xffu) << (8 * b);
                q[a] = r;
            }
            *reinterpret_cast<uint4 *>(y + i) = make_uint4(q[0], q[1], q[2], q[3]);
        }
    }
    // else eight at a time: straight-line code for several bytes overlaps their
    // steps, a byte's turn by itself takes half as long again
    for (; i + 8 <= L; i += 8) {
        uint32_t q[8];
#pragma unroll
        for (int b = 0; b < 8; ++b)
            q[b] = x[i + b];
#pragma unroll
        for (int b = 0; b < 8; ++b)
            y[i + b] = (uint8_t)f(q[b]);
    }
    for (; i < L; ++i)
        y[i] = (uint8_t)f(x[i]);
}

// Code each segment from its starting list.  Issue bound, about 45
// instructions a byte and a word-wise walk for the lanes beyond the 16th entry:
// 64 MiB of transformed text 1.80 -> 0.49 ms (before: a byte-wise walk of the
// list in shared memory, whose length the slowest lane of the warp set).  The
// whole stage, chaining included, took 3.08 -> 0.71 ms forward and 2.68 ->
// 0.45 ms back in 1 MiB blocks, 13.9 -> 0.79 and 9.0 -> 0.42 ms for one 16
// MiB block (before: one warp chained a block's segments).
__global__ void __launch_bounds__(kMtfThreads) k_mtf_encode(const uint8_t *in, Segs S,
                                                            const uint8_t *lists, uint8_t *out,
                                                            bool vec)
{
    __shared__ uint32_t cols[64 * kMtfThreads];  // [word][thread]
    const uint64_t g = (uint64_t)blockIdx.x * kMtfThreads + threadIdx.x;
    if (g >= S.count)
        return;
    List l;
    l.col = cols + threadIdx.x;
    const uint4 *src = reinterpret_cast<const uint4 *>(lists + g * 256);
    const uint4 head = src[0];
    l.w[0] = head.x, l.w[1] = head.y, l.w[2] = head.z, l.w[3] = head.w;
    for (int i = 1; i < 16; ++i) {
        const uint4 v = src[i];
        l.col[(4 * i) * kMtfThreads] = v.x;
        l.col[(4 * i + 1) * kMtfThreads] = v.y;
        l.col[(4 * i + 2) * kMtfThreads] = v.z;
        l.col[(4 * i + 3) * kMtfThreads] = v.w;
    }
    map_bytes(in + S.start(g), out + S.start(g), S.len(g), vec,
              [&](uint32_t c) { return find_and_move(l, c); });
}

// Decode each segment from the identity list: relative bytes and the final
// list (as indices into the starting list).
__global__ void __launch_bounds__(kMtfThreads) k_mtf_decode_rel(const uint8_t *in, Segs S,
                                                                uint8_t *rel, uint8_t *fin, bool vec)
{
    __shared__ uint32_t cols[64 * kMtfThreads];
    const uint64_t g = (uint64_t)blockIdx.x * kMtfThreads + threadIdx.x;
    if (g >= S.count)
        return;
    List l;
    l.col = cols + threadIdx.x;
    for (int i = 0; i < 64; ++i) {
        const uint32_t v = 0x03020100u + 0x04040404u * (uint32_t)i;
        if (i < kRegWords)
            l.w[i & (kRegWords - 1)] = v;
        else
            l.col[i * kMtfThreads] = v;
    }
    map_bytes(in + S.start(g), rel + S.start(g), S.len(g), vec,
              [&](uint32_t j) { return take_and_move(l, j); });
    uint4 *dst = reinterpret_cast<uint4 *>(fin + g * 256);
    dst[0] = make_uint4(l.w[0], l.w[1], l.w[2], l.w[3]);
    for (int i = 1; i < 16; ++i)
        dst[i] = make_uint4(l.col[(4 * i) * kMtfThreads], l.col[(4 * i + 1) * kMtfThreads],
                            l.col[(4 * i + 2) * kMtfThreads], l.col[(4 * i + 3) * kMtfThreads]);
}

// One step of the inverse lists: L_{j+1}[i] = L_j[F_j[i]], lane's eight
// entries of F_j in f; lst[cur] holds L_j, then L_{j+1}.
__device__ __forceinline__ void apply(uint8_t (*lst)[256], int &cur, uint2 f, int lane)
{
    uint32_t r[2] = {0, 0};
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const uint32_t i = ((t < 4 ? f.x : f.y) >> (8 * (t & 3))) & 0xffu;
        r[t >> 2] |= (uint32_t)lst[cur][i] << (8 * (t & 3));
    }
    reinterpret_cast<uint2 *>(lst[cur ^ 1])[lane] = make_uint2(r[0], r[1]);
    __syncwarp();
    cur ^= 1;
}

// cnt segments' permutations from `f` on, one after the other, the next
// loaded ahead; every list before its step goes to `out` where given.
__device__ __forceinline__ void compose(uint8_t (*lst)[256], int &cur, const uint8_t *f,
                                        uint32_t cnt, uint8_t *out, int lane)
{
    uint2 next = reinterpret_cast<const uint2 *>(f)[lane];
    for (uint32_t j = 0; j < cnt; ++j) {
        const uint2 v = next;
        if (j + 1 < cnt)
            next = reinterpret_cast<const uint2 *>(f + (j + 1) * 256)[lane];
        if (out)
            reinterpret_cast<uint2 *>(out + j * 256)[lane] =
                reinterpret_cast<const uint2 *>(lst[cur])[lane];
        apply(lst, cur, v, lane);
    }
}

__device__ __forceinline__ void identity(uint8_t *lst, int lane)
{
    const uint32_t b = 0x03020100u + 0x08080808u * (uint32_t)lane;
    reinterpret_cast<uint2 *>(lst)[lane] = make_uint2(b, b + 0x04040404u);
}

// Inverse step 1: the composition of every kSuper segments' permutations,
// into the list slot of the last of them.  (A segment without bytes has the
// identity.)
__global__ void __launch_bounds__(kListWarps * 32)
    k_mtf_supers_inv(const uint8_t *fin, Segs S, uint32_t supers, uint64_t total, uint8_t *lists)
{
    __shared__ __align__(16) uint8_t lst[kListWarps][2][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t v = (uint64_t)blockIdx.x * kListWarps + w;
    if (v >= total)
        return;
    const uint64_t first = (v / supers) * S.per_block + (v % supers) * kSuper;
    const uint64_t left = S.per_block - (v % supers) * kSuper;
    const uint32_t cnt = left < kSuper ? (uint32_t)left : kSuper;
    identity(lst[w][0], lane);
    int cur = 0;
    __syncwarp();
    compose(lst[w], cur, fin + first * 256, cnt, nullptr, lane);
    reinterpret_cast<uint2 *>(lists + (first + cnt - 1) * 256)[lane] =
        reinterpret_cast<const uint2 *>(lst[w][cur])[lane];
}

// Inverse step 2, one warp per block: every run's starting list, into the slot
// of its first segment.
__global__ void __launch_bounds__(kListWarps * 32)
    k_mtf_chain_supers_inv(Segs S, uint32_t supers, uint64_t blocks, uint8_t *lists)
{
    __shared__ __align__(16) uint8_t lst[kListWarps][2][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t b = (uint64_t)blockIdx.x * kListWarps + w;
    if (b >= blocks)
        return;
    uint8_t *base = lists + b * S.per_block * 256;
    identity(lst[w][0], lane);
    int cur = 0;
    __syncwarp();
    const uint64_t step = (uint64_t)kSuper * 256;
    uint2 next = reinterpret_cast<const uint2 *>(base + step - 256)[lane];
    for (uint32_t v = 0; v < supers; ++v) {
        const uint2 f = next;  // run v's composition (the last run's is not needed)
        if (v + 2 < supers)
            next = reinterpret_cast<const uint2 *>(base + (v + 2) * step - 256)[lane];
        reinterpret_cast<uint2 *>(base + v * step)[lane] =
            reinterpret_cast<const uint2 *>(lst[w][cur])[lane];
        apply(lst[w], cur, f, lane);
    }
}

// Inverse step 3 (or the only one), one warp per run.
__global__ void __launch_bounds__(kListWarps * 32)
    k_mtf_lists_inv(const uint8_t *fin, Segs S, uint32_t supers, uint64_t total, bool from_slot,
                    uint8_t *lists)
{
    __shared__ __align__(16) uint8_t lst[kListWarps][2][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t v = (uint64_t)blockIdx.x * kListWarps + w;
    if (v >= total)
        return;
    const uint64_t first = (v / supers) * S.per_block + (v % supers) * kSuper;
    const uint64_t left = S.per_block - (v % supers) * kSuper;
    const uint32_t cnt = left < kSuper ? (uint32_t)left : kSuper;
    if (from_slot)
        reinterpret_cast<uint2 *>(lst[w][0])[lane] =
            reinterpret_cast<const uint2 *>(lists + first * 256)[lane];
    else
        identity(lst[w][0], lane);
    int cur = 0;
    __syncwarp();
    compose(lst[w], cur, fin + first * 256, cnt, lists + first * 256, lane);
}

// out[p] = starting list of p's segment, at entry rel[p]: one warp per segment
__global__ void __launch_bounds__(kListWarps * 32) k_mtf_map(const uint8_t *rel, Segs S,
                                                             const uint8_t *lists, uint8_t *out,
                                                             bool vec)
{
    __shared__ __align__(16) uint8_t lst[kListWarps][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (uint64_t g = (uint64_t)blockIdx.x * kListWarps + w; g < S.count;
         g += (uint64_t)gridDim.x * kListWarps) {
        reinterpret_cast<uint2 *>(lst[w])[lane] =
            reinterpret_cast<const uint2 *>(lists + g * 256)[lane];
        __syncwarp();
        const uint64_t s0 = S.start(g);
        const uint32_t L = S.len(g);
        uint32_t i = 0;
        if (vec)
            for (; i + 512 <= L; i += 512)
                map_bytes(rel + s0 + i + 16 * lane, out + s0 + i + 16 * lane, 16, true,
                          [&](uint32_t c) { return (uint32_t)lst[w][c]; });
        for (i += lane; i < L; i += 32)
            out[s0 + i] = lst[w][rel[s0 + i]];
        __syncwarp();
    }
}

struct MtfWs {
    uint8_t *dist;      // 256 per segment: distinct bytes, or the final lists
    uint32_t *dcount;   // one per segment
    uint8_t *lists;     // 256 per segment: starting lists
    uint8_t *rel;       // n: relative bytes (inverse)
    uint64_t bytes;
};

MtfWs mtf_layout(uint8_t *base, uint64_t n, uint32_t block)
{
    const Segs S = make_segs(n, block);
    MtfWs w;
    uint64_t off = 0;
    auto carve = [&](uint64_t bytes) {
        uint8_t *p = base ? base + off : nullptr;
        off += (bytes + 255) & ~255ull;
        return p;
    };
    w.dist = carve(256 * S.count);
    w.dcount = reinterpret_cast<uint32_t *>(carve(4 * S.count));
    w.lists = carve(256 * S.count);
    w.rel = carve(n);
    w.bytes = off;
    return w;
}

bool mtf_args_ok(uint64_t n, uint32_t block) { return block >= 1 && n <= HUFF_BWT_MAX_N; }

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// runs of kSuper segments: per block, and in all
struct Runs {
    uint32_t supers;
    uint64_t total;
};
Runs make_runs(const Segs &S, uint64_t blocks)
{
    Runs R;
    R.supers = (S.per_block + kSuper - 1) / kSuper;
    R.total = blocks * R.supers;
    return R;
}

// every segment's bytes start 16-byte aligned
bool vector_ok(const void *in, const void *out, uint32_t block)
{
    return (block & 15u) == 0 && aligned16(in) && aligned16(out);
}

unsigned warp_ctas(uint64_t warps) { return (unsigned)((warps + kListWarps - 1) / kListWarps); }
unsigned warp_grid(uint64_t warps)
{
    const uint64_t most = (uint64_t)device_sm_count() * 16;  // 64 warps an SM
    const uint64_t ctas = (warps + kListWarps - 1) / kListWarps;
    return (unsigned)(ctas < most ? ctas : most ? most : 1);
}
unsigned seg_grid(uint64_t count) { return (unsigned)((count + kMtfThreads - 1) / kMtfThreads); }

}  // namespace
}  // namespace huff

using namespace huff;

extern "C" {

uint64_t huff_mtf_workspace_size(uint64_t n, uint32_t block)
{
    if (!mtf_args_ok(n, block))
        return 0;
    return mtf_layout(nullptr, n, block).bytes;
}

huff_status_t huff_mtf_forward(const uint8_t *d_in, uint64_t n, uint32_t block, uint8_t *d_out,
                               void *d_ws, uint64_t ws_bytes, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_mtf_forward");
    if (!mtf_args_ok(n, block) || (n && (!d_in || !d_out || !d_ws)) ||
        (n && ws_bytes < huff_mtf_workspace_size(n, block)) || (d_ws && !aligned16(d_ws)))
        return HUFF_ERR_INVALID_ARG;
    if (n == 0)
        return HUFF_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const Segs S = make_segs(n, block);
    const uint64_t blocks = (n + block - 1) / block;
    MtfWs w = mtf_layout(static_cast<uint8_t *>(d_ws), n, block);
    const Runs R = make_runs(S, blocks);
    const bool vec = vector_ok(d_in, d_out, block);
    k_mtf_distinct<<<warp_grid(S.count), kListWarps * 32, 0, s>>>(d_in, S, w.dist, w.dcount);
    if (R.supers > 1) {
        k_mtf_supers<<<warp_ctas(R.total), kListWarps * 32, 0, s>>>(w.dist, w.dcount, S, R.supers,
                                                                    R.total, w.lists);
        k_mtf_chain_supers<<<warp_ctas(blocks), kListWarps * 32, 0, s>>>(S, R.supers, blocks,
                                                                         w.lists);
    }
    k_mtf_lists<<<warp_ctas(R.total), kListWarps * 32, 0, s>>>(w.dist, w.dcount, S, R.supers, R.total,
                                                               R.supers > 1, w.lists);
    k_mtf_encode<<<seg_grid(S.count), kMtfThreads, 0, s>>>(d_in, S, w.lists, d_out, vec);
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

huff_status_t huff_mtf_inverse(const uint8_t *d_in, uint64_t n, uint32_t block, uint8_t *d_out,
                               void *d_ws, uint64_t ws_bytes, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_mtf_inverse");
    if (!mtf_args_ok(n, block) || (n && (!d_in || !d_out || !d_ws)) ||
        (n && ws_bytes < huff_mtf_workspace_size(n, block)) || (d_ws && !aligned16(d_ws)))
        return HUFF_ERR_INVALID_ARG;
    if (n == 0)
        return HUFF_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const Segs S = make_segs(n, block);
    const uint64_t blocks = (n + block - 1) / block;
    MtfWs w = mtf_layout(static_cast<uint8_t *>(d_ws), n, block);
    const Runs R = make_runs(S, blocks);
    // w.rel is 256-byte aligned
    k_mtf_decode_rel<<<seg_grid(S.count), kMtfThreads, 0, s>>>(d_in, S, w.rel, w.dist,
                                                               vector_ok(d_in, nullptr, block));
    if (R.supers > 1) {
        k_mtf_supers_inv<<<warp_ctas(R.total), kListWarps * 32, 0, s>>>(w.dist, S, R.supers, R.total,
                                                                        w.lists);
        k_mtf_chain_supers_inv<<<warp_ctas(blocks), kListWarps * 32, 0, s>>>(S, R.supers, blocks,
                                                                             w.lists);
    }
    k_mtf_lists_inv<<<warp_ctas(R.total), kListWarps * 32, 0, s>>>(w.dist, S, R.supers, R.total,
                                                                   R.supers > 1, w.lists);
    k_mtf_map<<<warp_grid(S.count), kListWarps * 32, 0, s>>>(w.rel, S, w.lists, d_out,
                                                             vector_ok(nullptr, d_out, block));
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

}  // extern "C"
