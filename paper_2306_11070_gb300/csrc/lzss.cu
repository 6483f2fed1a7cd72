// LZSS Method 2 on the GPU: the segmented parallel version of the paper's
// LZSS coder (Section III-B).  The data is cut into equal segments, each
// coded on its own against a sliding window of its W most recent bits, and
// the segments' code lengths and codes are packed together in order.
//
// Readings (the paper counts window and match lengths in bits; its example
// configuration "1024/24/12/8" is a 1024-bit window, matches of 12..24 bits
// and 8-bit literal blocks):
//  - bits are read most significant bit of each byte first;
//  - the window starts either from the counting numbers (bytes 0, 1, 2, ...
//    before the segment) or from the segment's first W bits, stored as they
//    are (then no match reaches before the segment);
//  - at each position the longest match of Lmin..min(Lmax, bits left) bits
//    is taken, the smallest distance among equally long ones, and a source
//    may run into the bits being coded; a match is the bit 1, distance - 1
//    in log2(W) bits and length - Lmin in ceil(log2(Lmax - Lmin + 1)) bits,
//    a literal the bit 0 and the next min(B, bits left) bits;
//  - container: a 48-byte header (n, segment bytes, W, Lmin, Lmax, B, the
//    dictionary mode, count), count u32 code lengths in bits, then each
//    segment's code packed MSB first into bytes from a 16-byte boundary,
//    zero padded to the next one.
//
// Compression: one warp per segment, or per part of a segment where there are
// few (see k_lzss_parts).  For each token the 32 lanes search the window
// together: for windows of 64 to 16384 bits from a ring in shared memory, all
// distances bit-parallel (a lane's 32-bit mask holds 32 sources) or, in narrow
// windows, a distance at a time; other windows so through L1.  Every lane keeps the same 64-bit
// output accumulator and lane 0 stores the completed words into the
// segment's worst-case slot of the workspace; a one-CTA scan then lays out
// the header and length table and a gather moves every code into place.
// Decompression: a one-CTA scan checks the header and table and finds every
// segment's start; then a CTA of two warps decodes each segment 32 tokens at
// a time, the first warp finding the tokens and reading their fields, the
// second copying a match's bits from the output it has written (a source
// that overlaps the bits being produced repeats with the match distance as
// its period).  Very many segments are decoded by a thread each instead.
#include <cstdint>
#include <type_traits>

#include "api_trace.h"
#include "huff_internal.cuh"

namespace huff {
namespace {

constexpr uint32_t kLzHead = 48;
constexpr int kLzWarps = 8;                // compress: segments per CTA
constexpr int kLzBlock = 32 * kLzWarps;
constexpr int kScanBlock = 1024;
constexpr uint32_t kMaxWindow = 65536;
constexpr uint32_t kRingMaxWindow = 16384;  // the shared-memory window ring
constexpr uint64_t kMaxSegment = 1ull << 24;
constexpr int kThrBlock = 32;             // thread-per-segment decompress: one warp per CTA
constexpr uint32_t kThrRing = 128;        // output words kept per thread (a power of two)
constexpr uint32_t kThrMaxWindow = 2048;  // windows whose words fit that ring with 4 to spare
constexpr uint32_t kLzInCells = 8;        // 16-byte cells of code staged per thread
constexpr uint32_t kLzInFlight = kLzInCells - 1;  // copies left in flight when a word is read
constexpr uint32_t kPathNone = 0, kPathWarps = 1, kPathThreads = 2;  // k_lzss_dlayout's choice
constexpr uint32_t kDecRing = 256;   // decompress: output words kept per warp (a power of two)
constexpr uint32_t kDecAhead = 66;   // 31 words not stored yet, 33 a batch of 32 tokens may fill, one begun
constexpr uint32_t kDecHistory = kDecRing - kDecAhead - 4;  // stored words that stay readable
constexpr uint32_t kCodeRing = 256;  // code words staged per warp (a power of two)
constexpr uint32_t kWalkBits = 64;   // code bits per lane and find_tokens
constexpr uint32_t kTokList = 2048;  // 31 tokens left and the kWalkBits * 32 / 2 of one find_tokens

struct LzParams {
    uint32_t W, lmin, lmax, blk, dict;
    uint32_t ob, lb;  // offset and length field bits
};

__host__ __device__ __forceinline__ int ilog2_exact(uint32_t w)
{
    int k = 0;
    while ((1u << k) < w && k < 31)
        ++k;
    return (1u << k) == w ? k : -1;
}
__host__ __device__ __forceinline__ int ceil_log2(uint32_t v)
{
    int k = 0;
    while ((1ull << k) < v)
        ++k;
    return k;
}
__host__ __device__ __forceinline__ bool params_ok(uint32_t W, uint32_t lmin, uint32_t lmax,
                                                   uint32_t blk, uint32_t dict)
{
    return W >= 2 && W <= kMaxWindow && ilog2_exact(W) > 0 && lmin >= 1 && lmin <= lmax &&
           lmax <= 32 && blk >= 1 && blk <= 32 && (dict == 1 || dict == 2);
}
__host__ __device__ __forceinline__ LzParams make_params(uint32_t W, uint32_t lmin, uint32_t lmax,
                                                         uint32_t blk, uint32_t dict)
{
    LzParams P;
    P.W = W;
    P.lmin = lmin;
    P.lmax = lmax;
    P.blk = blk;
    P.dict = dict;
    P.ob = (uint32_t)ilog2_exact(W);
    P.lb = (uint32_t)ceil_log2(lmax - lmin + 1);
    return P;
}
// upper bound of a segment's code bits: every token but the last literal
// codes at least min(B, Lmin) bits
__host__ __device__ __forceinline__ uint64_t max_bits(uint64_t m, const LzParams &P)
{
    const uint64_t step = P.blk < P.lmin ? P.blk : P.lmin;
    const uint64_t ref = 1 + P.ob + P.lb, lit = 1 + P.blk;
    return (8 * m / step + 2) * (ref > lit ? ref : lit) + P.W;
}
__host__ __device__ __forceinline__ uint64_t al16(uint64_t v) { return (v + 15) & ~15ull; }
// bytes of one segment's worst-case slot in the compression workspace
__host__ __device__ __forceinline__ uint64_t slot_bytes(uint64_t seg, const LzParams &P)
{
    return al16((max_bits(seg, P) + 7) / 8);
}

__device__ __forceinline__ uint32_t bswap32(uint32_t v) { return __byte_perm(v, 0u, 0x0123); }

// word q of the counting-numbers dictionary (bytes 4q .. 4q + 3, MSB first)
__device__ __forceinline__ uint32_t dict_word(uint32_t q)
{
    const uint32_t b = (4 * q) & 255;
    return (b << 24) | (((b + 1) & 255) << 16) | (((b + 2) & 255) << 8) | ((b + 3) & 255);
}

// Word q (bits 32q .. 32q + 31, MSB first) of an m-byte segment, zero past
// its end; the segment starts 16-byte aligned.
__device__ __forceinline__ uint32_t seg_word(const uint8_t *x, uint64_t m, uint64_t q)
{
    const uint64_t b = 4 * q;
    if (b + 4 <= m)
        return bswap32(__ldg(reinterpret_cast<const uint32_t *>(x + b)));
    uint32_t v = 0;
    for (int k = 0; k < 4; ++k)
        v = (v << 8) | (b + k < m ? (uint32_t)x[b + k] : 0u);
    return v;
}

// Word vw of the virtual bit string "window before the segment ++ segment"
// (the W dictionary bits occupy words 0 .. W/32 - 1; only used when W >= 32).
__device__ __forceinline__ uint32_t vword(const uint8_t *x, uint64_t m, uint32_t dwords, uint64_t vw)
{
    return vw < dwords ? dict_word((uint32_t)vw) : seg_word(x, m, vw - dwords);
}

// The 32 bits at bit position v of the virtual string (v may be at any bit)
__device__ __forceinline__ uint32_t vbits(const uint8_t *x, uint64_t m, uint32_t W, uint64_t v)
{
    // windows narrower than a word: handle the dictionary bit by bit
    if (W < 32 && v < W) {
        uint32_t out = 0;
        for (int i = 0; i < 32; ++i) {
            const uint64_t t = v + i;
            uint32_t b;
            if (t < W)
                b = (((uint32_t)(t >> 3) & 255) >> (7 - (t & 7))) & 1;
            else
                b = (seg_word(x, m, (t - W) >> 5) >> (31 - ((t - W) & 31))) & 1;
            out = (out << 1) | b;
        }
        return out;
    }
    const uint32_t dwords = W >= 32 ? W / 32 : 0;
    const uint64_t base = W >= 32 ? 0 : W;  // W < 32: the segment starts at virtual bit W
    const uint64_t u = v - base;
    const uint64_t q = u >> 5;
    const uint32_t sh = (uint32_t)(u & 31);
    const uint32_t a = vword(x, m, dwords, q), b = vword(x, m, dwords, q + 1);
    return sh ? __funnelshift_l(b, a, sh) : a;
}

// Bit accumulator that every lane of a warp keeps in step; lane 0 stores
// each completed 32-bit word (MSB-first bytes) into `out`.
struct WarpBits {
    uint64_t acc;
    uint32_t n;     // pending bits (< 32 between appends)
    uint64_t word;  // next word index
    uint32_t *out;
    __device__ __forceinline__ void put(uint32_t v, uint32_t k, bool leader)
    {
        if (k == 0)
            return;
        acc = (acc << k) | (uint64_t)(v >> (32 - k));  // the top k bits of v
        n += k;
        if (n >= 32) {
            n -= 32;
            if (leader)
                out[word] = bswap32((uint32_t)(acc >> n));
            ++word;
        }
    }
    // the last partial word and zero words up to the slot's 16-byte boundary
    __device__ __forceinline__ void finish(bool leader)
    {
        if (leader) {
            uint64_t w = word;
            if (n)
                out[w++] = bswap32((uint32_t)(acc << (32 - n)));
            while (w & 3)
                out[w++] = 0u;
        }
    }
};

// Ring words per warp (R, a power of two): the window's W/32 words, 34 ahead
// of the position and a batch of 128 loaded at once.  Stored twice, at i and
// i + R, so that neighbouring words are read at neighbouring addresses.
constexpr uint32_t kRingBatch = 128;
__host__ __device__ __forceinline__ uint32_t ring_words(uint32_t W)
{
    uint32_t r = 64;
    while (r < W / 32 + 36 + kRingBatch)
        r <<= 1;
    return r;
}
__host__ __device__ __forceinline__ bool ring_ok(const LzParams &P)
{
    return P.W >= 64 && P.W <= kRingMaxWindow;
}

// Whether the search takes a distance at a time instead of 1024 at once: about
// 8 instructions per 32 bits of window against 4 or 5 per bit of the longest
// match, of Lmin bits at least.  `many`: segments to fill the chip, so that
// instructions count and not a chain's length.  16 MiB of random bytes, ms by
// distances / at once (with one candidate a lane and step in all windows, before,
// 3.4 in 1 KiB segments of 64/4/11/8):
//               1 KiB segments  64 KiB segments
//   64/4/11/8     2.22 / 4.69     20.3 / 30.1
//   64/12/24/8    1.72 / 2.25     16.8 / 17.5
//   128/4/11/8    2.39 / 4.12     21.8 / 26.6
//   128/12/24/8   2.08 / 2.24     21.2 / 18.3
//   256/4/11/8    2.86 / 3.61     26.4 / 23.6
//   256/8/16/8    2.64 / 2.67     24.8 / 19.5
//   512/4/11/8    3.84 / 3.17     36.6 / 21.3
bool by_distance(const LzParams &P, bool many)
{
    return P.W <= (P.lmin < 8 ? 128u : 64u) << (many ? 1 : 0);
}

// The longest match of lo..maxlen bits over 1024 distances at once, the
// smallest distance among equally long ones.  Lane j holds 32 sources, the
// bits a:b (64 bits of the window from bit P - 32 j - 32 of position P); bit
// 31 - i of a mask stands for the source that starts i bits on.  After t
// steps a mask's bits are the sources that agree with the first t bits of the
// look-ahead X: step t ands it with the window shifted by t, complemented
// where X's bit is 0.  About four instructions a step for 1024 candidates,
// against six for 32 when each candidate is shifted into place and compared
// by itself.  One vote after the first 4 G0 steps (G0 = Lmin / 4, straight-line)
// ends most searches, with Lmin below 8 one after 12; else every lane finishes its steps and a warp maximum
// picks the match.  Returns its length << 10 | (1023 - (d - 1)) with d counted
// within the 1024, 0 for none of lo..maxlen bits.
__device__ __forceinline__ uint32_t sign_byte3(uint32_t v)  // the top bit, 32 times
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0xbbbb;" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t sign_byte2(uint32_t v)  // bit 23
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0xaaaa;" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t sign_byte1(uint32_t v)  // bit 15
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0x9999;" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t sign_byte0(uint32_t v)  // bit 7
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0x8888;" : "=r"(r) : "r"(v));
    return r;
}
template <int G0>
__device__ __forceinline__ uint32_t search_masks(uint32_t a, uint32_t b, uint32_t m, uint32_t X,
                                                 uint32_t lo, uint32_t maxlen, int lane)
{
    uint32_t nx[8];  // ~X shifted by 0..7: their bytes' top bits are its bits
#pragma unroll
    for (int i = 0; i < 8; ++i)
        nx[i] = ~X << i;
    auto step = [&](int t, uint32_t c) {
        const uint32_t v = nx[t & 7];
        const uint32_t no = t < 8    ? sign_byte3(v)
                            : t < 16 ? sign_byte2(v)
                            : t < 24 ? sign_byte1(v)
                                     : sign_byte0(v);
        return c & (__funnelshift_l(b, a, t) ^ no);
    };
#pragma unroll
    for (int t = 0; t < 4 * G0; ++t)
        m = step(t, m);
    if (G0 > 0 && !__any_sync(0xffffffffu, m != 0))
        return 0;
    uint32_t len = m ? 4 * G0 : 0, best = m;
#pragma unroll
    for (int t = 4 * G0; t < 32; ++t) {
        if ((t & 3) == 0 && (uint32_t)t >= maxlen)
            break;
        if (G0 < 2 && (t == 12 || t == 20) && !__any_sync(0xffffffffu, m != 0))
            break;  // (from so short a start few searches go on)
        m = step(t, m);
        if (m && (uint32_t)t < maxlen) {
            best = m;
            len = t + 1;
        }
    }
    const uint32_t key =
        len >= lo && len <= maxlen ? len << 10 | (1024u - 32u * lane - __ffs(best)) : 0u;
    return __reduce_max_sync(0xffffffffu, key);
}

// The same a distance at a time, lane's distances lane + 1, lane + 33, ... up to
// 32 * count: its sources start at bit `at` of the ring and every 32 bits before.
// Returns the length << 16 | (65535 - (d - 1)), whatever the length.
__device__ __forceinline__ uint32_t search_distances(const uint32_t *ring, uint32_t R, uint32_t at,
                                                     uint32_t count, uint32_t X, uint32_t maxlen,
                                                     int lane)
{
    const uint32_t sh = at & 31u;
    uint32_t i = (at >> 5) & (R - 1), best = 0, tag = 65535u - lane;
    uint32_t after = ring[i + 1];
#pragma unroll 2
    for (uint32_t k = 0; k < count; ++k) {
        const uint32_t w = ring[i];
        uint32_t len = __clz(__funnelshift_l(after, w, sh) ^ X);
        len = len < maxlen ? len : maxlen;
        const uint32_t key = (len << 16) + tag;
        best = key > best ? key : best;
        after = w;
        i = (i - 1) & (R - 1);
        tag -= 32;
    }
    return __reduce_max_sync(0xffffffffu, best);
}

// Output bits of one warp, the same in every lane: the pending n < 32 bits
// left-aligned in `top`, zeros below; lane 0 stores each completed word.
struct WarpOut {
    uint32_t top, n, word;
    uint32_t *out;
    // the top k (1..32) bits of v, zeros below them
    __device__ __forceinline__ void put(uint32_t v, uint32_t k, int lane)
    {
        const uint32_t t = top | (v >> n);
        const uint32_t rest = __funnelshift_lc(0u, v, 32u - n);  // 0 at n = 0
        n += k;
        if (n >= 32) {
            if (lane == 0)
                out[word] = bswap32(t);
            ++word;
            n -= 32;
            top = rest;
        } else {
            top = t;
        }
    }
};

// One warp's coder for windows of 64..16384 bits, the window in a ring in shared
// memory.  A token depends on its position alone (the window holds the data
// itself), so coding may begin anywhere in a segment.  Where the bits ahead
// repeat the bit before them (a zero run), distance 1 gives the longest match
// there is and no distance is smaller: all the tokens of the run that the
// ring shows (up to 1024 bits) are written at once, as the repeating words
// they form.
struct Coder {
    LzParams P;
    uint32_t *ring;
    uint32_t R, dwords, passes, len_ref, lit_mask;
    uint64_t run_rep;  // the token of a run (distance 1, the longest length), repeated
    uint32_t inv_ref, inv_max;  // x / len_ref, x / lmax as x * inv >> 20: exact up to 2^20 / 32
    const uint8_t *x;  // the segment
    uint32_t m, nbits;
    __device__ __forceinline__ void init(const LzParams &P_, uint32_t *ring_)
    {
        P = P_;
        ring = ring_;
        R = ring_words(P.W);
        dwords = P.W / 32;
        passes = (P.W + 1023) / 1024;
        len_ref = 1 + P.ob + P.lb;
        lit_mask = P.blk < 31 ? ~(0x7fffffffu >> P.blk) : ~0u;
        run_rep = (uint64_t)(0x80000000u | ((P.lmax - P.lmin) << (32 - len_ref))) << 32;
        for (uint32_t k = len_ref; k < 64; k <<= 1)
            run_rep |= run_rep >> k;
        inv_ref = ((1u << 20) + len_ref - 1) / len_ref;
        inv_max = ((1u << 20) + P.lmax - 1) / P.lmax;
    }
    // bits stored as they are before the first token
    __device__ __forceinline__ uint32_t raw() const
    {
        return P.dict != 2 ? 0u : nbits < P.W ? nbits : P.W;
    }
    __device__ __forceinline__ void put_raw(WarpOut &out, int lane) const
    {
        const uint32_t p = raw();
        for (uint32_t q = lane; q < p / 32; q += 32)
            out.out[q] = bswap32(seg_word(x, m, q));
        out.word = p / 32;
        out.n = p & 31u;
        out.top = out.n ? seg_word(x, m, p / 32) & ~(0xffffffffu >> out.n) : 0u;
    }
    // Code from bit p up to the first token that ends at or past `stop`, whose
    // end is returned; before(p) is asked ahead of every token (of a run, its
    // first) and ends the coding when true.
    template <int G0, class F>
    __device__ __forceinline__ uint32_t code(uint32_t p, uint32_t stop, WarpOut &out, int lane,
                                             F before) const
    {
        const uint32_t run_bits = 32 - P.lmax;
        // ring: words [hw - R, hw) of "dictionary ++ segment" (bit v = W + p);
        // pre: the next batch, loaded ahead
        __syncwarp();
        uint32_t hw = p >> 5;
        uint32_t pre[kRingBatch / 32];
#pragma unroll
        for (int k = 0; k < (int)kRingBatch / 32; ++k)
            pre[k] = vword(x, m, dwords, hw + 32 * k + lane);
        while (p < stop && !before(p)) {
            const uint32_t v = P.W + p, q = v >> 5, sh = v & 31u;
            if (hw < q + 34) {
                do {
#pragma unroll
                    for (int k = 0; k < (int)kRingBatch / 32; ++k) {
                        const uint32_t i = (hw + 32 * k + lane) & (R - 1);
                        ring[i] = pre[k];
                        ring[i + R] = pre[k];
                        pre[k] = vword(x, m, dwords, hw + kRingBatch + 32 * k + lane);
                    }
                    hw += kRingBatch;
                } while (hw < q + 34);
                __syncwarp();
            }
            const uint32_t r = nbits - p;
            const uint32_t *const cur = ring + (q & (R - 1));
            const uint32_t *const win = ring + ((q - lane - 1) & (R - 1));
            const uint32_t c0 = cur[0], X = __funnelshift_l(cur[1], c0, sh);  // the look-ahead bits
            const uint32_t w0 = win[0], w1 = win[1], w2 = win[2];
            // all ones or zeros, as the bit before the position
            const uint32_t prev = 0u - (__funnelshift_l(c0, cur[R - 1], sh) & 1u);
            if (((X ^ prev) >> run_bits) == 0 && r >= P.lmax) {
                const uint32_t *const z = ring + ((q + lane) & (R - 1));
                const uint32_t diff = __funnelshift_l(z[1], z[0], sh) ^ prev;
                const uint32_t other = __ballot_sync(0xffffffffu, diff != 0);
                const int f = other ? __ffs(other) - 1 : 31;
                uint32_t run = 32 * f + __shfl_sync(0xffffffffu, (uint32_t)__clz(diff), f);
                run = run < r ? run : r;
                const uint32_t k = run * inv_max >> 20;  // tokens, 1..1024
                p += k * P.lmax;
                const uint32_t total = out.n + k * len_ref, full = total >> 5;
                for (uint32_t i = lane; i <= full; i += 32) {
                    // word i of the pending bits and the repeated token
                    const uint32_t o = 32 * i - out.n;
                    uint32_t w = (uint32_t)(run_rep << (o - (o * inv_ref >> 20) * len_ref) >> 32);
                    if (i == 0)
                        w = out.top | (uint32_t)(run_rep >> 32 >> out.n);
                    if (i < full)
                        out.out[out.word + i] = bswap32(w);
                    else
                        out.top = w;
                }
                out.top = __shfl_sync(0xffffffffu, out.top, full & 31u);
                out.word += full;
                out.n = total & 31u;
                out.top &= ~__funnelshift_rc(0xffffffffu, 0u, out.n);
                continue;
            }
            const uint32_t maxlen = r < P.lmax ? r : P.lmax;
            uint32_t len = 0, dm1 = 0;
            if constexpr (G0 < 0) {
                const uint32_t key =
                    search_distances(ring, R, v - lane - 1, dwords, X, maxlen, lane);
                if (key >> 16 >= P.lmin) {
                    len = key >> 16;
                    dm1 = 65535u - (key & 65535u);
                }
            } else if (maxlen >= P.lmin) {
                uint32_t key = search_masks<G0>(__funnelshift_l(w1, w0, sh),
                                                __funnelshift_l(w2, w1, sh),
                                                lane < (int)dwords ? 0xffffffffu : 0u, X, P.lmin,
                                                maxlen, lane);
                if (key) {
                    len = key >> 10;
                    dm1 = 1023 - (key & 1023u);
                }
                for (uint32_t k = 1; k < passes && len < maxlen; ++k) {
                    const uint32_t *const w = ring + ((q - 32 * k - lane - 1) & (R - 1));
                    key = search_masks<G0>(__funnelshift_l(w[1], w[0], sh),
                                           __funnelshift_l(w[2], w[1], sh), 0xffffffffu, X,
                                           len ? len + 1 : P.lmin, maxlen, lane);
                    if (key) {  // longer than any nearer one
                        len = key >> 10;
                        dm1 = 1024 * k + 1023 - (key & 1023u);
                    }
                }
            }
            if (len) {  // a match: 1, d - 1, l - Lmin
                out.put(0x80000000u | (dm1 << (31 - P.ob)) |
                            (P.lb ? (len - P.lmin) << (32 - len_ref) : 0u),
                        len_ref, lane);
                p += len;
            } else if (r >= P.blk && P.blk < 32) {  // a literal: 0, the next B bits
                out.put((X >> 1) & lit_mask, P.blk + 1, lane);
                p += P.blk;
            } else {  // a literal of min(B, r) bits
                const uint32_t k = r < P.blk ? r : P.blk;
                out.put(0u, 1, lane);
                out.put(X & ~__funnelshift_rc(0xffffffffu, 0u, k), k, lane);
                p += k;
            }
        }
        return p;
    }
};

// Windows of 64..16384 bits, one warp per segment.  Bound by the latency of one
// token's steps (a warp alone issues about every 4.5 cycles) and, from some
// 8000 warps on, by instruction issue.  64 MiB of the bitstream stand-in with
// 1024/12/24/8: 13.1 -> 2.4 ms in 16 KiB segments, 10.4 -> 1.9 ms in 4 KiB
// (before: one candidate a lane and step); W = 4096 in 16 KiB segments 40.9 ->
// 4.6 ms.  With Lmin's steps not straight-line (a run-time bound on each) it
// took half as long again.
template <int G0>
__global__ void __launch_bounds__(32)
    k_lzss_compress_ring(const uint8_t *__restrict__ in, uint64_t n, uint64_t seg, LzParams P,
                         uint8_t *__restrict__ slots, uint32_t *__restrict__ bits_out,
                         const int32_t *status)
{
    if (chain_failed(status))
        return;
    extern __shared__ uint32_t ring[];
    const int lane = threadIdx.x;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t sbytes = slot_bytes(seg, P);
    Coder cd;
    cd.init(P, ring);
    for (uint64_t s = blockIdx.x; s < count; s += gridDim.x) {
        cd.x = in + s * seg;
        cd.m = (uint32_t)(s + 1 < count ? seg : n - s * seg);
        cd.nbits = 8 * cd.m;
        WarpOut out;
        out.out = reinterpret_cast<uint32_t *>(slots + s * sbytes);
        cd.put_raw(out, lane);
        cd.code<G0>(cd.raw(), cd.nbits, out, lane, [](uint32_t) { return false; });
        if (lane == 0) {  // the last word and zeros up to the slot's 16-byte boundary
            uint32_t w = out.word;
            if (out.n)
                out.out[w++] = bswap32(out.top);
            while (w & 3u)
                out.out[w++] = 0u;
            bits_out[s] = out.word * 32 + out.n;
        }
    }
}

// Few segments leave most of the chip idle, so a segment is coded in `parts` by
// a warp each.  A part begins at its cut whether or not a token does; since a
// token depends on its position alone, its code is right from the first of its
// tokens that begins where one of the segment's tokens does (chains of tokens
// from two starts meet after some tens of them, not counting runs).
// k_lzss_parts codes the parts, noting kMarks places where a token begins, the
// first kDense and then one in kSparse; k_lzss_join, a warp per segment, takes
// the parts in order: from where the one before ended it codes on until it
// meets a noted token (or, if it meets none, to the part's end);
// k_lzss_gather_parts puts the pieces together bit by bit. In a segment's slot,
// part k from byte k * stride on: {end, code bits, marks, 0}, the code, the
// bits before the meeting point, the marks {position, code bits before}.  Part
// 0 is right as it is; its marks' place holds the pieces {first bit in the
// slot, bits}, 2 per part.
constexpr uint32_t kMarks = 128, kDense = 96, kSparse = 16, kMaxParts = 8;
constexpr uint32_t kMinPart = 4096;  // bytes
struct PartsLayout {
    uint32_t parts;               // of a segment
    uint32_t code, head, stride;  // bytes of a part's code, its head, a part
};

__device__ __forceinline__ uint32_t part_cut(const Coder &cd, uint32_t parts, uint32_t k)
{
    const uint32_t raw = cd.raw();
    return raw + (uint32_t)((uint64_t)(cd.nbits - raw) * k / parts);
}

template <int G0>
__global__ void __launch_bounds__(32)
    k_lzss_parts(const uint8_t *__restrict__ in, uint64_t n, uint64_t seg, LzParams P, PartsLayout L,
                 uint8_t *__restrict__ slots, const int32_t *status)
{
    if (chain_failed(status))
        return;
    extern __shared__ uint32_t ring[];
    const int lane = threadIdx.x;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t sbytes = slot_bytes(seg, P);
    Coder cd;
    cd.init(P, ring);
    for (uint64_t i = blockIdx.x; i < count * L.parts; i += gridDim.x) {
        const uint64_t s = i / L.parts;
        const uint32_t k = (uint32_t)(i - s * L.parts);
        cd.x = in + s * seg;
        cd.m = (uint32_t)(s + 1 < count ? seg : n - s * seg);
        cd.nbits = 8 * cd.m;
        uint8_t *const part = slots + s * sbytes + (uint64_t)k * L.stride;
        uint2 *const marks = reinterpret_cast<uint2 *>(part + 16 + L.code + L.head);
        WarpOut out;
        out.out = reinterpret_cast<uint32_t *>(part + 16);
        out.top = out.n = out.word = 0;
        if (k == 0)
            cd.put_raw(out, lane);
        uint32_t nm = k == 0 ? kMarks : 0, skip = 0;
        const uint32_t end = cd.code<G0>(part_cut(cd, L.parts, k), part_cut(cd, L.parts, k + 1), out,
                                         lane, [&](uint32_t p) {
                                             if (nm < kMarks && skip-- == 0) {
                                                 if (lane == 0)
                                                     marks[nm] = make_uint2(p, 32 * out.word + out.n);
                                                 skip = ++nm < kDense ? 0 : kSparse - 1;
                                             }
                                             return false;
                                         });
        if (lane == 0) {
            if (out.n)
                out.out[out.word] = bswap32(out.top);
            *reinterpret_cast<uint4 *>(part) =
                make_uint4(end, 32 * out.word + out.n, k == 0 ? 0u : nm, 0u);
        }
    }
}

template <int G0>
__global__ void __launch_bounds__(32)
    k_lzss_join(const uint8_t *__restrict__ in, uint64_t n, uint64_t seg, LzParams P, PartsLayout L,
                uint8_t *__restrict__ slots, uint32_t *__restrict__ bits_out, const int32_t *status)
{
    if (chain_failed(status))
        return;
    extern __shared__ uint32_t ring[];
    const int lane = threadIdx.x;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t sbytes = slot_bytes(seg, P);
    Coder cd;
    cd.init(P, ring);
    // bits of a head that a step may begin at: a run's tokens still fit
    const uint32_t head_bits = 8 * L.head - 1024 / P.lmax * cd.len_ref - 96;
    for (uint64_t s = blockIdx.x; s < count; s += gridDim.x) {
        cd.x = in + s * seg;
        cd.m = (uint32_t)(s + 1 < count ? seg : n - s * seg);
        cd.nbits = 8 * cd.m;
        uint8_t *const slot = slots + s * sbytes;
        uint2 *const pieces = reinterpret_cast<uint2 *>(slot + 16 + L.code + L.head);
        const uint4 first = *reinterpret_cast<const uint4 *>(slot);
        uint32_t p = first.x, total = first.y;
        if (lane < 2)
            pieces[lane] = lane ? make_uint2(0, 0) : make_uint2(8 * 16, first.y);
        for (uint32_t k = 1; k < L.parts; ++k) {
            const uint32_t stop = part_cut(cd, L.parts, k + 1);
            const uint32_t at = k * L.stride;  // bytes
            uint2 head = make_uint2(0, 0), tail = make_uint2(0, 0);
            if (p < stop) {
                const uint4 part = *reinterpret_cast<const uint4 *>(slot + at);
                const uint2 *const marks =
                    reinterpret_cast<const uint2 *>(slot + at + 16 + L.code + L.head);
                WarpOut out;
                out.out = reinterpret_cast<uint32_t *>(slot + at + 16 + L.code);
                out.top = out.n = out.word = 0;
                uint32_t base = 0;  // lane's mark: base + lane
                uint2 mark = lane < part.z ? marks[lane] : make_uint2(0xffffffffu, 0);
                bool met = false, lost = false;
                const uint32_t end = cd.code<G0>(p, stop, out, lane, [&](uint32_t at_bit) {
                    uint32_t hit;
                    for (;;) {
                        hit = __ballot_sync(0xffffffffu, mark.x == at_bit);
                        if (hit || __any_sync(0xffffffffu, mark.x > at_bit))
                            break;
                        base += 32;
                        if (base >= part.z)
                            break;
                        mark = base + lane < part.z ? marks[base + lane] : make_uint2(0xffffffffu, 0);
                    }
                    met = hit != 0;
                    lost = !met && (base >= part.z || 32 * out.word + out.n > head_bits);
                    if (met)
                        tail.x = __shfl_sync(0xffffffffu, mark.y, __ffs(hit) - 1);
                    return met || lost;
                });
                if (lost) {  // the whole part again, over its code
                    out.out = reinterpret_cast<uint32_t *>(slot + at + 16);
                    out.top = out.n = out.word = 0;
                    p = cd.code<G0>(p, stop, out, lane, [](uint32_t) { return false; });
                    head = make_uint2(8 * (at + 16), 32 * out.word + out.n);
                } else {
                    head = make_uint2(8 * (at + 16 + L.code), 32 * out.word + out.n);
                    p = met ? part.x : end;
                    if (met)
                        tail = make_uint2(8 * (at + 16) + tail.x, part.y - tail.x);
                }
                if (lane == 0 && out.n)
                    out.out[out.word] = bswap32(out.top);
            }
            if (lane < 2)
                pieces[2 * k + lane] = lane ? tail : head;
            total += head.y + tail.y;
        }
        if (lane == 0)
            bits_out[s] = total;
    }
}

// Every segment's pieces to its place, zero padded to the 16-byte boundary.
__global__ void __launch_bounds__(256)
    k_lzss_gather_parts(uint64_t n, uint64_t seg, LzParams P, PartsLayout L,
                        const uint8_t *__restrict__ slots, const uint32_t *__restrict__ bits,
                        const uint64_t *__restrict__ start, uint8_t *__restrict__ out, uint64_t cap,
                        const int32_t *status)
{
    __shared__ uint2 piece[2 * kMaxParts];       // first bit in the slot, first bit of the code
    __shared__ uint32_t first[2 * kMaxParts + 1];
    if (chain_failed(status))
        return;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t sbytes = slot_bytes(seg, P);
    for (uint64_t s = blockIdx.x; s < count; s += gridDim.x) {
        const uint8_t *const slot = slots + s * sbytes;
        const uint32_t total = bits[s], words = (uint32_t)(al16(((uint64_t)total + 7) / 8) / 4);
        if (start[s] + 4ull * words > cap)
            continue;
        __syncthreads();
        if (threadIdx.x < 2 * L.parts)
            piece[threadIdx.x] =
                reinterpret_cast<const uint2 *>(slot + 16 + L.code + L.head)[threadIdx.x];
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t at = 0;
            for (uint32_t i = 0; i < 2 * L.parts; ++i) {
                first[i] = at;
                at += piece[i].y;
            }
            first[2 * L.parts] = at;
        }
        __syncthreads();
        uint32_t *const dst = reinterpret_cast<uint32_t *>(out + start[s]);
        const uint32_t *const src = reinterpret_cast<const uint32_t *>(slot);
        uint32_t i = 0;
        for (uint32_t j = threadIdx.x; j < words; j += blockDim.x) {
            uint32_t w = 0, got = 0;  // bits of the word so far
            const uint32_t at = 32 * j;
            while (i + 1 < 2 * L.parts && first[i + 1] <= at)
                ++i;
            for (uint32_t q = i; q < 2 * L.parts && got < 32; ++q) {
                const uint32_t from = at + got, to = first[q + 1];
                if (from >= to)
                    continue;
                const uint32_t b = piece[q].x + (from - first[q]), a = b >> 5;
                const uint32_t v = __funnelshift_l(bswap32(__ldcg(src + a + 1)), bswap32(__ldcg(src + a)),
                                                   b & 31u);
                const uint32_t take = to - from < 32 - got ? to - from : 32 - got;
                w |= (v & ~__funnelshift_rc(0xffffffffu, 0u, take)) >> got;
                got += take;
            }
            dst[j] = bswap32(w);
        }
    }
}

// Every other window: the words through L1, each lane trying its own distances
// one by one.
__global__ void __launch_bounds__(kLzBlock)
    k_lzss_compress(const uint8_t *__restrict__ in, uint64_t n, uint64_t seg, LzParams P,
                    uint8_t *__restrict__ slots, uint32_t *__restrict__ bits_out,
                    const int32_t *status)
{
    if (chain_failed(status))
        return;
    const int lane = threadIdx.x & 31;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t sbytes = slot_bytes(seg, P);
    const uint64_t nwarps = (uint64_t)gridDim.x * kLzWarps;
    for (uint64_t s = (uint64_t)blockIdx.x * kLzWarps + (threadIdx.x >> 5); s < count; s += nwarps) {
        const uint8_t *x = in + s * seg;
        const uint64_t m = s + 1 < count ? seg : n - s * seg;
        const uint64_t nbits = 8 * m;
        WarpBits out;
        out.acc = 0;
        out.n = 0;
        out.word = 0;
        out.out = reinterpret_cast<uint32_t *>(slots + s * sbytes);
        uint64_t p = 0;
        if (P.dict == 2) {  // the first W bits as they are
            const uint64_t raw = nbits < P.W ? nbits : P.W;
            for (uint64_t q = 0; q < raw; q += 32) {
                const uint32_t k = raw - q < 32 ? (uint32_t)(raw - q) : 32u;
                out.put(seg_word(x, m, q >> 5), k, lane == 0);
            }
            p = raw;
        }
        const uint64_t vbase = P.W;  // virtual bit of the segment's bit 0
        const uint32_t dwords = P.W >= 32 ? P.W / 32 : 0;
        const uint32_t nk = P.W >= 32 ? P.W / 32 : 1;  // candidates per lane
        while (p < nbits) {
            const uint64_t r = nbits - p;
            const uint32_t maxlen = r < P.lmax ? (uint32_t)r : P.lmax;
            const uint32_t X = vbits(x, m, P.W, vbase + p);  // the 32 look-ahead bits
            uint32_t key = 0;
            if (maxlen >= P.lmin) {
                // lane's sources: virtual bit v_k = vbase + p - (lane + 1) - 32 k
                const uint64_t v0 = vbase + p - (uint64_t)lane - 1;
                if (P.W >= 32) {
                    const uint32_t sh = (uint32_t)(v0 & 31);
                    uint64_t vw = v0 >> 5;
                    uint32_t hiw = vword(x, m, dwords, vw + 1);
                    for (uint32_t k = 0; k < nk; ++k, --vw) {
                        const uint32_t low = vword(x, m, dwords, vw);
                        const uint32_t src = sh ? __funnelshift_l(hiw, low, sh) : low;
                        hiw = low;
                        const uint32_t d = (uint32_t)lane + 1 + 32 * k;
                        uint32_t len = __clz(src ^ X);
                        len = len < maxlen ? len : maxlen;
                        const bool ok = (P.dict == 1 || d <= p) && len >= P.lmin;
                        const uint32_t kk = (len << 16) | (65535u - (d - 1));
                        key = ok && kk > key ? kk : key;
                    }
                } else if ((uint32_t)lane < P.W) {
                    const uint32_t d = (uint32_t)lane + 1;
                    const uint32_t src = vbits(x, m, P.W, v0);
                    uint32_t len = __clz(src ^ X);
                    len = len < maxlen ? len : maxlen;
                    if ((P.dict == 1 || d <= p) && len >= P.lmin)
                        key = (len << 16) | (65535u - (d - 1));
                }
                key = __reduce_max_sync(0xffffffffu, key);
            }
            if (key) {  // a match: 1, d - 1, l - Lmin
                const uint32_t len = key >> 16, dm1 = 65535u - (key & 0xffffu);
                out.put(1u << 31, 1, lane == 0);
                out.put(dm1 << (32 - P.ob), P.ob, lane == 0);
                out.put(P.lb ? (len - P.lmin) << (32 - P.lb) : 0u, P.lb, lane == 0);
                p += len;
            } else {  // a literal: 0, the next min(B, r) bits
                const uint32_t k = r < P.blk ? (uint32_t)r : P.blk;
                out.put(0u, 1, lane == 0);
                out.put(X, k, lane == 0);
                p += k;
            }
        }
        out.finish(lane == 0);
        if (lane == 0)
            bits_out[s] = (uint32_t)(out.word * 32 + out.n);
    }
}

// Exclusive sum of `own` over the CTA's kScanBlock threads; the total of all in
// `total`.  `part` holds 32 values.
__device__ __forceinline__ unsigned long long block_scan(unsigned long long own,
                                                         unsigned long long *part,
                                                         unsigned long long &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long incl = own;
    for (int k = 1; k < 32; k <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, k);
        if (lane >= k)
            incl += y;
    }
    __syncthreads();  // part's last readers
    if (lane == 31)
        part[warp] = incl;
    __syncthreads();
    unsigned long long p = part[lane];
    for (int k = 1; k < 32; k <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, p, k);
        if (lane >= k)
            p += y;
    }
    total = __shfl_sync(0xffffffffu, p, 31);
    const unsigned long long before = __shfl_sync(0xffffffffu, p, warp ? warp - 1 : 0);
    return (warp ? before : 0) + incl - own;
}

// Header, length table and segment starts of the container; the size into
// *out_bytes, HUFF_ERR_CAPACITY when it exceeds `cap`.
__global__ void __launch_bounds__(kScanBlock)
    k_lzss_layout(uint64_t n, uint64_t seg, LzParams P, const uint32_t *__restrict__ bits,
                  uint64_t *__restrict__ start, uint8_t *__restrict__ out, uint64_t cap,
                  unsigned long long *out_bytes, int32_t *status)
{
    __shared__ unsigned long long s_part[32];
    if (chain_failed(status))
        return;
    const int tid = threadIdx.x;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t head = al16(kLzHead + 4 * count);
    unsigned long long total = head;
    for (uint64_t i0 = 0; i0 < count; i0 += kScanBlock) {
        const uint64_t i = i0 + tid;
        unsigned long long sum;
        const unsigned long long at =
            block_scan(i < count ? al16(((uint64_t)bits[i] + 7) / 8) : 0, s_part, sum);
        if (i < count)
            start[i] = total + at;
        total += sum;
    }
    if (tid == 0) {
        *out_bytes = total;
        if (total > cap)
            set_status(status, HUFF_ERR_CAPACITY);
    }
    if (total > cap)
        return;
    for (uint64_t i = tid; i < head; i += kScanBlock) {  // header, table, padding
        uint8_t v = 0;
        if (i < kLzHead) {
            uint64_t f = 0;
            uint32_t o = (uint32_t)i;
            if (o < 8)
                f = n;
            else if (o < 16)
                f = seg, o -= 8;
            else if (o < 20)
                f = P.W, o -= 16;
            else if (o < 24)
                f = P.lmin, o -= 20;
            else if (o < 28)
                f = P.lmax, o -= 24;
            else if (o < 32)
                f = P.blk, o -= 28;
            else if (o < 36)
                f = P.dict, o -= 32;
            else if (o < 40)
                f = 0, o -= 36;
            else
                f = count, o -= 40;
            v = (uint8_t)(f >> (8 * (o & 7)));
        } else if (i < kLzHead + 4 * count) {
            const uint64_t j = (i - kLzHead) / 4;
            v = (uint8_t)(bits[j] >> (8 * ((i - kLzHead) & 3)));
        }
        out[i] = v;
    }
}

// Move every segment's code from its slot to its place (16-byte copies; the
// slot already holds the zero padding up to its 16-byte boundary).
__global__ void k_lzss_gather(uint64_t n, uint64_t seg, LzParams P, const uint8_t *__restrict__ slots,
                              const uint32_t *__restrict__ bits, const uint64_t *__restrict__ start,
                              uint8_t *__restrict__ out, uint64_t cap, const int32_t *status)
{
    if (chain_failed(status))
        return;
    const uint64_t count = n ? (n + seg - 1) / seg : 0;
    const uint64_t sbytes = slot_bytes(seg, P);
    for (uint64_t s = blockIdx.x; s < count; s += gridDim.x) {
        const uint64_t len = al16((bits[s] + 7) / 8);
        if (start[s] + len > cap)
            continue;
        const uint4 *src = reinterpret_cast<const uint4 *>(slots + s * sbytes);
        uint4 *dst = reinterpret_cast<uint4 *>(out + start[s]);
        for (uint64_t j = threadIdx.x; j < len / 16; j += blockDim.x)
            dst[j] = src[j];
    }
}

// ---------------------------------------------------------------- decompress
// Whether a thread per segment decodes faster than a CTA of two warps per
// segment.  A thread's tokens cost a fraction of the instructions (32 segments
// share each one), but every segment is one chain of some hundreds of cycles a
// token, so it takes very many segments to fill the chip; a CTA spends about 3
// ns of it on a segment however short, and on short tokens (Lmin up to 6 bits)
// as much per bit as the threads.  Measured thread / CTA times, bitstream
// stand-in:
//  - stored prefix, windows of 32..2048 bits, literals up to 31 bits (the
//    branch-free step of decode_fast): 1024/12/24/8 in 1 KiB segments 1.72 from
//    16384 segments, 1.05 from 49152, 0.76 from 131072; 64/4/11/8 0.86, 0.57
//    and 0.41.  From 320 segments per SM on, short tokens from 100.
//  - all others, token by token.  Short tokens: 64/4/11/8 and the counting
//    dictionary in 256 B segments 1.68 from 8192 segments, 0.76 from 32768, 0.62
//    from 262144, in 1 KiB segments 2.25, 0.88 and 0.70 (131072).  Longer ones
//    only where a segment is short: 1024/12/24/8 from 16384, 49152 and 262144
//    segments of 16 B 0.66, 0.46 and 0.34, 64 B 1.04, 0.66 and 0.53, 128 B 1.46,
//    0.87 and 0.74, 256 B 2.12, 1.29 and 1.03, 1 KiB 3.07, 1.85 and (131072) 1.43.
__device__ __forceinline__ bool threads_better(uint64_t count, uint64_t seg, const LzParams &P,
                                               uint32_t sms)
{
    const bool brief = P.lmin <= 6 && P.W <= kThrMaxWindow;
    uint32_t per_sm;  // from so many segments on
    if (P.dict == 2 && P.W >= 32 && P.W <= kThrMaxWindow && P.blk <= 31)
        per_sm = brief ? 100 : 320;
    else if (brief)
        per_sm = seg <= 64 ? 100 : 200;
    else
        per_sm = seg <= 32 ? 100 : seg <= 64 ? 200 : seg <= 128 ? 320 : seg <= 256 ? 1000 : ~0u;
    return per_sm != ~0u && count >= (uint64_t)per_sm * sms;
}

// Header and table checks, segment starts (scan), *d_n; statuses as the
// oracle's: CORRUPT for an inconsistent header or table, CAPACITY for n >
// cap.  *path: the decoder to run, kPathNone when the segments may not be
// decoded.
__global__ void __launch_bounds__(kScanBlock)
    k_lzss_dlayout(const uint8_t *__restrict__ c, uint64_t bytes, uint64_t cap,
                   uint64_t *__restrict__ start, uint64_t max_count,
                   unsigned long long *d_n, int32_t *status, uint32_t *path, uint32_t sms)
{
    __shared__ unsigned long long s_part[32];
    const int tid = threadIdx.x;
    if (tid == 0)
        *path = kPathNone;
    if (chain_failed(status))
        return;
    if (bytes < kLzHead) {
        if (tid == 0)
            set_status(status, HUFF_ERR_CORRUPT_STREAM);
        return;
    }
    const uint64_t n = *reinterpret_cast<const uint64_t *>(c);
    const uint64_t seg = *reinterpret_cast<const uint64_t *>(c + 8);
    const uint32_t *f = reinterpret_cast<const uint32_t *>(c + 16);
    const uint64_t count = *reinterpret_cast<const uint64_t *>(c + 40);
    const bool hdr_ok = params_ok(f[0], f[1], f[2], f[3], f[4]) && f[5] == 0 && seg >= 16 &&
                        seg % 16 == 0 && seg <= kMaxSegment &&
                        count == (n ? (n + seg - 1) / seg : 0) && count <= (bytes - kLzHead) / 4 &&
                        count <= max_count;
    if (!hdr_ok) {
        if (tid == 0)
            set_status(status, HUFF_ERR_CORRUPT_STREAM);
        return;
    }
    const uint8_t *tab = c + kLzHead;
    const uint64_t head = al16(kLzHead + 4 * count);
    unsigned long long total = head;
    for (uint64_t i0 = 0; i0 < count; i0 += kScanBlock) {
        const uint64_t i = i0 + tid;
        unsigned long long sum;
        const uint64_t nb = i < count ? *reinterpret_cast<const uint32_t *>(tab + 4 * i) : 0u;
        const unsigned long long at = block_scan(al16((nb + 7) / 8), s_part, sum);
        if (i < count)
            start[i] = total + at;
        total += sum;
    }
    if (tid == 0) {
        if (total != bytes) {
            set_status(status, HUFF_ERR_CORRUPT_STREAM);
        } else {
            *d_n = n;
            if (n > cap)
                set_status(status, HUFF_ERR_CAPACITY);
            else
                *path = threads_better(count, seg, make_params(f[0], f[1], f[2], f[3], f[4]), sms)
                            ? kPathThreads
                            : kPathWarps;
        }
    }
}

// Store output word q (MSB-first bytes) of an m-byte segment output.
__device__ __forceinline__ void store_out_word(uint8_t *y, uint32_t m, uint32_t q, uint32_t w)
{
    const uint32_t b = 4 * q;
    if (b + 4 <= m) {
        __stcg(reinterpret_cast<uint32_t *>(y) + q, bswap32(w));
    } else {
        for (uint32_t k = 0; k < 4; ++k)
            if (b + k < m)
                y[b + k] = (uint8_t)(w >> (24 - 8 * k));
    }
}

// Shared memory of one decoding CTA: a front warp and a copy warp, the first
// one batch of tokens ahead of the second.
struct alignas(16) DecShared {
    uint32_t out[kDecRing];    // copy warp: output word q at q mod kDecRing
    uint32_t code[kCodeRing];  // front warp: code word q at q mod kCodeRing
    uint16_t list[kTokList];   // front warp: token starts not decoded yet (position << 1 | flag)
    uint16_t exits[(kWalkBits + 33) * 32];  // front warp: [offset][lane], see find_tokens
    struct Batch {  // 32 tokens: place in the output, kTok* fields, distance or literal bits
        uint32_t o[32], info[32], x[32];
    } batch[2];
};
// a token's fields in Batch::info above its length (bits 0..5)
constexpr uint32_t kTokRef = 64, kTokValid = 128, kTokEnd = 256;

__device__ __forceinline__ uint32_t lds_u16(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
// named barriers of the two warps: 1, 2 a batch is full, 3, 4 it is read
// (ids as immediates: with an id in a register the kernel reserves all 16
// barriers, which leaves four CTAs per SM resident)
__device__ __forceinline__ void full_sync(uint32_t turn)
{
    if (turn & 1)
        asm volatile("bar.sync 2, 64;" ::: "memory");
    else
        asm volatile("bar.sync 1, 64;" ::: "memory");
}
__device__ __forceinline__ void full_arrive(uint32_t turn)
{
    if (turn & 1)
        asm volatile("bar.arrive 2, 64;" ::: "memory");
    else
        asm volatile("bar.arrive 1, 64;" ::: "memory");
}
__device__ __forceinline__ void read_sync(uint32_t turn)
{
    if (turn & 1)
        asm volatile("bar.sync 4, 64;" ::: "memory");
    else
        asm volatile("bar.sync 3, 64;" ::: "memory");
}
__device__ __forceinline__ void read_arrive(uint32_t turn)
{
    if (turn & 1)
        asm volatile("bar.arrive 4, 64;" ::: "memory");
    else
        asm volatile("bar.arrive 3, 64;" ::: "memory");
}

// The segment a CTA decodes.
struct SegIn {
    const uint32_t *w;  // the code's words (16-byte aligned, padded to a 16-byte boundary)
    uint32_t nw;        // their number; words past them read as zero
    uint32_t code_bits;
    uint8_t *y;         // the output, 16-byte aligned
    uint32_t m, nbits;  // its bytes and bits
    uint32_t raw;       // bits stored as they are before the tokens
    __device__ __forceinline__ uint32_t load(uint32_t i) const
    {
        return i < nw ? bswap32(__ldg(w + i)) : 0u;
    }
};

// The front warp's state.
struct Front {
    uint32_t bpos;        // code bits whose tokens are listed
    uint32_t loaded;      // code words staged
    uint32_t pre0, pre1;  // the next 64 code words, two per lane
    uint32_t head, avail; // the list's first token and its length
};

// exits[e] of one lane's kWalkBits bits (hi:lo), from the last offset back;
// G offsets at a time: no token is shorter than G bits, so the loads of a
// group do not depend on its own stores.
template <int G>
__device__ __forceinline__ void fill_exits(uint32_t col, uint32_t hi, uint32_t lo, uint32_t len_ref,
                                           uint32_t len_lit)
{
    const uint32_t cr = col + 64 * len_ref, cl = col + 64 * len_lit;
#pragma unroll
    for (int g = (int)kWalkBits - G; g >= 0; g -= G) {
        uint32_t v[G];
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const int p = g + j;
            const bool ref = ((p < 32 ? hi : lo) & (0x80000000u >> (p & 31))) != 0;
            v[j] = lds_u16((ref ? cr : cl) + 64 * p);
        }
#pragma unroll
        for (int j = 0; j < G; ++j)
            sts_u16(col + 64 * (g + j), v[j] + 0x100u);
    }
}

// List the starts of the tokens in the next kWalkBits * 32 code bits.  A
// token's length depends on its flag alone, so where a walk leaves a stretch
// of code is a function of where it enters.  Lane l takes the kWalkBits bits
// from bit kWalkBits * l on and fills, for every offset e, exits[e][l]: the
// offset in lane l + 1's bits at which a walk entering at e leaves, and the
// tokens it passes << 8 (exits[e] = exits[e + the length of the token at e]
// plus one token; offsets past the stretch map to themselves).  Then one
// chain of 32 loads gives every lane its true entry and its tokens' place in
// the list, and each lane walks only its own few tokens: a walk of all the
// tokens by itself costs one warp ~150 cycles a token.
__device__ __forceinline__ void find_tokens(const SegIn &sg, Front &fr, DecShared &sh,
                                            uint32_t len_ref, uint32_t len_lit, int lane)
{
    // the stretch, the longest token's rest past it and a word of slack
    while (fr.loaded < (fr.bpos >> 5) + kWalkBits + 4) {
        sh.code[(fr.loaded + lane) & (kCodeRing - 1)] = fr.pre0;
        sh.code[(fr.loaded + 32 + lane) & (kCodeRing - 1)] = fr.pre1;
        fr.loaded += 64;
        fr.pre0 = sg.load(fr.loaded + lane);
        fr.pre1 = sg.load(fr.loaded + 32 + lane);
    }
    __syncwarp();
    const uint32_t at = (fr.bpos & 31u) + kWalkBits * (uint32_t)lane;
    const uint32_t q = (fr.bpos >> 5) + (at >> 5);
    const uint32_t w0 = sh.code[q & (kCodeRing - 1)], w1 = sh.code[(q + 1) & (kCodeRing - 1)],
                   w2 = sh.code[(q + 2) & (kCodeRing - 1)];
    uint32_t hi = __funnelshift_l(w1, w0, at & 31u), lo = __funnelshift_l(w2, w1, at & 31u);
    const uint32_t tab = smem_u32(sh.exits);
    if (len_ref >= 8 && len_lit >= 8)
        fill_exits<8>(tab + 2 * lane, hi, lo, len_ref, len_lit);
    else
        fill_exits<2>(tab + 2 * lane, hi, lo, len_ref, len_lit);
    __syncwarp();
    uint32_t e = 0, acc = 0, mine = 0;  // acc, mine: tokens so far << 8 | entry
#pragma unroll
    for (int l = 0; l < 32; ++l) {
        mine = lane == l ? acc : mine;
        const uint32_t v = lds_u16(tab + e * 64 + 2 * l);
        e = v & 0xffu;
        acc = (acc & ~0xffu) + v;
    }
    uint32_t p = mine & 0xffu, i = fr.head + fr.avail + (mine >> 8);
    const uint32_t base = (fr.bpos + kWalkBits * (uint32_t)lane) << 1;
    const uint64_t b = (((uint64_t)hi << 32) | lo) << p;
    hi = (uint32_t)(b >> 32);
    lo = (uint32_t)b;
    while (p < kWalkBits) {
        const uint32_t flag = hi >> 31, step = flag ? len_ref : len_lit;
        sh.list[i & (kTokList - 1)] = (uint16_t)(base + 2 * p + flag);
        ++i;
        p += step;
        hi = __funnelshift_l(lo, hi, 1);
        lo <<= 1;
        hi = __funnelshift_lc(lo, hi, step - 1);  // step <= 33
        lo = __funnelshift_lc(0u, lo, step - 1);
    }
    fr.avail += acc >> 8;
    fr.bpos += 32 * kWalkBits + e;
    __syncwarp();
}

// Front warp: the segment's tokens, 32 per batch, to the copy warp.  `turn`
// counts the batches of the CTA.  False (warp-uniform) if the code is corrupt.
__device__ __forceinline__ bool read_segment(const SegIn &sg, DecShared &sh, const LzParams &P,
                                             int lane, uint32_t &turn)
{
    uint32_t opos = sg.raw, cpos = sg.raw;
    bool good = sg.raw <= sg.code_bits, ended = false;
    Front fr;
    fr.bpos = cpos;
    fr.loaded = cpos >> 5;
    fr.pre0 = sg.load(fr.loaded + lane);
    fr.pre1 = sg.load(fr.loaded + 32 + lane);
    fr.head = fr.avail = 0;
    const uint32_t len_ref = 1 + P.ob + P.lb, len_lit = 1 + P.blk;
    while (!ended) {
        uint32_t o = 0, info = kTokEnd, x = 0;
        if (good && opos < sg.nbits) {
            if (fr.avail < 32)
                find_tokens(sg, fr, sh, len_ref, len_lit, lane);
            const uint32_t tok = sh.list[(fr.head + lane) & (kTokList - 1)];
            const bool ref = tok & 1u;
            const uint32_t dc = ((tok >> 1) - cpos) & 0x7fffu;
            const uint32_t at = (cpos & 31u) + dc + 1;
            const uint32_t q = (cpos >> 5) + (at >> 5);
            const uint32_t body = __funnelshift_l(sh.code[(q + 1) & (kCodeRing - 1)],
                                                  sh.code[q & (kCodeRing - 1)], at & 31u);
            const uint32_t d = (body >> (32 - P.ob)) + 1;
            uint32_t len = ref ? (P.lb ? (body << P.ob) >> (32 - P.lb) : 0u) + P.lmin : P.blk;
            o = len;
#pragma unroll
            for (int k = 1; k < 32; k <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, o, k);
                if (lane >= k)
                    o += y;
            }
            o += opos - len;
            const bool valid = o < sg.nbits;
            const uint32_t room = sg.nbits - o, left = sg.code_bits - cpos;
            if (!ref && valid && len > room)
                len = room;
            const uint32_t used = ref ? len_ref : 1 + len;
            const bool bad = valid && (dc + used > left || (ref && (len > P.lmax || len > room ||
                                                                    (P.dict == 2 && d > o))));
            good = !__any_sync(0xffffffffu, bad);
            if (good) {
                const int last = 31 - __clz(__ballot_sync(0xffffffffu, valid));
                opos = __shfl_sync(0xffffffffu, o + len, last);
                cpos += __shfl_sync(0xffffffffu, dc + used, last);
                fr.head += last + 1;
                fr.avail -= last + 1;
                info = valid ? len | (ref ? kTokRef : 0u) | kTokValid : 0u;
                if (opos >= sg.nbits)
                    info |= kTokEnd;
                x = ref ? d : body;
            }
        }
        ended = !good || opos >= sg.nbits;
        if (turn >= 2)
            read_sync(turn);
        DecShared::Batch &bt = sh.batch[turn & 1];
        bt.o[lane] = o;
        bt.info[lane] = info;
        bt.x[lane] = x;
        __threadfence_block();
        full_arrive(turn);
        ++turn;
    }
    return good && cpos == sg.code_bits;
}

// Copy warp's view of the output.
struct Back {
    const uint32_t *ring;
    const uint8_t *y;
    uint32_t flushed;  // output words stored
    // output word q: the dictionary before the segment (q < 0), the ring, or,
    // for windows wider than the ring's history, the output already stored
    __device__ __forceinline__ uint32_t word_at(int32_t q, const LzParams &P) const
    {
        if (q < 0)
            return P.W >= 32 ? dict_word((uint32_t)(q + (int32_t)(P.W / 32)))
                             : dict_word(0) >> (32 - P.W);
        if (q + (int32_t)kDecHistory >= (int32_t)flushed)
            return ring[(uint32_t)q & (kDecRing - 1)];
        return bswap32(__ldcg(reinterpret_cast<const uint32_t *>(y) + q));
    }
    // the 32 bits at output bit s; near: they are in the ring
    __device__ __forceinline__ uint32_t bits_at(int32_t s, const LzParams &P, bool near) const
    {
        const int32_t q = s >> 5;  // floor
        uint32_t a, b;
        if (near) {
            a = ring[(uint32_t)q & (kDecRing - 1)];
            b = ring[(uint32_t)(q + 1) & (kDecRing - 1)];
        } else {
            a = word_at(q, P);
            b = word_at(q + 1, P);
        }
        return __funnelshift_l(b, a, (uint32_t)s & 31u);
    }
};

// Copy warp: write the segment's tokens as they come, 32 at a time.
// A literal is ready at once, a match once the bits it reads lie before the
// first token still waiting (rounds, at most 32; 1.2 on average on the
// bitstream stand-in).  Consecutive matches of one distance d -- the form a
// zero run or any longer repeat takes -- would wait on one another; each
// instead reads the period of d bits before the first of them, at its own
// phase, so the whole run is ready together.  Every 32 completed words leave
// with one coalesced store, and as many words ahead are cleared.
__device__ __forceinline__ void write_segment(const SegIn &sg, DecShared &sh, const LzParams &P,
                                              int lane, uint32_t &turn)
{
    uint32_t first = 0;  // the word being filled
    for (uint32_t q = (uint32_t)lane; q < (sg.raw >> 5); q += 32) {
        const uint32_t v = sg.load(q);
        sh.out[q & (kDecRing - 1)] = v;
        store_out_word(sg.y, sg.m, q, v);
    }
    if (sg.raw & 31u)
        first = sg.load(sg.raw >> 5) & ~(0xffffffffu >> (sg.raw & 31u));
    __syncwarp();
    // the word being filled and the words a batch may reach past it
    Back bk;
    bk.ring = sh.out;
    bk.y = sg.y;
    bk.flushed = sg.raw >> 5;
    for (uint32_t j = (uint32_t)lane; j <= kDecAhead; j += 32)
        sh.out[(bk.flushed + j) & (kDecRing - 1)] = j == 0 ? first : 0u;
    uint32_t opos = sg.raw;
    for (bool more = true; more;) {
        full_sync(turn);
        const DecShared::Batch &bt = sh.batch[turn & 1];
        const uint32_t o = bt.o[lane], info = bt.info[lane], x = bt.x[lane];
        read_arrive(turn);
        ++turn;
        const uint32_t len = info & 63u;
        const bool ref = (info & kTokRef) != 0;
        more = !(info & kTokEnd);  // the same in every lane
        uint32_t pend = __ballot_sync(0xffffffffu, (info & kTokValid) != 0);
        if (pend == 0)
            break;
        const uint32_t refs = __ballot_sync(0xffffffffu, ref);
        const int last = 31 - __clz(pend);
        const uint32_t d = x;  // of a match
        const uint32_t pd = __shfl_up_sync(0xffffffffu, x, 1);
        const bool cont = lane > 0 && ((refs >> lane) & (refs >> (lane - 1)) & 1u) && pd == d;
        const uint32_t heads = refs & ~__ballot_sync(0xffffffffu, cont);
        const uint32_t hl = heads & (0xffffffffu >> (31 - lane));
        const uint32_t o_r = __shfl_sync(0xffffffffu, o, hl ? 31 - __clz(hl) : 0);
        uint32_t phase = o - o_r;
        if (ref && phase >= d)
            phase %= d;
        // bits from the source up to the run's start, and where the reads end
        const uint32_t avail = d - phase;
        const bool wrap = ref && avail < len;  // the period starts again (avail < 32)
        const int32_t src = (int32_t)(o_r - avail), again = (int32_t)(o_r - d);
        const int32_t need = !ref ? INT32_MIN : (int32_t)(wrap ? o_r : o_r - avail + len);
        // the lowest word read: past the dictionary and in the ring?
        const int32_t low = (wrap ? again : src) >> 5;
        const bool near = !__any_sync(
            0xffffffffu, ref && (low < 0 || low + (int32_t)kDecHistory < (int32_t)bk.flushed));
        int32_t front = (int32_t)opos;  // the first token waiting
        for (;;) {
            const bool go = ((pend >> lane) & 1u) && need <= front;
            if (go) {
                uint32_t v = x;
                if (ref) {
                    v = bk.bits_at(src, P, near);
                    if (wrap) {
                        v = (v & ~(0xffffffffu >> avail)) | (bk.bits_at(again, P, near) >> avail);
                        if (d < len) {
                            v &= ~(0xffffffffu >> d);
                            for (uint32_t s = d; s < len; s <<= 1)
                                v |= v >> s;
                        }
                    }
                }
                v &= ~__funnelshift_rc(0xffffffffu, 0u, len);
                const uint32_t sft = o & 31u;
                const uint32_t hi = v >> sft, lo = __funnelshift_l(0u, v, 32u - sft);
                if (hi)
                    atomicOr(sh.out + ((o >> 5) & (kDecRing - 1)), hi);
                if (sft && lo)
                    atomicOr(sh.out + (((o >> 5) + 1) & (kDecRing - 1)), lo);
            }
            pend &= ~__ballot_sync(0xffffffffu, go);
            __syncwarp();
            if (!pend)
                break;
            front = (int32_t)__shfl_sync(0xffffffffu, o, __ffs(pend) - 1);
        }
        opos = __shfl_sync(0xffffffffu, o + len, last);
        if ((opos >> 5) - bk.flushed >= 32) {
            const uint32_t j = bk.flushed + lane;
            __stcg(reinterpret_cast<uint32_t *>(sg.y) + j, bswap32(sh.out[j & (kDecRing - 1)]));
            sh.out[(j + kDecAhead + 1) & (kDecRing - 1)] = 0u;
            bk.flushed += 32;
            __syncwarp();
        }
    }
    for (uint32_t j = bk.flushed + lane; 32 * j < opos; j += 32)
        store_out_word(sg.y, sg.m, j, sh.out[j & (kDecRing - 1)]);
    __syncwarp();
}

// One CTA of two warps per segment.  Bound by the latency of the two warps'
// steps at a thousand segments (64 MiB in 64 KiB segments: 7 CTAs per SM) and
// by instruction issue from about 4000 on.  64 MiB of the bitstream stand-in
// with 1024/12/24/8: 11.9 -> 0.90 ms in 64 KiB segments, 3.35 -> 0.69 ms in
// 16 KiB segments (before: a thread per segment); one warp doing both parts
// took 1.19 ms, and 3.1 ms with a walk over the token flags in registers.
__global__ void __launch_bounds__(64) k_lzss_decode(const uint8_t *__restrict__ c,
                                                    const uint64_t *__restrict__ start,
                                                    uint8_t *__restrict__ out, int32_t *status,
                                                    const uint32_t *path)
{
    __shared__ DecShared sh;
    if (*path != kPathWarps)
        return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t n = *reinterpret_cast<const uint64_t *>(c);
    const uint64_t seg = *reinterpret_cast<const uint64_t *>(c + 8);
    const uint32_t *f = reinterpret_cast<const uint32_t *>(c + 16);
    const LzParams P = make_params(f[0], f[1], f[2], f[3], f[4]);
    const uint64_t count = *reinterpret_cast<const uint64_t *>(c + 40);
    if (warp == 0)
        for (uint32_t e = 0; e < 33; ++e)  // a walk past its stretch has left it
            sh.exits[(kWalkBits + e) * 32 + lane] = (uint16_t)e;
    uint32_t turn = 0;
    for (uint64_t s = blockIdx.x; s < count; s += gridDim.x) {
        SegIn sg;
        sg.m = (uint32_t)(s + 1 < count ? seg : n - s * seg);
        sg.nbits = 8 * sg.m;
        sg.code_bits = *reinterpret_cast<const uint32_t *>(c + kLzHead + 4 * s);
        sg.w = reinterpret_cast<const uint32_t *>(c + start[s]);
        sg.nw = (uint32_t)(al16(((uint64_t)sg.code_bits + 7) / 8) / 4);
        sg.y = out + s * seg;
        sg.raw = P.dict == 2 ? (sg.nbits < P.W ? sg.nbits : P.W) : 0u;
        if (warp == 0) {
            if (!read_segment(sg, sh, P, lane, turn) && lane == 0)
                set_status(status, HUFF_ERR_CORRUPT_STREAM);
        } else {
            write_segment(sg, sh, P, lane, turn);
        }
    }
    if (warp == 0)  // the copy warp's last two reads
        for (uint32_t t = turn < 2 ? 0 : turn - 2; t < turn; ++t)
            read_sync(t);
}

// MSB-first bit reader over a segment's code: a 64-bit buffer refilled from
// the code's 32-bit words (the code starts 16-byte aligned and is padded
// with zeros to a 16-byte boundary; words past the padding read as zero).
// The word after the buffer is always loaded one refill ahead, so the
// load's latency is off the token chain.
struct CodeReader {
    const uint32_t *w;
    uint32_t nw;     // words of the padded code
    uint32_t next;   // next word to load
    uint32_t nxt;    // word next - 1, loaded ahead
    uint64_t buf;    // valid bits, left-aligned
    uint32_t have;
    uint32_t nbits;  // the segment's code length (< 2^28: segments are at most 16 MiB)
    uint32_t pos;    // bits consumed
    __device__ __forceinline__ uint32_t load(uint32_t i) const
    {
        return i < nw ? bswap32(__ldg(w + i)) : 0u;
    }
    __device__ __forceinline__ void init(const uint8_t *c, uint64_t code_bits)
    {
        w = reinterpret_cast<const uint32_t *>(c);
        nw = (uint32_t)(al16((code_bits + 7) / 8) / 4);
        buf = ((uint64_t)load(0) << 32) | load(1);
        have = 64;
        nxt = load(2);
        next = 3;
        nbits = (uint32_t)code_bits;
        pos = 0;
    }
    __device__ __forceinline__ uint32_t get(uint32_t k)  // k <= 32 bits, right-aligned
    {
        if (k == 0)
            return 0;
        const uint32_t v = (uint32_t)(buf >> (64 - k));
        buf <<= k;
        have -= k;
        pos += k;
        if (have <= 32) {  // refill: >= 32 valid bits for the next get
            buf |= (uint64_t)nxt << (32 - have);
            have += 32;
            nxt = load(next++);
        }
        return v;
    }
};

// The bits a thread has produced so far, read back: with kRing from the
// thread's ring of recent words in shared memory, else from the output; the
// word being filled is in a register, and bits before the segment are the
// dictionary's.  With the ring, completed words are written out four at a time
// with one 16-byte store.
template <bool kRing>
struct OutBits {
    uint8_t *y;      // the segment's output (16-byte aligned)
    uint32_t m;      // its bytes (at most 16 MiB)
    uint32_t W;
    uint32_t *ring;  // kThrRing words, word q at q mod kThrRing
    uint32_t pend;   // bits of the word being filled, left-aligned
    uint32_t npend;  // their count
    uint32_t pos;    // bits produced (< 2^27)
    __device__ __forceinline__ uint32_t word_at(int32_t q) const
    {
        const int32_t cur = (int32_t)(pos >> 5);
        if (q < 0)
            return W >= 32 ? dict_word((uint32_t)(q + (int32_t)(W / 32))) : dict_word(0) >> (32 - W);
        if (q >= cur)
            return q == cur ? pend : 0u;
        return kRing ? ring[(uint32_t)q & (kThrRing - 1)]
                     : bswap32(__ldcg(reinterpret_cast<const uint32_t *>(y) + q));
    }
    // the 32 bits at output bit s (at most W bits before the segment)
    __device__ __forceinline__ uint32_t bits_at(int32_t s) const
    {
        const int32_t q = s >> 5;  // floor
        return __funnelshift_l(word_at(q + 1), word_at(q), (uint32_t)s & 31u);
    }
    // append the top k (1..32) bits of v
    __device__ __forceinline__ void put(uint32_t v, uint32_t k)
    {
        v = k < 32 ? v & ~(0xffffffffu >> k) : v;
        const uint64_t acc = ((uint64_t)pend << 32) | ((uint64_t)v << (32 - npend));
        const uint32_t total = npend + k;
        if (total >= 32) {
            complete(pos >> 5, (uint32_t)(acc >> 32));
            pend = (uint32_t)acc;
            npend = total - 32;
        } else {
            pend = (uint32_t)(acc >> 32);
            npend = total;
        }
        pos += k;
    }
    __device__ __forceinline__ void complete(uint32_t q, uint32_t w) const
    {
        if (!kRing) {
            store_out_word(y, m, q, w);
            return;
        }
        ring[q & (kThrRing - 1)] = w;
        if ((q & 3) == 3) {  // a whole 16-byte group
            const uint32_t g = q >> 2;
            if (16 * g + 16 <= m) {
                const uint32_t r = (q - 3) & (kThrRing - 1);
                *reinterpret_cast<uint4 *>(y + 16 * g) =
                    make_uint4(bswap32(ring[r]), bswap32(ring[r + 1]), bswap32(ring[r + 2]),
                               bswap32(ring[r + 3]));
            } else {
                for (uint32_t j = q - 3; j <= q; ++j)
                    store_out_word(y, m, j, ring[j & (kThrRing - 1)]);
            }
        }
    }
    __device__ __forceinline__ void finish() const
    {
        const uint32_t q = pos >> 5;  // the word being filled
        if (kRing)  // completed words of the last, unfinished group
            for (uint32_t j = q & ~3u; j < q; ++j)
                store_out_word(y, m, j, ring[j & (kThrRing - 1)]);
        if (npend)
            store_out_word(y, m, q, pend);
    }
};

// The code words of the fast loop below come through a per-thread ring of
// kLzInCells 16-byte cells in shared memory ([cell][thread], 512-byte rows),
// filled by cp.async copies kept ahead of the reader: the 32 lanes of a warp
// refill at different tokens, and a refill that waited on a global load
// would wait on the one another lane issued a token before (the scoreboard
// is the warp's), which left most of the load latency exposed.
__device__ __forceinline__ void lz_cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void lz_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void lz_cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

struct CodeRing {
    uint32_t col;      // shared address of this thread's cell in row 0
    uint32_t fetched;  // cells requested so far (cell c holds code words 4c..4c+3)
    uint32_t ncells;   // cells of the segment's code (its 16-byte padded length)
    // request cells until the ring holds the kLzInCells from word w's on
    __device__ __forceinline__ void top_up(const uint32_t *w, uint32_t word)
    {
        while (fetched < (word >> 2) + kLzInCells && fetched < ncells) {
            lz_cp_async16(col + (fetched & (kLzInCells - 1)) * (kThrBlock * 16), w + 4 * fetched);
            lz_cp_commit();
            ++fetched;
        }
    }
    // code word `word` right after top_up(w, word): unless the code's last
    // cell has been requested, exactly kLzInFlight cells were requested after
    // word's (one copy group each), so waiting for all but that many to land
    // includes word's; after the last cell every copy is waited for.  A slot
    // is requested again only once the reader has left its cell.
    __device__ __forceinline__ uint32_t word_at(uint32_t word) const
    {
        if (fetched >= ncells)
            lz_cp_wait<0>();
        else
            lz_cp_wait<kLzInFlight>();
        return lds(col + ((word >> 2) & (kLzInCells - 1)) * (kThrBlock * 16) + (word & 3u) * 4);
    }
};

// Tokens far from both ends of a segment, for the shared-memory ring
// (windows of 32..2048 bits) with the stored-prefix window and literal blocks
// of at most 31 bits: at least 64 code bits and 32 output bits remain, so no
// bounds check applies, the window never reaches before the output (the
// prefix filled it) and a token is at most 32 bits of the reader's top 32.
// Branch free where the lanes of a warp (each on its own segment) would
// diverge: both the match and the literal are formed and the token
// selects.  False (and the caller's status) only for a length field above
// the longest match.
__device__ __forceinline__ bool decode_fast(CodeReader &rd, OutBits<true> &ob, const LzParams &P,
                                            uint32_t nbits, uint32_t in_col)
{
    CodeRing rg;
    rg.col = in_col;
    rg.fetched = rd.next >> 2;
    rg.ncells = rd.nw >> 2;
    rg.top_up(rd.w, rd.next);
    bool ok = true;
    while (rd.pos + 64 <= rd.nbits && ob.pos + 32 <= nbits) {
        const uint32_t t = (uint32_t)(rd.buf >> 32);  // >= 33 bits are valid
        const uint32_t flag = t >> 31;
        const uint32_t body = t << 1;  // the token after its flag, left-aligned
        const uint32_t d = (body >> (32 - P.ob)) + 1;
        const uint32_t len = (P.lb ? (body << P.ob) >> (32 - P.lb) : 0u) + P.lmin;
        if (flag && len > P.lmax) {
            ok = false;
            break;
        }
        const uint32_t used = flag ? 1u + P.ob + P.lb : 1u + P.blk;
        const uint32_t nout = flag ? len : P.blk;
        // the match's 32 source bits at ob.pos - d (at most W back, so inside
        // the output and the ring; read whether or not the token is a match)
        const uint32_t src = ob.pos - d;
        const uint32_t q = src >> 5, cur = ob.pos >> 5;
        const uint32_t wa = ob.ring[q & (kThrRing - 1)], wb = ob.ring[(q + 1) & (kThrRing - 1)];
        const uint32_t a = q == cur ? ob.pend : wa;
        const uint32_t b = q + 1 == cur ? ob.pend : (q + 1 > cur ? 0u : wb);
        uint32_t v = __funnelshift_l(b, a, src & 31u);
        // a source that runs into the bits being produced repeats with period d
        uint32_t vp = v & ~(0xffffffffu >> (d & 31u));
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const uint32_t sh = d << i;
            vp |= sh < len ? vp >> (sh & 31u) : 0u;
        }
        v = flag ? (d < len ? vp : v) : body;
        // consume the token: one refill keeps >= 33 bits; the next word
        // comes from the ring (zero past the padded code, as rd.load gives)
        rd.buf <<= used;
        rd.have -= used;
        rd.pos += used;
        if (rd.have <= 32) {
            rd.buf |= (uint64_t)rd.nxt << (32 - rd.have);
            rd.have += 32;
            uint32_t nw = 0u;
            if (rd.next < rd.nw) {
                rg.top_up(rd.w, rd.next);
                nw = bswap32(rg.word_at(rd.next));
            }
            rd.nxt = nw;
            ++rd.next;
        }
        ob.put(v, nout);
    }
    lz_cp_wait<0>();  // no copy in flight into the ring once the loop is left
    return ok;
}

// Decode one segment's tokens; false if the code is corrupt.
template <bool kRing>
__device__ __forceinline__ bool decode_segment(CodeReader &rd, OutBits<kRing> &ob, const LzParams &P,
                                               uint32_t nbits, uint32_t in_col)
{
    const uint32_t raw = P.dict != 2 ? 0u : nbits < P.W ? nbits : P.W;
    while (ob.pos < raw) {
        const uint32_t k = raw - ob.pos < 32 ? raw - ob.pos : 32u;
        if (rd.pos + k > rd.nbits)
            return false;
        ob.put(rd.get(k) << (32 - k), k);
    }
    if constexpr (kRing) {
        if (P.dict == 2 && P.blk <= 31 && !decode_fast(rd, ob, P, nbits, in_col))
            return false;
    }
    while (ob.pos < nbits) {
        if (rd.pos >= rd.nbits)
            return false;
        const uint32_t r = nbits - ob.pos;
        if (rd.get(1)) {
            if (rd.pos + P.ob + P.lb > rd.nbits)
                return false;
            const uint32_t d = rd.get(P.ob) + 1;
            const uint32_t len = rd.get(P.lb) + P.lmin;
            if (len > P.lmax || len > r || (P.dict == 2 && d > ob.pos))
                return false;
            uint32_t v = ob.bits_at((int32_t)ob.pos - (int32_t)d);
            if (d < len) {  // the source runs into these bits: period d
                v &= ~(0xffffffffu >> d);
                for (uint32_t sh = d; sh < len; sh <<= 1)
                    v |= v >> sh;
            }
            ob.put(v, len);
        } else {
            const uint32_t k = r < P.blk ? (uint32_t)r : P.blk;
            if (rd.pos + k > rd.nbits)
                return false;
            ob.put(rd.get(k) << (32 - k), k);
        }
    }
    return rd.pos == rd.nbits;
}

// One thread per segment, for very many segments (see threads_better).
__global__ void __launch_bounds__(kThrBlock)
    k_lzss_decode_threads(const uint8_t *__restrict__ c, const uint64_t *__restrict__ start,
                          uint8_t *__restrict__ out, int32_t *status, const uint32_t *path)
{
    // ring of thread t at t * (kThrRing + 1): the odd stride spreads the
    // threads' equal ring positions over the banks
    __shared__ uint32_t rings[kThrBlock * (kThrRing + 1)];
    __shared__ __align__(16) uint4 cells[kLzInCells * kThrBlock];  // [cell][thread]
    if (*path != kPathThreads)
        return;
    const uint32_t in_col = smem_u32(cells) + threadIdx.x * 16;
    const uint64_t n = *reinterpret_cast<const uint64_t *>(c);
    const uint64_t seg = *reinterpret_cast<const uint64_t *>(c + 8);
    const uint32_t *f = reinterpret_cast<const uint32_t *>(c + 16);
    const LzParams P = make_params(f[0], f[1], f[2], f[3], f[4]);
    const uint64_t count = *reinterpret_cast<const uint64_t *>(c + 40);
    const bool in_ring = P.W >= 32 && P.W <= kThrMaxWindow;
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < count;
         s += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t m = (uint32_t)(s + 1 < count ? seg : n - s * seg);
        CodeReader rd;
        rd.init(c + start[s], *reinterpret_cast<const uint32_t *>(c + kLzHead + 4 * s));
        auto decode = [&](auto ob) {
            ob.y = out + s * seg;
            ob.m = m;
            ob.W = P.W;
            ob.ring = rings + threadIdx.x * (kThrRing + 1);
            ob.pend = ob.npend = ob.pos = 0;
            const bool good = decode_segment(rd, ob, P, 8 * m, in_col);
            if (good)
                ob.finish();
            return good;
        };
        if (!(in_ring ? decode(OutBits<true>()) : decode(OutBits<false>())))
            set_status(status, HUFF_ERR_CORRUPT_STREAM);
    }
}

__global__ void k_lzss_set(int32_t *status, unsigned long long *p, uint64_t v)
{
    *status = 0;
    if (p)
        *p = v;
}

// Parts of a segment: 8 where that makes up to 15 warps per SM, 4 or 2 up to 27
// (more parts mean more joins one after the other, and a full chip gains
// nothing), of 4 KiB at least, if the slots hold them.  64 KiB segments with
// 1024/12/24/8, one warp a segment against parts: 64 segments 3.60 / 1.10 ms (8
// parts), 256: 3.80 / 1.57, 512: 3.82 / 2.03 (4 parts; 8: 2.18), 1024: 4.40 /
// 2.99 (4; 8: 3.14); 4096 segments of 16 KiB 2.38 / 2.80 (2 parts), so none.
PartsLayout parts_of(uint64_t n, uint64_t seg, uint64_t count, const LzParams &P, uint64_t sms)
{
    PartsLayout L = {1, 0, 0, 0};
    if (!ring_ok(P) || P.lmax < 8 || n == 0)
        return L;
    const uint64_t ref = 1 + P.ob + P.lb, lit = 1 + P.blk;
    for (uint64_t k = kMaxParts; k > 1; k >>= 1) {
        if (seg / k < kMinPart || count * k > (k > 4 ? 15 : 27) * sms)
            continue;
        // a part's bits, the last step's past its end, each at the rate of the
        // kind of token that grows it most
        const uint64_t bits = 8 * seg / k + 1 + 1024 + 64;
        const uint64_t code = (ref * P.blk > lit * P.lmin ? (bits * ref + P.lmin - 1) / P.lmin
                                                          : (bits * lit + P.blk - 1) / P.blk) +
                              2 * (ref > lit ? ref : lit) + P.W;
        const uint64_t bytes = al16(code / 8 + 16);
        // the rest of the slot for the bits before the meeting points: few
        // tokens but for the runs among them (28 K bits at most in 500 parts of
        // the stand-in)
        const uint64_t stride = (slot_bytes(seg, P) - 32) / k & ~15ull;
        const uint64_t fixed = 16 + bytes + 8 * kMarks;
        if (stride < fixed + bytes / 4 + 512 || 8 * k * stride >> 32)
            continue;  // (bit positions in a slot are 32 bits wide)
        const uint64_t head = stride - fixed;
        L.parts = (uint32_t)k;
        L.code = (uint32_t)bytes;
        L.head = (uint32_t)head;
        L.stride = (uint32_t)stride;
        return L;
    }
    return L;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool host_params(const huff_lzss_params_t *p, LzParams &P)
{
    if (!p || !params_ok(p->window, p->min_len, p->max_len, p->block, p->dict))
        return false;
    P = make_params(p->window, p->min_len, p->max_len, p->block, p->dict);
    return true;
}

bool seg_ok(uint64_t seg) { return seg >= 16 && seg % 16 == 0 && seg <= kMaxSegment; }

}  // namespace
}  // namespace huff

using namespace huff;

extern "C" {

uint64_t huff_lzss_max_size(uint64_t n, uint64_t segment_bytes, const huff_lzss_params_t *params)
{
    LzParams P;
    if (!host_params(params, P) || !seg_ok(segment_bytes))
        return 0;
    const uint64_t count = n ? (n + segment_bytes - 1) / segment_bytes : 0;
    return al16(kLzHead + 4 * count) + count * slot_bytes(segment_bytes, P);
}

uint64_t huff_lzss_workspace_size(uint64_t n, uint64_t segment_bytes,
                                  const huff_lzss_params_t *params)
{
    LzParams P;
    if (!host_params(params, P) || !seg_ok(segment_bytes))
        return 0;
    const uint64_t count = n ? (n + segment_bytes - 1) / segment_bytes : 0;
    // slots, then the bit lengths (u32) and the starts (u64)
    return count * slot_bytes(segment_bytes, P) + al16(4 * count) + 8 * count + 16;
}

huff_status_t huff_lzss_compress(const uint8_t *d_in, uint64_t n, uint64_t segment_bytes,
                                 const huff_lzss_params_t *params, uint8_t *d_out, uint64_t out_cap,
                                 uint64_t *d_out_bytes, void *d_ws, uint64_t ws_bytes,
                                 int32_t *d_status, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_lzss_compress");
    LzParams P;
    if (!host_params(params, P) || !seg_ok(segment_bytes) || !d_out || !d_out_bytes ||
        !d_status || (n && (!d_in || !aligned16(d_in))) || !aligned16(d_out) ||
        (n && (!d_ws || !aligned16(d_ws))) ||
        ws_bytes < huff_lzss_workspace_size(n, segment_bytes, params))
        return HUFF_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_lzss_set<<<1, 1, 0, s>>>(d_status, reinterpret_cast<unsigned long long *>(d_out_bytes), 0);
    const uint64_t count = n ? (n + segment_bytes - 1) / segment_bytes : 0;
    uint8_t *ws = static_cast<uint8_t *>(d_ws);
    uint8_t *slots = ws;
    uint32_t *bits = reinterpret_cast<uint32_t *>(ws + count * slot_bytes(segment_bytes, P));
    uint64_t *start = reinterpret_cast<uint64_t *>(reinterpret_cast<uint8_t *>(bits) + al16(4 * count));
    const int sms = device_sm_count();
    if (sms < 1)
        return HUFF_ERR_CUDA;
    const PartsLayout L = parts_of(n, segment_bytes, count, P, (uint64_t)sms);
    if (count) {
        if (ring_ok(P)) {
            const size_t smem = 2 * (size_t)ring_words(P.W) * 4;  // at most 8 KB
            const auto grid = [&](uint64_t warps) {
                return (unsigned)(warps < (uint64_t)sms * 64 ? warps : (uint64_t)sms * 64);
            };
            auto run = [&](auto g0) {
                constexpr int G0 = decltype(g0)::value;
                if (L.parts > 1) {
                    k_lzss_parts<G0><<<grid(count * L.parts), 32, smem, s>>>(
                        d_in, n, segment_bytes, P, L, slots, d_status);
                    k_lzss_join<G0><<<grid(count), 32, smem, s>>>(d_in, n, segment_bytes, P, L, slots,
                                                                  bits, d_status);
                } else {
                    k_lzss_compress_ring<G0><<<grid(count), 32, smem, s>>>(d_in, n, segment_bytes, P,
                                                                           slots, bits, d_status);
                }
            };
            const bool many = count >= 50 * (uint64_t)sms;
            switch (by_distance(P, many) ? -1 : (int)(P.lmin / 4)) {
            case -1: run(std::integral_constant<int, -1>()); break;
            case 0: run(std::integral_constant<int, 0>()); break;
            case 1: run(std::integral_constant<int, 1>()); break;
            case 2: run(std::integral_constant<int, 2>()); break;
            case 3: run(std::integral_constant<int, 3>()); break;
            case 4: run(std::integral_constant<int, 4>()); break;
            case 5: run(std::integral_constant<int, 5>()); break;
            default: run(std::integral_constant<int, 6>()); break;
            }
        } else {
            uint64_t grid = (count + kLzWarps - 1) / kLzWarps;
            if (grid > (uint64_t)sms * 64)
                grid = (uint64_t)sms * 64;
            k_lzss_compress<<<(unsigned)grid, kLzBlock, 0, s>>>(d_in, n, segment_bytes, P, slots,
                                                                bits, d_status);
        }
    }
    k_lzss_layout<<<1, kScanBlock, 0, s>>>(n, segment_bytes, P, bits, start, d_out, out_cap,
                                           reinterpret_cast<unsigned long long *>(d_out_bytes),
                                           d_status);
    if (count) {
        const uint64_t grid = count < (uint64_t)sms * 16 ? count : (uint64_t)sms * 16;
        if (L.parts > 1)
            k_lzss_gather_parts<<<(unsigned)grid, 256, 0, s>>>(n, segment_bytes, P, L, slots, bits,
                                                               start, d_out, out_cap, d_status);
        else
            k_lzss_gather<<<(unsigned)grid, 128, 0, s>>>(n, segment_bytes, P, slots, bits, start,
                                                         d_out, out_cap, d_status);
    }
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

uint64_t huff_lzss_decompress_workspace_size(uint64_t in_bytes)
{
    const uint64_t max_count = in_bytes > kLzHead ? (in_bytes - kLzHead) / 4 : 0;
    return 16 + 8 * max_count;
}

huff_status_t huff_lzss_decompress(const uint8_t *d_in, uint64_t in_bytes, uint8_t *d_out,
                                   uint64_t out_cap, uint64_t *d_n, void *d_ws, uint64_t ws_bytes,
                                   int32_t *d_status, huff_stream_t stream)
{
    HUFF_API_RANGE("huff_lzss_decompress");
    if (!d_in || !aligned16(d_in) || !d_n || !d_status || (out_cap && !d_out) ||
        (d_out && !aligned16(d_out)) || !d_ws || !aligned16(d_ws) ||
        ws_bytes < huff_lzss_decompress_workspace_size(in_bytes))
        return HUFF_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_lzss_set<<<1, 1, 0, s>>>(d_status, reinterpret_cast<unsigned long long *>(d_n), 0);
    const uint64_t max_count = in_bytes > kLzHead ? (in_bytes - kLzHead) / 4 : 0;
    const int sms = device_sm_count();
    if (sms < 1)
        return HUFF_ERR_CUDA;
    uint32_t *path = static_cast<uint32_t *>(d_ws);
    uint64_t *start = reinterpret_cast<uint64_t *>(static_cast<uint8_t *>(d_ws) + 16);
    k_lzss_dlayout<<<1, kScanBlock, 0, s>>>(d_in, in_bytes, out_cap, start, max_count,
                                            reinterpret_cast<unsigned long long *>(d_n), d_status,
                                            path, (uint32_t)sms);
    // the count is only known on the device, so bound the grids by the table
    // size; the decoder that k_lzss_dlayout did not choose returns at once
    uint64_t grid = max_count;
    if (grid > (uint64_t)sms * 32)
        grid = (uint64_t)sms * 32;
    if (grid < 1)
        grid = 1;
    k_lzss_decode<<<(unsigned)grid, 64, 0, s>>>(d_in, start, d_out, d_status, path);
    k_lzss_decode_threads<<<(unsigned)grid, kThrBlock, 0, s>>>(d_in, start, d_out, d_status, path);
    return cudaGetLastError() == cudaSuccess ? HUFF_OK : HUFF_ERR_CUDA;
}

}  // extern "C"
