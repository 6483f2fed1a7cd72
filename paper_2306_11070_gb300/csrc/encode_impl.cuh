// Encoder device routines, shared by the single-stream kernel (encode.cu)
// and the fused batched kernel (batch.cu).  See encode.cu for the design.
#pragma once

#include "huff_internal.cuh"

namespace huff {
namespace enc {

// 32 symbols per lane and step, 1024 per warp step, 16 steps per unit
constexpr int kStepSyms = 32;
constexpr int kStep = 32 * kStepSyms;
constexpr int kSteps = kUnitSymbols / kStep;
// 32-bit codes: 16 symbols per lane and step
constexpr int kLongSyms = 16;
constexpr int kLongStep = 32 * kLongSyms;
constexpr int kLongSteps = kUnitSymbols / kLongStep;
constexpr uint32_t kMadMaxLen = 31;  // a group's marker takes a bit
// warp buffer: a guard word, then a step of 1024 codes after < 32 carried bits
constexpr int kWarpObuf = 1 + kStep * (int)kMadMaxLen / 32 + 15;
// Code table: 256 rows of 64 words, of which a stream uses one half (16
// columns of two words: lanes l and l + 16 share a column, and still no lookup
// collides, because a warp's 64-bit loads are made for 16 lanes at a time).
// The two halves of a row belong to two streams where two are written at once.
constexpr int kTblRow = 64;
constexpr int kTblWords = 256 * kTblRow;  // 64 KiB

// One stream being written: input, unit offsets, output layout.
struct Job {
    const uint8_t *in;
    uint64_t n;
    uint32_t cs;
    const unsigned long long *unit_off;  // exclusive bit prefix per unit, total at [units]
    uint64_t units;
    uint8_t *out;
    uint64_t out_cap;
    uint64_t pay0;  // payload byte offset
    uint64_t cap_words;
    bool table_fits;
};

__device__ __forceinline__ Job make_job(const uint8_t *in, uint64_t n, uint32_t cs,
                                        const unsigned long long *unit_off, uint8_t *out,
                                        uint64_t out_cap)
{
    Job j;
    j.in = in;
    j.n = n;
    j.cs = cs;
    j.unit_off = unit_off;
    j.units = (n + kUnitSymbols - 1) / kUnitSymbols;
    j.out = out;
    j.out_cap = out_cap;
    const uint64_t chunks = n ? ceil_div_u64(n, cs) : 0;
    j.pay0 = kHeaderBytes + 8 * chunks;
    j.table_fits = j.pay0 <= out_cap;
    j.cap_words = j.table_fits ? (out_cap - j.pay0) / 4 : 0;
    return j;
}

// Header (threads 0..255 of the calling CTA) and the stream size.
__device__ __forceinline__ void write_header(const Job &J, const huff_codebook_t *cb,
                                             unsigned long long *out_bytes, int32_t *status)
{
    const int tid = threadIdx.x;
    if (J.out_cap >= kHeaderBytes) {
        if (tid < 256)
            J.out[tid] = cb->len[tid];
        if (tid == 0) {
            *reinterpret_cast<uint64_t *>(J.out + 256) = J.n;
            *reinterpret_cast<uint32_t *>(J.out + 264) = J.cs;
            *reinterpret_cast<uint32_t *>(J.out + 268) = cb->max_len;
        }
    }
    if (tid == 0) {
        const uint64_t total = J.units ? J.unit_off[J.units] : 0;
        *out_bytes = J.pay0 + 4 * ((total + 31) >> 5);
        if (!J.table_fits)
            set_status(status, HUFF_ERR_CAPACITY);
    }
}

// Zero this warp's buffer (kWarpObuf words at wob); every step leaves the
// words it used zero again, so this runs once per unit.
__device__ __forceinline__ void clear_buffer(uint32_t *wob, int lane)
{
    for (int j = lane; j < kWarpObuf; j += 32)
        wob[j] = 0u;
    __syncwarp();
}

template <int N>
__device__ __forceinline__ uint32_t byte_of(const uint32_t (&w)[N], int k)
{
    return __byte_perm(w[k >> 2], 0u, 0x4440u | (uint32_t)(k & 3));
}

__device__ __forceinline__ void red_or(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Shared per-unit state of the encoders below.
struct UnitState {
    uint64_t base;   // first symbol of the unit
    uint64_t gbit;   // stream bit of the next step's first symbol
    uint32_t carry;  // bits of the partial word before the step, high-aligned
    uint32_t lead;   // distance from the step start to the next chunk start
    uint64_t next_chunk;  // index of that chunk
};

// This lane's SPT input bytes of the step starting at symbol sb (m of them
// real, the rest zero), read straight from the input (partial steps only).
template <int SPT>
__device__ __forceinline__ int step_input_tail(const Job &J, uint64_t sb, int lane,
                                               uint32_t (&w)[SPT / 4])
{
    const uint64_t i0 = sb + (uint64_t)lane * SPT;
    const int m = i0 >= J.n ? 0 : (J.n - i0 >= (uint64_t)SPT ? SPT : (int)(J.n - i0));
#pragma unroll
    for (int j = 0; j < SPT / 4; ++j)
        w[j] = 0u;
#pragma unroll
    for (int k = 0; k < SPT; ++k)
        if (k < m)
            w[k >> 2] |= (uint32_t)J.in[i0 + k] << (8 * (k & 3));
    return m;
}

// Inclusive warp scan of the lanes' bit counts: (exclusive position, total).
__device__ __forceinline__ void scan_bits(uint32_t bits, int lane, uint32_t &pos, uint32_t &total)
{
    uint32_t incl = bits;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d)
            incl += v;
    }
    pos = incl - bits;
    total = __shfl_sync(0xffffffffu, incl, 31);
}

// Chunk offsets: the stream bit of every chunk that starts at one of this
// lane's symbols.  A chunk starts at a multiple of cs, itself a multiple of
// 16, so only at lane offset 0 or 16 (mid16: the bits of the lane's first 16
// symbols; only used when SPT = 32).
template <int SPT, int STEP>
__device__ __forceinline__ void step_chunks(const Job &J, const UnitState &st, uint64_t sb, int lane,
                                            uint32_t pos, uint32_t mid16)
{
    if (!J.table_fits || (J.cs >= (uint32_t)STEP && st.lead >= (uint32_t)STEP))
        return;
    uint64_t *offs = reinterpret_cast<uint64_t *>(J.out + kHeaderBytes);
#pragma unroll
    for (int off = 0; off < SPT; off += 16) {
        const uint32_t d = (uint32_t)lane * SPT + off;
        const uint64_t bit = st.gbit + pos + (off ? mid16 : 0u);
        if (J.cs >= (uint32_t)STEP) {  // at most one start per step
            stg64_if(d == st.lead && sb + d < J.n, offs + st.next_chunk, bit);
        } else if (d >= st.lead && (d - st.lead) % J.cs == 0 && sb + d < J.n) {
            offs[(sb + d) / J.cs] = bit;
        }
    }
}

template <int STEP>
__device__ __forceinline__ void step_advance(const Job &J, UnitState &st, uint32_t step_bits)
{
    st.gbit += step_bits;
    if (st.lead >= (uint32_t)STEP) {
        st.lead -= STEP;
    } else if (J.cs >= (uint32_t)STEP) {
        st.lead = J.cs - (STEP - st.lead);
        ++st.next_chunk;
    } else {
        st.lead = (J.cs - (STEP - st.lead) % J.cs) % J.cs;
    }
}

// Whole words of the step out (coalesced); the partial last word is carried
// into the next step, or left to the next unit's seam at the unit end.
// kChecked: bound checks against the output capacity (else the words surely
// fit) and every word read cleared again for the next step's OR-ing.
// Returns true on overflow.
template <bool kChecked>
__device__ __forceinline__ bool step_output(const Job &J, UnitState &st, bool last, uint32_t step_bits,
                                            uint32_t *wob, int lane)
{
    uint32_t *pay = reinterpret_cast<uint32_t *>(J.out + J.pay0);
    const uint32_t r = (uint32_t)(st.gbit & 31);
    const uint32_t nw = (r + step_bits + 31) >> 5;
    const uint32_t tail = (r + step_bits) & 31u;
    const uint32_t nwrite = (last || tail == 0) ? nw : nw - 1;
    const uint64_t wbase = st.gbit >> 5;
    bool overflow = false;
    const uint32_t carry = tail ? wob[nw - 1] : 0u;
    if (!kChecked || wbase + nwrite <= J.cap_words) {
        for (uint32_t j0 = 0; j0 < nw; j0 += 32) {
            const uint32_t j = j0 + lane;
            const uint32_t v = j < nw ? wob[j] : 0u;
            stg_if(j < nwrite, pay + wbase + j, v);
            if (kChecked && j < nw)
                wob[j] = 0u;
        }
    } else {
        for (uint32_t j = lane; j < nw; j += 32) {
            if (j < nwrite) {
                if (wbase + j < J.cap_words)
                    pay[wbase + j] = wob[j];
                else
                    overflow = true;
            }
            wob[j] = 0u;
        }
    }
    st.carry = carry;
    return overflow;
}

__device__ __forceinline__ void load32(const uint8_t *p, uint32_t (&w)[8])
{
    const uint4 a = ld_stream16(p), b = ld_stream16(p + 16);
    w[0] = a.x;
    w[1] = a.y;
    w[2] = a.z;
    w[3] = a.w;
    w[4] = b.x;
    w[5] = b.y;
    w[6] = b.z;
    w[7] = b.w;
}

// The steps of unit u that need no bound checks: those that lie inside the
// input, if the unit's words (a last partial word included) fit the output.
// Only what is left of the last unit takes the checked step, with its byte
// loads and shared ORs; checking that whole unit made one warp run 60 us at
// 64 MiB where the others took 41.
__device__ __forceinline__ int full_steps(const Job &J, uint64_t u)
{
    if (((J.unit_off[u + 1] + 31) >> 5) > J.cap_words)
        return 0;
    const uint64_t left = (J.n - u * kUnitSymbols) / kStep;
    return left < (uint64_t)kSteps ? (int)left : kSteps;
}

// ---- codes gathered by multiply-add ------------------------------------------
// A group of codes is gathered on the FMA pipe: the table holds (code, 2^len)
// per byte and column, and a = a * 2^len + code appends a code to the group's
// bits; a starts at 1, so its leading one marks the group's length (a group
// has at most 31 bits).  Per code that is one byte permutation (which is the
// table address), one table load (8 bytes) and one IMAD; only the group pays
// for its length, its place and the store.  (Two funnel shifts per code into a
// 64-bit window are bound by the ALU pipe: 4096 buffers of 2 GB in all take
// 1977 us instead of 1913.)  The groups of a lane are cut at its 16th
// symbol too, where a chunk may start.
//  - Longest code of at most 10 bits: groups of floor(31 / longest) codes, at
//    least 3, always fit.
//  - Longer codes are rare wherever there are any: the groups take 4 codes
//    where the average is at most 4 bits, else 3, and a multiply-add whose
//    high word is not zero shows the group that does not fit; its step and the
//    rest of the unit then go in pairs, if two codes always fit (at most 15
//    bits), else code by code.  On geometric bytes (longest 25 to 29 bits,
//    average 2) 64 MiB take 114 us instead of 211 and 1 GiB 911 instead of
//    2127.  The same guess for codes of at most 10 bits (4 for 3) gained 2 to
//    4% on text and lost as much on Zipf bytes, where every unit has a group
//    that does not fit: not done.

// How the codes of a stream are written: 32-bit codes one by one; 3 or 4 at a
// time because they nearly always fit, else one by one or in pairs; 3, 4, 8 or
// 16 at a time because they fit.
enum Plan { kLong, kTry3, kTry4, kPairs3, kPairs4, kFit3, kFit4, kFit8, kFit16 };

__device__ __forceinline__ int plan_of(const Job &J, uint32_t max_len)
{
    if (max_len > kMadMaxLen)
        return kLong;
    const uint32_t fit = max_len ? 31u / max_len : 16u;
    if (fit >= 3)
        return fit >= 16 ? kFit16 : fit >= 8 ? kFit8 : fit >= 4 ? kFit4 : kFit3;
    const bool four = J.units && J.unit_off[J.units] <= 4 * J.n;
    return fit == 2 ? (four ? kPairs4 : kPairs3) : four ? kTry4 : kTry3;
}

// A stream's half of the code table, built by threads tid = 0..nt-1: one or
// two threads per byte read its length and code once and fill the byte's 16
// columns with 16-byte stores, rotated by the byte so that a warp's stores
// spread over all eight 16-byte bank groups.  32-bit codes: 16 words of code,
// then 16 of length.
__device__ __forceinline__ void build_table(const huff_codebook_t *cb, uint32_t *tbl, bool pairs, int tid,
                                            int nt)
{
    for (int b = tid; b < 256; b += nt) {
        const uint32_t L = cb->len[b];
        const uint32_t c = L ? cb->code[b] : 0u;
        const uint32_t p = 1u << (L & 31u);  // 2^0 = 1 for a byte without a code: no bits
        uint4 *row = reinterpret_cast<uint4 *>(tbl + b * kTblRow);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = (j + b) & 7;
            row[k] = pairs ? make_uint4(c, p, c, p) : k < 4 ? make_uint4(c, c, c, c) : make_uint4(L, L, L, L);
        }
    }
}

// The last r (< 32) bits of the code stream before symbol `base` (> 0), as the
// high bits of a word: lane l re-codes byte base-1-l.  Warp-uniform result.
template <bool kPairs>
__device__ __forceinline__ uint32_t seam_word(const uint8_t *in, uint64_t base, uint32_t r,
                                              const uint32_t *tbl, int lane)
{
    const uint32_t *e = tbl + (uint32_t)in[base - 1 - lane] * kTblRow;
    uint32_t L, code;
    if (kPairs) {
        const uint2 x = reinterpret_cast<const uint2 *>(e)[lane & 15];
        code = x.x;
        L = 31u - __clz(x.y);
    } else {
        code = e[lane & 15];
        L = e[16 + (lane & 15)];
    }
    uint32_t sfx = L;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, sfx, d);
        if (lane >= d)
            sfx += v;
    }
    const uint32_t before = sfx - L;  // bits between this code's end and base
    const uint32_t part = (L && before < r) ? code << (32 - r + before) : 0u;
    return __reduce_or_sync(0xffffffffu, part);
}

template <bool kPairs>
__device__ __forceinline__ UnitState unit_start(const Job &J, uint64_t u, const uint32_t *tbl, int lane)
{
    UnitState st;
    st.base = u * kUnitSymbols;
    st.gbit = J.unit_off[u];
    st.carry = (st.base > 0 && (st.gbit & 31))
                   ? seam_word<kPairs>(J.in, st.base, (uint32_t)(st.gbit & 31), tbl, lane)
                   : 0u;
    const uint32_t umod = (uint32_t)(st.base % J.cs);
    st.lead = umod ? J.cs - umod : 0u;
    st.next_chunk = (st.base + st.lead) / J.cs;
    return st;
}

// st.shared of v at address a where w1 != w0.
__device__ __forceinline__ void sts_if_ne(uint32_t w1, uint32_t w0, uint32_t a, uint32_t v)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %0, %1;\n@p st.shared.u32 [%2], %3;\n}" ::"r"(w1),
                 "r"(w0), "r"(a), "r"(v)
                 : "memory");
}

// The 32 codes of a lane as groups of at most G codes (16 symbols, where a
// chunk may start, end a group).
template <int G>
struct Groups {
    static constexpr int NH = (16 + G - 1) / G;  // groups per 16 symbols
    static constexpr int NG = 2 * NH;
    uint32_t acc[NG];  // marker and bits
    uint32_t len[NG];
    uint32_t bits, mid16;  // of all 32 symbols and of the first 16
};

// Gather the codes of the lane's first m symbols.  A group's first kFirst
// codes have at most 31 bits together, whatever they are; a multiply-add of
// a later one whose high word is not zero has overflowed (the result, which
// the caller then throws away, is nonzero).
// The lane's column lies at shared address tcol_s + kImm, tcol_s with zeros in
// its second byte.
template <int G, int kFirst, bool kAll, uint32_t kImm>
__device__ __forceinline__ uint32_t mad_gather(Groups<G> &q, const uint32_t (&w)[8], int m,
                                               uint32_t tcol_s)
{
    constexpr int NH = Groups<G>::NH, NG = Groups<G>::NG;
    uint32_t over = 0;
    q.bits = 0;
#pragma unroll
    for (int g = 0; g < NG; ++g) {
        const int k0 = (g / NH) * 16 + (g % NH) * G;
        uint32_t a = 1u;
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const int k = k0 + j;
            if ((g % NH) * G + j < 16 && (kAll || k < m)) {
                uint2 x;
                asm("ld.shared.v2.u32 {%0, %1}, [%2+%3];"
                    : "=r"(x.x), "=r"(x.y)
                    : "r"(__byte_perm(w[k >> 2], tcol_s, 0x7604u | (uint32_t)(k & 3) << 4)), "n"(kImm));
                if (j >= kFirst) {
                    const uint64_t t = (uint64_t)a * x.y + x.x;
                    over |= (uint32_t)(t >> 32);
                    a = (uint32_t)t;
                } else {
                    a = a * x.y + x.x;
                }
            }
        }
        q.acc[g] = a;
        q.len[g] = 31u - __clz(a);
        q.bits += q.len[g];
        if (g == NH - 1)
            q.mid16 = q.bits;
    }
    return over;
}

// Pack and write the gathered step at symbol sb.  kInner: the step lies inside
// the input, the unit's words fit the output and every lane has at least 32
// bits, so the step needs no bound checks and every complete word is written
// by one plain store: of the lane that completes it, with zeros for the bits
// that are not its own.  After a warp barrier each lane ORs its last partial
// word into the next lane's first word (the last lane stores it: no lane
// writes that word), and lane 0 ORs the carried bits into word 0.  Otherwise a
// lane may have no bits at all, and all words are ORed into a zeroed buffer.
template <int G, bool kInner>
__device__ __forceinline__ bool mad_pack(const Job &J, UnitState &st, uint64_t sb, int lane,
                                         const Groups<G> &q, uint32_t wob_s, uint32_t *wob)
{
    uint32_t pos, step_bits;
    scan_bits(q.bits, lane, pos, step_bits);
    const uint32_t p0 = (uint32_t)(st.gbit & 31) + pos;
    step_chunks<kStepSyms, kStep>(J, st, sb, lane, pos, q.mid16);
    if (!kInner) {
        sts_if(lane == 0, wob_s, st.carry);  // word 0 starts with the carried bits
        __syncwarp();
    }
    // lom + 1 holds the lane's last 32 bits.  A group of L bits x (a = 2^L + x)
    // that takes the lane's end from E to E1 over a word boundary completes
    // the word (lom + 1) << d | x >> r, with r = E1 mod 32 bits left over and
    // d = L - r = -E mod 32; the marker's 2^d is the 2^d that lom lacks.  A group that crosses no boundary stores nothing (about one group in two
    // crosses on text), which keeps the warp-buffer stores off the L1 data
    // pipe; a predicated store, because some lane of 32 nearly always
    // crosses.
    uint32_t lom = ~0u, E = p0, nE = 0u - p0, wi = p0 >> 5;
#pragma unroll
    for (int g = 0; g < Groups<G>::NG; ++g) {
        const uint32_t L = q.len[g];
        const uint32_t v0 = __funnelshift_l(0u, lom, nE);  // lom << (-E mod 32)
        E = imad(L, kc[kOne], E);
        nE -= L;
        const uint32_t v = v0 + __funnelshift_r(q.acc[g], 0u, E);
        const uint32_t w1 = E >> 5, ad = imad(w1, kc[kFour], wob_s - 4);
        if (kInner)
            sts_if_ne(w1, wi, ad, v);
        else if (w1 != wi)
            red_or(ad, v);
        wi = w1;
        lom = (lom << L) + q.acc[g] - 1u;
    }
    const uint32_t part = __funnelshift_lc(0u, lom + 1u, 32u - (E & 31u));
    if (kInner) {
        __syncwarp();
        const uint32_t pa = imad(E >> 5, kc[kFour], wob_s);
        if (lane == 31)
            sts(pa, part);
        else
            red_or(pa, part);
        if (lane == 0)
            red_or(wob_s, st.carry);
    } else {
        red_or(imad(E >> 5, kc[kFour], wob_s), part);
    }
    __syncwarp();
    const bool last = sb + kStep >= J.n;
    const bool overflow = step_output<!kInner>(J, st, last, step_bits, wob, lane);
    __syncwarp();
    step_advance<kStep>(J, st, step_bits);
    return overflow;
}

// Steps [step, full) of a unit without bound checks; returns the first step
// that cannot be done so (a group overflows, or a lane has fewer than 32 bits
// because of bytes without a code), or full.
template <int G, int kFirst, uint32_t kImm>
__device__ __forceinline__ int mad_steps(const Job &J, UnitState &st, int step, int full, int lane,
                                         uint32_t tcol_s, uint32_t wob_s, uint32_t *wob)
{
    const uint8_t *p = J.in + st.base + lane * kStepSyms;
    uint32_t w[8];
    load32(p + step * kStep, w);
    for (; step < full; ++step) {
        uint32_t nx[8];
        if (step + 1 < full)
            load32(p + (step + 1) * kStep, nx);  // one step ahead
        Groups<G> q;
        const uint32_t over = mad_gather<G, kFirst, true, kImm>(q, w, kStepSyms, tcol_s);
        if (!__all_sync(0xffffffffu, q.bits >= (uint32_t)kStepSyms && over == 0u))
            break;
        mad_pack<G, true>(J, st, st.base + (uint64_t)step * kStep, lane, q, wob_s, wob);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            w[j] = nx[j];
    }
    return step;
}

// The steps of a unit from `step` on in groups of S codes, which always fit:
// the whole ones, then the checked rest.
template <int S, uint32_t kImm>
__device__ __noinline__ bool mad_rest(const Job J, UnitState st, int step, int full, int lane,
                                      uint32_t tcol_s, uint32_t wob_s, uint32_t *wob)
{
    bool overflow = false;
    if (step < full)
        step = mad_steps<S, S, kImm>(J, st, step, full, lane, tcol_s, wob_s, wob);
    if (step < kSteps && st.base + (uint64_t)step * kStep < J.n) {
        clear_buffer(wob - 1, lane);
        for (; step < kSteps; ++step) {
            const uint64_t sb = st.base + (uint64_t)step * kStep;
            if (sb >= J.n)
                break;  // warp-uniform
            uint32_t w[8];
            const int m = step_input_tail<kStepSyms>(J, sb, lane, w);
            Groups<S> q;
            mad_gather<S, S, false, kImm>(q, w, m, tcol_s);
            overflow |= mad_pack<S, false>(J, st, sb, lane, q, wob_s, wob);
        }
    }
    return overflow;
}

// Encode unit u of job J with the calling warp in groups of G codes, of which
// kFirst always fit; the steps with a group that does not fit, and all after
// them, in groups of S.  tbl is the stream's half of the table, wob the warp's
// buffer of kWarpObuf words (word 0 is the guard).  Returns true if a payload
// word fell outside the output capacity.
template <int G, int kFirst, int S, uint32_t kImm>
__device__ __forceinline__ bool encode_unit_mad(const Job &J, uint64_t u, const uint32_t *tbl, uint32_t *wob)
{
    const int lane = threadIdx.x & 31;
    const uint32_t tcol_s = smem_u32(tbl + 2 * (lane & 15)) - kImm, wob_s = smem_u32(wob + 1);
    UnitState st = unit_start<true>(J, u, tbl, lane);
    const int full = full_steps(J, u);
    int step = 0;
    if (full)  // warp-uniform
        step = mad_steps<G, kFirst, kImm>(J, st, 0, full, lane, tcol_s, wob_s, wob + 1);
    if (step < kSteps && st.base + (uint64_t)step * kStep < J.n)
        return mad_rest<S, kImm>(J, st, step, full, lane, tcol_s, wob_s, wob + 1);
    return false;
}

// The same for 32-bit codes: 16 symbols per lane and a 64-bit accumulator
// (rare: only very skewed inputs have codes this long).
__device__ __forceinline__ bool encode_unit_long(const Job &J, uint64_t u, const uint32_t *tbl,
                                                 uint32_t *wob_all)
{
    const int lane = threadIdx.x & 31;
    clear_buffer(wob_all, lane);
    uint32_t *wob = wob_all + 1;
    bool overflow = false;
    UnitState st = unit_start<false>(J, u, tbl, lane);
    for (int step = 0; step < kLongSteps; ++step) {
        const uint64_t sb = st.base + (uint64_t)step * kLongStep;
        if (sb >= J.n)
            break;  // warp-uniform
        uint32_t w[4];
        const int m = step_input_tail<kLongSyms>(J, sb, lane, w);
        uint32_t e[kLongSyms], l2[kLongSyms];
        uint32_t bits = 0;
        const int col = lane & 15;
#pragma unroll
        for (int k = 0; k < kLongSyms; ++k) {
            const uint32_t b = byte_of(w, k);
            e[k] = k < m ? tbl[b * kTblRow + col] : 0u;
            l2[k] = k < m ? tbl[b * kTblRow + 16 + col] : 0u;
            bits += l2[k];
        }
        uint32_t pos, step_bits;
        scan_bits(bits, lane, pos, step_bits);
        const uint32_t r = (uint32_t)(st.gbit & 31);
        if (lane == 0)
            wob[0] = st.carry;  // word 0 starts with the carried bits
        __syncwarp();
        step_chunks<kLongSyms, kLongStep>(J, st, sb, lane, pos, 0u);
        if (m > 0) {
            uint32_t wi = (r + pos) >> 5, nb = (r + pos) & 31u;
            uint64_t acc = 0;
#pragma unroll
            for (int k = 0; k < kLongSyms; ++k) {
                const uint32_t L = l2[k];
                acc = L ? ((acc << L) | e[k]) : acc;
                nb += L;
                if (nb >= 32) {
                    nb -= 32;
                    atomicOr(wob + wi, (uint32_t)(acc >> nb));
                    ++wi;
                }
            }
            if (nb)
                atomicOr(wob + wi, (uint32_t)acc << (32 - nb));
        }
        __syncwarp();
        overflow |= step_output<true>(J, st, sb + kLongStep >= J.n, step_bits, wob, lane);
        __syncwarp();
        step_advance<kLongStep>(J, st, step_bits);
    }
    return overflow;
}

}  // namespace enc
}  // namespace huff
