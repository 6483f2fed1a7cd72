// Codebook device routine (one CTA of 256 threads per histogram), shared by
// the single-stream kernel (codebook.cu) and the batched kernel (batch.cu).
// See codebook.cu for the method.
#pragma once

#include "huff_internal.cuh"

namespace huff {
namespace cbk {

struct CodebookShared {
    unsigned long long w[256];
    alignas(16) unsigned long long key[256];   // weight * 256 + byte, all ones if absent
    unsigned long long pm[2][512];             // package-merge: the previous and current list
    uint16_t pos[kMaxCodeLen + 1][256];        // package-merge: position of each leaf per list
    int pm_take[kMaxCodeLen + 1];              // package-merge: leaves taken from each list
    unsigned long long nw[511];  // [0,m): leaves by (weight, byte); [m,2m-1): merged
    int16_t par[511];
    int16_t dep[511];
    int16_t anc[511];
    uint8_t leaf_sym[256];
    uint8_t len_s[256];
    uint32_t bl[kMaxCodeLen + 1];
    uint32_t next_code[kMaxCodeLen + 1];
    int s_max;
    int q[3];  // the queues' heads and the next node, from a single thread's steps
};

// Code lengths of at most `limit` bits for the m leaves nw[0..m) (sorted by
// (weight, byte)), by package-merge (Larmore & Hirschberg 1990): list 1 =
// the leaves; list i = the leaves merged with the packages (sums of
// consecutive pairs) of list i-1, a leaf before a package of equal weight;
// the first 2m-2 items of list `limit` are taken and each taken package takes
// its two items of the list below.  A leaf's length is the number of lists
// it is taken from, and the leaves taken from a list are a prefix of the
// sorted leaves.  Every merge position is a binary search (one item per
// thread); 2 <= m <= 2^limit.
__device__ __forceinline__ void package_merge(int m, int limit, CodebookShared &sh)
{
    const int t = threadIdx.x;
    int cnt = m;  // items in the previous list
    if (t < m) {
        sh.pm[0][t] = sh.nw[t];
        sh.pos[1][t] = (uint16_t)t;
    }
    __syncthreads();
    for (int i = 2; i <= limit; ++i) {
        const unsigned long long *prev = sh.pm[(i - 2) & 1];
        unsigned long long *cur = sh.pm[(i - 1) & 1];
        const int np = cnt >> 1;
        if (t < m) {  // leaf t goes after the packages lighter than it
            const unsigned long long w = sh.nw[t];
            int lo = 0, hi = np;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (prev[2 * mid] + prev[2 * mid + 1] < w)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            cur[t + lo] = w;
            sh.pos[i][t] = (uint16_t)(t + lo);
        }
        if (t < np) {  // package t goes after the leaves not heavier than it
            const unsigned long long w = prev[2 * t] + prev[2 * t + 1];
            int lo = 0, hi = m;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (sh.nw[mid] <= w)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            cur[t + lo] = w;
        }
        cnt = m + np;
        __syncthreads();
    }
    if (t == 0) {  // walk down from the last list
        int take = 2 * m - 2;
        for (int i = limit; i >= 1; --i) {
            int lo = 0, hi = m;  // leaves among the first `take` items
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((int)sh.pos[i][mid] < take)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            sh.pm_take[i] = lo;
            take = 2 * (take - lo);
        }
    }
    __syncthreads();
    if (t < m) {
        int d = 0;
        for (int i = 1; i <= limit; ++i)
            d += t < sh.pm_take[i];
        sh.dep[t] = (int16_t)d;
    }
}

// Build *cb from hist (u64[256]); blockDim.x must be 256.  Huffman codes
// longer than `limit` (1..32) bits: without `limited` that is an error (*cb
// cleared, HUFF_ERR_CODE_TOO_LONG); with it the lengths are recomputed by
// package-merge (the error only if the bytes present exceed 2^limit).
__device__ __forceinline__ void build_codebook(const unsigned long long *hist, huff_codebook_t *cb,
                                               int32_t *status, CodebookShared &sh,
                                               int limit = (int)kMaxCodeLen, bool limited = false)
{
    if (chain_failed(status))
        return;
    const int t = threadIdx.x;
    const unsigned long long wt = hist[t];
    // (weight, byte) as one key where every weight is below 2^56 (any byte
    // count is)
    const unsigned long long kt = wt ? (wt << 8) | (unsigned long long)t : ~0ull;
    sh.w[t] = wt;
    sh.key[t] = kt;
    sh.len_s[t] = 0;
    if (t <= (int)kMaxCodeLen)
        sh.bl[t] = 0;
    if (t == 0)
        sh.s_max = 0;
    const int present = wt > 0;
    const int m = __syncthreads_count(present);
    const bool huge = __syncthreads_or((wt >> 56) != 0);  // weights the key cannot hold

    // 1. rank of byte t among present bytes, ordered by (weight, byte): the
    //    keys below its own (an absent byte's key is above every other)
    if (present) {
        int rank = 0;
        if (!huge) {
#pragma unroll 8
            for (int j = 0; j < 128; ++j) {
                const ulonglong2 k2 = reinterpret_cast<const ulonglong2 *>(sh.key)[j];
                rank += (k2.x < kt) + (k2.y < kt);
            }
        } else {
            for (int j = 0; j < 256; ++j) {
                const unsigned long long wj = sh.w[j];
                rank += (wj > 0) & ((wj < wt) | ((wj == wt) & (j < t)));
            }
        }
        sh.leaf_sym[rank] = (uint8_t)t;
        sh.nw[rank] = wt;
    }
    __syncthreads();

    if (m >= 2) {
        // 2. two-queue merge, in rounds: every node not heavier than the sum
        // T of the two lightest comes before the first new node (whose weight
        // is T and whose id is larger), so all of them are taken in pairs at
        // once, in (weight, id) order; one left over stays.  Rounds of fewer
        // than six pairs (weights that grow like powers of two) give way to 32
        // steps of one thread, a pair each; up to 64 byte values, and weights
        // that a sum could overflow, take no rounds at all.  The codebook of
        // 256 equally frequent bytes takes 7.2 us in rounds and 22 us step by
        // step, that of text (34 values) 8.3 and 6.5 us.
        constexpr unsigned long long kNone = ~0ull;
        uint16_t *const seq = sh.pos[0];  // 512 places
        const bool rounds = m > 64 && !huge;
        int li = 0, ii = m, ni = m;
        while (ni < 2 * m - 1) {  // (the same in every thread)
            int leaves = 0, merged = 0;
            bool leaf_in = false, merged_in = false;
            if (rounds) {
                const unsigned long long a0 = li < m ? sh.nw[li] : kNone;
                const unsigned long long a1 = li + 1 < m ? sh.nw[li + 1] : kNone;
                const unsigned long long b0 = ii < ni ? sh.nw[ii] : kNone;
                const unsigned long long b1 = ii + 1 < ni ? sh.nw[ii + 1] : kNone;
                const unsigned long long T = a0 <= b0 ? a0 + (a1 <= b0 ? a1 : b0) : b0 + (a0 <= b1 ? a0 : b1);
                leaf_in = li + t < m && sh.nw[li + t] <= T;
                merged_in = ii + t < ni && sh.nw[ii + t] <= T;
                leaves = __syncthreads_count(leaf_in);
                merged = __syncthreads_count(merged_in);
            }
            const int pairs = (leaves + merged) >> 1;
            if (pairs >= 6) {
                if (leaf_in) {  // after the merged nodes lighter than it
                    const unsigned long long w = sh.nw[li + t];
                    int lo = 0, hi = merged;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (sh.nw[ii + mid] < w)
                            lo = mid + 1;
                        else
                            hi = mid;
                    }
                    seq[t + lo] = (uint16_t)(li + t);
                }
                if (merged_in) {  // after the leaves not heavier than it
                    const unsigned long long w = sh.nw[ii + t];
                    int lo = 0, hi = leaves;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (sh.nw[li + mid] <= w)
                            lo = mid + 1;
                        else
                            hi = mid;
                    }
                    seq[t + lo] = (uint16_t)(ii + t);
                }
                __syncthreads();
                if (t < pairs) {
                    const int a = seq[2 * t], b = seq[2 * t + 1];
                    sh.nw[ni + t] = sh.nw[a] + sh.nw[b];
                    sh.par[a] = sh.par[b] = (int16_t)(ni + t);
                }
                if ((leaves + merged) & 1) {
                    if (seq[leaves + merged - 1] < m)
                        --leaves;
                    else
                        --merged;
                }
                li += leaves;
                ii += merged;
                ni += pairs;
                __syncthreads();
                continue;
            }
            const int left = 2 * m - 1 - ni, steps = rounds && left > 32 ? 32 : left;
            if (t == 0) {
                // the first two entries of each queue are kept in registers (all
                // ones past a queue's end), so that a take never waits for a
                // shared load: a leaf's weight is loaded two takes before it can
                // be needed, and a merged node's weight usually never is.  A tie
                // takes the leaf (the smaller id).
                unsigned long long l0 = li < m ? sh.nw[li] : kNone, l1 = li + 1 < m ? sh.nw[li + 1] : kNone;
                unsigned long long i0 = ii < ni ? sh.nw[ii] : kNone, i1 = ii + 1 < ni ? sh.nw[ii + 1] : kNone;
                for (int step = 0; step < steps; ++step) {
                    int ab[2];
                    unsigned long long wab[2];
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        // branch free: both refills are loaded (at in-range
                        // indices) and the take selects
                        const bool lf = l0 <= i0;
                        const unsigned long long nl = sh.nw[li + 2 < 510 ? li + 2 : 510];
                        const unsigned long long nq = sh.nw[ii + 2 < 510 ? ii + 2 : 510];
                        ab[k] = lf ? li : ii;
                        wab[k] = lf ? l0 : i0;
                        const unsigned long long l1n = li + 2 < m ? nl : kNone;
                        const unsigned long long i1n = ii + 2 < ni ? nq : kNone;
                        l0 = lf ? l1 : l0;
                        l1 = lf ? l1n : l1;
                        i0 = lf ? i0 : i1;
                        i1 = lf ? i1 : i1n;
                        li += lf;
                        ii += !lf;
                    }
                    const unsigned long long w2 = wab[0] + wab[1];
                    sh.nw[ni] = w2;
                    sh.par[ab[0]] = (int16_t)ni;
                    sh.par[ab[1]] = (int16_t)ni;
                    // the new node joins the merged queue at ni
                    i0 = ii == ni ? w2 : i0;
                    i1 = ii + 1 == ni ? w2 : i1;
                    ++ni;
                }
                sh.q[0] = li;
                sh.q[1] = ii;
                sh.q[2] = ni;
            }
            __syncthreads();
            li = sh.q[0];
            ii = sh.q[1];
            ni = sh.q[2];
        }
        if (t == 0)
            sh.par[2 * m - 2] = (int16_t)(2 * m - 2);  // the root points at itself
        __syncthreads();
        // 3. depth = distance to the root, by pointer jumping (9 rounds cover
        //    511 nodes; done early once every ancestor is the root)
        const int nn = 2 * m - 1, root = 2 * m - 2;
        for (int k = t; k < nn; k += 256) {
            sh.dep[k] = (k == root) ? 0 : 1;
            sh.anc[k] = sh.par[k];
        }
        __syncthreads();
        for (int round = 0; round < 9; ++round) {
            int16_t nd[2], na[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int k = t + j * 256;
                if (k < nn) {
                    nd[j] = (int16_t)(sh.dep[k] + sh.dep[sh.anc[k]]);
                    na[j] = sh.anc[sh.anc[k]];
                }
            }
            __syncthreads();
            bool at_root = true;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int k = t + j * 256;
                if (k < nn) {
                    sh.dep[k] = nd[j];
                    sh.anc[k] = na[j];
                    at_root &= na[j] == root;
                }
            }
            if (__syncthreads_and(at_root))
                break;
        }
        // the Huffman lengths, unless a limit below 32 is exceeded
        if (t < m)
            atomicMax(&sh.s_max, (int)sh.dep[t]);
        __syncthreads();
        if (limited && sh.s_max > limit && (limit >= 9 || m <= (1 << limit))) {
            __syncthreads();
            if (t == 0)
                sh.s_max = 0;
            package_merge(m, limit, sh);
            if (t < m)
                atomicMax(&sh.s_max, (int)sh.dep[t]);
        }
        if (t < m) {
            const int d = sh.dep[t];
            sh.len_s[sh.leaf_sym[t]] = (uint8_t)(d > 255 ? 255 : d);
        }
    } else if (m == 1 && present) {
        sh.len_s[t] = 1;  // one distinct byte: the 1-bit code "0"
        sh.s_max = 1;
    }
    __syncthreads();

    // 4. length limit, then canonical codes
    const int max_len = sh.s_max;
    if (max_len > limit) {
        set_status(status, HUFF_ERR_CODE_TOO_LONG);
        cb->len[t] = 0;
        cb->code[t] = 0;
        if (t == 0) {
            cb->nsym = 0;
            cb->max_len = 0;
        }
        return;
    }
    const int L = sh.len_s[t];
    if (L)
        atomicAdd(&sh.bl[L], 1u);
    __syncthreads();
    // next_code[b] = (next_code[b - 1] + bl[b - 1]) << 1, that is the sum of
    // bl[k] << (b - k) over the shorter lengths k, a length per thread; and the
    // bytes of each length per warp
    if (t >= 1 && t <= (int)kMaxCodeLen) {
        uint32_t code = 0;
        for (int k = 1; k < t; ++k)
            code = (code + sh.bl[k]) << 1;
        sh.next_code[t] = code;
    }
    const int lane = t & 31, warp = t >> 5;
    const uint32_t same = __match_any_sync(0xffffffffu, L);
    uint16_t *const of_len = sh.pos[0];  // [warp][length]
    if (t < 8 * (int)(kMaxCodeLen + 1))
        of_len[t] = 0;
    if (t + 256 < 8 * (int)(kMaxCodeLen + 1))
        of_len[t + 256] = 0;
    __syncthreads();
    if (lane == __ffs(same) - 1)
        of_len[warp * (kMaxCodeLen + 1) + L] = (uint16_t)__popc(same);
    __syncthreads();
    uint32_t code = 0;
    if (L) {
        uint32_t r = __popc(same & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w)
            r += of_len[w * (kMaxCodeLen + 1) + L];
        code = sh.next_code[L] + r;
    }
    cb->len[t] = (uint8_t)L;
    cb->code[t] = code;
    if (t == 0) {
        cb->nsym = (uint32_t)m;
        cb->max_len = (uint32_t)max_len;
    }
}

}  // namespace cbk
}  // namespace huff
