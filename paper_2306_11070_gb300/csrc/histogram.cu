// Byte histogram: the "probability of occurrence" step of the paper's
// Huffman Method 1 (Section III-A).
//
// HBM-bound: n bytes read once.  Each CTA keeps 32 private copies of the 256
// counters in shared memory, laid out [bin][lane], and lane l only touches
// column l, so the 32 shared-memory atomics of one warp instruction always
// fall in 32 different banks, whatever the data (a single repeated byte
// included).  Persistent CTAs take 16 KiB units round robin; each thread
// loads its four 16-byte pieces of the next unit before counting the current
// one.
//
// Optionally the kernel also writes every unit's own histogram (u16[256],
// 512 bytes per 16 KiB): the encoder turns these into the bit offset of each
// unit with a dot product against the code lengths, so it never has to wait
// on another CTA.  The shared-memory pipe bounds it (86% busy): 512 wavefronts
// count a unit, 256 fold its columns.  So two units share a fold: the first
// counts in the low, the second in the high half of the columns.  Folds are sums
// modulo 2^32 of columns that are never cleared, and their difference is the
// first unit's count plus 2^16 times the second's, both at most 16384.
// A compress call
// of 1 GiB takes 773 us instead of 786.
#include "hist_impl.cuh"

namespace huff {
namespace {

using namespace hst;

constexpr int kHistBlock = kThreads;

// Clears the totals (and the chain's status).  A kernel instead of memory sets,
// because the histogram can be launched behind it.
__global__ void __launch_bounds__(256) k_clear(unsigned long long *hist, int32_t *status)
{
    chain_next();
    hist[threadIdx.x] = 0;
    if (status && threadIdx.x == 0)
        *status = 0;
}

__global__ void __launch_bounds__(kHistBlock)
    k_histogram(const uint8_t *in, uint64_t n, unsigned long long *hist, uint16_t *unit_hist)
{
    __shared__ __align__(16) uint32_t cnt[256 * 32];
    chain_next();
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < 256 * 32; i += kHistBlock)
        cnt[i] = 0;
    chain_wait();
    const uint32_t col = smem_u32(cnt) + 4u * lane;  // this lane's column
    const uint64_t units = (n + kUnitSymbols - 1) / kUnitSymbols;
    uint32_t prev = 0, total = 0;  // this thread's bin: last fold, count so far
    const uint32_t one2 = unit_hist ? 1u << 16 : 1u;
    uint4 a[kVecPerThread];
    const uint64_t G = gridDim.x;
    uint64_t u = blockIdx.x;
    load_unit(in, n, u, a);
    __syncthreads();
    for (; u < units; u += 2 * G) {
        uint4 cur[kVecPerThread];
#pragma unroll
        for (int j = 0; j < kVecPerThread; ++j)
            cur[j] = a[j];
        load_unit(in, n, u + G, a);  // in flight while this unit is counted
        count_unit(in, n, u, cur, col, 1u);
        if (u + G < units) {
#pragma unroll
            for (int j = 0; j < kVecPerThread; ++j)
                cur[j] = a[j];
            load_unit(in, n, u + 2 * G, a);
            count_unit(in, n, u + G, cur, col, one2);
        }
        if (unit_hist) {
            __syncthreads();  // all counts of both units are in
            const uint32_t s = fold_bin(cnt, tid), d = s - prev;
            prev = s;
            unit_hist[u * 256 + tid] = (uint16_t)d;
            if (u + G < units)
                unit_hist[(u + G) * 256 + tid] = (uint16_t)(d >> 16);
            total += (d & 0xffffu) + (d >> 16);
            __syncthreads();  // folds read before the next unit's counts
        }
    }
    __syncthreads();
    if (!unit_hist)
        total = fold_bin(cnt, tid);
    if (total)
        atomicAdd(hist + tid, (unsigned long long)total);
}

}  // namespace

cudaError_t launch_histogram(const uint8_t *d_in, uint64_t n, unsigned long long *d_hist,
                             uint16_t *d_unit_hist, cudaStream_t s, int32_t *d_status)
{
    k_clear<<<1, 256, 0, s>>>(d_hist, d_status);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess || n == 0)
        return err;
    static KernelSetup setup;
    int per_sm = 0;
    err = kernel_setup(setup, (const void *)k_histogram, kHistBlock, 0, &per_sm);
    if (err != cudaSuccess)
        return err;
    const int sms = device_sm_count();
    if (sms < 1)
        return cudaErrorInvalidDevice;
    const uint64_t units = (n + kUnitSymbols - 1) / kUnitSymbols;
    const uint64_t cap = (uint64_t)sms * per_sm;
    const uint64_t grid = units < cap ? units : cap;
    return launch_chained(k_histogram, grid, kHistBlock, 0, s, d_in, n, d_hist, d_unit_hist);
}

}  // namespace huff
