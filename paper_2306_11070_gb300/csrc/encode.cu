// Encoder: the coding step of the paper's Huffman Method 1 (Section III-A)
// over Method 2's segments, which become chunks of `cs` symbols with stored
// bit offsets.
//
// Design (one pass over the input, n bytes read + payload written):
//  - The bit offset of every 16 KiB unit is known before this kernel starts
//    (offsets.cu: unit histograms or unit counts, then a scan), so no warp
//    ever waits on another.  Each warp encodes whole units by itself in 16
//    steps of 1024 symbols; the loop has no CTA barrier at all.
//  - A step: every lane loads its 32 bytes (two 16-byte loads, issued one
//    step ahead), gathers their codes into groups by multiply-add from a
//    table in shared memory that is replicated per lane, so that the 32
//    lookups of a warp never collide in a bank (see encode_impl.cuh), a warp
//    scan of the lanes' bit counts gives every lane its bit position, the
//    lanes pack their groups into the warp's word buffer in shared memory,
//    and the warp writes the whole words with coalesced stores.  The partial
//    last word is carried in a register into the next step.
//  - What bounds it: on text the shared-memory data pipe is 66% busy while a
//    unit runs (two wavefronts per 32 lookups, about 1.5 for the packed
//    words) and 57% of the issue slots are taken (64 MiB).
//  - The word a unit shares with the unit before it is completed by the later
//    unit: it re-codes the last <= 31 bits of its predecessor from the 32
//    input bytes before it, so no warp waits for another's output and the
//    payload needs no clearing pass.
#include "encode_impl.cuh"

namespace huff {
namespace {

using namespace enc;

// One CTA of 16 warps per SM: one copy of the 64 KiB code table per SM, and
// 16 warps are what fit without spills (18 or 20 warps of 96 registers: 1 GiB
// takes 1070 and 1030 us instead of 839).
constexpr int kEncBlock = 512;
constexpr int kEncWarps = kEncBlock / 32;
// the table, the padding before it, and the buffers if the gap is too small
constexpr int kEncObufBytes = kEncWarps * kWarpObuf * 4;
constexpr int kEncSmemBytes = 65536 + kTblWords * 4 + kEncObufBytes;

struct EncodeArgs {
    const uint8_t *in;
    uint64_t n;
    const huff_codebook_t *cb;
    const unsigned long long *unit_off;
    uint32_t cs;
    uint8_t *out;
    uint64_t out_cap;
    unsigned long long *out_bytes;
    int32_t *status;
};

// This warp's part of the CTA's dynamic shared memory, and the code table, which
// lies at a 64 KiB boundary of the shared window, so that the address of a
// byte's entry is one byte permutation of the data word and the lane's column
// (a multiply-add per symbol fewer); the warps' buffers take the gap before
// it.
struct Smem {
    uint32_t *tbl, *wob;
};

__device__ __forceinline__ Smem carve(uint4 *smem_raw)
{
    const uint32_t pad = (0u - smem_u32(smem_raw)) & 0xffffu;
    unsigned char *raw = reinterpret_cast<unsigned char *>(smem_raw);
    Smem m;
    m.tbl = reinterpret_cast<uint32_t *>(raw + pad);
    m.wob = reinterpret_cast<uint32_t *>(raw + (pad >= (uint32_t)kEncObufBytes ? 0u : pad + kTblWords * 4)) +
            (threadIdx.x >> 5) * kWarpObuf;
    return m;
}

// Units go to the CTAs first and to their warps second: a last wave that does
// not fill the chip leaves every SM with a few busy warps instead of some SMs
// with none, and a few units get an SM each (1 MiB: the call takes 62 us
// instead of 77).
#define FOR_UNITS(u, J)                                                                      \
    for (uint64_t u = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; u < (J).units; \
         u += (uint64_t)gridDim.x * kEncWarps)

// Codes of 11 to 31 bits, in groups of G that nearly always fit, else of S.
template <int G, int S>
__device__ __noinline__ void encode_try(const EncodeArgs &a)
{
    extern __shared__ uint4 smem_raw[];
    const Smem m = carve(smem_raw);
    const Job J = make_job(a.in, a.n, a.cs, a.unit_off, a.out, a.out_cap);
    bool overflow = false;
    FOR_UNITS(u, J)
        overflow |= encode_unit_mad<G, S, S, 0>(J, u, m.tbl, m.wob);
    if (overflow)
        set_status(a.status, HUFF_ERR_CAPACITY);
}

__device__ __noinline__ void encode_long(const EncodeArgs &a)
{
    extern __shared__ uint4 smem_raw[];
    const Smem m = carve(smem_raw);
    const Job J = make_job(a.in, a.n, a.cs, a.unit_off, a.out, a.out_cap);
    bool overflow = false;
    FOR_UNITS(u, J)
        overflow |= encode_unit_long(J, u, m.tbl, m.wob);
    if (overflow)
        set_status(a.status, HUFF_ERR_CAPACITY);
}

// A function, called once per unit, and the rarer plans in functions of their
// own: inlined into the kernel, all or each by itself, they spill or are
// scheduled worse (1 GiB of text: the call takes 810 to 1010 us instead of
// 795).
__device__ __noinline__ bool encode_unit_fit(const Job J, uint64_t u, const uint32_t *tbl, int plan,
                                                uint32_t *wob)
{
    switch (plan) {
    case kFit16: return encode_unit_mad<16, 16, 16, 0>(J, u, tbl, wob);
    case kFit8: return encode_unit_mad<8, 8, 8, 0>(J, u, tbl, wob);
    case kFit4: return encode_unit_mad<4, 4, 4, 0>(J, u, tbl, wob);
    default: return encode_unit_mad<3, 3, 3, 0>(J, u, tbl, wob);
    }
}

// One kernel for all code lengths: the host does not know them, and a second
// launch that only finds out that it does not apply costs 2 us or more.
__global__ void __launch_bounds__(kEncBlock, 1) k_encode(const __grid_constant__ EncodeArgs a)
{
    extern __shared__ uint4 smem_raw[];
    chain_wait();
    if (chain_failed(a.status))
        return;
    const Smem m = carve(smem_raw);
    const uint32_t max_len = a.cb->max_len;
    build_table(a.cb, m.tbl, max_len <= kMadMaxLen, threadIdx.x, kEncBlock);
    const Job J = make_job(a.in, a.n, a.cs, a.unit_off, a.out, a.out_cap);
    if (blockIdx.x == 0)
        write_header(J, a.cb, a.out_bytes, a.status);
    __syncthreads();  // the only CTA barrier: the table is ready
    bool overflow = false;
    const int plan = plan_of(J, max_len);
    if (plan < kFit3) {
        switch (plan) {
        case kPairs4: encode_try<4, 2>(a); break;
        case kPairs3: encode_try<3, 2>(a); break;
        case kTry4: encode_try<4, 1>(a); break;
        case kTry3: encode_try<3, 1>(a); break;
        default: encode_long(a);
        }
        return;
    }
    FOR_UNITS(u, J)
        overflow |= encode_unit_fit(J, u, m.tbl, plan, m.wob);
    if (overflow)
        set_status(a.status, HUFF_ERR_CAPACITY);
}

}  // namespace

uint64_t encode_workspace_bytes(uint64_t n)
{
    // unit bit counts (u32), unit offsets (u64, + total), the scan's tile sums
    const uint64_t units = (n + kUnitSymbols - 1) / kUnitSymbols;
    return ((4 * units + 255) & ~255ull) + ((8 * (units + 1) + 255) & ~255ull) +
           8 * unit_scan_tiles(units);
}

cudaError_t launch_encode(const uint8_t *d_in, uint64_t n, const huff_codebook_t *d_cb, uint32_t cs,
                          uint8_t *d_out, uint64_t out_cap, unsigned long long *d_out_bytes,
                          void *d_ws, const uint16_t *d_unit_hist, int32_t *d_status,
                          cudaStream_t s)
{
    static KernelSetup setup;
    int per_sm = 0;
    cudaError_t err = kernel_setup(setup, (const void *)k_encode, kEncBlock, kEncSmemBytes, &per_sm);
    if (err != cudaSuccess)
        return err;
    const int sms = device_sm_count();
    if (sms < 1)
        return cudaErrorInvalidDevice;
    const uint64_t units = (n + kUnitSymbols - 1) / kUnitSymbols;
    uint8_t *ws = static_cast<uint8_t *>(d_ws);
    uint32_t *unit_bits = reinterpret_cast<uint32_t *>(ws);
    unsigned long long *unit_off =
        reinterpret_cast<unsigned long long *>(ws + ((4 * units + 255) & ~255ull));
    unsigned long long *tile_sum = reinterpret_cast<unsigned long long *>(
        ws + ((4 * units + 255) & ~255ull) + ((8 * (units + 1) + 255) & ~255ull));
    err = launch_unit_offsets(d_in, n, d_unit_hist, d_cb, unit_bits, unit_off, tile_sum, d_status,
                              s);
    if (err != cudaSuccess)
        return err;
    EncodeArgs a;
    a.in = d_in;
    a.n = n;
    a.cb = d_cb;
    a.unit_off = unit_off;
    a.cs = cs;
    a.out = d_out;
    a.out_cap = out_cap;
    a.out_bytes = d_out_bytes;
    a.status = d_status;
    uint64_t grid = (uint64_t)sms * per_sm;
    if (grid > units)
        grid = units;
    if (grid < 1)
        grid = 1;
    return launch_chained(k_encode, grid, kEncBlock, kEncSmemBytes, s, a);
}

}  // namespace huff
