// Batched engine internals shared by batch.cu (kernels, plans) and
// server.cu (served rounds).
#pragma once

#include <vector>

#include "huff_internal.cuh"

namespace huff {

constexpr int kBatchBlock = 256;
constexpr int kBatchWarps = kBatchBlock / 32;
// The encode and decode phases run each half of a CTA on its own items
// (its own code or lookup table), so that small buffers leave fewer warps
// idle than with items of the whole CTA.
constexpr int kHalf = kBatchBlock / 2;
constexpr int kHalfWarps = kBatchWarps / 2;
constexpr int kUnitsPerItem = kHalfWarps;  // encode: one unit per warp of a half
constexpr int kTasksPerItem = kHalfWarps;  // decode: one task per warp of a half

// control words (device): barrier arrivals and generation, then three tickets
// and the lanes a buffer's decoding is spread over
enum { kCtlArrive = 0, kCtlGen = 1, kCtlTicket0 = 2, kCtlLanes = 5, kCtlWords = 8 };

struct BatchBuf {
    const uint8_t *in;
    uint64_t in_bytes;
    uint8_t *out;
    uint64_t out_cap;
    unsigned long long *out_bytes;
    int32_t *status;
};

struct BatchArgs {
    const BatchBuf *bufs;
    uint32_t count;
    uint32_t cs;                    // compress: chunk symbols
    const uint64_t *unit_base;      // compress: [count + 1] prefix of units
    const uint64_t *item_base;      // compress: [count + 1] prefix of encode items
    uint16_t *unit_hist;            // compress: [units][256]
    unsigned long long *unit_off;   // compress: per buffer units_b + 1 entries at unit_base[b] + b
    huff_codebook_t *cbs;           // compress: [count]
    uint4 *unit_owner;              // compress: [units] (its first input byte, low and high
                                    //   words; its bytes; its buffer), set in phase 0
    uint4 *item_owner;              // compress: [items] (buffer, item within it, its first
                                    //   unit's index in unit_base order, low and high words)
    uint64_t *dec_items;            // decompress: [count + 1] items, then their prefix
    uint32_t min_lanes;             // decompress: lanes per buffer to aim for,
    uint32_t own_lanes;             //   whatever the batch's size (the caller's own number)
    unsigned int *ctl;              // kCtlWords
    int32_t *fail;                  // whole-batch failure (barrier timeout)
    uint32_t barrier_extra;         // test hook: CTAs the barriers wait for beyond the grid
};

// Host-side description of a batch's device block (see batch_layout).
struct BatchLayout {
    uint32_t count;
    huff_op_t op;
    std::vector<BatchBuf> bufs;
    std::vector<uint64_t> unit_base, item_base;
    uint64_t o_ctl, o_bufs, o_ub, o_ib, o_di, o_uh, o_uo, o_cb, o_uw, o_iw;
    uint64_t bytes;         // device block size
    uint64_t upload_bytes;  // leading part filled from the host
};

// even: buffers of one size but for the last, kept in their order.
void batch_layout(const huff_batch_desc_t *descs, uint32_t count, huff_op_t op, BatchLayout &L,
                  bool even = false);
BatchArgs batch_args(const BatchLayout &L, void *d_block, uint32_t cs, uint32_t lanes, bool own_lanes,
                     uint32_t barrier_extra = 0);
cudaError_t batch_upload(const BatchLayout &L, void *d_block, uint8_t *host, cudaStream_t s);
int batch_occupancy(huff_op_t op);
inline huff_status_t batch_occupancy_error(int per_sm)
{
    return per_sm < 0 ? HUFF_ERR_UNSUPPORTED : HUFF_ERR_CUDA;
}
cudaError_t batch_launch(huff_op_t op, const BatchArgs &args, unsigned grid, cudaStream_t s);
// Run an even batch once, its lanes not a caller's own: with its device block in
// `scratch` (16-byte aligned) where it fits, else by a plan, which the caller
// destroys once the stream has passed it.  `host` is read by the upload until
// then too.
huff_status_t batch_once(const huff_batch_desc_t *descs, uint32_t count, huff_op_t op,
                         const huff_batch_params_t &prm, void *scratch, uint64_t scratch_bytes,
                         std::vector<uint8_t> &host, cudaStream_t s, huff_batch_plan_t **plan);
huff_status_t batch_check(const huff_batch_desc_t *descs, uint32_t count, huff_op_t op,
                          const huff_batch_params_t &prm);

// huff_segmented_compress / huff_segmented_decompress for a caller with device
// memory to spare: the batch's block (and decompression's per-segment words)
// go into scratch[0, scratch_bytes) where they fit, so that nothing is
// allocated.
huff_status_t segmented_compress(const uint8_t *d_in, uint64_t n, uint64_t segment_bytes,
                                 uint32_t chunk_symbols, uint8_t *d_out, uint64_t out_cap,
                                 uint64_t *d_out_bytes, void *d_ws, uint64_t ws_bytes,
                                 int32_t *d_status, cudaStream_t s, void *scratch,
                                 uint64_t scratch_bytes);
huff_status_t segmented_decompress(const uint8_t *d_in, uint64_t in_bytes, uint8_t *d_out,
                                   uint64_t out_cap, uint64_t *d_n, int32_t *d_status,
                                   cudaStream_t s, void *scratch, uint64_t scratch_bytes);

}  // namespace huff
