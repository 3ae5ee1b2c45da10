// Types and launchers of the block codec and the block pool (device side).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "qsim_internal.h"

namespace qsim {

// a compressed block to read
struct BlockRef {
    const uint8_t *ptr;
    uint64_t bytes;
};

// one entry of the block table (where block b's current stream lives)
struct BlockSlot {
    uint8_t *ptr;
    uint64_t bytes;
    uint32_t tier;  // 0 device, 1 pinned host
    uint32_t pad;
};

// where an encoder writes block j of a group
struct EncTarget {
    uint8_t *ptr;
    uint64_t cap;
    uint32_t tier;
    uint32_t pad;
};

struct EncResult {
    uint64_t total;      // stream bytes (also computed when the slot overflowed)
    uint32_t overflow;   // 1 if the stream did not fit the reserved slot
    uint32_t pad;
    double err_sq;       // sum (x - x')^2 over the block
    double norm_sq;      // sum x'^2 over the block
};

// per-stage running totals, updated by the encoder
struct StageAccum {
    uint64_t store_bytes;
    uint64_t reserved_bytes;
    uint64_t host_bytes;
    uint64_t blocks;
    uint64_t overflow_blocks;
    uint64_t pad;
    double err_sq;
    double norm_sq;
};

// a bump arena (device memory, or mapped pinned host memory)
struct ArenaDev {
    uint8_t *base;
    uint64_t cap;
    uint64_t *bump;  // device counter
};

// look-back scratch of the single-block encoder
struct LookbackScratch {
    uint64_t *state;    // one status word per frame
    uint32_t *ticket;   // left zero
    uint32_t *epoch;    // tags the status words; advanced by every launch
};

void count_launch();

// What a single-block call tells the host: written by the launch itself, to mapped pinned memory where the call may
// hold some, so that the call needs one launch and one synchronisation and no copy.
struct CallHost {
    uint64_t bytes;   // compressed size
    int32_t status;   // QSIM_OK or the first error
    uint32_t pad;
};
struct CallResult {
    int *status;       // device status word of the launch, left zero
    uint32_t *done;    // device counter, left zero
    CallHost *record;  // device address of the record
};

// Blocks b0 .. b0 + nblocks - 1 of a table decoded back to back. rel: the streams are QSZR (relative bound)
void launch_decode(const BlockSlot *table, uint64_t b0, uint32_t nblocks, int m, float2 *wv, int *status,
                   cudaStream_t s, bool rel = false);
// One block given by pointer, QSZ1 or QSZR by its magic number
void launch_decode_block(const BlockRef &in, int m, float2 *out, const CallResult &res, cudaStream_t s);
// Per-frame records of the encoder, in work-item order (blocks of more than one frame)
struct FrameRecords {
    uint8_t *side;        // image bytes before the bit-plane words (at most side_bytes)
    uint32_t side_bytes;  // 256, or kQszrSideBytes for the relative-bound codec
    uint32_t *len, *off;  // stream bytes, offset in the block's stream
    uint32_t *head;       // relative-bound codec: bytes in `side`
    float2 *part;         // (sum (x - x')^2, sum x'^2)
};
// Encode a batch of blocks with exact slots (see k_encode); wv is overwritten. Blocks of more than one frame need
// launch_frame_copy after it. arrive: one zero word per block, left zero. rel: QSZR (e is the shift k).
void launch_encode(float2 *wv, uint32_t nblocks, int m, int e, const ArenaDev &dev, const ArenaDev &host,
                   EncTarget *tgt, EncResult *res, const uint32_t *ids, BlockSlot *table, StageAccum *acc,
                   const FrameRecords &fr, uint64_t *arrive, int *status, cudaStream_t s, bool rel,
                   bool keep_fitting);
void launch_frame_copy(const float2 *wv, uint32_t nblocks, int m, int e, const EncTarget *tgt, EncResult *res,
                       const uint32_t *ids, BlockSlot *table, StageAccum *acc, const FrameRecords &fr, cudaStream_t s,
                       bool rel);
// One block into a caller's buffer (rel: QSZR, e is the shift k)
void launch_encode_block(const float2 *amps, int m, int e, uint8_t *out, uint64_t cap, const LookbackScratch &scr,
                         const CallResult &res, cudaStream_t s, bool rel = false);
// The compressed store of a basis state: block b0 holds amplitude 1 at index loc, the others are zero
void launch_init_store(uint64_t nblocks, uint64_t b0, uint64_t loc, int m, int e, BlockSlot *table,
                       const ArenaDev &dev, const ArenaDev &host, StageAccum *acc, int *status, cudaStream_t s,
                       bool rel);
// leading phase ops of a stage for the decoder (count <= kMaxPreOps)
struct OpDev;
struct PreOps {
    const OpDev *ops = nullptr;
    uint32_t count = 0;
    uint32_t G = 1;                   // blocks per group
    const float2 *mats = nullptr;
    const uint64_t *gbase = nullptr;  // per group of the batch
    uint64_t *reset = nullptr;        // two words set to zero by the launch (null: none)
};
// decode with the block references read from table[ids[j]]
void launch_decode_table(const BlockSlot *table, const uint32_t *ids, uint32_t nblocks, int m, float2 *wv,
                         uint32_t *hist, int *status, const PreOps &pre, cudaStream_t s, bool rel = false);
void launch_reserve(uint32_t nblocks, const float *pred_log2, double margin, uint64_t worst, const ArenaDev &dev,
                    const ArenaDev &host, EncTarget *tgt, EncResult *res, int *status, cudaStream_t s);
void launch_copy_out(const float2 *wv, uint32_t nblocks, int m, const EncTarget *tgt, const uint32_t *ids,
                     BlockSlot *table, StageAccum *acc, int *status, cudaStream_t s);
void launch_copy_in(const BlockRef *in, uint32_t nblocks, int m, float2 *wv, int *status, cudaStream_t s);
// Amplitudes idx[0 .. count - 1] of a state whose blocks are in `table` (device arrays)
void launch_amplitudes(const BlockSlot *table, const uint64_t *idx, uint64_t count, int m, float2 *out, int *status,
                       cudaStream_t s, uint32_t codec);
void launch_gather_refs(const BlockSlot *table, const uint32_t *ids, uint32_t count, BlockRef *out,
                        cudaStream_t s);

}  // namespace qsim
