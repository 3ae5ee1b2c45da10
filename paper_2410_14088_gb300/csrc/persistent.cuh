// Persistent stage kernel: work-item phases, arguments and launcher.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "codec.cuh"
#include "gates.cuh"
#include "mlp.cuh"

namespace qsim {

enum PhaseType : uint32_t {
    PH_DECODE = 0,   // frames_per_item frames (a team of threads each), leading phase ops applied
    PH_PASS = 1,     // one tile of gate pass `arg`
    PH_PREDICT = 2,  // one SV group: predicted sizes and slot reservation
    PH_ENCODE = 3,   // frames_per_item frames. Blocks of one frame go to their slots, reserved here. Larger blocks' images
                     // are staged; the unit's last item turns their lengths into frame offsets, reserves the blocks'
                     // exact slots (with learned sizing: keeps every predicted slot its block fits) and folds the error
                     // partials into the stage totals
    PH_COPY = 4      // frames_per_item staged frames copied into their slots (blocks of more than one frame)
};

// One step of the work queue: phase `phase` of a unit, `count` items from item `begin` on.
struct PStep {
    uint32_t begin, seg, grp;  // first item; segment (stage of a circuit); unit of the segment
    uint32_t phase, type, arg;
    uint32_t per;    // items per SV group of the unit
    uint32_t need;   // items of the unit's previous phase
    uint32_t count;
    uint32_t pad[3];
};
static_assert(sizeof(PStep) % 16 == 0, "steps are read as words");

constexpr int kMaxPhases = 128;
// threads per CTA: 128 in launches whose dense ops run on tcgen05 (one thread per index group of a width-5 op, four CTAs
// per SM filling its TMEM), else 256 (two CTAs per SM)
__host__ __device__ constexpr uint32_t persistent_threads(bool um) { return um ? 128u : 256u; }
constexpr uint32_t kNoGroup = 0xffffffffu;

// One stage of one circuit, its SV groups taken gpu at a time as units. Its units take the launch's numbers group_begin
// and on (working-vector slot and the done/arrive counters follow that number).
struct PSeg {
    uint32_t group_begin;
    uint32_t W, G, ngroups, m, nphases, npre, pre_begin, pbf16;  // ngroups: units
    uint32_t gpu;  // SV groups per unit
    int e;
    uint32_t stall_test;  // 1: group 0's second phase waits for a count never reached (bounded-wait test)
    const PassDev *passes;
    const OpDev *ops;
    const float2 *mats;
    const uint4 *blob;       // the plan's pass blobs
    const uint32_t *bfr;     // B-fragment tables of the tensor-core precisions
    const uint32_t *ids;     // group-major block ids of the stage
    const uint64_t *gbase;   // per group: full-index bits of its outer qubits
    BlockSlot *tab_in, *tab_out;
    StageAccum *acc;
    ArenaDev dev, host;
    uint64_t worst;
    // per block of the stage (group-major); the kernel leaves hist zeroed for the next stage
    EncTarget *tgt;
    EncResult *res;
    uint32_t *hist;
    // predictor
    const float *pparams;
    StageFeatures sf;
    double margin;
    // stage barrier within one launch: the previous stage of the same circuit
    // (null when it ran in an earlier launch) and this stage's own counters
    const uint32_t *prev_flag;  // becomes 1 once every group of the previous stage has finished
    uint32_t *fin_count;        // groups of this stage finished
    uint32_t *fin_flag;         // set to 1 after the last group (and the arena reset below)
    uint64_t *reset_bumps;      // two bump words zeroed when the stage is complete (null: none)
};

struct PLaunch {
    const PSeg *segs;
    const PStep *steps;      // in queue order
    uint32_t nsteps;
    uint64_t total_items;    // below 2^32
    uint32_t total_groups;
    // per unit of the launch (host-planned working-vector slots): amplitude offset of its slot in wv, frame offset of its
    // slot in the frame records, and the unit that used the slot before (kNoGroup: none)
    const uint64_t *g_wv;
    const uint32_t *g_frame;
    const uint32_t *g_prev;
    float2 *wv;
    // per slot frame (blocks of more than one frame): image bytes before the bit-plane words, stream bytes, offset in the
    // block's stream, bytes in `side` (relative codec), error partials
    uint8_t *side;
    uint32_t side_bytes;
    uint32_t *flen, *foff, *fhead;
    float2 *part;
    uint32_t *done, *arrive;  // per launch group x kMaxPhases each, zero at launch
    uint32_t *ctr;            // queue head, CTAs finished
    int *status;
    uint64_t wait_ns;         // limit of every dependency wait
};

// pass_bytes: the largest tile + pass blob + matrix area of the launch's passes
size_t persistent_smem_bytes(size_t pass_bytes, bool um);
// um: the launch's passes carry tcgen05 dense ops (TF32 widths 3 to 6, or split BF16 widths 3 to 5)
int prepare_stage_persistent(int prec, size_t smem, bool rel = false, bool um = false);
int launch_stage_persistent(const PLaunch &a, int prec, size_t smem, cudaStream_t s, int *grid, bool rel = false,
                            bool um = false);

}  // namespace qsim
