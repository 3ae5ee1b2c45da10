// Persistent stage kernel (sm_103a): one launch runs a whole stage.
//
// The paper overlaps the SV groups of a stage by dealing them round-robin to
// CUDA streams (Sec. 4.2). Here the same overlap happens inside one launch:
// every CTA repeatedly takes the next work item from a global queue of steps. A
// step is one phase of one unit: decode frames, [predict + reserve], a gate pass's
// tiles (pass by pass), encode frames, [copy frames to their slots]. A unit is one
// or more SV groups of the stage, together about 2^22 amplitudes, so that its
// phases are long enough to fill the GPU. A CTA waits (bounded spin) until the
// unit's previous phase is complete before running its item.
//
// Items are handed out in queue order, so the order decides what overlaps. Units
// that share working-vector slots form a lane, whose steps are in dependency order
// (stage after stage; within a stage as many units side by side as the lane has
// slots, phase by phase); a batch's small circuits have a lane each, and the lanes
// are merged by the fraction of their steps, so that while one circuit's phase
// drains the CTAs work on the others'. (With every circuit's stage in the queue as a
// whole, the time of a batch was the sum of its circuits' alone: 16 circuits of 17 to 22
// qubits took 14.4 ms, 6.4 ms as lanes; 48 ms with a warp per frame and a group per
// unit.) Every dependency
// points to an earlier item of the same lane, which was taken by a CTA that is
// already running: the schedule cannot deadlock even when not every CTA is resident.
//
// Data produced by other CTAs of the same launch is read through L2 (ld.cg),
// since the per-SM L1 caches are not coherent within a launch.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "codec.cuh"
#include "codec_dev.cuh"
#include "codec_team.cuh"
#include "device_common.cuh"
#include "gates.cuh"
#include "gates_dev.cuh"
#include "mlp.cuh"
#include "persistent.cuh"

namespace qsim {

namespace {

using cdev::FrameGeom;
using cdev::geom;

template <bool UM>
constexpr int kPT = int(persistent_threads(UM));

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ EncTarget load_target(const EncTarget *t) {
    EncTarget r;
    r.ptr = reinterpret_cast<uint8_t *>(__ldcg(reinterpret_cast<const unsigned long long *>(&t->ptr)));
    r.cap = __ldcg(reinterpret_cast<const unsigned long long *>(&t->cap));
    r.tier = __ldcg(&t->tier);
    r.pad = 0;
    return r;
}

// REL: the relative-bound codec (QSZR). UM: the plan's dense ops
// of width 3 to 5 (TF32 or split BF16) and 6 (TF32) run on tcgen05 (TMEM accumulator and MMA mbarrier held by each
// CTA for the launch).
template <int PREC, bool REL, bool UM>
__global__ void __launch_bounds__(kPT<UM>, 512 / kPT<UM>) k_stage_persistent(PLaunch L) {
    constexpr int PT = kPT<UM>;
    extern __shared__ float4 dsm[];
    __shared__ gdev::PassSmem PS;
    __shared__ OpDev s_pre[kMaxPreOps];
    __shared__ uint2 s_pre_ab[kMaxPreOps];
    __shared__ __align__(16) PSeg S;
    __shared__ cdev::TeamSmem s_team[PT / 32];
    __shared__ float s_pred[4 * kMlpHidden];  // predictor: features, hidden layers
    __shared__ uint32_t s_item, s_seg;
    __shared__ PStep s_step;
    __shared__ uint32_t s_pcache[2];  // key (segment x 256 + pass) of the pass staged in dsm; its B resident
    __shared__ int s_flag, s_abort;
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        s_seg = ~0u;
        s_step.begin = s_step.count = 0;
        s_pcache[0] = ~0u;
        s_pcache[1] = 0;
    }
    uint32_t mphase = 0;     // parity of the MMA mbarrier's next phase (UM)
    bool mma_ok = true;      // false after an MMA wait ran out (then a last bounded wait before TMEM is freed)
    if constexpr (UM) {
        if (warp == 0) umma::tmem_alloc(umma::smem_addr(&PS.tmem), gdev::umma_pass_tmem_cols(0));
        if (tid == 0) umma::mbar_init(umma::smem_addr(&PS.mbar), 1);
        umma::fence_before_sync();
    }
    __syncthreads();
    if constexpr (UM) umma::fence_after_sync();

    // Thread 0's words (cur: warp 0's), in shared memory: the passes are short of registers, and what is held through
    // an item in each thread's is spilled inside their loops.
    struct Own {
        // the (launch group, phase) whose dependencies this CTA last saw met; later items of the same phase of the
        // same group skip the wait (the counters only grow within a launch)
        uint64_t dep_key;
        // a done counter of a per-item phase whose increments this CTA holds back, and their number; they are added
        // (after a fence) when the CTA completes an item of another phase, before it waits on any dependency and when
        // it leaves, so a CTA that waits never holds counts another CTA waits for
        uint32_t *pend_done;
        uint32_t pend_cnt;
        // the next item, claimed one item ahead so that the claim's latency hides under the current item (every
        // dependency points to an earlier item, and the grid is one wave of resident CTAs, so the smallest unfinished
        // item is always some CTA's current item and the queue keeps moving)
        uint32_t nx_item;
        uint32_t cur;  // the step in s_step
    };
    __shared__ Own own;
    if (tid == 0) own = Own{~0ull, nullptr, 0u, atomicAdd(L.ctr, 1u), 0u};
    auto flush = [&]() {
        if (own.pend_cnt) {
            __threadfence();
            atomicAdd(own.pend_done, own.pend_cnt);
            own.pend_cnt = 0;
        }
    };
    // thread 0: wait for the item's dependencies (the group's previous phase; for its first phase the slot's
    // previous group and the circuit's previous stage); returns 1 when the item must skip its work (a device
    // error, or a wait that ran out)
    auto deps = [&]() -> int {
        const uint32_t q = S.group_begin + s_step.grp;
        const uint64_t key = uint64_t(q) * kMaxPhases + s_step.phase;
        if (key == own.dep_key) return ld_relaxed_u32(reinterpret_cast<const uint32_t *>(L.status)) != 0;
        flush();
        const uint32_t *flag = nullptr, *flag2 = nullptr;
        uint32_t need = 0;
        if (s_step.phase > 0) {
            flag = L.done + uint64_t(q) * kMaxPhases + s_step.phase - 1;
            need = s_step.need;
        } else {
            const uint32_t prev = L.g_prev[q];
            if (prev != kNoGroup) {  // the slot's previous unit must have finished
                flag = L.done + uint64_t(prev) * kMaxPhases + kMaxPhases - 1;
                need = 1;
            }
            flag2 = S.prev_flag;
        }
        if (S.stall_test && s_step.grp == 0 && s_step.phase == 1) ++need;  // never reached: exercises the time limit
        bool met = true;
        if (flag || flag2) {
            const uint64_t t0 = global_ns();
            while ((flag && ld_acquire_u32(flag) < need) || (flag2 && ld_acquire_u32(flag2) == 0)) {
                if (global_ns() - t0 > L.wait_ns) {
                    raise_status(L.status, QSIM_E_TIMEOUT);
                    met = false;
                    break;
                }
                __nanosleep(256);
            }
        }
        if (met) own.dep_key = key;
        // after any device error the remaining items only keep the schedule going
        return (!met || ld_relaxed_u32(reinterpret_cast<const uint32_t *>(L.status)) != 0) ? 1 : 0;
    };

    while (true) {
        if (warp == 0) {
            __syncwarp();  // thread 0 has written own and read s_step
            const uint32_t it = own.nx_item;
            // a CTA's items only move forward, mostly within one step: then s_step holds it
            if (it < L.total_items && it - s_step.begin >= s_step.count) {
                uint32_t cur = own.cur;
                for (;;) {  // the last step that begins at or before the item, 32 steps at a look
                    const uint32_t k = cur + uint32_t(tid);
                    const uint32_t begin = k < L.nsteps ? __ldg(&L.steps[k].begin) : 0xffffffffu;
                    const uint32_t ahead = __popc(__ballot_sync(kFull, begin <= it)) - 1;
                    cur += ahead;
                    if (ahead < 31) break;
                }
                __syncwarp();
                if (tid == 0) own.cur = cur;
                if (tid < int(sizeof(PStep) / 4))
                    reinterpret_cast<uint32_t *>(&s_step)[tid] = __ldg(reinterpret_cast<const uint32_t *>(L.steps + cur) + tid);
            }
            __syncwarp();
            if (tid == 0) {
                s_item = it;
                if (it < L.total_items) {
                    own.nx_item = atomicAdd(L.ctr, 1u);
                    // the current segment's descriptor is in S: check the dependencies before the barrier
                    if (s_step.seg == s_seg) s_abort = deps();
                }
            }
        }
        __syncthreads();
        const uint32_t item = s_item;
        if (item >= L.total_items) break;
        const uint32_t want = s_step.seg;
        if (want != s_seg) {  // uniform: a new segment, load its descriptor and leading phase ops
            const unsigned long long *src = reinterpret_cast<const unsigned long long *>(L.segs + want);
            unsigned long long *dst = reinterpret_cast<unsigned long long *>(&S);
            for (int t = tid; t < int(sizeof(PSeg) / 8); t += PT) dst[t] = __ldg(src + t);
            __syncthreads();
            if (tid < int(S.npre)) {
                s_pre[tid] = S.ops[S.pre_begin + tid];
                s_pre_ab[tid] = cdev::pre_setup(S.ops[S.pre_begin + tid]);
            }
            if (tid == 0) {
                s_seg = want;
                s_abort = deps();
            }
            __syncthreads();
        }
        const FrameGeom g = geom(int(S.m));
        const uint32_t gframes = S.G * g.nframes;
        const uint32_t grp = s_step.grp, q = S.group_begin + grp;  // the unit's number in the stage and the launch
        const uint32_t type = s_step.type, i = item - s_step.begin;
        const bool abort_item = s_abort != 0;
        // the item's SV group in the unit and its place among the group's items of this phase. Every divisor here is a
        // power of two: shifts, except in the tcgen05 forms, where they cost registers (26-qubit random brick in one
        // group: 26.1 -> 25.5 ms in FP32, 16.7 -> 16.3 in TF32 warp MMAs; tcgen05 1 to 2 % slower with them)
        const uint32_t gi = UM ? i / s_step.per : S.gpu == 1u ? 0u : i / s_step.per;
        const uint32_t ii = UM ? i % s_step.per : i - gi * s_step.per;
        const uint64_t sg = uint64_t(grp) * S.gpu + gi;  // SV group of the stage
        float2 *wv = L.wv + L.g_wv[q] + (uint64_t(gi) << S.W);
        const uint32_t *ids = S.ids + sg * S.G;
        const uint64_t gb = S.gbase[sg];
        const uint64_t bbase = sg * S.G;  // per-group block arrays
        const uint32_t sf0 = L.g_frame[q] + gi * gframes;  // the group's first frame in the frame records
        const bool by_arrival = type == PH_ENCODE || type == PH_COPY;
        // frame-parallel items: a team per frame, each with its own tile in dsm
        const uint32_t tl = 31u - uint32_t(__clz(cdev::team_threads(g.C)));
        const uint32_t tn = UM ? cdev::team_threads(g.C) : 1u << tl, team = UM ? uint32_t(tid) / tn : uint32_t(tid) >> tl;
        const cdev::Team tm{UM ? uint32_t(tid) % tn : uint32_t(tid) & (tn - 1u), tn, 1u + team};
        uint8_t *tile = reinterpret_cast<uint8_t *>(dsm) + team * cdev::team_tile_bytes(g.C);
        const uint32_t fi = ii * (UM ? PT / tn : PT >> tl) + team;
        const uint32_t jj = UM ? fi / g.nframes : fi >> (S.m - uint32_t(g.fl));
        const uint32_t f = UM ? fi % g.nframes : fi & (g.nframes - 1u);
        const uint64_t a0 = (uint64_t(jj) << S.m) + uint64_t(f) * g.F;
        if (type != PH_PASS && tid == 0) s_pcache[0] = ~0u;  // dsm is overwritten: no pass stays staged
        if (abort_item) {
            // skip the work, keep the counts
        } else if (type == PH_DECODE) {
            if (fi < gframes) {
                const BlockSlot sl = S.tab_in[ids[jj]];
                cdev::decode_frame_team<kMaxPreOps, REL>(tm, s_team[team], tile, sl.ptr, sl.bytes, g, int(S.m), f,
                                                         wv + a0, S.hist ? S.hist + (bbase + jj) * 32 : nullptr,
                                                         L.status, s_pre, s_pre_ab, S.npre,
                                                         reinterpret_cast<const uint8_t *>(S.mats),
                                                         uint64_t(jj) << S.m, gb);
            }
        } else if (type == PH_PASS) {
            if constexpr (UM) {
                // tile loads by cp.async (L1-cached): the item's dependencies were acquired by thread 0 (for this
                // group and phase, in this item or an earlier one of this CTA) before the CTA barrier above, so the
                // memory model orders them after the previous phase's writes; L1 starts empty at the launch
                mma_ok &= gdev::pass_tile<PT, 5, PREC, false, true>(wv, S.passes[s_step.arg], S.blob, S.mats, S.bfr,
                                                                   ii, gb, PS, reinterpret_cast<float2 *>(dsm),
                                                                   L.status, &mphase, s_pcache,
                                                                   s_seg * 256u + s_step.arg);
            } else {
                gdev::pass_tile<PT, 5, PREC, false>(wv, S.passes[s_step.arg], S.blob, S.mats, S.bfr, ii, gb, PS,
                                                   reinterpret_cast<float2 *>(dsm), L.status, nullptr, s_pcache,
                                                   s_seg * 256u + s_step.arg);
            }
        } else if (type == PH_ENCODE) {
            if (fi < gframes) {
                cdev::load_rows_team(tm, tile, wv + a0, g.C);
                const cdev::EncFrame r = cdev::encode_frame_team<REL>(tm, s_team[team], tile, g, S.e, L.status);
                if (g.nframes == 1) {
                    // a block of one frame: straight to its slot
                    if (tm.t == 0) {
                        const uint32_t total = uint32_t(g.data_start) + r.len;
                        const EncTarget t = cdev::reserve_block(total, S.pparams != nullptr, &S.tgt[bbase + jj], S.dev,
                                                                S.host, S.acc, L.status);
                        EncResult out{};
                        out.err_sq = r.err_sq;
                        out.norm_sq = r.norm_sq;
                        s_team[team].bc = reinterpret_cast<uint64_t>(
                            cdev::finish_single_frame(total, t, out, S.tab_out + ids[jj], S.acc));
                        S.res[bbase + jj] = out;
                        atomicAdd(&S.acc->err_sq, out.err_sq);
                        atomicAdd(&S.acc->norm_sq, out.norm_sq);
                    }
                    tm.sync();
                    cdev::store_single_frame<REL>(tm, tile, g, int(S.m), S.e, r.len,
                                                  reinterpret_cast<uint8_t *>(s_team[team].bc));
                } else {
                    cdev::stage_frame(tm, tile, r, wv + a0, L.side + uint64_t(sf0 + fi) * L.side_bytes);
                    if (tm.t == 0) {
                        L.flen[sf0 + fi] = r.len;
                        if (REL) L.fhead[sf0 + fi] = r.head;
                        L.part[sf0 + fi] = make_float2(r.err_sq, r.norm_sq);
                        __threadfence();  // read by the phase's last item and the copy phase on other CTAs
                    }
                }
            }
        } else if (type == PH_COPY) {
            if (fi < gframes)  // frames of 4096 amplitudes: teams of 128
                cdev::copy_frame_team<REL>(tm, wv + a0, L.side + uint64_t(sf0 + fi) * L.side_bytes,
                                           __ldcg(L.flen + sf0 + fi), REL ? __ldcg(L.fhead + sf0 + fi) : 256u,
                                           __ldcg(L.foff + sf0 + fi), g, int(S.m), S.e, f,
                                           load_target(&S.tgt[bbase + jj]), &S.res[bbase + jj], S.tab_out + ids[jj],
                                           S.acc);
        } else if (type == PH_PREDICT) {
            // one SV group: its blocks share every input of the predictor, so one forward pass sizes them all. Weights in
            // dsm, W2's rows padded to 65 words (lanes walk rows)
            constexpr int IN = kMlpIn, HID = kMlpHidden, OB1 = HID * IN, OW2 = OB1 + HID, OB2 = OW2 + HID * (HID + 1),
                          OW3 = OB2 + HID, OB3 = OW3 + HID, FW2 = HID * IN + HID;
            float *w = reinterpret_cast<float *>(dsm), *x = s_pred, *h1 = s_pred + HID, *h2 = s_pred + 2 * HID;
            for (int t = tid; t < kMlpParams; t += PT) {
                const float v = S.pparams[t];
                const int o = t < FW2 ? t : t < FW2 + HID * HID ? t + (t - FW2) / HID : t + HID;
                w[o] = S.pbf16 ? __bfloat162float(__float2bfloat16_rn(v)) : v;
            }
            if (tid < 32) {
                uint32_t c = 0;
                for (uint32_t k = 0; k < S.G; ++k) c += __ldcg(S.hist + (bbase + k) * 32 + tid);
                x[tid] = float(c) * (1.0f / (float(S.G) * float(2ull << S.m)));
                const uint32_t nz = __ballot_sync(kFull, c != 0);
                if (tid == 0) x[32] = float(nz ? 31 - __clz(nz) : 0) / 32.f;
                if (tid < 8) x[33 + tid] = S.sf.v[tid];
            }
            __syncthreads();
            if (tid < HID) {
                float a = w[OB1 + tid];
                for (int j = 0; j < IN; ++j) a = fmaf(w[tid * IN + j], x[j], a);
                h1[tid] = fmaxf(a, 0.f);
            }
            __syncthreads();
            if (tid < HID) {
                float a = w[OB2 + tid];
                for (int j = 0; j < HID; ++j) a = fmaf(w[OW2 + tid * (HID + 1) + j], h1[j], a);
                h2[tid] = fmaxf(a, 0.f);
            }
            __syncthreads();
            float y = w[OB3];
            for (int j = 0; j < HID; ++j) y = fmaf(w[OW3 + j], h2[j], y);  // as mlp_forward_one
            double pr = double(y) + double(S.m + 3);
            pr = pr < 0 ? 0 : (pr > 40 ? 40 : pr);
            const double want_b = exp2(pr) * (1.0 + S.margin);
            const uint64_t want = want_b >= double(S.worst) ? S.worst : uint64_t(want_b);
            for (uint32_t k = tid; k < S.G; k += PT) cdev::reserve_slot(want, S.dev, S.host, &S.tgt[bbase + k], L.status);
            // the group's histograms are consumed: leave them zero for the next stage
            for (uint32_t t = tid; t < S.G * 32; t += PT) S.hist[bbase * 32 + t] = 0;
        }
        // ---- completion ----
        __syncthreads();
        // The step's numbers are read from s_step again. Warp 0 overwrites it at the loop's top: after thread 0's reads
        // here, and after one more barrier where every thread reads.
        if (!by_arrival) {
            if (tid == 0) {
                uint32_t *done = L.done + uint64_t(S.group_begin + s_step.grp) * kMaxPhases + s_step.phase;
                if (done != own.pend_done) {
                    flush();
                    own.pend_done = done;
                }
                ++own.pend_cnt;
            }
            continue;
        }
        const uint32_t p = s_step.phase, count = s_step.count, dq = S.group_begin + s_step.grp;
        uint32_t *done = L.done + uint64_t(dq) * kMaxPhases + p;
        if (tid == 0) {
            __threadfence();
            s_flag = atomicAdd(L.arrive + uint64_t(dq) * kMaxPhases + p, 1u) == count - 1;
        }
        __syncthreads();
        if (!s_flag) continue;
        __threadfence();
        if (!abort_item && type == PH_ENCODE && g.nframes > 1) {
            // the unit's frame lengths are complete: frame offsets, the blocks' slots (with learned sizing every
            // predicted slot its block fits is kept) and the stage's error sums, a team of 128 per block
            const uint32_t f0 = L.g_frame[dq];
            const uint64_t b0 = uint64_t(grp) * S.gpu * S.G;
            for (uint32_t k = team; k < S.gpu * S.G; k += PT / 128) {
                double a, b;
                const uint32_t fk = f0 + k * g.nframes;
                const uint32_t total = cdev::block_offsets_team(tm, s_team[team], L.flen + fk, L.part + fk, L.foff + fk,
                                                                g.nframes, uint32_t(g.data_start), a, b);
                if (tm.t == 0) {
                    cdev::reserve_block(total, S.pparams != nullptr, &S.tgt[b0 + k], S.dev, S.host, S.acc, L.status);
                    EncResult out{};
                    out.err_sq = a;
                    out.norm_sq = b;
                    S.res[b0 + k] = out;
                    atomicAdd(&S.acc->err_sq, a);
                    atomicAdd(&S.acc->norm_sq, b);
                }
                tm.sync();
            }
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            atomicExch(done, count);
            if (p == S.nphases - 1) {
                // the group is finished: its slot may be reused; the stage may be complete
                atomicExch(L.done + uint64_t(dq) * kMaxPhases + kMaxPhases - 1, 1u);
                if (atomicAdd(S.fin_count, 1u) == S.ngroups - 1) {
                    if (S.reset_bumps) {
                        // every group of the stage has read its input arena: the next stage writes there
                        S.reset_bumps[0] = 0;
                        S.reset_bumps[1] = 0;
                    }
                    __threadfence();
                    atomicExch(S.fin_flag, 1u);
                }
            }
        }
    }
    if (tid == 0) flush();
    if constexpr (UM) {
        // after an MMA wait that ran out, wait (bounded) once more for that op's MMAs before TMEM is freed
        if (!mma_ok) umma::mbar_wait(umma::smem_addr(&PS.mbar), mphase ^ 1u, gdev::kUmmaWaitNs);
        umma::fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            umma::fence_after_sync();
            umma::tmem_dealloc(PS.tmem, gdev::umma_pass_tmem_cols(0));
        }
    }
    // the last CTA out resets the queue
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(L.ctr + 1, 1u) == gridDim.x - 1) {
            L.ctr[0] = 0;
            L.ctr[1] = 0;
        }
    }
}

template <int PREC, bool REL, bool UM>
struct LaunchShape {  // of a device; mu guards the two values (runs on several threads)
    std::mutex mu;
    int grid = 0;
    size_t attr_smem = 0;
    static LaunchShape &current() {
        static LaunchShape shapes[64];
        int dev = 0;
        cudaGetDevice(&dev);
        return shapes[dev & 63];
    }
};

// kernel attributes and the grid (one wave of resident CTAs); done outside any stream capture
template <int PREC, bool REL, bool UM>
int prepare_prec(size_t smem) {
    LaunchShape<PREC, REL, UM> &shape = LaunchShape<PREC, REL, UM>::current();
    std::lock_guard<std::mutex> lk(shape.mu);
    if (shape.attr_smem < smem) {
        if (cudaFuncSetAttribute(k_stage_persistent<PREC, REL, UM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(smem)) != cudaSuccess)
            return QSIM_E_CUDA;
        shape.attr_smem = smem;
        shape.grid = 0;
    }
    if (!shape.grid) {
        // resident CTAs per SM from the kernel's registers and shared memory and the SM's limits (65536 registers,
        // 2048 threads, 228 KB of shared memory with 1 KB reserved per CTA); the runtime's occupancy query was
        // seen to answer 1 where more CTAs were resident
        int per_sm = 1;
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, k_stage_persistent<PREC, REL, UM>) == cudaSuccess) {
            const int regs = ((fa.numRegs > 0 ? fa.numRegs : 255) + 7) & ~7;
            constexpr int PT = kPT<UM>;
            const int by_regs = 65536 / (regs * PT);
            const int by_smem = int((228u * 1024u) / (smem + fa.sharedSizeBytes + 1024u));
            per_sm = by_regs < by_smem ? by_regs : by_smem;
            if (per_sm > 2048 / PT) per_sm = 2048 / PT;
            // each CTA of a tcgen05 launch holds its TMEM columns for the launch: no more than the SM's 512
            if (UM && per_sm > int(512u / gdev::umma_pass_tmem_cols(0))) per_sm = int(512u / gdev::umma_pass_tmem_cols(0));
            if (per_sm < 1) per_sm = 1;
        }
        shape.grid = num_sms() * per_sm;
    }
    return QSIM_OK;
}

template <int PREC, bool REL, bool UM>
int launch_stage_prec(const PLaunch &a, size_t smem, cudaStream_t s, int *grid_out) {
    LaunchShape<PREC, REL, UM> &shape = LaunchShape<PREC, REL, UM>::current();
    int grid;
    {
        std::lock_guard<std::mutex> lk(shape.mu);
        if (shape.attr_smem < smem || !shape.grid) return QSIM_E_INVALID;
        grid = shape.grid;
    }
    k_stage_persistent<PREC, REL, UM><<<grid, kPT<UM>, smem, s>>>(a);
    if (grid_out) *grid_out = grid;
    count_launch();
    return QSIM_OK;
}

// um: the tcgen05 forms, TF32 and split BF16, with 128-thread CTAs; the others have 256 threads
template <bool REL>
int prepare_codec(int prec, size_t smem, bool um) {
    if (prec == QSIM_PREC_TF32)
        return um ? prepare_prec<QSIM_PREC_TF32, REL, true>(smem) : prepare_prec<QSIM_PREC_TF32, REL, false>(smem);
    if (prec == QSIM_PREC_BF16X3)
        return um ? prepare_prec<QSIM_PREC_BF16X3, REL, true>(smem) : prepare_prec<QSIM_PREC_BF16X3, REL, false>(smem);
    return prepare_prec<QSIM_PREC_FP32, REL, false>(smem);
}

template <bool REL>
int launch_codec(const PLaunch &a, int prec, size_t smem, cudaStream_t s, int *grid, bool um) {
    if (prec == QSIM_PREC_TF32)
        return um ? launch_stage_prec<QSIM_PREC_TF32, REL, true>(a, smem, s, grid)
                  : launch_stage_prec<QSIM_PREC_TF32, REL, false>(a, smem, s, grid);
    if (prec == QSIM_PREC_BF16X3)
        return um ? launch_stage_prec<QSIM_PREC_BF16X3, REL, true>(a, smem, s, grid)
                  : launch_stage_prec<QSIM_PREC_BF16X3, REL, false>(a, smem, s, grid);
    return launch_stage_prec<QSIM_PREC_FP32, REL, false>(a, smem, s, grid);
}

}  // namespace

size_t persistent_smem_bytes(size_t pass_bytes, bool um) {
    const size_t mlp = size_t(kMlpParams + kMlpHidden) * sizeof(float);
    // a tile per team: threads / max(32, C) of them, most in all at C = 32
    const size_t tiles = size_t(persistent_threads(um) / 32) * cdev::team_tile_bytes(32);
    return std::max(std::max(pass_bytes, mlp), tiles);
}

int prepare_stage_persistent(int prec, size_t smem, bool rel, bool um) {
    return rel ? prepare_codec<true>(prec, smem, um) : prepare_codec<false>(prec, smem, um);
}

int launch_stage_persistent(const PLaunch &a, int prec, size_t smem, cudaStream_t s, int *grid, bool rel, bool um) {
    return rel ? launch_codec<true>(a, prec, smem, s, grid, um) : launch_codec<false>(a, prec, smem, s, grid, um);
}

}  // namespace qsim
