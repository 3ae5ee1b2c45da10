// Device functions of the QSZ1 codec (shared by the codec kernels and the
// persistent stage kernel). The format and the method are described in codec.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "codec.cuh"
#include "device_common.cuh"
#include "gates.cuh"

namespace qsim {
namespace cdev {


constexpr uint32_t kFlagA = 1u, kFlagP = 2u;
constexpr uint32_t kEpochMask = (1u << 30) - 1;
constexpr long long kSpinLimit = 1ll << 22;
constexpr uint64_t kLookbackWaitNs = 2000000000ull;  // 2 s

__device__ __forceinline__ uint64_t lb_word(uint32_t epoch, uint32_t flag, uint32_t value) {
    return (uint64_t(epoch & kEpochMask) << 34) | (uint64_t(flag) << 32) | value;
}

struct FrameGeom {
    int fl;
    uint32_t F, C, nframes;
    uint64_t data_start;
};

__device__ __forceinline__ FrameGeom geom(int m) {
    FrameGeom g;
    g.fl = m < 12 ? m : 12;
    g.F = 1u << g.fl;
    g.C = g.F / 32;
    g.nframes = 1u << (m - g.fl);
    g.data_start = 32 + ((4ull * (g.nframes + 1) + 15) & ~15ull);
    return g;
}

// QSZR (relative bound): code range, |x| < 2^64
constexpr uint32_t kQszrMaxU = 0x5F800000u;

// sign chunk type: 0 all clear, 1 all set (Algorithm 2's pre-scan), 3 run-coded (the signs change 1 to 3 times
// between neighbours), 2 stored word
__device__ __forceinline__ uint32_t sign_type(uint32_t w) {
    if (w == 0u) return 0u;
    if (w == 0xFFFFFFFFu) return 1u;
    return __popc((w ^ (w >> 1)) & 0x7FFFFFFFu) <= 3 ? 3u : 2u;
}

// run record of a run-coded sign word: bit 15 = sign of value 0, bits 0-4 / 5-9 / 10-14 the run boundaries
// p1 < p2 < p3 (value p differs from value p - 1), unused fields zero
__device__ __forceinline__ uint32_t sign_run_record(uint32_t w) {
    uint32_t t = (w ^ (w >> 1)) & 0x7FFFFFFFu;
    const uint32_t p1 = __ffs(t);
    t &= t - 1u;
    const uint32_t p2 = __ffs(t);
    t &= t - 1u;
    const uint32_t p3 = __ffs(t);
    return ((w & 1u) << 15) | p1 | (p2 << 5) | (p3 << 10);
}

// sign word of a run record; ok false for a record no encoder writes
__device__ __forceinline__ uint32_t sign_run_word(uint32_t rec, bool &ok) {
    const uint32_t p1 = rec & 31u, p2 = (rec >> 5) & 31u, p3 = (rec >> 10) & 31u;
    ok = p1 != 0u && (p2 == 0u ? p3 == 0u : (p2 > p1 && (p3 == 0u || p3 > p2)));
    uint32_t w = (rec >> 15) ? 0xFFFFFFFFu : 0u;
    if (p1) w ^= 0xFFFFFFFFu << p1;
    if (p2) w ^= 0xFFFFFFFFu << p2;
    if (p3) w ^= 0xFFFFFFFFu << p3;
    return w;
}

// packed sign-section counts of a frame: stored words Re | Im << 8, run records Re << 16 | Im << 24
__device__ __forceinline__ uint32_t sign_section_bytes(uint32_t mixed) {
    const uint32_t nw = (mixed & 0xffu) + ((mixed >> 8) & 0xffu), nr = ((mixed >> 16) & 0xffu) + (mixed >> 24);
    return (4u * nw + 2u * nr + 15u) & ~15u;
}

__device__ __forceinline__ uint32_t zigzag(int32_t d) {
    return (uint32_t(d) << 1) ^ uint32_t(d >> 31);
}

__device__ __forceinline__ int32_t unzigzag(uint32_t z) {
    return int32_t((z >> 1) ^ (0u - (z & 1u)));
}

// ---------------------------------------------------------------------------
// Leading phase ops of a stage, applied by the decoder. The phase index of a
// diagonal op splits into bits fixed for the frame (working bits >= the frame
// log, and outer qubits from the group), the lane's bits 0..4 and the chunk's
// bits 5.. ; the host builds the lane and chunk parts as byte tables (32 + 128
// bytes at float2 offset op.dlut of the phase area). pre_setup gives each op
// its tables' place (in the phase area, or staged in shared memory), pre_frame
// its per-lane register for the frame, and pre_chunk applies the ops to one
// chunk's amplitude.
// ---------------------------------------------------------------------------
constexpr uint32_t kPreFlip = 0xFFFFFFFFu;  // pre_ab[o].y of a phase flip
constexpr uint32_t kPreNone = 0xFFFFFFFFu;  // register of a flip whose amplitude is not in this lane
constexpr uint32_t kPreTabBytes = 160u + 8u * 256u;  // an op's staged tables: index bytes, phases

// ab.x: byte offset of a diagonal op's lane and chunk tables from the tables' base; ab.y: of its phases, or kPreFlip for
// a phase flip.
__device__ __forceinline__ uint2 pre_setup(const OpDev &op) {
    return op.type == OP_DIAG ? make_uint2(uint32_t(op.dlut) * 8u, uint32_t(op.mat) * 8u) : make_uint2(0u, kPreFlip);
}

// Per-lane register of each op for the frame whose first working index is w0f: a diagonal op's frame
// and lane bits of the phase index; for a phase flip, the chunk of the marked amplitude in the lane that
// holds it (kPreNone elsewhere).
template <int NP>
__device__ __forceinline__ void pre_frame(uint32_t (&cl)[NP > 0 ? NP : 1], const OpDev *ops, uint32_t nops,
                                          const uint2 *pre_ab, const uint8_t *tabs, uint64_t w0f, uint32_t fl,
                                          uint32_t lane, uint64_t gb) {
#pragma unroll
    for (int o = 0; o < NP; ++o) {
        cl[o] = kPreNone;
        if (uint32_t(o) >= nops) continue;
        const OpDev &op = ops[o];
        if (op.type == OP_DIAG) {
            uint32_t idx = 0;
            for (uint32_t j = 0; j < op.k; ++j) {
                const uint32_t src = op.dsrc[j];
                if (src < fl) continue;
                const uint64_t bit = src < 64 ? (w0f >> src) & 1ull : (gb >> (src - 64)) & 1ull;
                idx |= uint32_t(bit) << j;
            }
            cl[o] = idx | tabs[pre_ab[o].x + lane];
        } else if (op.basis_in_stage && gb == op.basis_outer && op.basis_w >= w0f &&
                   op.basis_w - w0f < (uint64_t(1) << fl)) {
            const uint32_t off = uint32_t(op.basis_w - w0f);
            if ((off & 31u) == lane) cl[o] = off >> 5;
        }
    }
}

template <int NP>
__device__ __forceinline__ float2 pre_chunk(float2 v, const uint32_t (&cl)[NP > 0 ? NP : 1], const uint2 *pre_ab,
                                            uint32_t nops, uint32_t c, const uint8_t *tabs) {
#pragma unroll
    for (int o = 0; o < NP; ++o) {
        if (uint32_t(o) >= nops) break;
        const uint2 ab = pre_ab[o];
        if (ab.y != kPreFlip) {
            const uint32_t idx = cl[o] | tabs[ab.x + 32u + c];
            const float2 ph = reinterpret_cast<const float2 *>(tabs + ab.y)[idx];
            v = make_float2(ph.x * v.x - ph.y * v.y, ph.x * v.y + ph.y * v.x);
        } else if (c == cl[o]) {
            v = make_float2(-v.x, -v.y);
        }
    }
    return v;
}

// ---------------------------------------------------------------------------
// Reservation of one block's slot from the two-tier pool: device arena
// first, then the pinned host arena; slots are padded to 256 bytes.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void reserve_slot(uint64_t want, const ArenaDev &dev, const ArenaDev &host, EncTarget *t,
                                             int *status) {
    const uint64_t sz = (want + 255) & ~255ull;
    uint64_t off = atomicAdd(reinterpret_cast<unsigned long long *>(dev.bump), sz);
    if (off + sz <= dev.cap) {
        t->ptr = dev.base + off;
        t->cap = sz;
        t->tier = 0;
        return;
    }
    if (host.base) {
        off = atomicAdd(reinterpret_cast<unsigned long long *>(host.bump), sz);
        if (off + sz <= host.cap) {
            t->ptr = host.base + off;
            t->cap = sz;
            t->tier = 1;
            return;
        }
    }
    t->ptr = nullptr;
    t->cap = 0;
    t->tier = 0;
    raise_status(status, QSIM_E_NOMEM);
}

// ---------------------------------------------------------------------------
// Relative-bound variant (QSZR, Sec. 4.3 Eq. 1-2 and Algorithm 2). The code of
// a component x is its FP32 magnitude bit pattern U = bits(|x|) (exponent plus
// linear mantissa: log2|x| up to a scale and offset) rounded to a multiple of
// 2^k: q = (U + 2^(k-1)) >> k; the sign (1 for x < 0 with q != 0) goes to a
// per-chunk sign word W = ballot(sign): chunks of all clear or all set signs
// store only their 2-bit type (0, 1: Algorithm 2's pre-scan); the others are
// coded losslessly, as a 2-byte run record when the signs change 1 to 3 times
// between neighbours (type 3), else as the raw word (type 2). Reconstruction
// |x'| = float(bits q << k).
// ---------------------------------------------------------------------------

// code of one component; bad collects QSIM_E_INVALID (non-finite, wins) or QSIM_E_RANGE
template <bool REL>
__device__ __forceinline__ int32_t quantize_one(float x, float inv_step, uint32_t k, int &bad) {
    if constexpr (REL) {
        const uint32_t U = __float_as_uint(x) & 0x7FFFFFFFu;
        if (U >= kQszrMaxU) {
            bad = U >= 0x7F800000u ? QSIM_E_INVALID : (bad ? bad : QSIM_E_RANGE);
            return 0;
        }
        return int32_t((U + (1u << (k - 1))) >> k);
    } else {
        const float tq = x * inv_step;  // exact: power-of-two scaling
        if (!(fabsf(tq) < 1073741824.0f)) {  // NaN, Inf or out of range
            bad = isfinite(x) ? (bad ? bad : QSIM_E_RANGE) : QSIM_E_INVALID;
            return 0;
        }
        return __float2int_rn(tq);
    }
}

// Warp look-back over the preceding frames of the block (status words of lb_block,
// tagged with epoch): publishes frame f's length, returns the bytes of frames 0..f-1.
// Every wait is time-bounded (QSIM_E_TIMEOUT).
__device__ __forceinline__ uint32_t lookback_warp(uint64_t *lb_block, uint32_t f, uint32_t epoch, uint32_t len,
                                                  int *status) {
    const int lane = threadIdx.x & 31;
    uint64_t *st = lb_block;
    if (f == 0) {
        if (lane == 0) st_relaxed_u64(st, lb_word(epoch, kFlagP, len));
        return 0;
    }
    if (lane == 0) st_relaxed_u64(st + f, lb_word(epoch, kFlagA, len));
    uint64_t excl = 0;
    int64_t end = int64_t(f) - 1;
    bool timed_out = false;
    while (true) {
        const int64_t p = end - lane;
        uint32_t flag = kFlagP, val = 0;
        if (p >= 0) {
            long long spins = 0;
            const uint64_t t0 = global_ns();
            while (true) {
                const uint64_t w = ld_relaxed_u64(st + p);
                const uint32_t fl = uint32_t(w >> 32) & 3u;
                if (fl != 0 && uint32_t(w >> 34) == epoch) {
                    flag = fl;
                    val = uint32_t(w);
                    break;
                }
                if (++spins > kSpinLimit || global_ns() - t0 > kLookbackWaitNs) {
                    timed_out = true;
                    flag = kFlagP;
                    val = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        const uint32_t pmask = __ballot_sync(kFull, flag == kFlagP);
        const int first = pmask ? __ffs(pmask) - 1 : 32;
        uint64_t contrib = lane <= first ? val : 0;
#pragma unroll
        for (int o = 16; o; o >>= 1) contrib += __shfl_xor_sync(kFull, contrib, o);
        excl += contrib;
        if (pmask) break;
        end -= 32;
    }
    if (__any_sync(kFull, timed_out) && lane == 0) raise_status(status, QSIM_E_TIMEOUT);
    if (lane == 0) st_relaxed_u64(st + f, lb_word(epoch, kFlagP, uint32_t(excl + len)));
    return uint32_t(excl);
}

}  // namespace cdev
}  // namespace qsim
