// QSZ1 block codec kernels (sm_103a).
//
// The paper compresses every SV block with a GPU lossy compressor under a
// point-wise error bound (Sec. 4.3) and notes that sign runs are detected with
// warp votes. QSZ1 is this library's own absolute-bound format:
//   step s = 2^e, e = the largest integer with 2^e <= 2 eb (so s/2 <= eb);
//   q = round-half-even(x / s) in int32, |q| < 2^30;  x' = q * s exactly;
//   planes Re and Im; chunks of 32 values; d_0 = q_0, d_j = q_j - q_{j-1};
//   z = zigzag(d); w = bit length of OR z; bit planes W_b = ballot(bit b of z).
// Stream: 32-byte header (u32 magic "QSZ1", u16 version 1, u16 flags 0, u8 m,
// u8 frame_log, i8 e, u8 0, u32 nframes, u64 total_bytes, u64 0), u32
// offsets[nframes+1] padded to 16 bytes, then frames of F = min(4096, 2^m)
// amplitudes: u8 widths[2C] (C = F/32, Re then Im) padded to 16, the words of
// each chunk (Re chunks then Im chunks), padded to 16. A frame whose widths
// are all zero has length 0 (the all-zero run elision).
//
// A frame is coded by a team of threads, one per chunk pair (codec_team.cuh).
#include <cuda_runtime.h>
#include <stdint.h>

#include "codec.cuh"
#include "codec_dev.cuh"
#include "codec_team.cuh"
#include "device_common.cuh"
#include "gates.cuh"

namespace qsim {

namespace {

using namespace cdev;

// One frame per team of max(32, C) threads, which is the CTA. Blocks are read from table[ids[j]] (ids null: block
// b0 + j). NP: the most leading phase ops the kernel applies (pre.count <= NP). Five CTAs of 128 threads per SM (35 KB of tile
// each would fit six) leave 102 registers, of which a chunk pair's 64 bit-plane words (the wide path) and the rest take
// 91 to 96; only the relative codec's form with more than two leading ops spills (68 bytes a thread). A launch
// of few frames is one chain of latencies, so its CTAs are as many as its frames: one 1024-amplitude frame per CTA took
// 6 us where a warp per frame took 22.
template <int NP, bool REL>
__global__ void __launch_bounds__(kTeamMax, 5) k_decode(const BlockSlot *__restrict__ table,
                                                        const uint32_t *__restrict__ ids, uint64_t b0,
                                                        uint32_t nblocks, int m, float2 *__restrict__ wv,
                                                        uint32_t *__restrict__ hist, int *status, PreOps pre) {
    extern __shared__ __align__(16) uint8_t tile[];
    const FrameGeom g = geom(m);
    __shared__ OpDev s_pre[NP > 0 ? NP : 1];
    __shared__ uint2 s_pre_ab[NP > 0 ? NP : 1];
    __shared__ TeamSmem S;
    const Team tm{threadIdx.x, blockDim.x, 1};
    if (pre.reset && blockIdx.x == 0 && threadIdx.x < 2) pre.reset[threadIdx.x] = 0;
    // the leading ops' descriptors and tables, staged once per CTA beside its tile
    uint8_t *tabs = tile + team_tile_bytes(g.C);
    if (NP > 0) {
        constexpr uint32_t W = sizeof(OpDev) / 4;
        for (uint32_t i = threadIdx.x; i < pre.count * W; i += blockDim.x)
            reinterpret_cast<uint32_t *>(s_pre)[i] = __ldg(reinterpret_cast<const uint32_t *>(pre.ops) + i);
        __syncthreads();
        for (uint32_t o = 0; o < pre.count; ++o) {
            const bool diag = s_pre[o].type == OP_DIAG;
            if (threadIdx.x == 0)
                s_pre_ab[o] = make_uint2(o * kPreTabBytes, diag ? o * kPreTabBytes + 160u : kPreFlip);
            if (!diag) continue;
            uint64_t *d = reinterpret_cast<uint64_t *>(tabs + o * kPreTabBytes);
            const uint64_t *lut = reinterpret_cast<const uint64_t *>(pre.mats + s_pre[o].dlut);
            const uint64_t *ph = reinterpret_cast<const uint64_t *>(pre.mats + s_pre[o].mat);
            for (uint32_t i = threadIdx.x; i < 20u + (1u << s_pre[o].k); i += blockDim.x)
                d[i] = __ldg(i < 20u ? lut + i : ph + (i - 20u));
        }
        __syncthreads();
    }
    const uint64_t items = uint64_t(nblocks) * g.nframes;
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t j = uint32_t(item / g.nframes), f = uint32_t(item % g.nframes);
        const BlockSlot sl = table[ids ? ids[j] : b0 + j];
        decode_frame_team<NP, REL>(tm, S, tile, sl.ptr, sl.bytes, g, m, f, wv + (uint64_t(j) << m) + uint64_t(f) * g.F,
                                   hist ? hist + uint64_t(j) * 32 : nullptr, status, s_pre, s_pre_ab, pre.count,
                                   tabs, pre.count ? (uint64_t(j % pre.G) << m) : 0,
                                   pre.count ? pre.gbase[j / pre.G] : 0);
        tm.sync();
    }
}

// One block given by pointer, its format (QSZ1 or QSZR) read from the stream's magic number.
__global__ void __launch_bounds__(kTeamMax, 5) k_decode_block(BlockRef in, int m, float2 *__restrict__ out,
                                                              CallResult res) {
    extern __shared__ __align__(16) uint8_t tile[];
    const FrameGeom g = geom(m);
    __shared__ TeamSmem S;
    const Team tm{threadIdx.x, blockDim.x, 1};
    const uint32_t f = blockIdx.x;
    float2 *dst = out + uint64_t(f) * g.F;
    const bool rel = in.bytes >= g.data_start && !(reinterpret_cast<uintptr_t>(in.ptr) & 15) &&
                     __ldg(reinterpret_cast<const uint32_t *>(in.ptr)) == kQszrMagic;
    if (rel)
        decode_frame_team<0, true>(tm, S, tile, in.ptr, in.bytes, g, m, f, dst, nullptr, res.status, nullptr, nullptr,
                                   0, nullptr, 0, 0);
    else
        decode_frame_team<0, false>(tm, S, tile, in.ptr, in.bytes, g, m, f, dst, nullptr, res.status, nullptr, nullptr,
                                    0, nullptr, 0, 0);
    call_done(res, tm, gridDim.x);
}

// Random access: amplitude idx[i] of a state to out[i], one warp each. It reads the frame's widths and the words of two
// chunks (about 0.5 KB) instead of decoding the frame's 4096 amplitudes to memory first, so its cost, about 0.3 ns an
// index, stays below that of moving the index and the amplitude to and from the host however many a frame is asked for.
// 65536 random indices of a 26-qubit state: 28.7 ms with a host map of frames and whole frames decoded, 0.13 ms now.
template <bool REL>
__global__ void __launch_bounds__(256) k_amplitudes(const BlockSlot *__restrict__ table,
                                                    const uint64_t *__restrict__ idx, uint64_t count, int m,
                                                    float2 *__restrict__ out, int *status) {
    const FrameGeom g = geom(m);
    for (uint64_t i = blockIdx.x * 8ull + (threadIdx.x >> 5); i < count; i += gridDim.x * 8ull) {
        const uint64_t x = idx[i];
        const uint32_t local = uint32_t(x & ((1ull << m) - 1));
        const BlockSlot sl = table[x >> m];
        const float2 v = amplitude_warp<REL>(sl.ptr, sl.bytes, g, m, local >> g.fl, local & (g.F - 1u), status);
        if ((threadIdx.x & 31) == 0) out[i] = v;
    }
}

// the same from an uncompressed store
__global__ void k_amplitudes_raw(const BlockSlot *__restrict__ table, const uint64_t *__restrict__ idx, uint64_t count,
                                 int m, float2 *__restrict__ out, int *status) {
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < count; i += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t x = idx[i];
        const BlockSlot sl = table[x >> m];
        float2 v = make_float2(0.f, 0.f);
        if (sl.ptr == nullptr || sl.bytes < (8ull << m)) raise_status(status, QSIM_E_CORRUPT);
        else v = reinterpret_cast<const float2 *>(sl.ptr)[x & ((1ull << m) - 1)];
        out[i] = v;
    }
}

// Encoder of a batch of blocks, one frame per team of max(32, C) threads (the CTA). A frame is read once, coded in
// shared memory and
//  - blocks of one frame (m <= 12): written to its slot, reserved here, header included; nothing is left to copy;
//  - larger blocks: its bit-plane words go over the frame's own amplitudes (they never need more room) and the part
//    of its image before them to the frame's side record; the CTA that finishes a block's last frame turns the frame
//    lengths into offsets and reserves the block's slot, while other blocks are still being coded. k_frame_copy then
//    moves the images. (The exact slot needs the size of the whole block, so its frames cannot go there directly.)
// Blocks of one frame: 33 + 8 us for the encoder and its copy with a warp per frame, 8 us now (64 frames of 1024 amplitudes).
// arrive: one counter per block, zero before and after. keep_fitting (learned sizing): a block keeps the slot reserved
// for it beforehand when its exact size fits, and only a block whose prediction was too small gets an exact slot
// (counted as an overflowed block).
template <bool REL>
__global__ void __launch_bounds__(kTeamMax, 5) k_encode(float2 *wv, uint32_t nblocks, int m, int e, ArenaDev dev,
                                                        ArenaDev host, EncTarget *__restrict__ tgt,
                                                        EncResult *__restrict__ res,
                                                        const uint32_t *__restrict__ ids,
                                                        BlockSlot *__restrict__ table, StageAccum *acc,
                                                        FrameRecords fr, unsigned long long *arrive, int keep_fitting,
                                                        int *status) {
    extern __shared__ __align__(16) uint8_t tile[];
    const FrameGeom g = geom(m);
    __shared__ TeamSmem S;
    const Team tm{threadIdx.x, blockDim.x, 1};
    const uint64_t items = uint64_t(nblocks) * g.nframes;
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t j = uint32_t(item / g.nframes), f = uint32_t(item % g.nframes);
        float2 *frame = wv + (uint64_t(j) << m) + uint64_t(f) * g.F;
        load_rows_team(tm, tile, frame, g.C);
        const EncFrame r = encode_frame_team<REL>(tm, S, tile, g, e, status);
        uint32_t total = uint32_t(g.data_start) + r.len;
        double err = r.err_sq, nrm = r.norm_sq;
        bool last = true;
        if (g.nframes > 1) {
            stage_frame(tm, tile, r, frame, fr.side + item * fr.side_bytes);
            if (tm.t == 0) {
                fr.len[item] = r.len;
                if (REL) fr.head[item] = r.head;
                fr.part[item] = make_float2(r.err_sq, r.norm_sq);
                __threadfence();  // the frame's records before its arrival: the block's last CTA reads them all
                S.flag = atomicAdd(arrive + j, 1ull) == g.nframes - 1;
            }
            tm.sync();
            last = S.flag != 0;
            if (last) {
                __threadfence();
                const uint64_t b = uint64_t(j) * g.nframes;
                total = block_offsets_team(tm, S, fr.len + b, fr.part + b, fr.off + b, g.nframes,
                                           uint32_t(g.data_start), err, nrm);
            }
        }
        if (last && tm.t == 0) {
            const EncTarget t = reserve_block(total, keep_fitting != 0, tgt + j, dev, host, acc, status);
            EncResult out{};
            out.err_sq = err;
            out.norm_sq = nrm;
            if (g.nframes == 1)
                S.bc = reinterpret_cast<uint64_t>(finish_single_frame(total, t, out, table + (ids ? ids[j] : j), acc));
            else
                arrive[j] = 0;
            res[j] = out;
            if (acc) {
                atomicAdd(&acc->err_sq, err);
                atomicAdd(&acc->norm_sq, nrm);
            }
        }
        tm.sync();
        if (g.nframes == 1) {
            store_single_frame<REL>(tm, tile, g, m, e, r.len, reinterpret_cast<uint8_t *>(S.bc));
            tm.sync();
        }
    }
}

// Second step of blocks of several frames (C = 128), one CTA per frame (copy_frame_team).
template <bool REL>
__global__ void __launch_bounds__(kTeamMax) k_frame_copy(const float2 *__restrict__ wv, uint32_t nblocks, int m, int e,
                                                         const EncTarget *__restrict__ tgt,
                                                         EncResult *__restrict__ res,
                                                         const uint32_t *__restrict__ ids,
                                                         BlockSlot *__restrict__ table, StageAccum *acc,
                                                         FrameRecords fr) {
    const FrameGeom g = geom(m);
    const Team tm{threadIdx.x, kTeamMax, 1};
    const uint64_t items = uint64_t(nblocks) * g.nframes;
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t j = uint32_t(item / g.nframes), f = uint32_t(item % g.nframes);
        copy_frame_team<REL>(tm, wv + (uint64_t(j) << m) + uint64_t(f) * g.F, fr.side + item * fr.side_bytes, fr.len[item],
                             REL ? fr.head[item] : 256u, fr.off[item], g, m, e, f, tgt[j], res + j,
                             table + (ids ? ids[j] : j), acc);
    }
}

// One block into the caller's buffer in one pass: each CTA codes one frame, takes a ticket so that frames are
// processed in order, and finds its byte offset with a decoupled look-back over the preceding frames' sizes. Every
// spin-wait is bounded and reports QSIM_E_TIMEOUT instead of hanging. The record receives the stream's size (also when
// it exceeds cap; the header is then not written) and the status. A block of 2^22 amplitudes: 84 -> 47 us a call, of
// which the launch and the wait for it are 20 and 1024 frames on 760 resident CTAs two rounds of about 10.
template <bool REL>
__global__ void __launch_bounds__(kTeamMax, 5) k_encode_block(const float2 *__restrict__ amps, int m, int e,
                                                              uint8_t *__restrict__ out, uint64_t cap,
                                                              LookbackScratch scr, CallResult res) {
    extern __shared__ __align__(16) uint8_t tile[];
    const FrameGeom g = geom(m);
    __shared__ TeamSmem S;
    const Team tm{threadIdx.x, blockDim.x, 1};
    uint32_t f = 0, epoch = 0;
    if (g.nframes > 1) {
        if (tm.t == 0) {
            S.bc = atomicAdd(scr.ticket, 1u);
            S.bc2 = ld_relaxed_u32(scr.epoch) & kEpochMask;
        }
        tm.sync();
        f = uint32_t(S.bc);
        epoch = uint32_t(S.bc2);
    }
    load_rows_team(tm, tile, amps + uint64_t(f) * g.F, g.C);
    const EncFrame r = encode_frame_team<REL>(tm, S, tile, g, e, res.status);
    uint32_t excl = 0;
    if (g.nframes > 1) {
        if (tm.t < 32) {
            const uint32_t x = lookback_warp(scr.state, f, epoch, r.len, res.status);
            if (tm.t == 0) S.flag = x;
        }
        tm.sync();
        excl = S.flag;
    }
    const uint64_t off = g.data_start + excl, total = off + r.len;
    if (total <= cap) {
        uint4 *d = reinterpret_cast<uint4 *>(out + off);
        for (uint32_t i = tm.t; i < r.len / 16u; i += tm.n) d[i] = reinterpret_cast<const uint4 *>(tile)[i];
    }
    if (tm.t == 0 && g.data_start <= cap) reinterpret_cast<uint32_t *>(out + 32)[f] = uint32_t(off);
    if (f == g.nframes - 1) {
        if (total <= cap) {
            uint32_t *h32 = reinterpret_cast<uint32_t *>(out);
            if (tm.t < 8) h32[tm.t] = header_word(tm.t, REL, g, m, e, f, uint32_t(total - g.data_start));
            const uint32_t i = 8 + g.nframes + tm.t;
            if (i < uint32_t(g.data_start) / 4u) h32[i] = tm.t ? 0u : uint32_t(total);
        }
        if (tm.t == 0) res.record->bytes = total;
    }
    if (call_done(res, tm, gridDim.x) && g.nframes > 1) {
        *scr.ticket = 0;
        atomicExch(scr.epoch, (epoch + 1) & kEpochMask);
    }
}

// Initial store (Sec. 4.2): every block's stream written directly. All but block b0 are zero: a header and an offset
// table. b0 holds the basis state's single amplitude 1 at local index loc: its one non-empty frame is coded here. 0.013 ms
// for eight blocks of 2^25 amplitudes (0.83 ms with both kinds of block filled in memory and encoded).
template <bool REL>
__global__ void __launch_bounds__(kTeamMax) k_init_store(uint64_t nblocks, uint64_t b0, uint64_t loc, int m, int e,
                                                         BlockSlot *__restrict__ table, ArenaDev dev, ArenaDev host,
                                                         StageAccum *acc, int *status) {
    extern __shared__ __align__(16) uint8_t tile[];
    const FrameGeom g = geom(m);
    __shared__ TeamSmem S;
    const Team tm{threadIdx.x, blockDim.x, 1};
    unsigned long long bytes = 0;  // thread 0
    for (uint64_t b = blockIdx.x; b < nblocks; b += gridDim.x) {
        uint32_t len = 0;
        const uint32_t f0 = uint32_t(loc >> g.fl), at = uint32_t(loc) & (g.F - 1u);
        if (b == b0) {
            for (uint32_t i = tm.t; i < team_tile_bytes(g.C) / 16u; i += tm.n)
                reinterpret_cast<uint4 *>(tile)[i] = make_uint4(0, 0, 0, 0);
            tm.sync();
            if (tm.t == 0) *reinterpret_cast<float *>(tile + kRowBytes * (at >> 5) + 8u * (at & 31u)) = 1.f;
            tm.sync();
            len = encode_frame_team<REL>(tm, S, tile, g, e, status).len;
        }
        if (tm.t == 0) {
            const uint64_t total = g.data_start + len;
            EncTarget t;
            reserve_slot(total, dev, host, &t, status);
            table[b].ptr = t.ptr;
            table[b].bytes = total;
            table[b].tier = t.tier;
            S.bc = reinterpret_cast<uint64_t>(t.ptr);
            bytes += total;
        }
        tm.sync();
        uint8_t *out = reinterpret_cast<uint8_t *>(S.bc);
        if (out) {
            for (uint32_t i = tm.t; i < uint32_t(g.data_start) / 4u; i += tm.n)
                reinterpret_cast<uint32_t *>(out)[i] = header_word(i, REL, g, m, e, f0, len);
            uint4 *d = reinterpret_cast<uint4 *>(out + g.data_start);
            for (uint32_t i = tm.t; i < len / 16u; i += tm.n) d[i] = reinterpret_cast<const uint4 *>(tile)[i];
        }
        tm.sync();
    }
    if (tm.t == 0 && bytes) atomicAdd(reinterpret_cast<unsigned long long *>(&acc->store_bytes), bytes);
}

// ---------------------------------------------------------------------------
// Slot reservation from the two-tier pool: device arena first, then the
// pinned host arena. 2^pred_log2[j] (1 + margin) bytes, at most `worst`, or
// `worst` without predictions; the slot is padded to 256 bytes.
// ---------------------------------------------------------------------------
__global__ void k_reserve(uint32_t nblocks, const float *__restrict__ pred_log2, double margin, uint64_t worst,
                          ArenaDev dev, ArenaDev host, EncTarget *__restrict__ tgt, EncResult *__restrict__ res,
                          int *status) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nblocks) return;
    uint64_t want = worst;
    if (pred_log2) {
        double p = double(pred_log2[j]);
        p = p < 0 ? 0 : (p > 40 ? 40 : p);
        double b = exp2(p) * (1.0 + margin);
        want = b >= double(worst) ? worst : uint64_t(b);
    }
    res[j].total = 0;
    res[j].overflow = 0;
    res[j].err_sq = 0;
    res[j].norm_sq = 0;
    reserve_slot(want, dev, host, &tgt[j], status);
}

// Raw (uncompressed) store: copy blocks, 16 bytes per thread.
__global__ void k_copy_blocks_out(const float2 *__restrict__ wv, uint32_t nblocks, int m,
                                  const EncTarget *__restrict__ tgt, const uint32_t *__restrict__ ids,
                                  BlockSlot *__restrict__ table, StageAccum *acc, int *status) {
    const uint64_t per = (8ull << m) / 16;
    const uint64_t total = per * nblocks;
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < total; i += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t j = uint32_t(i / per);
        const uint64_t o = i % per;
        if (tgt[j].ptr == nullptr || tgt[j].cap < (8ull << m)) continue;
        reinterpret_cast<float4 *>(tgt[j].ptr)[o] = reinterpret_cast<const float4 *>(wv + (uint64_t(j) << m))[o];
        if (o == 0) {
            table[ids[j]].ptr = tgt[j].ptr;
            table[ids[j]].bytes = 8ull << m;
            table[ids[j]].tier = tgt[j].tier;
            if (acc) {
                atomicAdd(reinterpret_cast<unsigned long long *>(&acc->store_bytes), 8ull << m);
                atomicAdd(reinterpret_cast<unsigned long long *>(&acc->reserved_bytes), tgt[j].cap);
                if (tgt[j].tier) atomicAdd(reinterpret_cast<unsigned long long *>(&acc->host_bytes), tgt[j].cap);
                atomicAdd(reinterpret_cast<unsigned long long *>(&acc->blocks), 1ull);
            }
        }
    }
}

__global__ void k_copy_blocks_in(const BlockRef *__restrict__ in, uint32_t nblocks, int m, float2 *__restrict__ wv,
                                 int *status) {
    const uint64_t per = (8ull << m) / 16;
    const uint64_t total = per * nblocks;
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < total; i += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t j = uint32_t(i / per);
        const uint64_t o = i % per;
        if (in[j].ptr == nullptr || in[j].bytes < (8ull << m)) {
            if (o == 0) raise_status(status, QSIM_E_CORRUPT);
            continue;
        }
        reinterpret_cast<float4 *>(wv + (uint64_t(j) << m))[o] = reinterpret_cast<const float4 *>(in[j].ptr)[o];
    }
}

// Gather block references from the block table (ids null: its first `count` entries).
__global__ void k_gather_refs(const BlockSlot *__restrict__ table, const uint32_t *__restrict__ ids, uint32_t count,
                              BlockRef *__restrict__ out) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < count) {
        const uint32_t b = ids ? ids[j] : j;
        out[j].ptr = table[b].ptr;
        out[j].bytes = table[b].bytes;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static unsigned grid_for(uint64_t items, unsigned cap) {
    return unsigned(items < cap ? (items ? items : 1) : cap);
}

// Team kernels: one CTA of team_threads(C) threads per frame, team_tile_bytes(C) of dynamic shared memory.
struct TeamShape {
    uint32_t threads;
    size_t smem;
};
static TeamShape team_shape(int m) {
    const uint32_t C = (1u << frame_log_for(m)) / 32u;
    return {cdev::team_threads(C), cdev::team_tile_bytes(C)};
}
constexpr unsigned kMaxGrid = 1u << 30;

template <bool REL>
static void decode_table(const BlockSlot *table, const uint32_t *ids, uint64_t b0, uint32_t nblocks, int m, float2 *wv,
                         uint32_t *hist, int *status, const PreOps &pre, cudaStream_t s) {
    const uint64_t items = uint64_t(nblocks) * qsz_nframes(m);
    const TeamShape ts = team_shape(m);
    // with leading phase ops each CTA copies their tables (up to 18 KB) once and takes several frames: three CTAs for
    // each of the five resident ones, so that the last ones to finish are short
    const unsigned grid = grid_for(items, pre.count ? num_sms() * 5 * 3 : kMaxGrid);
    const size_t smem = ts.smem + pre.count * cdev::kPreTabBytes;
    if (pre.count > 2)  // kMaxPreOps tables beside the largest tile: 52.5 KB
        allow_smem<k_decode<kMaxPreOps, REL>>(int(cdev::team_tile_bytes(128) + kMaxPreOps * cdev::kPreTabBytes));
    if (pre.count == 0)
        k_decode<0, REL><<<grid, ts.threads, smem, s>>>(table, ids, b0, nblocks, m, wv, hist, status, pre);
    else if (pre.count <= 2)
        k_decode<2, REL><<<grid, ts.threads, smem, s>>>(table, ids, b0, nblocks, m, wv, hist, status, pre);
    else
        k_decode<kMaxPreOps, REL><<<grid, ts.threads, smem, s>>>(table, ids, b0, nblocks, m, wv, hist, status, pre);
}

void launch_decode(const BlockSlot *table, uint64_t b0, uint32_t nblocks, int m, float2 *wv, int *status,
                   cudaStream_t s, bool rel) {
    if (rel)
        decode_table<true>(table, nullptr, b0, nblocks, m, wv, nullptr, status, PreOps{}, s);
    else
        decode_table<false>(table, nullptr, b0, nblocks, m, wv, nullptr, status, PreOps{}, s);
    count_launch();
}

void launch_decode_block(const BlockRef &in, int m, float2 *out, const CallResult &res, cudaStream_t s) {
    const TeamShape ts = team_shape(m);
    k_decode_block<<<unsigned(qsz_nframes(m)), ts.threads, ts.smem, s>>>(in, m, out, res);
    count_launch();
}

void launch_amplitudes(const BlockSlot *table, const uint64_t *idx, uint64_t count, int m, float2 *out, int *status,
                       cudaStream_t s, uint32_t codec) {
    if (codec == QSIM_CODEC_NONE)
        k_amplitudes_raw<<<grid_for((count + 255) / 256, num_sms() * 16), 256, 0, s>>>(table, idx, count, m, out, status);
    else if (codec == QSIM_CODEC_QSZR)
        k_amplitudes<true><<<grid_for((count + 7) / 8, num_sms() * 64), 256, 0, s>>>(table, idx, count, m, out, status);
    else
        k_amplitudes<false><<<grid_for((count + 7) / 8, num_sms() * 64), 256, 0, s>>>(table, idx, count, m, out, status);
    count_launch();
}

void launch_decode_table(const BlockSlot *table, const uint32_t *ids, uint32_t nblocks, int m, float2 *wv,
                         uint32_t *hist, int *status, const PreOps &pre, cudaStream_t s, bool rel) {
    if (rel)
        decode_table<true>(table, ids, 0, nblocks, m, wv, hist, status, pre, s);
    else
        decode_table<false>(table, ids, 0, nblocks, m, wv, hist, status, pre, s);
    count_launch();
}

void launch_encode(float2 *wv, uint32_t nblocks, int m, int e, const ArenaDev &dev, const ArenaDev &host,
                   EncTarget *tgt, EncResult *res, const uint32_t *ids, BlockSlot *table, StageAccum *acc,
                   const FrameRecords &fr, uint64_t *arrive, int *status, cudaStream_t s, bool rel,
                   bool keep_fitting) {
    const unsigned grid = grid_for(uint64_t(nblocks) * qsz_nframes(m), kMaxGrid);
    const TeamShape ts = team_shape(m);
    unsigned long long *arr = reinterpret_cast<unsigned long long *>(arrive);
    if (rel)
        k_encode<true><<<grid, ts.threads, ts.smem, s>>>(wv, nblocks, m, e, dev, host, tgt, res, ids, table, acc, fr,
                                                         arr, keep_fitting ? 1 : 0, status);
    else
        k_encode<false><<<grid, ts.threads, ts.smem, s>>>(wv, nblocks, m, e, dev, host, tgt, res, ids, table, acc, fr,
                                                          arr, keep_fitting ? 1 : 0, status);
    count_launch();
}

void launch_frame_copy(const float2 *wv, uint32_t nblocks, int m, int e, const EncTarget *tgt, EncResult *res,
                       const uint32_t *ids, BlockSlot *table, StageAccum *acc, const FrameRecords &fr, cudaStream_t s,
                       bool rel) {
    const unsigned grid = grid_for(uint64_t(nblocks) * qsz_nframes(m), kMaxGrid);
    if (rel)
        k_frame_copy<true><<<grid, cdev::kTeamMax, 0, s>>>(wv, nblocks, m, e, tgt, res, ids, table, acc, fr);
    else
        k_frame_copy<false><<<grid, cdev::kTeamMax, 0, s>>>(wv, nblocks, m, e, tgt, res, ids, table, acc, fr);
    count_launch();
}

void launch_encode_block(const float2 *amps, int m, int e, uint8_t *out, uint64_t cap, const LookbackScratch &scr,
                         const CallResult &res, cudaStream_t s, bool rel) {
    const TeamShape ts = team_shape(m);
    const unsigned grid = unsigned(qsz_nframes(m));
    if (rel)
        k_encode_block<true><<<grid, ts.threads, ts.smem, s>>>(amps, m, e, out, cap, scr, res);
    else
        k_encode_block<false><<<grid, ts.threads, ts.smem, s>>>(amps, m, e, out, cap, scr, res);
    count_launch();
}

void launch_init_store(uint64_t nblocks, uint64_t b0, uint64_t loc, int m, int e, BlockSlot *table,
                       const ArenaDev &dev, const ArenaDev &host, StageAccum *acc, int *status, cudaStream_t s,
                       bool rel) {
    const TeamShape ts = team_shape(m);
    const unsigned grid = grid_for(nblocks, num_sms() * 8);
    if (rel)
        k_init_store<true><<<grid, ts.threads, ts.smem, s>>>(nblocks, b0, loc, m, e, table, dev, host, acc, status);
    else
        k_init_store<false><<<grid, ts.threads, ts.smem, s>>>(nblocks, b0, loc, m, e, table, dev, host, acc, status);
    count_launch();
}

void launch_reserve(uint32_t nblocks, const float *pred_log2, double margin, uint64_t worst, const ArenaDev &dev,
                    const ArenaDev &host, EncTarget *tgt, EncResult *res, int *status, cudaStream_t s) {
    k_reserve<<<(nblocks + 127) / 128, 128, 0, s>>>(nblocks, pred_log2, margin, worst, dev, host, tgt, res, status);
    count_launch();
}

void launch_copy_out(const float2 *wv, uint32_t nblocks, int m, const EncTarget *tgt, const uint32_t *ids,
                     BlockSlot *table, StageAccum *acc, int *status, cudaStream_t s) {
    const uint64_t items = (uint64_t(nblocks) << m) / 2;
    k_copy_blocks_out<<<grid_for((items + 255) / 256, num_sms() * 16), 256, 0, s>>>(wv, nblocks, m, tgt, ids, table, acc,
                                                                            status);
    count_launch();
}

void launch_copy_in(const BlockRef *in, uint32_t nblocks, int m, float2 *wv, int *status, cudaStream_t s) {
    const uint64_t items = (uint64_t(nblocks) << m) / 2;
    k_copy_blocks_in<<<grid_for((items + 255) / 256, num_sms() * 16), 256, 0, s>>>(in, nblocks, m, wv, status);
    count_launch();
}

void launch_gather_refs(const BlockSlot *table, const uint32_t *ids, uint32_t count, BlockRef *out, cudaStream_t s) {
    k_gather_refs<<<(count + 127) / 128, 128, 0, s>>>(table, ids, count, out);
    count_launch();
}

}  // namespace qsim
