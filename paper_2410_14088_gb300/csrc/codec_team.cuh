// Frame coder of the QSZ1 / QSZR block codec, one thread per chunk pair.
//
// A team of max(32, C) threads (C = chunks per plane of the frame, 128 in frames of 4096 amplitudes) codes one frame
// staged in shared memory; thread t owns Re chunk t and Im chunk t, 32 values each, in registers. The 32 x 32 bit
// transpose between codes and bit planes is then a register transpose of one thread (256 byte-permute, shift and
// select instructions for a chunk pair whose codes fit 16 bits), the Lorenzo difference and its inverse are one add
// per value, a chunk's width is one count-leading-zeros of the OR of its codes, and the team meets only for the one
// scan that turns the chunks' widths into word offsets. A warp-per-frame coder spends 5-step shuffle networks on each
// of those (transpose, prefix sums, width votes) and walks its 128 chunk pairs one after the other.
//
// What bounds it: instruction issue and shared memory (the frame passes through shared memory once each way, plus its
// words), close to the HBM time of the frame. Per 32-value chunk pair 49 warp instructions decode and 56 encode, against
// 143 and 115 with a warp per frame; launches of 4096 dense frames (2^24 amplitudes) take 39 us instead of 155 and 46
// instead of 133, 2^28 amplitudes of early frames 0.30 ms to decode (7.0 TB/s) and 0.57 ms to encode (4.9 TB/s; 1.26 before).
//
// Layout: chunk t's amplitudes at byte 272 t of the tile (256 bytes and 16 of padding): a thread walks its row 16
// bytes at a time and eight threads' rows fall on all 32 banks, and rows are read and written coalesced. The frame's
// compressed image (at most 272 C + 64 bytes) takes the same memory before the decoder writes the rows and after the
// encoder has read them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "codec.cuh"
#include "codec_dev.cuh"
#include "device_common.cuh"

namespace qsim {
namespace cdev {

constexpr uint32_t kRowBytes = 272;
constexpr uint32_t kTeamMax = 128;
// Tile bytes of a frame of C chunks per plane. The largest QSZR image, 256 C + pad16(2C) + pad16(C/2) + pad16(8C),
// is at most 272 C + 64 for every C = 1, 2, 4, ..., 128 (the QSZ1 image lacks the last two terms).
__host__ __device__ constexpr uint32_t team_tile_bytes(uint32_t C) { return kRowBytes * C + 64u; }
__host__ __device__ constexpr uint32_t team_threads(uint32_t C) { return C < 32u ? 32u : C; }

// small shared memory of a team
struct TeamSmem {
    uint32_t w[4], s[4], x[4];  // per warp: width sums, sign-section counts, largest width
    float err[4], nrm[4];
    double da[4], db[4];
    uint64_t bc, bc2;           // broadcast from thread 0
    uint32_t flag;
    uint32_t hist[32];
};

// n threads (a multiple of 32, numbered t) meeting on hardware barrier `bar` (1 to 4; unused by a team of one warp)
struct Team {
    uint32_t t, n, bar;
    __device__ __forceinline__ void sync() const {
        // barrier ids 1 to 4 as constants: an id in a register would reserve all sixteen for the CTA
        if (n == 32u) __syncwarp();
        else if (bar == 1u) asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
        else if (bar == 2u) asm volatile("bar.sync 2, %0;" ::"r"(n) : "memory");
        else if (bar == 3u) asm volatile("bar.sync 3, %0;" ::"r"(n) : "memory");
        else asm volatile("bar.sync 4, %0;" ::"r"(n) : "memory");
    }
};

__device__ __forceinline__ void team_cp16(void *smem, const void *gmem) {
    const uint32_t sa = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void team_cp_wait() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Transpose the 32 x 32 bit matrix in v (row r = v[r], column = bit): block swaps of 16, 8, 4, 2 and 1 rows, the
// first two as byte permutes.
__device__ __forceinline__ void transpose32(uint32_t (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const uint32_t a = v[i], b = v[i + 16];
        v[i] = __byte_perm(a, b, 0x5410);
        v[i + 16] = __byte_perm(a, b, 0x7632);
    }
#pragma unroll
    for (int k = 0; k < 32; k += 16)
#pragma unroll
        for (int i = k; i < k + 8; ++i) {
            const uint32_t a = v[i], b = v[i + 8];
            v[i] = __byte_perm(a, b, 0x6240);
            v[i + 8] = __byte_perm(a, b, 0x7351);
        }
#pragma unroll
    for (int s = 4; s >= 1; s >>= 1) {
        const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int k = 0; k < 32; k += 2 * s)
#pragma unroll
            for (int i = k; i < k + s; ++i) {
                const uint32_t a = v[i], b = v[i + s];
                v[i] = (a & m) | ((b << s) & ~m);
                v[i + s] = ((a >> s) & m) | (b & ~m);
            }
    }
}

// 1.5 * 2^23: adding it to |y| < 2^22 rounds y to the nearest integer (ties to even, as __float2int_rn), which then
// sits in the low mantissa bits; subtracting it (scaled) gives the value back exactly
constexpr float kRound = 12582912.0f;
constexpr int32_t kRoundBits = 0x4B400000;

// End of a single-block call's CTA: the last one to arrive reports the launch's status in the call's record and leaves
// the device words zero for the next call (calls on one context do not overlap). True in that CTA's thread 0.
__device__ __forceinline__ bool call_done(const CallResult &res, const Team &tm, uint32_t nctas) {
    tm.sync();  // every thread's raise_status came before
    if (tm.t != 0) return false;
    if (nctas > 1) {  // a call of one frame has nobody to wait for
        __threadfence();
        if (atomicAdd(res.done, 1u) != nctas - 1) return false;
        __threadfence();
        *res.done = 0;
    }
    res.record->status = atomicExch(res.status, 0);
    __threadfence_system();
    return true;
}

// ---------------------------------------------------------------------------
// decode
// ---------------------------------------------------------------------------
struct FrameHead {
    bool ok;          // the stream's header and frame f's offsets are consistent
    uint32_t fa, fb;  // frame f's image in the stream
    int e;            // step exponent (QSZ1) or code shift (QSZR)
};

// Header and offsets of frame f of a stream, read and checked by a whole warp, one load per lane.
template <bool REL>
__device__ __forceinline__ FrameHead frame_head(const uint8_t *sp, uint64_t bytes, const FrameGeom &g, int m, uint32_t f) {
    const uint32_t lane = threadIdx.x & 31u, C = g.C;
    const uint32_t padw = (2u * C + 15u) & ~15u;
    const uint32_t tbp = REL ? ((((2u * C + 3u) / 4u) + 15u) & ~15u) : 0u;  // sign chunk types, padded
    const bool can = sp != nullptr && !(reinterpret_cast<uintptr_t>(sp) & 15) && bytes >= g.data_start;
    uint32_t hv = 0;
    if (can) {
        const uint32_t *h32 = reinterpret_cast<const uint32_t *>(sp);
        if (lane < 8) hv = h32[lane];
        else if (lane == 8) hv = h32[8];               // offsets[0]
        else if (lane == 9) hv = h32[8 + f];           // offsets[f]
        else if (lane == 10) hv = h32[8 + f + 1];      // offsets[f+1]
        else if (lane == 11) hv = h32[8 + g.nframes];  // offsets[nframes]
    }
    const uint32_t magic = __shfl_sync(kFull, hv, 0), w1 = __shfl_sync(kFull, hv, 1);
    const uint32_t w2 = __shfl_sync(kFull, hv, 2), nfr = __shfl_sync(kFull, hv, 3);
    const uint64_t total = uint64_t(__shfl_sync(kFull, hv, 4)) | (uint64_t(__shfl_sync(kFull, hv, 5)) << 32);
    const uint64_t rsv = uint64_t(__shfl_sync(kFull, hv, 6)) | (uint64_t(__shfl_sync(kFull, hv, 7)) << 32);
    const uint32_t o0 = __shfl_sync(kFull, hv, 8), on = __shfl_sync(kFull, hv, 11);
    FrameHead r;
    r.fa = __shfl_sync(kFull, hv, 9);
    r.fb = __shfl_sync(kFull, hv, 10);
    r.e = REL ? int(uint8_t(w2 >> 16)) : int(int8_t(uint8_t(w2 >> 16)));
    r.ok = can && magic == (REL ? kQszrMagic : kQszMagic) && w1 == 1u && (w2 & 0xff) == uint32_t(m) &&
           ((w2 >> 8) & 0xff) == uint32_t(g.fl) && (w2 >> 24) == 0 && nfr == g.nframes && rsv == 0 &&
           (REL ? (r.e >= kQszrKMin && r.e <= kQszrKMax) : (r.e >= kQszEMin && r.e <= kQszEMax)) && total <= bytes &&
           total >= g.data_start && o0 == g.data_start && on == total && r.fb >= r.fa && r.fb <= total &&
           r.fa >= g.data_start && !((r.fa | r.fb) & 15u) &&
           (r.fb == r.fa || (r.fb - r.fa >= padw + tbp && r.fb - r.fa <= team_tile_bytes(C)));
    return r;
}

// The amplitude at index `at` of frame f of one block, decoded by a whole warp from the two chunks that hold it: the
// widths are read 8 per lane and scanned for the chunks' words, each plane's words go through one transpose, and the
// codes up to the index are summed. Every lane returns the amplitude.
template <bool REL>
__device__ __forceinline__ float2 amplitude_warp(const uint8_t *sp, uint64_t bytes, const FrameGeom &g, int m,
                                                 uint32_t f, uint32_t at, int *status) {
    const uint32_t lane = threadIdx.x & 31u, C = g.C, c = at >> 5, l = at & 31u;
    const uint32_t padw = (2u * C + 15u) & ~15u;
    const uint32_t tbp = REL ? ((((2u * C + 3u) / 4u) + 15u) & ~15u) : 0u;
    const FrameHead fh = frame_head<REL>(sp, bytes, g, m, f);
    bool ok = fh.ok;
    const uint32_t flen = ok ? fh.fb - fh.fa : 0u;
    if (ok && !flen) return make_float2(0.f, 0.f);
    const uint8_t *img = sp + fh.fa;
    uint64_t wb = 0;  // widths 8 lane .. 8 lane + 7 (bytes past 2C are zero padding)
    if (ok && 8u * lane < 2u * C) wb = *reinterpret_cast<const uint64_t *>(img + 8u * lane);
    uint32_t sum = 0, mx = 0;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
        const uint32_t w = uint32_t(wb >> (8u * k)) & 0xffu;
        sum += w;
        mx = max(mx, w);
    }
    uint32_t tw = 0, cnt = 0;  // REL: sign chunk types 16 lane .. 16 lane + 15; stored words | run records << 16
    if constexpr (REL) {
        if (ok && 16u * lane < 2u * C) tw = *reinterpret_cast<const uint32_t *>(img + padw + 4u * lane);
        const uint32_t hi = tw & 0xAAAAAAAAu, t3 = hi & (tw << 1);
        cnt = __popc(hi ^ t3) | (__popc(t3) << 16);
    }
    uint32_t incl = sum, icnt = cnt;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(kFull, incl, o);
        const uint32_t b = REL ? __shfl_up_sync(kFull, icnt, o) : 0u;
        if (lane >= o) {
            incl += a;
            icnt += b;
        }
    }
    const uint32_t words = __shfl_sync(kFull, incl, 31), ctot = __shfl_sync(kFull, icnt, 31);
    const uint32_t n2 = ctot & 0xffffu, n3 = ctot >> 16, signs = REL ? (4u * n2 + 2u * n3 + 15u) & ~15u : 0u;
    ok = ok && __reduce_max_sync(kFull, mx) <= 32 && words > 0 &&
         uint64_t(flen) == padw + tbp + signs + ((4ull * words + 15) & ~15ull);
    if (!ok) {
        if (lane == 0) raise_status(status, QSIM_E_CORRUPT);
        return make_float2(0.f, 0.f);
    }
    const uint32_t *pay = reinterpret_cast<const uint32_t *>(img + padw + tbp + signs);
    float v[2];
    bool bad = false;
#pragma unroll
    for (uint32_t p = 0; p < 2; ++p) {
        const uint32_t i = p * C + c;  // the chunk among the frame's 2C
        const uint64_t own = __shfl_sync(kFull, wb, i >> 3);
        uint32_t off = __shfl_sync(kFull, incl - sum, i >> 3);
        for (uint32_t k = 0; k < (i & 7u); ++k) off += uint32_t(own >> (8u * k)) & 0xffu;
        const uint32_t w = uint32_t(own >> (8u * (i & 7u))) & 0xffu;
        const uint32_t z = warp_bit_transpose(lane < w ? __ldg(pay + off + lane) : 0u, int(lane));
        const int32_t q = __reduce_add_sync(kFull, lane <= l ? unzigzag(z) : 0);
        if constexpr (REL) {
            const uint32_t types = __shfl_sync(kFull, tw, i >> 4), s = 2u * (i & 15u);
            const uint32_t before = __shfl_sync(kFull, icnt - cnt, i >> 4), below = (1u << s) - 1u;
            const uint32_t t3 = types & 0xAAAAAAAAu & (types << 1), t2 = (types & 0xAAAAAAAAu) ^ t3;
            const uint32_t ty = (types >> s) & 3u;
            const uint32_t *mixw = reinterpret_cast<const uint32_t *>(img + padw + tbp);
            uint32_t sw = ty == 1u ? 0xFFFFFFFFu : 0u;
            if (ty == 2u) sw = __ldg(mixw + (before & 0xffffu) + __popc(t2 & below));
            if (ty == 3u) {
                bool rok;
                const uint16_t *runw = reinterpret_cast<const uint16_t *>(mixw + n2);
                sw = sign_run_word(__ldg(runw + (before >> 16) + __popc(t3 & below)), rok);
                bad |= !rok;
            }
            bad |= uint32_t(q) > (kQszrMaxU >> fh.e);
            v[p] = __uint_as_float((uint32_t(q) << fh.e) ^ (((sw >> l) & 1u) << 31));
        } else {
            v[p] = float(q) * exp2i(fh.e);
        }
    }
    if (bad && lane == 0) raise_status(status, QSIM_E_CORRUPT);
    return make_float2(v[0], v[1]);
}

// Frame f of one block (stream sp, `bytes` long) into dst (F amplitudes). tile: team_tile_bytes(C), 16-byte aligned.
// hist_j (nullable): the block's code-width histogram. pre_*: leading phase ops, their tables at byte offsets pre_ab of
// tabs. The team may
// reuse tile and S after its next sync().
template <int NP, bool REL>
__device__ __forceinline__ void decode_frame_team(const Team &tm, TeamSmem &S, uint8_t *tile, const uint8_t *sp,
                                                  uint64_t bytes, const FrameGeom &g, int m, uint32_t f,
                                                  float2 *__restrict__ dst, uint32_t *hist_j, int *status,
                                                  const OpDev *pre_ops, const uint2 *pre_ab, uint32_t npre,
                                                  const uint8_t *tabs, uint64_t wbase, uint64_t gb) {
    const uint32_t t = tm.t, lane = t & 31u, warp = t >> 5, nw = tm.n >> 5, C = g.C;
    const uint32_t padw = (2u * C + 15u) & ~15u;
    const uint32_t tbp = REL ? ((((2u * C + 3u) / 4u) + 15u) & ~15u) : 0u;  // sign chunk types, padded
    const FrameHead fh = frame_head<REL>(sp, bytes, g, m, f);  // every warp of the team reads it
    const uint32_t fa = fh.fa;
    const int e = fh.e;
    bool ok = fh.ok;
    const uint32_t flen = ok ? fh.fb - fa : 0u;
    // ---- the frame's image to shared memory ----
    for (uint32_t i = t; i < flen / 16u; i += tm.n) team_cp16(tile + 16u * i, sp + fa + 16u * i);
    team_cp_wait();
    tm.sync();
    const bool act = t < C;
    uint32_t wr = 0, wi = 0, tr = 0, ti = 0, cnt = 0;
    if (flen && act) {
        wr = tile[t];
        wi = tile[C + t];
        if constexpr (REL) {
            const uint32_t i = C + t;
            tr = (tile[padw + (t >> 2)] >> (2u * (t & 3u))) & 3u;
            ti = (tile[padw + (i >> 2)] >> (2u * (i & 3u))) & 3u;
            // stored words Re | Im << 8, run records Re << 16 | Im << 24
            cnt = uint32_t(tr == 2u) | (uint32_t(ti == 2u) << 8) | (uint32_t(tr == 3u) << 16) | (uint32_t(ti == 3u) << 24);
        }
    }
    // ---- word offsets: one scan of (Re width, Im width) over the team (sums below 2^16 even in a corrupt frame) ----
    const uint32_t wp = wr | (wi << 16);
    uint32_t incl = wp, icnt = cnt;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(kFull, incl, o);
        const uint32_t b = REL ? __shfl_up_sync(kFull, icnt, o) : 0u;
        if (lane >= o) {
            incl += a;
            icnt += b;
        }
    }
    const uint32_t mx = __reduce_max_sync(kFull, max(wr, wi));
    if (lane == 31) {
        S.w[warp] = incl;
        S.s[warp] = icnt;
        S.x[warp] = mx;
    }
    if (hist_j && t < 32) S.hist[t] = 0;
    tm.sync();
    uint32_t base = 0, tot = 0, cbase = 0, ctot = 0, maxw = 0;
#pragma unroll
    for (uint32_t w = 0; w < 4; ++w)
        if (w < nw) {
            if (w == warp) {
                base = tot;
                cbase = ctot;
            }
            tot += S.w[w];
            ctot += S.s[w];
            maxw = max(maxw, S.x[w]);
        }
    const uint32_t words = (tot & 0xffffu) + (tot >> 16);
    const uint32_t signs = REL ? sign_section_bytes(ctot) : 0u;
    if (flen) ok = maxw <= 32 && words > 0 && uint64_t(flen) == padw + tbp + signs + ((4ull * words + 15) & ~15ull);
    if (!ok && t == 0) raise_status(status, QSIM_E_CORRUPT);
    const bool wide_dst = !(reinterpret_cast<uintptr_t>(dst) & 15);
    if (!ok || !flen) {  // an all-zero frame (or a corrupt one)
        if (wide_dst) {
            float4 *d4 = reinterpret_cast<float4 *>(dst);
            for (uint32_t i = t; i < 16u * C; i += tm.n) d4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            for (uint32_t i = t; i < 32u * C; i += tm.n) dst[i] = make_float2(0.f, 0.f);
        }
        if (hist_j && t == 0) atomicAdd(&hist_j[0], 2 * g.F);
        return;
    }
    if (hist_j && act) {  // the chunks' code widths, 32 values each
        atomicAdd(&S.hist[min(wr, 31u)], 32u);
        atomicAdd(&S.hist[min(wi, 31u)], 32u);
    }
    base += incl - wp;
    const uint32_t offr = base & 0xffffu, offi = (tot & 0xffffu) + (base >> 16);
    const uint32_t *pay = reinterpret_cast<const uint32_t *>(tile + padw + tbp + signs);
    uint8_t *row = tile + kRowBytes * t;
    const float step = REL ? 0.f : exp2i(e);
    // planes 0..15 of the Re chunk in rows 0..15 and of the Im chunk in rows 16..31: the transposed word j holds both
    // codes' low halves
    uint32_t lo[32];
#pragma unroll
    for (uint32_t b = 0; b < 16; ++b) {
        lo[b] = b < wr ? pay[offr + b] : 0u;
        lo[16 + b] = b < wi ? pay[offi + b] : 0u;
    }
    if (!REL && maxw <= 16u) {
        transpose32(lo);
        tm.sync();  // every word is in registers: the rows take the image's place
        if (act) {
            // |q| <= 32 * 2^15: the running sums start at kRoundBits, so that each one reinterpreted as a float is
            // kRound + q, and one FMA gives q * step exactly
            const float off = -kRound * step;
            int32_t ar = kRoundBits, ai = kRoundBits;
#pragma unroll
            for (uint32_t j = 0; j < 32; j += 2) {
                float4 o;
                ar += unzigzag(lo[j] & 0xffffu);
                ai += unzigzag(lo[j] >> 16);
                o.x = fmaf(__int_as_float(ar), step, off);
                o.y = fmaf(__int_as_float(ai), step, off);
                ar += unzigzag(lo[j + 1] & 0xffffu);
                ai += unzigzag(lo[j + 1] >> 16);
                o.z = fmaf(__int_as_float(ar), step, off);
                o.w = fmaf(__int_as_float(ai), step, off);
                *reinterpret_cast<float4 *>(row + 8u * j) = o;
            }
        }
    } else {
        uint32_t hi[32];  // planes 16..31, laid out like lo
#pragma unroll
        for (uint32_t b = 0; b < 16; ++b) {
            hi[b] = 16u + b < wr ? pay[offr + 16u + b] : 0u;
            hi[16 + b] = 16u + b < wi ? pay[offi + 16u + b] : 0u;
        }
        uint32_t swr = 0, swi = 0;  // REL: sign words of the two chunks
        bool bad = false;
        if constexpr (REL) {
            cbase += icnt - cnt;
            const uint32_t n2 = (ctot & 0xffu) + ((ctot >> 8) & 0xffu), n3r = (ctot >> 16) & 0xffu;
            const uint32_t *mixw = reinterpret_cast<const uint32_t *>(tile + padw + tbp);
            const uint16_t *runw = reinterpret_cast<const uint16_t *>(mixw + n2);
            swr = tr == 1u ? 0xFFFFFFFFu : 0u;
            swi = ti == 1u ? 0xFFFFFFFFu : 0u;
            if (tr == 2u) swr = mixw[cbase & 0xffu];
            if (ti == 2u) swi = mixw[(ctot & 0xffu) + ((cbase >> 8) & 0xffu)];
            bool rok = true;
            if (tr == 3u) {
                swr = sign_run_word(runw[(cbase >> 16) & 0xffu], rok);
                bad |= !rok;
            }
            if (ti == 3u) {
                swi = sign_run_word(runw[n3r + (cbase >> 24)], rok);
                bad |= !rok;
            }
        }
        transpose32(lo);
        transpose32(hi);
        tm.sync();
        if (act) {
            uint32_t qr = 0, qi = 0;
#pragma unroll
            for (uint32_t j = 0; j < 32; j += 2) {
                float v[4];
#pragma unroll
                for (uint32_t k = 0; k < 2; ++k) {
                    const uint32_t l = lo[j + k], h = hi[j + k];
                    qr += uint32_t(unzigzag((l & 0xffffu) | (h << 16)));
                    qi += uint32_t(unzigzag((l >> 16) | (h & 0xffff0000u)));
                    if constexpr (REL) {
                        bad |= qr > (kQszrMaxU >> e) || qi > (kQszrMaxU >> e);
                        v[2 * k] = __uint_as_float((qr << e) ^ (((swr >> (j + k)) & 1u) << 31));
                        v[2 * k + 1] = __uint_as_float((qi << e) ^ (((swi >> (j + k)) & 1u) << 31));
                    } else {
                        v[2 * k] = float(int32_t(qr)) * step;
                        v[2 * k + 1] = float(int32_t(qi)) * step;
                    }
                }
                *reinterpret_cast<float4 *>(row + 8u * j) = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
        if (REL && bad) raise_status(status, QSIM_E_CORRUPT);
    }
    // ---- rows to memory, 16 bytes per thread (two amplitudes: the thread's columns stay the same) ----
    uint32_t p0[NP > 0 ? NP : 1], p1[NP > 0 ? NP : 1];
    if (NP > 0 && npre) {
        const uint64_t w0f = wbase | (uint64_t(f) * g.F);
        pre_frame<NP>(p0, pre_ops, npre, pre_ab, tabs, w0f, g.fl, 2u * (t & 15u), gb);
        pre_frame<NP>(p1, pre_ops, npre, pre_ab, tabs, w0f, g.fl, 2u * (t & 15u) + 1u, gb);
    }
    tm.sync();
    const uint8_t *col = tile + 16u * (t & 15u);
#pragma unroll 4
    for (uint32_t i = t; i < 16u * C; i += tm.n) {
        float4 v = *reinterpret_cast<const float4 *>(col + kRowBytes * (i >> 4));
        if (NP > 0 && npre) {
            const float2 a = pre_chunk<NP>(make_float2(v.x, v.y), p0, pre_ab, npre, i >> 4, tabs);
            const float2 b = pre_chunk<NP>(make_float2(v.z, v.w), p1, pre_ab, npre, i >> 4, tabs);
            v = make_float4(a.x, a.y, b.x, b.y);
        }
        if (wide_dst) {
            reinterpret_cast<float4 *>(dst)[i] = v;
        } else {
            dst[2u * i] = make_float2(v.x, v.y);
            dst[2u * i + 1u] = make_float2(v.z, v.w);
        }
    }
    if (hist_j && t < 32) {  // every add to S.hist came before the last sync
        const uint32_t v = S.hist[t];
        if (v) atomicAdd(&hist_j[t], v);
    }
}

// ---------------------------------------------------------------------------
// encode
// ---------------------------------------------------------------------------
// A frame's amplitudes (16-byte aligned) into the tile's rows.
__device__ __forceinline__ void load_rows_team(const Team &tm, uint8_t *tile, const float2 *src, uint32_t C) {
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint8_t *col = tile + 16u * (tm.t & 15u);
#pragma unroll 4
    for (uint32_t i = tm.t; i < 16u * C; i += tm.n) team_cp16(col + kRowBytes * (i >> 4), s4 + i);
    team_cp_wait();
    tm.sync();
}

struct EncFrame {
    uint32_t len;   // stream bytes of the frame (0: every code is zero)
    uint32_t head;  // bytes of its image before the bit-plane words
    float err_sq, norm_sq;  // thread 0: sums of (x - x')^2 and x'^2
};

// Codes the frame in the tile's rows (visible to the team) and leaves its image in the tile, visible to the team. e:
// the step exponent (QSZ1) or the code shift k (REL).
template <bool REL>
__device__ __forceinline__ EncFrame encode_frame_team(const Team &tm, TeamSmem &S, uint8_t *tile, const FrameGeom &g,
                                                      int e, int *status) {
    const uint32_t t = tm.t, lane = t & 31u, warp = t >> 5, nw = tm.n >> 5, C = g.C;
    const uint32_t padw = (2u * C + 15u) & ~15u;
    const uint32_t tbp = REL ? ((((2u * C + 3u) / 4u) + 15u) & ~15u) : 0u;
    const float inv_step = REL ? 0.f : exp2i(-e), step = REL ? 0.f : exp2i(e);
    const bool act = t < C;
    const float4 *row = reinterpret_cast<const float4 *>(tile + kRowBytes * t);
    // x - x' is exact in FP32 (|x - x'| <= s/2 <= |x'|/2 when q != 0, x' = 0 otherwise); a thread sums 64 values
    float err_sq = 0.f, norm_sq = 0.f;
    uint32_t wr = 0, wi = 0, swr = 0, swi = 0;
    uint32_t lo[32], hi[32];  // codes, then bit planes: 0..15 of Re | 0..15 of Im; hi likewise planes 16..31
    bool narrow = false;
    if constexpr (!REL) {
        // codes below 2^14 in magnitude: rounded by one FMA into the low mantissa bits (the difference of two such
        // floats' bits is the difference of the codes), differences and zigzag codes of Re and Im packed in one word
        bool fits = true;
        uint32_t any = 0;
        if (act) {
            const float lim = 16383.f * step, off = -kRound * step;
            int32_t pr = kRoundBits, pi = kRoundBits;
#pragma unroll
            for (uint32_t j = 0; j < 32; j += 2) {
                const float4 v = row[j / 2];
                const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (uint32_t k = 0; k < 2; ++k) {
                    const float xr = x[2 * k], xi = x[2 * k + 1];
                    fits = fits && fabsf(xr) <= lim && fabsf(xi) <= lim;  // false for NaN
                    const float fr = fmaf(xr, inv_step, kRound), fi = fmaf(xi, inv_step, kRound);
                    const float yr = fmaf(fr, step, off), yi = fmaf(fi, step, off);  // exact
                    const float er = xr - yr, ei = xi - yi;
                    err_sq = fmaf(er, er, err_sq);
                    norm_sq = fmaf(yr, yr, norm_sq);
                    err_sq = fmaf(ei, ei, err_sq);
                    norm_sq = fmaf(yi, yi, norm_sq);
                    const int32_t br = __float_as_int(fr), bi = __float_as_int(fi);
                    const uint32_t p = __byte_perm(uint32_t(br - pr), uint32_t(bi - pi), 0x5410);
                    pr = br;
                    pi = bi;
                    const uint32_t sg = ((p >> 15) & 0x00010001u) * 0xffffu;
                    lo[j + k] = ((p << 1) & 0xfffefffeu) ^ sg;
                    any |= lo[j + k];
                }
            }
        } else {
#pragma unroll
            for (uint32_t j = 0; j < 32; ++j) lo[j] = 0;
        }
        narrow = __all_sync(kFull, fits);
        if (narrow) {
            wr = 32 - __clz(any & 0xffffu);
            wi = 32 - __clz(any >> 16);
            transpose32(lo);
        }
    }
    if (!narrow) {
        int bad = 0;
        err_sq = norm_sq = 0.f;
        uint32_t anyr = 0, anyi = 0;
        int32_t pr = 0, pi = 0;
#pragma unroll
        for (uint32_t j = 0; j < 32; ++j) {
            lo[j] = hi[j] = 0;
            if (!act) continue;
            const float2 v = reinterpret_cast<const float2 *>(row)[j];
            const float x[2] = {v.x, v.y};
            int32_t q[2];
#pragma unroll
            for (uint32_t p = 0; p < 2; ++p) {
                q[p] = quantize_one<REL>(x[p], inv_step, uint32_t(e), bad);
                float y;
                if constexpr (REL) {
                    const bool neg = x[p] < 0.f && q[p] != 0;
                    if (p) swi |= uint32_t(neg) << j;
                    else swr |= uint32_t(neg) << j;
                    const float mag = __uint_as_float(uint32_t(q[p]) << e);
                    y = neg ? -mag : mag;
                } else {
                    y = float(q[p]) * step;
                }
                const float d = x[p] - y;
                err_sq = fmaf(d, d, err_sq);
                norm_sq = fmaf(y, y, norm_sq);
            }
            const uint32_t zr = zigzag(int32_t(uint32_t(q[0]) - uint32_t(pr)));
            const uint32_t zi = zigzag(int32_t(uint32_t(q[1]) - uint32_t(pi)));
            pr = q[0];
            pi = q[1];
            anyr |= zr;
            anyi |= zi;
            lo[j] = __byte_perm(zr, zi, 0x5410);
            hi[j] = __byte_perm(zr, zi, 0x7632);
        }
        if (bad) raise_status(status, bad);
        wr = 32 - __clz(anyr);
        wi = 32 - __clz(anyi);
        transpose32(lo);
        transpose32(hi);
    }
    uint32_t tr = 0, ti = 0, cnt = 0;
    if constexpr (REL) {
        if (act) {
            tr = sign_type(swr);
            ti = sign_type(swi);
        }
        cnt = uint32_t(tr == 2u) | (uint32_t(ti == 2u) << 8) | (uint32_t(tr == 3u) << 16) | (uint32_t(ti == 3u) << 24);
    }
    // ---- word offsets ----
    const uint32_t wp = wr | (wi << 16);
    uint32_t incl = wp, icnt = cnt;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(kFull, incl, o);
        const uint32_t b = REL ? __shfl_up_sync(kFull, icnt, o) : 0u;
        if (lane >= o) {
            incl += a;
            icnt += b;
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        err_sq += __shfl_xor_sync(kFull, err_sq, o);
        norm_sq += __shfl_xor_sync(kFull, norm_sq, o);
    }
    if (lane == 31) {
        S.w[warp] = incl;
        S.s[warp] = icnt;
        S.err[warp] = err_sq;
        S.nrm[warp] = norm_sq;
    }
    tm.sync();  // every row is in registers: the image takes the rows' place
    uint32_t base = 0, tot = 0, cbase = 0, ctot = 0;
    EncFrame r{};
#pragma unroll
    for (uint32_t w = 0; w < 4; ++w)
        if (w < nw) {
            if (w == warp) {
                base = tot;
                cbase = ctot;
            }
            tot += S.w[w];
            ctot += S.s[w];
            r.err_sq += S.err[w];
            r.norm_sq += S.nrm[w];
        }
    const uint32_t words = (tot & 0xffffu) + (tot >> 16);
    const uint32_t signs = REL ? sign_section_bytes(ctot) : 0u;
    r.head = padw + tbp + signs;
    r.len = words ? r.head + ((4u * words + 15u) & ~15u) : 0u;
    if (act) {
        tile[t] = uint8_t(wr);
        tile[C + t] = uint8_t(wi);
    }
    for (uint32_t b = 2u * C + t; b < padw; b += tm.n) tile[b] = 0;
    if constexpr (REL) {
        // the 2-bit types of four chunks per byte (frames of fewer than four chunks: all of them in byte 0)
        uint8_t *types = tile + padw;
        if (C >= 4) {
            uint32_t a = tr << (2u * (t & 3u)), b = ti << (2u * (t & 3u));
            a |= __shfl_xor_sync(kFull, a, 1);
            b |= __shfl_xor_sync(kFull, b, 1);
            a |= __shfl_xor_sync(kFull, a, 2);
            b |= __shfl_xor_sync(kFull, b, 2);
            if (act && !(t & 3u)) {
                types[t >> 2] = uint8_t(a);
                types[(C + t) >> 2] = uint8_t(b);
            }
        } else {
            uint32_t a = act ? (tr << (2u * t)) | (ti << (2u * (C + t))) : 0u;
            a |= __shfl_xor_sync(kFull, a, 1);
            if (t == 0) types[0] = uint8_t(a);
        }
        for (uint32_t b = (2u * C + 3u) / 4u + t; b < tbp; b += tm.n) types[b] = 0;
        cbase += icnt - cnt;
        const uint32_t n2r = ctot & 0xffu, n2 = n2r + ((ctot >> 8) & 0xffu);
        const uint32_t n3r = (ctot >> 16) & 0xffu, n3 = n3r + (ctot >> 24);
        uint32_t *mixw = reinterpret_cast<uint32_t *>(types + tbp);
        uint16_t *runw = reinterpret_cast<uint16_t *>(mixw + n2);
        if (tr == 2u) mixw[cbase & 0xffu] = swr;
        if (ti == 2u) mixw[n2r + ((cbase >> 8) & 0xffu)] = swi;
        if (tr == 3u) runw[(cbase >> 16) & 0xffu] = uint16_t(sign_run_record(swr));
        if (ti == 3u) runw[n3r + (cbase >> 24)] = uint16_t(sign_run_record(swi));
        for (uint32_t b = n3 + t; b < (signs - 4u * n2) / 2u; b += tm.n) runw[b] = 0;
    }
    base += incl - wp;
    uint32_t *pay = reinterpret_cast<uint32_t *>(tile + r.head);
    uint32_t *pr = pay + (base & 0xffffu), *pi = pay + (tot & 0xffffu) + (base >> 16);
#pragma unroll
    for (uint32_t b = 0; b < 16; ++b) {
        if (b < wr) pr[b] = lo[b];
        if (b < wi) pi[b] = lo[16 + b];
    }
    if (!narrow) {
#pragma unroll
        for (uint32_t b = 0; b < 16; ++b) {
            if (16u + b < wr) pr[16 + b] = hi[b];
            if (16u + b < wi) pi[16 + b] = hi[16 + b];
        }
    }
    if (words + t < ((words + 3u) & ~3u)) pay[words + t] = 0;
    tm.sync();
    return r;
}

// Frame offsets of one block from its frames' lengths (data_start first), and the FP64 sums of the frames' error
// partials. Returns the block's stream bytes; a and b in thread 0. nframes a power of two above 1.
__device__ __forceinline__ uint32_t block_offsets_team(const Team &tm, TeamSmem &S, const uint32_t *flen,
                                                       const float2 *part, uint32_t *foff, uint32_t nframes,
                                                       uint32_t data_start, double &a, double &b) {
    const uint32_t t = tm.t, lane = t & 31u, warp = t >> 5, nw = tm.n >> 5;
    uint32_t run = data_start;
    a = b = 0;
    for (uint32_t f0 = 0; f0 < nframes; f0 += 4u * tm.n) {
        uint32_t v[4], sum = 0;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t f = f0 + 4u * t + k;
            v[k] = 0;
            if (f < nframes) {
                v[k] = __ldcg(flen + f);
                const float2 p = __ldcg(part + f);
                a += double(p.x);
                b += double(p.y);
            }
            sum += v[k];
        }
        uint32_t incl = sum;
#pragma unroll
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) S.w[warp] = incl;
        tm.sync();
        uint32_t off = run + incl - sum;
        for (uint32_t w = 0; w < nw; ++w) {
            if (w < warp) off += S.w[w];
            run += S.w[w];
        }
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t f = f0 + 4u * t + k;
            if (f < nframes) foff[f] = off;
            off += v[k];
        }
        tm.sync();
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(kFull, a, o);
        b += __shfl_xor_sync(kFull, b, o);
    }
    if (lane == 0) {
        S.da[warp] = a;
        S.db[warp] = b;
    }
    tm.sync();
    a = b = 0;
    for (uint32_t w = 0; w < nw; ++w) {
        a += S.da[w];
        b += S.db[w];
    }
    return run;
}

// Reserve block j's slot for `total` bytes (thread 0). keep: it keeps the slot reserved for it beforehand when it fits,
// and is counted as overflowed when it does not.
__device__ __forceinline__ EncTarget reserve_block(uint32_t total, bool keep, EncTarget *tgt_j, const ArenaDev &dev,
                                                   const ArenaDev &host, StageAccum *acc, int *status) {
    EncTarget t{};
    if (keep) {
        t.ptr = reinterpret_cast<uint8_t *>(__ldcg(reinterpret_cast<const unsigned long long *>(&tgt_j->ptr)));
        t.cap = __ldcg(reinterpret_cast<const unsigned long long *>(&tgt_j->cap));
        t.tier = __ldcg(&tgt_j->tier);
    }
    if (!keep || t.ptr == nullptr || total > t.cap) {
        if (keep && acc) atomicAdd(reinterpret_cast<unsigned long long *>(&acc->overflow_blocks), 1ull);
        reserve_slot(total, dev, host, &t, status);
        *tgt_j = t;
    }
    return t;
}

// 32-bit word i of a stream's header and offset table (data_start bytes) for a block whose frames up to f0 are empty,
// frame f0 has len bytes and the later ones are empty
__device__ __forceinline__ uint32_t header_word(uint32_t i, bool rel, const FrameGeom &g, int m, int e, uint32_t f0,
                                                uint32_t len) {
    const uint32_t ds = uint32_t(g.data_start);
    switch (i) {
        case 0: return rel ? kQszrMagic : kQszMagic;
        case 1: return 1u;  // version 1, flags 0
        case 2: return uint32_t(m) | (uint32_t(g.fl) << 8) | (uint32_t(uint8_t(int8_t(e))) << 16);
        case 3: return g.nframes;
        case 4: return ds + len;  // total bytes (below 2^32 for every m <= 26)
        case 5: case 6: case 7: return 0u;
        default: return i - 8u > g.nframes ? 0u : i - 8u > f0 ? ds + len : ds;
    }
}

// the stage's totals for one block of `total` stream bytes in slot t
__device__ __forceinline__ void count_block(StageAccum *acc, uint64_t total, const EncTarget &t) {
    atomicAdd(reinterpret_cast<unsigned long long *>(&acc->store_bytes), total);
    atomicAdd(reinterpret_cast<unsigned long long *>(&acc->reserved_bytes), t.cap);
    if (t.tier) atomicAdd(reinterpret_cast<unsigned long long *>(&acc->host_bytes), t.cap);
    atomicAdd(reinterpret_cast<unsigned long long *>(&acc->blocks), 1ull);
}

// A one-frame block (header, offsets and the frame's image in the tile) to its slot `out` (null: nothing).
template <bool REL>
__device__ __forceinline__ void store_single_frame(const Team &tm, const uint8_t *tile, const FrameGeom &g, int m, int e,
                                                   uint32_t len, uint8_t *out) {
    if (!out) return;
    for (uint32_t i = tm.t; i < uint32_t(g.data_start) / 4u; i += tm.n)
        reinterpret_cast<uint32_t *>(out)[i] = header_word(i, REL, g, m, e, 0, len);
    uint4 *d = reinterpret_cast<uint4 *>(out + g.data_start);
    for (uint32_t i = tm.t; i < len / 16u; i += tm.n) d[i] = reinterpret_cast<const uint4 *>(tile)[i];
}

// Thread 0 after a one-frame block's slot is known: result, table slot and totals. Returns the slot, null when the
// reservation failed.
__device__ __forceinline__ uint8_t *finish_single_frame(uint32_t total, const EncTarget &t, EncResult &out,
                                                        BlockSlot *slot, StageAccum *acc) {
    const bool fits = t.ptr != nullptr && total <= t.cap;
    out.total = total;
    out.overflow = fits ? 0u : 1u;
    if (fits) {
        slot->ptr = t.ptr;
        slot->bytes = total;
        slot->tier = t.tier;
        if (acc) count_block(acc, total, t);
    } else if (acc) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&acc->overflow_blocks), 1ull);
    }
    return fits ? t.ptr : nullptr;
}

// The frame's image from the tile to where the copy step finds it: the bit-plane words over the frame's own amplitudes
// (they never need more room), the part before them to the side record.
__device__ __forceinline__ void stage_frame(const Team &tm, const uint8_t *tile, const EncFrame &r, float2 *frame,
                                            uint8_t *side) {
    uint4 *pay = reinterpret_cast<uint4 *>(frame), *s = reinterpret_cast<uint4 *>(side);
    const uint4 *img = reinterpret_cast<const uint4 *>(tile);
    const uint32_t h = r.head / 16u, n = r.len / 16u;  // n = 0 for an all-zero frame
    for (uint32_t i = tm.t; i < n; i += tm.n) {
        if (i < h) s[i] = img[i];
        else pay[i - h] = img[i];
    }
}

// Second step of blocks of several frames: frame f's staged image (read through L2) to its offset in the block's slot t;
// the block's last frame writes the header, the table slot and the totals. 128 threads.
template <bool REL>
__device__ __forceinline__ void copy_frame_team(const Team &tm, const float2 *frame, const uint8_t *side, uint32_t len,
                                                uint32_t head, uint32_t off, const FrameGeom &g, int m, int e, uint32_t f,
                                                const EncTarget &t, EncResult *res_j, BlockSlot *slot, StageAccum *acc) {
    const bool fits = t.ptr != nullptr && uint64_t(off) + len <= t.cap;
    if (fits && len) {
        const uint4 *s = reinterpret_cast<const uint4 *>(side), *pay = reinterpret_cast<const uint4 *>(frame);
        uint4 *d = reinterpret_cast<uint4 *>(t.ptr + off);
        const uint32_t h = head / 16u, n = len / 16u;
#pragma unroll 4
        for (uint32_t i = tm.t; i < n; i += tm.n) d[i] = __ldcg(i < h ? s + i : pay + (i - h));
    }
    if (tm.t != 0) return;
    if (!fits) atomicOr(&res_j->overflow, 1u);
    if (t.ptr && g.data_start <= t.cap) reinterpret_cast<uint32_t *>(t.ptr + 32)[f] = off;
    if (f != g.nframes - 1) return;
    const uint64_t total = uint64_t(off) + len;
    res_j->total = total;
    if (t.ptr && total <= t.cap) {
        uint32_t *h32 = reinterpret_cast<uint32_t *>(t.ptr);
        for (uint32_t i = 0; i < 8; ++i) h32[i] = header_word(i, REL, g, m, e, f, uint32_t(total - g.data_start));
        for (uint32_t i = 8 + g.nframes; i < uint32_t(g.data_start) / 4u; ++i)
            h32[i] = i == 8 + g.nframes ? uint32_t(total) : 0u;
        slot->ptr = t.ptr;
        slot->bytes = total;
        slot->tier = t.tier;
        if (acc) count_block(acc, total, t);
    } else if (acc) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&acc->overflow_blocks), 1ull);
    }
}

}  // namespace cdev
}  // namespace qsim
