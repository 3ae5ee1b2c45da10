// Tile passes that keep the tile in registers (sm_103a, tcgen05).
//
// A pass of 4096-amplitude tiles whose ops are width-5 dense ops on the tensor cores and runs of degree-2 diagonal ops
// needs shared memory only to hand a tile from one dense op's index groups to the next one's. Thread g of a tile's 128
// owns index group g of the current dense op, its 32 amplitudes in registers: it loads them straight from the working
// vector for the first op and stores them straight back after the last one (its neighbours in the warp hold the tile's
// low three bits, so a row of 8 amplitudes is one 64-byte access), the diagonal runs before and after a dense op are
// applied to the registers, and between two dense ops each thread scatters its group and gathers the next one. The
// staged form of these passes (gates_dev.cuh) moves the tile through shared memory once more at each end, twice more
// for every diagonal run, and is bound by exactly that.
//
// The index groups are those of the staged form, so the operands of every MMA, the order of its K steps, the phases
// and the rounding of every product are the same, and so are the results. Per 2^28 amplitudes, staged and in registers:
// one op 0.82 and 0.75 ms (5.7 TB/s; a copy takes 0.63), two 1.04 and 0.90, two and a run 1.80 and 1.31. What bounds the
// rest is the chain of load, MMA, read-back and store at 16 warps per SM.
//
// A CTA works on HALVES tiles at a time, 128 threads each, that share the dense ops' B operands and the tables. With
// two halves every op's B stays in shared memory (passes of up to two TF32 ops); with one, B is reloaded per op into
// one buffer as soon as the previous op's MMAs have read it. Either way four tiles are in flight per SM, which fills
// its 512 TMEM columns.
#pragma once

#include "gates_dev.cuh"

namespace qsim {
namespace gdev {

template <int H>
struct RegSmem {
    uint64_t mbar[H];
    uint32_t tmem;
    uint32_t next[H][2];                   // a half's next tile, by iteration parity
    uint32_t pa[H][2][kRegMaxPoly][13];    // by parity: a run's linear coefficients and constant on this tile
};

// one half's 128 threads (barrier ids as constants: an id in a register would reserve all sixteen for the CTA)
__device__ __forceinline__ void half_sync(uint32_t h) {
    if (h == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
}
__device__ __forceinline__ bool half_all(uint32_t h, bool ok) {
    uint32_t r;
    if (h == 0)
        asm volatile(
            "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 1, 128, p;\n\t"
            "selp.u32 %0, 1, 0, q;\n\t}\n"
            : "=r"(r)
            : "r"(uint32_t(ok))
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 2, 128, p;\n\t"
            "selp.u32 %0, 1, 0, q;\n\t}\n"
            : "=r"(r)
            : "r"(uint32_t(ok))
            : "memory");
    return r != 0;
}

template <int PREC>
__host__ __device__ constexpr uint32_t reg_b_bytes() {
    return umma_b_bytes<PREC>();
}

// Dynamic shared memory of a register pass: B operands, one 32 KB tile per half when the pass needs it, tables, and
// seven words per thread and diagonal run.
struct RegShape {
    bool resident;  // every dense op's B operand stays (else one buffer, reloaded per op)
    bool tile;
    uint32_t bytes;
};
template <int PREC, int H>
__host__ __device__ constexpr RegShape reg_shape(uint32_t ndense, uint32_t npoly, uint32_t flags, uint32_t words) {
    RegShape s{};
    s.resident = H == 2 || ndense == 1;
    s.tile = PREC == QSIM_PREC_BF16X3 || ndense > 1 || flags != (kRegIn | kRegOut);
    s.bytes = 1024u + (s.resident ? ndense : 1u) * reg_b_bytes<PREC>() + (s.tile ? H * 32768u : 0u) + words * 4u +
              npoly * 7u * 512u;
    return s;
}

// The 32 x 32 complex product of the half's 128 index groups: (re, im) of thread g's group in, out in place. The
// operands and their order are those of apply_dense_umma / apply_dense_umma3. `between` runs after every thread of
// the half has entered the op and before any leaves it. False when the wait for the MMAs ran out (status set).
template <int PREC, class F>
__device__ __forceinline__ bool dense_regs(float (&re)[32], float (&im)[32], uint8_t *tile, bool gathered, uint32_t bsm,
                                           uint32_t tmem, uint32_t mbar, uint32_t &phase, uint32_t h, bool hook,
                                           int *status, F between) {
    const uint32_t g = threadIdx.x & 127u;
    const uint32_t lane = (32u * (g >> 5)) << 16;
    bool ok = true;
    auto wait = [&]() {
        // one warp polls, the others wait at the barrier
        ok = half_all(h, g >= 32u || umma::mbar_wait(mbar, phase, kUmmaWaitNs));
        phase ^= 1u;
        if (!ok && g == 0) raise_status(status, QSIM_E_TIMEOUT);
    };
    if constexpr (PREC == QSIM_PREC_TF32) {
        {
            uint32_t a[32];
#pragma unroll
            for (uint32_t j = 0; j < 32; ++j) a[j] = f32_to_tf32(re[j]);
            umma::tmem_st32(tmem + lane + kUmmaACol, a);
#pragma unroll
            for (uint32_t j = 0; j < 32; ++j) a[j] = f32_to_tf32(im[j]);
            umma::tmem_st32(tmem + lane + kUmmaACol + 32u, a);
            umma::tmem_wait_st();
        }
        cp_async_wait_all();  // this thread's share of B
        umma::fence_proxy_async_smem();
        umma::fence_before_sync();
        half_sync(h);
        if (g == 0 && !hook) {  // the test hook issues nothing
            umma::fence_after_sync();
#pragma unroll
            for (uint32_t s = 0; s < 8; ++s) {
                const uint64_t db = umma::desc_kmajor_sw128(bsm + (s >> 2) * 8192u + (s & 3u) * 32u);
                umma::mma_tf32_ts(tmem, tmem + kUmmaACol + 8u * s, db, kUmmaIdesc, s);
            }
            umma::commit(mbar);
        }
        between();
        wait();
    } else {
        if (gathered) half_sync(h);  // every thread has read the tile: A takes its place
        uint8_t *arow = tile + (g >> 3) * 1024u + (g & 7u) * 128u;
        uint32_t mid[32];
#pragma unroll
        for (uint32_t c = 0; c < 8; ++c) {  // 16-byte chunk c = K elements 8c .. 8c + 7 (Re parts, then Im parts)
            uint32_t hi[4], lo[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t k = 8 * c + 2 * q;
                const float x0 = k < 32 ? re[k & 31] : im[k & 31], x1 = k < 32 ? re[(k + 1) & 31] : im[(k + 1) & 31];
                __nv_bfloat16 h0, m0, l0, h1, m1, l1;
                split3(x0, h0, m0, l0);
                split3(x1, h1, m1, l1);
                hi[q] = pack_bf16(h0, h1);
                lo[q] = pack_bf16(l0, l1);
                mid[4 * c + q] = pack_bf16(m0, m1);
            }
            const uint32_t o = (c ^ (g & 7u)) << 4;
            *reinterpret_cast<uint4 *>(arow + o) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4 *>(arow + 16384u + o) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        cp_async_wait_all();
        umma::fence_proxy_async_smem();
        umma::fence_before_sync();
        half_sync(h);
        const uint32_t a0 = umma::smem_addr(tile);
        auto product = [&](uint32_t a_half, uint32_t b_part, uint32_t first) {
#pragma unroll
            for (uint32_t s = 0; s < 4; ++s) {
                const uint64_t da = umma::desc_kmajor_sw128(a0 + a_half * 16384u + s * 32u);
                const uint64_t db = umma::desc_kmajor_sw128(bsm + b_part * 8192u + s * 32u);
                umma::mma_bf16_ss(tmem, da, db, kUmmaIdescBf16, first && s == 0 ? 0u : 1u);
            }
        };
        if (g == 0 && !hook) {
            umma::fence_after_sync();
            product(1, 0, 1);  // lo x B_hi (the first product overwrites D)
            product(0, 2, 0);  // hi x B_lo
            umma::commit(mbar);
        }
        between();
        wait();
        if (!ok) return false;
#pragma unroll
        for (uint32_t c = 0; c < 8; ++c) {
            const uint32_t o = (c ^ (g & 7u)) << 4;
            *reinterpret_cast<uint4 *>(arow + 16384u + o) =
                make_uint4(mid[4 * c], mid[4 * c + 1], mid[4 * c + 2], mid[4 * c + 3]);
        }
        umma::fence_proxy_async_smem();
        half_sync(h);
        if (g == 0 && !hook) {
            umma::fence_after_sync();
            product(1, 1, 0);  // mid x B_mid
            product(1, 0, 0);  // mid x B_hi
            product(0, 1, 0);  // hi x B_mid
            product(0, 0, 0);  // hi x B_hi
            umma::commit(mbar);
        }
        wait();
    }
    if (!ok) return false;
    umma::fence_after_sync();
    uint32_t d[32];
    umma::tmem_ld32(tmem + lane, d);
#pragma unroll
    for (uint32_t j = 0; j < 32; ++j) re[j] = __uint_as_float(d[j]);
    umma::tmem_ld32(tmem + lane + 32u, d);
#pragma unroll
    for (uint32_t j = 0; j < 32; ++j) im[j] = __uint_as_float(d[j]);
    umma::fence_before_sync();  // the next op's barrier orders these reads before its MMAs
    return true;
}

// A diagonal run on thread g's amplitudes: one phase exp(2 pi i P) each, P the run's polynomial in 32-bit fixed-point
// turns. pa: its coefficients on this tile; pc: the tile-independent part of P that the group's bits decide, summed once
// per CTA (the quadratic terms among them, theirs with each matrix bit, and the row of T).
__device__ __forceinline__ void poly_regs(float (&re)[32], float (&im)[32], const uint32_t *pw, const uint32_t *pa,
                                          const uint32_t *pc) {
    const uint32_t g = threadIdx.x & 127u;
    uint32_t ang = pa[12] + pc[g], beta[5];
#pragma unroll
    for (uint32_t t = 0; t < 7; ++t) ang += (g >> t) & 1u ? pa[t] : 0u;
#pragma unroll
    for (uint32_t b = 0; b < 5; ++b) beta[b] = pa[7 + b] + pc[128u * (1u + b) + g];
    const uint32_t *tr = pw + pc[768u + g];
#pragma unroll
    for (uint32_t i = 0; i < 32; ++i) {  // Gray-code order: one linear coefficient in or out per step
        const uint32_t j = gray5(i);
        if (i) ang = (j >> ctz5(i)) & 1u ? ang + beta[ctz5(i)] : ang - beta[ctz5(i)];
        float sn, cs;
        __sincosf(6.28318530717958648f * 2.3283064365386963e-10f * float(int32_t(ang + tr[j])), &sn, &cs);
        const float2 v = make_float2(re[j], im[j]);
        re[j] = cs * v.x - sn * v.y;
        im[j] = cs * v.y + sn * v.x;
    }
}

template <int PREC, int H>
__device__ __forceinline__ void pass_reg_tiles(float2 *__restrict__ wv, uint32_t W, uint64_t ntiles, const PassDev &P,
                                               const uint4 *__restrict__ gblob, const uint32_t *__restrict__ bfr,
                                               const uint64_t *__restrict__ gbase, RegSmem<H> &S, uint8_t *dyn,
                                               uint32_t *ctr, int *status) {
    const uint32_t tid = threadIdx.x, g = tid & 127u, h = tid >> 7;
    constexpr uint32_t NT = 128u * H;
    const bool hook = (P.umma & 2u) != 0;
    uint8_t *mem = dyn + ((1024u - (umma::smem_addr(dyn) & 1023u)) & 1023u);
    const RegShape shape = reg_shape<PREC, H>(P.reg_dense, P.reg_poly, P.reg_flags, P.reg_words);
    uint8_t *tiles = mem + (shape.resident ? P.reg_dense : 1u) * reg_b_bytes<PREC>();
    uint32_t *tab = reinterpret_cast<uint32_t *>(tiles + (shape.tile ? H * 32768u : 0u));
    uint32_t *pc = tab + P.reg_words;
    // ---- once per CTA: tables, B operands, TMEM, mbarriers, the tile-independent parts of the runs ----
    for (uint32_t i = tid; i < P.reg_words / 4u; i += NT) cp_async16(reinterpret_cast<uint4 *>(tab) + i, gblob + P.reg_off + i);
    if (tid < 32) umma::tmem_alloc(umma::smem_addr(&S.tmem), 128u * H);
    if (tid < uint32_t(H)) umma::mbar_init(umma::smem_addr(&S.mbar[tid]), 1);
    cp_async_wait_all();
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t ndense = tab[1], npoly = tab[2], steps = tab[0], flags = tab[3];
    auto load_b = [&](uint32_t d, uint8_t *dst, uint32_t t0, uint32_t n) {
        const uint4 *src = reinterpret_cast<const uint4 *>(bfr + tab[kRegHead + kRegDense * d + 133]);
        for (uint32_t i = t0; i < reg_b_bytes<PREC>() / 16u; i += n) cp_async16(reinterpret_cast<uint4 *>(dst) + i, src + i);
        cp_async_commit();
    };
    if (shape.resident)
        for (uint32_t d = 0; d < ndense; ++d) load_b(d, mem + d * reg_b_bytes<PREC>(), tid, NT);
    else
        load_b(0, mem, tid, NT);
    for (uint32_t p = h; p < npoly; p += H) {
        const uint32_t *pw = tab + tab[52 + p];
        uint32_t th = 0, beta[5] = {};
        for (uint32_t t = 0; t < 7; ++t) {
            if (!((g >> t) & 1u)) continue;
            for (uint32_t t2 = t + 1; t2 < 7; ++t2)
                if ((g >> t2) & 1u) th += pw[12 * t + t2];
#pragma unroll
            for (uint32_t b = 0; b < 5; ++b) beta[b] += pw[12 * t + 7 + b];
        }
        uint32_t row = 0, nr = 0;
        for (uint32_t t = 0; t < 7; ++t)
            if ((pw[205] >> t) & 1u) row |= ((g >> t) & 1u) << nr++;
        pc[896u * p + g] = th;
#pragma unroll
        for (uint32_t b = 0; b < 5; ++b) pc[896u * p + 128u * (1u + b) + g] = beta[b];
        pc[896u * p + 768u + g] = pw[206] + kRegRow * row;
    }
    auto init_pa = [&](uint32_t par) {
        if (g < 13)
            for (uint32_t p = 0; p < npoly; ++p) S.pa[h][par][p][g] = tab[tab[52 + p] + (g < 12 ? 192 + g : 204)];
    };
    init_pa(0);
    uint32_t off_in = 0, off_out = 0;  // working offset of the thread's group in the first and the last dense op
#pragma unroll
    for (uint32_t t = 0; t < 7; ++t) {
        off_in |= ((g >> t) & 1u) << tab[28 + t];
        off_out |= ((g >> t) & 1u) << tab[40 + t];
    }
    cp_async_wait_all();
    __syncthreads();
    uint8_t *tile8 = tiles + h * 32768u;
    float2 *tile = reinterpret_cast<float2 *>(tile8);
    const uint32_t tmem = S.tmem + 128u * h, mbar = umma::smem_addr(&S.mbar[h]);
    auto dense_tab = [&](uint32_t d) { return tab + kRegHead + kRegDense * d; };
    auto group_base = [&](uint32_t d) { return dense_tab(d)[g & 63u] ^ dense_tab(d)[64u + (g >> 6)]; };
    const uint32_t lane = tid & 31u, out_pos = lane < P.nout ? P.out_pos[lane] : 64u;
    const uint64_t tmask = (1ull << P.nout) - 1;
    // working index of element 0 of a tile: lane b places bit b of the tile's number
    auto tile_base = [&](uint64_t t) {
        const uint64_t b = out_pos < 64u ? ((t & tmask) >> lane & 1ull) << out_pos : 0ull;
        uint64_t r = __reduce_or_sync(kFull, uint32_t(b));
        if (W > 32) r |= uint64_t(__reduce_or_sync(kFull, uint32_t(b >> 32))) << 32;
        return r;
    };
    uint32_t phase = 0;
    bool ok = true;
    uint32_t it = 0;
    for (uint64_t t = uint64_t(blockIdx.x) * H + h; t < ntiles; ++it) {
        if (g == 0) S.next[h][it & 1u] = gridDim.x * H + atomicAdd(ctr, 1u);  // read after this tile's barriers
        const uint64_t grp = t >> P.nout, base = tile_base(t);
        float2 *gp = wv + (grp << W) + base;
        const uint64_t gb = gbase ? gbase[grp] : 0ull;
        float re[32], im[32];
        // ---- the first dense op's groups ----
        bool gathered = false;
        if (flags & kRegIn) {
            const float2 *src = gp + off_in;
            uint32_t o = 0, bit[5];
#pragma unroll
            for (uint32_t b = 0; b < 5; ++b) bit[b] = 1u << tab[35 + b];
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) {
                if (i) o ^= bit[ctz5(i)];
                const float2 v = src[o];
                re[gray5(i)] = v.x;
                im[gray5(i)] = v.y;
            }
        } else {
            uint32_t o = 0;
#pragma unroll
            for (uint32_t b = 0; b < 7; ++b) o |= ((g >> b) & 1u) << P.tile_pos[b];
            const uint32_t tq = swz_thread<128>(g);
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) {
                if (i) o ^= 1u << P.tile_pos[7 + ctz5(i)];
                cp_async8(&tile[(tq ^ swz_u<128>(gray5(i))) + 128u * gray5(i)], gp + o);
            }
        }
        // the runs' coefficients on this tile: every term whose constant bits are 1 here
        for (uint32_t p = 0; p < npoly; ++p) {
            const uint32_t *tr = tab + tab[52 + p] + kPolyHeadWords;
            for (uint32_t i = g; i < tab[56 + p]; i += 128) {
                const uint32_t k = tr[4 * i], s1 = tr[4 * i + 1], s2 = tr[4 * i + 2];
                const uint64_t b1 = s1 < 64 ? (base >> s1) & 1ull : (gb >> (s1 - 64)) & 1ull;
                const uint64_t b2 = s2 == kNoSrc ? 1ull : s2 < 64 ? (base >> s2) & 1ull : (gb >> (s2 - 64)) & 1ull;
                if (b1 & b2) atomicAdd(&S.pa[h][it & 1u][p][k == kPolyConst ? 12u : k], tr[4 * i + 3]);
            }
        }
        auto gather = [&](uint32_t d) {
            uint32_t a = group_base(d), bit[5];
#pragma unroll
            for (uint32_t b = 0; b < 5; ++b) bit[b] = dense_tab(d)[128 + b];
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) {
                if (i) a ^= bit[ctz5(i)];
                const float2 v = tile[a];
                re[gray5(i)] = v.x;
                im[gray5(i)] = v.y;
            }
            gathered = true;
        };
        auto scatter = [&](uint32_t d) {
            uint32_t a = group_base(d), bit[5];
#pragma unroll
            for (uint32_t b = 0; b < 5; ++b) bit[b] = dense_tab(d)[128 + b];
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) {
                if (i) a ^= bit[ctz5(i)];
                tile[a] = make_float2(re[gray5(i)], im[gray5(i)]);
            }
        };
        if (!(flags & kRegIn)) {
            cp_async_wait_all();
            half_sync(h);
            gather(0);
        } else if (tab[4] & kRegPoly) {
            half_sync(h);  // the first step reads the coefficients
        }
        // ---- the ops ----
        uint32_t done = 0;  // dense ops done
        for (uint32_t s = 0; s < steps && ok; ++s) {
            const uint32_t st = tab[4 + s];
            if (st & kRegPoly) {
                const uint32_t p = st & 0xffffu;
                poly_regs(re, im, tab + tab[52 + p], S.pa[h][it & 1u][p], pc + 896u * p);
                continue;
            }
            if (done) {
                scatter(st - 1);
                half_sync(h);
                gather(st);
            }
            ok = dense_regs<PREC>(re, im, tile8, gathered, umma::smem_addr(mem) + (shape.resident ? st * reg_b_bytes<PREC>() : 0u),
                                  tmem, mbar, phase, h, hook, status, [&]() {
                                      // the other parity's coefficients are free (every thread has left the last
                                      // tile) and are next added to after this op's wait
                                      if (done == 0) init_pa((it + 1) & 1u);
                                  });
            if (ok && !shape.resident) load_b(st + 1 < ndense ? st + 1 : 0, mem, g, 128);
            ++done;
        }
        if (!ok) break;  // uniform in the half: the MMA wait ran out (status set)
        // ---- the last dense op's groups ----
        if (flags & kRegOut) {
            float2 *dst = gp + off_out;
            uint32_t o = 0, bit[5];
#pragma unroll
            for (uint32_t b = 0; b < 5; ++b) bit[b] = 1u << tab[47 + b];
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) {
                if (i) o ^= bit[ctz5(i)];
                dst[o] = make_float2(re[gray5(i)], im[gray5(i)]);
            }
        } else {
            scatter(ndense - 1);
            half_sync(h);
            uint32_t o = 0;
#pragma unroll
            for (uint32_t b = 0; b < 7; ++b) o |= ((g >> b) & 1u) << P.tile_pos[b];
            const uint32_t tq = swz_thread<128>(g);
#pragma unroll
            for (uint32_t i = 0; i < 32; ++i) {
                if (i) o ^= 1u << P.tile_pos[7 + ctz5(i)];
                gp[o] = tile[(tq ^ swz_u<128>(gray5(i))) + 128u * gray5(i)];
            }
            half_sync(h);  // the next tile's loads overwrite this one
        }
        t = S.next[h][it & 1u];
    }
    cp_async_wait_all();  // a reload of B may be in flight
    // after a wait that ran out, wait (bounded) once more for the MMAs in flight before TMEM is freed
    if (!ok) umma::mbar_wait(mbar, phase ^ 1u, kUmmaWaitNs);
    umma::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
        // every tile claimed by this CTA precedes its arrival; the last CTA to arrive resets both counters
        __threadfence();
        if (atomicAdd(ctr + 1, 1u) == gridDim.x - 1) {
            atomicExch(ctr, 0u);
            atomicExch(ctr + 1, 0u);
        }
    }
    if (tid < 32) {
        umma::fence_after_sync();
        umma::tmem_dealloc(S.tmem, 128u * H);
    }
}

}  // namespace gdev
}  // namespace qsim
