// Gate passes on FP32 CUDA cores (sm_103a).
//
// The state update of Sec. 2.1 multiplies, for every index group that agrees
// outside the target bits, the 2^k amplitudes of the group by the gate matrix.
// Here a stage's gates arrive fused into dense ops of <= k qubits (plus
// diagonal phase ops and phase flips). A pass loads one tile of 2^T
// amplitudes of the working vector into shared memory (the tile's low bits
// are contiguous working-index bits, so the loads are coalesced), applies
// every op of the pass in shared memory, and stores the tile back: one read
// and one write of the working vector per pass instead of one per gate.
//
// Shared memory layout is XOR-swizzled (bits 4-7, 8-11, 12-15 folded into the
// low four bits of the float2 index) so that the lanes of a warp, which walk
// different index groups, hit different banks.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <map>
#include <mutex>

#include "codec.cuh"
#include "device_common.cuh"
#include "gates.cuh"
#include "gates_dev.cuh"
#include "gates_reg.cuh"

namespace qsim {

namespace {

using namespace gdev;
constexpr int NT = 128;
constexpr int kPassSmemMost = 220 * 1024;  // dynamic shared memory of a pass, 6 KB of PassSmem beside it

// One wave of resident CTAs, each looping over tiles of all the launch's groups
// (one tile buffer per CTA; several resident CTAs per SM keep loads, ops and
// stores of different tiles in flight). The pass set-up, the pass blob, TMEM
// and a single tcgen05 op's B operand are staged once per CTA rather than once
// per tile. (A variant with two tile buffers per CTA and cp.async prefetch of
// the next tile ran slower on GB300: fewer resident CTAs, 3.1 against 4.3 TB/s
// on load/store-only passes.)
// UM: the pass's k = 5 dense ops run on tcgen05 (a separate instantiation, so that the warp-MMA kernels
// keep their own register allocation)
// Teams of 128 threads per CTA, a tile each, at most. On CUDA cores four share one pass blob: a blob of many ops (56 KB
// in the 28-op passes of a random circuit) beside every 32 KB tile left two tiles, 8 warps, per SM; four tiles beside one
// blob are the 16 warps that 128 registers a thread allow (26-qubit random brick in FP32 with the groups of
// apply_dense_groups: 21.8 -> 18.2 ms; four teams of 64 threads with twice the groups: 22.1). One team per CTA elsewhere:
// width 6 takes 255 registers, the tcgen05 forms size TMEM and B by the tile, and the warp-level MMAs hold their matrix
// in registers, where a team's own tile, barrier and counters cost spills (whole runs of 26 qubits, several teams and
// one: random brick in TF32 at width 5 13.2 and 11.75 ms, at width 3 16.8 and 15.6, in split BF16 at width 5 21.7 and
// 19.3, at width 4 19.6 and 17.5; QFT in split BF16 21.4 and 18.8).
template <int KMAX, int PREC, bool UM>
__host__ __device__ constexpr int pass_teams() {
    return UM || KMAX >= 6 || PREC != QSIM_PREC_FP32 ? 1 : 4;
}
// CTAs of one team that fit an SM by registers
template <int KMAX, int PREC, bool UM>
__host__ __device__ constexpr int pass_min_blocks() {
    return pass_teams<KMAX, PREC, UM>() > 1 ? 1 : KMAX >= 6 ? 2 : (PREC == QSIM_PREC_BF16X3 && KMAX >= 4) ? 3 : 4;
}

template <int KMAX, int PREC, bool UM>
__global__ void __launch_bounds__(NT * pass_teams<KMAX, PREC, UM>(), pass_min_blocks<KMAX, PREC, UM>())
    k_pass(float2 *__restrict__ wv, uint32_t W, uint64_t ntiles, const __grid_constant__ PassDev P,
           const uint4 *__restrict__ blob, const float2 *__restrict__ mats, const uint32_t *__restrict__ bfr,
           const uint64_t *__restrict__ gbase, uint32_t *ctr, int *status) {
    extern __shared__ float4 dyn_smem[];
    constexpr int TEAMS = pass_teams<KMAX, PREC, UM>();
    __shared__ PassSmem S[TEAMS];
    pass_tiles<NT, KMAX, PREC, UM, TEAMS>(wv, W, ntiles, P, blob, mats, bfr, gbase, S[threadIdx.x / NT],
                                          reinterpret_cast<float2 *>(dyn_smem), ctr, status);
}

// Resident CTAs per SM of one k_pass instantiation at a given dynamic shared memory size (cached), from the
// kernel's registers and static shared memory and the SM's limits (65536 registers, 2048 threads, 32 CTAs,
// 228 KB of shared memory with 1 KB reserved per CTA). (The runtime's occupancy query answered 1 here where
// 4 CTAs per SM were resident.)
template <int KMAX, int PREC, bool UM>
int pass_blocks_per_sm(size_t smem, int nt) {
    static std::mutex mu;
    static std::map<std::pair<size_t, int>, int> cache;
    std::lock_guard<std::mutex> lk(mu);
    const std::pair<size_t, int> key(smem, nt);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    cudaFuncAttributes fa{};
    int nb = 1;
    if (cudaFuncGetAttributes(&fa, k_pass<KMAX, PREC, UM>) == cudaSuccess) {
        const int regs = ((fa.numRegs > 0 ? fa.numRegs : 255) + 7) & ~7;
        const int by_regs = 65536 / (regs * nt);
        const int by_smem = int((228u * 1024u) / (smem + fa.sharedSizeBytes + 1024u));
        nb = std::max(1, std::min(std::min(by_regs, by_smem), std::min(2048 / nt, 32)));
    }
    cache[key] = nb;
    return nb;
}

template <int KMAX, int PREC, bool UM>
void launch_pass_ku(dim3 grid, cudaStream_t s, float2 *wv, uint32_t W, const PassDev &P, const uint4 *blob,
                    const float2 *mats, const uint32_t *bfr, const uint64_t *gbase, uint32_t *ctr, int *status) {
    allow_smem<k_pass<KMAX, PREC, UM>>(kPassSmemMost, true);  // the resident CTAs are limited by their tiles
    int teams = pass_teams<KMAX, PREC, UM>();
    while (teams > 1 && pass_smem_bytes(P, teams) > size_t(kPassSmemMost)) --teams;  // tiles of 2^13 amplitudes
    const size_t smem = pass_smem_bytes(P, teams);
    // grid.x tiles per group, grid.y groups: the resident CTAs loop over all of them. The grid is twice the
    // resident count so that an underestimate of it cannot leave SMs short of CTAs (measured on the 32-qubit
    // QAOA passes: one CTA per SM 0.85 ms, one resident wave 0.41 ms, two 0.41 ms, one tile per CTA 0.46 ms);
    // CTAs that start after the tiles have run out leave at once. CTAs of several teams: one wave.
    const uint64_t ntiles = uint64_t(grid.x) * grid.y;
    const uint64_t resident = (teams > 1 ? 1ull : 2ull) * uint64_t(pass_blocks_per_sm<KMAX, PREC, UM>(smem, NT * teams)) * num_sms();
    const uint32_t nctas = uint32_t(ntiles < resident ? ntiles : resident);
    k_pass<KMAX, PREC, UM><<<nctas, NT * teams, smem, s>>>(wv, W, ntiles, P, blob, mats, bfr, gbase, ctr, status);
}

template <int KMAX, int PREC>
void launch_pass_k(dim3 grid, cudaStream_t s, float2 *wv, uint32_t W, const PassDev &P,
                   const uint4 *blob, const float2 *mats, const uint32_t *bfr, const uint64_t *gbase, uint32_t *ctr,
                   int *status) {
    if constexpr ((PREC == QSIM_PREC_TF32 || PREC == QSIM_PREC_BF16X3) && KMAX >= 5) {
        if (P.umma) {
            launch_pass_ku<KMAX, PREC, true>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status);
            return;
        }
    }
    launch_pass_ku<KMAX, PREC, false>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status);
}

template <int PREC, int H>
__global__ void __launch_bounds__(128 * H, 4 / H)
    k_pass_reg(float2 *__restrict__ wv, uint32_t W, uint64_t ntiles, const __grid_constant__ PassDev P,
               const uint4 *__restrict__ blob, const uint32_t *__restrict__ bfr, const uint64_t *__restrict__ gbase,
               uint32_t *ctr, int *status) {
    extern __shared__ float4 dyn_smem[];
    __shared__ RegSmem<H> S;
    pass_reg_tiles<PREC, H>(wv, W, ntiles, P, blob, bfr, gbase, S, reinterpret_cast<uint8_t *>(dyn_smem), ctr, status);
}

// Shared memory a CTA of k_pass_reg may take for two (H = 2) to be resident: 228 KB per SM, 1 KB reserved per CTA, and
// RegSmem.
constexpr uint32_t kRegSmemTwo = 228u * 512u - 1024u - uint32_t(sizeof(RegSmem<2>)) - 64u;

// Two tiles per CTA when every dense op's B operand fits beside them at two CTAs per SM (four tiles in flight, B read
// once per CTA); else one tile per CTA and B reloaded per op.
template <int PREC>
bool reg_two(const PassDev &P) {
    return reg_shape<PREC, 2>(P.reg_dense, P.reg_poly, P.reg_flags, P.reg_words).bytes <= kRegSmemTwo;
}

template <int PREC, int H>
void launch_reg(uint64_t ntiles, cudaStream_t s, float2 *wv, uint32_t W, const PassDev &P, const uint4 *blob,
                const uint32_t *bfr, const uint64_t *gbase, uint32_t *ctr, int *status) {
    allow_smem<k_pass_reg<PREC, H>>(200 * 1024, true);
    const uint32_t smem = reg_shape<PREC, H>(P.reg_dense, P.reg_poly, P.reg_flags, P.reg_words).bytes;
    const uint64_t by_smem = (228u * 1024u) / (smem + sizeof(RegSmem<H>) + 1024u);
    const uint64_t per_sm = std::max<uint64_t>(1, std::min<uint64_t>(by_smem, 4 / H));
    // twice the resident CTAs, as launch_pass_ku
    const uint64_t want = (ntiles + H - 1) / H, resident = 2 * per_sm * num_sms();
    k_pass_reg<PREC, H><<<unsigned(std::min(want, resident)), 128 * H, smem, s>>>(wv, W, ntiles, P, blob, bfr, gbase,
                                                                                 ctr, status);
}

template <int PREC>
void launch_reg_prec(uint64_t ntiles, cudaStream_t s, float2 *wv, uint32_t W, const PassDev &P, const uint4 *blob,
                     const uint32_t *bfr, const uint64_t *gbase, uint32_t *ctr, int *status) {
    if (reg_two<PREC>(P)) launch_reg<PREC, 2>(ntiles, s, wv, W, P, blob, bfr, gbase, ctr, status);
    else launch_reg<PREC, 1>(ntiles, s, wv, W, P, blob, bfr, gbase, ctr, status);
}

template <int PREC>
void launch_pass_prec(uint32_t kmax, dim3 grid, cudaStream_t s, float2 *wv, uint32_t W,
                      const PassDev &P, const uint4 *blob, const float2 *mats, const uint32_t *bfr,
                      const uint64_t *gbase, uint32_t *ctr, int *status) {
    switch (kmax) {
        case 0: launch_pass_k<0, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
        case 1: launch_pass_k<1, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
        case 2: launch_pass_k<2, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
        case 3: launch_pass_k<3, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
        case 4: launch_pass_k<4, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
        case 5: launch_pass_k<5, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
        default: launch_pass_k<6, PREC>(grid, s, wv, W, P, blob, mats, bfr, gbase, ctr, status); break;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host: B-fragment tables
// ---------------------------------------------------------------------------
static uint32_t f32_bits(float f) {
    uint32_t u;
    memcpy(&u, &f, 4);
    return u;
}
static float bits_f32(uint32_t u) {
    float f;
    memcpy(&f, &u, 4);
    return f;
}
// round to TF32 (10 explicit mantissa bits), nearest with ties away from zero
static uint32_t to_tf32(float x) { return (f32_bits(x) + 0x1000u) & ~0x1FFFu; }
// round to BF16, nearest even
static uint16_t to_bf16(float x) {
    const uint32_t u = f32_bits(x);
    return uint16_t((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
}
static float from_bf16(uint16_t h) { return bits_f32(uint32_t(h) << 16); }

size_t bfrag_words(uint32_t k, int prec) {
    const size_t n2 = size_t(2) << k;
    return prec == QSIM_PREC_TF32 ? n2 * n2 : 3 * n2 * n2 / 2;
}

void build_bfrag_table(const double *u, uint32_t k, int prec, uint32_t *out) {
    const uint32_t D = 1u << k, N2 = 2 * D, NTILES = N2 / 8;
    // U_r^T[kk][n] = U_r[n][kk] as float
    auto ur = [&](uint32_t n, uint32_t kk) -> float {
        const uint32_t r = n % D, c = kk % D;
        const double re = u[2 * (size_t(r) * D + c)], im = u[2 * (size_t(r) * D + c) + 1];
        if (n < D) return float(kk < D ? re : -im);
        return float(kk < D ? im : re);
    };
    if (prec == QSIM_PREC_TF32) {
        const uint32_t KS = N2 / 8;
        for (uint32_t ks = 0; ks < KS; ++ks)
            for (uint32_t nt = 0; nt < NTILES; ++nt)
                for (uint32_t lane = 0; lane < 32; ++lane) {
                    const uint32_t g = lane / 4, t = lane % 4;
                    uint32_t *o = out + ((size_t(ks) * NTILES + nt) * 32 + lane) * 2;
                    o[0] = to_tf32(ur(nt * 8 + g, ks * 8 + t));
                    o[1] = to_tf32(ur(nt * 8 + g, ks * 8 + t + 4));
                }
        return;
    }
    const uint32_t KS = N2 / 16;
    const size_t part = size_t(KS) * NTILES * 32 * 2;
    for (uint32_t ks = 0; ks < KS; ++ks)
        for (uint32_t nt = 0; nt < NTILES; ++nt)
            for (uint32_t lane = 0; lane < 32; ++lane) {
                const uint32_t g = lane / 4, t = lane % 4;
                for (int r = 0; r < 2; ++r) {
                    uint16_t h[2], m[2], l[2];
                    for (int q = 0; q < 2; ++q) {
                        const float x = ur(nt * 8 + g, ks * 16 + 2 * t + q + 8 * r);
                        h[q] = to_bf16(x);
                        const float r1 = x - from_bf16(h[q]);
                        m[q] = to_bf16(r1);
                        l[q] = to_bf16(r1 - from_bf16(m[q]));
                    }
                    const size_t e = ((size_t(ks) * NTILES + nt) * 32 + lane) * 2 + r;
                    out[e] = uint32_t(h[0]) | (uint32_t(h[1]) << 16);
                    out[part + e] = uint32_t(m[0]) | (uint32_t(m[1]) << 16);
                    out[2 * part + e] = uint32_t(l[0]) | (uint32_t(l[1]) << 16);
                }
            }
}

size_t umma_pass_smem(uint32_t umma_bits) {
    return (umma_bits & 1u) ? size_t(umma_pass_b_bytes(umma_bits)) + 1024 : 0;
}

size_t pass_smem_bytes(const PassDev &P, int teams) {
    const size_t um = umma_pass_smem(P.umma);
    return (size_t(teams) << P.T) * sizeof(float2) + um + size_t(P.blob_words) * 16 +
           size_t(teams) * P.mat_elems * sizeof(float2);
}

// A pass takes the register form while three CTAs of its reload form fit an SM (75 KB each). Past that two tiles would be
// in flight where the staged form keeps three. The line goes by the tiles in flight: no plan of the benchmark's circuits
// reaches it (their fullest passes, three ops and one run, take 1.53 ms per 2^28 amplitudes against 1.55 staged).
bool reg_pass_fits(const PassDev &P, int prec) {
    constexpr uint32_t most = 228u * 1024u / 3u - 1024u - uint32_t(sizeof(RegSmem<1>)) - 64u;
    if (prec == QSIM_PREC_TF32)
        return reg_two<QSIM_PREC_TF32>(P) ||
               reg_shape<QSIM_PREC_TF32, 1>(P.reg_dense, P.reg_poly, P.reg_flags, P.reg_words).bytes <= most;
    return prec == QSIM_PREC_BF16X3 &&
           (reg_two<QSIM_PREC_BF16X3>(P) ||
            reg_shape<QSIM_PREC_BF16X3, 1>(P.reg_dense, P.reg_poly, P.reg_flags, P.reg_words).bytes <= most);
}

void build_umma_b(const double *u, uint32_t *out) {
    constexpr uint32_t D = 32;
    for (uint32_t n = 0; n < 2 * D; ++n)
        for (uint32_t kk = 0; kk < 2 * D; ++kk) {
            const uint32_t r = n % D, c = kk % D;
            const double re = u[2 * (size_t(r) * D + c)], im = u[2 * (size_t(r) * D + c) + 1];
            const double v = n < D ? (kk < D ? re : -im) : (kk < D ? im : re);
            const uint32_t a = kk / 32, ch = (kk % 32) / 4, w = kk % 4;
            const size_t byte = size_t(a) * 8192 + (n / 8) * 1024 + (n % 8) * 128 + ((ch ^ (n % 8)) * 16) + w * 4;
            out[byte / 4] = to_tf32(float(v));
        }
}

void build_umma_b6(const double *u, uint32_t *out) {
    constexpr uint32_t D = 64;
    for (uint32_t n = 0; n < 2 * D; ++n)
        for (uint32_t kk = 0; kk < 2 * D; ++kk) {
            const uint32_t r = n % D, c = kk % D;
            const double re = u[2 * (size_t(r) * D + c)], im = u[2 * (size_t(r) * D + c) + 1];
            const double v = n < D ? (kk < D ? re : -im) : (kk < D ? im : re);
            const uint32_t a = kk / 32, ch = (kk % 32) / 4, w = kk % 4;
            const size_t byte = size_t(a) * 16384 + (n / 8) * 1024 + (n % 8) * 128 + ((ch ^ (n % 8)) * 16) + w * 4;
            out[byte / 4] = to_tf32(float(v));
        }
}

void build_umma_b3(const double *u, uint32_t *out) {
    constexpr uint32_t D = 32;
    uint16_t *o16 = reinterpret_cast<uint16_t *>(out);
    for (uint32_t n = 0; n < 2 * D; ++n)
        for (uint32_t kk = 0; kk < 2 * D; ++kk) {
            const uint32_t r = n % D, c = kk % D;
            const double re = u[2 * (size_t(r) * D + c)], im = u[2 * (size_t(r) * D + c) + 1];
            const float x = float(n < D ? (kk < D ? re : -im) : (kk < D ? im : re));
            const uint16_t h = to_bf16(x);
            const float r1 = x - from_bf16(h);
            const uint16_t m = to_bf16(r1);
            const uint16_t l = to_bf16(r1 - from_bf16(m));
            const uint32_t ch = kk / 8, w = kk % 8;
            const size_t off = (n / 8) * 1024 + (n % 8) * 128 + ((ch ^ (n % 8)) * 16) + w * 2;  // bytes in a part
            o16[(0 * 8192 + off) / 2] = h;
            o16[(1 * 8192 + off) / 2] = m;
            o16[(2 * 8192 + off) / 2] = l;
        }
}

void launch_pass(float2 *wv, uint32_t W, uint32_t ngroups, const PassDev *pass_host, const uint4 *blob_dev,
                 const float2 *mats_dev, const uint32_t *bfr_dev, const uint64_t *gbase_dev, int prec,
                 cudaStream_t s, uint32_t *ctr, int *status) {
    const PassDev &P = *pass_host;
    if (P.reg_words) {
        const uint64_t ntiles = uint64_t(ngroups) << P.nout;
        if (prec == QSIM_PREC_TF32)
            launch_reg_prec<QSIM_PREC_TF32>(ntiles, s, wv, W, P, blob_dev, bfr_dev, gbase_dev, ctr, status);
        else
            launch_reg_prec<QSIM_PREC_BF16X3>(ntiles, s, wv, W, P, blob_dev, bfr_dev, gbase_dev, ctr, status);
        count_launch();
        return;
    }
    dim3 grid(1u << P.nout, ngroups);
    const uint32_t kmax = P.kmax;
    if (prec == QSIM_PREC_TF32 && kmax >= 3)
        launch_pass_prec<QSIM_PREC_TF32>(kmax, grid, s, wv, W, P, blob_dev, mats_dev, bfr_dev, gbase_dev, ctr, status);
    else if (prec == QSIM_PREC_BF16X3 && kmax >= 3)
        launch_pass_prec<QSIM_PREC_BF16X3>(kmax, grid, s, wv, W, P, blob_dev, mats_dev, bfr_dev, gbase_dev, ctr, status);
    else
        launch_pass_prec<QSIM_PREC_FP32>(kmax, grid, s, wv, W, P, blob_dev, mats_dev, bfr_dev, gbase_dev, ctr, status);
    count_launch();
}

}  // namespace qsim
