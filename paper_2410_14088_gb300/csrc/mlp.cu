// Learned block-size predictor: a 41 -> 64 -> 64 -> 1 ReLU MLP, with its own
// forward, loss/gradient and Adam kernels (sm_103a).
//
// The paper handles the unpredictable size of compressed blocks with a second
// memory level (Sec. 4.4). Here the size of each block's next stream is
// predicted from cheap statistics so that a slot can be reserved before the
// block is encoded; a block whose size was under-estimated gets a slot of its
// exact size.
//
// Inputs (x, 41 floats): the 32-bin histogram of code bit lengths
// (bit length of |q|, as fractions of the 2^(m+1) values of each block of the
// block's SV group, which the stage mixes), the largest bit length / 32, and
// 8 stage features. Output: log2(stream bytes) - (m + 3),
// i.e. minus the log2 of the block's compression ratio.
// Parameter layout (6913 floats): W1[64][41], b1[64], W2[64][64], b2[64],
// W3[64], b3.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "codec.cuh"
#include "device_common.cuh"
#include "mlp.cuh"

namespace qsim {

namespace {

constexpr int IN = kMlpIn, HID = kMlpHidden, NP = kMlpParams;
constexpr int OW1 = 0, OB1 = OW1 + HID * IN, OW2 = OB1 + HID, OB2 = OW2 + HID * HID, OW3 = OB2 + HID,
              OB3 = OW3 + HID;

__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ void load_weights(float *w, const float *params, bool bf16) {
    for (int i = threadIdx.x; i < NP; i += blockDim.x) w[i] = bf16 ? round_bf16(params[i]) : params[i];
}

__global__ void k_mlp_forward(const float *__restrict__ params, const float *__restrict__ x, uint32_t batch,
                              float *__restrict__ y, int bf16) {
    __shared__ float w[NP];
    load_weights(w, params, bf16 != 0);
    __syncthreads();
    for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < batch; b += gridDim.x * blockDim.x) {
        float xs[IN];
        for (int j = 0; j < IN; ++j) xs[j] = x[uint64_t(b) * IN + j];
        y[b] = mlp_forward_one(w, xs);
    }
}

// Features of each block of a batch from the decoder's bit-length histogram,
// then the prediction; optionally the features are also written out (for
// the training log, completed by the target once the exact size is known).
// One warp per block: the features (the SV group's width histogram, the largest
// populated bin, the stage features), then the forward pass with the hidden
// units spread over the lanes (two per lane per layer).
__global__ void __launch_bounds__(128) k_predict_sizes(const uint32_t *__restrict__ hist, uint32_t nblocks,
                                                       uint32_t G, int m, StageFeatures sf,
                                                       const float *__restrict__ params, int bf16,
                                                       float *__restrict__ pred, float *__restrict__ feat_out) {
    __shared__ float w[NP];
    __shared__ float xs[4][IN + 1];
    __shared__ float hs[4][HID];
    if (params) load_weights(w, params, bf16 != 0);
    __syncthreads();
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const float inv = 1.0f / (float(G) * float(2ull << m));
    for (uint32_t j = blockIdx.x * 4 + wi; j < nblocks; j += gridDim.x * 4) {
        // a stage mixes the G blocks of an SV group, so the histogram is the group's
        const uint64_t g0 = uint64_t(j / G) * G;
        uint32_t c = 0;
        for (uint32_t jj = 0; jj < G; ++jj) c += __ldcg(hist + (g0 + jj) * 32 + lane);
        const uint32_t nz = __ballot_sync(0xffffffffu, c != 0);
        xs[wi][lane] = float(c) * inv;
        if (lane == 0) xs[wi][32] = float(nz ? 31 - __clz(nz) : 0) / 32.f;
        if (lane < 8) xs[wi][33 + lane] = sf.v[lane];
        __syncwarp();
        if (feat_out)
            for (int t = lane; t < IN; t += 32) feat_out[uint64_t(j) * (IN + 1) + t] = xs[wi][t];
        if (params && pred) {
            float a0 = w[OB1 + lane], a1 = w[OB1 + lane + 32];
            for (int t = 0; t < IN; ++t) {
                const float x = xs[wi][t];
                a0 = fmaf(w[OW1 + lane * IN + t], x, a0);
                a1 = fmaf(w[OW1 + (lane + 32) * IN + t], x, a1);
            }
            hs[wi][lane] = fmaxf(a0, 0.f);
            hs[wi][lane + 32] = fmaxf(a1, 0.f);
            __syncwarp();
            float b0 = w[OB2 + lane], b1 = w[OB2 + lane + 32];
            for (int t = 0; t < HID; ++t) {
                const float h = hs[wi][t];
                b0 = fmaf(w[OW2 + lane * HID + t], h, b0);
                b1 = fmaf(w[OW2 + (lane + 32) * HID + t], h, b1);
            }
            float y = w[OW3 + lane] * fmaxf(b0, 0.f) + w[OW3 + lane + 32] * fmaxf(b1, 0.f);
#pragma unroll
            for (int o = 16; o; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
            if (lane == 0) pred[j] = y + w[OB3] + float(m + 3);
        }
        __syncwarp();
    }
}

// Writes the training target log2(bytes) - (m + 3) beside each logged feature row.
__global__ void k_log_targets(const EncResult *__restrict__ res, uint32_t nblocks, int m, float *__restrict__ rows) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < nblocks) rows[uint64_t(j) * (IN + 1) + IN] = log2f(float(res[j].total)) - float(m + 3);
}

// ---------------------------------------------------------------------------
// Training. One cluster of eight CTAs runs a whole sequence of steps. A batch is taken in chunks of 64 samples: each CTA
// takes eight of them through the forward and backward pass with its own copy of the weights in shared memory, then every
// CTA collects what its eighth of the weight rows needs of all 64 through distributed shared memory, sums the gradient
// of those rows over the samples, applies Adam to them, whose moments it keeps in registers, and writes the new weights
// into all eight copies. Two cluster barriers per chunk, no launch and no global round trip. Every sum that the weights
// depend on runs in the order of a loop over its terms: inputs, units, and samples within a chunk, whose sums are added
// in the chunks' order. A training run amplifies the rounding of its first steps, so a sum split over threads or CTAs
// ends in other weights. (The reported loss is no such sum: k_mlp_loss adds its CTAs' shares in any order, in FP64.) A step of 64 samples is 1.3 MFLOP in a chain of six dependent phases:
// latency and shared-memory reads bound it. 800 steps of 64 samples: 72 ms with two launches and one CTA per step,
// 8.3 ms now (the call).
// ---------------------------------------------------------------------------
constexpr int CR = 8;                            // CTAs of the cluster
constexpr int SB = 8;                            // samples a CTA takes at a time
constexpr int CH = CR * SB;                      // of a chunk
constexpr int TT = 256;                          // threads
constexpr int RW = HID / CR;                     // weight rows a CTA owns, one per warp
constexpr int XS = 44, W2S = HID + 4, H2S = HID + 4;  // words of a row: eight rows' 16-byte reads fall on all banks
static_assert(XS >= IN && RW == TT / 32 && IN > 32 && IN <= 32 + 9, "a warp's lanes cover a row of W1 in two rounds");

struct __align__(16) TrainParams {
    float w1[HID * XS], b1[HID], w2[HID * W2S], b2[HID], w3[HID], b3[4];
};
struct __align__(16) TrainSmem : TrainParams {
    // this CTA's samples
    float x[SB][XS], h1[SB][HID], h2[SB][H2S], d1[SB][HID], d2[SB][HID], dy[SB], t[SB], sq[SB];
    // the chunk's, where it is about this CTA's weight rows by row
    float ax[CH][XS], ah1[CH][HID], at1[RW][CH], at2[RW][CH], ah2[RW][CH], ady[CH];
    float one[4];
    float loss;
};

// parameter i's place in a TrainParams, in floats
__device__ __forceinline__ int train_place(int i) {
    constexpr int P1 = HID * XS, P2 = P1 + HID, P3 = P2 + HID * W2S;
    if (i < OB1) return i / IN * XS + i % IN;
    if (i < OW2) return P1 + (i - OB1);
    if (i < OB2) return P2 + (i - OW2) / HID * W2S + (i - OW2) % HID;
    return P3 + (i - OB2);  // b2, W3 and b3 follow one another
}
__device__ __forceinline__ float *train_flat(TrainParams &p) { return reinterpret_cast<float *>(&p); }

__device__ __forceinline__ void train_load(TrainSmem &S, const float *params) {
    for (int i = threadIdx.x; i < SB * XS; i += TT) S.x[0][i] = 0.f;  // the rows' ends too
    if (threadIdx.x == 0) S.one[0] = 1.f, S.loss = 0.f;
    float *w = train_flat(S);
    for (int i = threadIdx.x; i < NP; i += TT) w[train_place(i)] = params[i];
    __syncthreads();
}

// The rows of the samples a CTA takes at once, two values per thread (IN features and the target per sample), held in
// registers so that a step's rows are on their way while the step before it is computed: first where they are (the
// sample order is a load of its own), half a step later the rows.
struct TrainRows {
    float v[2];
};
struct TrainAt {
    uint64_t s[2];
    uint32_t n;
};
__device__ __forceinline__ TrainAt train_at(const uint32_t *perm, uint64_t first, uint32_t n) {
    TrainAt a{{0, 0}, n};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t b = (threadIdx.x + TT * k) / (IN + 1);
        if (b < n && b < uint32_t(SB)) a.s[k] = perm ? __ldg(perm + first + b) : first + b;
    }
    return a;
}
__device__ __forceinline__ TrainRows train_fetch(const float *x, uint32_t xstride, const float *t, uint32_t tstride,
                                                 const TrainAt &a) {
    TrainRows r{{0.f, 0.f}};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t i = threadIdx.x + TT * k, b = i / (IN + 1), j = i % (IN + 1);
        if (b < a.n && b < uint32_t(SB))
            r.v[k] = j < uint32_t(IN) ? __ldg(x + a.s[k] * xstride + j) : __ldg(t + a.s[k] * tstride);
    }
    return r;
}
__device__ __forceinline__ void train_put(TrainSmem &S, const TrainRows &r) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t i = threadIdx.x + TT * k, b = i / (IN + 1), j = i % (IN + 1);
        if (b >= uint32_t(SB)) continue;
        if (j < uint32_t(IN)) S.x[b][j] = r.v[k];
        else S.t[b] = r.v[k];
    }
}

__device__ __forceinline__ float train_fma4(const float4 &a, const float4 &b, float c) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

// Forward pass of the n (<= SB) samples in S.x; each sample's residual y - t to S.dy (0 past n). A thread takes one unit
// of two samples. Ends unsynchronised: thread b wrote sample b's.
__device__ __forceinline__ void train_forward(TrainSmem &S, uint32_t n) {
    const int tid = threadIdx.x, h = tid & (HID - 1), q = tid / HID;
    float a0 = S.b1[h], a1 = a0;
    const float *w = S.w1 + h * XS;
#pragma unroll
    for (int j = 0; j < IN / 4 * 4; j += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(w + j);
        a0 = train_fma4(v, *reinterpret_cast<const float4 *>(&S.x[q][j]), a0);
        a1 = train_fma4(v, *reinterpret_cast<const float4 *>(&S.x[q + 4][j]), a1);
    }
#pragma unroll
    for (int j = IN / 4 * 4; j < IN; ++j) {
        a0 = fmaf(w[j], S.x[q][j], a0);
        a1 = fmaf(w[j], S.x[q + 4][j], a1);
    }
    S.h1[q][h] = fmaxf(a0, 0.f);
    S.h1[q + 4][h] = fmaxf(a1, 0.f);
    __syncthreads();
    a0 = a1 = S.b2[h];
    w = S.w2 + h * W2S;
#pragma unroll
    for (int j = 0; j < HID; j += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(w + j);
        a0 = train_fma4(v, *reinterpret_cast<const float4 *>(&S.h1[q][j]), a0);
        a1 = train_fma4(v, *reinterpret_cast<const float4 *>(&S.h1[q + 4][j]), a1);
    }
    S.h2[q][h] = fmaxf(a0, 0.f);
    S.h2[q + 4][h] = fmaxf(a1, 0.f);
    __syncthreads();
    if (tid < SB) {
        float y = S.b3[0];
#pragma unroll
        for (int j = 0; j < HID; j += 4)
            y = train_fma4(*reinterpret_cast<const float4 *>(S.w3 + j), *reinterpret_cast<const float4 *>(&S.h2[tid][j]), y);
        S.dy[tid] = uint32_t(tid) < n ? y - S.t[tid] : 0.f;
    }
}

// Forward and backward pass of the n samples in S.x (inv_b: 1 / the batch's samples); `half` is called in between.
template <class F>
__device__ __forceinline__ void train_samples(TrainSmem &S, uint32_t n, float inv_b, F half) {
    const int tid = threadIdx.x, h = tid & (HID - 1), q = tid / HID;
    train_forward(S, n);
    if (tid < SB) {
        const float r = S.dy[tid];
        S.dy[tid] = r * inv_b;
        S.sq[tid] = 0.5f * r * r * inv_b;
    }
    half();
    __syncthreads();
#pragma unroll
    for (int b = q; b < SB; b += 4) S.d2[b][h] = S.h2[b][h] > 0.f ? S.dy[b] * S.w3[h] : 0.f;
    __syncthreads();
    float a0 = 0.f, a1 = 0.f;  // back through W2
#pragma unroll
    for (int i = 0; i < HID; i += 4) {
        const float4 w = make_float4(S.w2[i * W2S + h], S.w2[(i + 1) * W2S + h], S.w2[(i + 2) * W2S + h],
                                     S.w2[(i + 3) * W2S + h]);
        a0 = train_fma4(*reinterpret_cast<const float4 *>(&S.d2[q][i]), w, a0);
        a1 = train_fma4(*reinterpret_cast<const float4 *>(&S.d2[q + 4][i]), w, a1);
    }
    S.d1[q][h] = S.h1[q][h] > 0.f ? a0 : 0.f;
    S.d1[q + 4][h] = S.h1[q + 4][h] > 0.f ? a1 : 0.f;
}

// `total` samples in the order of perm (null: as they are), `batch` per step; TRAIN: Adam's step number t0 + 1 and on,
// params, m1 and m2 updated at the end. Else one batch of all samples: gradient and loss.
template <bool TRAIN>
__global__ void __cluster_dims__(CR, 1, 1) __launch_bounds__(TT, 1)
    k_mlp_train(float *__restrict__ params, const float *__restrict__ x, uint32_t xstride, const float *__restrict__ t,
                uint32_t tstride, const uint32_t *__restrict__ perm, uint64_t total, uint32_t epoch, uint32_t batch,
                float *__restrict__ m1, float *__restrict__ m2, int t0, float lr, float beta1, float beta2, float eps,
                float *__restrict__ grad, float *__restrict__ loss_out) {
    extern __shared__ __align__(16) uint8_t train_smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(train_smem);
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const uint32_t rank = cl.block_rank();
    const int tid = threadIdx.x, row = tid >> 5, lane = tid & 31, unit = RW * int(rank) + row;
    train_load(S, params);
    // the thread's parameters, of weight rows `unit`: two neighbours of W2, one of W1, and one of the row's end of W1, of
    // b2, b1, W3 or b3
    int own[4] = {OW2 + unit * HID + 2 * lane, OW2 + unit * HID + 2 * lane + 1, OW1 + unit * IN + lane, -1};
    if (lane < IN - 32) own[3] = OW1 + unit * IN + 32 + lane;
    else if (lane == 9) own[3] = OB2 + unit;
    else if (lane == 10) own[3] = OB1 + unit;
    else if (lane == 11) own[3] = OW3 + unit;
    else if (lane == 12 && unit == 0) own[3] = OB3;
    // the last one's factors by sample
    const float *pf = lane == 9 ? S.at2[row] : lane == 11 || lane == 12 ? S.ady : S.at1[row];
    const float *qf = lane < IN - 32 ? &S.ax[0][32 + lane] : lane == 11 ? S.ah2[row] : S.one;
    const int qs = lane < IN - 32 ? XS : lane == 11 ? 1 : 0;
    int place[4];
    float p[4] = {}, ma[4] = {}, mb[4] = {}, g[4] = {};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        place[k] = train_place(max(own[k], 0));
        if (own[k] < 0) continue;
        p[k] = params[own[k]];
        if (TRAIN) {
            ma[k] = m1[own[k]];
            mb[k] = m2[own[k]];
        }
    }
    // batches do not cross epochs: the last one of an epoch may be smaller
    uint64_t pos = 0;
    uint32_t in_epoch = 0;
    int step = t0;
    auto batch_at = [&](uint32_t e) { return min(batch, epoch - e); };
    // this CTA's samples of the chunk that starts `left` samples before its batch's end
    auto share = [&](uint32_t left) { return left > SB * rank ? min(left - SB * rank, uint32_t(SB)) : 0u; };
    TrainRows next = train_fetch(x, xstride, t, tstride, train_at(perm, SB * rank, share(batch_at(0))));
    cl.sync();
    while (pos < total) {
        const uint32_t nb = batch_at(in_epoch);
        const float inv_b = 1.0f / float(nb);
        const uint64_t npos = pos + nb;
        const uint32_t nin = in_epoch + nb == epoch ? 0u : in_epoch + nb;
#pragma unroll
        for (int k = 0; k < 4; ++k) g[k] = 0.f;
        for (uint32_t c = 0; c < nb; c += CH) {
            if (c) cl.sync();  // every CTA has collected the chunk before
            train_put(S, next);
            __syncthreads();
            TrainAt at{{0, 0}, 0};
            if (c + CH < nb) at = train_at(perm, pos + c + CH + SB * rank, share(nb - c - CH));
            else if (npos < total) at = train_at(perm, npos + SB * rank, share(batch_at(nin)));
            train_samples(S, share(nb - c), inv_b, [&] { next = train_fetch(x, xstride, t, tstride, at); });
            cl.sync();  // every CTA's samples are done
            {           // collect: sample b of the chunk is sample b % SB of CTA b / SB
                float4 vh[CH * HID / 4 / TT], vx[3], vd[3];
#pragma unroll
                for (int k = 0; k < CH * HID / 4 / TT; ++k) {
                    const int i = tid + TT * k, b = i / (HID / 4);
                    vh[k] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(&S.h1[b % SB][i % (HID / 4) * 4], b / SB));
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int i = tid + TT * k, b = i / (XS / 4);
                    if (b < CH)
                        vx[k] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(&S.x[b % SB][i % (XS / 4) * 4], b / SB));
                }
                const int b = (tid / 2) & (CH - 1), o = RW * int(rank) + 4 * (tid & 1);  // threads 0 .. 127
                float yv = 0.f;
                if (tid < 2 * CH) {
                    vd[0] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(&S.d1[b % SB][o], b / SB));
                    vd[1] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(&S.d2[b % SB][o], b / SB));
                    vd[2] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(&S.h2[b % SB][o], b / SB));
                    yv = *cl.map_shared_rank(&S.dy[b % SB], b / SB);
                }
#pragma unroll
                for (int k = 0; k < CH * HID / 4 / TT; ++k)
                    reinterpret_cast<float4 *>(S.ah1[0])[tid + TT * k] = vh[k];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if ((tid + TT * k) / (XS / 4) < CH) reinterpret_cast<float4 *>(S.ax[0])[tid + TT * k] = vx[k];
                if (tid < 2 * CH) {
                    const int r = 4 * (tid & 1);
                    S.at1[r][b] = vd[0].x, S.at1[r + 1][b] = vd[0].y, S.at1[r + 2][b] = vd[0].z, S.at1[r + 3][b] = vd[0].w;
                    S.at2[r][b] = vd[1].x, S.at2[r + 1][b] = vd[1].y, S.at2[r + 2][b] = vd[1].z, S.at2[r + 3][b] = vd[1].w;
                    S.ah2[r][b] = vd[2].x, S.ah2[r + 1][b] = vd[2].y, S.ah2[r + 2][b] = vd[2].z, S.ah2[r + 3][b] = vd[2].w;
                    if (!(tid & 1)) S.ady[b] = yv;
                }
            }
            if (!TRAIN && tid == 0)
                for (int b = 0; b < SB; ++b) S.loss += S.sq[b];
            __syncthreads();
            float a[4] = {};  // samples past the batch's end have zero derivatives
            const int cn = int(min(nb - c, uint32_t(CH)));
#pragma unroll 4
            for (int b = 0; b < cn; ++b) {
                const float2 hv = *reinterpret_cast<const float2 *>(&S.ah1[b][2 * lane]);
                const float e2 = S.at2[row][b];
                a[0] = fmaf(e2, hv.x, a[0]);
                a[1] = fmaf(e2, hv.y, a[1]);
                a[2] = fmaf(S.at1[row][b], S.ax[b][lane], a[2]);
                a[3] = fmaf(pf[b], qf[b * qs], a[3]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) g[k] += a[k];
        }
        ++step;
        const float c1 = TRAIN ? 1.f - powf(beta1, float(step)) : 1.f, c2 = TRAIN ? 1.f - powf(beta2, float(step)) : 1.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (own[k] < 0) continue;
            if (TRAIN) {
                const float gi = g[k];
                const float a = beta1 * ma[k] + (1.f - beta1) * gi;
                const float b = beta2 * mb[k] + (1.f - beta2) * gi * gi;
                ma[k] = a;
                mb[k] = b;
                p[k] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
#pragma unroll
                for (int r = 0; r < CR; ++r) cl.map_shared_rank(train_flat(S), r)[place[k]] = p[k];
            } else {
                grad[own[k]] = g[k];
            }
        }
        cl.sync();  // the new weights are in every copy, the chunk has been collected
        if (!TRAIN && rank == 0 && tid == 0 && loss_out) {
            float ls = 0.f;
            for (int r = 0; r < CR; ++r) ls += *cl.map_shared_rank(&S.loss, r);
            *loss_out = ls;
        }
        pos = npos;
        in_epoch = nin;
    }
    if (!TRAIN) cl.sync();  // no CTA leaves while its loss may be read
    if (TRAIN) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (own[k] >= 0) {
                params[own[k]] = p[k];
                m1[own[k]] = ma[k];
                m2[own[k]] = mb[k];
            }
    }
}

// Loss 0.5/B sum (y - t)^2 over count samples, summed in FP64 (loss: one zero double).
__global__ void __launch_bounds__(TT) k_mlp_loss(const float *__restrict__ params, const float *__restrict__ x,
                                                 uint32_t xstride, const float *__restrict__ t, uint32_t tstride,
                                                 uint64_t count, double *loss) {
    extern __shared__ __align__(16) uint8_t train_smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(train_smem);
    train_load(S, params);
    double sum = 0;
    for (uint64_t c = uint64_t(blockIdx.x) * SB; c < count; c += uint64_t(gridDim.x) * SB) {
        const uint32_t n = uint32_t(min(count - c, uint64_t(SB)));
        train_put(S, train_fetch(x, xstride, t, tstride, train_at(nullptr, c, n)));
        __syncthreads();
        train_forward(S, n);
        __syncthreads();
        if (threadIdx.x == 0)
            for (int b = 0; b < SB; ++b) sum += 0.5 * double(S.dy[b]) * double(S.dy[b]) / double(count);
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, sum);
}

// Adam (Kingma & Ba 2015) with bias correction; t is 1-based.
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m1,
                       float *__restrict__ m2, uint32_t n, int t, float lr, float beta1, float beta2, float eps) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float c1 = 1.f - powf(beta1, float(t)), c2 = 1.f - powf(beta2, float(t));
    const float gi = g[i];
    const float a = beta1 * m1[i] + (1.f - beta1) * gi;
    const float b = beta2 * m2[i] + (1.f - beta2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    p[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
}

}  // namespace

void launch_mlp_forward(const float *params, const float *x, uint32_t batch, float *y, int bf16, cudaStream_t s) {
    const unsigned grid = (batch + 127) / 128;
    k_mlp_forward<<<grid ? grid : 1, 128, 0, s>>>(params, x, batch, y, bf16);
    count_launch();
}

void launch_predict_sizes(const uint32_t *hist, uint32_t nblocks, uint32_t G, int m, const StageFeatures &sf,
                          const float *params, int bf16, float *pred, float *feat_out, cudaStream_t s) {
    const unsigned grid = (nblocks + 3) / 4;
    k_predict_sizes<<<grid ? grid : 1, 128, 0, s>>>(hist, nblocks, G, m, sf, params, bf16, pred, feat_out);
    count_launch();
}

void launch_log_targets(const EncResult *res, uint32_t nblocks, int m, float *rows, cudaStream_t s) {
    k_log_targets<<<(nblocks + 127) / 128, 128, 0, s>>>(res, nblocks, m, rows);
    count_launch();
}

int launch_mlp_loss_grad(const float *params, const float *x, uint32_t xstride, const float *t, uint32_t tstride,
                         uint32_t count, float *grad, float *loss, cudaStream_t s) {
    if (!allow_smem<k_mlp_train<false>>(int(sizeof(TrainSmem)))) return QSIM_E_CUDA;
    k_mlp_train<false><<<CR, TT, sizeof(TrainSmem), s>>>(const_cast<float *>(params), x, xstride, t, tstride, nullptr,
                                                         count, count, count, nullptr, nullptr, 0, 0.f, 0.f, 0.f, 0.f,
                                                         grad, loss);
    count_launch();
    return QSIM_OK;
}

int launch_mlp_train(float *params, const float *rows, uint32_t stride, const uint32_t *perm, uint64_t total,
                     uint32_t epoch, uint32_t batch, float *m1, float *m2, int t0, float lr, float beta1, float beta2,
                     float eps, cudaStream_t s) {
    if (!allow_smem<k_mlp_train<true>>(int(sizeof(TrainSmem)))) return QSIM_E_CUDA;
    k_mlp_train<true><<<CR, TT, sizeof(TrainSmem), s>>>(params, rows, stride, rows + IN, stride, perm, total, epoch,
                                                        batch, m1, m2, t0, lr, beta1, beta2, eps, nullptr, nullptr);
    count_launch();
    return QSIM_OK;
}

int launch_mlp_loss(const float *params, const float *rows, uint32_t stride, uint64_t count, double *loss,
                    cudaStream_t s) {
    if (!allow_smem<k_mlp_loss>(int(sizeof(TrainSmem)))) return QSIM_E_CUDA;
    const uint64_t chunks = (count + SB - 1) / SB;
    k_mlp_loss<<<unsigned(chunks < 304 ? chunks : 304), TT, sizeof(TrainSmem), s>>>(params, rows, stride, rows + IN,
                                                                                   stride, count, loss);
    count_launch();
    return QSIM_OK;
}

void launch_adam(float *p, const float *g, float *m1, float *m2, uint32_t n, int t, float lr, float beta1, float beta2,
                 float eps, cudaStream_t s) {
    k_adam<<<(n + 255) / 256, 256, 0, s>>>(p, g, m1, m2, n, t, lr, beta1, beta2, eps);
    count_launch();
}

}  // namespace qsim
