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
// Training. One cluster of eight CTAs runs a whole sequence of steps: each CTA takes an eighth of a batch's samples
// through the forward and backward pass with its own copy of the weights in shared memory, the gradient is reduced
// through distributed shared memory (each CTA sums an eighth of the parameters over the eight partials, in rank
// order, so the result is deterministic), and the same CTA applies Adam to that eighth, whose moments it keeps in
// registers, and writes the new weights into all eight copies. Two cluster barriers per step, no launch and no global
// round trip. A step of 64 samples is 1.3 MFLOP in a chain of six dependent phases: latency and shared-memory reads
// bound it, so the split is the smallest that leaves every phase two outputs per thread (8 samples x 64 units on 256
// threads) and every product is tiled in registers over 128-bit reads. 800 steps of 64 samples: 72 ms with two launches
// and one CTA per step, 5.9 ms of kernel now (8.1 ms the call).
// ---------------------------------------------------------------------------
constexpr int CR = 8;                            // CTAs of the cluster
constexpr int SB = 8;                            // samples a CTA takes at a time (one warp each in the output layer)
constexpr int TT = 256;                          // threads
constexpr int IN4 = (IN + 3) / 4;                // float4s of a row of W1
constexpr int NV = HID * IN4 + HID / 4 + HID * HID / 4 + (2 * HID + 4) / 4;  // float4s of the parameters in shared memory
constexpr int SHARD = (NV + CR - 1) / CR;        // of them a CTA's, one per thread
static_assert(SHARD <= TT, "a thread owns at most one");
constexpr int XS = (IN + 15) / 16 * 16;          // words of an input row and of a row of W1, zeros past IN
constexpr int W2S = HID + 16;                    // words of a row of W2
static_assert(XS % 32 == 16 && W2S % 32 == 16, "two rows read together must fall on different halves of the banks");

struct __align__(16) TrainParams {
    float w1[HID * XS], b1[HID], w2[HID * W2S], b2[HID], w3[HID], b3[4];
};
struct __align__(16) TrainSmem : TrainParams {
    TrainParams g;                               // partial gradient
    float x[SB][XS];
    float h1[SB][HID], h2[SB][HID], d1[SB][HID], d2[SB][HID];
    float t[SB], dy[SB], sq[SB];
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

// the place of the v-th float4 of the parameters (rows' ends past IN / 4 and HID / 4 left out)
__device__ __forceinline__ int train_vec(int v) {
    constexpr int P1 = HID * XS, P2 = P1 + HID, P3 = P2 + HID * W2S;
    constexpr int V1 = HID * IN4, V2 = V1 + HID / 4, V3 = V2 + HID * HID / 4;
    if (v < V1) return v / IN4 * XS + v % IN4 * 4;
    if (v < V2) return P1 + (v - V1) * 4;
    if (v < V3) return P2 + (v - V2) / (HID / 4) * W2S + (v - V2) % (HID / 4) * 4;
    return P3 + (v - V3) * 4;
}
// the parameter at a place train_vec names or the three after it; -1: none (a row's end)
__device__ __forceinline__ int train_param(int at) {
    constexpr int P1 = HID * XS, P2 = P1 + HID, P3 = P2 + HID * W2S;
    if (at < P1) return at % XS < IN ? at / XS * IN + at % XS : -1;
    if (at < P2) return OB1 + (at - P1);
    if (at < P3) return OW2 + (at - P2) / W2S * HID + (at - P2) % W2S;
    return OB2 + (at - P3) < NP ? OB2 + (at - P3) : -1;
}
__device__ __forceinline__ float *train_flat(TrainParams &p) { return reinterpret_cast<float *>(&p); }

// The weights into S, zeros into the rows' ends.
__device__ __forceinline__ void train_load(TrainSmem &S, const float *params) {
    float *w = train_flat(S);
    for (int i = threadIdx.x; i < HID * XS; i += TT) w[i] = 0.f;
    for (int i = threadIdx.x; i < SB * XS; i += TT) S.x[0][i] = 0.f;
    if (threadIdx.x < 4) S.b3[threadIdx.x] = S.g.b3[threadIdx.x] = 0.f;
    __syncthreads();
    for (int i = threadIdx.x; i < NP; i += TT) w[train_place(i)] = params[i];
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

// The sums over K terms of v[b][k] * w[u * S + k] for the 8 samples and 64 units, put(b, u, sum) for each. The phase is
// bound by shared-memory reads: a thread takes two units of four samples over a quarter of the terms in 128-bit reads,
// K / 16 * 6 of them for 2 K products (one unit of two samples at a time took 3 K reads for the same 2 K). The
// quarters are neighbouring lanes, whose reads of two rows of w fill the 32 banks (S = 16 mod 32).
template <int K, int S, class F>
__device__ __forceinline__ void train_rows(const float *w, const float *v, int vs, F put) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane & 3;
    const int u0 = (lane >> 2) + 8 * (warp & 3), b0 = 4 * (warp >> 2);
    float acc[2][4] = {};
#pragma unroll
    for (int t = 0; t < K / 16; ++t) {
        const int k = 16 * t + 4 * q;
        const float4 wa = *reinterpret_cast<const float4 *>(w + u0 * S + k);
        const float4 wb = *reinterpret_cast<const float4 *>(w + (u0 + HID / 2) * S + k);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float4 x = *reinterpret_cast<const float4 *>(v + (b0 + b) * vs + k);
            acc[0][b] = fmaf(wa.w, x.w, fmaf(wa.z, x.z, fmaf(wa.y, x.y, fmaf(wa.x, x.x, acc[0][b]))));
            acc[1][b] = fmaf(wb.w, x.w, fmaf(wb.z, x.z, fmaf(wb.y, x.y, fmaf(wb.x, x.x, acc[1][b]))));
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {  // lane q of the four ends with sample b0 + q
        float r[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float keep = q & 2 ? acc[i][2 + j] : acc[i][j], give = q & 2 ? acc[i][j] : acc[i][2 + j];
            r[j] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
        }
        const float keep = q & 1 ? r[1] : r[0], give = q & 1 ? r[0] : r[1];
        put(b0 + q, u0 + HID / 2 * i, keep + __shfl_xor_sync(0xffffffffu, give, 1));
    }
}

// The sums over i of d2[b][i] * W2[i][j], put(b, j, sums of j and j + 1). As above with the threads along W2's rows: four
// units of two samples over a quarter of the terms.
template <class F>
__device__ __forceinline__ void train_cols(const TrainSmem &S, F put) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 3;
    const int j0 = 4 * ((lane & 7) + 8 * (warp & 1)), b0 = 2 * (warp >> 1);
    float acc[2][4] = {};
#pragma unroll
    for (int t = 0; t < HID / 16; ++t) {
        const int k = HID / 4 * q + 4 * t;
        float x[2][4];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const float4 d = *reinterpret_cast<const float4 *>(&S.d2[b0 + b][k]);
            x[b][0] = d.x;
            x[b][1] = d.y;
            x[b][2] = d.z;
            x[b][3] = d.w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 w = *reinterpret_cast<const float4 *>(S.w2 + (k + i) * W2S + j0);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                acc[b][0] = fmaf(w.x, x[b][i], acc[b][0]);
                acc[b][1] = fmaf(w.y, x[b][i], acc[b][1]);
                acc[b][2] = fmaf(w.z, x[b][i], acc[b][2]);
                acc[b][3] = fmaf(w.w, x[b][i], acc[b][3]);
            }
        }
    }
    float r[4], s[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // quarters 2 and 3 end with sample b0 + 1
        const float keep = q & 2 ? acc[1][j] : acc[0][j], give = q & 2 ? acc[0][j] : acc[1][j];
        r[j] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {  // odd quarters with units j0 + 2 and j0 + 3
        const float keep = q & 1 ? r[2 + j] : r[j], give = q & 1 ? r[j] : r[2 + j];
        s[j] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
    put(b0 + (q >> 1), j0 + 2 * (q & 1), s[0], s[1]);
}

// What a thread writes of the partial gradient: four neighbours, first ? v : what is there + v.
__device__ __forceinline__ void train_put4(float *at, bool first, const float *v) {
    float4 o = make_float4(v[0], v[1], v[2], v[3]);
    if (!first) {
        const float4 w = *reinterpret_cast<float4 *>(at);
        o = make_float4(o.x + w.x, o.y + w.y, o.z + w.z, o.w + w.w);
    }
    *reinterpret_cast<float4 *>(at) = o;
}

// The outer products of a and x, four by four (rows r0 .., columns c0 ..), summed over the samples.
__device__ __forceinline__ void train_outer(const float *a, const float *x, int xs, int r0, int c0, float (&acc)[4][4]) {
#pragma unroll
    for (int b = 0; b < SB; ++b) {
        const float4 d = *reinterpret_cast<const float4 *>(a + b * HID + r0);
        const float4 e = *reinterpret_cast<const float4 *>(x + b * xs + c0);
        const float dd[4] = {d.x, d.y, d.z, d.w}, xx[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(dd[i], xx[j], acc[i][j]);
    }
}

// Forward pass of the n (<= SB) samples in S.x; each sample's residual y - t to S.dy (0 past n). Ends unsynchronised:
// warp b wrote sample b's.
__device__ __forceinline__ void train_forward(TrainSmem &S, uint32_t n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    train_rows<XS, XS>(S.w1, S.x[0], XS, [&](int b, int u, float v) { S.h1[b][u] = fmaxf(v + S.b1[u], 0.f); });
    __syncthreads();
    train_rows<HID, W2S>(S.w2, S.h1[0], HID, [&](int b, int u, float v) { S.h2[b][u] = fmaxf(v + S.b2[u], 0.f); });
    __syncthreads();
    float y = S.w3[lane] * S.h2[warp][lane] + S.w3[lane + 32] * S.h2[warp][lane + 32];
#pragma unroll
    for (int o = 16; o; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    if (lane == 0) S.dy[warp] = uint32_t(warp) < n ? y + S.b3[0] - S.t[warp] : 0.f;
    __syncwarp();
}

// Gradient of the chunk in S.x (n samples), written to S.g (first) or added; the loss terms go to S.loss. `half` is
// called between the forward and the backward pass.
template <class F>
__device__ __forceinline__ void train_chunk(TrainSmem &S, uint32_t n, float inv_b, bool first, F half) {
    const int tid = threadIdx.x, h = tid & (HID - 1), q = tid / HID, lane = tid & 31, warp = tid >> 5;
    train_forward(S, n);
    half();
    {
        const float r = S.dy[warp], dy = r * inv_b;
        __syncwarp();
        if (lane == 0) {
            S.dy[warp] = dy;
            S.sq[warp] = 0.5f * r * dy;
        }
        S.d2[warp][lane] = S.h2[warp][lane] > 0.f ? dy * S.w3[lane] : 0.f;
        S.d2[warp][lane + 32] = S.h2[warp][lane + 32] > 0.f ? dy * S.w3[lane + 32] : 0.f;
    }
    __syncthreads();
    train_cols(S, [&](int b, int j, float v0, float v1) {  // back through W2
        const float2 a = *reinterpret_cast<const float2 *>(&S.h1[b][j]);
        *reinterpret_cast<float2 *>(&S.d1[b][j]) = make_float2(a.x > 0.f ? v0 : 0.f, a.y > 0.f ? v1 : 0.f);
    });
    auto put = [&](float *at, float v) { *at = first ? v : *at + v; };
    {  // W2: a 4 x 4 tile per thread
        const int r0 = (tid >> 4) * 4, c0 = (tid & 15) * 4;
        float acc[4][4] = {};
        train_outer(S.d2[0], S.h1[0], HID, r0, c0, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) train_put4(S.g.w2 + (r0 + i) * W2S + c0, first, acc[i]);
    }
    if (q == 0) {  // W3, b2 and b3
        float gw = 0.f, gb = 0.f;
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            gw = fmaf(S.dy[b], S.h2[b][h], gw);
            gb += S.d2[b][h];
        }
        put(S.g.w3 + h, gw);
        put(S.g.b2 + h, gb);
        if (h == 0) {
            float g3 = 0.f, ls = 0.f;
#pragma unroll
            for (int b = 0; b < SB; ++b) {
                g3 += S.dy[b];
                ls += S.sq[b];
            }
            put(S.g.b3, g3);
            S.loss = first ? ls : S.loss + ls;
        }
    }
    __syncthreads();
    constexpr int T1 = XS / 4;  // tiles along a row of W1
    if (tid < 16 * T1) {        // W1
        const int r0 = tid / T1 * 4, c0 = tid % T1 * 4;
        float acc[4][4] = {};
        train_outer(S.d1[0], S.x[0], XS, r0, c0, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) train_put4(S.g.w1 + (r0 + i) * XS + c0, first, acc[i]);
    } else if (tid - 16 * T1 < HID) {  // b1
        const int u = tid - 16 * T1;
        float v = 0.f;
#pragma unroll
        for (int b = 0; b < SB; ++b) v += S.d1[b][u];
        put(S.g.b1 + u, v);
    }
}
static_assert(16 * (XS / 4) + HID <= TT, "W1's tiles and b1 share the threads");

// Samples [r0, r0 + per) of a batch of nb belong to rank r.
__device__ __forceinline__ void train_share(uint32_t nb, uint32_t rank, uint32_t &r0, uint32_t &per) {
    const uint32_t each = (nb + CR - 1) / CR;
    r0 = min(each * rank, nb);
    per = min(each, nb - r0);
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
    const int tid = threadIdx.x;
    train_load(S, params);
    // the thread's parameters: float4 SHARD * rank + tid of them
    const int vec = SHARD * int(rank) + tid;
    const bool owner = tid < SHARD && vec < NV;
    const int place = owner ? train_vec(vec) : 0;
    float p[4] = {}, ma[4] = {}, mb[4] = {};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = train_param(place + k);
        if (!owner || i < 0) continue;
        p[k] = params[i];
        if (TRAIN) {
            ma[k] = m1[i];
            mb[k] = m2[i];
        }
    }
    // batches do not cross epochs: the last one of an epoch may be smaller
    uint64_t pos = 0;
    uint32_t in_epoch = 0;
    int step = t0;
    auto batch_at = [&](uint32_t e) { return min(batch, epoch - e); };
    uint32_t r0, per;
    train_share(batch_at(0), rank, r0, per);
    TrainRows next = train_fetch(x, xstride, t, tstride, train_at(perm, r0, min(per, uint32_t(SB))));
    cl.sync();
    while (pos < total) {
        const uint32_t nb = batch_at(in_epoch);
        train_share(nb, rank, r0, per);
        const float inv_b = 1.0f / float(nb);
        const uint64_t npos = pos + nb;
        const uint32_t nin = in_epoch + nb == epoch ? 0u : in_epoch + nb;
        uint32_t nr0 = 0, nper = 0;
        if (npos < total) train_share(batch_at(nin), rank, nr0, nper);
        // at least one chunk: a rank without samples contributes zeros
        for (uint32_t c = 0; c == 0 || c < per; c += SB) {
            const uint32_t n = per > c ? min(per - c, uint32_t(SB)) : 0u;
            train_put(S, next);
            __syncthreads();
            TrainAt at{{0, 0}, 0};
            if (c + SB < per) at = train_at(perm, pos + r0 + c + SB, min(per - c - SB, uint32_t(SB)));
            else if (npos < total) at = train_at(perm, npos + nr0, min(nper, uint32_t(SB)));
            train_chunk(S, n, inv_b, c == 0, [&] { next = train_fetch(x, xstride, t, tstride, at); });
            __syncthreads();
        }
        ++step;
        const float c1 = TRAIN ? 1.f - powf(beta1, float(step)) : 1.f, c2 = TRAIN ? 1.f - powf(beta2, float(step)) : 1.f;
        cl.sync();  // every rank's partial gradient is complete
        float4 part[CR];  // every remote read in flight before the first sum
#pragma unroll
        for (int r = 0; r < CR; ++r) part[r] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(train_flat(S.g), r) + place);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float g = 0.f;
#pragma unroll
            for (int r = 0; r < CR; ++r) g += k == 0 ? part[r].x : k == 1 ? part[r].y : k == 2 ? part[r].z : part[r].w;
            const int i = train_param(place + k);
            if (TRAIN) {
                const float a = beta1 * ma[k] + (1.f - beta1) * g;
                const float b = beta2 * mb[k] + (1.f - beta2) * g * g;
                ma[k] = a;
                mb[k] = b;
                if (i >= 0) p[k] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
            } else if (owner && i >= 0) {
                grad[i] = g;
            }
        }
        if (TRAIN && owner) {
            const float4 w = make_float4(p[0], p[1], p[2], p[3]);
#pragma unroll
            for (int r = 0; r < CR; ++r) *reinterpret_cast<float4 *>(cl.map_shared_rank(train_flat(S), r) + place) = w;
        }
        if (!TRAIN && rank == 0 && tid == 0 && loss_out) {
            float ls = 0.f;
            for (int r = 0; r < CR; ++r) ls += *cl.map_shared_rank(&S.loss, r);
            *loss_out = ls;
        }
        cl.sync();  // the new weights are in every copy, the partials have been read
        pos = npos;
        in_epoch = nin;
    }
    if (TRAIN) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (const int i = train_param(place + k); owner && i >= 0) {
                params[i] = p[k];
                m1[i] = ma[k];
                m2[i] = mb[k];
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
