// Surrogate network: an ensemble of 4 -> 64 -> 64 -> 2 perceptrons with
// GELU hidden layers, bfloat16 weights (float master copies) and float
// accumulation, trained by full-batch Adam on the mean squared error of
// standardised outputs. Forward, backward and update are this file's kernels;
// the ensemble spread is the prediction's uncertainty.
//
// Parameter layout per member (TDPD_MLP_NPARAM floats): W1[64][4], b1[64],
// W2[64][64], b2[64], W3[2][64], b3[2], rows = outputs.
#include <cuda_bf16.h>

#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "launch.h"

using namespace tdpd;

namespace {

constexpr int IN = TDPD_MLP_IN, HID = TDPD_MLP_HIDDEN, OUT = TDPD_MLP_OUT;
constexpr int NP = TDPD_MLP_NPARAM;
constexpr int OW1 = 0, OB1 = OW1 + HID * IN, OW2 = OB1 + HID, OB2 = OW2 + HID * HID,
              OW3 = OB2 + HID, OB3 = OW3 + OUT * HID;
static_assert(OB3 + OUT == NP, "parameter layout");
constexpr int TPB = 128;

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Means and deviations of the training set's inputs and outputs.
struct Standard {
    double mx[IN], sx[IN], my[OUT], sy[OUT];
};

// The shared part of both kernels. A CTA of TPB threads works on CH samples of
// one member as small matrix products from shared memory: thread t owns the
// samples s0..s0+3 (s0 = 4 (t & 7)) and, of the 64 features, 4 to..4 to + 3
// (to = t >> 3) in the products that end in layer 1 and to, to + 16, ... in
// those that end in layer 2 (the strided rows keep the 68-float weight rows on
// distinct banks). A 4 x 4 tile per thread takes 8 16-byte shared loads per 64
// multiply-adds.
constexpr int CH = 32;           // samples per CTA
constexpr int LDS_ = CH + 4;     // padded row of a feature-major activation (16-byte rows)
constexpr int LDW = HID + 4;     // padded row of W2

// (aligned for the 16-byte accesses, and every row of them)
struct alignas(16) NetSmem {
    float W2[HID][LDW];
    float W1[HID][IN];
    float b1[HID], b2[HID], W3[OUT][HID], b3[OUT], pad[2];
    float X[IN][LDS_];
    float H1[HID][LDS_];
    float Y[TPB / 32][OUT][CH];  // each warp's share of the outputs
};

static_assert(offsetof(NetSmem, W1) % 16 == 0 && offsetof(NetSmem, X) % 16 == 0 && offsetof(NetSmem, H1) % 16 == 0 &&
              offsetof(NetSmem, Y) % 16 == 0 && LDW % 4 == 0 && LDS_ % 4 == 0 && CH % 4 == 0 && IN == 4,
              "16-byte rows");

__device__ __forceinline__ void load_net(NetSmem &S, const float *__restrict__ p)
{
    const int t = threadIdx.x;
    for (int k = t; k < HID * HID; k += TPB) S.W2[k >> 6][k & 63] = bf16r(p[OW2 + k]);
    for (int k = t; k < HID * IN; k += TPB) S.W1[k >> 2][k & 3] = bf16r(p[OW1 + k]);
    if (t < HID) {
        S.b1[t] = bf16r(p[OB1 + t]);
        S.b2[t] = bf16r(p[OB2 + t]);
        S.W3[0][t] = bf16r(p[OW3 + t]);
        S.W3[1][t] = bf16r(p[OW3 + HID + t]);
        if (t < OUT) S.b3[t] = bf16r(p[OB3 + t]);
    }
}

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}

// GELU of z and (GRAD) its derivative, one error function for both.
template <bool GRAD>
__device__ __forceinline__ float gelu_both(float z, float &g)
{
    const float e = 1.0f + erff(z * 0.70710678118654752f);
    if (GRAD) g = 0.5f * e + z * expf(-0.5f * z * z) * 0.39894228040143268f;
    return 0.5f * z * e;
}

// Forward pass: h2[q][r] of feature to + 16 q and sample s0 + r, the
// derivatives g1[u][r] (feature 4 to + u) and g2[q][r], H1 and the warps' shares
// of the outputs in shared memory (complete after the caller's barrier).
template <bool GRAD>
__device__ __forceinline__ void forward(NetSmem &S, int s0, int to, float (&g1)[4][4], float (&h2)[4][4],
                                        float (&g2)[4][4])
{
    {
        float4 x[IN];
#pragma unroll
        for (int c = 0; c < IN; ++c) x[c] = ld4(&S.X[c][s0]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int o = 4 * to + u;
            const float4 w = ld4(S.W1[o]);
            const float b = S.b1[o];
            float z[4] = {b, b, b, b}, h[4];
            const float wc[IN] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int c = 0; c < IN; ++c) {
                z[0] = fmaf(wc[c], x[c].x, z[0]);
                z[1] = fmaf(wc[c], x[c].y, z[1]);
                z[2] = fmaf(wc[c], x[c].z, z[2]);
                z[3] = fmaf(wc[c], x[c].w, z[3]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) h[r] = gelu_both<GRAD>(z[r], g1[u][r]);
            st4(&S.H1[o][s0], h[0], h[1], h[2], h[3]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float b = S.b2[to + 16 * q];
#pragma unroll
        for (int r = 0; r < 4; ++r) h2[q][r] = b;
    }
#pragma unroll 4
    for (int i = 0; i < HID; i += 4) {
        float4 w[4], h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = ld4(&S.W2[to + 16 * q][i]);
#pragma unroll
        for (int u = 0; u < 4; ++u) h[u] = ld4(&S.H1[i + u][s0]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float wv = u == 0 ? w[q].x : u == 1 ? w[q].y : u == 2 ? w[q].z : w[q].w;
                h2[q][0] = fmaf(wv, h[u].x, h2[q][0]);
                h2[q][1] = fmaf(wv, h[u].y, h2[q][1]);
                h2[q][2] = fmaf(wv, h[u].z, h2[q][2]);
                h2[q][3] = fmaf(wv, h[u].w, h2[q][3]);
            }
    }
    float y[OUT][4];
#pragma unroll
    for (int k = 0; k < OUT; ++k)
#pragma unroll
        for (int r = 0; r < 4; ++r) y[k][r] = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float w0 = S.W3[0][to + 16 * q], w1 = S.W3[1][to + 16 * q];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            h2[q][r] = gelu_both<GRAD>(h2[q][r], g2[q][r]);
            y[0][r] = fmaf(w0, h2[q][r], y[0][r]);
            y[1][r] = fmaf(w1, h2[q][r], y[1][r]);
        }
    }
    // the four features' groups of the warp (lane bits 3 and 4)
#pragma unroll
    for (int k = 0; k < OUT; ++k)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            y[k][r] += __shfl_xor_sync(0xffffffffu, y[k][r], 8);
            y[k][r] += __shfl_xor_sync(0xffffffffu, y[k][r], 16);
        }
    if ((threadIdx.x & 24) == 0)
#pragma unroll
        for (int k = 0; k < OUT; ++k) st4(&S.Y[threadIdx.x >> 5][k][s0], y[k][0], y[k][1], y[k][2], y[k][3]);
}

// Output k of sample s: the bias and the warps' shares in warp order.
__device__ __forceinline__ float output(const NetSmem &S, int k, int s)
{
    float y = S.b3[k];
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) y += S.Y[w][k][s];
    return y;
}

// Prediction: the CTA's CH samples through one member; X: raw inputs,
// standardised here in binary64 and rounded once. Bound by the two products'
// multiply-adds and the error function; 2048 samples x 5 members: 320 CTAs, all
// resident.
__global__ void __launch_bounds__(TPB) k_mlp_fwd(const float *__restrict__ params, const float *__restrict__ X,
                                                 Standard st, int n, float *Y)
{
    __shared__ NetSmem S;
    const int mbr = blockIdx.y, t = threadIdx.x;
    load_net(S, params + (size_t)mbr * NP);
    {
        const int s = t >> 2, c = t & 3, smp = blockIdx.x * CH + s;
        S.X[c][s] = smp < n ? (float)((X[(size_t)smp * IN + c] - st.mx[c]) / st.sx[c]) : 0.0f;
    }
    __syncthreads();
    float g1[4][4], g2[4][4], h2[4][4];
    forward<false>(S, 4 * (t & 7), t >> 3, g1, h2, g2);
    __syncthreads();
    const int s = t >> 1, k = t & 1, smp = blockIdx.x * CH + s;
    if (s < CH && smp < n) Y[((size_t)mbr * n + smp) * OUT + k] = output(S, k, s);
}

// Ensemble statistics of the predictions in binary64: Y becomes each member's
// output in raw units, mean and rel the ensemble's mean and relative spread.
__global__ void __launch_bounds__(TPB) k_mlp_stats(float *Y, Standard st, int members, int n, float *mean, float *rel)
{
    pdl_enter();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;      // (sample, output)
    if (e >= n * OUT) return;
    const int c = e % OUT;
    double s = 0.0, s2 = 0.0;
    for (int k = 0; k < members; ++k) {
        const size_t at = (size_t)k * n * OUT + e;
        const double y = Y[at] * st.sy[c] + st.my[c];
        Y[at] = (float)y;
        s += y;
        s2 += y * y;
    }
    const double mu = s / members, size = fabs(mu);
    const double var = members > 1 ? fmax(0.0, (s2 - members * mu * mu) / (members - 1)) : 0.0;
    mean[e] = (float)mu;
    // (compared, not fmax, which drops a NaN: a mean that is NaN has a NaN spread, for
    // the callers trust a point by its small spread)
    rel[e] = (float)(sqrt(var) / (size < 1e-30 ? 1e-30 : size));
}

// One training pass over a chunk of CH samples of one member: forward,
// back-propagation, and the chunk's share of every parameter's gradient, in one
// launch. The error signals of layer 2 and the activations of layer 1 meet in
// shared memory for the 64 x 64 gradient; everything else stays in registers
// and is summed over the chunk's samples by shuffles in a fixed tree.
// k_mlp_reduce adds the chunks in a fixed order (float-float), so the gradient
// is deterministic.
// Bound by the multiply-adds (3 x 4096 per sample) and the error functions
// (128 per sample); about 5300 instructions per warp. Chunks of 32 samples at
// 128 threads put four or five CTAs of 40 KB on each SM for 5 x 4096 samples: 25
// us (one thread per sample with 154 KB of shared memory left four warps on an SM
// and a second, nearly empty wave: 88 us); 49 % of the issue slots.
struct TrainSmem {
    NetSmem N;
    float D2[HID][LDS_];
};
static_assert(alignof(TrainSmem) >= 16 && offsetof(TrainSmem, D2) % 16 == 0, "16-byte rows");

// PARTS: the launch takes every PARTS-th chunk, from `first` on, and (first > 0) adds
// its sums to the row of the chunk before, so that a row of part holds PARTS chunks.
template <int PARTS>
__global__ void __launch_bounds__(TPB, 5) k_mlp_chunk(const float *__restrict__ params, const float *__restrict__ X,
                                                      const float *__restrict__ T, int n, float *part,
                                                      float *loss_part, int first, int nch)
{
    __shared__ TrainSmem Q;
    NetSmem &S = Q.N;
    const int mbr = blockIdx.y, row = blockIdx.x, c = row * PARTS + first;
    const int t = threadIdx.x;
    const int s0 = 4 * (t & 7), to = t >> 3;
    {
        // the samples do not depend on the previous launch, the weights do
        const int s = t >> 2, k = t & 3, smp = c * CH + s;
        S.X[k][s] = smp < n ? X[(size_t)smp * IN + k] : 0.0f;
    }
    pdl_enter();
    load_net(S, params + (size_t)mbr * NP);
    __syncthreads();
    float g1[4][4], g2[4][4], h2[4][4];
    forward<true>(S, s0, to, g1, h2, g2);
    __syncthreads();

    float d3[OUT][4], err2 = 0.0f;
    const float sc = 2.0f / (float)(n * OUT);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int smp = c * CH + s0 + r;
        const bool valid = smp < n;
        const float2 y = valid ? *reinterpret_cast<const float2 *>(T + (size_t)smp * OUT) : make_float2(0.f, 0.f);
        const float e0 = output(S, 0, s0 + r) - y.x, e1 = output(S, 1, s0 + r) - y.y;
        d3[0][r] = valid ? sc * e0 : 0.0f;
        d3[1][r] = valid ? sc * e1 : 0.0f;
        err2 += valid ? e0 * e0 + e1 * e1 : 0.0f;
    }
    float *out = part + ((size_t)mbr * gridDim.x + row) * NP;
    auto put = [&](int k, float v) {
        if (PARTS > 1 && first > 0) v += out[k];
        out[k] = v;
    };
    // sum of a value over the chunk's samples: the thread's four, then the
    // eight sample groups of the feature (lane bits 0-2)
    auto over_samples = [](float v) {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        return v;
    };
    const bool writer = (t & 7) == 0;
    {
        const float l = over_samples(err2), b0 = over_samples((d3[0][0] + d3[0][1]) + (d3[0][2] + d3[0][3])),
                    b1 = over_samples((d3[1][0] + d3[1][1]) + (d3[1][2] + d3[1][3]));
        if (t == 0) {
            if (PARTS == 1 || c < nch) loss_part[(size_t)mbr * nch + c] = l;
            put(OB3, b0);
            put(OB3 + 1, b1);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int o = to + 16 * q;
        const float w0 = S.W3[0][o], w1 = S.W3[1][o];
        float d2[4], a0 = 0.0f, a1 = 0.0f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            d2[r] = fmaf(d3[0][r], w0, d3[1][r] * w1) * g2[q][r];
            a0 = fmaf(d3[0][r], h2[q][r], a0);
            a1 = fmaf(d3[1][r], h2[q][r], a1);
        }
        st4(&Q.D2[o][s0], d2[0], d2[1], d2[2], d2[3]);
        a0 = over_samples(a0);
        a1 = over_samples(a1);
        const float b2 = over_samples((d2[0] + d2[1]) + (d2[2] + d2[3]));
        if (writer) {
            put(OW3 + o, a0);
            put(OW3 + HID + o, a1);
            put(OB2 + o, b2);
        }
    }
    __syncthreads();
    {
        // error signals of layer 1: features 4 to + u
        float a[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int r = 0; r < 4; ++r) a[u][r] = 0.0f;
#pragma unroll 8
        for (int o = 0; o < HID; ++o) {
            const float4 w = ld4(&S.W2[o][4 * to]), d = ld4(&Q.D2[o][s0]);
            const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u][0] = fmaf(d.x, wv[u], a[u][0]);
                a[u][1] = fmaf(d.y, wv[u], a[u][1]);
                a[u][2] = fmaf(d.z, wv[u], a[u][2]);
                a[u][3] = fmaf(d.w, wv[u], a[u][3]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = 4 * to + u;
            float d1[4], b = 0.0f;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                d1[r] = a[u][r] * g1[u][r];
                b += d1[r];
            }
            b = over_samples(b);
            float w1[IN];
#pragma unroll
            for (int k = 0; k < IN; ++k) {
                const float4 x = ld4(&S.X[k][s0]);
                w1[k] = over_samples(fmaf(d1[3], x.w, fmaf(d1[2], x.z, fmaf(d1[1], x.y, d1[0] * x.x))));
            }
            if (writer) {
                put(OB1 + i, b);
#pragma unroll
                for (int k = 0; k < IN; ++k) put(OW1 + i * IN + k, w1[k]);
            }
        }
    }
    {
        // dW2[o][i] = sum_s d2[o][s] h1[i][s]: features o = to + 16 q of layer
        // 2 and i = (t & 7) + 8 p of layer 1
        const int ii = t & 7;
        float acc[4][8];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 8; ++p) acc[q][p] = 0.0f;
#pragma unroll 2
        for (int s = 0; s < CH; s += 4) {
            float4 d[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) d[q] = ld4(&Q.D2[to + 16 * q][s]);
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const float4 h = ld4(&S.H1[ii + 8 * p][s]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    acc[q][p] = fmaf(d[q].w, h.w, fmaf(d[q].z, h.z, fmaf(d[q].y, h.y, fmaf(d[q].x, h.x, acc[q][p]))));
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 8; ++p) put(OW2 + (to + 16 * q) * HID + ii + 8 * p, acc[q][p]);
    }
}

// Each parameter's gradient: its chunks' sums added in float-float, eight warps
// taking every eighth chunk and their sums added in warp order (a fixed order
// for a given chunk count; 32 parameters per CTA, so a warp reads 128 bytes per
// chunk and the eight warps keep enough loads in flight: 12 MB for 5 x 4096
// samples, 6.5 us). With adam, the Adam step (Kingma & Ba) on the float master weights,
// bc1 and bc2 being the bias corrections 1 - beta^t.
constexpr int RED_WARPS = 8;
__global__ void __launch_bounds__(32 * RED_WARPS) k_mlp_reduce(const float *__restrict__ part, int nch, int total,
                                                               float *grad, int adam, float *params, float *m,
                                                               float *v, float lr, float beta1, float beta2,
                                                               float eps, float bc1, float bc2)
{
    pdl_enter();
    __shared__ FF sum[RED_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    FF acc{0.0f, 0.0f};
    if (k < total) {
        const int mbr = k / NP;
        const float *p = part + (size_t)mbr * nch * NP + (k - mbr * NP);
#pragma unroll 8
        for (int c = w; c < nch; c += RED_WARPS) acc = ff_add(acc, p[(size_t)c * NP]);
    }
    sum[w][lane] = acc;
    __syncthreads();
    if (w != 0 || k >= total) return;
#pragma unroll
    for (int u = 1; u < RED_WARPS; ++u) acc = ff_add(acc, sum[u][lane]);
    const float g = acc.hi + acc.lo;
    grad[k] = g;
    if (adam) {
        const float mk = fmaf(beta1, m[k], (1.0f - beta1) * g);
        const float vk = fmaf(beta2, v[k], (1.0f - beta2) * g * g);
        m[k] = mk;
        v[k] = vk;
        params[k] -= lr * (mk / bc1) / (sqrtf(vk / bc2) + eps);
    }
}

}  // namespace

struct tdpd_mlp {
    int members = 0, n = 0, cap = 0;
    int64_t t = 0;
    float *params = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
    float *X = nullptr, *T = nullptr, *loss_part = nullptr;
    float *gpart = nullptr;     // [members][chunks][NP] per-chunk gradient sums
    Standard sd = {};
    float *base = nullptr;      // one allocation: params, m, v, grad, the first workspace
    // prediction workspace, kept between calls up to PRED_KEEP floats: inputs,
    // then mean, relative spread and the members' outputs. One call at a time uses
    // it, from its copy of the inputs to the read of its results (pred_use), so that
    // threads may predict with one handle; the calls share the handle's stream anyway
    float *pred = nullptr, *pred_own = nullptr;
    std::mutex pred_use;
    size_t pred_floats = 0;
    // samples to train on in X and T; a standardisation to predict with (it outlives
    // the samples when a larger set does not fit)
    bool have_data = false, have_std = false;
    cudaStream_t st = nullptr;
};

namespace {

tdpd_status mfail(tdpd_status c, const std::string &msg)
{
    set_thread_error(msg.c_str());
    return c;
}

#define MCU(call)                                                                             \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess) return mfail(TDPD_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

void free_data(tdpd_mlp *m)
{
    cudaFree(m->gpart);
    m->cap = m->n = 0;
    m->X = m->T = m->loss_part = m->gpart = nullptr;
    m->have_data = false;
}

// Rows of the per-chunk gradient sums: a chunk each up to ROWS_MAX chunks (262,144
// samples; 151 MB per member), above that four chunks each, which bounds the memory
// at 144 bytes per sample and member (a row per chunk: 576).
constexpr int ROWS_MAX = 8192;
int grad_parts(int nch) { return nch <= ROWS_MAX ? 1 : 4; }

// Buffers for n samples in one allocation, nearly all of it gradient rows (the first 512
// samples of five members set in 96 us, with four allocations 107; most of it maps
// the rows' 1.5 MB, four times those of 128-sample chunks, which took 35). On failure the
// handle has no samples.
tdpd_status alloc_data(tdpd_mlp *m, int n)
{
    if (n <= m->cap) return TDPD_OK;
    cudaStreamSynchronize(m->st);
    free_data(m);
    const size_t M = m->members, nch = (size_t)(n + CH - 1) / CH;
    // (fewer samples later may take more rows)
    const size_t rows = nch <= (size_t)ROWS_MAX ? nch : std::max((nch + 3) / 4, (size_t)ROWS_MAX);
    const auto padded = [](size_t floats) { return (floats + 63) / 64 * 64; };
    const size_t part = padded(M * rows * NP), x = padded((size_t)n * IN), t = padded((size_t)n * OUT);
    if (cudaMalloc((void **)&m->gpart, (part + x + t + M * nch) * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();                       // (not the next call's error)
        m->gpart = nullptr;
        return mfail(TDPD_ENOMEM, "tdpd_mlp: device allocation failed");
    }
    m->X = m->gpart + part;
    m->T = m->X + x;
    m->loss_part = m->T + t;
    m->cap = n;
    return TDPD_OK;
}

// The prediction workspace, at least `need` floats: PRED_MIN of them come with
// the handle, more are allocated once. (Two allocations and their release on every
// call, the standardisation and the ensemble statistics on the host took 250 us of
// a call that ranks 2048 points with five members.)
constexpr size_t PRED_MIN = (size_t)1 << 16, PRED_KEEP = (size_t)1 << 22;
tdpd_status pred_workspace(tdpd_mlp *m, size_t need)
{
    if (need <= m->pred_floats) return TDPD_OK;
    void *d = nullptr;
    if (cudaMalloc(&d, need * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        return mfail(TDPD_ENOMEM, "tdpd_mlp_predict: device allocation failed");
    }
    if (m->pred_own) cudaFree(m->pred_own);       // (every call waits for its work before it lets go)
    m->pred = m->pred_own = (float *)d;
    m->pred_floats = need;
    return TDPD_OK;
}

// One pass over the data: the chunks' gradients, then their sums (and, with
// lr > 0, one Adam step); loss (may be NULL) receives each member's loss.
tdpd_status pass(tdpd_mlp *m, float lr, double *loss)
{
    const int nch = (m->n + CH - 1) / CH;
    const int parts = grad_parts(nch), rows = (nch + parts - 1) / parts;
    if (parts == 1)
        launch_pdl(k_mlp_chunk<1>, dim3(nch, m->members), TPB, m->st, m->params, m->X, m->T, m->n, m->gpart,
                   m->loss_part, 0, nch);
    else
        for (int k = 0; k < parts; ++k)
            launch_pdl(k_mlp_chunk<4>, dim3(rows, m->members), TPB, m->st, m->params, m->X, m->T, m->n, m->gpart,
                       m->loss_part, k, nch);
    const int total = m->members * NP;
    float bc1 = 1.0f, bc2 = 1.0f;
    if (lr > 0.0f) {
        ++m->t;
        bc1 = (float)(1.0 - std::pow(0.9, (double)m->t));
        bc2 = (float)(1.0 - std::pow(0.999, (double)m->t));
    }
    launch_pdl(k_mlp_reduce, (total + 31) / 32, 32 * RED_WARPS, m->st, m->gpart, rows, total, m->grad,
               lr > 0.0f ? 1 : 0, m->params, m->m, m->v, lr, 0.9f, 0.999f, 1e-8f, bc1, bc2);
    MCU(cudaGetLastError());
    if (loss) {
        std::vector<float> part((size_t)m->members * nch);
        MCU(cudaMemcpyAsync(part.data(), m->loss_part, part.size() * sizeof(float), cudaMemcpyDeviceToHost, m->st));
        MCU(cudaStreamSynchronize(m->st));
        for (int k = 0; k < m->members; ++k) {
            double sum = 0.0;
            for (int c = 0; c < nch; ++c) sum += part[(size_t)k * nch + c];
            loss[k] = sum / ((double)m->n * OUT);
        }
    }
    return TDPD_OK;
}

}  // namespace

extern "C" {

tdpd_status tdpd_mlp_create(tdpd_mlp **out, int members)
{
    if (!out || members < 1 || members > 64) return mfail(TDPD_EINVAL, "tdpd_mlp_create: 1..64 members");
    *out = nullptr;
    tdpd_mlp *m = new (std::nothrow) tdpd_mlp;
    if (!m) return mfail(TDPD_ENOMEM, "host allocation failed");
    m->members = members;
    const size_t par = (size_t)members * NP;
    void *p = nullptr;
    if (cudaMalloc(&p, (4 * par + PRED_MIN) * sizeof(float)) != cudaSuccess) {
        delete m;
        return mfail(TDPD_ENOMEM, "tdpd_mlp_create: device allocation failed");
    }
    m->base = m->params = (float *)p;
    m->m = m->params + par;
    m->v = m->m + par;
    m->grad = m->v + par;
    m->pred = m->grad + par;
    m->pred_floats = PRED_MIN;
    if (cudaStreamCreateWithFlags(&m->st, cudaStreamNonBlocking) != cudaSuccess ||
        cudaMemset(m->params, 0, 3 * par * sizeof(float)) != cudaSuccess) {
        cudaFree(m->base);
        delete m;
        return mfail(TDPD_ECUDA, "tdpd_mlp_create: stream or memset failed");
    }
    *out = m;
    return TDPD_OK;
}

tdpd_status tdpd_mlp_set_params(tdpd_mlp *m, const float *params)
{
    if (!m || !params) return mfail(TDPD_EINVAL, "null argument");
    const size_t bytes = (size_t)m->members * NP * sizeof(float);
    MCU(cudaMemcpyAsync(m->params, params, bytes, cudaMemcpyHostToDevice, m->st));
    MCU(cudaMemsetAsync(m->m, 0, bytes, m->st));
    MCU(cudaMemsetAsync(m->v, 0, bytes, m->st));
    MCU(cudaStreamSynchronize(m->st));
    m->t = 0;
    return TDPD_OK;
}

tdpd_status tdpd_mlp_get_params(tdpd_mlp *m, float *params)
{
    if (!m || !params) return mfail(TDPD_EINVAL, "null argument");
    MCU(cudaMemcpyAsync(params, m->params, (size_t)m->members * NP * sizeof(float), cudaMemcpyDeviceToHost, m->st));
    MCU(cudaStreamSynchronize(m->st));
    return TDPD_OK;
}

tdpd_status tdpd_mlp_set_data(tdpd_mlp *m, int n, const float *X, const float *Y)
{
    if (!m || n < 2 || !X || !Y) return mfail(TDPD_EINVAL, "tdpd_mlp_set_data: need n >= 2 samples");
    tdpd_status rc = alloc_data(m, n);
    if (rc) return rc;
    // standardisation: mean and population deviation of each column
    for (int k = 0; k < IN + OUT; ++k) {
        const float *src = k < IN ? X : Y;
        const int w = k < IN ? IN : OUT, c = k < IN ? k : k - IN;
        double s = 0.0, s2 = 0.0;
        for (int i = 0; i < n; ++i) s += src[(size_t)i * w + c];
        const double mean = s / n;
        for (int i = 0; i < n; ++i) {
            const double d = src[(size_t)i * w + c] - mean;
            s2 += d * d;
        }
        const double sd = std::sqrt(s2 / n) + 1e-12;
        if (k < IN) { m->sd.mx[c] = mean; m->sd.sx[c] = sd; }
        else { m->sd.my[c] = mean; m->sd.sy[c] = sd; }
    }
    std::vector<float> xs((size_t)n * IN), ys((size_t)n * OUT);
    for (int i = 0; i < n; ++i) {
        for (int c = 0; c < IN; ++c) xs[(size_t)i * IN + c] = (float)((X[(size_t)i * IN + c] - m->sd.mx[c]) / m->sd.sx[c]);
        for (int c = 0; c < OUT; ++c) ys[(size_t)i * OUT + c] = (float)((Y[(size_t)i * OUT + c] - m->sd.my[c]) / m->sd.sy[c]);
    }
    MCU(cudaMemcpyAsync(m->X, xs.data(), xs.size() * sizeof(float), cudaMemcpyHostToDevice, m->st));
    MCU(cudaMemcpyAsync(m->T, ys.data(), ys.size() * sizeof(float), cudaMemcpyHostToDevice, m->st));
    MCU(cudaStreamSynchronize(m->st));
    m->n = n;
    m->have_data = m->have_std = true;
    return TDPD_OK;
}

tdpd_status tdpd_mlp_loss_grad(tdpd_mlp *m, double *loss, float *grad)
{
    if (!m || !m->have_data) return mfail(TDPD_ESTATE, "tdpd_mlp_loss_grad: no data set");
    tdpd_status rc = pass(m, 0.0f, loss);
    if (rc) return rc;
    if (grad) {
        MCU(cudaMemcpyAsync(grad, m->grad, (size_t)m->members * NP * sizeof(float), cudaMemcpyDeviceToHost, m->st));
        MCU(cudaStreamSynchronize(m->st));
    }
    return TDPD_OK;
}

tdpd_status tdpd_mlp_train(tdpd_mlp *m, int steps, float lr, double *loss)
{
    if (!m || !m->have_data) return mfail(TDPD_ESTATE, "tdpd_mlp_train: no data set");
    if (steps < 0 || !(lr > 0)) return mfail(TDPD_EINVAL, "tdpd_mlp_train: steps >= 0, lr > 0");
    for (int k = 0; k < steps; ++k) {
        tdpd_status rc = pass(m, lr, nullptr);
        if (rc) return rc;
    }
    if (loss) return pass(m, 0.0f, loss);
    MCU(cudaStreamSynchronize(m->st));
    return TDPD_OK;
}

tdpd_status tdpd_mlp_predict(tdpd_mlp *m, int n, const float *X, float *mean, float *rel_spread, float *member_out)
{
    if (!m || n < 1 || !X || !mean) return mfail(TDPD_EINVAL, "tdpd_mlp_predict: bad arguments");
    if (!m->have_std) return mfail(TDPD_ESTATE, "tdpd_mlp_predict: no standardisation (set data first)");
    const size_t N = (size_t)n, in = N * IN, ens = 2 * N * OUT, each = (size_t)m->members * N * OUT;
    const size_t need = in + ens + each;
    // a call beyond the kept workspace allocates for itself
    const bool keep = need <= PRED_KEEP;
    std::unique_lock<std::mutex> use(m->pred_use, std::defer_lock);
    float *d = nullptr;
    if (keep) {
        use.lock();
        tdpd_status rc = pred_workspace(m, need);
        if (rc) return rc;
        d = m->pred;
    } else if (cudaMallocAsync((void **)&d, need * sizeof(float), m->st) != cudaSuccess) {
        cudaGetLastError();                       // (not the next call's error)
        return mfail(TDPD_ENOMEM, "tdpd_mlp_predict: device allocation failed");
    }
    float *dmean = d + in, *drel = dmean + N * OUT, *dY = drel + N * OUT;
    MCU(cudaMemcpyAsync(d, X, in * sizeof(float), cudaMemcpyHostToDevice, m->st));
    k_mlp_fwd<<<dim3((n + CH - 1) / CH, m->members), TPB, 0, m->st>>>(m->params, d, m->sd, n, dY);
    launch_pdl(k_mlp_stats, (unsigned)((N * OUT + TPB - 1) / TPB), TPB, m->st, dY, m->sd, m->members, n, dmean, drel);
    MCU(cudaGetLastError());
    MCU(cudaMemcpyAsync(mean, dmean, N * OUT * sizeof(float), cudaMemcpyDeviceToHost, m->st));
    if (rel_spread) MCU(cudaMemcpyAsync(rel_spread, drel, N * OUT * sizeof(float), cudaMemcpyDeviceToHost, m->st));
    if (member_out) MCU(cudaMemcpyAsync(member_out, dY, each * sizeof(float), cudaMemcpyDeviceToHost, m->st));
    if (!keep) MCU(cudaFreeAsync(d, m->st));
    MCU(cudaStreamSynchronize(m->st));
    return TDPD_OK;
}

void tdpd_mlp_destroy(tdpd_mlp *m)
{
    if (!m) return;
    cudaStreamSynchronize(m->st);
    free_data(m);
    if (m->pred_own) cudaFree(m->pred_own);
    cudaFree(m->base);
    cudaStreamDestroy(m->st);
    delete m;
}

}  // extern "C"
