// zf_mlp.cu -- the learned selector: a 32 -> 64 -> 64 -> 12 perceptron
// (ReLU hidden layers, FP32) with hand-written forward, backward and Adam
// kernels, and the host loops that train it and use it in zf_plan.
//
// Parameters are one flat FP32 vector: W1[64][32], b1[64], W2[64][64], b2[64],
// W3[12][64], b3[12] (7,052 values).  The loss is the softmax cross-entropy
// over the classes each sample allows (others masked), averaged over the
// batch.  Gradients are summed in a fixed order (eight samples in a CTA, then
// the CTAs), so training is deterministic.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <numeric>
#include <vector>

#include "zf_internal.h"

namespace {

constexpr int IN = 32, HID = 64, OUT = 12;
constexpr int OW1 = 0, OB1 = OW1 + HID * IN, OW2 = OB1 + HID, OB2 = OW2 + HID * HID, OW3 = OB2 + HID,
              OB3 = OW3 + OUT * HID, NP = OB3 + OUT;
static_assert(NP == 7052, "parameter layout");

// A CTA of 256 threads takes kTile samples with the weights in shared memory
// (rows padded by one, so that both a row and a column are read without bank
// conflicts): thread (j, g) owns hidden unit j for samples 2g and 2g + 1, and a
// weight read serves both.  Activations are kept unit by unit, kTile samples
// side by side.  What bounds it is latency -- a batch of 256 is 32 CTAs and 11
// MFLOP -- so the batch is spread thin.  One CTA per sample, with weights read
// from global memory column-wise and 28 KB of gradient written per sample for
// a second kernel to add up, wrote and read 14 MB a step instead of 1.8.
constexpr int kTile = 8, kThreads = 256;
constexpr int kPart = NP + 4;   // floats of a CTA's partial result: the gradient, the summed loss, padding

struct MlpSmem {
    float w1[HID * (IN + 1)], w2[HID * (HID + 1)], w3[OUT * (HID + 1)], b1[HID], b2[HID], b3[OUT];
    alignas(16) float x[IN * kTile];
    alignas(16) float h1[HID * kTile], h2[HID * kTile], d1[HID * kTile], d2[HID * kTile];
    alignas(16) float z[OUT * kTile];
    alignas(16) float loss[kTile];
};

// The rows a launch reads: row r of the batch is row order[r] of X (row r
// where order is null), standardized as (x - mean) / sd where scaled.
struct Rows {
    const float* X;
    const uint32_t* order;
    uint32_t n;
    bool scaled;
    float mean[IN], sd[IN];
};

__device__ __forceinline__ uint32_t row_of(const Rows& r, uint32_t i) { return r.order ? r.order[i] : i; }

// Loads the weights and the CTA's samples (zeros past the batch) and computes the logits sm.z.
__device__ __forceinline__ void forward_tile(const float* __restrict__ p, const Rows& r, MlpSmem& sm) {
    const int tid = threadIdx.x;
    const uint32_t s0 = blockIdx.x * kTile;
    // every load is under way before the first value is stored: a thread's 28 weights, a bias and an input value
    // one after another held up a batch of up to 64 samples by 2 us
    static_assert(kThreads == IN * kTile, "one input value per thread");
    const int s = tid / IN, f = tid % IN;
    float x = s0 + s < r.n ? r.X[(size_t)row_of(r, s0 + s) * IN + f] : 0.0f;
    constexpr int N1 = HID * IN / kThreads, N2 = HID * HID / kThreads, N3 = OUT * HID / kThreads;
    float w1[N1], w2[N2], w3[N3], b = 0.0f;
#pragma unroll
    for (int q = 0; q < N1; q++) w1[q] = p[OW1 + tid + q * kThreads];
#pragma unroll
    for (int q = 0; q < N2; q++) w2[q] = p[OW2 + tid + q * kThreads];
#pragma unroll
    for (int q = 0; q < N3; q++) w3[q] = p[OW3 + tid + q * kThreads];
    if (tid < HID) b = p[OB1 + tid];
    else if (tid < 2 * HID) b = p[OB2 + tid - HID];
    else if (tid < 2 * HID + OUT) b = p[OB3 + tid - 2 * HID];
#pragma unroll
    for (int q = 0; q < N1; q++) sm.w1[(tid + q * kThreads) / IN * (IN + 1) + (tid + q * kThreads) % IN] = w1[q];
#pragma unroll
    for (int q = 0; q < N2; q++) sm.w2[(tid + q * kThreads) / HID * (HID + 1) + (tid + q * kThreads) % HID] = w2[q];
#pragma unroll
    for (int q = 0; q < N3; q++) sm.w3[(tid + q * kThreads) / HID * (HID + 1) + (tid + q * kThreads) % HID] = w3[q];
    if (tid < HID) sm.b1[tid] = b;
    else if (tid < 2 * HID) sm.b2[tid - HID] = b;
    else if (tid < 2 * HID + OUT) sm.b3[tid - 2 * HID] = b;
    if (r.scaled) x = (x - r.mean[f]) / r.sd[f];
    sm.x[f * kTile + s] = x;
    __syncthreads();
    const int j = tid & (HID - 1), g = tid / HID * 2;
    {
        float a0 = sm.b1[j], a1 = a0;
#pragma unroll 8
        for (int i = 0; i < IN; i++) {
            const float w = sm.w1[j * (IN + 1) + i];
            const float2 x = *reinterpret_cast<const float2*>(&sm.x[i * kTile + g]);
            a0 += w * x.x;
            a1 += w * x.y;
        }
        *reinterpret_cast<float2*>(&sm.h1[j * kTile + g]) = make_float2(fmaxf(a0, 0.0f), fmaxf(a1, 0.0f));
    }
    __syncthreads();
    {
        float a0 = sm.b2[j], a1 = a0;
#pragma unroll 8
        for (int i = 0; i < HID; i++) {
            const float w = sm.w2[j * (HID + 1) + i];
            const float2 x = *reinterpret_cast<const float2*>(&sm.h1[i * kTile + g]);
            a0 += w * x.x;
            a1 += w * x.y;
        }
        *reinterpret_cast<float2*>(&sm.h2[j * kTile + g]) = make_float2(fmaxf(a0, 0.0f), fmaxf(a1, 0.0f));
    }
    __syncthreads();
    if (tid < OUT * kTile) {
        const int k = tid / kTile, s = tid % kTile;
        float a = sm.b3[k];
#pragma unroll 8
        for (int i = 0; i < HID; i++) a += sm.w3[k * (HID + 1) + i] * sm.h2[i * kTile + s];
        sm.z[tid] = a;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kThreads) mlp_forward(const float* __restrict__ p, const __grid_constant__ Rows r,
                                                        float* __restrict__ Z) {
    __shared__ MlpSmem sm;
    forward_tile(p, r, sm);
    const uint32_t s0 = blockIdx.x * kTile;
    const int s = threadIdx.x / OUT, k = threadIdx.x % OUT;
    if (threadIdx.x < OUT * kTile && s0 + s < r.n) Z[(size_t)(s0 + s) * OUT + k] = sm.z[k * kTile + s];
}

// The CTA's samples' share of the gradient of the batch-mean masked
// cross-entropy, and the sum of their losses, into part[blockIdx.x].
__global__ void __launch_bounds__(kThreads) mlp_grad_part(const float* __restrict__ p, const __grid_constant__ Rows r,
                                                          const int32_t* __restrict__ Y, const uint8_t* __restrict__ MK,
                                                          float* __restrict__ part) {
    __shared__ MlpSmem sm;
    forward_tile(p, r, sm);
    const int tid = threadIdx.x;
    const uint32_t s0 = blockIdx.x * kTile;
    float* out = part + (size_t)blockIdx.x * kPart;
    if (tid < kTile) {
        float l = 0.0f, dz[OUT];
        for (int k = 0; k < OUT; k++) dz[k] = 0.0f;
        if (s0 + tid < r.n) {
            const uint32_t row = row_of(r, s0 + tid);
            const int y = Y[row];
            const uint8_t* mk = MK + (size_t)row * OUT;
            float mx = -INFINITY;
            for (int k = 0; k < OUT; k++)
                if (mk[k]) mx = fmaxf(mx, sm.z[k * kTile + tid]);
            float sum = 0.0f, ey = 0.0f;
            for (int k = 0; k < OUT; k++) {
                dz[k] = mk[k] ? expf(sm.z[k * kTile + tid] - mx) : 0.0f;
                sum += dz[k];
                if (k == y) ey = dz[k];
            }
            for (int k = 0; k < OUT; k++) dz[k] = (dz[k] / sum - (k == y ? 1.0f : 0.0f)) / (float)r.n;
            l = -logf(ey / sum);
        }
        for (int k = 0; k < OUT; k++) sm.z[k * kTile + tid] = dz[k];   // from here on the gradient of the logits
        sm.loss[tid] = l;
    }
    __syncthreads();
    const int j = tid & (HID - 1), g = tid / HID * 2;
    {
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
        for (int k = 0; k < OUT; k++) {
            const float w = sm.w3[k * (HID + 1) + j];
            const float2 d = *reinterpret_cast<const float2*>(&sm.z[k * kTile + g]);
            a0 += w * d.x;
            a1 += w * d.y;
        }
        const float2 h = *reinterpret_cast<const float2*>(&sm.h2[j * kTile + g]);
        *reinterpret_cast<float2*>(&sm.d2[j * kTile + g]) = make_float2(h.x > 0.0f ? a0 : 0.0f, h.y > 0.0f ? a1 : 0.0f);
    }
    __syncthreads();
    {
        float a0 = 0.0f, a1 = 0.0f;
#pragma unroll 8
        for (int i = 0; i < HID; i++) {
            const float w = sm.w2[i * (HID + 1) + j];
            const float2 d = *reinterpret_cast<const float2*>(&sm.d2[i * kTile + g]);
            a0 += w * d.x;
            a1 += w * d.y;
        }
        const float2 h = *reinterpret_cast<const float2*>(&sm.h1[j * kTile + g]);
        *reinterpret_cast<float2*>(&sm.d1[j * kTile + g]) = make_float2(h.x > 0.0f ? a0 : 0.0f, h.y > 0.0f ? a1 : 0.0f);
    }
    // a weight's gradient: the sum over the samples of its row's gradient times its column's input
    auto dot = [](const float* a, const float* b) {
        float t = 0.0f;
#pragma unroll
        for (int s = 0; s < kTile; s += 4) {
            const float4 u = *reinterpret_cast<const float4*>(a + s), v = *reinterpret_cast<const float4*>(b + s);
            t += u.x * v.x;
            t += u.y * v.y;
            t += u.z * v.z;
            t += u.w * v.w;
        }
        return t;
    };
    auto total = [](const float* a) {
        float t = 0.0f;
#pragma unroll
        for (int s = 0; s < kTile; s++) t += a[s];
        return t;
    };
    for (int i = tid; i < OUT * HID; i += kThreads) out[OW3 + i] = dot(&sm.z[i / HID * kTile], &sm.h2[i % HID * kTile]);
    for (int i = tid; i < HID * HID; i += kThreads) out[OW2 + i] = dot(&sm.d2[i / HID * kTile], &sm.h1[i % HID * kTile]);
    __syncthreads();
    for (int i = tid; i < HID * IN; i += kThreads) out[OW1 + i] = dot(&sm.d1[i / IN * kTile], &sm.x[i % IN * kTile]);
    if (tid < HID) out[OB1 + tid] = total(&sm.d1[tid * kTile]);
    else if (tid < 2 * HID) out[OB2 + tid - HID] = total(&sm.d2[(tid - HID) * kTile]);
    else if (tid < 2 * HID + OUT) out[OB3 + tid - 2 * HID] = total(&sm.z[(tid - 2 * HID) * kTile]);
    else if (tid == kThreads - 1) out[NP] = total(sm.loss);
}

// Forward pass and the argmax over each sample's allowed classes.
__global__ void __launch_bounds__(kThreads) mlp_predict(const float* __restrict__ p, const __grid_constant__ Rows r,
                                                        const uint8_t* __restrict__ MK, int32_t* __restrict__ C) {
    __shared__ MlpSmem sm;
    forward_tile(p, r, sm);
    const uint32_t row = blockIdx.x * kTile + threadIdx.x;
    if (threadIdx.x < kTile && row < r.n) {
        int best = -1;
        float zb = 0.0f;
        for (int k = 0; k < OUT; k++) {
            const float z = sm.z[k * kTile + threadIdx.x];
            if (MK[(size_t)row * OUT + k] && (best < 0 || z > zb)) {
                best = k;
                zb = z;
            }
        }
        C[row] = best;
    }
}

// Sum of the CTAs' parts of value i, in their order.
__device__ __forceinline__ float sum_parts(const float* __restrict__ part, uint32_t nparts, int i) {
    float s = 0.0f;
#pragma unroll 8
    for (uint32_t c = 0; c < nparts; c++) s += part[(size_t)c * kPart + i];
    return s;
}

__global__ void mlp_reduce(const float* __restrict__ part, uint32_t nparts, uint32_t B, float* __restrict__ grad,
                           float* __restrict__ loss) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NP) grad[i] = sum_parts(part, nparts, i);
    if (i == NP && loss) *loss = sum_parts(part, nparts, NP) / (float)B;
}

__device__ __forceinline__ void adam_value(float& p, float& m, float& v, float gi, float lr, float b1, float b2, float eps,
                                           float c1, float c2) {
    m = b1 * m + (1.0f - b1) * gi;
    v = b2 * v + (1.0f - b2) * gi * gi;
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__device__ __forceinline__ void adam_one(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v, int i,
                                         float gi, float lr, float b1, float b2, float eps, float c1, float c2) {
    float pi = p[i], mi = m[i], vi = v[i];
    adam_value(pi, mi, vi, gi, lr, b1, b2, eps, c1, c2);
    p[i] = pi;
    m[i] = mi;
    v[i] = vi;
}

// A training step after mlp_grad_part: the gradient's sum and the Adam update in one pass.
__global__ void mlp_reduce_adam(const float* __restrict__ part, uint32_t nparts, uint32_t B, float* __restrict__ loss,
                                float* __restrict__ p, float* __restrict__ m, float* __restrict__ v, float lr, float b1,
                                float b2, float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NP) adam_one(p, m, v, i, sum_parts(part, nparts, i), lr, b1, b2, eps, c1, c2);
    if (i == NP && loss) *loss = sum_parts(part, nparts, NP) / (float)B;
}

__global__ void mlp_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                         const float* __restrict__ g, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NP) adam_one(p, m, v, i, g[i], lr, b1, b2, eps, c1, c2);
}

// ---------------------------------------------------------------- training in one cluster
// Steps of up to kClusterBatch samples run inside one kernel: a cluster of
// kRanks CTAs keeps the weights in every CTA's shared memory and each rank a
// sixteenth of the Adam state in registers.  Per step a rank takes a sixteenth
// of the batch (16 samples at a time), leaves its share of the gradient in its
// shared memory, and after a cluster barrier every rank sums the sixteen shares
// of its sixteenth of the parameters, updates them and stores them into all
// CTAs' weights.  The next step's rows are loaded while a step computes.  A
// layer takes one unit and kSpt samples per thread, a weight gradient 4 x 4
// values per thread.  What bounds it is the latency of a step's layers and two
// cluster barriers (28% of issue slots busy): a step of 256 samples takes 13.5
// us, 25 as two launches.  Eight ranks of 32 samples took 23.
constexpr int kRanks = 16, kCt = 512, kSamples = 16;
constexpr int kSpt = kSamples * HID / kCt;          // samples of a thread (of one unit)
constexpr int kSt = kSamples + 4, kUt = HID + 4;    // a unit's samples and a sample's units, padded
constexpr uint32_t kClusterBatch = 2 * kRanks * kSamples;
constexpr int kOwn = (NP + kRanks - 1) / kRanks, kPer = (kOwn + kCt - 1) / kCt;   // parameters of a rank, of a thread
static_assert(kSpt == 2 || kSpt == 4, "vector loads of a thread's samples");

struct TrainSmem {
    float w1[HID * (IN + 1)], w2[HID * (HID + 1)], w3[OUT * (HID + 1)], b1[HID], b2[HID], b3[OUT];
    alignas(16) float x[IN * kSt];                                                // unit by unit
    alignas(16) float h1[HID * kSt], h2[HID * kSt], d2[HID * kSt], z[OUT * kSt];
    alignas(16) float xs[kSamples * kUt], h1s[kSamples * kUt], h2s[kSamples * kUt];   // sample by sample
    alignas(16) float d1s[kSamples * kUt], d2s[kSamples * kUt], zs[kSamples * 16];
    alignas(16) float grad[NP];
    float loss[kSamples];
    float total_loss;
    uint32_t mask[kSamples];
    int32_t y[kSamples];
};

struct TrainArgs {
    const float* X;
    const int32_t* Y;
    const uint8_t* MK;
    const uint32_t* order;    // the epochs' sample orders, `count` each
    const float* c1;          // Adam's bias corrections of every step
    const float* c2;
    float* losses;            // one per step
    float *p, *m, *v;
    uint32_t count, batch, epochs;
    float lr, b1, b2, eps;
    float mean[IN], sd[IN];
};

// Where parameter i lies in the padded weights.
__device__ __forceinline__ float* weight(TrainSmem& sm, int i) {
    if (i < OB1) return &sm.w1[i / IN * (IN + 1) + i % IN];
    if (i < OW2) return &sm.b1[i - OB1];
    if (i < OB2) return &sm.w2[(i - OW2) / HID * (HID + 1) + (i - OW2) % HID];
    if (i < OW3) return &sm.b2[i - OB2];
    if (i < OB3) return &sm.w3[(i - OW3) / HID * (HID + 1) + (i - OW3) % HID];
    return &sm.b3[i - OB3];
}

// A thread's kSpt samples of one unit.
struct Vals {
    float v[kSpt];
};
__device__ __forceinline__ Vals load_vals(const float* p) {
    Vals r;
    if constexpr (kSpt == 4) *reinterpret_cast<float4*>(r.v) = *reinterpret_cast<const float4*>(p);
    else *reinterpret_cast<float2*>(r.v) = *reinterpret_cast<const float2*>(p);
    return r;
}
__device__ __forceinline__ void store_vals(float* p, const Vals& r) {
    if constexpr (kSpt == 4) *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(r.v);
    else *reinterpret_cast<float2*>(p) = *reinterpret_cast<const float2*>(r.v);
}

// Samples g.. of one unit of a layer: a + the sum over i of w[i * ws] * in[i][g..].
template <int N>
__device__ __forceinline__ Vals layer(const float* w, int ws, const float* in, int g, float a) {
    Vals r;
#pragma unroll
    for (int s = 0; s < kSpt; s++) r.v[s] = a;
#pragma unroll 16
    for (int i = 0; i < N; i++) {
        const float u = w[i * ws];
        const Vals x = load_vals(&in[i * kSt + g]);
#pragma unroll
        for (int s = 0; s < kSpt; s++) r.v[s] += u * x.v[s];
    }
    return r;
}

// A 4 x 4 piece of a weight gradient: the sum over n samples of a[s][0..3] times
// b[s][0..3] (rows of `as` and kUt floats), written to rows of `gs` floats at g
// (added there where `add`).
__device__ __forceinline__ void grad_tile(const float* a, int as, const float* b, int n, float* g, int gs, bool add) {
    float t[4][4] = {};
#pragma unroll 4
    for (int s = 0; s < n; s++) {
        const float4 u = *reinterpret_cast<const float4*>(a + s * as), v = *reinterpret_cast<const float4*>(b + s * kUt);
        const float uu[4] = {u.x, u.y, u.z, u.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int c = 0; c < 4; c++) t[r][c] += uu[r] * vv[c];
    }
#pragma unroll
    for (int r = 0; r < 4; r++) {
        float4* o = reinterpret_cast<float4*>(g + r * gs);
        float4 w = make_float4(t[r][0], t[r][1], t[r][2], t[r][3]);
        if (add) {
            const float4 q = *o;
            w = make_float4(q.x + w.x, q.y + w.y, q.z + w.z, q.w + w.w);
        }
        *o = w;
    }
}

__global__ void __launch_bounds__(kCt, 1) mlp_train_cluster(const __grid_constant__ TrainArgs t) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem[];
    TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, rank = (int)cluster.block_rank();
    for (int i = tid; i < NP; i += kCt) *weight(sm, i) = t.p[i];
    float pp[kPer], pm[kPer], pv[kPer];   // the thread's parameters rank * kOwn + tid + kCt q
    int own[kPer];
#pragma unroll
    for (int q = 0; q < kPer; q++) {
        const int k = tid + kCt * q, i = rank * kOwn + k;
        own[q] = k < kOwn && i < NP ? i : -1;
        pp[q] = own[q] >= 0 ? t.p[i] : 0.0f;
        pm[q] = own[q] >= 0 ? t.m[i] : 0.0f;
        pv[q] = own[q] >= 0 ? t.v[i] : 0.0f;
    }
    const uint32_t per_epoch = (t.count + t.batch - 1) / t.batch, steps = per_epoch * t.epochs;
    // first sample (in the orders) and samples of this rank in step k
    auto share = [&](uint32_t k, uint32_t& first, uint32_t& B) -> uint32_t {
        const uint32_t e = k / per_epoch, b0 = (k % per_epoch) * t.batch;
        B = min(t.batch, t.count - b0);
        const uint32_t per = (B + kRanks - 1) / kRanks, r0 = min(B, per * rank);
        first = e * t.count + b0 + r0;
        return min(per, B - r0);
    };
    // the thread's input values of a pass and, for the first threads, their sample's label and mask
    constexpr int kX = kSamples * IN / kCt, kRow = kCt / IN;   // values of a thread, samples between them
    const int xs = tid / IN, xi = tid % IN;
    const float mu = t.mean[xi], sd = t.sd[xi];
    float nx[kX];
    uint32_t row[kX], lrow = 0;      // their rows in X, loaded a pass ahead: a row waits for its index, the thread does not
    int32_t ny = 0;
    uint32_t nm = 0;
    auto fetch_rows = [&](uint32_t first, uint32_t n) {
#pragma unroll
        for (int q = 0; q < kX; q++) row[q] = (uint32_t)(xs + kRow * q) < n ? t.order[first + xs + kRow * q] : 0xFFFFFFFFu;
        lrow = tid < kSamples && (uint32_t)tid < n ? t.order[first + tid] : 0xFFFFFFFFu;
    };
    auto fetch = [&]() {
#pragma unroll
        for (int q = 0; q < kX; q++) nx[q] = row[q] != 0xFFFFFFFFu ? t.X[(size_t)row[q] * IN + xi] : mu;
        ny = 0;
        nm = 0;
        if (lrow != 0xFFFFFFFFu) {
            ny = t.Y[lrow];
            const uint32_t* mk = reinterpret_cast<const uint32_t*>(t.MK + (size_t)lrow * OUT);
            const uint32_t m0 = mk[0], m1 = mk[1], m2 = mk[2];
#pragma unroll
            for (int k = 0; k < 4; k++)
                nm |= ((m0 >> (8 * k)) & 0xFFu ? 1u << k : 0u) | ((m1 >> (8 * k)) & 0xFFu ? 16u << k : 0u) |
                      ((m2 >> (8 * k)) & 0xFFu ? 256u << k : 0u);
        }
    };
    const int j = tid % HID, g = tid / HID * kSpt;   // the thread's unit and first sample
    // a layer's result in both orders
    auto keep = [&](const Vals& r, float* by_unit, float* by_sample) {
        if (by_unit) store_vals(&by_unit[j * kSt + g], r);
#pragma unroll
        for (int s = 0; s < kSpt; s++) by_sample[(g + s) * kUt + j] = r.v[s];
    };
    uint32_t first, B, n = share(0, first, B);
    auto first_rows = [&](uint32_t k) {              // of step k, if there is one
        uint32_t f2, B2;
        const uint32_t n2 = k < steps ? share(k, f2, B2) : 0;
        fetch_rows(f2, min(n2, (uint32_t)kSamples));
    };
    fetch_rows(first, min(n, (uint32_t)kSamples));
    fetch();
    if (n <= kSamples) first_rows(1);
    float* const mine = own[0] >= 0 ? weight(sm, own[0]) : nullptr;
    for (uint32_t k = 0; k < steps; k++) {
        if (tid == 0) sm.total_loss = 0.0f;
        // at least one pass, so that a rank without samples leaves a gradient of zero
        for (uint32_t s0 = 0; s0 == 0 || s0 < n; s0 += kSamples) {
            const uint32_t ns = n > s0 ? min(n - s0, (uint32_t)kSamples) : 0u;
            if (s0) {
                fetch_rows(first + s0, ns);
                fetch();
                if (s0 + kSamples >= n) first_rows(k + 1);
            }
#pragma unroll
            for (int q = 0; q < kX; q++) {
                const float v = (nx[q] - mu) / sd;   // samples past ns are zeros
                sm.x[xi * kSt + xs + kRow * q] = v;
                sm.xs[(xs + kRow * q) * kUt + xi] = v;
            }
            if (tid < kSamples) {
                sm.y[tid] = ny;
                sm.mask[tid] = nm;
            }
            __syncthreads();
            if (s0 + kSamples >= n && k + 1 < steps) {           // the next step's first rows, and the indices after them
                fetch();
                uint32_t f2, B2;
                if (share(k + 1, f2, B2) <= kSamples) first_rows(k + 2);
            }
            Vals h1 = layer<IN>(&sm.w1[j * (IN + 1)], 1, sm.x, g, sm.b1[j]);
#pragma unroll
            for (int s = 0; s < kSpt; s++) h1.v[s] = fmaxf(h1.v[s], 0.0f);
            keep(h1, sm.h1, sm.h1s);
            __syncthreads();
            Vals h2 = layer<HID>(&sm.w2[j * (HID + 1)], 1, sm.h1, g, sm.b2[j]);
#pragma unroll
            for (int s = 0; s < kSpt; s++) h2.v[s] = fmaxf(h2.v[s], 0.0f);
            keep(h2, sm.h2, sm.h2s);
            __syncthreads();
            // logits and their gradient: 16 lanes per sample, one class each
            if (tid < 16 * kSamples) {
                const int s = tid / 16, o = tid % 16;
                const bool in = (uint32_t)s < ns, cls = o < OUT;
                float z = cls ? sm.b3[o] : 0.0f;
                if (cls) {
#pragma unroll 16
                    for (int i = 0; i < HID; i++) z += sm.w3[o * (HID + 1) + i] * sm.h2[i * kSt + s];
                }
                const bool allowed = in && cls && ((sm.mask[s] >> o) & 1u);
                float mx = allowed ? z : -INFINITY;
#pragma unroll
                for (int d = 8; d; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, d));
                const float e = allowed ? expf(z - mx) : 0.0f;
                float sum = e;
#pragma unroll
                for (int d = 8; d; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
                const int y = sm.y[s];
                const bool label = o == y;
                const float dz = in && cls ? (e / sum - (label ? 1.0f : 0.0f)) / (float)B : 0.0f;
                if (cls) {
                    sm.z[o * kSt + s] = dz;
                    sm.zs[s * 16 + o] = dz;
                    if (label || (o == 0 && (uint32_t)y >= OUT)) sm.loss[s] = in ? -logf((label ? e : 0.0f) / sum) : 0.0f;
                }
            }
            __syncthreads();
            if (tid < 32) {
                float l = tid < (int)ns ? sm.loss[tid] : 0.0f;
#pragma unroll
                for (int d = 16; d; d >>= 1) l += __shfl_down_sync(0xFFFFFFFFu, l, d);
                if (tid == 0) sm.total_loss += l;
            }
            Vals d2 = layer<OUT>(&sm.w3[j], HID + 1, sm.z, g, 0.0f);
#pragma unroll
            for (int s = 0; s < kSpt; s++) d2.v[s] = h2.v[s] > 0.0f ? d2.v[s] : 0.0f;
            keep(d2, sm.d2, sm.d2s);
            __syncthreads();
            Vals d1 = layer<HID>(&sm.w2[j], HID + 1, sm.d2, g, 0.0f);
#pragma unroll
            for (int s = 0; s < kSpt; s++) d1.v[s] = h1.v[s] > 0.0f ? d1.v[s] : 0.0f;
            keep(d1, nullptr, sm.d1s);
            __syncthreads();
            // the rank's share of the gradient: 256 threads for W2, 128 for W1, 48 for W3, the rest for the biases
            const bool add = s0 != 0;
            if (tid < 256) {
                const int r = tid / 16 * 4, c = tid % 16 * 4;
                grad_tile(&sm.d2s[r], kUt, &sm.h1s[c], (int)ns, &sm.grad[OW2 + r * HID + c], HID, add);
            } else if (tid < 384) {
                const int r = (tid - 256) / 8 * 4, c = (tid - 256) % 8 * 4;
                grad_tile(&sm.d1s[r], kUt, &sm.xs[c], (int)ns, &sm.grad[OW1 + r * IN + c], IN, add);
            } else if (tid < 432) {
                const int r = (tid - 384) / 16 * 4, c = (tid - 384) % 16 * 4;
                grad_tile(&sm.zs[r], 16, &sm.h2s[c], (int)ns, &sm.grad[OW3 + r * HID + c], HID, add);
            } else {
                for (int i = tid - 432; i < 2 * HID + OUT; i += kCt - 432) {
                    const float* a = i < HID ? &sm.d1s[i] : i < 2 * HID ? &sm.d2s[i - HID] : &sm.zs[i - 2 * HID];
                    const int st = i < 2 * HID ? kUt : 16, at = i < HID ? OB1 + i : i < 2 * HID ? OB2 + i - HID : OB3 + i - 2 * HID;
                    float r = add ? sm.grad[at] : 0.0f;
                    for (int s = 0; s < (int)ns; s++) r += a[s * st];
                    sm.grad[at] = r;
                }
            }
            __syncthreads();
        }
        cluster.sync();   // every rank's share is in its shared memory
        const float c1 = t.c1[k], c2 = t.c2[k];
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            if (own[q] < 0) continue;
            float gi = 0.0f;
#pragma unroll
            for (int r = 0; r < kRanks; r++) gi += *cluster.map_shared_rank(&sm.grad[own[q]], r);
            adam_value(pp[q], pm[q], pv[q], gi, t.lr, t.b1, t.b2, t.eps, c1, c2);
            float* w = q ? weight(sm, own[q]) : mine;
#pragma unroll
            for (int r = 0; r < kRanks; r++) *cluster.map_shared_rank(w, r) = pp[q];
        }
        if (rank == 0 && tid == kCt - 1) {
            float l = 0.0f;
            for (int r = 0; r < kRanks; r++) l += *cluster.map_shared_rank(&sm.total_loss, r);
            t.losses[k] = l / (float)B;
        }
        if (k + 1 < steps) n = share(k + 1, first, B);
        cluster.sync();   // the weights are the next step's; no rank reads a gradient any more
    }
#pragma unroll
    for (int q = 0; q < kPer; q++)
        if (own[q] >= 0) {
            t.p[own[q]] = pp[q];
            t.m[own[q]] = pm[q];
            t.v[own[q]] = pv[q];
        }
}

uint64_t splitmix(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

double unit_of(uint64_t h) { return ((h >> 11) + 0.5) / 9007199254740992.0; }
double unit(uint64_t seed, uint64_t i) { return unit_of(splitmix(seed ^ splitmix(i))); }

}  // namespace

struct zf_mlp {
    int device = 0;
    float* p = nullptr;       // parameters
    float* m = nullptr;       // Adam first moment
    float* v = nullptr;       // Adam second moment
    float* part = nullptr;    // the CTAs' partial gradients of a batch
    uint32_t cap = 0;         // CTAs `part` holds
    uint8_t* data = nullptr;  // zf_mlp_train's and zf_mlp_predict's rows on the device, kept for the next call
    size_t data_cap = 0;
    std::mutex data_mu;       // held by the calls that use `data`
    cudaEvent_t copied[2] = {nullptr, nullptr};   // zf_mlp_train's uploads, two in turn: the copy has read its source
    int cluster = -1;         // whether mlp_train_cluster fits the device (-1: not asked yet)
    uint32_t step = 0;
    // input standardization (x - mean) / std, fitted by zf_mlp_train on its
    // rows and applied by zf_mlp_train and zf_mlp_predict
    bool scaled = false;
    float mean[32] = {0}, sd[32] = {0};
};

namespace {
uint32_t tiles(uint32_t B) { return B / kTile + (B % kTile != 0); }

zf_status ensure_batch(zf_mlp* n, uint32_t B) {
    const uint32_t t = tiles(B);
    if (t <= n->cap) return ZF_OK;
    if (n->part) cudaFree(n->part);
    n->part = nullptr;
    n->cap = 0;
    if (cudaMalloc(&n->part, (size_t)t * kPart * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        return ZF_ENOMEM;
    }
    n->cap = t;
    return ZF_OK;
}

// Device room for the rows of one call, cut into pieces of at least the given
// sizes; kept by the network up to kKeepData and given back with it.
constexpr size_t kKeepData = 64u << 20;
zf_status ensure_data(zf_mlp* n, const size_t (&bytes)[5], void** const (&out)[5]) {
    size_t total = 0;
    for (size_t b : bytes) total += (b + 255) & ~size_t(255);
    if (total > n->data_cap) {
        if (n->data) cudaFree(n->data);
        n->data = nullptr;
        n->data_cap = 0;
        if (cudaMalloc(&n->data, total) != cudaSuccess) {
            cudaGetLastError();
            return ZF_ENOMEM;
        }
        n->data_cap = total;
    }
    size_t pos = 0;
    for (int i = 0; i < 5; i++) {
        *out[i] = n->data + pos;
        pos += (bytes[i] + 255) & ~size_t(255);
    }
    return ZF_OK;
}
void release_large(zf_mlp* n) {
    if (n->data_cap > kKeepData) {
        cudaFree(n->data);
        n->data = nullptr;
        n->data_cap = 0;
    }
}

cudaLaunchConfig_t cluster_config(cudaLaunchAttribute* at) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(kRanks);
    c.blockDim = dim3(kCt);
    c.dynamicSmemBytes = sizeof(TrainSmem);
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim = {kRanks, 1, 1};
    c.attrs = at;
    c.numAttrs = 1;
    return c;
}
// Whether the current device runs a cluster of kRanks such CTAs (more than eight are a device's choice).
bool cluster_fits() {
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t c = cluster_config(&at);
    int most = 0;
    if (cudaFuncSetAttribute(mlp_train_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)) != cudaSuccess ||
        cudaFuncSetAttribute(mlp_train_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&most, mlp_train_cluster, &c) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return most > 0;
}
cudaError_t launch_cluster(const TrainArgs& args) {
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t c = cluster_config(&at);
    return cudaLaunchKernelEx(&c, mlp_train_cluster, args);
}

Rows plain_rows(const float* X, uint32_t n) {
    Rows r{};
    r.X = X;
    r.n = n;
    return r;
}
}  // namespace

extern "C" {

zf_status zf_mlp_create(int device, uint64_t seed, zf_mlp** out) {
    zf::KeepDevice keep_device;
    if (!out) return ZF_EINVAL;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return ZF_ECUDA;
    auto* n = new zf_mlp();
    n->device = device;
    if (cudaMalloc(&n->p, NP * sizeof(float)) != cudaSuccess || cudaMalloc(&n->m, NP * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&n->v, NP * sizeof(float)) != cudaSuccess ||
        cudaEventCreateWithFlags(&n->copied[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&n->copied[1], cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        zf_mlp_destroy(n);
        return ZF_ENOMEM;
    }
    // He-normal weights (Box-Muller on a counter-based generator), zero biases
    std::vector<float> h(NP, 0.0f);
    auto fill = [&](int off, int rows, int cols) {
        for (int i = 0; i < rows * cols; i++) {
            const double u1 = unit(seed, 2ull * (off + i)), u2 = unit(seed, 2ull * (off + i) + 1);
            const double z = std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
            h[off + i] = (float)(z * std::sqrt(2.0 / cols));
        }
    };
    fill(OW1, HID, IN);
    fill(OW2, HID, HID);
    fill(OW3, OUT, HID);
    zf_status st = zf_mlp_set_params(n, h.data());
    if (st) {
        zf_mlp_destroy(n);
        return st;
    }
    *out = n;
    return ZF_OK;
}

zf_status zf_mlp_destroy(zf_mlp* n) {
    zf::KeepDevice keep_device;
    if (!n) return ZF_OK;
    cudaSetDevice(n->device);
    for (void* q : {(void*)n->p, (void*)n->m, (void*)n->v, (void*)n->part, (void*)n->data})
        if (q) cudaFree(q);
    for (cudaEvent_t e : n->copied)
        if (e) cudaEventDestroy(e);
    delete n;
    return ZF_OK;
}

zf_status zf_mlp_get_params(const zf_mlp* n, float* host) {
    zf::KeepDevice keep_device;
    if (!n || !host) return ZF_EINVAL;
    cudaSetDevice(n->device);
    return cudaMemcpy(host, n->p, NP * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? ZF_OK : ZF_ECUDA;
}

zf_status zf_mlp_set_params(zf_mlp* n, const float* host) {
    zf::KeepDevice keep_device;
    if (!n || !host) return ZF_EINVAL;
    cudaSetDevice(n->device);
    if (cudaMemcpy(n->p, host, NP * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(n->m, 0, NP * sizeof(float)) != cudaSuccess || cudaMemset(n->v, 0, NP * sizeof(float)) != cudaSuccess)
        return ZF_ECUDA;
    n->step = 0;
    n->scaled = false;   // parameters from elsewhere: inputs are taken as given
    return ZF_OK;
}

zf_status zf_mlp_forward(zf_mlp* n, const float* d_x, uint32_t batch, float* d_logits, void* stream) {
    if (!n || (batch && (!d_x || !d_logits))) return ZF_EINVAL;
    if (!batch) return ZF_OK;
    mlp_forward<<<tiles(batch), kThreads, 0, (cudaStream_t)stream>>>(n->p, plain_rows(d_x, batch), d_logits);
    return cudaGetLastError() == cudaSuccess ? ZF_OK : ZF_ECUDA;
}

zf_status zf_mlp_grad(zf_mlp* n, const float* d_x, const int32_t* d_y, const uint8_t* d_mask, uint32_t batch,
                      float* d_grad, float* d_loss, void* stream) {
    if (!n || !batch || !d_x || !d_y || !d_mask || !d_grad) return ZF_EINVAL;
    zf_status st = ensure_batch(n, batch);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    mlp_grad_part<<<tiles(batch), kThreads, 0, s>>>(n->p, plain_rows(d_x, batch), d_y, d_mask, n->part);
    mlp_reduce<<<(NP + 256) / 256, 256, 0, s>>>(n->part, tiles(batch), batch, d_grad, d_loss);
    return cudaGetLastError() == cudaSuccess ? ZF_OK : ZF_ECUDA;
}

zf_status zf_mlp_adam(zf_mlp* n, const float* d_grad, float lr, void* stream) {
    if (!n || !d_grad) return ZF_EINVAL;
    n->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)n->step)), c2 = (float)(1.0 - std::pow(0.999, (double)n->step));
    mlp_adam<<<(NP + 255) / 256, 256, 0, (cudaStream_t)stream>>>(n->p, n->m, n->v, d_grad, lr, b1, b2, 1e-8f, c1, c2);
    return cudaGetLastError() == cudaSuccess ? ZF_OK : ZF_ECUDA;
}

// Mini-batch training on the GPU: the sample order of every epoch is a
// seeded shuffle.  The rows are on the device once, and the host does not wait
// for a step: batches of up to kClusterBatch samples run inside one launch per
// group of epochs (mlp_train_cluster; the next group's orders are shuffled
// meanwhile), larger ones as two launches a step; the losses come back at the
// end.  Three copies and three launches a step, each step waited for, took
// 1,367 us for two epochs of eight batches of 256, two launches a step 509;
// this takes 325.
zf_status zf_mlp_train(zf_mlp* n, const float* h_x, const int32_t* h_y, const uint8_t* h_mask, uint32_t count,
                       uint32_t epochs, uint32_t batch, float lr, uint64_t seed, float* h_losses) {
    zf::KeepDevice keep_device;
    if (!n || !h_x || !h_y || !h_mask || !count || !batch) return ZF_EINVAL;
    cudaSetDevice(n->device);
    std::lock_guard<std::mutex> lock(n->data_mu);
    batch = std::min(batch, count);
    if (n->cluster < 0) n->cluster = cluster_fits();
    const bool cluster = batch <= kClusterBatch && n->cluster;
    const uint32_t steps = count / batch + (count % batch != 0);   // of an epoch
    // epochs whose losses come back at once, and epochs of one launch or upload at most
    const uint32_t back = std::max(1u, std::min(epochs, (1u << 20) / steps));
    const uint32_t most = cluster ? std::max(1u, std::min(std::min(epochs, 64u), (1u << 18) / count)) : 1u;
    const size_t words = (size_t)most * (count + 2 * (size_t)steps);   // orders, then c1 and c2 of every step
    float *dx = nullptr, *dl = nullptr;
    int32_t* dy = nullptr;
    uint8_t* dm = nullptr;
    uint32_t* dord = nullptr;
    zf_status st = cluster ? ZF_OK : ensure_batch(n, batch);
    if (!st)
        st = ensure_data(n, {(size_t)count * IN * sizeof(float), (size_t)count * sizeof(int32_t), (size_t)count * OUT,
                             words * sizeof(uint32_t), (size_t)back * steps * sizeof(float)},
                         {(void**)&dx, (void**)&dy, (void**)&dm, (void**)&dord, (void**)&dl});
    if (st) return st;
    auto done = [&](zf_status s) {
        if (s != ZF_OK) cudaDeviceSynchronize();   // uploads in flight read this call's memory
        release_large(n);
        return s;
    };
    // per-feature mean and standard deviation of the training rows (a
    // constant feature keeps std 1), kept by the network for inference
    double s1[IN] = {0}, s2[IN] = {0};
    for (uint32_t r = 0; r < count; r++)
        for (uint32_t f = 0; f < IN; f++) {
            const double v = h_x[(size_t)r * IN + f];
            s1[f] += v;
            s2[f] += v * v;
        }
    Rows rows = plain_rows(dx, 0);
    rows.scaled = true;
    for (uint32_t f = 0; f < IN; f++) {
        const double mu = s1[f] / count, var = std::max(0.0, s2[f] / count - mu * mu);
        rows.mean[f] = n->mean[f] = (float)mu;
        rows.sd[f] = n->sd[f] = var > 0 ? (float)std::sqrt(var) : 1.0f;
    }
    n->scaled = true;
    if (cudaMemcpy(dx, h_x, (size_t)count * IN * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(dy, h_y, (size_t)count * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(dm, h_mask, (size_t)count * OUT, cudaMemcpyHostToDevice) != cudaSuccess)
        return done(ZF_ECUDA);
    TrainArgs args{};
    if (cluster) {
        args = TrainArgs{dx, dy, dm, nullptr, nullptr, nullptr, nullptr, n->p, n->m, n->v, count, batch, 0,
                         lr, 0.9f, 0.999f, 1e-8f, {}, {}};
        std::copy(rows.mean, rows.mean + IN, args.mean);
        std::copy(rows.sd, rows.sd + IN, args.sd);
    }
    std::vector<uint64_t> hash(count + 1);   // of the counter generator, the same every epoch
    for (uint32_t i = 2; i <= count; i++) hash[i] = splitmix(i);
    // An upload may still be reading its host buffer when cudaMemcpyAsync returns: two take turns, and one is refilled
    // after the event behind its copy
    std::vector<uint32_t> up[2];
    uint32_t uploads = 0;
    std::vector<float> losses((size_t)back * steps);
    uint32_t group = 1;                      // the first launch starts after one shuffle, later ones are larger
    for (uint32_t e0 = 0; e0 < epochs; e0 += back) {
        const uint32_t e1 = std::min(epochs, e0 + back);
        for (uint32_t e = e0; e < e1;) {
            const uint32_t ne = std::min(std::min(group, most), e1 - e);
            std::vector<uint32_t>& buf = up[uploads & 1];
            const cudaEvent_t copied = n->copied[uploads & 1];
            if (uploads >= 2 && cudaEventSynchronize(copied) != cudaSuccess) return done(ZF_ECUDA);
            uploads++;
            buf.resize(words);
            for (uint32_t q = 0; q < ne; q++) {
                uint32_t* order = buf.data() + (size_t)q * count;
                std::iota(order, order + count, 0u);
                for (uint32_t i = count; i > 1; i--) {   // Fisher-Yates with the counter generator
                    const uint32_t j = (uint32_t)(unit_of(splitmix((seed + e + q) ^ hash[i])) * i);
                    std::swap(order[i - 1], order[std::min(j, i - 1)]);
                }
            }
            float* c = reinterpret_cast<float*>(buf.data() + (size_t)ne * count);
            const uint32_t ns = ne * steps;
            for (uint32_t k = 0; k < ns; k++) {
                n->step++;
                c[k] = (float)(1.0 - std::pow(0.9, (double)n->step));
                c[ns + k] = (float)(1.0 - std::pow(0.999, (double)n->step));
            }
            float* dloss = dl + (size_t)(e - e0) * steps;
            if (cudaMemcpyAsync(dord, buf.data(), ((size_t)ne * count + 2 * (size_t)ns) * sizeof(uint32_t), cudaMemcpyHostToDevice,
                                0) != cudaSuccess ||
                cudaEventRecord(copied, 0) != cudaSuccess)
                return done(ZF_ECUDA);
            if (cluster) {
                args.order = dord;
                args.c1 = reinterpret_cast<const float*>(dord + (size_t)ne * count);
                args.c2 = args.c1 + ns;
                args.losses = dloss;
                args.epochs = ne;
                if (launch_cluster(args) != cudaSuccess) return done(ZF_ECUDA);
            } else {
                for (uint32_t k = 0; k < ns; k++) {
                    const uint32_t b0 = k % steps * batch;
                    rows.n = std::min(batch, count - b0);
                    rows.order = dord + (size_t)(k / steps) * count + b0;
                    mlp_grad_part<<<tiles(rows.n), kThreads>>>(n->p, rows, dy, dm, n->part);
                    mlp_reduce_adam<<<(NP + 256) / 256, 256>>>(n->part, tiles(rows.n), rows.n, dloss + k, n->p, n->m, n->v, lr,
                                                               0.9f, 0.999f, 1e-8f, c[k], c[ns + k]);
                }
            }
            if (cudaGetLastError() != cudaSuccess) return done(ZF_ECUDA);
            e += ne;
            group = std::min(2 * group, most);
        }
        if (!h_losses) continue;
        if (cudaMemcpy(losses.data(), dl, (size_t)(e1 - e0) * steps * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
            return done(ZF_ECUDA);
        for (uint32_t e = e0; e < e1; e++) {
            double esum = 0;
            for (uint32_t k = 0; k < steps; k++) esum += losses[(size_t)(e - e0) * steps + k];
            h_losses[e] = (float)(esum / steps);
        }
    }
    return done(cudaDeviceSynchronize() == cudaSuccess ? ZF_OK : ZF_ECUDA);
}

// Class of each row of h_x (count x 32): the argmax of the logits over the
// classes h_mask allows (-1 if none), computed on the GPU.
zf_status zf_mlp_predict(zf_mlp* n, const float* h_x, const uint8_t* h_mask, uint32_t count, int32_t* h_class) {
    zf::KeepDevice keep_device;
    if (!n || !h_x || !h_mask || !h_class) return ZF_EINVAL;
    if (!count) return ZF_OK;
    cudaSetDevice(n->device);
    std::lock_guard<std::mutex> lock(n->data_mu);
    float* dx = nullptr;
    uint8_t* dm = nullptr;
    int32_t* dc = nullptr;
    void* none = nullptr;
    const zf_status st = ensure_data(n, {(size_t)count * IN * sizeof(float), (size_t)count * OUT, (size_t)count * sizeof(int32_t), 0, 0},
                                     {(void**)&dx, (void**)&dm, (void**)&dc, &none, &none});
    if (st) return st;
    auto done = [&](zf_status s) {
        release_large(n);
        return s;
    };
    Rows rows = plain_rows(dx, count);
    rows.scaled = n->scaled;   // the standardization fitted by zf_mlp_train
    std::copy(n->mean, n->mean + IN, rows.mean);
    std::copy(n->sd, n->sd + IN, rows.sd);
    if (cudaMemcpy(dx, h_x, (size_t)count * IN * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(dm, h_mask, (size_t)count * OUT, cudaMemcpyHostToDevice) != cudaSuccess)
        return done(ZF_ECUDA);
    mlp_predict<<<tiles(count), kThreads>>>(n->p, rows, dm, dc);
    if (cudaGetLastError() != cudaSuccess) return done(ZF_ECUDA);
    if (cudaMemcpy(h_class, dc, (size_t)count * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
        return done(ZF_ECUDA);
    return done(ZF_OK);
}

zf_status zf_mlp_get_scaling(const zf_mlp* n, float* mean, float* std_) {
    if (!n || !mean || !std_) return ZF_EINVAL;
    for (uint32_t f = 0; f < IN; f++) {
        mean[f] = n->scaled ? n->mean[f] : 0.0f;
        std_[f] = n->scaled ? n->sd[f] : 1.0f;
    }
    return ZF_OK;
}

}  // extern "C"
