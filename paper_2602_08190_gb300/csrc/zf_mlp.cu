// zf_mlp.cu -- the learned selector: a 32 -> 64 -> 64 -> 12 perceptron
// (ReLU hidden layers, FP32) with hand-written forward, backward and Adam
// kernels, and the host loops that train it and use it in zf_plan.
//
// Parameters are one flat FP32 vector: W1[64][32], b1[64], W2[64][64], b2[64],
// W3[12][64], b3[12] (7,052 values).  The loss is the softmax cross-entropy
// over the classes each sample allows (others masked), averaged over the
// batch.  Gradients are summed in a fixed order (eight samples in a CTA, then
// the CTAs), so training is deterministic.
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

// The rows a launch reads: row r of the batch is row inl[r] of X where
// `listed` (a batch of up to kListed rows: its order travels as parameters, so
// no copy stands between the steps), else order[r], or r where order is null.
// They are standardized as (x - mean) / sd where scaled.
constexpr uint32_t kListed = 512;
struct Rows {
    const float* X;
    const uint32_t* order;
    uint32_t n;
    bool scaled, listed;
    float mean[IN], sd[IN];
    uint32_t inl[kListed];
};

__device__ __forceinline__ uint32_t row_of(const Rows& r, uint32_t i) {
    return r.listed ? r.inl[i] : r.order ? r.order[i] : i;
}

// Loads the weights and the CTA's samples (zeros past the batch) and computes the logits sm.z.
__device__ __forceinline__ void forward_tile(const float* __restrict__ p, const Rows& r, MlpSmem& sm) {
    const int tid = threadIdx.x;
    const uint32_t s0 = blockIdx.x * kTile;
    for (int i = tid; i < HID * IN; i += kThreads) sm.w1[i / IN * (IN + 1) + i % IN] = p[OW1 + i];
    for (int i = tid; i < HID * HID; i += kThreads) sm.w2[i / HID * (HID + 1) + i % HID] = p[OW2 + i];
    for (int i = tid; i < OUT * HID; i += kThreads) sm.w3[i / HID * (HID + 1) + i % HID] = p[OW3 + i];
    if (tid < HID) sm.b1[tid] = p[OB1 + tid];
    else if (tid < 2 * HID) sm.b2[tid - HID] = p[OB2 + tid - HID];
    else if (tid < 2 * HID + OUT) sm.b3[tid - 2 * HID] = p[OB3 + tid - 2 * HID];
    {
        static_assert(kThreads == IN * kTile, "one input value per thread");
        const int s = tid / IN, i = tid % IN;
        float v = s0 + s < r.n ? r.X[(size_t)row_of(r, s0 + s) * IN + i] : 0.0f;
        if (r.scaled) v = (v - r.mean[i]) / r.sd[i];
        sm.x[i * kTile + s] = v;
    }
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

__device__ __forceinline__ void adam_one(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v, int i,
                                         float gi, float lr, float b1, float b2, float eps, float c1, float c2) {
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
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

uint64_t splitmix(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

double unit(uint64_t seed, uint64_t i) { return ((splitmix(seed ^ splitmix(i)) >> 11) + 0.5) / 9007199254740992.0; }

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
        cudaMalloc(&n->v, NP * sizeof(float)) != cudaSuccess) {
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
// seeded shuffle; a step is two launches, and the host does not wait for any
// of them: the rows are on the device once, a batch's order is a parameter of
// its launch, and the losses come back at the end.  Three copies and three
// launches a step, each step waited for, took 1,367 us for two epochs of
// eight batches of 256; this takes 509 us.
zf_status zf_mlp_train(zf_mlp* n, const float* h_x, const int32_t* h_y, const uint8_t* h_mask, uint32_t count,
                       uint32_t epochs, uint32_t batch, float lr, uint64_t seed, float* h_losses) {
    zf::KeepDevice keep_device;
    if (!n || !h_x || !h_y || !h_mask || !count || !batch) return ZF_EINVAL;
    cudaSetDevice(n->device);
    std::lock_guard<std::mutex> lock(n->data_mu);
    const uint32_t steps = count / batch + (count % batch != 0);   // of an epoch
    const uint32_t group = std::max(1u, std::min(epochs, (1u << 20) / steps));   // epochs whose losses come back at once
    const bool listed = std::min(batch, count) <= kListed;
    float *dx = nullptr, *dl = nullptr;
    int32_t* dy = nullptr;
    uint8_t* dm = nullptr;
    uint32_t* dord = nullptr;
    zf_status st = ensure_batch(n, std::min(batch, count));
    if (!st)
        st = ensure_data(n, {(size_t)count * IN * sizeof(float), (size_t)count * sizeof(int32_t), (size_t)count * OUT,
                             listed ? 0 : (size_t)count * sizeof(uint32_t), (size_t)group * steps * sizeof(float)},
                         {(void**)&dx, (void**)&dy, (void**)&dm, (void**)&dord, (void**)&dl});
    if (st) return st;
    auto done = [&](zf_status s) {
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
    rows.listed = listed;
    std::vector<uint32_t> order(count);
    std::vector<float> losses((size_t)group * steps);
    for (uint32_t e0 = 0; e0 < epochs; e0 += group) {
        const uint32_t ne = std::min(group, epochs - e0);
        for (uint32_t e = 0; e < ne; e++) {
            std::iota(order.begin(), order.end(), 0u);
            for (uint32_t i = count; i > 1; i--) {   // Fisher-Yates with the counter generator
                const uint32_t j = (uint32_t)(unit(seed + e0 + e, i) * i);
                std::swap(order[i - 1], order[std::min(j, i - 1)]);
            }
            if (!listed && cudaMemcpy(dord, order.data(), (size_t)count * sizeof(uint32_t), cudaMemcpyHostToDevice) != cudaSuccess)
                return done(ZF_ECUDA);
            for (uint32_t k = 0; k < steps; k++) {
                rows.n = std::min(batch, count - k * batch);
                if (listed) std::copy_n(order.begin() + (size_t)k * batch, rows.n, rows.inl);
                else rows.order = dord + (size_t)k * batch;
                n->step++;
                const float c1 = (float)(1.0 - std::pow(0.9, (double)n->step));
                const float c2 = (float)(1.0 - std::pow(0.999, (double)n->step));
                mlp_grad_part<<<tiles(rows.n), kThreads>>>(n->p, rows, dy, dm, n->part);
                mlp_reduce_adam<<<(NP + 256) / 256, 256>>>(n->part, tiles(rows.n), rows.n, dl + (size_t)e * steps + k,
                                                           n->p, n->m, n->v, lr, 0.9f, 0.999f, 1e-8f, c1, c2);
            }
        }
        if (cudaGetLastError() != cudaSuccess) return done(ZF_ECUDA);
        if (!h_losses) continue;
        if (cudaMemcpy(losses.data(), dl, (size_t)ne * steps * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
            return done(ZF_ECUDA);
        for (uint32_t e = 0; e < ne; e++) {
            double esum = 0;
            for (uint32_t k = 0; k < steps; k++) esum += losses[(size_t)e * steps + k];
            h_losses[e0 + e] = (float)(esum / steps);
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
