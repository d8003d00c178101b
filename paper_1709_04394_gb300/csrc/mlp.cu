// mlp.cu -- the schedule MLP: 6 -> 64 tanh -> 64 tanh -> 1, fp32 master
// parameters, forward and backward with their bf16 roundings and fp32
// accumulation, Adam. Parameters are one flat vector
// [W1 (64x6 row-major), b1 (64), W2 (64x64), b2 (64), W3 (64), b3 (1)].
// The network proposes the next annealing step (Sec. 5.4 cites adaptive
// steps); the histogram overlap judges every proposal.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "device.cuh"
#include "internal.h"

namespace gbmc {

namespace cg = cooperative_groups;

namespace {
// Adam's 1 - beta^k of the steps of one training launch.
constexpr uint64_t kMlpStepsPerLaunch = 256;
struct MlpBias {
    float c1[kMlpStepsPerLaunch], c2[kMlpStepsPerLaunch];
};
}  // namespace

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ---- one thread block: 16 samples, 256 threads ----
//
// Thread t computes hidden unit t & 63 of the samples t >> 6, + 4, + 8, + 12: four
// sums per weight read. The weights lie in shared memory rounded to bf16; rows of W2
// are 68 words apart, so that 128-bit reads of 32 rows and 32-bit reads along a row are
// both free of conflicts. Shared-memory reads bound the layers: four at a time.
constexpr int kMlpThreads = 256, kMlpSamples = 16, kMlpW2Row = kMlpHidden + 4;
constexpr int kMlpCtas = (int)kMlpMaxBatch / kMlpSamples;  // of a gradient's cluster: 8

struct alignas(16) MlpWeights {
    float W1[kMlpHidden * kMlpIn], b1[kMlpHidden], W2[kMlpHidden * kMlpW2Row], b2[kMlpHidden], W3[kMlpHidden], b3[1];
};
// Offset in floats of parameter q within MlpWeights.
__device__ __forceinline__ uint32_t mlp_slot(uint32_t q) {
    if (q < (uint32_t)kOffW2) return q;
    if (q < (uint32_t)kOffB2) {
        const uint32_t e = q - kOffW2;
        return kOffW2 + (e / kMlpHidden) * kMlpW2Row + e % kMlpHidden;
    }
    return q + kMlpHidden * (kMlpW2Row - kMlpHidden);
}

struct alignas(16) MlpSamples {
    float x[kMlpSamples][kMlpIn], h1[kMlpSamples][kMlpHidden], h2[kMlpSamples][kMlpHidden], y[kMlpSamples];
};

__device__ __forceinline__ void mlp_load_weights(MlpWeights& w, const float* __restrict__ p) {
    float* f = reinterpret_cast<float*>(&w);
    for (uint32_t q = threadIdx.x; q < (uint32_t)kMlpParams; q += kMlpThreads) f[mlp_slot(q)] = bf(p[q]);
}

// Loads n <= 16 samples (the others as zeros) and runs them forward; whole block.
__device__ __forceinline__ void mlp_forward_block(const MlpWeights& w, MlpSamples& s, const float* __restrict__ X,
                                                  uint32_t n) {
    const uint32_t t = threadIdx.x, j = t & 63u, g = t >> 6;
    for (uint32_t i = t; i < kMlpSamples * kMlpIn; i += kMlpThreads)
        s.x[i / kMlpIn][i % kMlpIn] = i < n * kMlpIn ? X[i] : 0.f;
    __syncthreads();  // (the weights too)
    float a[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        a[m] = w.b1[j];
#pragma unroll
        for (int i = 0; i < kMlpIn; ++i) a[m] += w.W1[j * kMlpIn + i] * s.x[g + 4 * m][i];
        s.h1[g + 4 * m][j] = tanhf(a[m]);
        a[m] = w.b2[j];
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kMlpHidden; k += 4) {
        const float4 wk = *reinterpret_cast<const float4*>(&w.W2[j * kMlpW2Row + k]);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float4 h = *reinterpret_cast<const float4*>(&s.h1[g + 4 * m][k]);
            a[m] += wk.x * h.x;
            a[m] += wk.y * h.y;
            a[m] += wk.z * h.z;
            a[m] += wk.w * h.w;
        }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) s.h2[g + 4 * m][j] = tanhf(a[m]);
    __syncthreads();
    // outputs: a warp per sample
    const uint32_t lane = t & 31u;
    for (uint32_t b = t >> 5; b < kMlpSamples; b += kMlpThreads / 32) {
        const float v = warp_sum(w.W3[lane] * s.h2[b][lane] + w.W3[lane + 32] * s.h2[b][lane + 32]);
        if (lane == 0) s.y[b] = v + w.b3[0];
    }
    __syncthreads();
}

// Batch inference, 16 samples per block: 1517 samples 114 us (one thread each) -> 8.6 us.
__global__ void __launch_bounds__(kMlpThreads) k_mlp_forward(const float* __restrict__ p, const float* __restrict__ X,
                                                             uint32_t B, float* __restrict__ Y) {
    __shared__ MlpWeights w;
    __shared__ MlpSamples s;
    mlp_load_weights(w, p);
    for (uint32_t b0 = blockIdx.x * kMlpSamples; b0 < B; b0 += gridDim.x * kMlpSamples) {
        const uint32_t n = B - b0 < (uint32_t)kMlpSamples ? B - b0 : (uint32_t)kMlpSamples;
        mlp_forward_block(w, s, X + (uint64_t)b0 * kMlpIn, n);
        if (threadIdx.x < n) Y[b0 + threadIdx.x] = s.y[threadIdx.x];
        __syncthreads();  // before the next samples overwrite these
    }
}

cudaError_t launch_mlp_forward(const float* p, const float* X, uint32_t B, float* Y, cudaStream_t s) {
    const uint32_t blocks = (B + kMlpSamples - 1) / kMlpSamples;
    k_mlp_forward<<<blocks < 1216u ? blocks : 1216u, kMlpThreads, 0, s>>>(p, X, B, Y);
    count_launch();
    return cudaGetLastError();
}

// ---- gradients and training: one cluster of eight blocks ----
//
// Gradient of (1/B) sum_b (y_b - t_b)^2 / 2 over a minibatch of B <= 128 samples:
// block r takes samples 16 r .. 16 r + 15 and sums their share of every parameter's
// gradient in its shared memory; after a cluster barrier block r adds up the eight
// shares (in block order: deterministic) of its eighth of the parameters. Training
// goes on from there without leaving the chip: the block applies Adam to its eighth
// (parameter and moments in registers for the whole launch), writes the rounded
// weights into the shared memory of all eight blocks, and a second cluster barrier
// starts the next step.
//
// Bound: latency (a step is 1.7 million multiply-adds over eight SMs; a dozen block
// barriers, two cluster barriers, remote reads and writes). One block with one thread
// per sample, and a launch each for gradient and Adam, took 174 us per gradient of 128
// samples and 182 us per training step; this takes 14 us (launch included) and 7.1 us.
struct alignas(16) MlpShared {
    MlpWeights w;
    MlpSamples s;
    float dz2[kMlpSamples][kMlpHidden], dz1[kMlpSamples][kMlpHidden];
    float part[kMlpParams + 3];  // this block's share of the gradient
    float dy[kMlpSamples], loss;
};
constexpr uint32_t kMlpSlice = (kMlpParams + kMlpCtas - 1) / kMlpCtas;       // parameters per block: 585
constexpr int kMlpOwn = (int)((kMlpSlice + kMlpThreads - 1) / kMlpThreads);  // and per thread: 3

// This block's share of the gradient and loss over samples [16 r, B); whole block.
__device__ __forceinline__ void mlp_backward_block(MlpShared& S, const float* __restrict__ X, const float* __restrict__ T,
                                                   uint32_t B, uint32_t rank) {
    const uint32_t t = threadIdx.x, j = t & 63u, g = t >> 6;
    const uint32_t b0 = rank * kMlpSamples, n = b0 >= B ? 0u : B - b0 < (uint32_t)kMlpSamples ? B - b0 : kMlpSamples;
    mlp_forward_block(S.w, S.s, X + (uint64_t)b0 * kMlpIn, n);
    if (t < 32) {
        const float d = t < n ? S.s.y[t] - T[b0 + t] : 0.f;
        if (t < kMlpSamples) S.dy[t] = d / (float)B;
        const float l = warp_sum(0.5f * d * d);
        if (t == 0) S.loss = l;
    }
    __syncthreads();
    // back through layer 3 and the second tanh
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const float hv = S.s.h2[g + 4 * m][j];
        S.dz2[g + 4 * m][j] = S.dy[g + 4 * m] * S.w.W3[j] * (1.f - hv * hv);
    }
    __syncthreads();
    // through layer 2 and the first tanh
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int i = 0; i < kMlpHidden; i += 4) {
        float wi[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) wi[k] = S.w.W2[(i + k) * kMlpW2Row + j];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float4 z = *reinterpret_cast<const float4*>(&S.dz2[g + 4 * m][i]);
            a[m] += z.x * wi[0];
            a[m] += z.y * wi[1];
            a[m] += z.z * wi[2];
            a[m] += z.w * wi[3];
        }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const float hv = S.s.h1[g + 4 * m][j];
        S.dz1[g + 4 * m][j] = a[m] * (1.f - hv * hv);
    }
    __syncthreads();
    // W2: row t >> 2, columns 4 (t & 3) + 16 i .. + 3
    {
        float4 acc[4] = {};
        const uint32_t c = 4u * (t & 3u);
#pragma unroll 4
        for (int b = 0; b < kMlpSamples; ++b) {
            const float z = S.dz2[b][t >> 2];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 h = *reinterpret_cast<const float4*>(&S.s.h1[b][c + 16 * i]);
                acc[i].x += z * h.x;
                acc[i].y += z * h.y;
                acc[i].z += z * h.z;
                acc[i].w += z * h.w;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4*>(&S.part[kOffW2 + (t >> 2) * kMlpHidden + c + 16 * i]) = acc[i];
    }
    // the others: 384 of W1, 64 each of b1, b2, W3, one b3
    for (uint32_t q = t; q < 577u; q += kMlpThreads) {
        float acc = 0.f;
        uint32_t at;
        if (q < 384u) {
            for (int b = 0; b < kMlpSamples; ++b) acc += S.dz1[b][q / kMlpIn] * S.s.x[b][q % kMlpIn];
            at = kOffW1 + q;
        } else if (q < 448u) {
            for (int b = 0; b < kMlpSamples; ++b) acc += S.dz1[b][q - 384u];
            at = kOffB1 + q - 384u;
        } else if (q < 512u) {
            for (int b = 0; b < kMlpSamples; ++b) acc += S.dz2[b][q - 448u];
            at = kOffB2 + q - 448u;
        } else if (q < 576u) {
            for (int b = 0; b < kMlpSamples; ++b) acc += S.dy[b] * S.s.h2[b][q - 512u];
            at = kOffW3 + q - 512u;
        } else {
            for (int b = 0; b < kMlpSamples; ++b) acc += S.dy[b];
            at = kOffB3;
        }
        S.part[at] = acc;
    }
}

__global__ void __cluster_dims__(kMlpCtas, 1, 1) __launch_bounds__(kMlpThreads)
    k_mlp_grad(const float* __restrict__ p, const float* __restrict__ X, const float* __restrict__ T, uint32_t B,
               float* __restrict__ g, float* __restrict__ loss) {
    extern __shared__ __align__(16) unsigned char raw[];
    MlpShared& S = *reinterpret_cast<MlpShared*>(raw);
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank();
    mlp_load_weights(S.w, p);
    mlp_backward_block(S, X, T, B, rank);
    cluster.sync();
    for (uint32_t i = threadIdx.x; i < kMlpSlice && rank * kMlpSlice + i < (uint32_t)kMlpParams; i += kMlpThreads) {
        const uint32_t q = rank * kMlpSlice + i;
        float a = 0.f;
#pragma unroll
        for (int r = 0; r < kMlpCtas; ++r) a += *cluster.map_shared_rank(&S.part[q], r);
        g[q] = a;
    }
    if (rank == 0 && threadIdx.x == 0) {
        float l = 0.f;
#pragma unroll
        for (int r = 0; r < kMlpCtas; ++r) l += *cluster.map_shared_rank(&S.loss, r);
        loss[0] = l / (float)B;
    }
    cluster.sync();  // no block leaves while others read its shared memory
}

cudaError_t launch_mlp_grad(const float* p, const float* X, const float* T, uint32_t B, float* g, float* loss,
                            cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpShared));
    if (e != cudaSuccess) return e;
    k_mlp_grad<<<kMlpCtas, kMlpThreads, sizeof(MlpShared), s>>>(p, X, T, B, g, loss);
    count_launch();
    return cudaGetLastError();
}

// Adam of one parameter; c1, c2: 1 - beta^k.
__device__ __forceinline__ void adam_update(float& p, float g, float& m, float& v, float lr, float c1, float c2) {
    m = 0.9f * m + 0.1f * g;
    v = 0.999f * v + 0.001f * g * g;
    p -= lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
}

// n_steps training steps from minibatch `batch0` of an epoch of nb on.
__global__ void __cluster_dims__(kMlpCtas, 1, 1) __launch_bounds__(kMlpThreads)
    k_mlp_train(float* __restrict__ p, float* __restrict__ m_all, float* __restrict__ v_all, const float* __restrict__ X,
                const float* __restrict__ T, uint32_t n, uint32_t batch, uint32_t batch0, uint32_t n_steps, float lr,
                float* __restrict__ losses, const __grid_constant__ MlpBias bias) {
    extern __shared__ __align__(16) unsigned char raw[];
    MlpShared& S = *reinterpret_cast<MlpShared*>(raw);
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), nb = (n + batch - 1u) / batch;
    float pq[kMlpOwn], mq[kMlpOwn], vq[kMlpOwn];
#pragma unroll
    for (int i = 0; i < kMlpOwn; ++i) {
        const uint32_t o = threadIdx.x + i * kMlpThreads, q = rank * kMlpSlice + o;
        const bool has = o < kMlpSlice && q < (uint32_t)kMlpParams;
        pq[i] = has ? p[q] : 0.f;
        mq[i] = has ? m_all[q] : 0.f;
        vq[i] = has ? v_all[q] : 0.f;
    }
    mlp_load_weights(S.w, p);
    cluster.sync();
    for (uint32_t k = 0; k < n_steps; ++k) {
        const uint32_t first = (batch0 + k) % nb * batch, B = n - first < batch ? n - first : batch;
        mlp_backward_block(S, X + (uint64_t)first * kMlpIn, T + first, B, rank);
        cluster.sync();
#pragma unroll
        for (int i = 0; i < kMlpOwn; ++i) {
            const uint32_t o = threadIdx.x + i * kMlpThreads, q = rank * kMlpSlice + o;
            if (o >= kMlpSlice || q >= (uint32_t)kMlpParams) continue;
            float g = 0.f;
#pragma unroll
            for (int r = 0; r < kMlpCtas; ++r) g += *cluster.map_shared_rank(&S.part[q], r);
            adam_update(pq[i], g, mq[i], vq[i], lr, bias.c1[k], bias.c2[k]);
            float* f = reinterpret_cast<float*>(&S.w) + mlp_slot(q);
            const float rounded = bf(pq[i]);
#pragma unroll
            for (int r = 0; r < kMlpCtas; ++r) *cluster.map_shared_rank(f, r) = rounded;
        }
        if (losses && rank == 0 && threadIdx.x == 0) {
            float l = 0.f;
#pragma unroll
            for (int r = 0; r < kMlpCtas; ++r) l += *cluster.map_shared_rank(&S.loss, r);
            losses[k] = l / (float)B;
        }
        cluster.sync();
    }
#pragma unroll
    for (int i = 0; i < kMlpOwn; ++i) {
        const uint32_t o = threadIdx.x + i * kMlpThreads, q = rank * kMlpSlice + o;
        if (o >= kMlpSlice || q >= (uint32_t)kMlpParams) continue;
        p[q] = pq[i];
        m_all[q] = mq[i];
        v_all[q] = vq[i];
    }
}

static void adam_bias(uint32_t k, float& c1, float& c2) {
    c1 = 1.0f - (float)pow(0.9, (double)k);
    c2 = 1.0f - (float)pow(0.999, (double)k);
}

cudaError_t launch_mlp_train(float* p, float* m, float* v, const float* X, const float* T, uint32_t n, uint32_t epochs,
                             uint32_t batch, float lr, float* losses, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpShared));
    if (e != cudaSuccess) return e;
    const uint64_t nb = (n + batch - 1u) / batch, steps = nb * epochs;
    for (uint64_t k0 = 0; k0 < steps; k0 += kMlpStepsPerLaunch) {
        const uint32_t ns = (uint32_t)(steps - k0 < kMlpStepsPerLaunch ? steps - k0 : kMlpStepsPerLaunch);
        MlpBias bias;
        for (uint32_t k = 0; k < ns; ++k) adam_bias((uint32_t)(k0 + k + 1), bias.c1[k], bias.c2[k]);
        k_mlp_train<<<kMlpCtas, kMlpThreads, sizeof(MlpShared), s>>>(p, m, v, X, T, n, batch, (uint32_t)(k0 % nb), ns, lr,
                                                                    losses ? losses + k0 : nullptr, bias);
        count_launch();
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

__global__ void k_mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, float lr, float c1, float c2) {
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (uint32_t)kMlpParams) return;
    float pq = p[q], mq = m[q], vq = v[q];
    adam_update(pq, g[q], mq, vq, lr, c1, c2);
    m[q] = mq;
    v[q] = vq;
    p[q] = pq;
}

cudaError_t launch_mlp_adam(float* p, const float* g, float* m, float* v, uint32_t k, float lr, cudaStream_t s) {
    float c1, c2;
    adam_bias(k, c1, c2);
    k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, s>>>(p, g, m, v, lr, c1, c2);
    count_launch();
    return cudaGetLastError();
}

}  // namespace gbmc
