// Training and scoring of the learned decision heuristic (not in the paper):
// a 16-64-1 MLP, ReLU hidden layer, logistic output, trained by minibatch SGD
// with momentum on binary cross-entropy.  Training is one persistent kernel
// for all minibatches of all epochs (mlp_train_kernel); scoring is one pass
// over the rows (mlp_score_kernel).  Both read the caller's rows in host
// memory directly where the GPU can (host_readable).  The solver evaluates the
// trained network with bf16 weights and fp32 accumulation (mlp.cuh, mlp_score).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "aspgpu.h"
#include "device.cuh"
#include "mlp.cuh"

namespace aspgpu {

int internal_fail(int code, const char *msg);

namespace {

// Weights by value in the launch: 4.6 KB (fp32) or 2.3 KB (bf16) of kernel
// parameters instead of an allocation and a copy per call.
struct MlpWeights { float w[MLP_PARAMS]; };
struct MlpWeightsBf16 { uint16_t w[MLP_PARAMS]; };

constexpr int TRAIN_BATCH = 4096;                        // samples of one SGD step
constexpr int TRAIN_ROWS = 128, TRAIN_THREADS = 512;     // samples and threads of one CTA
constexpr int TRAIN_CTAS = TRAIN_BATCH / TRAIN_ROWS;
constexpr int TRAIN_TERMS = N_FEATURES + 2;              // per hidden unit: 16 of W1, b1, w2
constexpr int TRAIN_GRADS = N_HIDDEN * TRAIN_TERMS;      // the gradient without b2's entry
constexpr int TRAIN_SLOT = 1156;                         // words of one CTA's gradient (b2's last)
constexpr int TRAIN_ROW = 20;                            // words of a padded row in shared memory
static_assert(TRAIN_GRADS + 1 <= TRAIN_SLOT && TRAIN_THREADS == 4 * TRAIN_ROWS && N_HIDDEN == 64, "layout");
// shared memory: weight rows | feature rows | partial logits | activations,
// later the per-group gradients | dLoss/dlogit
constexpr int TRAIN_SMEM_WORDS = N_HIDDEN * TRAIN_ROW + TRAIN_ROWS * TRAIN_ROW + 4 * TRAIN_ROWS + 8 * TRAIN_GRADS + TRAIN_ROWS + 4;
static_assert(8 * TRAIN_GRADS >= TRAIN_ROWS * (N_HIDDEN + 1), "activations fit where the gradients go");

struct TrainSync { unsigned int count, err; };

// Arrival of every CTA at barrier number gen; false (and a sticky error flag)
// if the others do not come within 20 s.
__device__ bool train_sync(TrainSync *s, unsigned int gen)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned int target = (gen + 1u) * gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(&s->count) : "memory");
        unsigned long long t0 = 0;
        for (unsigned int spins = 1;; spins++) {
            unsigned int c;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&s->count) : "memory");
            if ((int)(c - target) >= 0) break;
            if ((spins & 255u) == 0u) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                if (*(volatile unsigned int *)&s->err || now - t0 > 20000000000ull) {
                    atomicExch(&s->err, 1u);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// All SGD steps of all epochs in one launch.  A step is a chain that nothing
// but the next step's rows can overlap (forward, gradient, sum over CTAs,
// update), about 9.4 MFMA in all, so it is bound by the latency of that chain.
// 32 CTAs hold 128 samples each: fewer CTAs make the arithmetic longer, more
// make the sum longer (every CTA reads every CTA's 4.6 KB).  Forward: four
// threads per sample, 16 hidden units each, weight rows broadcast from shared
// memory.  Gradient: thread (k, group of 16 samples) keeps the 18 sums of
// hidden unit k in registers, so no shuffle and no atomic is needed: with the
// kept mask m = d [a_k > 0], dW1[k] = w2[k] sum m x, db1[k] = w2[k] sum m,
// dw2[k] = sum d h.  Each CTA writes its sums to a slot; after one grid
// barrier every CTA adds the slots in the same order and applies the same
// update to its own copy of the weights and momentum, so weights never leave
// the chip and results do not depend on timing.  The next step's rows load
// while the barrier waits.
__global__ void __launch_bounds__(TRAIN_THREADS, 1)
mlp_train_kernel(const __grid_constant__ MlpWeights P, const float4 *X, const float *Y, int64_t n, int epochs, float lr,
                 float momentum, float *slots, TrainSync *sync, float *out)
{
    extern __shared__ float4 train_smem[];
    float *wr = reinterpret_cast<float *>(train_smem);           // [64][20]: W1 row, b1, w2
    float *xs = wr + N_HIDDEN * TRAIN_ROW;                       // [128][20]
    float *part = xs + TRAIN_ROWS * TRAIN_ROW;                   // [4][128]
    float *as = part + 4 * TRAIN_ROWS;                           // [128][65] hidden activations
    float *red = as;                                             // [8][18][64], after the activations
    float *ds = as + 8 * TRAIN_GRADS;                            // [128], then b2
    const int tid = threadIdx.x;
    // this thread's parameters: entries e of the gradient, e = term * 64 + k
    // (term 0..15: W1[k][term], 16: b1[k], 17: w2[k]), the last one b2
    float w[3], v[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int e = tid + i * TRAIN_THREADS, k = e & 63, j = e >> 6;
        if (e > TRAIN_GRADS) continue;
        const int p = e == TRAIN_GRADS ? MLP_PARAMS - 1 : j < N_FEATURES ? k * N_FEATURES + j : N_FEATURES * N_HIDDEN + (j - N_FEATURES) * N_HIDDEN + k;
        w[i] = P.w[p];
        if (e == TRAIN_GRADS) ds[TRAIN_ROWS] = w[i];
        else wr[k * TRAIN_ROW + j] = w[i];
    }
    const int64_t batches = (n + TRAIN_BATCH - 1) / TRAIN_BATCH, steps = batches * epochs;
    const int row = tid >> 2, col = tid & 3;
    float4 px = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float py = 0.0f;
    auto fetch = [&](int64_t step) {
        const int64_t b0 = (step % batches) * TRAIN_BATCH + (int64_t)blockIdx.x * TRAIN_ROWS;
        px = b0 + row < n ? X[(b0 + row) * 4 + col] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (tid < TRAIN_ROWS) py = b0 + tid < n ? Y[b0 + tid] : 0.0f;
    };
    fetch(0);
    for (int64_t step = 0; step < steps; step++) {
        const int64_t b0 = (step % batches) * TRAIN_BATCH;
        const int nb = (int)(n - b0 < TRAIN_BATCH ? n - b0 : TRAIN_BATCH);
        const float inv = 1.0f / (float)nb;
        *reinterpret_cast<float4 *>(xs + row * TRAIN_ROW + 4 * col) = px;
        const float y = py;
        __syncthreads();
        {   // forward: sample s, hidden units 16 kg .. 16 kg + 15
            const int s = tid & (TRAIN_ROWS - 1), kg = tid >> 7;
            float x[N_FEATURES];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 f = *reinterpret_cast<const float4 *>(xs + s * TRAIN_ROW + 4 * q);
                x[4 * q] = f.x; x[4 * q + 1] = f.y; x[4 * q + 2] = f.z; x[4 * q + 3] = f.w;
            }
            float z = 0.0f;
#pragma unroll 4
            for (int kk = 0; kk < 16; kk++) {
                const int k = kg * 16 + kk;
                const float4 *r = reinterpret_cast<const float4 *>(wr + k * TRAIN_ROW);
                const float4 bw = r[4];
                float a = bw.x;
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float4 f = r[q];
                    a = fmaf(f.x, x[4 * q], a); a = fmaf(f.y, x[4 * q + 1], a);
                    a = fmaf(f.z, x[4 * q + 2], a); a = fmaf(f.w, x[4 * q + 3], a);
                }
                const float h = fmaxf(a, 0.0f);
                as[s * (N_HIDDEN + 1) + k] = h;
                z = fmaf(bw.y, h, z);
            }
            part[kg * TRAIN_ROWS + s] = z;
        }
        __syncthreads();
        if (tid < TRAIN_ROWS) {
            const float z = ds[TRAIN_ROWS] + ((part[tid] + part[TRAIN_ROWS + tid]) + (part[2 * TRAIN_ROWS + tid] + part[3 * TRAIN_ROWS + tid]));
            const float p = 1.0f / (1.0f + expf(-z));
            ds[tid] = (int)blockIdx.x * TRAIN_ROWS + tid < nb ? (p - y) * inv : 0.0f;
        }
        __syncthreads();
        const int k = tid & 63, sg = tid >> 6;
        float acc[TRAIN_TERMS];
#pragma unroll
        for (int q = 0; q < TRAIN_TERMS; q++) acc[q] = 0.0f;
#pragma unroll 4
        for (int i = 0; i < 16; i++) {
            const int s = sg * 16 + i;
            const float d = ds[s], h = as[s * (N_HIDDEN + 1) + k], m = h > 0.0f ? d : 0.0f;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 f = *reinterpret_cast<const float4 *>(xs + s * TRAIN_ROW + 4 * q);
                acc[4 * q] = fmaf(m, f.x, acc[4 * q]); acc[4 * q + 1] = fmaf(m, f.y, acc[4 * q + 1]);
                acc[4 * q + 2] = fmaf(m, f.z, acc[4 * q + 2]); acc[4 * q + 3] = fmaf(m, f.w, acc[4 * q + 3]);
            }
            acc[16] += m;
            acc[17] = fmaf(d, h, acc[17]);
        }
        __syncthreads();                                     // the activations are read
#pragma unroll
        for (int q = 0; q < TRAIN_TERMS; q++) red[sg * TRAIN_GRADS + q * 64 + k] = acc[q];
        __syncthreads();
        float *slot = slots + ((size_t)(step & 1) * gridDim.x + blockIdx.x) * TRAIN_SLOT;
        for (int e = tid; e < TRAIN_GRADS; e += TRAIN_THREADS) {
            float g[8];
#pragma unroll
            for (int q = 0; q < 8; q++) g[q] = red[q * TRAIN_GRADS + e];
            const float sum = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]));
            slot[e] = (e >> 6) < N_FEATURES + 1 ? sum * wr[(e & 63) * TRAIN_ROW + N_FEATURES + 1] : sum;
        }
        if (tid >= TRAIN_THREADS - 32) {                     // b2: the sum of dLoss/dlogit
            const int lane = tid & 31;
            float g = (ds[lane] + ds[lane + 32]) + (ds[lane + 64] + ds[lane + 96]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xFFFFFFFFu, g, o);
            if (lane == 0) slot[TRAIN_GRADS] = g;
        }
        if (step + 1 < steps) fetch(step + 1);
        if (!train_sync(sync, (unsigned int)step)) return;
        const float *all = slots + (size_t)(step & 1) * gridDim.x * TRAIN_SLOT;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const int e = tid + i * TRAIN_THREADS;
            if (e > TRAIN_GRADS) continue;
            float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
            for (int c = 0; c < (int)gridDim.x; c += 4)
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (c + q < (int)gridDim.x) g[q] += __ldcg(all + (size_t)(c + q) * TRAIN_SLOT + e);
            v[i] = momentum * v[i] + ((g[0] + g[1]) + (g[2] + g[3]));
            w[i] -= lr * v[i];
            if (e == TRAIN_GRADS) ds[TRAIN_ROWS] = w[i];
            else wr[(e & 63) * TRAIN_ROW + (e >> 6)] = w[i];
        }
    }
    if (blockIdx.x != 0) return;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int e = tid + i * TRAIN_THREADS, k = e & 63, j = e >> 6;
        if (e > TRAIN_GRADS) continue;
        out[e == TRAIN_GRADS ? MLP_PARAMS - 1 : j < N_FEATURES ? k * N_FEATURES + j : N_FEATURES * N_HIDDEN + (j - N_FEATURES) * N_HIDDEN + k] = w[i];
    }
}

// Inference with the solver's arithmetic (mlp_score): bf16 weights, fp32
// accumulation in the same order, so the scores are the same bits.  Bound by
// reading the rows (64 B each, over the CPU-GPU link when they are in host
// memory); the weights are widened once per CTA and read as broadcast rows.
__global__ void __launch_bounds__(256) mlp_score_kernel(const __grid_constant__ MlpWeightsBf16 P, const float4 *X, int n,
                                                        float *out)
{
    __shared__ float4 rows[N_HIDDEN * TRAIN_ROW / 4];
    float *wr = reinterpret_cast<float *>(rows);
    for (int p = threadIdx.x; p < MLP_PARAMS - 1; p += blockDim.x) {
        const int k = p < N_FEATURES * N_HIDDEN ? p / N_FEATURES : p & 63;
        const int j = p < N_FEATURES * N_HIDDEN ? p % N_FEATURES : N_FEATURES + (p - N_FEATURES * N_HIDDEN) / N_HIDDEN;
        wr[k * TRAIN_ROW + j] = __uint_as_float((uint32_t)P.w[p] << 16);
    }
    const float b2 = __uint_as_float((uint32_t)P.w[MLP_PARAMS - 1] << 16);
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float x[N_FEATURES];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 f = X[(size_t)i * 4 + q];
            x[4 * q] = f.x; x[4 * q + 1] = f.y; x[4 * q + 2] = f.z; x[4 * q + 3] = f.w;
        }
        float y = b2;
#pragma unroll 4
        for (int k = 0; k < N_HIDDEN; k++) {
            const float4 *r = rows + k * (TRAIN_ROW / 4);
            const float4 bw = r[4];
            float a = bw.x;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 f = r[q];
                a = fmaf(f.x, x[4 * q], a); a = fmaf(f.y, x[4 * q + 1], a);
                a = fmaf(f.z, x[4 * q + 2], a); a = fmaf(f.w, x[4 * q + 3], a);
            }
            y = fmaf(bw.y, fmaxf(a, 0.0f), y);
        }
        out[i] = y;
    }
}

// Static prior of heuristic 3: feature 0 + log sigmoid(MLP) per row.
__global__ void mlp_prior_kernel(const uint16_t *Wb, const float *X, int n, float *out)
{
    __shared__ __nv_bfloat16 w[MLP_PARAMS];
    for (int p = threadIdx.x; p < MLP_PARAMS; p += blockDim.x) w[p] = __ushort_as_bfloat16(Wb[p]);
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float x[N_FEATURES];
#pragma unroll
        for (int q = 0; q < N_FEATURES; q++) x[q] = X[(size_t)i * N_FEATURES + q];
        const float z = mlp_score(w, x);
        const float log_p = z >= 0.0f ? -log1pf(__expf(-z)) : z - log1pf(__expf(z));
        out[i] = x[0] + log_p;
    }
}

}  // namespace

// Per-rule prior of heuristic 3 on the device: features uploaded from the
// host, bf16 weights already on the device, result left in d_out.
int mlp_prior(const uint16_t *d_w, const std::vector<float> &features, int64_t n, float *d_out, cudaStream_t st)
{
    if (n <= 0) return ASP_OK;
    float *dX = nullptr;
    const size_t bx = (size_t)n * N_FEATURES * sizeof(float);
    if (cudaMalloc(&dX, bx) != cudaSuccess) { cudaGetLastError(); return internal_fail(ASP_E_OOM, "device allocation failed (prior)"); }
    cudaError_t e = cudaMemcpyAsync(dX, features.data(), bx, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        mlp_prior_kernel<<<(int)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, st>>>(d_w, dX, (int)n, d_out);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(dX);
    if (e != cudaSuccess) return internal_fail(ASP_E_CUDA, cudaGetErrorString(e));
    return ASP_OK;
}

namespace {

// The rows of a host array as the kernels read them: in place where the GPU
// reads pageable host memory through the host's page tables (Grace; 64 MB in
// 340 us, against 386 us for a copy of it and 87 us for the copy's buffer),
// else, or where the rows are not 16-byte aligned, from a device copy.
struct HostRows {
    const float *p = nullptr;
    float *copy = nullptr;
    cudaError_t take(const float *src, size_t bytes)
    {
        int dev = 0, direct = 0, tables = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&direct, cudaDevAttrPageableMemoryAccess, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&tables, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev);
        if (e != cudaSuccess) return e;
        p = src;
        if (direct && tables && (reinterpret_cast<uintptr_t>(src) & 15u) == 0u) return cudaSuccess;
        e = cudaMalloc(&copy, bytes);
        if (e == cudaSuccess) e = cudaMemcpy(copy, src, bytes, cudaMemcpyHostToDevice);
        p = copy;
        return e;
    }
    ~HostRows() { if (copy) cudaFree(copy); }
};

int mlp_fail(cudaError_t e)
{
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return internal_fail(ASP_E_OOM, "device allocation failed");
    }
    return internal_fail(ASP_E_CUDA, cudaGetErrorString(e));
}

}  // namespace

}  // namespace aspgpu

extern "C" int asp_mlp_score(const float *weights, const float *features, int64_t n, float *scores)
{
    using namespace aspgpu;
    if (!weights || !features || !scores || n <= 0 || n > (1ll << 30)) return internal_fail(ASP_E_ARG, "bad argument");
    MlpWeightsBf16 W;
    for (int i = 0; i < MLP_PARAMS; i++) {
        uint32_t u;
        std::memcpy(&u, weights + i, 4);
        W.w[i] = (uint16_t)((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
    }
    HostRows X;
    float *dO = nullptr;
    cudaError_t e = X.take(features, (size_t)n * N_FEATURES * sizeof(float));
    // the scores go through at most 1 MB of device memory, a size that costs
    // 2 us to allocate and free (5 MB: 58 us), a chunk of rows at a time;
    // they are not stored to the host's pages from the kernel, where first
    // touches of fresh pages fault (27 ms for 64 MB)
    const int64_t chunk = std::min<int64_t>(n, 1 << 18);
    if (e == cudaSuccess) e = cudaMalloc(&dO, (size_t)chunk * sizeof(float));
    for (int64_t i = 0; i < n && e == cudaSuccess; i += chunk) {
        const int m = (int)std::min(chunk, n - i);
        mlp_score_kernel<<<(m + 255) / 256, 256>>>(W, reinterpret_cast<const float4 *>(X.p + i * N_FEATURES), m, dO);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpy(scores + i, dO, (size_t)m * sizeof(float), cudaMemcpyDeviceToHost);
    }
    if (dO) cudaFree(dO);
    return e == cudaSuccess ? ASP_OK : mlp_fail(e);
}

extern "C" int asp_train_mlp(const float *features, const float *labels, int64_t n, int32_t epochs,
                             float learning_rate, float *weights)
{
    using namespace aspgpu;
    if (!features || !labels || !weights || n <= 0 || n > (1ll << 30) || epochs < 0)
        return internal_fail(ASP_E_ARG, "bad argument");
    if (epochs == 0) return ASP_OK;
    MlpWeights W;
    std::memcpy(W.w, weights, sizeof(W.w));
    HostRows X, Y;
    cudaError_t e = X.take(features, (size_t)n * N_FEATURES * sizeof(float));
    if (e == cudaSuccess) e = Y.take(labels, (size_t)n * sizeof(float));
    const int grid = (int)std::min<int64_t>(TRAIN_CTAS, (n + TRAIN_ROWS - 1) / TRAIN_ROWS);
    // device memory: slots of two steps | trained weights | barrier
    const size_t words = (size_t)2 * grid * TRAIN_SLOT + TRAIN_SLOT;
    float *mem = nullptr;
    if (e == cudaSuccess) e = cudaMalloc(&mem, words * sizeof(float) + sizeof(TrainSync));
    TrainSync *sync = reinterpret_cast<TrainSync *>(mem + words), host_sync{};
    if (e == cudaSuccess) e = cudaMemsetAsync(sync, 0, sizeof(TrainSync));
    const size_t smem = TRAIN_SMEM_WORDS * sizeof(float);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) {
        const float4 *x4 = reinterpret_cast<const float4 *>(X.p);
        float momentum = 0.9f, *out = mem + (size_t)2 * grid * TRAIN_SLOT;
        int ep = epochs;
        void *args[] = {&W, &x4, &Y.p, &n, &ep, &learning_rate, &momentum, &mem, &sync, &out};
        e = cudaLaunchCooperativeKernel((void *)mlp_train_kernel, dim3(grid), dim3(TRAIN_THREADS), args, smem, 0);
        if (e == cudaSuccess) e = cudaMemcpy(&host_sync, sync, sizeof(TrainSync), cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && !host_sync.err) e = cudaMemcpy(weights, out, MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToHost);
    }
    if (mem) cudaFree(mem);
    if (e != cudaSuccess) return mlp_fail(e);
    return host_sync.err ? internal_fail(ASP_E_DEVICE, "training stopped: a barrier wait ran out") : ASP_OK;
}
