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

constexpr int ROW_WORDS = 20;                            // words of a padded weight row in shared memory
constexpr int TRAIN_BATCH = 4096;                        // samples of one SGD step
constexpr int TRAIN_THREADS = 512, TRAIN_WARPS = TRAIN_THREADS / 32;
constexpr int TRAIN_TERMS = N_FEATURES + 2;              // per hidden unit: 16 of W1, b1, w2
constexpr int TRAIN_GRADS = N_HIDDEN * TRAIN_TERMS;      // the gradient without b2's entry
constexpr int TRAIN_PART = TRAIN_GRADS + 4;              // words of one warp's gradient (b2's after the others)
constexpr int TRAIN_CHUNK = 16;                          // samples of a warp in shared memory at a time
static_assert(N_HIDDEN == 64 && N_FEATURES == 16, "layout");
// shared memory: weight rows and b2 | the warps' rows | the warps' gradients
constexpr int TRAIN_W_WORDS = N_HIDDEN * ROW_WORDS + 4;
constexpr int TRAIN_SMEM_WORDS = TRAIN_W_WORDS + TRAIN_WARPS * (TRAIN_CHUNK * N_FEATURES + TRAIN_PART);

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cluster_ctas()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// Barrier of every thread of the cluster; shared-memory writes before it are
// seen after it in every CTA.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Address of the CTA's shared word p in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t remote_shared(const float *p, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

// two fp32 FMAs in one instruction: d = a * b + c by halves
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n\t.reg .b64 x, y, z, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
        "fma.rn.f32x2 w, x, y, z;\n\tmov.b64 {%0, %1}, w;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

// All SGD steps of all epochs in one launch of one cluster.  A step is a chain
// that nothing but the next step's rows can overlap (forward, gradient, sum,
// update), 9.4 MFMA in all, so it is bound by its latency; the weights, the
// momentum and every sum stay on the chip, and cluster barriers (0.3 us) stand
// where a grid barrier and slots in L2 cost about 6 us of a step.
//  - A warp takes a contiguous part of the batch's samples; lane l keeps the
//    weight rows and the 18 gradient sums of hidden units l and l + 32 in
//    registers, so a sample's row is read once (broadcast) for its forward pass
//    and its gradient, and the logit is a warp sum.  With m = d [a_k > 0]:
//    dW1[k] = w2[k] sum m x, db1[k] = w2[k] sum m, dw2[k] = sum d h.
//  - The warps' sums are added per CTA, then each CTA adds its share of the
//    parameters over the CTAs (distributed shared memory), applies the momentum
//    step and stores the new weights into every CTA.
// All sums have a fixed order: results do not depend on timing.  The next
// step's first rows load while the sums are made.
__global__ void __launch_bounds__(TRAIN_THREADS, 1)
mlp_train_kernel(const __grid_constant__ MlpWeights P, const float4 *X, const float *Y, int64_t n, int epochs, float lr,
                 float momentum, float *out)
{
    extern __shared__ float4 train_smem[];
    float *wr = reinterpret_cast<float *>(train_smem);           // [64][20]: W1 row, b1, w2; then b2
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *xs = wr + TRAIN_W_WORDS + warp * (TRAIN_CHUNK * N_FEATURES);                       // this warp's rows
    float *parts = wr + TRAIN_W_WORDS + TRAIN_WARPS * (TRAIN_CHUNK * N_FEATURES);             // [warp][TRAIN_PART]
    const uint32_t rank = cluster_rank(), ctas = cluster_ctas();
    // gradient entry e = term * 64 + k (term 0..15: W1[k][term], 16: b1[k],
    // 17: w2[k]), then b2's: its parameter and its place in the rows
    auto param = [](int e) {
        const int k = e & 63, j = e >> 6;
        return e == TRAIN_GRADS ? MLP_PARAMS - 1 : j < N_FEATURES ? k * N_FEATURES + j : N_FEATURES * N_HIDDEN + (j - N_FEATURES) * N_HIDDEN + k;
    };
    auto place = [](int e) { return e == TRAIN_GRADS ? N_HIDDEN * ROW_WORDS : (e & 63) * ROW_WORDS + (e >> 6); };
    for (int e = tid; e <= TRAIN_GRADS; e += TRAIN_THREADS) wr[place(e)] = P.w[param(e)];
    // this CTA's share of the entries: [e0, e1), `ctas` lanes each
    const int share = (TRAIN_GRADS + 1 + (int)ctas - 1) / (int)ctas, e0 = (int)rank * share;
    const int e1 = min(e0 + share, TRAIN_GRADS + 1), per = TRAIN_THREADS / (int)ctas;
    constexpr int OWN = 3;                                       // entries of a group of lanes (16 CTAs: 73 over 32 groups; 8: 145 over 64)
    float w[OWN], v[OWN];
#pragma unroll
    for (int i = 0; i < OWN; i++) {
        const int e = e0 + tid / (int)ctas + i * per;
        w[i] = e < e1 ? P.w[param(e)] : 0.0f;
        v[i] = 0.0f;
    }
    const int64_t batches = (n + TRAIN_BATCH - 1) / TRAIN_BATCH, steps = batches * epochs;
    const int gw = (int)rank * TRAIN_WARPS + warp, nw = (int)ctas * TRAIN_WARPS;
    float4 px[2];
    float py = 0.0f;
    // rows [r0, r0 + 16) below r1 of the batch at b0
    auto fetch = [&](int64_t b0, int r0, int r1) {
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int r = r0 + (lane >> 2) + 8 * q;
            px[q] = r < r1 ? X[(b0 + r) * 4 + (lane & 3)] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        py = lane < TRAIN_CHUNK && r0 + lane < r1 ? Y[b0 + r0 + lane] : 0.0f;
    };
    auto range = [&](int64_t step, int64_t &b0, int &nb, int &r0, int &r1) {
        b0 = (step % batches) * TRAIN_BATCH;
        nb = (int)(n - b0 < TRAIN_BATCH ? n - b0 : TRAIN_BATCH);
        const int each = (nb + nw - 1) / nw;
        r0 = min(gw * each, nb);
        r1 = min(r0 + each, nb);
    };
    int64_t b0;
    int nb, r0, r1;
    range(0, b0, nb, r0, r1);
    fetch(b0, r0, r1);
    cluster_sync();                                              // every CTA has started and has its weights
    for (int64_t step = 0; step < steps; step++) {
        const float inv = 1.0f / (float)nb;
        float2 W[2][8], S[2][8];
        float b1[2], w2[2], sb[2] = {0.0f, 0.0f}, sh[2] = {0.0f, 0.0f}, sd = 0.0f;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const float4 *r = reinterpret_cast<const float4 *>(wr + (lane + 32 * u) * ROW_WORDS);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 f = r[q];
                W[u][2 * q] = make_float2(f.x, f.y);
                W[u][2 * q + 1] = make_float2(f.z, f.w);
                S[u][2 * q] = S[u][2 * q + 1] = make_float2(0.0f, 0.0f);
            }
            const float4 f = r[4];
            b1[u] = f.x;
            w2[u] = f.y;
        }
        const float b2 = wr[N_HIDDEN * ROW_WORDS];
        for (int c0 = r0; c0 < r1; c0 += TRAIN_CHUNK) {
            if (c0 > r0) fetch(b0, c0, r1);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 2; q++) *reinterpret_cast<float4 *>(xs + ((lane >> 2) + 8 * q) * N_FEATURES + 4 * (lane & 3)) = px[q];
            const float yc = py;
            __syncwarp();
            const int rows = min(TRAIN_CHUNK, r1 - c0);
#pragma unroll 2
            for (int s = 0; s < rows; s++) {
                float2 x[8];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const float4 f = *reinterpret_cast<const float4 *>(xs + s * N_FEATURES + 4 * q);
                    x[2 * q] = make_float2(f.x, f.y);
                    x[2 * q + 1] = make_float2(f.z, f.w);
                }
                float h[2], z = 0.0f;
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    // one chain in the order of mlp_score: near a kink another
                    // rounding puts a sample on the other side of it
                    float a = b1[u];
#pragma unroll
                    for (int q = 0; q < 8; q++) a = fmaf(W[u][q].y, x[q].y, fmaf(W[u][q].x, x[q].x, a));
                    h[u] = fmaxf(a, 0.0f);
                    z = fmaf(w2[u], h[u], z);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
                const float d = (1.0f / (1.0f + expf(-(z + b2))) - __shfl_sync(0xFFFFFFFFu, yc, s)) * inv;
                sd += d;
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const float m = h[u] > 0.0f ? d : 0.0f;
                    const float2 mm = make_float2(m, m);
#pragma unroll
                    for (int q = 0; q < 8; q++) S[u][q] = fma2(mm, x[q], S[u][q]);
                    sb[u] += m;
                    sh[u] = fmaf(d, h[u], sh[u]);
                }
            }
        }
        float *part = parts + warp * TRAIN_PART;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = lane + 32 * u;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                part[(2 * q) * 64 + k] = S[u][q].x;
                part[(2 * q + 1) * 64 + k] = S[u][q].y;
            }
            part[16 * 64 + k] = sb[u];
            part[17 * 64 + k] = sh[u];
        }
        if (lane == 0) part[TRAIN_GRADS] = sd;
        if (step + 1 < steps) {
            range(step + 1, b0, nb, r0, r1);
            fetch(b0, r0, r1);
        }
        __syncthreads();
        // the CTA's sums, in the first warp's place
        for (int e = tid; e <= TRAIN_GRADS; e += TRAIN_THREADS) {
            float g[TRAIN_WARPS];
#pragma unroll
            for (int q = 0; q < TRAIN_WARPS; q++) g[q] = parts[q * TRAIN_PART + e];
#pragma unroll
            for (int o = TRAIN_WARPS / 2; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < o; q++) g[q] += g[q + o];
            parts[e] = e < (N_FEATURES + 1) * 64 ? g[0] * wr[(e & 63) * ROW_WORDS + N_FEATURES + 1] : g[0];
        }
        cluster_sync();
        // this CTA's share: lane c of a group reads CTA c's sum, the group adds
        // them up, applies the step, and lane c stores the weight in CTA c
#pragma unroll
        for (int i = 0; i < OWN; i++) {
            const int e = e0 + tid / (int)ctas + i * per;
            const uint32_t c = (uint32_t)tid % ctas;
            if (i * per >= share) break;                         // the same on every thread
            float g = 0.0f;
            if (e < e1) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(g) : "r"(remote_shared(parts + e, c)) : "memory");
            for (uint32_t o = ctas / 2u; o > 0u; o >>= 1) g += __shfl_xor_sync(0xFFFFFFFFu, g, o);
            v[i] = momentum * v[i] + g;
            w[i] -= lr * v[i];
            if (e < e1) asm volatile("st.shared::cluster.f32 [%0], %1;" :: "r"(remote_shared(wr + place(e), c)), "f"(w[i]) : "memory");
        }
        cluster_sync();
    }
#pragma unroll
    for (int i = 0; i < OWN; i++) {
        const int e = e0 + tid / (int)ctas + i * per;
        if (e < e1 && (uint32_t)tid % ctas == 0u) out[param(e)] = w[i];
    }
}

constexpr int SCORE_THREADS = 256, SCORE_EACH = 2, SCORE_TILE = SCORE_THREADS * SCORE_EACH;   // rows of a tile, two a thread
constexpr int SCORE_SMEM_WORDS = (N_HIDDEN + SCORE_TILE) * ROW_WORDS;

// Inference with the solver's arithmetic (mlp_score): bf16 weights, fp32
// accumulation in the same order, so the scores are the same bits.  Bound by
// reading the rows (64 B each, over the CPU-GPU link when they are in host
// memory): a tile of 512 rows loads coalesced, the next one while this one is
// computed, and goes through shared memory to the threads.  A broadcast weight
// row serves two rows a thread: with one, the reads of shared memory alone took
// 140 us for 1M rows.
__global__ void __launch_bounds__(SCORE_THREADS) mlp_score_kernel(const __grid_constant__ MlpWeightsBf16 P, const float4 *X, int n,
                                                                 float *out)
{
    extern __shared__ float4 score_smem[];
    float *wr = reinterpret_cast<float *>(score_smem), *xs = wr + N_HIDDEN * ROW_WORDS;
    for (int p = threadIdx.x; p < MLP_PARAMS - 1; p += blockDim.x) {
        const int k = p < N_FEATURES * N_HIDDEN ? p / N_FEATURES : p & 63;
        const int j = p < N_FEATURES * N_HIDDEN ? p % N_FEATURES : N_FEATURES + (p - N_FEATURES * N_HIDDEN) / N_HIDDEN;
        wr[k * ROW_WORDS + j] = __uint_as_float((uint32_t)P.w[p] << 16);
    }
    const float b2 = __uint_as_float((uint32_t)P.w[MLP_PARAMS - 1] << 16);
    constexpr int LOADS = SCORE_TILE * N_FEATURES / 4 / SCORE_THREADS;
    float4 next[LOADS];
    const long long words = (long long)n * (N_FEATURES / 4);
    auto fetch = [&](long long tile) {
#pragma unroll
        for (int q = 0; q < LOADS; q++) {
            const long long i = tile * (SCORE_TILE * N_FEATURES / 4) + q * SCORE_THREADS + threadIdx.x;
            next[q] = i < words ? X[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    };
    const long long tiles = ((long long)n + SCORE_TILE - 1) / SCORE_TILE;
    fetch(blockIdx.x);
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < LOADS; q++) {
            const int i = q * SCORE_THREADS + threadIdx.x;
            *reinterpret_cast<float4 *>(xs + (i >> 2) * ROW_WORDS + 4 * (i & 3)) = next[q];
        }
        __syncthreads();
        if (t + gridDim.x < tiles) fetch(t + gridDim.x);
        float x[SCORE_EACH][N_FEATURES], y[SCORE_EACH];
#pragma unroll
        for (int u = 0; u < SCORE_EACH; u++) {
            y[u] = b2;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 f = *reinterpret_cast<const float4 *>(xs + (threadIdx.x + u * SCORE_THREADS) * ROW_WORDS + 4 * q);
                x[u][4 * q] = f.x; x[u][4 * q + 1] = f.y; x[u][4 * q + 2] = f.z; x[u][4 * q + 3] = f.w;
            }
        }
#pragma unroll 4
        for (int k = 0; k < N_HIDDEN; k++) {
            const float4 *r = reinterpret_cast<const float4 *>(wr + k * ROW_WORDS);
            const float4 bw = r[4];
            float a[SCORE_EACH];
#pragma unroll
            for (int u = 0; u < SCORE_EACH; u++) a[u] = bw.x;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float4 f = r[q];
#pragma unroll
                for (int u = 0; u < SCORE_EACH; u++) {
                    a[u] = fmaf(f.x, x[u][4 * q], a[u]); a[u] = fmaf(f.y, x[u][4 * q + 1], a[u]);
                    a[u] = fmaf(f.z, x[u][4 * q + 2], a[u]); a[u] = fmaf(f.w, x[u][4 * q + 3], a[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < SCORE_EACH; u++) y[u] = fmaf(bw.y, fmaxf(a[u], 0.0f), y[u]);
        }
#pragma unroll
        for (int u = 0; u < SCORE_EACH; u++) {
            const long long i = t * SCORE_TILE + u * SCORE_THREADS + threadIdx.x;
            if (i < n) out[i] = y[u];
        }
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
    // the scores go through device memory, at most 4 MB, a chunk of rows at a
    // time; they are not stored to the host's pages from the kernel, where
    // first touches of fresh pages fault (27 ms for 64 MB)
    const int64_t chunk = std::min<int64_t>(n, 1 << 20);
    const size_t smem = SCORE_SMEM_WORDS * sizeof(float);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaMalloc(&dO, (size_t)chunk * sizeof(float));
    for (int64_t i = 0; i < n && e == cudaSuccess; i += chunk) {
        const int m = (int)std::min(chunk, n - i);
        mlp_score_kernel<<<std::min((m + SCORE_TILE - 1) / SCORE_TILE, 608), SCORE_THREADS, smem>>>(W, reinterpret_cast<const float4 *>(X.p + i * N_FEATURES), m, dO);
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
    // one cluster: 16 CTAs where the GPU can place them together, else 8
    const size_t smem = TRAIN_SMEM_WORDS * sizeof(float);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.blockDim = dim3(TRAIN_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    int ctas = 16, fit = 0;
    for (; e == cudaSuccess && ctas >= 8; ctas /= 2) {
        at.val.clusterDim.x = (unsigned)ctas;
        cfg.gridDim = dim3(ctas);
        if (cudaOccupancyMaxActiveClusters(&fit, mlp_train_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); fit = 0; }
        if (fit > 0) break;
    }
    if (e == cudaSuccess && fit < 1) return internal_fail(ASP_E_CUDA, "the training kernel's cluster cannot be resident");
    float *out = nullptr;
    if (e == cudaSuccess) e = cudaMalloc(&out, MLP_PARAMS * sizeof(float));
    if (e == cudaSuccess)
        e = cudaLaunchKernelEx(&cfg, mlp_train_kernel, W, reinterpret_cast<const float4 *>(X.p), Y.p, n, (int)epochs, learning_rate, 0.9f, out);
    if (e == cudaSuccess) e = cudaMemcpy(weights, out, MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToHost);
    if (out) cudaFree(out);
    return e == cudaSuccess ? ASP_OK : mlp_fail(e);
}
