// Search state around a launch: the reset before a solve, and the exchange of
// a partial assignment and its closure for asp_debug_propagate.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "device.cuh"
#include "store.h"

namespace aspgpu {

namespace {

__device__ __forceinline__ void first_control(const Dev &D, uint32_t n_input)
{
    Ctl c{};
    D.ctl[1] = c;
    c.op = OP_INIT;
    c.cdl = 1u;
    c.tc = c.tb = n_input;
    c.lfill = D.lits_static;
    D.ctl[0] = c;
    Acc a{};
    a.ckey = a.cslot[0] = a.cslot[1] = a.cslot[2] = NO_KEY;
    a.minU = 0xFFFFFFFFu;
    for (int i = 0; i < 4; i++) D.acc[i] = a;
    *D.stats = DevStats{};
    *D.bar = Barrier{};
}

// Clears what a search starts from and writes the first control block: one
// launch where nine memsets and copies stood (about 1 us each on the stream).
// codes: the assignment and levels too (a propagation sets them from its
// input).
__global__ void __launch_bounds__(256) reset_kernel(Dev D, bool codes, uint32_t n_input)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    if (codes) {
        for (uint32_t w = t; w <= D.asg_words; w += nt) D.asg[w] = 0u;
        for (uint32_t v = t; v <= D.nv; v += nt) D.dl[v] = 0;
    }
    for (uint32_t j = t; j < D.J + 2u; j += nt) D.act[j] = 0u;
    for (uint32_t j = t; j < D.J + 4u; j += nt) D.level_start[j] = 0u;
    if (t == 0) first_control(D, n_input);
}

// variables of one block of the input kernels: 256 threads x 32
constexpr uint32_t IN_VARS = 8192;

// The codes (8 per word), levels and reasons of the input, and the number of
// assigned variables of each block of IN_VARS.
__global__ void __launch_bounds__(256) input_codes_kernel(Dev D, const int8_t *partial, uint32_t *counts)
{
    __shared__ uint32_t s_n;
    if (threadIdx.x == 0) s_n = 0u;
    __syncthreads();
    uint32_t n = 0;
    const uint32_t w0 = blockIdx.x * (IN_VARS / 8u);
    for (uint32_t w = w0 + threadIdx.x; w < min(w0 + IN_VARS / 8u, D.asg_words); w += blockDim.x) {
        uint32_t m = 0;
        for (uint32_t q = 0; q < 8u; q++) {
            const uint32_t v = 8u * w + q;
            const int8_t x = v < D.nv ? partial[v] : (int8_t)0;
            if (x) { m |= (x > 0 ? V_T : V_F) << (4u * q); n++; }
        }
        D.asg[w] = m;
    }
    const uint32_t v0 = blockIdx.x * IN_VARS;
    for (uint32_t v = v0 + threadIdx.x; v < min(v0 + IN_VARS, D.nv); v += blockDim.x) {
        D.dl[v] = partial[v] ? 1 : 0;
        D.reason[v] = R_INPUT;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) D.asg[D.asg_words] = 0u;
    if (n) atomicAdd(&s_n, n);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = s_n;
}

// The input's variables on the trail in ascending order: a block starts after
// the counts of the blocks before it, and a warp after those of its block.
// The last block writes the first control block.
__global__ void __launch_bounds__(256) input_trail_kernel(Dev D, const int8_t *partial, const uint32_t *counts)
{
    __shared__ uint32_t s_base, s_warp[8];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_base = 0u;
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t b = threadIdx.x; b < blockIdx.x; b += blockDim.x) before += counts[b];
    if (before) atomicAdd(&s_base, before);
    // the warp's variables: 1024, a row of 32 at a time
    const uint32_t v0 = blockIdx.x * IN_VARS + warp * 1024u;
    uint32_t n = 0;
    for (uint32_t r = 0; r < 32u; r++) {
        const uint32_t v = v0 + 32u * r + lane;
        n += __popc(__ballot_sync(0xFFFFFFFFu, v < D.nv && partial[v] != 0));
    }
    if (lane == 0) s_warp[warp] = n;
    __syncthreads();
    uint32_t pos = s_base;
    for (uint32_t i = 0; i < warp; i++) pos += s_warp[i];
    for (uint32_t r = 0; r < 32u; r++) {
        const uint32_t v = v0 + 32u * r + lane;
        const int8_t x = v < D.nv ? partial[v] : (int8_t)0;
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, x != 0);
        if (x) D.trail[pos + __popc(m & ((1u << lane) - 1u))] = v | (x < 0 ? TRAIL_F : 0u);
        pos += (uint32_t)__popc(m);
    }
    if (blockIdx.x == gridDim.x - 1u && threadIdx.x == blockDim.x - 1u) first_control(D, pos);
}

// The closure, one byte per variable: 1 true, -1 false, 2 both, 0 unassigned.
__global__ void __launch_bounds__(256) closure_kernel(Dev D, int8_t *closure)
{
    const uint32_t nt = gridDim.x * blockDim.x;
    for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < D.asg_words; w += nt) {
        const uint32_t m = D.asg[w];
        unsigned long long out = 0;
        for (uint32_t q = 0; q < 8u; q++) {
            const uint32_t c = (m >> (4u * q)) & 3u;
            out |= (unsigned long long)(uint8_t)(c == V_F ? -1 : c == 3u ? 2 : (int)c) << (8u * q);
        }
        reinterpret_cast<unsigned long long *>(closure)[w] = out;   // the buffer holds 8 x asg_words bytes
    }
}

// literals (and words of the scan) of one block of the occurrence kernels
constexpr uint32_t OCC_BLOCK = 2048;

__global__ void __launch_bounds__(256) occ_count_kernel(Dev D, uint32_t n_lits, uint32_t *count)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_lits; i += gridDim.x * blockDim.x)
        atomicAdd(count + __ldg(D.lits + i), 1u);
}

// Exclusive scan of the n counts into off in three launches: sums of blocks
// of OCC_BLOCK, their scan (one block), then each block's scan on its base.
__global__ void __launch_bounds__(256) occ_sums_kernel(const uint32_t *count, uint32_t n, uint32_t *sums)
{
    __shared__ uint32_t s;
    if (threadIdx.x == 0) s = 0u;
    __syncthreads();
    uint32_t x = 0;
    for (uint32_t i = blockIdx.x * OCC_BLOCK + threadIdx.x; i < min((blockIdx.x + 1u) * OCC_BLOCK, n); i += 256u) x += count[i];
    x = __reduce_add_sync(0xFFFFFFFFu, x);
    if ((threadIdx.x & 31u) == 0u) atomicAdd(&s, x);
    __syncthreads();
    if (threadIdx.x == 0) sums[blockIdx.x] = s;
}

// Exclusive scan over a block of 256 threads; *total its sum.
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t *total)
{
    __shared__ uint32_t s_w[8];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t y = x;
    for (uint32_t o = 1; o < 32u; o <<= 1) {
        const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, y, o);
        if (lane >= o) y += z;
    }
    __syncthreads();
    if (lane == 31u) s_w[warp] = y;
    __syncthreads();
    uint32_t base = 0, sum = 0;
    for (uint32_t i = 0; i < 8u; i++) {
        if (i < warp) base += s_w[i];
        sum += s_w[i];
    }
    *total = sum;
    return base + y - x;
}

__global__ void __launch_bounds__(256) occ_base_kernel(uint32_t *sums, uint32_t n)
{
    uint32_t run = 0;
    for (uint32_t i0 = 0; i0 < n; i0 += 256u) {
        const uint32_t i = i0 + threadIdx.x, x = i < n ? sums[i] : 0u;
        uint32_t total;
        const uint32_t at = run + block_scan(x, &total);
        if (i < n) sums[i] = at;
        run += total;
    }
}

__global__ void __launch_bounds__(256) occ_offsets_kernel(const uint32_t *count, uint32_t n, const uint32_t *sums, uint32_t *off)
{
    uint32_t run = sums[blockIdx.x];
    for (uint32_t i0 = blockIdx.x * OCC_BLOCK; i0 < (blockIdx.x + 1u) * OCC_BLOCK; i0 += 256u) {
        const uint32_t i = i0 + threadIdx.x, x = i < n ? count[i] : 0u;
        uint32_t total;
        const uint32_t at = run + block_scan(x, &total);
        if (i < n) off[i] = at;
        if (i + 1u == n) off[n] = at + x;
        run += total;
    }
}

// First word of bucket L's literals in the rows of the nogoods of more than
// eight literals.
struct RowBase { uint32_t at[BUCKET_MAX + 1]; };

// The entry of literal word i, and its word of the rows.
__device__ __forceinline__ void occ_fill(const Dev &D, uint32_t i, const RowBase &R, const uint32_t *off, uint32_t *count,
                                         Occurrence *occ, uint32_t *rows)
{
    uint32_t L = 2;
    for (uint32_t q = 3; q <= (uint32_t)BUCKET_MAX; q++)
        if (i >= D.bk_base[q]) L = q;
    const uint32_t n = D.bk_n[L], r = i - D.bk_base[L], q = r / n, k = r % n;
    const uint32_t *base = D.lits + D.bk_base[L] + k;
    const uint32_t l = __ldg(D.lits + i);
    uint32_t w[8] = {bucket_nogood_id(L, k), PAD_LIT, PAD_LIT, PAD_LIT, PAD_LIT, PAD_LIT, PAD_LIT, PAD_LIT};
    if (L <= 8u) {
#pragma unroll
        for (uint32_t j = 1; j < 8u; j++)
            if (j < L) w[j] = __ldg(base + (size_t)(q + j < L ? q + j : q + j - L) * n);
    } else {
        w[1] = END_BIT | L;
        w[2] = R.at[L] + k * L;
        rows[w[2] + q] = l;
    }
    uint4 *e = reinterpret_cast<uint4 *>(occ + (__ldcg(off + l) + atomicSub(count + l, 1u) - 1u));
    e[0] = make_uint4(w[0], w[1], w[2], w[3]);
    e[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

__global__ void __launch_bounds__(256) occ_fill_kernel(Dev D, uint32_t n_lits, RowBase R, const uint32_t *off, uint32_t *count,
                                                       Occurrence *occ, uint32_t *rows)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_lits; i += gridDim.x * blockDim.x) occ_fill(D, i, R, off, count, occ, rows);
}

// The whole construction by one block, for small programs: one launch instead
// of six (loading a 20-atom program took 12 % longer with those).
__global__ void __launch_bounds__(256) occ_small_kernel(Dev D, uint32_t n_lits, RowBase R, uint32_t *off, uint32_t *count,
                                                        Occurrence *occ, uint32_t *rows)
{
    const uint32_t n = 2u * D.nv;
    for (uint32_t i = threadIdx.x; i < n; i += 256u) count[i] = 0u;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_lits; i += 256u) atomicAdd(count + __ldg(D.lits + i), 1u);
    __syncthreads();
    uint32_t run = 0;
    for (uint32_t i0 = 0; i0 < n; i0 += 256u) {
        const uint32_t i = i0 + threadIdx.x, x = i < n ? __ldcg(count + i) : 0u;
        uint32_t total;
        const uint32_t at = run + block_scan(x, &total);
        if (i < n) off[i] = at;
        run += total;
    }
    if (threadIdx.x == 0) off[n] = run;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_lits; i += 256u) occ_fill(D, i, R, off, count, occ, rows);
}

// Where each program's models go in the packed words (-1: they do not fit,
// or there are none), by one block: a scan over the programs in order.
__global__ void __launch_bounds__(256) pack_places_kernel(const Dev *devs, uint32_t n, const long long *results, long long *places,
                                                          long long packed)
{
    __shared__ long long s_w[256];
    long long run = 0;
    for (uint32_t i0 = 0; i0 < n; i0 += 256u) {
        const uint32_t i = i0 + threadIdx.x;
        const long long words = i < n ? min(results[4ull * i + 1], devs[i].models_cap) * (long long)((devs[i].na + 63u) / 64u) : 0;
        s_w[threadIdx.x] = words;
        __syncthreads();
        for (uint32_t d = 1; d < 256u; d <<= 1) {
            const long long x = threadIdx.x >= d ? s_w[threadIdx.x - d] : 0;
            __syncthreads();
            s_w[threadIdx.x] += x;
            __syncthreads();
        }
        const long long end = run + s_w[threadIdx.x];
        if (i < n) places[i] = words > 0 && end <= packed ? end - words : -1;
        run += s_w[255];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(128) pack_models_kernel(const Dev *devs, uint32_t n, const long long *results, const long long *places,
                                                          unsigned long long *models)
{
    for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) {
        if (places[i] < 0) continue;
        const long long words = min(results[4ull * i + 1], devs[i].models_cap) * (long long)((devs[i].na + 63u) / 64u);
        for (long long w = threadIdx.x; w < words; w += blockDim.x) models[places[i] + w] = devs[i].models[w];
    }
}

}  // namespace

// After a batch: every program's models into one array, so that one copy
// brings them to the host.
cudaError_t launch_batch_pack(const Dev *devs, uint32_t n, const long long *results, long long *places,
                              unsigned long long *models, int64_t packed, cudaStream_t st)
{
    pack_places_kernel<<<1, 256, 0, st>>>(devs, n, results, places, packed);
    pack_models_kernel<<<(int)std::min<uint32_t>(n, 1216u), 128, 0, st>>>(devs, n, results, places, models);
    return cudaGetLastError();
}

// Words of the rows of the bucket nogoods of more than eight literals.
uint32_t row_words(const Dev &D)
{
    uint32_t w = 0;
    for (uint32_t L = 9; L <= (uint32_t)BUCKET_MAX; L++) w += L * D.bk_n[L];
    return w;
}

// The occurrence lists (device.cuh): off of 2 nv + 1 words, n_lits entries,
// row_words(D) words of rows.  count: 2 nv words, sums: one word per 2048 of
// them.  (On the host this was a random pass over the store, 0.1 s for 8M
// literals.)
cudaError_t launch_occurrences(const Dev &D, uint32_t n_lits, uint32_t *off, Occurrence *occ, uint32_t *rows, uint32_t *count,
                               uint32_t *sums, cudaStream_t st)
{
    RowBase R{};
    for (uint32_t L = 9, w = 0; L <= (uint32_t)BUCKET_MAX; L++) {
        R.at[L] = w;
        w += L * D.bk_n[L];
    }
    const uint32_t n = 2u * D.nv, blocks = (n + OCC_BLOCK - 1u) / OCC_BLOCK;
    // one block also clears and scans the counters of literals without an
    // occurrence.  A load of 4k literals by one block and by six launches: 0.456
    // and 0.470 ms with 20k atoms, 1.33 and 1.20 with 100k, 48.6 and 42.1 with 4M
    if (n_lits <= 8192u && n <= 65536u) {
        occ_small_kernel<<<1, 256, 0, st>>>(D, n_lits, R, off, count, occ, rows);
        return cudaGetLastError();
    }
    const int grid = (int)std::max<uint32_t>(1u, std::min<uint32_t>((n_lits + 255u) / 256u, 4864u));
    cudaError_t e = cudaMemsetAsync(count, 0, (size_t)n * 4, st);
    if (e != cudaSuccess) return e;
    occ_count_kernel<<<grid, 256, 0, st>>>(D, n_lits, count);
    occ_sums_kernel<<<blocks, 256, 0, st>>>(count, n, sums);
    occ_base_kernel<<<1, 256, 0, st>>>(sums, blocks);
    occ_offsets_kernel<<<blocks, 256, 0, st>>>(count, n, sums, off);
    occ_fill_kernel<<<grid, 256, 0, st>>>(D, n_lits, R, off, count, occ, rows);
    return cudaGetLastError();
}

cudaError_t launch_reset(const Dev &D, bool codes, cudaStream_t st)
{
    const uint32_t n = std::max(codes ? D.nv : 0u, D.J + 4u);
    reset_kernel<<<(int)std::min<uint32_t>((n + 255u) / 256u, 1216u), 256, 0, st>>>(D, codes, 0u);
    return cudaGetLastError();
}

// Blocks of the input kernels (one count word each).
uint32_t input_blocks(const Dev &D) { return std::max<uint32_t>(1u, (D.nv + IN_VARS - 1u) / IN_VARS); }

// The state of a propagation from the partial assignment on the device.
cudaError_t launch_input(const Dev &D, const int8_t *partial, uint32_t *counts, cudaStream_t st)
{
    cudaError_t e = launch_reset(D, false, st);
    if (e != cudaSuccess) return e;
    input_codes_kernel<<<input_blocks(D), 256, 0, st>>>(D, partial, counts);
    input_trail_kernel<<<input_blocks(D), 256, 0, st>>>(D, partial, counts);
    return cudaGetLastError();
}

cudaError_t launch_closure(const Dev &D, int8_t *closure, cudaStream_t st)
{
    closure_kernel<<<(int)std::max<uint32_t>(1u, std::min<uint32_t>((D.asg_words + 255u) / 256u, 1216u)), 256, 0, st>>>(D, closure);
    return cudaGetLastError();
}

}  // namespace aspgpu
