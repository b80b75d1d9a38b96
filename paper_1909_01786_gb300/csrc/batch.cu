// Batched solving: many programs in one launch, one CTA per program.  The
// kernel (kernels.cuh) is compiled once per configuration and frontier mode
// in batch_kernel.cu; this unit dispatches to those instantiations.
#include <cuda_runtime.h>

#include "device.cuh"

namespace aspgpu {

// Batch kernel configurations: threads per CTA and the CTAs per SM the
// register budget is compiled for.
//   0: 256 threads, 3 per SM (programs up to ~66 KB of view)
//   1: 128 threads, 6 per SM (twice the programs in flight, ~30 KB views)
//   2: 768 threads, 1 per SM (lists only; configuration 0 of autotuned batches of
//      no more programs than SMs, where a second CTA per SM would have no work)
int batch_threads(int config) { return config == 2 ? 768 : config == 1 ? 128 : 256; }

// batch_kernel.cu, compiled with BATCH_CONFIG = c and BATCH_LISTS = l
#define ASP_BATCH_DECL(c, l)                                                                                  \
    cudaError_t batch_configure_c##c##_l##l(size_t smem, int *blocks_per_sm);                                   \
    cudaError_t launch_batch_c##c##_l##l(const Dev *devs, const uint32_t *order, uint32_t n, unsigned int *queue, \
                                         int grid, size_t smem, cudaStream_t st);
ASP_BATCH_DECL(0, 0)
ASP_BATCH_DECL(0, 1)
ASP_BATCH_DECL(1, 0)
ASP_BATCH_DECL(1, 1)
ASP_BATCH_DECL(2, 1)
#undef ASP_BATCH_DECL

// lists: the kernels that follow occurrence lists only
cudaError_t batch_configure(int config, bool lists, size_t smem, int *blocks_per_sm)
{
    if (config == 2) return batch_configure_c2_l1(smem, blocks_per_sm);
    if (config == 1) return lists ? batch_configure_c1_l1(smem, blocks_per_sm) : batch_configure_c1_l0(smem, blocks_per_sm);
    return lists ? batch_configure_c0_l1(smem, blocks_per_sm) : batch_configure_c0_l0(smem, blocks_per_sm);
}

cudaError_t launch_batch(int config, bool lists, const Dev *devs, const uint32_t *order, uint32_t n,
                         unsigned int *queue, int grid, size_t smem, cudaStream_t st)
{
    if (config == 2) return launch_batch_c2_l1(devs, order, n, queue, grid, smem, st);
    if (config == 1)
        return lists ? launch_batch_c1_l1(devs, order, n, queue, grid, smem, st)
                     : launch_batch_c1_l0(devs, order, n, queue, grid, smem, st);
    return lists ? launch_batch_c0_l1(devs, order, n, queue, grid, smem, st)
                 : launch_batch_c0_l0(devs, order, n, queue, grid, smem, st);
}

}  // namespace aspgpu
