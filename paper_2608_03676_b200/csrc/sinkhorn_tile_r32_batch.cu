// Register-tile Sinkhorn kernel, up to 32 ranks, register-capped build for large batches (32 problems per SM).
#include "sinkhorn_tile.cuh"

int taot_launch_sinkhorn_tile_r32_batch(const SinkArgs& a, int32_t B, int sm_count, cudaStream_t st)
{
    if (a.tol > 0.0f) TAOT_CUDA_OK(taot_launch_chained(sinkhorn_tile_kernel<1, 1, 4, 8, 16, 32, true>, B, 32, 0, st, a, (int64_t)B));
    else TAOT_CUDA_OK(taot_launch_chained(sinkhorn_tile_kernel<1, 1, 4, 8, 16, 32, false>, B, 32, 0, st, a, (int64_t)B));
    TAOT_CUDA_OK(cudaGetLastError());
    return 1;
}
