// Phase 1 of a few problems of at most 32 ranks.
#include "sinkhorn_split.cuh"

int taot_launch_sinkhorn_tile_r32(const SinkArgs& a, int32_t B, cudaStream_t st)
{
    if (a.tol > 0.0f) TAOT_CUDA_OK(taot_launch_chained(sinkhorn_tile_kernel<32, 128, true>, B, 128, 0, st, a));
    else TAOT_CUDA_OK(taot_launch_chained(sinkhorn_tile_kernel<32, 128, false>, B, 128, 0, st, a));
    TAOT_CUDA_OK(cudaGetLastError());
    return 1;
}
