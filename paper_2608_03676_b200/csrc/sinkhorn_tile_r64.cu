// Phase 1 of a few problems of at most 64 ranks.
#include "sinkhorn_split.cuh"

int taot_launch_sinkhorn_tile_r64(const SinkArgs& a, int32_t B, int sm_count, cudaStream_t st)
{
    // Two CTAs of 128 threads fit on an SM (the builds take 181 to 201 registers); of 64 threads, whose set-up takes longer, four.
    const bool few = B <= 2 * sm_count;
    const unsigned nt = few ? 128 : 64;
    if (a.tol > 0.0f) TAOT_CUDA_OK(taot_launch_chained(few ? sinkhorn_tile_kernel<64, 128, true> : sinkhorn_tile_kernel<64, 64, true>, B, nt, 0, st, a));
    else TAOT_CUDA_OK(taot_launch_chained(few ? sinkhorn_tile_kernel<64, 128, false> : sinkhorn_tile_kernel<64, 64, false>, B, nt, 0, st, a));
    TAOT_CUDA_OK(cudaGetLastError());
    return 1;
}
