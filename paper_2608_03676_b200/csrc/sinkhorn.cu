// Phase 1: the kernel that takes any problem (sinkhorn_generic.cuh) and the choice of kernels.
#include "sinkhorn_generic.cuh"

namespace {

__global__ void __launch_bounds__(1024) sinkhorn_kernel(SinkArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (a.early) taot_release();
    taot_await();
    taot_release();
    if (a.only_marked && a.iters[blockIdx.x] != kHandBack) return;
    generic_problem(a, blockIdx.x, smem_raw);
}

}  // namespace

int taot_launch_sinkhorn_tile(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st);
int taot_launch_sinkhorn_cluster(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st, bool finish = false);
int taot_launch_sinkhorn_tiered(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st);
int taot_launch_sinkhorn_wide(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st);
int taot_launch_sinkhorn_class(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st);
int taot_launch_sinkhorn_dense_tc(taot_handle_t h, const SinkArgs& a, int32_t B, float* ws_tc, cudaStream_t st);

// Caller-supplied supply / demand vectors (the stand-alone entry point; inside taot_plan they come from integer
// loads and are always finite): a problem whose s or d holds a NaN or an infinity has no solution.  One warp per
// problem rereads the inputs after the solve; for such a problem it clears the plan, reports 0 iterations and sets
// TAOT_INFO_NONFINITE.  The solve kernels themselves never index with a value derived from s or d and all their
// loops are bounded, so whatever they computed on that problem before is harmless and is overwritten here.
__global__ void __launch_bounds__(128)
sinkhorn_input_guard_kernel(const float* __restrict__ s, const float* __restrict__ d, int32_t B, int32_t R,
                            float* plan, int32_t* iters, float* row_err, int32_t* info)
{
    const int lane = threadIdx.x & 31;
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    taot_await();
    if (b >= B) return;
    bool bad = false;
    for (int r = lane; r < R; r += 32) bad |= !isfinite(s[b * R + r]) || !isfinite(d[b * R + r]);
    if (!__any_sync(0xffffffffu, bad)) return;
    float* out = plan + b * (int64_t)R * R;
    for (int64_t q = lane; q < (int64_t)R * R; q += 32) out[q] = 0.0f;
    if (lane == 0) {
        iters[b] = 0;
        row_err[b] = 0.0f;
        atomicOr(info + b, TAOT_INFO_NONFINITE);
    }
}

int taot_launch_sinkhorn_guard(taot_handle_t h, const float* d_s, const float* d_d, int32_t B, float* d_plan,
                               int32_t* d_iters, float* d_row_err, int32_t* d_info, cudaStream_t st)
{
    TAOT_CUDA_OK(taot_launch_chained(sinkhorn_input_guard_kernel, (B + 3) / 4, 128, 0, st, d_s, d_d, B, h->p.R, d_plan, d_iters, d_row_err, d_info));
    return 1;
}

// Costs with classes of interchangeable ranks: the class kernels beyond 256 ranks and, up to there, for a caller's own
// batch with a fixed iteration count (R > 32: below, the register tiles are as fast).  Inside taot_plan, and in tolerance mode,
// Phase 1 stays on the tile and tier-sum kernels: the placement that follows decides exact ties (experts of one node's
// ranks on one cold rank) by the last bits of the hint, so its kernel is part of the result.
bool taot_sinkhorn_takes_classes(taot_handle_t h, bool from_loads)
{
    const taot_params& p = h->p;
    return h->cls_kind && (p.R > 256 || (!from_loads && p.tol <= 0.0f && p.R > 32));
}

int taot_launch_sinkhorn(taot_handle_t h, const float* d_s, const float* d_d, int32_t B, float* d_plan,
                         int32_t* d_iters, float* d_row_err, int32_t* d_info, float* d_kt, cudaStream_t st, float* d_tc, bool from_loads,
                         bool early)
{
    const taot_params& p = h->p;
    SinkArgs a;
    a.C = h->d_C; a.rowlse0 = h->d_rowlse0;
    a.R = p.R; a.kcap = h->kcap;
    a.inv_eps = 1.0 / (double)p.eps;
    a.eps0 = p.eps0; a.max_iters = p.max_iters; a.tol = p.tol;
    a.check_every = p.check_every < 1 ? 1 : p.check_every;
    a.skip_solved = 0;
    a.early = early ? 1 : 0;
    // Problems with ranks that have both supply and demand can be larger than the capacity.  Up to 256 ranks those of at most
    // 128 supply ranks, which the register tiles hold, are solved whichever kernel handed them back; beyond 256 ranks all are.
    a.plan_rows = p.R > 256 ? p.R : (p.R > 128 ? 128 : 0);
    a.kt_global = h->kcap_global > 0 ? d_kt : nullptr;
    a.kcap_global = h->kcap_global;
    const int NT = p.R <= 32 ? 32 : (p.R <= 64 ? 128 : (p.R <= 128 ? 256 : (p.R <= 256 ? 512 : 1024)));
    const size_t smem = generic_smem_bytes(p.R, NT, h->kcap);
    TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int launched = 0;
    // the global scratch (if any) holds p.L problems: larger batches go through in slices
    const int32_t slice = a.kt_global ? p.L : B;
    for (int32_t b0 = 0; b0 < B; b0 += slice) {
        const int32_t nb = (B - b0) < slice ? (B - b0) : slice;
        a.s = d_s + (int64_t)b0 * p.R; a.d = d_d + (int64_t)b0 * p.R;
        a.plan = d_plan + (int64_t)b0 * p.R * p.R; a.iters = d_iters + b0; a.row_err = d_row_err + b0;
        a.info = d_info + b0;
        a.skip_solved = 0;
        const bool classes = taot_sinkhorn_takes_classes(h, from_loads);
        const int nt = classes ? taot_launch_sinkhorn_class(h, a, nb, st) : taot_launch_sinkhorn_tiered(h, a, nb, st);
        if (nt < 0) return nt;
        if (nt > 0) {
            // complete, except for problems handed back: with classes those that have a rank with both supply and demand, which
            // beyond 256 ranks go to the clusters below (one problem of 1024 ranks 1.8 ms there, 12.4 in the kernel at the
            // end), and what does not fit there to the same solve as at the end, in the same launch (one more launch would
            // cost every call 2 us)
            launched += nt;
            a.only_marked = 1;
            if (p.R > 256) {
                a.skip_solved = 1;
                const int n = taot_launch_sinkhorn_cluster(h, a, nb, st, true);
                if (n < 0) return n;
                launched += n;
                if (n > 0) continue;
            }
        } else if (p.R <= 256) {
            // fast path: kernel matrix in registers; problems it cannot hold (or whose fp32 sums leave the
            // safe range) come back marked and are solved by the shared-memory kernel below
            a.only_marked = 1;
            const int n = taot_launch_sinkhorn_tile(h, a, nb, st);
            if (n < 0) return n;
            launched += n;
        } else {
            // beyond 256 ranks.  A large batch with a short fixed count and a Gibbs kernel inside fp32 (or more than 512
            // ranks): the whole batch as dense products on the tensor cores (complete: nothing is handed on)
            if (p.R > 512 || p.max_iters < TAOT_WIDE_MIN_ITERS) {
                const int ntc = taot_launch_sinkhorn_dense_tc(h, a, nb, d_tc, st);
                if (ntc < 0) return ntc;
                if (ntc > 0) { launched += ntc; continue; }
            }
            // otherwise up to 512 ranks one CTA holds the compacted matrix in its registers and shared memory, whatever
            // the number of supply ranks; what it hands back (supports that overlap), and larger problems, go to four-CTA
            // clusters that hold it in distributed shared memory; what those hand back (or everything, if no slice fits) to
            // the kernel below with the matrix in workspace
            a.skip_solved = 0;
            const int nw = taot_launch_sinkhorn_wide(h, a, nb, st);
            if (nw < 0) return nw;
            a.skip_solved = nw;
            const int n = taot_launch_sinkhorn_cluster(h, a, nb, st);
            if (n < 0) return n;
            launched += nw + n;
            a.only_marked = nw + n > 0 ? 1 : 0;
        }
        // This kernel may release the one behind it before it has waited only with a kernel in front that has waited for the merge:
        // the matching kernel, set up from there, reads loads that the merge wrote
        SinkArgs last = a;
        last.early = a.early && launched > 0;
        TAOT_CUDA_OK(taot_launch_chained(sinkhorn_kernel, nb, NT, smem, st, last));
        launched += 1;
    }
    return launched;
}
