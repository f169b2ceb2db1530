// Internal definitions shared by the translation units of libtaot (never installed).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "taot.h"
#include "taot_measure.h"

// Elements of topk_idx one CTA of the histogram / reassignment kernels owns.  A chunk never
// crosses a (layer, source rank) segment, so a segment of SEG = (T/R)*k elements has
// NC = ceil(SEG / TAOT_CHUNK) chunks, the last one possibly short.
#define TAOT_CHUNK 16384
#define TAOT_STREAM_THREADS 256            // threads of the streaming kernels: 64 elements each
#define TAOT_MAX_TIERS 8                   // distinct bonus values the bit-set auction handles
#define TAOT_MERGE_PARTS 8                 // CTAs that share the merge of one layer's chunk counts (256-rank tables)
#define TAOT_HOST_GROUP_BYTES (2 << 20)    // routing table from which a host call is split into layer groups
// Costs without structure at 257 to 512 ranks, large batches with a fixed count: from this many iterations on the kernel with the
// matrix in one CTA (sinkhorn_wide.cu), below it the dense products on the tensor cores (sinkhorn_dense_tc.cu), whose time does
// not depend on the supports.  512 ranks, 54 / 256 supply ranks against the dense products, ms:
//   iterations       256 problems          1024 problems          4096 problems
//       10        0.21 / 0.57 : 0.70     0.65 / 1.86 : 1.21      2.5 / 7.2 : 3.6
//       40        0.25 / 0.75 : 1.93     0.77 / 2.50 : 2.43      3.0 / 9.8 : 5.9
//       64        0.28 / 0.90 : 2.91     0.91 / 3.04 : 3.42      3.5 / 11.9 : 7.8
//      500        1.01 / 3.64 : 20.8     3.46 / 12.6 : 21.3     13.8 / 50.2 : 41.7
// So it is no line at which one becomes faster: with few supply ranks the one-CTA kernel always is.  From 64 iterations on it is
// up to 1024 problems whatever the loads; below, the dense products are up to twice as fast where half of the ranks have
// supply, and 1.4 to 8 times as slow where a tenth has.
#define TAOT_WIDE_MIN_ITERS 64
#define TAOT_MAX_GROUPS 6                  // layer groups taot_plan overlaps on internal streams

struct taot_handle_s {
    taot_params p;
    int device;
    int sm_count;
    // topology, device copies
    int32_t* d_e2r;          // [E]
    float* d_C;              // [R,R]
    float* d_B;              // [R,R] topology preference (given or derived)
    double* d_rowlse0;       // [R]  LSE_j(-C_ij/eps) over all ranks j: the first u-update with v = 1
    float* d_gibbs;          // [4][R,R] exp(-C/eps) and its transpose, each as TF32-exact high and low parts (tensor-core
                             // solve: where a call can take it and max C/eps <= 20), else null
    int32_t* d_rank_off;     // [R+1] CSR of experts by home rank
    int32_t* d_rank_list;    // [E]
    uint32_t* d_tiermask;    // [ntiers][W][R hosts] bit r of word w set iff bonus(32w + r -> host) == tierval[t]; null if ntiers == 0
    int32_t* d_torder;       // [E+S+1] target at each position
    int32_t* d_tdest;        // [E+S+1] destination rank of each target (R for the undeliverable bin)
    float* d_tierval;        // [ntiers] distinct values of the auction bonus matrix, descending
    int32_t ntiers;          // 0: too many distinct values, the auction scans densely
    uint32_t* d_bidlist;     // [nbid] every (tier, win count) pair, best score first: w << 8 | t, bit 31 = next has the same score
    uint32_t* d_bident;      // [ntiers][S+1] the same by pair: position << 16 | tie << 14 | tiers that score higher << 11 | w
    int32_t* d_hostcls;      // [R] hosts that see every rank at the same bonus share a number
    int32_t bid_ties;        // some pairs have equal scores
    int32_t nbid;            // 0: no list (no tiers, or price step <= 0): the auction scans densely
    int32_t* d_merge_part;   // [L][TAOT_MERGE_PARTS][E] expert loads of the parts of a layer's merge, or null (one CTA per layer)
    int32_t* d_merge_cnt;    // [L] parts of a layer's merge that are done; zero between calls
    // Classes of interchangeable ranks of the cost matrix, for the class kernels of Phase 1 (sinkhorn_class.cu)
    int32_t cls_kind;        // 0 none, 1 dense (at most 32 classes), 2 tree (three tiers between the classes)
    int32_t cls_nc, cls_gpl, cls_npg;
    float cls_tier[3];
    uint16_t* d_cls;         // [R] slot of each rank's class
    int32_t* d_cls_off;      // [slots + 1] CSR of ranks by slot
    uint16_t* d_cls_list;    // [R]
    double* d_cls_lse0;      // [slots]
    float* d_cls_cost;       // [nc][nc] (dense)
    int32_t tier_ok;         // 1: C has a node / rail-group structure the tier-by-tier kernels are built for and R is 256, 512 or 1024
    float tier_cost[3];      // its three costs off the diagonal: same node, same rail group, otherwise
    int32_t tier_node, tier_group;   // ranks per node and per rail group of that structure (8 / 32, 4 / 16, 4 / 32 or 16 / 32)
    // derived sizes
    int64_t seg;             // elements per (layer, rank) segment
    int32_t nc;              // chunks per segment
    int32_t kcap;            // Sinkhorn kernel-matrix capacity in floats per problem (shared memory)
    int64_t kcap_global;     // same, global-memory scratch per problem (R > 256 only), else 0
    // workspace layout (byte offsets)
    size_t off_cc, off_excess, off_spare, off_s, off_d, off_nrem, off_t12, off_kt, off_dc, off_wp, off_cyc, off_tc;
    size_t off_tb, off_tbflag;   // one-byte copy of the routing table (see tb_ok) and one flag per chunk (a value that is no expert)
    int32_t wp_ok;               // 1: dispatch keeps its counting pass's counts by warp for the scatter (off_wp)
    int32_t tb_ok;               // 1: the histogram pass also leaves the table as one byte per entry (E <= 256 experts,
                                 // segments of a multiple of 16 entries) for the reassignment to read instead of the table
    size_t ws_bytes;
    // host-call staging layout (byte offsets into d_ws of taot_plan_host)
    size_t hoff_topk, hoff_new, hoff_n, hoff_el, hoff_rl, hoff_ex, hoff_sp, hoff_plan, hoff_it, hoff_err,
           hoff_se, hoff_st, hoff_X, hoff_rounds, hoff_info, hoff_ws;
    size_t host_ws_bytes;
    int32_t last_launches;
    int32_t profiling;
    cudaEvent_t ev[6];
    // Layer groups of taot_plan (large routing tables only): group g is a view of this handle on layers
    // [group_l0[g], group_l0[g] + group[g]->p.L) -- same topology pointers, workspace offsets moved to the group's
    // first layer -- planned on a stream of its own so that the bandwidth-bound stages of one group run under the
    // latency-bound stages of another.  ngroups <= 1: one group on the caller's stream.
    int32_t is_view;                           // a view owns nothing
    int32_t ngroups;
    taot_handle_s* group[TAOT_MAX_GROUPS];
    int32_t group_l0[TAOT_MAX_GROUPS];
    int32_t group_len[TAOT_MAX_GROUPS];
    cudaStream_t gstream[TAOT_MAX_GROUPS];     // [0] unused: group 0 runs on the caller's stream
    cudaEvent_t ev_fork, ev_hist[TAOT_MAX_GROUPS], ev_join[TAOT_MAX_GROUPS];
    // Layer groups of the host calls (tables of at least TAOT_HOST_GROUP_BYTES): views like the ones above, each on a stream
    // of its own (gstream), so that copies in, kernels and copies out of different groups run side by side.  hgroups is set by
    // taot_create, the rest when a host call is in sight.
    int32_t hgroups;
    taot_handle_s* hgroup[TAOT_MAX_GROUPS];
    int32_t hgroup_l0[TAOT_MAX_GROUPS + 1];
    cudaStream_t bstream;                      // the one-byte copies of the groups' tables are made here, after all histograms
    cudaEvent_t ev_bytes[TAOT_MAX_GROUPS];     // group g's copy is there
};

static inline size_t taot_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// kernel launchers (each returns the number of kernels it enqueued, or a negative taot_status)
// d_info == nullptr: the flags of the chunks are all that is left of values that are no expert
int taot_launch_histogram(taot_handle_t h, const int32_t* d_topk, int32_t* d_cc, int32_t* d_info, cudaStream_t st,
                          void* ws = nullptr, bool write_bytes = true);
// the table as one byte per entry, by a few CTAs that leave the other SMs alone (returns 0 if this handle keeps no such copy)
int taot_launch_table_bytes(taot_handle_t h, const int32_t* d_topk, void* ws, cudaStream_t st);
int taot_launch_merge(taot_handle_t h, const int32_t* d_cc, int32_t* d_n, int32_t* d_expert_load,
                      int32_t* d_rank_load, int32_t* d_excess, int32_t* d_spare, float* d_s, float* d_d,
                      cudaStream_t st, int32_t* d_info = nullptr, const int32_t* d_chunk_bad = nullptr,
                      int32_t* d_info_out = nullptr);   // d_info_out: starts the call's status words from the chunks' flags
int taot_launch_excess_spare(taot_handle_t h, const int32_t* d_rank_load, int32_t B, int32_t* d_excess,
                             int32_t* d_spare, float* d_s, float* d_d, cudaStream_t st);
int taot_launch_sinkhorn(taot_handle_t h, const float* d_s, const float* d_d, int32_t B, float* d_plan,
                         int32_t* d_iters, float* d_row_err, int32_t* d_info, float* d_kt, cudaStream_t st,
                         float* d_tc = nullptr, bool from_loads = false, bool early = false);   // from_loads: called by taot_plan; early: its kernels
                                                                                       // let the matching kernel be set up beside them
bool taot_sinkhorn_takes_classes(taot_handle_t h, bool from_loads);
size_t taot_sinkhorn_tc_ws_floats(int32_t R, int32_t B);
int taot_launch_sinkhorn_guard(taot_handle_t h, const float* d_s, const float* d_d, int32_t B, float* d_plan,
                               int32_t* d_iters, float* d_row_err, int32_t* d_info, cudaStream_t st);
int taot_launch_match(taot_handle_t h, const int32_t* d_n, const int32_t* d_expert_load,
                      const int32_t* d_rank_load, const float* d_plan, int32_t* d_slot_expert,
                      int32_t* d_slot_tokens, int32_t* d_X, int32_t* d_rounds, int32_t* d_info,
                      int32_t* d_nrem, float* d_t12, cudaStream_t st, long long* d_cyc = nullptr,
                      bool early = false);   // early: behind a Phase 1 launched with `early`, see match_kernel
int taot_launch_assign(taot_handle_t h, const int32_t* d_topk, void* ws, const int32_t* d_slot_expert,
                       const int32_t* d_X, int32_t* d_new_idx, int32_t* d_info, cudaStream_t st);

int taot_launch_report(taot_handle_t h, const int32_t* d_expert_load, const int32_t* d_rank_load,
                       const int32_t* d_slot_expert, const int32_t* d_X, double lambda, taot_report_row* d_rows,
                       int32_t* d_spill, int32_t* d_load_after, int32_t* d_slot_moved, int32_t* d_slot_kind,
                       cudaStream_t st);

// Whether the counting pass of dispatch leaves its counts by warp span, 16 bytes per bin and chunk, for the scatter, which otherwise
// counts its spans again: not where a chunk has fewer entries than half the bins, and not where one scatter CTA fills an SM
// (beyond 1816 bins: nothing hides those reads) unless a chunk has eight entries per bin.  Kept against counted again, us, by
// entries per segment (layers x ranks chunks as in brackets):
//     385 bins, 64 ranks     256: 56.9 : 57.1 [3840]     1024:  87 :  97 [3840]     16384: 51 : 59 [192]
//    1281 bins, 256 ranks    256:  118 : 109  [2048]     1024: 143 : 158 [2048]     16384: 43 : 44 [256]
//    2049 bins, 256 ranks    256:  212 : 169  [2048]     4096: 257 : 199 [1792]     16384: 56 : 55 [256]
//    3073 bins, 256 ranks    256:  328 : 244  [2048]     4096: 386 : 298 [1792]     16384: 84 : 80 [256]
static inline bool taot_dispatch_keeps_counts(int64_t bins, int64_t seg)
{
    const int64_t entries = seg < TAOT_CHUNK ? seg : TAOT_CHUNK;
    return bins <= 1816 ? 2 * entries >= bins : entries >= 8 * bins;
}
int taot_launch_dispatch(taot_handle_t h, const int32_t* d_new_idx, int32_t* d_send_counts, int32_t* d_target_counts,
                         int32_t* d_perm, int32_t* d_info, void* ws, cudaStream_t st);

// Launch of a kernel that may be set up while the kernel before it on the stream still runs (programmatic dependent launch):
// its blocks are placed once every block of that kernel has called taot_release() or ended, and wait in taot_await() until that
// kernel has ended and its writes are visible.  Every kernel of a chain calls taot_await() before it reads or writes anything
// of the call; launched the ordinary way both are no-ops.
__device__ __forceinline__ void taot_await() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void taot_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t taot_launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// the same as clusters of `cluster` CTAs
template <class... P, class... A>
cudaError_t taot_launch_chained_cluster(void (*kernel)(P...), unsigned grid, unsigned block, unsigned cluster, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

#define TAOT_CUDA_OK(expr)                              \
    do {                                                \
        cudaError_t _e = (expr);                        \
        if (_e != cudaSuccess) return TAOT_ERR_CUDA;    \
    } while (0)
