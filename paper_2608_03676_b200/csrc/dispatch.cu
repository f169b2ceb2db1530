// Dispatch metadata after the planner (what the token all-to-all that follows needs; the paper's system passes
// the rewritten routing to its dispatcher, Method / System Design).  For every source rank: how many of its
// entries execute on each rank, how many go to each target (expert or guest slot), and the position of every
// entry in the rank's send buffer ordered by (destination rank, target, original order) -- a stable counting
// sort with E + S keys, done as three passes over chunks of <= 16384 entries:
//   dispatch_count_kernel    one CTA per chunk, every warp over its own contiguous span: counts over the E + S targets, with
//                            one more bin for values that are no target, and their sums over the spans before
//   dispatch_offsets_kernel  one CTA per (layer, source rank): totals, exclusive scan in destination order,
//                            per-chunk bases (in place), send counts per destination rank
//   dispatch_scatter_kernel  one CTA per chunk: each warp walks its span in order, 32 entries at a time; the lanes with
//                            the same target inside a step are found by OR-ing lane bits into a shared-memory
//                            word per target and ranked by lane, so the order stays stable
// 12 bytes of HBM traffic per entry (two reads of the table, one write of the positions), but what bounds it is random access
// to shared memory: 32 lanes on 385 targets meet in the same bank 3.3 deep, and a step makes five such accesses beside the
// count's one.  The count is made by warp, so that the scatter need not count its spans again where a chunk has entries
// enough for its bins (taot_dispatch_keeps_counts): 64 ranks x 58 layers (1 GB) 877 -> 757 us.  (One cluster per segment that reads the table once was built and made the same accesses in the same time:
// 0.83 to 1.05 ms at 64 ranks x 58 layers; finding the lanes by votes 1.05, by match 1.8 ms.)
#include "taot_internal.cuh"

namespace {

constexpr int kThreads = TAOT_STREAM_THREADS;
constexpr int kWarps = kThreads / 32;
constexpr int kWarpSpan = TAOT_CHUNK / kWarps;

struct DispatchArgs {
    const int32_t* idx;        // [L,T,k] rewritten routing table
    int32_t* dc;               // [L,R,NC,NB] chunk counts, then chunk bases
    uint16_t* wp;              // [L,R,NC,kWarps,NB] entries of the bin in the spans of the chunk before this warp's, or null
    const int32_t* torder;     // [NB] bin at each sorted position
    const int32_t* tdest;      // [NB] destination rank of each bin (R for the undeliverable bin)
    int32_t* send_counts;      // [L,R,R]
    int32_t* target_counts;    // [L,R,NB-1] or null
    int32_t* perm;             // [L,T,k]
    int32_t* info;
    int64_t layer_elems, seg;
    int32_t nc, R, NB;
    int32_t vec_ok;            // the table's chunks start on 16-byte boundaries
};

__device__ __forceinline__ void chunk_span(const DispatchArgs& a, int64_t id, int64_t& goff, int32_t& len)
{
    const int32_t c = (int32_t)(id % a.nc);
    const int64_t lr = id / a.nc;
    const int64_t start = (int64_t)c * TAOT_CHUNK;
    len = (int32_t)((a.seg - start) < (int64_t)TAOT_CHUNK ? (a.seg - start) : (int64_t)TAOT_CHUNK);
    goff = (lr / a.R) * a.layer_elems + (lr % a.R) * a.seg + start;
}

__device__ __forceinline__ int bin_of(int32_t v, int NB) { return (unsigned)v < (unsigned)(NB - 1) ? v : NB - 1; }

__device__ __forceinline__ void count_add(uint32_t addr) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory"); }

// a warp's counts over its contiguous span of n entries
__device__ __forceinline__ void count_span(const int32_t* src, int n, int32_t* counts, int NB, bool vec_ok)
{
    const int lane = threadIdx.x & 31;
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(counts);
    int i = 0;
    if (vec_ok && n == kWarpSpan) {
        const int4* src4 = reinterpret_cast<const int4*>(src) + lane;
#pragma unroll 1
        for (int h = 0; h < kWarpSpan / 128; h += 8) {
            int4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = __ldcs(src4 + (h + u) * 32);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                count_add(mine + 4u * (uint32_t)bin_of(x[u].x, NB));
                count_add(mine + 4u * (uint32_t)bin_of(x[u].y, NB));
                count_add(mine + 4u * (uint32_t)bin_of(x[u].z, NB));
                count_add(mine + 4u * (uint32_t)bin_of(x[u].w, NB));
            }
        }
        i = kWarpSpan;
    }
    for (i += lane; i < n; i += 32) count_add(mine + 4u * (uint32_t)bin_of(__ldcs(src + i), NB));
}

// Counts of a chunk by warp, each over its contiguous span, and from them the chunk's counts and (a.wp) the sums over the spans
// before each warp's.  (At most 16384 entries before a span: 16 bits.)
__global__ void __launch_bounds__(kThreads)
dispatch_count_kernel(DispatchArgs a)
{
    extern __shared__ int32_t wh[];            // [kWarps][NB]
    const int tid = threadIdx.x, warp = tid >> 5, NB = a.NB;
    const int64_t id = blockIdx.x;
    int64_t goff; int32_t len;
    chunk_span(a, id, goff, len);
    for (int q = tid; q < kWarps * NB; q += kThreads) wh[q] = 0;
    __syncthreads();
    taot_await();
    taot_release();
    const int s0 = warp * kWarpSpan;
    count_span(a.idx + goff + s0, min(len - s0, kWarpSpan), wh + warp * NB, NB, a.vec_ok);
    __syncthreads();
    int32_t* out = a.dc + id * NB;
    if (!a.wp) {
        for (int b = tid; b < NB; b += kThreads) {
            int32_t run = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) run += wh[w * NB + b];
            out[b] = run;
        }
        return;
    }
    uint16_t* wp = a.wp + id * kWarps * NB;
    for (int b = tid; b < NB; b += kThreads) {
        int32_t run = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            wp[w * NB + b] = (uint16_t)run;
            run += wh[w * NB + b];
        }
        out[b] = run;
    }
}

__global__ void __launch_bounds__(kThreads)
dispatch_offsets_kernel(DispatchArgs a)
{
    extern __shared__ int32_t sh[];
    const int NB = a.NB, R = a.R, NC = a.nc;
    int32_t* tot = sh;                 // [NB] totals by bin
    int32_t* pref = tot + NB;          // [NB] exclusive prefix by bin, in destination order
    int32_t* sc = pref + NB;           // [R + 1] entries per destination rank (+ undeliverable)
    __shared__ int32_t wsum[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t lr = blockIdx.x;
    int32_t* dc = a.dc + lr * NC * (int64_t)NB;
    taot_await();
    taot_release();
    for (int r = tid; r <= R; r += kThreads) sc[r] = 0;
    for (int b = tid; b < NB; b += kThreads) {
        int32_t t = 0;
        for (int c = 0; c < NC; ++c) t += dc[(int64_t)c * NB + b];
        tot[b] = t;
    }
    __syncthreads();
    // exclusive scan of the totals taken in destination order: thread t owns sorted positions [t*per, (t+1)*per)
    const int per = (NB + kThreads - 1) / kThreads;
    const int p0 = tid * per, p1 = min(NB, p0 + per);
    int32_t local = 0;
    for (int p = p0; p < p1; ++p) local += tot[a.torder[p]];
    int32_t inc = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int32_t run = inc - local;
    for (int w = 0; w < warp; ++w) run += wsum[w];
    for (int p = p0; p < p1; ++p) {
        const int b = a.torder[p];
        pref[b] = run;
        run += tot[b];
    }
    __syncthreads();
    for (int b = tid; b < NB; b += kThreads) {
        int32_t base = pref[b];
        for (int c = 0; c < NC; ++c) {
            const int32_t t = dc[(int64_t)c * NB + b];
            dc[(int64_t)c * NB + b] = base;
            base += t;
        }
        if (tot[b] != 0) atomicAdd(&sc[a.tdest[b]], tot[b]);
        if (a.target_counts && b < NB - 1) a.target_counts[lr * (int64_t)(NB - 1) + b] = tot[b];
    }
    __syncthreads();
    for (int r = tid; r < R; r += kThreads) a.send_counts[lr * R + r] = sc[r];
    if (tid == 0 && sc[R] != 0) atomicOr(a.info + (int32_t)(lr / R), TAOT_INFO_BAD_INDEX);
}

// ALT: the mask words of consecutive ranking steps sit in alternating rows (one warp barrier fewer per step); otherwise one
// row, for target counts whose three rows would not fit in shared memory.
// PRE: where a warp's entries start comes from the counting pass (a.wp); otherwise the spans are counted again here.
template <bool ALT, bool PRE>
__global__ void __launch_bounds__(kThreads)
dispatch_scatter_kernel(DispatchArgs a)
{
    extern __shared__ int32_t wh[];            // [kWarps][NB]: running positions;
                                               // then (ALT: 2 x) [kWarps][NB] lane masks of the steps being ranked
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NB = a.NB;
    const int64_t id = blockIdx.x;
    int64_t goff; int32_t len;
    chunk_span(a, id, goff, len);
    const int s0 = warp * kWarpSpan, n = min(len - s0, kWarpSpan);
    const int32_t* src = a.idx + goff + s0;
    int32_t* dst = a.perm + goff + s0;
    for (int q = (PRE ? kWarps * NB : 0) + tid; q < (ALT ? 3 : 2) * kWarps * NB; q += kThreads) wh[q] = 0;
    if constexpr (!PRE) __syncthreads();
    taot_await();
    if constexpr (!PRE) {
        count_span(src, n, wh + warp * NB, NB, a.vec_ok);
        __syncthreads();
        const int32_t* base = a.dc + id * (int64_t)NB;
        for (int b = tid; b < NB; b += kThreads) {
            int32_t run = base[b];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const int32_t t = wh[w * NB + b];
                wh[w * NB + b] = run;
                run += t;
            }
        }
    } else {
        const int32_t* base = a.dc + id * (int64_t)NB;
        const uint16_t* wp = a.wp + id * kWarps * (int64_t)NB;
        for (int b = tid; b < NB; b += kThreads) {
            const int32_t first = base[b];
            uint32_t before[kWarps];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) before[w] = wp[w * NB + b];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) wh[w * NB + b] = first + (int32_t)before[w];
        }
    }
    __syncthreads();
    const unsigned bit = 1u << lane, lt = bit - 1u;
    int32_t* const mine = wh + warp * NB;
    const uint32_t a_pos = (uint32_t)__cvta_generic_to_shared(mine);
    const uint32_t a_mask = a_pos + 4u * (uint32_t)(kWarps * NB), a_alt = ALT ? 4u * (uint32_t)(kWarps * NB) : 0u;
    constexpr int U = 8;
    int i0 = 0;
    // Whole steps of 32 entries, every lane the same instructions: OR my bit into the target's word (a set: the order does not
    // matter), read the word and the target's running position, then all of a target's lanes store the same new position and
    // clear the word.  The word is next written two steps later (ALT), the position next read behind the next barrier.
    for (; i0 + 32 * U <= n; i0 += 32 * U) {
        uint32_t b4[U];
#pragma unroll
        for (int u = 0; u < U; ++u) b4[u] = 4u * (uint32_t)bin_of(__ldcs(src + i0 + u * 32 + lane), NB);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t am = a_mask + ((u & 1) ? a_alt : 0u) + b4[u], ap = a_pos + b4[u];
            asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(am), "r"(bit) : "memory");
            __syncwarp();
            uint32_t peers, first;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(peers) : "r"(am) : "memory");
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(first) : "r"(ap) : "memory");
            __syncwarp();
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(am), "r"(0u) : "memory");
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(ap), "r"(first + (uint32_t)__popc(peers)) : "memory");
            if (!ALT) __syncwarp();
            __stcs(dst + i0 + u * 32 + lane, (int32_t)(first + (uint32_t)__popc(peers & lt)));
        }
    }
    __syncwarp();
    for (; i0 < n; i0 += 32) {                 // what is left of a short span
        const int i = i0 + lane;
        const bool ok = i < n;
        const int b = ok ? bin_of(__ldcs(src + i), NB) : 0;
        unsigned* const word = reinterpret_cast<unsigned*>(mine + kWarps * NB) + b;
        if (ok) atomicOr(word, bit);
        __syncwarp();
        const unsigned peers = ok ? *word : bit;
        const int32_t first = mine[b];
        __syncwarp();
        if (ok) {
            *word = 0u;
            mine[b] = first + __popc(peers);
            dst[i] = first + __popc(peers & lt);
        }
        __syncwarp();
    }
}

}  // namespace

int taot_launch_dispatch(taot_handle_t h, const int32_t* d_new_idx, int32_t* d_send_counts, int32_t* d_target_counts,
                         int32_t* d_perm, int32_t* d_info, void* ws, cudaStream_t st)
{
    const taot_params& p = h->p;
    DispatchArgs a;
    a.idx = d_new_idx;
    a.dc = reinterpret_cast<int32_t*>(static_cast<char*>(ws) + h->off_dc);
    a.wp = h->wp_ok ? reinterpret_cast<uint16_t*>(static_cast<char*>(ws) + h->off_wp) : nullptr;
    a.torder = h->d_torder; a.tdest = h->d_tdest;
    a.send_counts = d_send_counts; a.target_counts = d_target_counts; a.perm = d_perm; a.info = d_info;
    a.layer_elems = p.T * p.k; a.seg = h->seg; a.nc = h->nc; a.R = p.R; a.NB = p.E + p.R * p.K + 1;
    const unsigned chunks = (unsigned)((int64_t)p.L * p.R * h->nc);
    a.vec_ok = ((reinterpret_cast<uintptr_t>(d_new_idx) & 15) == 0 && h->seg % 4 == 0) ? 1 : 0;
    const size_t sm1 = sizeof(int32_t) * (size_t)kWarps * a.NB;
    const size_t sm2 = sizeof(int32_t) * (2 * (size_t)a.NB + p.R + 1);
    const bool alt = sizeof(int32_t) * 3 * (size_t)kWarps * a.NB <= 64 * 1024;
    const size_t sm3 = sizeof(int32_t) * (alt ? 3 : 2) * (size_t)kWarps * a.NB;
    const auto scatter = [&](auto kernel) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm3);
        return e == cudaSuccess ? taot_launch_chained(kernel, chunks, kThreads, sm3, st, a) : e;
    };
    TAOT_CUDA_OK(cudaFuncSetAttribute(dispatch_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm1));
    TAOT_CUDA_OK(taot_launch_chained(dispatch_count_kernel, chunks, kThreads, sm1, st, a));
    TAOT_CUDA_OK(taot_launch_chained(dispatch_offsets_kernel, (unsigned)((int64_t)p.L * p.R), kThreads, sm2, st, a));
    if (a.wp) TAOT_CUDA_OK(alt ? scatter(dispatch_scatter_kernel<true, true>) : scatter(dispatch_scatter_kernel<false, true>));
    else TAOT_CUDA_OK(alt ? scatter(dispatch_scatter_kernel<true, false>) : scatter(dispatch_scatter_kernel<false, false>));
    return 3;
}
