// Phase 1 for few problems of at most 64 ranks (Appendix A.2): what a plan of such a job calls.  A handful of problems, up to
// 1000 dependent iterations each, an SM to itself for every problem: the time is the length of one iteration's chain.
//
// The sums are those of the 4 x 8 lane grid (sinkhorn_tile.cuh, which keeps the batches that fill the GPU) to the last bit: the
// placement that follows decides exact ties by the last bits of the hint.  A row sum is eight chains of multiply-adds over the
// columns j = 8 cg + lc, one per lc, added as a balanced tree; a column sum four chains over the rows i = 4 ra + lr, added the
// same way.  On the grid these trees are shuffles between lanes, 29 cycles a level and five levels an iteration, and every lane
// issues the instructions of NRA rows and NCG columns.  Here a lane holds a row (beyond 32 ranks two lanes a half each) and, in a
// second set of registers, a column of K~ (two beyond 32 ranks): the trees are additions inside a lane, 4 cycles a level, and
// what changes hands is u~ and v~, written to shared memory (28 cycles there and back) and read four values per load (8 cycles
// each more).  ns per iteration, grid -> here, with a tolerance: 8 ranks 137 -> 92, 16 162 -> 106, 32 175 -> 109, 64 253 -> 145;
// fixed count: 119 -> 86, 125 -> 107, 140 -> 107, 188 -> 143.  What is left of the chain at 16 ranks: two exchanges 56, six loads
// 48, two reciprocals with their products 46, chains and trees 32, the look at the end of a group 10, of 204 cycles.
// More than 16 supply ranks (only beyond 32 ranks) take two warps and named barriers: there a lone warp would hold two rows a lane,
// 193 ns an iteration against 165 (with up to 16 the two are as fast).  A branch in the loop that the compiler cannot prove
// uniform costs 25 to 50 cycles with the warp barrier behind it.
//
// Set-up is spread over the CTA's warps: the cost matrix is in shared memory before the kernels in front have ended, and an
// exponential of the first iteration and of K~ is one thread's work each (64 ranks: 27 -> 16 us for all but the iterations).
#pragma once
#include "sinkhorn_common.cuh"

using namespace taot_sk;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSplitThreads = 128;         // of the widest build
constexpr int kSplitGroup = 8;             // iterations between two looks at drift, tolerance and cap (even)
constexpr int kSplitRows = 32;             // most supply ranks; a problem with more is handed back

__device__ __forceinline__ float rcp_fast(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int RMAX>
struct SplitSmem {
    static constexpr int KS = RMAX + 4;    // row stride of K
    double alpha[kSplitRows], beta[RMAX], mx[kSplitThreads], logd[RMAX];
    alignas(16) float C[RMAX * RMAX];
    alignas(16) float K[kSplitRows * KS];
    alignas(16) float v[2][RMAX];          // v~ by parity of the iterate
    alignas(16) float u[kSplitRows], e[kSplitGroup][kSplitRows];   // u~ and the rows' errors
    float st[kSplitRows], dd[RMAX], fg[RMAX];
    int32_t hot[kSplitRows], cold[RMAX];
    uint32_t bits[2];                      // what the eight iterations met, by warp
    int32_t fill;                          // what the other warps are to do: rebuild the tile, or go on behind the loop
    float err;                             // how the loop ended: row error of the iterate,
    int32_t status, t;                     // 1 solved, 0 handed back, and the iterate
};

// K~ by `nt` threads, a multiple of RMAX: the first `rows` rows (all of them at first: zero off the problem's block)
template <int RMAX>
__device__ __forceinline__ void split_fill(const SinkArgs& a, SplitSmem<RMAX>& sm, int Hn, int Cn, int rows, int tid, int nt)
{
    const int j = tid & (RMAX - 1);
    const bool col = j < Cn;
    const double be = col ? sm.beta[j] : 0.0;
    const float* C = sm.C + (col ? sm.cold[j] : 0);
#pragma unroll 4
    for (int i = tid / RMAX; i < rows; i += nt / RMAX) {
        float v = 0.0f;
        if (i < Hn && col) {
            const double c = (double)C[sm.hot[i] * a.R] * a.inv_eps;
            v = exp_split(sm.alpha[i] + be - c);
        }
        sm.K[i * SplitSmem<RMAX>::KS + j] = v;
    }
}

template <int NT>
__device__ __forceinline__ void split_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

// sum of the rows' errors in the grid's order
template <int NRA>
__device__ __forceinline__ float split_error(const float* e)
{
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll
    for (int ra = 0; ra < NRA; ++ra) {
        const float4 x = reinterpret_cast<const float4*>(e)[ra];
        s0 += x.x; s1 += x.y; s2 += x.z; s3 += x.w;
    }
    return (s0 + s1) + (s2 + s3);
}

// The iterations, by NW warps.  LR lanes hold a row, a lane CPL columns; NRA: rows / 4, NCG: columns / 8.
//
// Eight iterations at a time run without a branch on drift, tolerance or cap (a vote and a branch cost about 25 cycles); one look
// at the end tells whether there was anything, and if there was the eight are taken back and done again one by one.  A row error
// above the tolerance settles that the sum is; only if no row has one are the sums formed.
template <int RMAX, int NT, int NW, int LR, int NRA, int NCG, bool TOL>
__device__ __forceinline__ void split_loop(const SinkArgs& a, SplitSmem<RMAX>& sm, const int Hn, const int Cn, const float tol_abs_f)
{
    constexpr int NL = 32 * NW, CPL = RMAX / NL;
    constexpr int Q = 2 / LR;                          // float4 of v~ per cg that a row's lane reads
    constexpr int KS = SplitSmem<RMAX>::KS;
    const int lane = threadIdx.x;                      // (beyond 31 in the second warp)
    const int row = lane / LR, half = lane & (LR - 1);
    const auto sync = [&]() {
        if (NW == 1) __syncwarp();
        else asm volatile("bar.sync 2, %0;" ::"n"(NL) : "memory");
    };
    const auto any = [&](bool p) -> bool {
        if (NW == 1) {
            __syncwarp();                              // (a vote orders no memory; the barrier below does)
            return __any_sync(kFull, p);
        }
        int r;
        asm volatile("{ .reg .pred p, q; setp.ne.s32 p, %1, 0; barrier.cta.red.or.pred q, 3, %2, p; selp.s32 %0, 1, 0, q; }"
                     : "=r"(r) : "r"((int)p), "n"(NL) : "memory");
        return r != 0;
    };
    const bool row_ok = row < Hn;
    bool col_ok[CPL];
    // Off the problem's block u~ and v~ are 0: no select (the compiler makes it a branch around the reciprocal, and the warp barrier
    // behind a branch another 25 cycles).  The sums there must not be 0, so the lane's own copy of K~ begins with a 1.
    const float st = row_ok ? sm.st[row] : 0.0f;
    float dd[CPL];
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
        col_ok[q] = lane + NL * q < Cn;
        dd[q] = col_ok[q] ? sm.dd[lane + NL * q] : 0.0f;
    }
    const uint32_t lo_bits = __float_as_uint(kDriftLo), span_bits = __float_as_uint(kDriftHi) - lo_bits;
    const auto drifted = [&](float x) { return (__float_as_uint(x) - lo_bits) > span_bits; };
    const auto in_range = [](float x) { return x > kSumLo && x < kSumHi; };
    float4 Kr[NCG][Q], Kc[CPL][NRA];
    const auto load_tile = [&]() {
#pragma unroll
        for (int cg = 0; cg < NCG; ++cg)
#pragma unroll
            for (int q = 0; q < Q; ++q) Kr[cg][q] = *reinterpret_cast<const float4*>(&sm.K[row * KS + cg * 8 + (half + q) * 4]);
        if (!row_ok) Kr[0][0].x = 1.0f;
#pragma unroll
        for (int q = 0; q < CPL; ++q) {
#pragma unroll
            for (int ra = 0; ra < NRA; ++ra) {
                const float* k = &sm.K[ra * 4 * KS + lane + NL * q];
                Kc[q][ra] = make_float4(k[0], k[KS], k[2 * KS], k[3 * KS]);
            }
            if (!col_ok[q]) Kc[q][0].x = 1.0f;
        }
    };
    // (products and sums that the grid rounds apart are rounded apart)
    const auto chain = [](float4& p, const float4 k, const float4 x, bool first) {
        if (first) {
            p = make_float4(__fmul_rn(k.x, x.x), __fmul_rn(k.y, x.y), __fmul_rn(k.z, x.z), __fmul_rn(k.w, x.w));
        } else {
            p.x = fmaf(k.x, x.x, p.x);
            p.y = fmaf(k.y, x.y, p.y);
            p.z = fmaf(k.z, x.z, p.z);
            p.w = fmaf(k.w, x.w, p.w);
        }
    };
    const auto tree = [](const float4 p) { return __fadd_rn(__fadd_rn(p.x, p.y), __fadd_rn(p.z, p.w)); };
    float uo = row_ok ? 1.0f : 0.0f, un = 0.0f, r = 1.0f, vcol[CPL], cp[CPL];       // uo, vcol: iterate t in this lane's row and columns
    const auto new_rows = [&](const float* v) {
        const float4* vb = reinterpret_cast<const float4*>(v) + half;
        float4 p[Q];
#pragma unroll
        for (int cg = 0; cg < NCG; ++cg)
#pragma unroll
            for (int q = 0; q < Q; ++q) chain(p[q], Kr[cg][q], vb[cg * 2 + q], cg == 0);
        r = tree(p[0]);
        if constexpr (LR == 1) r = __fadd_rn(r, tree(p[Q - 1]));
        else r = __fadd_rn(r, __shfl_xor_sync(kFull, r, 1));
        un = __fmul_rn(st, rcp_fast(r));
    };
    const auto new_columns = [&](float* v) {
        float4 c[CPL];
#pragma unroll
        for (int ra = 0; ra < NRA; ++ra) {
            const float4 x = reinterpret_cast<const float4*>(sm.u)[ra];
#pragma unroll
            for (int q = 0; q < CPL; ++q) chain(c[q], Kc[q][ra], x, ra == 0);
        }
#pragma unroll
        for (int q = 0; q < CPL; ++q) {
            cp[q] = tree(c[q]);
            vcol[q] = __fmul_rn(dd[q], rcp_fast(cp[q]));
            v[lane + NL * q] = vcol[q];
        }
    };
    // the new u~ and, with a tolerance, the row's error of iterate t (a row's lanes hold the same); true: it is above the tolerance
    const auto put_rows = [&](float* e) {
        sm.u[row] = un;
        if (!TOL) return false;
        const float x = fabsf(fmaf(uo, r, -st));
        e[row] = x;
        return x > tol_abs_f;
    };
    const auto any_drift = [&]() {
        bool d = row_ok & drifted(uo);
#pragma unroll
        for (int q = 0; q < CPL; ++q) d |= col_ok[q] & drifted(vcol[q]);
        return d;
    };
    load_tile();
#pragma unroll
    for (int q = 0; q < CPL; ++q) vcol[q] = 1.0f;
    int t = 1;
    for (;;) {
        const int t_end = t + kSplitGroup;
        if (t_end <= a.max_iters) {                    // (the last iterate is one of those below)
            const float u0 = uo;
            float v0[CPL];
#pragma unroll
            for (int q = 0; q < CPL; ++q) v0[q] = vcol[q];
            float* va = sm.v[t & 1];
            float* vb = sm.v[(t + 1) & 1];
            bool odd = false, above[kSplitGroup];
#pragma unroll
            for (int g = 0; g < kSplitGroup; ++g) {
                new_rows(g & 1 ? vb : va);
                above[g] = put_rows(sm.e[g]);
                odd |= any_drift();
                uo = un;
                sync();
                new_columns(g & 1 ? va : vb);
                if (NW == 1 || g < kSplitGroup - 1) sync();
            }
            bool met, near = false;
            if (NW == 1) {
                met = __any_sync(kFull, odd);
                if (TOL) {
#pragma unroll
                    for (int g = 0; g < kSplitGroup; ++g) near |= !__any_sync(kFull, above[g]);
                }
            } else {
                uint32_t bits = odd ? 1u << kSplitGroup : 0u;
                if (TOL) {
#pragma unroll
                    for (int g = 0; g < kSplitGroup; ++g) bits |= above[g] ? 1u << g : 0u;
                }
                bits = __reduce_or_sync(kFull, bits);
                if ((lane & 31) == 0) sm.bits[lane >> 5] = bits;
                sync();
                bits = sm.bits[0] | sm.bits[1];
                met = (bits >> kSplitGroup) != 0u;
                near = TOL && (~bits & ((1u << kSplitGroup) - 1u)) != 0u;
            }
            if (TOL) {
                if (near) {
#pragma unroll
                    for (int g = 0; g < kSplitGroup; ++g) met |= split_error<NRA>(sm.e[g]) <= tol_abs_f;
                    sync();                            // every warp has the same sums before the next group writes over the errors
                }
            }
            if (!met) {
                t = t_end;
                continue;
            }
            sync();
            uo = u0;
#pragma unroll
            for (int q = 0; q < CPL; ++q) va[lane + NL * q] = vcol[q] = v0[q];
            sync();
        }
        // ---- one by one, until something has been seen to
        float usave = 1.0f, rsave = 1.0f;
        bool odd_p = false, due = false;               // of the iterate before this one
        for (;; ++t) {
            new_rows(sm.v[t & 1]);                     // half-step 1: r = K~ v~, u' = s~ / r; r are the row sums of iterate t
            // what iteration t - 1 left to decide
            const bool stop = TOL && due && split_error<NRA>(sm.e[0]) <= tol_abs_f, last = t > a.max_iters;
            if (stop || last) {                        // iterate t - 1 is the result
                const bool bad = any(row_ok && !in_range(rsave));
                if (!TOL) sm.e[0][row] = row_ok ? fabsf(fmaf(usave, rsave, -st)) : 0.0f;
                if (row_ok && half == 0) sm.alpha[row] += log((double)usave);
#pragma unroll
                for (int q = 0; q < CPL; ++q)
                    if (col_ok[q]) sm.beta[lane + NL * q] += log((double)sm.v[(t - 1) & 1][lane + NL * q]);
                sync();
                if (lane == 0) {
                    sm.err = split_error<NRA>(sm.e[0]);
                    sm.status = bad ? 0 : 1;
                    sm.t = t - 1;
                }
                return;
            }
            if (odd_p) {
                // u~, v~ merely drifted: fold them into the potentials and rebuild the tile; or a sum left the range in which
                // fp32 products are trustworthy: hand the problem back
                bool bad = row_ok && !in_range(rsave);
#pragma unroll
                for (int q = 0; q < CPL; ++q) bad |= col_ok[q] && !in_range(cp[q]);
                if (any(bad)) {
                    if (lane == 0) sm.status = 0;
                    return;
                }
                if (row_ok && half == 0) sm.alpha[row] += log((double)uo);
                uo = row_ok ? 1.0f : 0.0f;
#pragma unroll
                for (int q = 0; q < CPL; ++q) {
                    if (col_ok[q]) sm.beta[lane + NL * q] += log((double)vcol[q]);
                    sm.v[t & 1][lane + NL * q] = vcol[q] = 1.0f;
                }
                if (lane == 0) sm.fill = 1;
                split_sync<NT>();
                split_fill<RMAX>(a, sm, Hn, Cn, Hn, lane, NT);
                split_sync<NT>();
                load_tile();
                break;
            }
            if (t == t_end) {
                if (TOL) sync();                       // (the errors that `stop` read, and the next group's)
                break;
            }
            due = t % a.check_every == 0;
            odd_p = any(any_drift());
            put_rows(sm.e[0]);                         // half-step 2: c = K~^T u', v' = d / c
            usave = uo; uo = un; rsave = r;
            sync();
            new_columns(sm.v[(t + 1) & 1]);
            sync();
        }
    }
}

// The smallest build that holds the problem.  What the finer steps are worth, ns an iteration with the step : with the next larger build
// (8 problems, 2048 iterations, with a tolerance as without):
//   32 ranks  12 rows  102 : 105 (7 columns), 110 : 113 (20)             24 columns  107 : 118 (7 or 8 rows), 113 : 124 (14)
//   64 ranks  12 rows  127 : 132 (30 columns), 133 : 138 (46)            56 columns  132 : 138 (7 rows), 144 : 148 (14)
//             20 rows  133 : 147 (30), 141 : 154 (46)   24 rows  137 : 147 (30), 143 : 154 (42)
template <int RMAX, int NT, bool TOL>
__device__ __forceinline__ void split_dispatch(const SinkArgs& a, SplitSmem<RMAX>& sm, int Hn, int Cn, float tol_abs_f)
{
#define TAOT_SPLIT(NW, LR, NRA, NCG) return split_loop<RMAX, NT, NW, LR, NRA, NCG, TOL>(a, sm, Hn, Cn, tol_abs_f)
    if constexpr (RMAX == 32) {
#define TAOT_SPLIT_ROWS(NCG)                           \
        if (Hn <= 4) TAOT_SPLIT(1, 1, 1, NCG);        \
        if (Hn <= 8) TAOT_SPLIT(1, 1, 2, NCG);        \
        if (Hn <= 12) TAOT_SPLIT(1, 1, 3, NCG);       \
        if (Hn <= 16) TAOT_SPLIT(1, 1, 4, NCG);       \
        TAOT_SPLIT(1, 1, 8, NCG);
        if (Cn <= 8) { TAOT_SPLIT_ROWS(1) }
        if (Cn <= 16) { TAOT_SPLIT_ROWS(2) }
        if (Cn <= 24) { TAOT_SPLIT_ROWS(3) }
        TAOT_SPLIT_ROWS(4)
#undef TAOT_SPLIT_ROWS
    } else {
#define TAOT_SPLIT_ROWS(NCG)                           \
        if (Hn <= 8) TAOT_SPLIT(1, 2, 2, NCG);         \
        if (Hn <= 12) TAOT_SPLIT(1, 2, 3, NCG);        \
        if (Hn <= 16) TAOT_SPLIT(1, 2, 4, NCG);        \
        if (Hn <= 20) TAOT_SPLIT(2, 2, 5, NCG);        \
        if (Hn <= 24) TAOT_SPLIT(2, 2, 6, NCG);        \
        TAOT_SPLIT(2, 2, 8, NCG);
        if (Cn <= 32) { TAOT_SPLIT_ROWS(4) }
        if (Cn <= 48) { TAOT_SPLIT_ROWS(6) }
        if (Cn <= 56) { TAOT_SPLIT_ROWS(7) }
        TAOT_SPLIT_ROWS(8)
#undef TAOT_SPLIT_ROWS
    }
#undef TAOT_SPLIT
}

// one problem per CTA of NT threads (the name is that of the register-tile kernels it stands beside)
template <int RMAX, int NT, bool TOL>
__global__ void __launch_bounds__(NT, RMAX == 32 ? 4 : 2)
sinkhorn_tile_kernel(SinkArgs a)
{
    __shared__ SplitSmem<RMAX> sm;
    constexpr int NE = RMAX / 32;                      // ranks per lane
    const int R = a.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t b = blockIdx.x;
    // the topology, which no kernel in front writes
    if ((R & 1) == 0) {
        for (int q = tid; q < R * R / 4; q += NT) reinterpret_cast<float4*>(sm.C)[q] = reinterpret_cast<const float4*>(a.C)[q];
    } else {
        for (int q = tid; q < R * R; q += NT) sm.C[q] = a.C[q];
    }
    double lse0[NE];
#pragma unroll
    for (int k = 0; k < NE; ++k) lse0[k] = lane + 32 * k < R ? a.rowlse0[lane + 32 * k] : 0.0;
    taot_await();
    if (a.early) taot_release();
    float sv[NE], dv[NE];
    double ps = 0.0, pd = 0.0;
#pragma unroll
    for (int k = 0; k < NE; ++k) {
        const int i = lane + 32 * k;
        sv[k] = i < R ? a.s[b * R + i] : 0.0f;
        dv[k] = i < R ? a.d[b * R + i] : 0.0f;
    }
    float* out = a.plan + b * (int64_t)R * R;
    if ((reinterpret_cast<uintptr_t>(out) & 15) == 0 && (R & 1) == 0) {
        for (int q = tid; q < R * R / 4; q += NT) reinterpret_cast<float4*>(out)[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    } else {
        for (int q = tid; q < R * R; q += NT) out[q] = 0.0f;
    }
    // ---- supply scaling gamma = min(1, sum d / max(sum s, eps0)), compaction of supply / demand ranks: by every warp alike
#pragma unroll
    for (int k = 0; k < NE; ++k) {
        ps += sv[k] > 0.0f ? (double)sv[k] : 0.0;
        pd += dv[k] > 0.0f ? (double)dv[k] : 0.0;
    }
    for (int o = 16; o > 0; o >>= 1) {
        ps += __shfl_xor_sync(kFull, ps, o);
        pd += __shfl_xor_sync(kFull, pd, o);
    }
    const double gamma = fmin(1.0, pd / fmax(ps, (double)a.eps0));
    const unsigned lt = (1u << lane) - 1u;
    int Hn = 0, Cn = 0, hpos[NE], cpos[NE];
#pragma unroll
    for (int k = 0; k < NE; ++k) {
        sv[k] = sv[k] > 0.0f ? (float)(gamma * (double)sv[k]) : 0.0f;
        dv[k] = dv[k] > 0.0f ? dv[k] : 0.0f;
        const unsigned hm = __ballot_sync(kFull, sv[k] > 0.0f), cm = __ballot_sync(kFull, dv[k] > 0.0f);
        hpos[k] = Hn + __popc(hm & lt);
        cpos[k] = Cn + __popc(cm & lt);
        Hn += __popc(hm);
        Cn += __popc(cm);
    }
    int info = ps > pd ? TAOT_INFO_SUPPLY_SCALED : 0;
    if (Hn > kSplitRows || Hn == 0 || Cn == 0) {
        if (tid == 0) {
            if (Hn > kSplitRows) {
                a.iters[b] = kHandBack;
            } else {
                a.iters[b] = 0;
                a.row_err[b] = 0.0f;
                if (info) atomicOr(a.info + b, info);
            }
        }
        return;
    }
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NE; ++k)
            if (sv[k] > 0.0f) {
                sm.hot[hpos[k]] = lane + 32 * k;
                sm.st[hpos[k]] = sv[k];
                sm.alpha[hpos[k]] = log((double)sv[k]) - lse0[k];
            }
    } else if (warp == 1) {
#pragma unroll
        for (int k = 0; k < NE; ++k)
            if (dv[k] > 0.0f) {
                sm.cold[cpos[k]] = lane + 32 * k;
                sm.dd[cpos[k]] = dv[k];
                sm.logd[cpos[k]] = log((double)dv[k]);
            }
    }
    if (tid < RMAX) sm.v[0][tid] = sm.v[1][tid] = 1.0f;
    double sum_st = 0.0;
#pragma unroll
    for (int k = 0; k < NE; ++k) sum_st += (double)sv[k];
    for (int o = 16; o > 0; o >>= 1) sum_st += __shfl_xor_sync(kFull, sum_st, o);
    __syncthreads();
    // ---- iteration 1 in the log domain (v = 1 on every rank): phi = log s~ - LSE_j(-C_ij/eps) over all j,
    //      psi_j = log d_j - LSE_i(phi_i - C_ij/eps)
    {
        constexpr int P = NT / RMAX;
        const int j = tid & (RMAX - 1), p = tid / RMAX;
        const float* C = sm.C + (j < Cn ? sm.cold[j] : 0);
        double mx = -INFINITY;
        if (j < Cn) {
#pragma unroll 2
            for (int i = p; i < Hn; i += P) {
                const double x = sm.alpha[i] - (double)C[sm.hot[i] * R] * a.inv_eps;
                mx = x > mx ? x : mx;
            }
        }
        sm.mx[tid] = mx;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const double x = sm.mx[k * RMAX + j];
            mx = x > mx ? x : mx;
        }
        if (j < Cn) {
#pragma unroll 2
            for (int i = p; i < Hn; i += P) sm.K[i * SplitSmem<RMAX>::KS + j] = exp_split(sm.alpha[i] - (double)C[sm.hot[i] * R] * a.inv_eps - mx);
        }
        __syncthreads();
        if (p == 0 && j < Cn) {
            double acc = 0.0;
#pragma unroll 4
            for (int i = 0; i < Hn; ++i) acc += (double)sm.K[i * SplitSmem<RMAX>::KS + j];
            sm.beta[j] = sm.logd[j] - (mx + log(acc));
        }
        __syncthreads();
    }
    split_fill<RMAX>(a, sm, Hn, Cn, kSplitRows, tid, NT);
    __syncthreads();
    // one warp iterates; the others wait until a fold wants the tile rebuilt (64 ranks, 1000 iterations with a dozen folds: 2 us each
    // by the one warp)
    if (warp < (RMAX > 32 && Hn > 16 ? 2 : 1)) {
        split_dispatch<RMAX, NT, TOL>(a, sm, Hn, Cn, (float)((double)a.tol * sum_st));
        if (tid == 0) sm.fill = 0;
        split_sync<NT>();
    } else {
        for (split_sync<NT>(); sm.fill; split_sync<NT>()) {
            split_fill<RMAX>(a, sm, Hn, Cn, Hn, tid, NT);
            split_sync<NT>();
        }
    }
    __syncthreads();
    taot_release();
    if (sm.status == 0) {
        if (tid == 0) a.iters[b] = kHandBack;
        return;
    }
    // ---- T = diag(u) M diag(v) from the total potentials, then the column cap
    split_fill<RMAX>(a, sm, Hn, Cn, Hn, tid, NT);
    __syncthreads();
    if (tid < Cn) {
        float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, c3 = 0.0f;
        const float* k = &sm.K[tid];
        for (int i = 0; i < Hn; i += 4, k += 4 * SplitSmem<RMAX>::KS) {
            c0 += k[0];
            c1 += k[SplitSmem<RMAX>::KS];
            c2 += k[2 * SplitSmem<RMAX>::KS];
            c3 += k[3 * SplitSmem<RMAX>::KS];
        }
        const float acc = (c0 + c1) + (c2 + c3);
        sm.fg[tid] = (float)fmin(1.0, (double)sm.dd[tid] / ((double)acc + (double)a.eps0));
    }
    __syncthreads();
    int nonfinite = 0;
    const int j = tid & (RMAX - 1);
    if (j < Cn) {
        const float fg = sm.fg[j];
        float* ocol = out + sm.cold[j];
        for (int i = tid / RMAX; i < Hn; i += NT / RMAX) {
            const float val = sm.K[i * SplitSmem<RMAX>::KS + j] * fg;
            if (!isfinite(val)) nonfinite = 1;
            ocol[(int64_t)sm.hot[i] * R] = val;
        }
    }
    nonfinite = __syncthreads_or(nonfinite);
    if (tid == 0) {
        if (nonfinite) info |= TAOT_INFO_NONFINITE;
        const float err = sm.err;
        if (TOL && !(err <= (float)((double)a.tol * sum_st))) info |= TAOT_INFO_SINKHORN_CAP;
        a.iters[b] = sm.t;
        a.row_err[b] = (float)((double)err / sum_st);
        if (info) atomicOr(a.info + b, info);
    }
}

}  // namespace
