// Sinkhorn-Knopp (Appendix A.2) for a cost without structure at 257 to 512 ranks: the absorbed kernel matrix of a problem,
// compacted to the ranks with supply x the ranks with demand, in the registers of one CTA.
//
// Loads that follow a power law leave few ranks above the mean: 54 of 512 against 458 below, a tenth of the full matrix.  Thread
// (warp w, row lane rl = lane % 8, column lane cl = lane / 8) holds rows rl * RT + a (a < RT) of columns 32 w + 8 cl + g (g < 8)
// as packed pairs, so that
//   column sums end inside the warp: RT multiply-adds per column, then 7 shuffles (a transposing butterfly over the 8 row
//   lanes) leave one column of the warp's 32 in each lane, which divides, and the warp exchanges its 32 new factors by shared
//   memory without a block barrier;
//   row sums cross the warps: 8 multiply-adds per row, a butterfly over the 4 column lanes, one 8-byte store per two rows,
//   a barrier, two threads per row add the warps' parts and divide, a barrier.
// Bound: fp32 multiply-adds, 2 |H||C| an iteration over four schedulers, plus the latency of the two barriers.
//
// The same absorbed form, drift fold, stopping rule and hand-back as the register-tile kernels (sinkhorn_tile.cuh); problems
// with more than 64 supply ranks go to the kernels behind it (iters = -1).
//
// Measured (B200, 512 ranks, 256 problems, 500 iterations): 20.7 -> 1.03 ms (dense products over all R x R on the tensor cores
// before); 3.4 us an iteration over the batch, two waves of problems, about 1600 cycles an iteration.
#include "sinkhorn_common.cuh"

using namespace taot_sk;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxR = 512, kMaxRows = 64, kMaxWarps = kMaxR / 32;
typedef unsigned long long u64;

__device__ __forceinline__ float rcp_fast(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ u64 pack2(float x, float y)
{
    u64 p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(x), "f"(y));
    return p;
}
__device__ __forceinline__ void unpack2(u64 p, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(p)); }
__device__ __forceinline__ void fma2(u64& acc, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ u64 mul2(u64 a, u64 b)
{
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ bool in_window(float x)
{
    return (__float_as_uint(x) - __float_as_uint(kDriftLo)) <= (__float_as_uint(kDriftHi) - __float_as_uint(kDriftLo));
}
__device__ __forceinline__ bool in_range(float x) { return x > kSumLo && x < kSumHi; }

struct WideSmem {
    double alpha[kMaxRows], beta[kMaxR], red[2][kMaxWarps + 1];
    float st[kMaxRows], dd[kMaxR];
    __align__(16) float u[2][kMaxRows / 8 * 20 + 16 * 8];   // u~ by parity of the iteration, each twice (a packed operand), by row lane
                                                   // with a stride of 2 RT + 4 (no bank conflicts between the row lanes)
    __align__(16) float v[kMaxR];                  // v~
    __align__(16) float part[kMaxWarps][80];       // row sums by warp (stride: the two readers of a row meet no bank conflict)
    float err[kMaxRows];
    int32_t hot[kMaxR], cold[kMaxR], hpos[kMaxR], cpos[kMaxR], wcnt[32];
    int event[2];                                  // iteration after which an event is due: [0] drift, [1] stop
    int bad;
};

// The iteration for up to 8 * RT supply ranks.  `tile`: [8 RT][32 NW] staging in shared memory.  False: hand the problem back.
template <int RT, bool TOL>
__device__ __forceinline__ bool wide_solve(const SinkArgs& a, WideSmem& sm, float* tile, const int NW, const int Hn, const int Cn,
                                           const double sum_st, int info, float* out, const int64_t b)
{
    constexpr int NR = 8 * RT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, R = a.R, NC = NW * 32;
    const bool mainw = warp < NW;                  // with a tolerance one more warp sums the row error beside the iteration
    const int rl = lane & 7, cl = lane >> 3;
    const float tol_abs = (float)((double)a.tol * sum_st);
    const int col = warp * 32 + lane;              // the column whose sum this lane ends up with
    const bool col_ok = mainw && col < Cn;
    const float dd = col_ok ? sm.dd[col] : 1.0f;
    u64 K[RT][4];                                  // rows rl * RT + a, columns 32 warp + 8 cl + (2k, 2k + 1)
    u64 v2[4];                                     // v~ of those columns
    float vo = 1.0f, vprev = 1.0f;                 // v~ of column `col`: iterate t, iterate t - 1

    auto build = [&](const bool staged) {          // block-wide: the tile from the potentials (staged: it holds the costs)
        __syncthreads();
#pragma unroll 4
        for (int q = tid; q < NR * NC; q += NT) {
            const int i = q / NC, j = q - i * NC;
            const bool ok = i < Hn && j < Cn;
            const double c = (double)(staged ? tile[q] : a.C[(int64_t)sm.hot[ok ? i : 0] * R + sm.cold[ok ? j : 0]]) * a.inv_eps;
            const float e = exp_split(sm.alpha[ok ? i : 0] + sm.beta[ok ? j : 0] - c);
            tile[q] = ok ? e : 0.0f;
        }
        __syncthreads();
    };
    auto load_tile = [&]() {
        if (mainw) {
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const ulonglong2* p = reinterpret_cast<const ulonglong2*>(tile + (rl * RT + r) * NC + warp * 32 + cl * 8);
                const ulonglong2 x = p[0], y = p[1];
                K[r][0] = x.x; K[r][1] = x.y; K[r][2] = y.x; K[r][3] = y.y;
            }
        }
    };
    auto share_v = [&](float v) {                  // a warp's 32 new factors, to the lanes that multiply by them
        sm.v[col] = v;
        __syncwarp();
        const ulonglong2* p = reinterpret_cast<const ulonglong2*>(sm.v + warp * 32 + cl * 8);
        const ulonglong2 x = p[0], y = p[1];
        v2[0] = x.x; v2[1] = x.y; v2[2] = y.x; v2[3] = y.y;
        __syncwarp();
    };
    auto row_parts = [&]() {                       // this warp's part of the row sums
        float p[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            u64 acc = mul2(K[r][0], v2[0]);
#pragma unroll
            for (int k = 1; k < 4; ++k) fma2(acc, K[r][k], v2[k]);
            float x, y;
            unpack2(acc, x, y);
            p[r] = x + y;
        }
        // butterfly over the column lanes, halving the rows a lane keeps
        const bool up4 = (lane & 16) != 0, up3 = (lane & 8) != 0;
#pragma unroll
        for (int r = 0; r < RT / 2; ++r) {
            const float send = up4 ? p[r] : p[r + RT / 2], keep = up4 ? p[r + RT / 2] : p[r];
            p[r] = keep + __shfl_xor_sync(kFull, send, 16);
        }
        if constexpr (RT >= 4) {
#pragma unroll
            for (int r = 0; r < RT / 4; ++r) {
                const float send = up3 ? p[r] : p[r + RT / 4], keep = up3 ? p[r + RT / 4] : p[r];
                p[r] = keep + __shfl_xor_sync(kFull, send, 8);
            }
            const int a0 = (up4 ? RT / 2 : 0) + (up3 ? RT / 4 : 0);
            if constexpr (RT == 8) *reinterpret_cast<float2*>(&sm.part[warp][rl * RT + a0]) = make_float2(p[0], p[1]);
            else sm.part[warp][rl * RT + a0] = p[0];
        } else {
            p[0] += __shfl_xor_sync(kFull, p[0], 8);
            if (!up3) sm.part[warp][rl * RT + (up4 ? 1 : 0)] = p[0];
        }
    };
    // two threads per row add the warps' parts: the row sum in both (threads below 2 NR)
    auto row_total = [&]() {
        const int row = tid >> 1;
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < kMaxWarps / 2; ++k) {
            const int w = 2 * k + (tid & 1);
            if (w < NW) s += sm.part[w][row];
        }
        return s + __shfl_xor_sync(kFull, s, 1);
    };
    const int uq = (tid >> 1) / RT * (2 * RT + 4) + (tid >> 1) % RT * 2 + (tid & 1);      // this thread's place in u
    const bool totals = tid < 2 * NR;              // whole warps: NR is a multiple of 16
    const int row = tid >> 1;
    const bool row_ok = totals && row < Hn;
    const float st = row_ok ? sm.st[row] : 1.0f;

    // the rows of the plan without supply, a row per warp and iteration, while the iterations run
    const bool wide4 = R % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    int zero_row = mainw ? warp : R;
    auto write_zero_row = [&]() {
        if (sm.hpos[zero_row] < 0) {
            float* o = out + (int64_t)zero_row * R;
            if (wide4) {
                for (int j = lane * 4; j < R; j += 128) *reinterpret_cast<float4*>(o + j) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            } else {
                for (int j = lane; j < R; j += 32) o[j] = 0.0f;
            }
        }
        zero_row += NW;
    };

    // ---- the costs into the staging, and iteration 1 in the log domain (v = 1 on every rank): phi = log s~ -
    //      LSE_j(-C_ij/eps) over all j (the caller's), psi_j = log d_j - LSE_i(phi_i - C_ij/eps)
#pragma unroll 8
    for (int q = tid; q < NR * NC; q += NT) {
        const int i = q / NC, j = q - i * NC;
        const bool ok = i < Hn && j < Cn;
        tile[q] = a.C[(int64_t)sm.hot[ok ? i : 0] * R + sm.cold[ok ? j : 0]];
    }
    __syncthreads();
    for (int j = tid; j < Cn; j += NT) {
        double mx = -INFINITY;
#pragma unroll 4
        for (int i = 0; i < Hn; ++i) mx = fmax(mx, sm.alpha[i] - (double)tile[i * NC + j] * a.inv_eps);
        double acc = 0.0;
#pragma unroll 4
        for (int i = 0; i < Hn; ++i) acc += (double)exp_split(sm.alpha[i] - (double)tile[i * NC + j] * a.inv_eps - mx);
        sm.beta[j] = log((double)sm.dd[j]) - (mx + log(acc));
    }
    build(true);
    load_tile();
    if (totals) sm.u[1][uq] = 1.0f;               // iterate 1
    if (tid == 0) { sm.event[0] = -1; sm.event[1] = -1; sm.bad = 0; }
    if (mainw) share_v(1.0f);
    __syncthreads();

    int t = 1, until_check = a.check_every;
    float err_out = 0.0f;
    for (;;) {
        // ================= half-step 1: row sums of iterate t
        if (mainw) row_parts();
        __syncthreads();
        const int ev_drift = sm.event[0], ev_stop = TOL ? sm.event[1] : -1;
        if (ev_drift == t || ev_stop == t || t >= a.max_iters) {
            if (TOL && ev_stop == t) {             // iterate t - 1 met the tolerance: back to it
                --t;
                vo = vprev;
            } else if (ev_drift == t) {
                // u~ or v~ of iterate t left the window: fold it into the potentials, or hand the problem back if a sum left
                // the range in which fp32 products are trustworthy
                const float un = row_ok ? sm.u[t & 1][uq] : 1.0f;
                if (!in_range(un) || !in_range(vo)) sm.bad = 1;
                __syncthreads();
                if (sm.bad) return false;
                if (row_ok && !(tid & 1)) sm.alpha[row] += log((double)un);
                if (col_ok) sm.beta[col] += log((double)vo);
                __syncthreads();
                if (totals) sm.u[t & 1][uq] = 1.0f;
                if (tid == 0) sm.event[0] = -1;
                vo = 1.0f;
                if (mainw) share_v(1.0f);
                build(false);
                load_tile();
                continue;
            }
            // ---- the result is iterate t: its row sums and error
            if (mainw) share_v(vo);
            __syncthreads();
            if (mainw) row_parts();
            __syncthreads();
            double e = 0.0;
            if (totals) {
                const float r = row_total();
                if (row_ok) {
                    if (!in_range(r)) sm.bad = 1;
                    if (!(tid & 1)) e = (double)fabsf(fmaf(sm.u[t & 1][uq], r, -st));
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
            if (lane == 0) sm.red[0][warp] = e;
            __syncthreads();
            if (sm.bad) return false;
            e = 0.0;
            for (int w = 0; w < (NT >> 5); ++w) e += sm.red[0][w];
            err_out = (float)(e / sum_st);
            if (TOL && !((float)e <= tol_abs)) info |= TAOT_INFO_SINKHORN_CAP;
            break;
        }
        bool check_now = false;
        if (TOL) {
            check_now = --until_check == 0;
            if (check_now) until_check = a.check_every;
        }
        if (totals) {
            const float r = row_total();
            const float un = row_ok ? st * rcp_fast(r) : 1.0f;
            if (TOL && check_now && !(tid & 1)) sm.err[row] = row_ok ? fabsf(fmaf(sm.u[t & 1][uq], r, -st)) : 0.0f;
            sm.u[(t + 1) & 1][uq] = un;
            if (!in_window(un)) sm.event[0] = t + 1;
        }
        __syncthreads();
        // ================= half-step 2: column sums, inside the warp
        if (mainw) {
            float q[8];
            {
                u64 q2[4];
                const ulonglong2* up = reinterpret_cast<const ulonglong2*>(&sm.u[(t + 1) & 1][rl * (2 * RT + 4)]);
#pragma unroll
                for (int r = 0; r < RT; r += 2) {
                    const ulonglong2 uu = up[r / 2];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (r == 0) q2[k] = mul2(K[0][k], uu.x);
                        else fma2(q2[k], K[r][k], uu.x);
                        fma2(q2[k], K[r + 1][k], uu.y);
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) unpack2(q2[k], q[2 * k], q[2 * k + 1]);
            }
#pragma unroll
            for (int off = 4; off >= 1; off >>= 1) {
                const bool up = (rl & off) != 0;
#pragma unroll
                for (int k = 0; k < off; ++k) {
                    const float send = up ? q[k] : q[k + off], keep = up ? q[k + off] : q[k];
                    q[k] = keep + __shfl_xor_sync(kFull, send, off);
                }
            }
            vprev = vo;
            vo = col_ok ? dd * rcp_fast(q[0]) : 1.0f;
            if (!in_window(vo)) sm.event[0] = t + 1;
            share_v(vo);
            if (zero_row < R) write_zero_row();
        } else if (TOL && check_now) {             // the error warp: the 64 terms of iterate t
            float e = 0.0f;
            for (int i = lane; i < NR; i += 32) e += sm.err[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
            if (lane == 0 && e <= tol_abs) sm.event[1] = t + 1;
        }
        ++t;
    }

    // ---- T = diag(u) M diag(v) from the total potentials, then the column cap
    if (row_ok && !(tid & 1)) sm.alpha[row] += log((double)sm.u[t & 1][uq]);
    if (col_ok) sm.beta[col] += log((double)vo);
    while (zero_row < R) write_zero_row();
    build(false);
    for (int j = tid; j < NC; j += NT) {
        float acc = 0.0f;
        for (int i = 0; i < Hn; ++i) acc += tile[i * NC + j];
        sm.v[j] = j < Cn ? (float)fmin(1.0, (double)sm.dd[j] / ((double)acc + (double)a.eps0)) : 0.0f;
    }
    __syncthreads();
    int nonfinite = 0;
    for (int i = warp; i < R; i += NT >> 5) {
        const int h = sm.hpos[i];
        float* o = out + (int64_t)i * R;
        if (h < 0) continue;
#pragma unroll 4
        for (int j = lane; j < R; j += 32) {
            const int c = sm.cpos[j];
            const float w = c >= 0 ? tile[h * NC + c] * sm.v[c] : 0.0f;
            if (!isfinite(w)) nonfinite = 1;
            o[j] = w;
        }
    }
    if (__syncthreads_or(nonfinite)) info |= TAOT_INFO_NONFINITE;
    if (tid == 0) {
        a.iters[b] = t;
        a.row_err[b] = err_out;
        if (info) atomicOr(a.info + b, info);
    }
    return true;
}

template <bool TOL>
__global__ void __launch_bounds__(kMaxR + (TOL ? 32 : 0), 1)
sinkhorn_wide_kernel(SinkArgs a, int64_t nprob)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WideSmem& sm = *reinterpret_cast<WideSmem*>(smem_raw);
    float* tile = reinterpret_cast<float*>(smem_raw + ((sizeof(WideSmem) + 15) & ~(size_t)15));
    const int R = a.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, NW = (R + 31) >> 5;
    const int64_t b = blockIdx.x;
    taot_await();
    if (b >= nprob) return;

    // ---- supply scaling gamma = min(1, sum d / max(sum s, eps0)), compaction of the ranks with supply / demand
    double ps = 0.0, pd = 0.0;
    for (int i = tid; i < R; i += NT) {
        const float sv = a.s[b * R + i], dv = a.d[b * R + i];
        ps += sv > 0.0f ? (double)sv : 0.0;
        pd += dv > 0.0f ? (double)dv : 0.0;
    }
    for (int o = 16; o > 0; o >>= 1) {
        ps += __shfl_xor_sync(kFull, ps, o);
        pd += __shfl_xor_sync(kFull, pd, o);
    }
    if (lane == 0) { sm.red[0][warp] = ps; sm.red[1][warp] = pd; }
    __syncthreads();
    double sum_s = 0.0, sum_d = 0.0;
    for (int w = 0; w < (NT >> 5); ++w) { sum_s += sm.red[0][w]; sum_d += sm.red[1][w]; }
    const double gamma = fmin(1.0, sum_d / fmax(sum_s, (double)a.eps0));
    float* sv_all = tile;                          // (the staging is free here)
    float* dv_all = tile + R;
    for (int i = tid; i < R; i += NT) {
        const float sv = a.s[b * R + i], dv = a.d[b * R + i];
        sv_all[i] = sv > 0.0f ? (float)(gamma * (double)sv) : 0.0f;
        dv_all[i] = dv > 0.0f ? dv : 0.0f;
    }
    __syncthreads();
    const int Hn = compact_positive(sv_all, R, sm.hot, sm.hpos, sm.wcnt);
    const int Cn = compact_positive(dv_all, R, sm.cold, sm.cpos, sm.wcnt);
    if (Hn > kMaxRows && Cn > 0) {                 // another kernel takes it
        if (tid == 0) a.iters[b] = kHandBack;
        return;
    }
    for (int i = tid; i < Hn; i += NT) sm.st[i] = sv_all[sm.hot[i]];
    for (int j = tid; j < Cn; j += NT) sm.dd[j] = dv_all[sm.cold[j]];
    __syncthreads();
    int info = 0;
    if (sum_s > sum_d) info |= TAOT_INFO_SUPPLY_SCALED;
    float* out = a.plan + b * (int64_t)R * R;
    if (Hn == 0 || Cn == 0) {
        for (int q = tid; q < R * R; q += NT) out[q] = 0.0f;
        if (tid == 0) {
            a.iters[b] = 0;
            a.row_err[b] = 0.0f;
            if (info) atomicOr(a.info + b, info);
        }
        return;
    }
    double sum_st = 0.0;
    for (int i = 0; i < Hn; ++i) sum_st += (double)sm.st[i];          // same order in every thread

    for (int i = tid; i < Hn; i += NT) sm.alpha[i] = log((double)sm.st[i]) - a.rowlse0[sm.hot[i]];
    __syncthreads();
    bool done;
    if (Hn <= 16) done = wide_solve<2, TOL>(a, sm, tile, NW, Hn, Cn, sum_st, info, out, b);
    else if (Hn <= 32) done = wide_solve<4, TOL>(a, sm, tile, NW, Hn, Cn, sum_st, info, out, b);
    else done = wide_solve<8, TOL>(a, sm, tile, NW, Hn, Cn, sum_st, info, out, b);
    if (!done && tid == 0) a.iters[b] = kHandBack;
}

}  // namespace

// Launches the kernel for 257 to 512 ranks (returns 1), otherwise nothing (0).
//
// Against the dense tensor-core solve (sinkhorn_dense_tc.cu), which multiplies all R x R entries whatever the supports: that
// one keeps the solves of fewer than kWideMinIters iterations it applies to (a few milliseconds at most; its cost does not
// depend on how many ranks have supply, and its row error is measured on the plan itself), this one takes the long ones.
int taot_launch_sinkhorn_wide(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st)
{
    if (a.R <= 256 || a.R > kMaxR) return 0;
    const int NW = (a.R + 31) / 32;
    const size_t smem = ((sizeof(WideSmem) + 15) & ~(size_t)15) + sizeof(float) * kMaxRows * 32 * NW;
    if (a.tol > 0.0f) {
        TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_wide_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        TAOT_CUDA_OK(taot_launch_chained(sinkhorn_wide_kernel<true>, B, NW * 32 + 32, smem, st, a, (int64_t)B));
    } else {
        TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_wide_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        TAOT_CUDA_OK(taot_launch_chained(sinkhorn_wide_kernel<false>, B, NW * 32, smem, st, a, (int64_t)B));
    }
    TAOT_CUDA_OK(cudaGetLastError());
    return 1;
}
