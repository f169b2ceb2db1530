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
// Beyond 64 supply ranks (loads that are nearly even put half of the ranks above the mean) the warps that the columns leave idle
// take further blocks of 64 rows, and the rows that are left sit in shared memory (wide_solve_tall): every problem whose supports
// are disjoint fits one SM.  Bound there: the latency of four barriers and of one pass over shared memory per half-step, each
// warp a chain of its own (7000 cycles an iteration at 256 x 256, 42 % of the issue slots, hardly a bank conflict).
//
// Against 64-bit arithmetic (2-norm of the plan, 200 to 500 iterations, 70 to 288 supply ranks): 0.7 to 1.0e-7, the clusters 0.8
// to 1.4e-7; with the column sums of the cap in fp32 it was up to 2.2e-7.
//
// The same absorbed form, drift fold, stopping rule and hand-back as the register-tile kernels (sinkhorn_tile.cuh); problems
// whose supports overlap so far that their rows do not fit go to the kernels behind it (iters = -1).
//
// Measured (B200, 512 ranks, 256 problems, 500 iterations): 20.7 -> 1.03 ms (dense products over all R x R on the tensor cores
// before); 3.4 us an iteration over the batch, two waves of problems, about 1600 cycles an iteration.  By supply ranks, against
// the four-CTA clusters (which took what had more than 64) and the dense products, ms for 500 iterations:
//   problems   supply ranks    16     54     65     96    128    256    288    384    clusters at 96 / 256    dense products
//        256                 0.62   1.02   2.02   2.56   2.90   3.64   4.19   3.32          10.4 / 14.6              20.8
//       1024                 2.09   3.47   6.93   8.84   10.0   12.6   14.5   11.5          41.7 / 58.4              21.3
#include <algorithm>
#include <type_traits>

#include "sinkhorn_common.cuh"

using namespace taot_sk;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxR = 512, kMaxRows = 64, kMaxWarps = kMaxR / 32, kMaxBlocks = kMaxWarps / 4;
typedef unsigned long long u64;

__device__ __forceinline__ float rcp_fast(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// a / b to the last half bit or so (operands well inside the range of fp32)
__device__ __forceinline__ float div_fast(float a, float b)
{
    const float r = rcp_fast(b), q = a * r;
    return fmaf(fmaf(-b, q, a), r, q);
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
// blocks of 64 rows that the registers of NW warps hold for Cn columns: a warp for 32 columns of a block, two threads per
// row for the totals
__host__ __device__ inline int row_blocks(int NW, int Cn)
{
    const int by_columns = NW / ((Cn + 31) / 32), by_rows = NW / 4;
    return by_columns < by_rows ? by_columns : by_rows;
}
__device__ __forceinline__ bool in_range(float x) { return x > kSumLo && x < kSumHi; }

struct WideSmem {
    double alpha[kMaxR], beta[kMaxR], red[2][kMaxWarps + 1];
    float st[kMaxR];
    __align__(16) float u[2][kMaxBlocks][kMaxRows / 8 * 20];   // u~ by parity of the iteration, each twice (a packed operand), by
                                                   // row lane with a stride of 2 RT + 4 (no bank conflicts between the row lanes)
    __align__(16) float ux[3][kMaxR - kMaxRows];   // u~ of the rows in shared memory: iterates t - 1, t, t + 1 in turn
    __align__(16) float v[kMaxR];                  // v~
    __align__(16) float part[kMaxWarps][80];       // row sums by warp (stride: the two readers of a row meet no bank conflict)
    float err[kMaxRows];                           // error terms by row, or (beyond 64 rows) by warp
    int16_t hot[kMaxR], cold[kMaxR], hpos[kMaxR], cpos[kMaxR];
    int32_t wcnt[32];
    int event[3];                                  // iteration after which an event is due: [0] drift, [1] stop, [2] drift (odd)
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
    const float* dem = a.d + b * R;                // demand: positive on the columns
    const float dd = col_ok ? dem[sm.cold[col]] : 1.0f;
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
        sm.beta[j] = log((double)dem[sm.cold[j]]) - (mx + log(acc));
    }
    build(true);
    load_tile();
    if (totals) sm.u[1][0][uq] = 1.0f;               // iterate 1
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
                const float un = row_ok ? sm.u[t & 1][0][uq] : 1.0f;
                if (!in_range(un) || !in_range(vo)) sm.bad = 1;
                __syncthreads();
                if (sm.bad) return false;
                if (row_ok && !(tid & 1)) sm.alpha[row] += log((double)un);
                if (col_ok) sm.beta[col] += log((double)vo);
                __syncthreads();
                if (totals) sm.u[t & 1][0][uq] = 1.0f;
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
                    if (!(tid & 1)) e = (double)fabsf(fmaf(sm.u[t & 1][0][uq], r, -st));
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
            if (TOL && check_now && !(tid & 1)) sm.err[row] = row_ok ? fabsf(fmaf(sm.u[t & 1][0][uq], r, -st)) : 0.0f;
            sm.u[(t + 1) & 1][0][uq] = un;
            if (!in_window(un)) sm.event[0] = t + 1;
        }
        __syncthreads();
        // ================= half-step 2: column sums, inside the warp
        if (mainw) {
            float q[8];
            {
                u64 q2[4];
                const ulonglong2* up = reinterpret_cast<const ulonglong2*>(&sm.u[(t + 1) & 1][0][rl * (2 * RT + 4)]);
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
    if (row_ok && !(tid & 1)) sm.alpha[row] += log((double)sm.u[t & 1][0][uq]);
    if (col_ok) sm.beta[col] += log((double)vo);
    while (zero_row < R) write_zero_row();
    build(false);
    for (int j = tid; j < NC; j += NT) {
        float acc = 0.0f;
        for (int i = 0; i < Hn; ++i) acc += tile[i * NC + j];
        sm.v[j] = j < Cn ? (float)fmin(1.0, (double)dem[sm.cold[j]] / ((double)acc + (double)a.eps0)) : 0.0f;
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

// The same beyond 64 supply ranks.  Warp (row block rb, column warp cw) holds rows 64 rb .. 64 rb + 63 of its 32 columns in
// registers, as above; there are as many row blocks as the columns leave warps for (at most NW / 4).  The other rows are in shared
// memory, `tile`, [rows][ldx].  An iteration, a block barrier behind each part: row sums (the rows in shared memory, one
// warp each, which also divides); the rows in registers totalled and divided, and meanwhile the columns' sums over the rows in
// shared memory; the columns' sums over the rows in registers; (more than one row block) added and divided.
template <bool TOL>
__device__ __forceinline__ bool wide_solve_tall(const SinkArgs& a, WideSmem& sm, float* tile, const int NW, const int Hn, const int Cn,
                                                const double sum_st, int info, float* out, const int64_t b)
{
    constexpr int RT = 8, NR = 8 * RT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, R = a.R;
    const bool mainw = warp < NW;                  // with a tolerance one more warp sums the row error beside the iteration
    const int CW = (Cn + 31) >> 5, NB = row_blocks(NW, Cn);
    const int rb = warp / CW, cw = warp - rb * CW;
    const bool holds = mainw && rb < NB, owner = rb == 0;       // owner: divides the columns
    const int rl = lane & 7, cl = lane >> 3;
    const int XN = max(0, Hn - NB * NR), ldx = (Cn + 3) & ~3, X0 = NB * NR;
    const float tol_abs = (float)((double)a.tol * sum_st);
    const int col = cw * 32 + lane;                // the column whose sum this lane ends up with
    const bool col_ok = owner && col < Cn;
    const float* dem = a.d + b * R;                // demand: positive on the columns
    const float dd = col_ok ? dem[sm.cold[col]] : 1.0f;
    u64 K[RT][4];                                  // rows 64 rb + rl * RT + a, columns 32 cw + 8 cl + (2k, 2k + 1)
    float vo = 1.0f, vprev = 1.0f;                 // v~ of column `col`: iterate t, iterate t - 1
    float *ux_p = sm.ux[0], *ux_t = sm.ux[1], *ux_n = sm.ux[2];
    const bool totals = tid < 2 * NR * NB;         // two threads per row in registers: whole warps
    const int row = tid >> 1;
    const bool row_ok = totals && row < Hn;
    const float st = row_ok ? sm.st[row] : 1.0f;
    const int ub = (row >> 6) & (kMaxBlocks - 1), uq = (row & 63) / RT * (2 * RT + 4) + (row & 63) % RT * 2 + (tid & 1);

    auto entry = [&](const int i, const int j) {   // row i, column j of K~; zero off the block
        const bool ok = i < Hn && j < Cn;
        const double c = (double)a.C[(int64_t)sm.hot[ok ? i : 0] * R + sm.cold[ok ? j : 0]] * a.inv_eps;
        const float e = exp_split(sm.alpha[ok ? i : 0] + sm.beta[ok ? j : 0] - c);
        return ok ? e : 0.0f;
    };
    auto build_rows = [&]() {                      // block-wide: the rows in shared memory from the potentials
        __syncthreads();
#pragma unroll 4
        for (int q = tid; q < XN * ldx; q += NT) {
            const int i = q / ldx;
            tile[q] = entry(X0 + i, q - i * ldx);
        }
    };
    auto row_parts = [&]() {                       // this warp's part of the sums of its rows
        float p[RT];
        u64 v2[4];
        const ulonglong2* vp = reinterpret_cast<const ulonglong2*>(sm.v + cw * 32 + cl * 8);
        const ulonglong2 v01 = vp[0], v23 = vp[1];
        v2[0] = v01.x; v2[1] = v01.y; v2[2] = v23.x; v2[3] = v23.y;
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            u64 acc = mul2(K[r][0], v2[0]);
#pragma unroll
            for (int k = 1; k < 4; ++k) fma2(acc, K[r][k], v2[k]);
            float x, y;
            unpack2(acc, x, y);
            p[r] = x + y;
        }
        const bool up4 = (lane & 16) != 0, up3 = (lane & 8) != 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float send = up4 ? p[r] : p[r + 4], keep = up4 ? p[r + 4] : p[r];
            p[r] = keep + __shfl_xor_sync(kFull, send, 16);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float send = up3 ? p[r] : p[r + 2], keep = up3 ? p[r + 2] : p[r];
            p[r] = keep + __shfl_xor_sync(kFull, send, 8);
        }
        *reinterpret_cast<float2*>(&sm.part[warp][rl * RT + (up4 ? 4 : 0) + (up3 ? 2 : 0)]) = make_float2(p[0], p[1]);
    };
    const float* part_at = &sm.part[min(ub * CW + (tid & 1), kMaxWarps - 1)][row & 63];
    // two threads per row add the warps' parts: the row sum in both (threads below 2 NR NB)
    auto row_total = [&]() {
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < kMaxWarps / 2; ++k)
            if (2 * k + (tid & 1) < CW) s += part_at[2 * k * (int)(sizeof(sm.part[0]) / sizeof(float))];
        return s + __shfl_xor_sync(kFull, s, 1);
    };
    // row sums of the rows in shared memory, every NW-th row a warp's: take(row beyond X0, sum) in one lane each.  As many rows at a
    // time as a warp has, up to 8 (4 with a tolerance: registers): a lone row of a warp takes a third of the time of eight
    auto some_rows = [&](auto rows, const int x0, auto take) {
        constexpr int RX = decltype(rows)::value;
        const float* k[RX];
        u64 acc[RX];
#pragma unroll
        for (int r = 0; r < RX; ++r) { k[r] = tile + min(x0 + r * NW, XN - 1) * ldx; acc[r] = 0; }
#pragma unroll 1
        for (int j = lane * 4; j < ldx; j += 128) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(sm.v + j);
            ulonglong2 x[RX];
#pragma unroll
            for (int r = 0; r < RX; ++r) x[r] = *reinterpret_cast<const ulonglong2*>(k[r] + j);
#pragma unroll
            for (int r = 0; r < RX; ++r) fma2(acc[r], x[r].x, w.x);
#pragma unroll
            for (int r = 0; r < RX; ++r) fma2(acc[r], x[r].y, w.y);
        }
        float p[RX];
#pragma unroll
        for (int r = 0; r < RX; ++r) {
            float x, y;
            unpack2(acc[r], x, y);
            p[r] = x + y;
        }
        // a transposing butterfly: lane l ends with row l / (32 / RX)
        int o = 16;
#pragma unroll
        for (int h = RX / 2; h > 0; h >>= 1, o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int r = 0; r < h; ++r) {
                const float send = up ? p[r] : p[r + h], keep = up ? p[r + h] : p[r];
                p[r] = keep + __shfl_xor_sync(kFull, send, o);
            }
        }
#pragma unroll
        for (int q = 32 / RX / 2; q > 0; q >>= 1) p[0] += __shfl_xor_sync(kFull, p[0], q);
        const int x = x0 + lane / (32 / RX) * NW;
        if (lane % (32 / RX) == 0 && x < XN) take(x, p[0]);
    };
    auto shared_rows = [&](auto take) {
        constexpr int most = TOL ? 4 : 8;
        for (int x0 = warp; x0 < XN; x0 += NW * most) {
            const int left = XN - x0 + warp;       // rows of all warps from here on
            if (left <= NW) some_rows(std::integral_constant<int, 1>(), x0, take);
            else if (left <= 2 * NW) some_rows(std::integral_constant<int, 2>(), x0, take);
            else if (TOL || left <= 4 * NW) some_rows(std::integral_constant<int, 4>(), x0, take);
            else some_rows(std::integral_constant<int, most>(), x0, take);
        }
    };
    // this block's share of those rows in the sum of this lane's column: lane 8 s + c takes columns 4 c .. 4 c + 3 of every
    // fourth row, then the four s are added and every lane gets its column
    const int per = ((XN + NB - 1) / NB + 3) & ~3, xa = min(XN, rb * per), xe = min(XN, xa + per);
    const int xcol = min(cw * 32 + rl * 4, ldx - 4), from = ((lane & 3) << 3) | (lane >> 2);
    auto shared_column = [&](const float* w) {
        u64 c01 = 0, c23 = 0;
        const float* k = tile + (xa + cl) * ldx + xcol;
#pragma unroll 8
        for (int x = xa + cl; x < xe; x += 4, k += 4 * ldx) {
            const ulonglong2 k4 = *reinterpret_cast<const ulonglong2*>(k);
            const u64 u2 = pack2(w[x], w[x]);
            fma2(c01, k4.x, u2);
            fma2(c23, k4.y, u2);
        }
        float c[4];
        unpack2(c01, c[0], c[1]);
        unpack2(c23, c[2], c[3]);
        const bool up4 = (lane & 16) != 0, up3 = (lane & 8) != 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float send = up4 ? c[i] : c[i + 2], keep = up4 ? c[i + 2] : c[i];
            c[i] = keep + __shfl_xor_sync(kFull, send, 16);
        }
        const float send = up3 ? c[0] : c[1], keep = up3 ? c[1] : c[0];
        return __shfl_sync(kFull, keep + __shfl_xor_sync(kFull, send, 8), from);
    };

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

    // ---- iteration 1 in the log domain, second half: eight rows at a time, rescaled when the maximum moves
    for (int j = tid; j < Cn; j += NT) {
        const float* cj = a.C + sm.cold[j];
        double mx = -INFINITY, acc = 0.0;
        for (int i0 = 0; i0 < Hn; i0 += 8) {
            double x[8], m8 = -INFINITY;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = min(i0 + q, Hn - 1);
                x[q] = i0 + q < Hn ? sm.alpha[i] - (double)cj[(int64_t)sm.hot[i] * R] * a.inv_eps : -INFINITY;
                m8 = fmax(m8, x[q]);
            }
            if (m8 > mx) { acc *= mx == -INFINITY ? 0.0 : (double)exp_split(mx - m8); mx = m8; }
#pragma unroll
            for (int q = 0; q < 8; ++q) acc += i0 + q < Hn ? (double)exp_split(x[q] - mx) : 0.0;
        }
        sm.beta[j] = log((double)dem[sm.cold[j]]) - (mx + log(acc));
    }
    for (int x = tid; x < XN; x += NT) ux_t[x] = 1.0f;            // iterate 1
    if (totals) sm.u[1][ub][uq] = 1.0f;
    if (tid == 0) { sm.event[0] = -1; sm.event[1] = -1; sm.event[2] = -1; sm.bad = 0; }
    if (holds && owner) sm.v[col] = 1.0f;

    int t = 1, until_check = a.check_every;
    float err_out = 0.0f;
    for (;;) {
    build_rows();
    if (holds) {
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = rb * NR + rl * RT + r, j = cw * 32 + cl * 8 + 2 * k;
                K[r][k] = pack2(entry(i, j), entry(i, j + 1));
            }
    }
    int ev_drift, ev_stop;
#pragma unroll 1
    for (;;) {
        __syncthreads();
        // ================= half-step 1: row sums of iterate t.  (The rows in shared memory already get u~ of t + 1, in the buffer
        // of t - 2; their drift goes to the word of the other parity: this iteration's events are looked at below)
        float e = 0.0f;                            // this lane's error terms of iterate t
        if (holds) row_parts();
        if (mainw)
            shared_rows([&](const int x, const float z) {
                const float s = sm.st[X0 + x], un = div_fast(s, z);
                if (TOL) e += fabsf(fmaf(ux_t[x], z, -s));
                ux_n[x] = un;
                if (!in_window(un)) sm.event[(t & 1) ? 0 : 2] = t + 1;
            });
        __syncthreads();
        ev_drift = sm.event[(t & 1) ? 2 : 0];
        ev_stop = TOL ? sm.event[1] : -1;
        if (ev_drift == t || ev_stop == t || t >= a.max_iters) break;
        bool check_now = false;
        if (TOL) {
            check_now = --until_check == 0;
            if (check_now) until_check = a.check_every;
        }
        if (totals) {
            const float r = row_total();
            const float un = row_ok ? div_fast(st, r) : 1.0f;
            if (TOL && row_ok && !(tid & 1)) e += fabsf(fmaf(sm.u[t & 1][ub][uq], r, -st));
            sm.u[(t + 1) & 1][ub][uq] = un;
            if (!in_window(un)) sm.event[(t & 1) ? 0 : 2] = t + 1;
        }
        if (TOL && check_now && mainw) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
            if (lane == 0) sm.err[warp] = e;
        }
        const float xc = holds ? shared_column(ux_n) : 0.0f;
        __syncthreads();
        // ================= half-step 2: column sums
        float q[8];
        if (holds) {
            u64 q2[4];
            const ulonglong2* up = reinterpret_cast<const ulonglong2*>(&sm.u[(t + 1) & 1][rb][rl * (2 * RT + 4)]);
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
#pragma unroll
            for (int off = 4; off >= 1; off >>= 1) {
                const bool up = (rl & off) != 0;
#pragma unroll
                for (int k = 0; k < off; ++k) {
                    const float send = up ? q[k] : q[k + off], keep = up ? q[k + off] : q[k];
                    q[k] = keep + __shfl_xor_sync(kFull, send, off);
                }
            }
            q[0] += xc;
            if (!owner) sm.part[warp][lane] = q[0];
        } else if (TOL && check_now && !mainw) {   // the error warp: the terms of iterate t
            float s = lane < NW ? sm.err[lane] : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
            if (lane == 0 && s <= tol_abs) sm.event[1] = t + 1;
        }
        if (NB > 1) __syncthreads();
        if (holds && owner) {
            for (int g = 1; g < NB; ++g) q[0] += sm.part[g * CW + cw][lane];
            vprev = vo;
            vo = col_ok ? div_fast(dd, q[0]) : 1.0f;
            if (!in_window(vo)) sm.event[(t & 1) ? 0 : 2] = t + 1;
            sm.v[col] = vo;
        }
        if (zero_row < R) write_zero_row();
        { float* x = ux_p; ux_p = ux_t; ux_t = ux_n; ux_n = x; }
        ++t;
    }
    if (TOL && ev_stop == t) {             // iterate t - 1 met the tolerance: back to it
        --t;
        vo = vprev;
        ux_t = ux_p;
    } else if (ev_drift == t) {
        // u~ or v~ of iterate t left the window: fold it into the potentials, or hand the problem back if a sum left
        // the range in which fp32 products are trustworthy
        const float un = row_ok ? sm.u[t & 1][ub][uq] : 1.0f;
        if (!in_range(un) || !in_range(vo)) sm.bad = 1;
        for (int x = tid; x < XN; x += NT)
            if (!in_range(ux_t[x])) sm.bad = 1;
        __syncthreads();
        if (sm.bad) return false;
        if (row_ok && !(tid & 1)) sm.alpha[row] += log((double)un);
        if (col_ok) sm.beta[col] += log((double)vo);
        for (int x = tid; x < XN; x += NT) { sm.alpha[X0 + x] += log((double)ux_t[x]); ux_t[x] = 1.0f; }
        if (totals) sm.u[t & 1][ub][uq] = 1.0f;
        if (tid == 0) { sm.event[0] = -1; sm.event[2] = -1; }
        vo = 1.0f;
        if (holds && owner) sm.v[col] = 1.0f;
        continue;
    }
    // ---- the result is iterate t: its row sums and error
    if (holds && owner) sm.v[col] = vo;
    __syncthreads();
    double ed = 0.0;
    if (holds) row_parts();
    if (mainw)
        shared_rows([&](const int x, const float z) {
            if (!in_range(z)) sm.bad = 1;
            ed += (double)fabsf(fmaf(ux_t[x], z, -sm.st[X0 + x]));
        });
    __syncthreads();
    if (totals) {
        const float r = row_total();
        if (row_ok) {
            if (!in_range(r)) sm.bad = 1;
            if (!(tid & 1)) ed += (double)fabsf(fmaf(sm.u[t & 1][ub][uq], r, -st));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ed += __shfl_xor_sync(kFull, ed, o);
    if (lane == 0) sm.red[0][warp] = ed;
    __syncthreads();
    if (sm.bad) return false;
    ed = 0.0;
    for (int w = 0; w < (NT >> 5); ++w) ed += sm.red[0][w];
    err_out = (float)(ed / sum_st);
    if (TOL && !((float)ed <= tol_abs)) info |= TAOT_INFO_SINKHORN_CAP;
    break;
    }

    // ---- T = diag(u) M diag(v) from the total potentials, then the column cap.  (The rows that were in registers are formed where
    //      they are needed, twice.)
    if (row_ok && !(tid & 1)) sm.alpha[row] += log((double)sm.u[t & 1][ub][uq]);
    if (col_ok) sm.beta[col] += log((double)vo);
    for (int x = tid; x < XN; x += NT) sm.alpha[X0 + x] += log((double)ux_t[x]);
    while (zero_row < R) write_zero_row();
    build_rows();
    __syncthreads();
    for (int j = tid; j < Cn; j += NT) {
        double acc = 0.0;                          // (hundreds of terms: their rounding in fp32 would show in the cap)
#pragma unroll 4
        for (int i = 0; i < min(X0, Hn); ++i) acc += (double)entry(i, j);
        for (int x = 0; x < XN; ++x) acc += (double)tile[x * ldx + j];
        sm.v[j] = (float)fmin(1.0, (double)dem[sm.cold[j]] / (acc + (double)a.eps0));
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
            float w = 0.0f;
            if (c >= 0) w = (h < X0 ? entry(h, c) : tile[(h - X0) * ldx + c]) * sm.v[c];
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
sinkhorn_wide_kernel(SinkArgs a, int64_t nprob, int32_t cap)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WideSmem& sm = *reinterpret_cast<WideSmem*>(smem_raw);
    float* tile = reinterpret_cast<float*>(smem_raw + ((sizeof(WideSmem) + 15) & ~(size_t)15));
    const int R = a.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, NW = (R + 31) >> 5;
    const int64_t b = blockIdx.x;
    taot_await();
    if (b >= nprob) return;                        // cap: floats of `tile`

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
    const bool tall = Hn > kMaxRows && Cn > 0;
    const int rest = tall ? Hn - row_blocks(NW, Cn) * kMaxRows : 0;      // rows in shared memory
    if (rest > 0 && rest * ((Cn + 3) & ~3) > cap) {               // another kernel takes it
        if (tid == 0) a.iters[b] = kHandBack;
        return;
    }
    for (int i = tid; i < Hn; i += NT) sm.st[i] = sv_all[sm.hot[i]];
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
    else if (!tall) done = wide_solve<8, TOL>(a, sm, tile, NW, Hn, Cn, sum_st, info, out, b);
    else done = wide_solve_tall<TOL>(a, sm, tile, NW, Hn, Cn, sum_st, info, out, b);
    if (!done && tid == 0) a.iters[b] = kHandBack;
}

}  // namespace

// Launches the kernel for 257 to 512 ranks (returns 1), otherwise nothing (0).
//
// Against the dense tensor-core solve (sinkhorn_dense_tc.cu), which multiplies all R x R entries whatever the supports: see
// TAOT_WIDE_MIN_ITERS.
int taot_launch_sinkhorn_wide(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st)
{
    if (a.R <= 256 || a.R > kMaxR) return 0;
    const int NW = (a.R + 31) / 32;
    // the staging of 64 rows, or the rows beyond 64 of disjoint supports with one row block: (h - 64) (c rounded up to 4) where
    // h + c <= R and c takes more than half of the warps
    const size_t state = (sizeof(WideSmem) + 15) & ~(size_t)15;
    int32_t cap = kMaxRows * 32 * NW;
    for (int c = 1; c < a.R - kMaxRows; ++c) {
        const int rest = a.R - c - row_blocks(NW, c) * kMaxRows;
        cap = std::max(cap, rest * ((c + 3) & ~3));
    }
    const size_t smem = state + sizeof(float) * (size_t)cap;
    if (a.tol > 0.0f) {
        TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_wide_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        TAOT_CUDA_OK(taot_launch_chained(sinkhorn_wide_kernel<true>, B, NW * 32 + 32, smem, st, a, (int64_t)B, cap));
    } else {
        TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_wide_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        TAOT_CUDA_OK(taot_launch_chained(sinkhorn_wide_kernel<false>, B, NW * 32, smem, st, a, (int64_t)B, cap));
    }
    TAOT_CUDA_OK(cudaGetLastError());
    return 1;
}
