// Phase 1: batched entropic optimal transport by Sinkhorn-Knopp (Appendix A.2).
//
// One CTA per problem.  The paper's iteration u = s~/(M v), v = d/(M^T u) is carried in the
// "absorbed" form: total log-potentials are split as  log u = alpha + log u~,  log v = beta +
// log v~  with (alpha, beta) in fp64 and (u~, v~) in fp32 near 1, and the kernel matrix held on
// chip is  K~_ij = exp(alpha_i + beta_j - C_ij/eps)  rounded to fp32.  A half-step is then an
// fp32 mat-vec over K~ followed by a divide, exactly the paper's GEMV form, but it cannot
// under- or overflow for any C/eps: whenever u~ or v~ drifts outside [e^-40, e^40] the factors
// are folded into (alpha, beta) and K~ is rebuilt (fp64 exp, a few times per solve).  Only rows
// with supply and columns with demand carry flow, so K~ is compacted to |hot| x |cold|.
// The first iteration (v = 1 on every rank) is done in the log domain in fp64; so is any
// iteration whose fp32 sums leave the safe range, which makes the solve total.
//
// Stopping: half-step 1 of iteration t+1 produces the row sums of iterate t for free
// (rowsum_i = u~_i * (K~ v~)_i), so the tolerance test costs nothing extra.
//
// The solve that takes any problem: the last kernel of every chain (sinkhorn.cu), and the end of the four-CTA clusters' kernel
// behind the class kernels (sinkhorn_cluster.cu).
#pragma once

#include "sinkhorn_common.cuh"

using namespace taot_sk;

namespace {

struct Smem {
    double* alpha;   // [R] by compact hot index
    double* beta;    // [R] by compact cold index
    double* phin;    // [R] scratch: new log-potential of the rows (slow path)
    double* errp;    // [32]
    float* st;       // [R] scaled supply, compact
    float* dd;       // [R] demand, compact
    float* u;        // [R]
    float* un;       // [R]
    float* v;        // [R]
    float* vn;       // [R]
    float* part;     // [max(NT, R)]
    int32_t* hot;    // [R] compact -> rank
    int32_t* cold;   // [R]
    int32_t* hpos;   // [R] rank -> compact or -1
    int32_t* cpos;   // [R]
    int32_t* wcnt;   // [32]
    int32_t* flags;  // [4]: 0 bad sum, 1 drift
    float* Kt;       // [kcap]
};

__device__ __forceinline__ Smem carve(unsigned char* base, int R, int NT)
{
    Smem m;
    double* dp = reinterpret_cast<double*>(base);
    m.alpha = dp; dp += R;
    m.beta = dp; dp += R;
    m.phin = dp; dp += R;
    m.errp = dp; dp += 32;
    float* fp = reinterpret_cast<float*>(dp);
    m.st = fp; fp += R;
    m.dd = fp; fp += R;
    m.u = fp; fp += R;
    m.un = fp; fp += R;
    m.v = fp; fp += R;
    m.vn = fp; fp += R;
    m.part = fp; fp += (NT > R ? NT : R);
    int32_t* ip = reinterpret_cast<int32_t*>(fp);
    m.hot = ip; ip += R;
    m.cold = ip; ip += R;
    m.hpos = ip; ip += R;
    m.cpos = ip; ip += R;
    m.wcnt = ip; ip += 32;
    m.flags = ip; ip += 4;
    m.Kt = reinterpret_cast<float*>(ip);
    return m;
}

inline size_t generic_smem_bytes(int R, int NT, int kcap)
{
    return sizeof(double) * (3 * R + 32) + sizeof(float) * (6 * R + (NT > R ? NT : R)) +
           sizeof(int32_t) * (4 * R + 36) + sizeof(float) * (size_t)kcap;
}

// K~_ij = exp(alpha_i + beta_j - C_ij/eps), fp64 exponent and exp, rounded once to fp32
__device__ void rebuild_kernel(const Smem& m, const SinkArgs& a, int Hn, int Cn)
{
    for (int q = threadIdx.x; q < Hn * Cn; q += blockDim.x) {
        const int i = q / Cn, j = q - i * Cn;
        const double c = (double)a.C[(int64_t)m.hot[i] * a.R + m.cold[j]] * a.inv_eps;
        m.Kt[q] = (float)exp(m.alpha[i] + m.beta[j] - c);
    }
}

// slow path, rows: L_i = LSE_j(psi_j - C_ij/eps) with psi = beta + log v~;  phin_i = log s~_i - L_i;
// contributes |exp(phi_i + L_i) - s~_i| to the row violation (phi = alpha + log u~).
__device__ void slow_half1(const Smem& m, const SinkArgs& a, int Hn, int Cn)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double e = 0.0;
    for (int i = tid; i < Hn; i += blockDim.x) {
        const float* crow = a.C + (int64_t)m.hot[i] * a.R;
        double mx = -INFINITY;
        for (int j = 0; j < Cn; ++j) {
            const double x = m.beta[j] + log((double)m.v[j]) - (double)crow[m.cold[j]] * a.inv_eps;
            mx = x > mx ? x : mx;
        }
        double acc = 0.0;
        for (int j = 0; j < Cn; ++j) {
            const double x = m.beta[j] + log((double)m.v[j]) - (double)crow[m.cold[j]] * a.inv_eps;
            acc += exp(x - mx);
        }
        const double L = mx + log(acc);
        const double phi = m.alpha[i] + log((double)m.u[i]);
        e += fabs(exp(phi + L) - (double)m.st[i]);
        m.phin[i] = log((double)m.st[i]) - L;
    }
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) m.errp[warp] = e;
}

// slow path, columns: beta_j = log d_j - LSE_i(phin_i - C_ij/eps); then alpha = phin, u~ = v~ = 1
__device__ void slow_half2(const Smem& m, const SinkArgs& a, int Hn, int Cn)
{
    for (int j = threadIdx.x; j < Cn; j += blockDim.x) {
        const int cj = m.cold[j];
        double mx = -INFINITY;
        for (int i = 0; i < Hn; ++i) {
            const double x = m.phin[i] - (double)a.C[(int64_t)m.hot[i] * a.R + cj] * a.inv_eps;
            mx = x > mx ? x : mx;
        }
        double acc = 0.0;
        for (int i = 0; i < Hn; ++i) {
            const double x = m.phin[i] - (double)a.C[(int64_t)m.hot[i] * a.R + cj] * a.inv_eps;
            acc += exp(x - mx);
        }
        m.beta[j] = log((double)m.dd[j]) - (mx + log(acc));
        m.v[j] = 1.0f;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < Hn; i += blockDim.x) { m.alpha[i] = m.phin[i]; m.u[i] = 1.0f; }
    __syncthreads();
    rebuild_kernel(m, a, Hn, Cn);
    __syncthreads();
}

// The solve of problem b by the whole CTA.
__device__ void generic_problem(const SinkArgs& a, const int64_t b, unsigned char* smem_raw)
{
    const int R = a.R, NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = NT >> 5;
    Smem m = carve(smem_raw, R, NT);
    __shared__ double s_sum[2];

    // ---- supply scaling gamma = min(1, sum d / max(sum s, eps0)), compaction
    if (tid == 0) { s_sum[0] = 0.0; s_sum[1] = 0.0; }
    __syncthreads();
    {
        double ps = 0.0, pd = 0.0;
        for (int i = tid; i < R; i += NT) {
            const float sv = a.s[b * R + i], dv = a.d[b * R + i];
            ps += sv > 0.0f ? (double)sv : 0.0;
            pd += dv > 0.0f ? (double)dv : 0.0;
        }
        for (int o = 16; o > 0; o >>= 1) {
            ps += __shfl_xor_sync(0xffffffffu, ps, o);
            pd += __shfl_xor_sync(0xffffffffu, pd, o);
        }
        if (lane == 0) { m.errp[warp] = ps; m.phin[warp] = pd; }   // phin is free here
        __syncthreads();
        if (tid == 0) {
            double S = 0.0, D = 0.0;
            for (int w = 0; w < NW; ++w) { S += m.errp[w]; D += m.phin[w]; }
            s_sum[0] = S; s_sum[1] = D;
        }
        __syncthreads();
    }
    const double sum_s = s_sum[0], sum_d = s_sum[1];
    const double gamma = fmin(1.0, sum_d / fmax(sum_s, (double)a.eps0));
    // scaled supply and demand by rank, in un[] / vn[] for the compaction
    for (int i = tid; i < R; i += NT) {
        const float sv = a.s[b * R + i], dv = a.d[b * R + i];
        m.un[i] = sv > 0.0f ? (float)(gamma * (double)sv) : 0.0f;
        m.vn[i] = dv > 0.0f ? dv : 0.0f;
    }
    __syncthreads();
    const int Hn = compact_positive(m.un, R, m.hot, m.hpos, m.wcnt);
    const int Cn = compact_positive(m.vn, R, m.cold, m.cpos, m.wcnt);
    for (int i = tid; i < Hn; i += NT) m.st[i] = m.un[m.hot[i]];
    for (int j = tid; j < Cn; j += NT) m.dd[j] = m.vn[m.cold[j]];
    __syncthreads();

    int info = 0;
    if (sum_s > sum_d) info |= TAOT_INFO_SUPPLY_SCALED;
    const bool empty = (Hn == 0) || (Cn == 0);
    bool too_big = (int64_t)Hn * Cn > (int64_t)a.kcap;
    if (too_big && a.kt_global != nullptr && (int64_t)Hn * Cn <= a.kcap_global) {
        m.Kt = a.kt_global + b * a.kcap_global;           // kernel matrix in global memory (L2 when the batch is small)
        too_big = false;
    }
    float* out = a.plan + b * (int64_t)R * R;
    const bool in_plan = too_big && Hn <= a.plan_rows;        // |hot| x |cold| <= R x R: the plan's own block always holds it
    if (in_plan) { m.Kt = out; too_big = false; }
    if (too_big) info |= TAOT_INFO_SINKHORN_SIZE;

    int t = 0;
    float err_out = 0.0f;
    if (!empty && !too_big) {
        double sum_st = 0.0;
        for (int i = 0; i < Hn; ++i) sum_st += (double)m.st[i];      // same order in every thread
        const double tol_abs = (double)a.tol * sum_st;

        // ---- iteration 1 in the log domain: v = 1 on EVERY rank, so the row normaliser is the
        //      precomputed LSE_j(-C_ij/eps) over all j
        for (int i = tid; i < Hn; i += NT) {
            m.phin[i] = log((double)m.st[i]) - a.rowlse0[m.hot[i]];
            m.u[i] = 1.0f;
        }
        __syncthreads();
        slow_half2(m, a, Hn, Cn);
        t = 1;

        // half-step-2 thread layout: G row groups x Cnp columns
        const int Cnp = (Cn + 31) & ~31;
        const int G = NT >= Cnp ? NT / Cnp : 1;
        const int cstride = NT >= Cnp ? Cnp : NT;
        const int g = tid / cstride, j0 = tid - g * cstride;

        for (;;) {
            // ================= half-step 1: r = K~ v~ ; rows of iterate t; u' = s~ / r
            if (tid < 4) m.flags[tid] = 0;
            __syncthreads();
            {
                double e = 0.0;
                for (int i = warp; i < Hn; i += NW) {
                    const float* krow = m.Kt + i * Cn;
                    float p = 0.0f;
                    for (int j = lane; j < Cn; j += 32) p = fmaf(krow[j], m.v[j], p);
                    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
                    if (lane == 0) {
                        if (!(p > kSumLo && p < kSumHi)) m.flags[0] = 1;
                        const float un = m.st[i] / p;
                        if (!(un > kDriftLo && un < kDriftHi)) m.flags[1] = 1;
                        m.un[i] = un;
                        e += (double)fabsf(fmaf(m.u[i], p, -m.st[i]));
                    }
                }
                if (lane == 0) m.errp[warp] = e;
            }
            __syncthreads();
            bool slow = m.flags[0] != 0;
            if (slow) {                    // redo the rows exactly, from the iterate that is still intact
                __syncthreads();
                slow_half1(m, a, Hn, Cn);
                __syncthreads();
            }
            double err = 0.0;
            for (int w = 0; w < NW; ++w) err += m.errp[w];
            const bool check = a.tol > 0.0f && (t % a.check_every == 0);
            if (t >= a.max_iters || (check && err <= tol_abs)) {
                err_out = (float)(err / sum_st);
                if (a.tol > 0.0f && !(err <= tol_abs)) info |= TAOT_INFO_SINKHORN_CAP;
                break;
            }
            // ================= half-step 2: c = K~^T u' ; v' = d / c
            if (!slow) {
                for (int j = j0; j < Cn && g < G; j += cstride) {
                    float p = 0.0f;
                    for (int i = g; i < Hn; i += G) p = fmaf(m.Kt[i * Cn + j], m.un[i], p);
                    m.part[g * Cn + j] = p;
                }
                __syncthreads();
                for (int j = tid; j < Cn; j += NT) {
                    float c = 0.0f;
                    for (int gg = 0; gg < G; ++gg) c += m.part[gg * Cn + j];
                    if (!(c > kSumLo && c < kSumHi)) m.flags[0] = 1;
                    const float vn = m.dd[j] / c;
                    if (!(vn > kDriftLo && vn < kDriftHi)) m.flags[1] = 1;
                    m.vn[j] = vn;
                }
                __syncthreads();
                if (m.flags[0]) {          // columns left the safe range: finish this iteration exactly
                    slow = true;
                    for (int i = tid; i < Hn; i += NT) m.phin[i] = m.alpha[i] + log((double)m.un[i]);
                    __syncthreads();
                }
            }
            if (slow) {
                slow_half2(m, a, Hn, Cn);
            } else {
                // commit (u', v'); fold them into (alpha, beta) if they drifted
                const bool drift = m.flags[1] != 0;
                __syncthreads();
                if (drift) {
                    for (int i = tid; i < Hn; i += NT) { m.alpha[i] += log((double)m.un[i]); m.u[i] = 1.0f; }
                    for (int j = tid; j < Cn; j += NT) { m.beta[j] += log((double)m.vn[j]); m.v[j] = 1.0f; }
                    __syncthreads();
                    rebuild_kernel(m, a, Hn, Cn);
                } else {
                    for (int i = tid; i < Hn; i += NT) m.u[i] = m.un[i];
                    for (int j = tid; j < Cn; j += NT) m.v[j] = m.vn[j];
                }
                __syncthreads();
            }
            ++t;
        }

        // ---- T = diag(u) M diag(v) from the total potentials, then the column cap
        __syncthreads();
        for (int i = tid; i < Hn; i += NT) m.alpha[i] += log((double)m.u[i]);
        for (int j = tid; j < Cn; j += NT) m.beta[j] += log((double)m.v[j]);
        __syncthreads();
        rebuild_kernel(m, a, Hn, Cn);
        __syncthreads();
        for (int j = tid; j < Cn; j += NT) {
            double cs = 0.0;
            for (int i = 0; i < Hn; ++i) cs += (double)m.Kt[i * Cn + j];
            m.vn[j] = (float)fmin(1.0, (double)m.dd[j] / (cs + (double)a.eps0));
        }
        __syncthreads();
    }

    // ---- write the full R x R plan (zeros off the hot x cold block)
    int nonfinite = 0;
    if (in_plan && !empty) {
        // The compact matrix is where the plan goes: a row at a time, the last one first.  Row i is written to [iR, iR + R), and
        // what is still to be read, the rows of the supply ranks up to i, ends at (supply ranks below i) |cold| <= iR, but for
        // row i itself, which is in registers by then.
        for (int i = R - 1; i >= 0; --i) {
            const int hp = m.hpos[i], cp = tid < R ? m.cpos[tid] : -1;           // a thread per column (R <= NT)
            const float val = hp >= 0 && cp >= 0 ? m.Kt[hp * Cn + cp] * m.vn[cp] : 0.0f;
            if (!isfinite(val)) nonfinite = 1;
            __syncthreads();
            if (tid < R) out[(int64_t)i * R + tid] = val;
            __syncthreads();
        }
    }
    for (int q = tid; q < R * R && !(in_plan && !empty); q += NT) {
        const int i = q / R, j = q - i * R;
        float val = 0.0f;
        if (!empty && !too_big) {
            const int hp = m.hpos[i], cp = m.cpos[j];
            if (hp >= 0 && cp >= 0) val = m.Kt[hp * Cn + cp] * m.vn[cp];
        }
        if (!isfinite(val)) nonfinite = 1;
        out[q] = val;
    }
    nonfinite = __syncthreads_or(nonfinite);
    if (nonfinite) info |= TAOT_INFO_NONFINITE;
    if (tid == 0) {
        a.iters[b] = t;
        a.row_err[b] = err_out;
        if (info) atomicOr(a.info + b, info);
    }
}

}  // namespace
