// Sinkhorn-Knopp (Appendix A.2) on classes of ranks: one warp per problem, one class per lane.
//
// Two ranks whose rows and columns of the cost matrix agree off the pair itself are interchangeable for Phase 1: with
// supply and demand on disjoint ranks (the diagonal then never takes part) the iteration
//     u_i = s~_i / sum_j K_ij v_j,     v_j = d_j / sum_i K_ij u_i,     K = exp(-C/eps)
// keeps u_i = s~_i phi_a for every supply rank i of class a and v_j = d_j psi_b for every demand rank j of class b, for
// ALL iterates, with
//     phi_a = 1 / sum_b K_ab D_b psi_b,    psi_b = 1 / sum_a K_ab S_a phi_a,    S_a, D_b = mass of a class.
// In a topology cost the classes are the nodes: a solve over R ranks is a solve over R / 8 numbers, in exact
// arithmetic the same iterates, the same row error sum_a S_a |phi_a x_a - 1| and the same plan s~_i phi_a K_ab psi_b d_j.
// (First iteration: v = 1 on every rank gives phi_a = 1 / sum_j K_aj over all ranks, equal inside a class.)
//
// The numbers are carried in the absorbed form of the other kernels: phi = e^alpha u~, psi = e^beta v~ with fp64 alpha,
// beta and fp32 u~, v~ near 1; the matrices Kr_ab = e^(alpha_a + beta_b - C_ab/eps) D_b and Kc_ab = same S_a sit in
// registers, so a half-step is an exchange of 32 values inside the warp, NC multiply-adds and one reciprocal -- no
// multiplication by the masses and no block barrier.  A solve is one dependent chain, so the loop holds only that chain;
// both tests ride beside it: the drift vote of an iterate is consumed after the next half-step's exchange has been
// issued, and the row error is summed by one integer reduction (redux.sync over shares scaled to 2^20 parts of the
// tolerance, 3e-5 of the tolerance exact) that is consumed half an iteration later.  An iterate that leaves the fp32
// window is taken again in the log domain in fp64, so no problem is handed on except one that has a rank with both
// supply and demand.
//
// Measured (B200, 500 iterations, whole call): 64 ranks, one problem 125 -> 56 us (register tile before; 150 cycles per
// iteration against 370); 256 ranks, 1024 problems 283 -> 137 to 148 us; 1024 ranks, 64 problems 373 -> 160 us (tier sums over
// eight warps before; 340 cycles per iteration against 1400; of the last 18 us, clusters that share the supply rows and
// fp32 exponentials in the log-domain half-steps).  What is left at 1024 ranks: 87 us of iterations, the rest loading,
// the log-domain half-steps and the supply rows, which only the SMs of the problem can write.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "sinkhorn_class.h"
#include "sinkhorn_common.cuh"

using namespace taot_sk;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;             // the solving warps, and warps that write the plan
constexpr uint32_t kTolParts = 1u << 20;  // the tolerance as an integer
constexpr float kShareCap = 33554432.0f;  // 2^25: 32 saturated shares stay below 2^31

__device__ __forceinline__ float rcp_fast(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ bool in_window(float x)            // [e^-40, e^40], false for everything that is no such number
{
    return (__float_as_uint(x) - __float_as_uint(kDriftLo)) <= (__float_as_uint(kDriftHi) - __float_as_uint(kDriftLo));
}
// smallest and largest of a run of scaling factors; not-a-number stays one
template <int VPL>
struct Span {
    float lo = 1.0f, hi = 1.0f;
    __device__ __forceinline__ void take(const float (&x)[VPL])
    {
        if constexpr (VPL == 1) {
            asm("min.NaN.f32 %0, %0, %1;" : "+f"(lo) : "f"(x[0]));
            asm("max.NaN.f32 %0, %0, %1;" : "+f"(hi) : "f"(x[0]));
        } else {
#pragma unroll
            for (int i = 0; i < VPL; i += 2) {
                asm("min.NaN.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(x[i]), "f"(x[i + 1]));
                asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(x[i]), "f"(x[i + 1]));
            }
        }
    }
    __device__ __forceinline__ bool out() const { return !(lo >= kDriftLo && hi <= kDriftHi); }
};
__device__ __forceinline__ bool in_range(float x) { return x > kSumLo && x < kSumHi; }

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

struct ClassArgs {
    SinkArgs a;
    const uint16_t* cls;      // [R] slot of each rank's class
    const int32_t* off;       // [slots + 1] members of a slot (empty for a slot without a class)
    const uint16_t* list;     // [R] ranks by slot (the kernels stage cls, off and list in shared memory)
    const double* lse0;       // [slots] log-sum-exp of -C_ij/eps over all ranks j, for the ranks i of the slot
    const float* cost;        // dense kernel: [NC][NC] cost between classes; tree kernel: unused
    double c1, c2, c3;        // tree kernel: cost / eps inside a class, inside a group, elsewhere
    int32_t wide;             // rows of the plan can be written 16 bytes at a time
    int32_t solvers;          // CTAs of the problems; any beyond them write the rows without supply
    int32_t cluster;          // tree kernel: CTAs per problem
};

// what a problem's solve leaves in shared memory for the warps that write the plan
struct Verdict {
    int32_t state;            // 0 solved, 1 nothing to move or no solution (all zero), 2 not written here
    int32_t flags;            // while loading: bit 0 a value that is not finite, bit 1 a rank with both
    int32_t iters, info;
    float row_err;
    double gamma;             // supply scaling
};

// ---- loading: supply and demand of a problem into shared memory, negative values as zero
__device__ __forceinline__ void load_masses(const SinkArgs& a, int64_t b, float* st, float* dm, Verdict* v)
{
    int fl = 0;
    for (int i = threadIdx.x; i < a.R; i += kThreads) {
        const float sv = a.s[b * a.R + i], dv = a.d[b * a.R + i];
        if (!isfinite(sv) || !isfinite(dv)) fl |= 1;
        if (sv > 0.0f && dv > 0.0f) fl |= 2;
        st[i] = sv > 0.0f ? sv : 0.0f;
        dm[i] = dv > 0.0f ? dv : 0.0f;
    }
    if (fl) atomicOr(&v->flags, fl);
}

// rows of the plan that no supply rank owns, while the solving warps iterate (most of the plan's bytes)
__device__ __forceinline__ void zero_rows(float* out, const float* st, int R, int wide, int w, int nw)
{
    const int lane = threadIdx.x & 31;
    for (int row = w; row < R; row += nw) {
        if (st[row] > 0.0f) continue;
        float* o = out + (int64_t)row * R;
        if (wide) {
            for (int j = lane * 4; j < R; j += 128) *reinterpret_cast<float4*>(o + j) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        } else {
            for (int j = lane; j < R; j += 32) o[j] = 0.0f;
        }
    }
}

// the same by CTAs of their own, on SMs no problem sits on: a warp takes 32 rows of the batch at a time
__device__ __forceinline__ void zero_rows_of_batch(const SinkArgs& a, int64_t nprob, int wide, int64_t w, int64_t nw)
{
    const int lane = threadIdx.x & 31, R = a.R;
    for (int64_t r0 = w * 32; r0 < nprob * R; r0 += nw * 32) {
        const int64_t r = r0 + lane;
        unsigned todo = __ballot_sync(kFull, r < nprob * R && !(a.s[r < nprob * R ? r : 0] > 0.0f));
        while (todo) {
            const int q = __ffs(todo) - 1;
            todo &= todo - 1;
            float* o = a.plan + (r0 + q) * R;
            if (wide) {
                for (int j = lane * 4; j < R; j += 128) *reinterpret_cast<float4*>(o + j) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            } else {
                for (int j = lane; j < R; j += 32) o[j] = 0.0f;
            }
        }
    }
}

// ---- masses of the classes, supply scaling gamma = min(1, sum d / max(sum s, eps0)) (Appendix A.2): one thread per class of
// the CTA's problems, one warp per problem for the totals.  Block-wide.  S and D receive [PPC][slots] masses, the supply
// scaled; st is scaled by the caller's writers later (ver[p].gamma).
template <int PPC>
__device__ __forceinline__ void class_masses(const ClassArgs& k, const int32_t* off, const uint16_t* list, const float* st,
                                             const float* dm, int dstride, int slots, double* S, double* D, int64_t nprob_here, Verdict* ver)
{
    const SinkArgs& a = k.a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < PPC * slots; q += kThreads) {
        const int p = q / slots, s = q - p * slots;
        double ps = 0.0, pd = 0.0;
        if (p < nprob_here)
            for (int e = off[s]; e < off[s + 1]; ++e) {
                const int r = list[e];
                ps += (double)st[p * a.R + r];
                pd += (double)dm[p * dstride + r];
            }
        S[q] = ps; D[q] = pd;
    }
    __syncthreads();
    if (warp < PPC && warp < nprob_here) {
        double ps = 0.0, pd = 0.0;
        for (int s = lane; s < slots; s += 32) { ps += S[warp * slots + s]; pd += D[warp * slots + s]; }
        const double sum_s = warp_sum(ps), sum_d = warp_sum(pd);
        const double gamma = fmin(1.0, sum_d / fmax(sum_s, (double)a.eps0));
        if (lane == 0) {
            Verdict& v = ver[warp];
            const int fl = v.flags;
            v.gamma = gamma;
            v.state = fl == 0 && sum_s > 0.0 && sum_d > 0.0 ? 0 : ((fl & 1) || !(fl & 2) ? 1 : 2);
            v.iters = 0;
            v.row_err = 0.0f;
            v.info = (fl & 1) ? TAOT_INFO_NONFINITE : (sum_s > sum_d ? TAOT_INFO_SUPPLY_SCALED : 0);
        }
    }
    __syncthreads();
    for (int q = tid; q < PPC * slots; q += kThreads) {
        const int p = q / slots, s = q - p * slots;
        if (p >= nprob_here) continue;
        const double gamma = ver[p].gamma;
        if (gamma >= 1.0) continue;
        double ps = 0.0;
        for (int e = off[s]; e < off[s + 1]; ++e) ps += (double)(float)(gamma * (double)st[p * a.R + list[e]]);
        S[q] = ps;
    }
    __syncthreads();
}

// log of a scaling factor inside the window: exponent times ln 2 in fp64, logf of a mantissa in [0.75, 1.5) (3e-8 absolute)
__device__ __forceinline__ double log_factor(float x)
{
    const int e = (__float_as_int(x) - 0x3f400000) >> 23;
    return (double)e * 0.693147180559945309417 + (double)logf(__int_as_float(__float_as_int(x) - (e << 23)));
}

// share of the row error of a class, in parts of the tolerance (saturated; not a number counts as saturated)
template <int VPL>
__device__ __forceinline__ uint32_t error_parts(float share, float scale)
{
    return (uint32_t)fminf(share * scale, kShareCap / VPL);
}

// The iteration, common to both kernels.  `half(rows, w, x)` forms the row (rows) or column sums x of this lane's classes
// from the scaling factors w of the other side; `fold()` moves u, v into the potentials and rebuilds the factors;
// `exact()` takes one whole iteration in the log domain from the potentials alone and rebuilds.  On return (u, v) is
// the result, x its row sums and t its number.
template <int VPL, bool TOL, class Half, class Fold, class Exact>
__device__ __forceinline__ void iterate(const SinkArgs& a, const bool counts, const float (&S)[VPL], const float tol_scale,
                                        float (&u)[VPL], float (&v)[VPL], float (&x)[VPL], int& t, const Half& half,
                                        const Fold& fold, const Exact& exact)
{
    float up[VPL], vp[VPL];                       // the iterate before (u, v): what an iterate outside the window is retaken from
#pragma unroll
    for (int i = 0; i < VPL; ++i) { up[i] = u[i]; vp[i] = v[i]; }
    t = 1;
    if (!TOL) {
        // Fixed count: four iterations without a vote or a branch, then one vote on whether any u or v of the four left the
        // window; if so the four are taken again one by one (a vote per iteration, consumed at its end, costs 70 cycles)
        while (t < a.max_iters) {
            const int n = a.max_iters - t < 4 ? a.max_iters - t : 4;
#pragma unroll
            for (int i = 0; i < VPL; ++i) { up[i] = u[i]; vp[i] = v[i]; }
            bool out = n < 4;
            if (!out) {
                Span<VPL> span;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    half(true, v, x);
#pragma unroll
                    for (int i = 0; i < VPL; ++i) u[i] = rcp_fast(x[i]);
                    half(false, u, x);
                    span.take(u);
#pragma unroll
                    for (int i = 0; i < VPL; ++i) v[i] = rcp_fast(x[i]);
                    span.take(v);
                }
                out = span.out();
            }
            if (__any_sync(kFull, out)) {
#pragma unroll
                for (int i = 0; i < VPL; ++i) { u[i] = up[i]; v[i] = vp[i]; }
#pragma unroll 1
                for (int j = 0; j < n; ++j) {
                    float un[VPL], vn[VPL];
                    bool drift = false, bad = false;
                    half(true, v, x);
#pragma unroll
                    for (int i = 0; i < VPL; ++i) { un[i] = rcp_fast(x[i]); drift = drift || !in_window(un[i]); bad = bad || !in_range(un[i]); }
                    half(false, un, x);
#pragma unroll
                    for (int i = 0; i < VPL; ++i) { vn[i] = rcp_fast(x[i]); drift = drift || !in_window(vn[i]); bad = bad || !in_range(vn[i]); }
                    if (__any_sync(kFull, bad)) {
                        fold();
                        exact();
                    } else {
#pragma unroll
                        for (int i = 0; i < VPL; ++i) { u[i] = un[i]; v[i] = vn[i]; }
                        if (__any_sync(kFull, drift)) fold();
                    }
                }
            }
            t += n;
        }
        half(true, v, x);                         // the result's row sums
        return;
    }
    int until_check = a.check_every;
    bool event = false;                           // some u or v of iterate t left the window
    for (;;) {
        half(true, v, x);                         // row sums of iterate t
        if (event) {
            event = false;
            bool ok = true;
#pragma unroll
            for (int i = 0; i < VPL; ++i) ok = ok && in_range(u[i]) && in_range(v[i]);
            if (__all_sync(kFull, ok)) {
                fold();
            } else {
#pragma unroll
                for (int i = 0; i < VPL; ++i) { u[i] = up[i]; v[i] = vp[i]; }
                fold();
                exact();
            }
#pragma unroll
            for (int i = 0; i < VPL; ++i) { up[i] = u[i]; vp[i] = v[i]; }
            continue;
        }
        if (t >= a.max_iters) return;
        float un[VPL], y[VPL];
#pragma unroll
        for (int i = 0; i < VPL; ++i) un[i] = rcp_fast(x[i]);
        uint32_t parts = kTolParts + 1u;
        if (TOL) {
            if (--until_check == 0) {
                until_check = a.check_every;
                uint32_t q = 0u;
#pragma unroll
                for (int i = 0; i < VPL; ++i) q += error_parts<VPL>(S[i] * fabsf(fmaf(u[i], x[i], -1.0f)), tol_scale);
                parts = __reduce_add_sync(kFull, counts ? q : 0u);
            }
        }
        half(false, un, y);
        float vn[VPL];
#pragma unroll
        for (int i = 0; i < VPL; ++i) vn[i] = rcp_fast(y[i]);
        if (TOL && parts <= kTolParts) return;    // iterate t meets the tolerance
        bool out = false;
#pragma unroll
        for (int i = 0; i < VPL; ++i) {
            up[i] = u[i]; vp[i] = v[i];
            u[i] = un[i]; v[i] = vn[i];
            out = out || !in_window(un[i]) || !in_window(vn[i]);
        }
        event = __any_sync(kFull, out);
        ++t;
    }
}

// relative row error of the result from its row sums, and the cap flag
template <int VPL>
__device__ __forceinline__ void finish(const SinkArgs& a, const bool counts, const double (&S)[VPL], const double sum_st,
                                       const float (&u)[VPL], const float (&x)[VPL], int t, Verdict* v)
{
    double e = 0.0;
#pragma unroll
    for (int i = 0; i < VPL; ++i) e += counts ? S[i] * (double)fabsf(fmaf(u[i], x[i], -1.0f)) : 0.0;
    e = warp_sum(e);
    if ((threadIdx.x & 31) == 0) {
        v->iters = t;
        v->row_err = sum_st > 0.0 ? (float)(e / sum_st) : 0.0f;
        if (a.tol > 0.0f && !(e <= (double)a.tol * sum_st)) v->info |= TAOT_INFO_SINKHORN_CAP;
    }
}

// =====================================================================================================================
// Dense kernel: at most 32 classes, any cost between them.  One class per lane (two classes: both in every lane, no
// exchange at all).  PPC problems per CTA, one warp each.

template <int NC, int VPL>
struct DenseSmem {
    double al[NC], be[NC], ls[NC], ld[NC];        // potentials and log masses by class
    float S[NC], D[NC], yc[NC];
    __align__(16) float x[2][32];                 // exchange buffers
    float E[NC][NC + 1];                          // e^(alpha + beta - C/eps)
};

// sum of m[b] * w_b over the NC classes of the other side, w in shared memory: 16-byte broadcast loads and packed
// multiply-adds in two chains (measured per iteration: 8 classes 138 cycles, 32 classes 237; the same gather by shuffles
// takes 190 and more than 1000)
template <int NC>
__device__ __forceinline__ float dot(const unsigned long long (&m)[NC / 2], const float* w)
{
    unsigned long long acc[2];
#pragma unroll
    for (int q = 0; q < NC / 4; ++q) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(w + 4 * q);
        if (q == 0) {
            asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(acc[0]) : "l"(m[0]), "l"(v.x));
            asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(acc[1]) : "l"(m[1]), "l"(v.y));
        } else {
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[0]) : "l"(m[2 * q]), "l"(v.x));
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[1]) : "l"(m[2 * q + 1]), "l"(v.y));
        }
    }
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[0]) : "l"(acc[1]));
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(acc[0]));
    return x + y;
}
__device__ __forceinline__ unsigned long long pack2(float x, float y)
{
    unsigned long long p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(x), "f"(y));
    return p;
}

template <int NC, int VPL, bool TOL, int PPC>
__global__ void __launch_bounds__(kThreads)
sinkhorn_class_kernel(ClassArgs k, int64_t nprob)
{
    constexpr int LPP = NC / VPL;                 // lanes that own classes; the others hold copies
    const SinkArgs& a = k.a;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int R = a.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t b0 = (int64_t)blockIdx.x * PPC;
    taot_await();
    if (blockIdx.x >= k.solvers) {
        zero_rows_of_batch(a, nprob, k.wide, (int64_t)(blockIdx.x - k.solvers) * (kThreads / 32) + warp,
                           (int64_t)(gridDim.x - k.solvers) * (kThreads / 32));
        return;
    }
    float* st = reinterpret_cast<float*>(smem_raw);                 // [PPC][R] supply; scaled at the end
    float* dm = st + PPC * R;                                       // [PPC][R] demand; at the end times the column cap
    uint16_t* cls = reinterpret_cast<uint16_t*>(dm + PPC * R);      // [R]
    uint16_t* list = cls + R;                                       // [R]
    __shared__ int32_t off[NC + 1];
    __shared__ DenseSmem<NC, VPL> sm[PPC];
    __shared__ double cost[NC * NC];               // over eps
    __shared__ double mS[PPC * NC], mD[PPC * NC];
    __shared__ Verdict ver[PPC];

    if (tid < PPC) { ver[tid].flags = 0; ver[tid].state = 1; }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PPC; ++p)
        if (b0 + p < nprob) load_masses(a, b0 + p, st + p * R, dm + p * R, &ver[p]);
    for (int i = tid; i < R; i += kThreads) { cls[i] = k.cls[i]; list[i] = k.list[i]; }
    for (int i = tid; i <= NC; i += kThreads) off[i] = k.off[i];
    for (int i = tid; i < NC * NC; i += kThreads) cost[i] = (double)k.cost[i] * a.inv_eps;
    __syncthreads();
    class_masses<PPC>(k, off, list, st, dm, R, NC, mS, mD, nprob - b0, ver);

    if (warp < PPC) {
        if (b0 + warp < nprob) {
            DenseSmem<NC, VPL>& m = sm[warp];
            const int slot0 = (lane % LPP) * VPL;
            const bool counts = lane < LPP;
            if (ver[warp].state == 0) {
                double S[VPL], D[VPL], sum_st = 0.0;
#pragma unroll
                for (int i = 0; i < VPL; ++i) {
                    S[i] = mS[warp * NC + slot0 + i]; D[i] = mD[warp * NC + slot0 + i];
                    sum_st += counts ? S[i] : 0.0;
                }
                sum_st = warp_sum(sum_st);
                unsigned long long Kr[VPL][NC / 2], Kc[VPL][NC / 2];       // pairs of entries
                float Sf[VPL], u[VPL], v[VPL], x[VPL];
#pragma unroll
                for (int i = 0; i < VPL; ++i) {
                    const int q = slot0 + i;
                    Sf[i] = (float)S[i];
                    u[i] = 1.0f; v[i] = 1.0f;
                    m.S[q] = Sf[i]; m.D[q] = (float)D[i];
                    m.ls[q] = S[i] > 0.0 ? log(S[i]) : -INFINITY;
                    m.ld[q] = D[i] > 0.0 ? log(D[i]) : -INFINITY;
                    m.al[q] = -k.lse0[q];                            // iteration 1, first half: v = 1 on every rank
                    m.be[q] = 0.0;
                }
                __syncwarp();
                // -log-sum-exp over the other side from its log masses and potentials: one exact half-step
                auto exact_half = [&](const bool rows) {
                    double res[VPL];
#pragma unroll
                    for (int i = 0; i < VPL; ++i) {
                        const int q = slot0 + i;
                        const double* lm = rows ? m.ld : m.ls;
                        const double* po = rows ? m.be : m.al;
                        double mx = -INFINITY;
                        for (int j = 0; j < NC; ++j)
                            mx = fmax(mx, lm[j] + po[j] - cost[rows ? q * NC + j : j * NC + q]);
                        double acc = 0.0;
                        for (int j = 0; j < NC; ++j) {
                            const double e = lm[j] + po[j] - cost[rows ? q * NC + j : j * NC + q];
                            if (e > -INFINITY) acc += (double)exp_split(e - mx);
                        }
                        res[i] = -(mx + log(acc));
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < VPL; ++i) {
                        if (rows) { if (S[i] > 0.0) m.al[slot0 + i] = res[i]; }
                        else if (D[i] > 0.0) m.be[slot0 + i] = res[i];
                    }
                    __syncwarp();
                };
                auto rebuild = [&]() {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < VPL; ++i) {
                        const int q = slot0 + i;
                        const double al = m.al[q];
#pragma unroll 8
                        for (int j = 0; j < NC; ++j) {
                            const float e = exp_split(al + m.be[j] - cost[q * NC + j]);
                            m.E[q][j] = (S[i] > 0.0 && m.D[j] > 0.0f) ? e : 0.0f;
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < VPL; ++i)
#pragma unroll
                        for (int j = 0; j < NC; j += 2) {
                            // a class without supply (demand) copies its other factor: 1 / v, which no sum takes in
                            const int q = slot0 + i;
                            const float r0 = S[i] > 0.0 ? m.E[q][j] * m.D[j] : (j == q ? 1.0f : 0.0f);
                            const float r1 = S[i] > 0.0 ? m.E[q][j + 1] * m.D[j + 1] : (j + 1 == q ? 1.0f : 0.0f);
                            const float c0 = D[i] > 0.0 ? m.E[j][q] * m.S[j] : (j == q ? 1.0f : 0.0f);
                            const float c1 = D[i] > 0.0 ? m.E[j + 1][q] * m.S[j + 1] : (j + 1 == q ? 1.0f : 0.0f);
                            Kr[i][j / 2] = pack2(r0, r1);
                            Kc[i][j / 2] = pack2(c0, c1);
                        }
                };
                auto fold = [&]() {
#pragma unroll
                    for (int i = 0; i < VPL; ++i) {
                        // (the lanes that hold copies of a class hold the same factors; one of them adds)
                        if (counts && S[i] > 0.0) m.al[slot0 + i] += log_factor(u[i]);
                        if (counts && D[i] > 0.0) m.be[slot0 + i] += log_factor(v[i]);
                        u[i] = 1.0f; v[i] = 1.0f;
                    }
                    rebuild();
                };
                auto exact = [&]() { exact_half(true); exact_half(false); rebuild(); };
                int buf = 0;
                auto half = [&](const bool rows, const float (&w)[VPL], float (&out)[VPL]) {
                    if constexpr (VPL == 2 && NC == 2) {                  // both classes in every lane: no exchange
#pragma unroll
                        for (int i = 0; i < VPL; ++i) {
                            float m0, m1;
                            asm("mov.b64 {%0, %1}, %2;" : "=f"(m0), "=f"(m1) : "l"(rows ? Kr[i][0] : Kc[i][0]));
                            out[i] = fmaf(m1, w[1], m0 * w[0]);
                        }
                    } else {
                        float* x = m.x[buf];
                        buf ^= 1;
                        x[lane] = w[0];                                   // (copies write behind the classes)
                        __syncwarp();
                        out[0] = rows ? dot<NC>(Kr[0], x) : dot<NC>(Kc[0], x);
                    }
                };
                exact_half(false);                                    // iteration 1, second half
                rebuild();
                int t;
                iterate<VPL, TOL>(a, counts, Sf, (float)((double)kTolParts / ((double)a.tol * sum_st)), u, v, x, t, half, fold, exact);
                finish<VPL>(a, counts, S, sum_st, u, x, t, &ver[warp]);
                // the plan is written from fp64 potentials: E anew, and the column sums of E for the cap
                fold();
#pragma unroll
                for (int i = 0; i < VPL; ++i) {
                    float y = 0.0f;
                    for (int j = 0; j < NC; ++j) y = fmaf(m.E[j][slot0 + i], m.S[j], y);
                    m.yc[slot0 + i] = y;
                }
            }
        }
    } else if (gridDim.x == k.solvers) {
        for (int p = 0; p < PPC; ++p)
            if (b0 + p < nprob)
                zero_rows(a.plan + (b0 + p) * (int64_t)R * R, st + p * R, R, k.wide, warp - PPC, kThreads / 32 - PPC);
    }
    __syncthreads();

    // ---- column cap: T_ij *= min(1, d_j / (colsum_j + eps0)), colsum_j = d_j * (column sum of E over the supply)
    for (int i = tid; i < PPC * R; i += kThreads) {
        const int p = i / R, j = i - p * R;
        if (b0 + p < nprob && ver[p].state == 0) {
            const float d = dm[i], sv = st[i];
            if (sv > 0.0f) st[i] = fmaxf((float)(ver[p].gamma * (double)sv), 1.17549435e-38f);
            dm[i] = d * (float)fmin(1.0, (double)d / ((double)d * (double)sm[p].yc[cls[j]] + (double)a.eps0));
        }
    }
    __syncthreads();
    int nonfinite = 0;
    for (int p = 0; p < PPC; ++p) {
        if (b0 + p >= nprob || ver[p].state == 2) continue;
        const bool solved = ver[p].state == 0;
        float* out = a.plan + (b0 + p) * (int64_t)R * R;
        const float* dp = dm + p * R;
        for (int row = warp; row < R; row += kThreads / 32) {
            const float sv = st[p * R + row];
            if (!(sv > 0.0f)) continue;
            float* o = out + (int64_t)row * R;
            const float si = solved ? sv : 0.0f;
            const float* er = sm[p].E[cls[row]];
            if (k.wide) {
#pragma unroll 2
                for (int j = lane * 4; j < R; j += 128) {
                    const float4 d4 = *reinterpret_cast<const float4*>(dp + j);
                    const ushort4 c4 = *reinterpret_cast<const ushort4*>(cls + j);
                    float4 w = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (solved) w = make_float4(si * (er[c4.x] * d4.x), si * (er[c4.y] * d4.y), si * (er[c4.z] * d4.z), si * (er[c4.w] * d4.w));
                    if (!isfinite((w.x + w.y) + (w.z + w.w))) nonfinite |= 1 << p;
                    *reinterpret_cast<float4*>(o + j) = w;
                }
            } else {
                for (int j = lane; j < R; j += 32) {
                    const float w = solved ? si * (er[cls[j]] * dp[j]) : 0.0f;
                    if (!isfinite(w)) nonfinite |= 1 << p;
                    o[j] = w;
                }
            }
        }
    }
    if (nonfinite) {
#pragma unroll
        for (int p = 0; p < PPC; ++p)
            if ((nonfinite >> p) & 1) atomicOr(&ver[p].info, TAOT_INFO_NONFINITE);
    }
    __syncthreads();
    if (tid < PPC && b0 + tid < nprob) {
        const Verdict& v = ver[tid];
        a.iters[b0 + tid] = v.state == 2 ? kHandBack : v.iters;
        if (v.state != 2) {
            a.row_err[b0 + tid] = v.row_err;
            if (v.info) atomicOr(a.info + b0 + tid, v.info);
        }
    }
}

// =====================================================================================================================
// Tree kernel: more than 32 classes, a cost with three tiers between them (inside a class c1, inside a group of classes
// c2, elsewhere c3; c2 = c3 if there is no group tier).  A lane holds GPL groups of up to NPG classes, so class and
// group sums are lane-local and one exchange of 32 lane totals completes a half-step:
//     x_n = kA_n v_n + kB_n G_g(n) + k3_n T,   G_g = sum over the classes of g of q_m v_m,   T = sum of F_g G_g,
//     q_n = e^(beta_n - m_g) D_n,  m_g = max beta in g,  F_g = e^(m_g - m),  m = max m_g,
//     kA = A1 - A2 q,  kB = A2 - A3 F,  k3 = A3,
//     A1 = e^(alpha + beta - c1) D,  A2 = e^(alpha - c2 + m_g),  A3 = e^(alpha - c3 + m)
// (column sums the same with the sides exchanged).  A1 >= A2 q e^(c2 - c1) and A2 >= A3 F e^(c3 - c2): the differences
// lose nothing that counts in the row sum.

template <int NS>
struct TreeSmem {
    double al[NS], be[NS];
    float S[NS], D[NS];
    float e1[NS], e2[NS], e3[NS], q[NS], Q[NS], yc[NS];    // what the plan's entries are products of
    float p[NS], b2[NS], b3[NS];
    __align__(16) float x[2][32];
};

// sum of one value per lane, the same bits in every lane (packed additions)
__device__ __forceinline__ float exchange_sum(float p, float* buf)
{
    buf[threadIdx.x & 31] = p;
    __syncwarp();
    unsigned long long t[16];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(buf + 4 * q);
        t[2 * q] = v.x; t[2 * q + 1] = v.y;
    }
#pragma unroll
    for (int w = 8; w > 0; w >>= 1)
#pragma unroll
        for (int q = 0; q < w; ++q) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(t[q]) : "l"(t[q + w]));
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(t[0]));
    return x + y;
}

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ float exp_or_zero(double x) { return x == -INFINITY ? 0.0f : exp_split(x); }

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// the same word of the shared memory of the cluster's first CTA
__device__ __forceinline__ float leader_f32(const float* p)
{
    uint32_t at;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
    return v;
}

template <int GPL, int NPG, bool TOL, int PPC>
__global__ void __launch_bounds__(kThreads)
sinkhorn_class_tree_kernel(ClassArgs k, int64_t nprob)
{
    constexpr int NPL = GPL * NPG, NS = 32 * NPL;
    const SinkArgs& a = k.a;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int R = a.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // PPC == 1: the problem's CTA may lead a cluster (k.cluster CTAs): the others write the rows without supply meanwhile
    // and, once it is solved, their share of the supply rows, from factors they fetch from the leader
    const int crank = PPC == 1 ? (int)(blockIdx.x % k.cluster) : 0, csize = PPC == 1 ? (int)k.cluster : 1;
    const int64_t b0 = (int64_t)blockIdx.x / csize * PPC;
    taot_await();
    if (blockIdx.x >= k.solvers) {
        zero_rows_of_batch(a, nprob, k.wide, (int64_t)(blockIdx.x - k.solvers) * (kThreads / 32) + warp,
                           (int64_t)(gridDim.x - k.solvers) * (kThreads / 32));
        return;
    }
    TreeSmem<NS>* sm = reinterpret_cast<TreeSmem<NS>*>(smem_raw);   // [PPC]
    double* mS = reinterpret_cast<double*>(sm + PPC);               // [PPC][NS] masses by class
    double* mD = mS + PPC * NS;
    float* st = reinterpret_cast<float*>(mD + PPC * NS);            // [PPC][R] supply; scaled at the end
    float* dm = st + PPC * R;                                       // [PPC][3][R] demand; at the end the column factors by tier
    uint16_t* cls = reinterpret_cast<uint16_t*>(dm + 3 * PPC * R);  // [R]
    uint16_t* list = cls + R;                                       // [R]
    __shared__ int32_t off[NS + 1];
    __shared__ Verdict ver[PPC];

    if (tid < PPC) { ver[tid].flags = 0; ver[tid].state = 1; ver[tid].info = 0; }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PPC; ++p)
        if (b0 + p < nprob) load_masses(a, b0 + p, st + p * R, dm + 3 * p * R, &ver[p]);
    for (int i = tid; i < R; i += kThreads) { cls[i] = k.cls[i]; list[i] = k.list[i]; }
    for (int i = tid; i <= NS; i += kThreads) off[i] = k.off[i];
    __syncthreads();
    if (crank == 0) class_masses<PPC>(k, off, list, st, dm, 3 * R, NS, mS, mD, nprob - b0, ver);

    if (crank > 0) {
        zero_rows(a.plan + b0 * (int64_t)R * R, st, R, k.wide, (crank - 1) * (kThreads / 32) + warp, (csize - 1) * (kThreads / 32));
    } else if (warp < PPC) {
        if (b0 + warp < nprob) {
            TreeSmem<NS>& m = sm[warp];
            const int slot0 = lane * NPL;
            if (ver[warp].state == 0) {
                double S[NPL], D[NPL], sum_st = 0.0;
#pragma unroll
                for (int i = 0; i < NPL; ++i) {
                    S[i] = mS[warp * NS + slot0 + i]; D[i] = mD[warp * NS + slot0 + i];
                    sum_st += S[i];
                }
                sum_st = warp_sum(sum_st);
                float Sf[NPL], u[NPL], v[NPL], x[NPL];
                float rA[NPL], rB[NPL], r3[NPL], rq[NPL], cA[NPL], cB[NPL], c3[NPL], cq[NPL], rF[GPL], cF[GPL];
                unsigned hot = 0u, cold = 0u;
#pragma unroll
                for (int i = 0; i < NPL; ++i) {
                    const int q = slot0 + i;
                    Sf[i] = (float)S[i];
                    m.S[q] = Sf[i]; m.D[q] = (float)D[i];
                    hot |= (S[i] > 0.0 ? 1u : 0u) << i;
                    cold |= (D[i] > 0.0 ? 1u : 0u) << i;
                    m.al[q] = -k.lse0[q];
                    m.be[q] = 0.0;
                    u[i] = 1.0f; v[i] = 1.0f;
                }
                __syncwarp();
                // one half-step in the log domain, by tiers (each lane only reads and writes its own slots)
                auto exact_half = [&](const bool rows) {
                    const unsigned src = rows ? cold : hot, dst = rows ? hot : cold;
                    // (exponentials as fp32 factors of an exact fp64 scale, and no branch around any of them: with fp64 exp
                    // behind branches a half-step took 5 us)
                    double lt[NPL], gm[GPL], gs[GPL];       // log terms of the other side, their group maxima and sums
                    float F[GPL];
                    double tm = -INFINITY;
#pragma unroll
                    for (int i = 0; i < NPL; ++i) {
                        const bool on = (src >> i) & 1u;
                        const double l = log(on ? (double)(rows ? m.D[slot0 + i] : m.S[slot0 + i]) : 1.0) + (rows ? m.be[slot0 + i] : m.al[slot0 + i]);
                        lt[i] = on ? l : -INFINITY;
                    }
#pragma unroll
                    for (int g = 0; g < GPL; ++g) {
                        gm[g] = -INFINITY; gs[g] = 0.0;
#pragma unroll
                        for (int n = 0; n < NPG; ++n) gm[g] = fmax(gm[g], lt[g * NPG + n]);
                        const double base = gm[g] > -INFINITY ? gm[g] : 0.0;
#pragma unroll
                        for (int n = 0; n < NPG; ++n) {
                            const float w = exp_or_zero(lt[g * NPG + n] - base);
                            m.e1[slot0 + g * NPG + n] = w;
                            gs[g] += (double)w;
                        }
                        tm = fmax(tm, gm[g]);
                    }
                    tm = warp_max(tm);
                    const double tbase = tm > -INFINITY ? tm : 0.0;
                    double ts = 0.0;
#pragma unroll
                    for (int g = 0; g < GPL; ++g) {
                        F[g] = exp_or_zero(gm[g] - tbase);
                        ts += (double)F[g] * gs[g];
                    }
                    ts = warp_sum(ts);
#pragma unroll 1
                    for (int i = 0; i < NPL; ++i) {
                        const int g = i / NPG;
                        double own = lt[0], gmi = gm[0], gsi = gs[0];
                        float Fi = F[0];
#pragma unroll
                        for (int j = 1; j < NPL; ++j) own = j == i ? lt[j] : own;
#pragma unroll
                        for (int j = 1; j < GPL; ++j)
                            if (j == g) { gmi = gm[j]; gsi = gs[j]; Fi = F[j]; }
                        double grp = 0.0;
#pragma unroll
                        for (int n = 0; n < NPG; ++n) grp += g * NPG + n != i ? (double)m.e1[slot0 + g * NPG + n] : 0.0;
                        const double rest = ts - (double)Fi * gsi;
                        const double l1 = own - k.c1;
                        const double g2 = log(grp > 0.0 ? grp : 1.0), g3 = log(rest > 0.0 ? rest : 1.0);
                        const double l2 = grp > 0.0 ? gmi + g2 - k.c2 : -INFINITY;
                        const double l3 = rest > 0.0 ? tm + g3 - k.c3 : -INFINITY;
                        const double mx = fmax(l1, fmax(l2, l3)), base = mx > -INFINITY ? mx : 0.0;
                        const double sum = (double)exp_or_zero(l1 - base) + (double)exp_or_zero(l2 - base) + (double)exp_or_zero(l3 - base);
                        const double res = -(mx + log(sum > 0.0 ? sum : 1.0));
                        if ((dst >> i) & 1u) (rows ? m.al : m.be)[slot0 + i] = res;
                    }
                    __syncwarp();
                };
                auto rebuild = [&]() {
                    double m2[GPL], p2[GPL], m3 = -INFINITY, p3 = -INFINITY;
#pragma unroll
                    for (int g = 0; g < GPL; ++g) {
                        m2[g] = -INFINITY; p2[g] = -INFINITY;
#pragma unroll
                        for (int n = 0; n < NPG; ++n) {
                            const int i = g * NPG + n;
                            if ((cold >> i) & 1u) m2[g] = fmax(m2[g], m.be[slot0 + i]);
                            if ((hot >> i) & 1u) p2[g] = fmax(p2[g], m.al[slot0 + i]);
                        }
                        m3 = fmax(m3, m2[g]); p3 = fmax(p3, p2[g]);
                    }
                    m3 = warp_max(m3); p3 = warp_max(p3);
#pragma unroll
                    for (int g = 0; g < GPL; ++g) {
                        rF[g] = exp_or_zero(m2[g] == -INFINITY ? -INFINITY : m2[g] - m3);
                        cF[g] = exp_or_zero(p2[g] == -INFINITY ? -INFINITY : p2[g] - p3);
                    }
                    // (a rolled loop: the code runs a few times per solve, and fetching it unrolled costs more than it saves)
#pragma unroll 1
                    for (int i = 0; i < NPL; ++i) {
                        const int s = slot0 + i;
                        double mg = m2[0], pg = p2[0];
                        float Fg = rF[0];
#pragma unroll
                        for (int g = 1; g < GPL; ++g)
                            if (i / NPG == g) { mg = m2[g]; pg = p2[g]; Fg = rF[g]; }
                        const bool ish = (hot >> i) & 1u, isc = (cold >> i) & 1u;
                        const bool gc = mg > -INFINITY, gh = pg > -INFINITY;
                        mg = gc ? mg : 0.0; pg = gh ? pg : 0.0;
                        const double al = m.al[s], be = m.be[s];
                        // (eight exponentials side by side, then the selection: behind branches they would run one by one)
                        const float x0 = exp_split(be - mg), x1 = exp_split(al - pg), x2 = exp_split(al + be - k.c1),
                                    x3 = exp_split(al - k.c2 + mg), x4 = exp_split(al - k.c3 + m3),
                                    x5 = exp_split(be - k.c2 + pg), x6 = exp_split(be - k.c3 + p3);
                        m.q[s] = isc ? x0 : 0.0f;
                        m.Q[s] = isc ? x0 * Fg : 0.0f;
                        m.p[s] = ish ? x1 : 0.0f;
                        m.e1[s] = ish && isc ? x2 : 0.0f;
                        m.e2[s] = ish && gc ? x3 : 0.0f;
                        m.e3[s] = ish ? x4 : 0.0f;
                        m.b2[s] = isc && gh ? x5 : 0.0f;
                        m.b3[s] = isc ? x6 : 0.0f;
                    }
                    // a class without supply (demand) copies its other factor: 1 / v, which no sum takes in
#pragma unroll
                    for (int i = 0; i < NPL; ++i) {
                        const int s = slot0 + i, g = i / NPG;
                        rq[i] = m.q[s] * m.D[s]; cq[i] = m.p[s] * m.S[s];
                        const float a2 = m.e2[s], a3 = m.e3[s], b2 = m.b2[s], b3 = m.b3[s];
                        rA[i] = ((hot >> i) & 1u) ? fmaf(-a2, rq[i], m.e1[s] * m.D[s]) : 1.0f;
                        cA[i] = ((cold >> i) & 1u) ? fmaf(-b2, cq[i], m.e1[s] * m.S[s]) : 1.0f;
                        rB[i] = fmaf(-a3, rF[g], a2); r3[i] = a3;
                        cB[i] = fmaf(-b3, cF[g], b2); c3[i] = b3;
                    }
                };
                auto fold = [&]() {
#pragma unroll
                    for (int i = 0; i < NPL; ++i) { m.e1[slot0 + i] = u[i]; m.e2[slot0 + i] = v[i]; u[i] = 1.0f; v[i] = 1.0f; }
#pragma unroll 1
                    for (int s = slot0; s < slot0 + NPL; ++s) {
                        if (m.S[s] > 0.0f) m.al[s] += log_factor(m.e1[s]);
                        if (m.D[s] > 0.0f) m.be[s] += log_factor(m.e2[s]);
                    }
                    rebuild();
                };
                auto exact = [&]() { exact_half(true); exact_half(false); rebuild(); };
                int buf = 0;
                auto half = [&](const bool rows, const float (&w)[NPL], float (&out)[NPL]) {
                    float p = 0.0f;
#pragma unroll
                    for (int g = 0; g < GPL; ++g) {
                        float t[NPG];
#pragma unroll
                        for (int n = 0; n < NPG; ++n) t[n] = (rows ? rq[g * NPG + n] : cq[g * NPG + n]) * w[g * NPG + n];
#pragma unroll
                        for (int h = NPG / 2; h > 0; h >>= 1)
#pragma unroll
                            for (int n = 0; n < h; ++n) t[n] += t[n + h];
                        p = g == 0 ? (rows ? rF[0] : cF[0]) * t[0] : fmaf(rows ? rF[g] : cF[g], t[0], p);
#pragma unroll
                        for (int n = 0; n < NPG; ++n) {
                            const int i = g * NPG + n;
                            out[i] = fmaf(rows ? rA[i] : cA[i], w[i], (rows ? rB[i] : cB[i]) * t[0]);
                        }
                    }
                    const float T = exchange_sum(p, m.x[buf]);
                    buf ^= 1;
#pragma unroll
                    for (int i = 0; i < NPL; ++i) out[i] = fmaf(rows ? r3[i] : c3[i], T, out[i]);
                };
                exact_half(false);                                    // iteration 1, second half
                rebuild();
                int t;
                iterate<NPL, TOL>(a, true, Sf, (float)((double)kTolParts / ((double)a.tol * sum_st)), u, v, x, t, half, fold, exact);
                finish<NPL>(a, true, S, sum_st, u, x, t, &ver[warp]);
                fold();
                half(false, u, x);                                    // column sums of the plan's own factors (u = 1)
#pragma unroll
                for (int i = 0; i < NPL; ++i) m.yc[slot0 + i] = x[i];
            }
        }
    } else if (gridDim.x == k.solvers && csize == 1) {
        for (int p = 0; p < PPC; ++p)
            if (b0 + p < nprob)
                zero_rows(a.plan + (b0 + p) * (int64_t)R * R, st + p * R, R, k.wide, warp - PPC, kThreads / 32 - PPC);
    }
    __syncthreads();

    // ---- column cap, then the factors of a column by tier
    for (int i = tid; crank == 0 && i < PPC * R; i += kThreads) {
        const int p = i / R, j = i - p * R;
        if (b0 + p < nprob && ver[p].state == 0) {
            const int c = cls[j];
            float* col = dm + 3 * p * R + j;
            const float d = col[0], sv = st[i];
            if (sv > 0.0f) st[i] = fmaxf((float)(ver[p].gamma * (double)sv), 1.17549435e-38f);
            const float w = d * (float)fmin(1.0, (double)d / ((double)d * (double)sm[p].yc[c] + (double)a.eps0));
            col[0] = w; col[R] = w * sm[p].q[c]; col[2 * R] = w * sm[p].Q[c];
        }
    }
    __syncthreads();
    if (csize > 1) {
        cluster_arrive(); cluster_wait();                               // the leader's factors are there
        if (crank > 0) {
            for (int i = tid; i < 4 * R; i += kThreads) st[i] = leader_f32(st + i);      // st, then dm
            for (int i = tid; i < 3 * NS; i += kThreads) sm[0].e1[i] = leader_f32(sm[0].e1 + i);
            if (tid == 0) ver[0].state = __float_as_int(leader_f32(reinterpret_cast<const float*>(&ver[0].state)));
        }
        __syncthreads();
        cluster_arrive();                                               // (the leader must not go before they are read)
    }
    int nonfinite = 0;
    for (int p = 0; p < PPC; ++p) {
        if (b0 + p >= nprob || ver[p].state == 2) continue;
        const bool solved = ver[p].state == 0;
        float* out = a.plan + (b0 + p) * (int64_t)R * R;
        const float* col = dm + 3 * p * R;
        for (int row = crank * (kThreads / 32) + warp; row < R; row += csize * (kThreads / 32)) {
            const float sv = st[p * R + row];
            if (!(sv > 0.0f)) continue;
            float* o = out + (int64_t)row * R;
            const int c = cls[row], g = c / NPG;
            const float si = solved ? sv : 0.0f;
            const float f1 = si * sm[p].e1[c], f2 = si * sm[p].e2[c], f3 = solved ? si * sm[p].e3[c] : 0.0f;
            bool fine = true;
            // the far tier for all columns, then the columns of the row's own group again
            if (k.wide) {
#pragma unroll 4
                for (int j = lane * 4; j < R; j += 128) {
                    const float4 q4 = *reinterpret_cast<const float4*>(col + 2 * R + j);
                    const float4 w = solved ? make_float4(f3 * q4.x, f3 * q4.y, f3 * q4.z, f3 * q4.w) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    fine = fine && isfinite((w.x + w.y) + (w.z + w.w));
                    *reinterpret_cast<float4*>(o + j) = w;
                }
            } else {
                for (int j = lane; j < R; j += 32) {
                    const float w = solved ? f3 * col[2 * R + j] : 0.0f;
                    fine = fine && isfinite(w);
                    o[j] = w;
                }
            }
            __syncwarp();
            if (solved)
                for (int q = off[g * NPG] + lane; q < off[(g + 1) * NPG]; q += 32) {
                    const int j = list[q];
                    const float w = cls[j] == c ? f1 * col[j] : f2 * col[R + j];
                    fine = fine && isfinite(w);
                    o[j] = w;
                }
            if (!fine) nonfinite |= 1 << p;
        }
    }
    if (nonfinite) {
#pragma unroll
        for (int p = 0; p < PPC; ++p)
            if ((nonfinite >> p) & 1) atomicOr(&ver[p].info, TAOT_INFO_NONFINITE);
    }
    if (csize > 1) cluster_wait();
    __syncthreads();
    if (crank > 0) {
        if (tid == 0 && (ver[0].info & TAOT_INFO_NONFINITE)) atomicOr(a.info + b0, TAOT_INFO_NONFINITE);
    } else if (tid < PPC && b0 + tid < nprob) {
        const Verdict& v = ver[tid];
        a.iters[b0 + tid] = v.state == 2 ? kHandBack : v.iters;
        if (v.state != 2) {
            a.row_err[b0 + tid] = v.row_err;
            if (v.info) atomicOr(a.info + b0 + tid, v.info);
        }
    }
}

template <int NC, int VPL, bool TOL, int PPC>
int launch_dense(const ClassArgs& k, int32_t B, int32_t zeroers, cudaStream_t st)
{
    const size_t smem = (size_t)k.a.R * (PPC * 2 * sizeof(float) + 2 * sizeof(uint16_t));
    TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_class_kernel<NC, VPL, TOL, PPC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    TAOT_CUDA_OK(taot_launch_chained(sinkhorn_class_kernel<NC, VPL, TOL, PPC>, (unsigned)(k.solvers + zeroers), kThreads, smem, st, k, (int64_t)B));
    return 1;
}

template <int GPL, int NPG, bool TOL, int PPC>
int launch_tree(ClassArgs& k, int32_t B, int32_t zeroers, int32_t cluster, cudaStream_t st)
{
    size_t smem = PPC * (sizeof(TreeSmem<32 * GPL * NPG>) + 2 * sizeof(double) * 32 * GPL * NPG) + (size_t)k.a.R * (PPC * 4 * sizeof(float) + 2 * sizeof(uint16_t));
    k.cluster = PPC == 1 ? cluster : 1;
    if (k.cluster > 1) {
        k.solvers = B * k.cluster;
        zeroers = 0;
        if (smem < 120 * 1024) smem = 120 * 1024;              // one CTA per SM: a solving SM's stores slow its exchanges down
    }
    TAOT_CUDA_OK(cudaFuncSetAttribute(sinkhorn_class_tree_kernel<GPL, NPG, TOL, PPC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    TAOT_CUDA_OK(taot_launch_chained_cluster(sinkhorn_class_tree_kernel<GPL, NPG, TOL, PPC>, (unsigned)(k.solvers + zeroers), kThreads,
                                             (unsigned)k.cluster, smem, st, k, (int64_t)B));
    return 1;
}

template <bool TOL, int PPC>
int launch_kind(const taot_handle_s* h, ClassArgs& k, int32_t B, int32_t zeroers, int32_t cluster, cudaStream_t st)
{
    k.solvers = (B + PPC - 1) / PPC;
    if (h->cls_kind == 1) {
        switch (h->cls_nc) {
            case 2: return launch_dense<2, 2, TOL, PPC>(k, B, zeroers, st);
            case 4: return launch_dense<4, 1, TOL, PPC>(k, B, zeroers, st);
            case 8: return launch_dense<8, 1, TOL, PPC>(k, B, zeroers, st);
            case 16: return launch_dense<16, 1, TOL, PPC>(k, B, zeroers, st);
            default: return launch_dense<32, 1, TOL, PPC>(k, B, zeroers, st);
        }
    }
    if (h->cls_npg == 8) return launch_tree<1, 8, TOL, PPC>(k, B, zeroers, cluster, st);
    switch (h->cls_gpl) {
        case 1: return launch_tree<1, 4, TOL, PPC>(k, B, zeroers, cluster, st);
        case 2: return launch_tree<2, 4, TOL, PPC>(k, B, zeroers, cluster, st);
        default: return launch_tree<4, 4, TOL, PPC>(k, B, zeroers, cluster, st);
    }
}

}  // namespace

// Launches the class kernels if the handle's cost has classes they hold (taot_build_classes); returns the number of
// kernels launched, 0 if there are none.  Problems with a rank that has both supply and demand come back marked.
int taot_launch_sinkhorn_class(taot_handle_t h, const SinkArgs& a, int32_t B, cudaStream_t st)
{
    if (!h->cls_kind) return 0;
    ClassArgs k;
    k.a = a;
    k.cls = h->d_cls; k.off = h->d_cls_off; k.list = h->d_cls_list; k.lse0 = h->d_cls_lse0; k.cost = h->d_cls_cost;
    k.c1 = (double)h->cls_tier[0] * a.inv_eps;
    k.c2 = (double)h->cls_tier[1] * a.inv_eps;
    k.c3 = (double)h->cls_tier[2] * a.inv_eps;
    k.wide = (a.R % 4 == 0 && (reinterpret_cast<uintptr_t>(a.plan) & 15) == 0) ? 1 : 0;
    // A problem alone on an SM has one warp that iterates and seven that write; from two problems per SM on, four of
    // them share a CTA, so that their warps sit on the SM's four schedulers instead of all on the first
    const bool share = B >= 2 * h->sm_count;
    // While SMs are left over they write the rows without supply (a solving SM's own stores slow its exchanges down);
    // otherwise the writing warps of the solving CTAs do
    const int32_t left = h->sm_count - B;
    const int32_t zeroers = left > 0 && (int64_t)B * a.R * a.R >= (1 << 20) ? 2 * left : 0;
    // The supply rows can only be written when their problem is solved, and one SM stores about 60 GB/s: from plans of 1 MB on
    // (512 ranks: 5 us and more) a problem takes a cluster of as many SMs as there are for each, 2, 4 or 8 (some less than
    // sm_count / B, since a cluster sits in one GPC)
    const int32_t per = h->sm_count / (B > 0 ? B : 1);
    const int32_t cluster = h->cls_kind == 2 && (int64_t)a.R * a.R >= (1 << 18) && per >= 2 ? (per >= 10 ? 8 : (per >= 5 ? 4 : 2)) : 1;
    if (a.tol > 0.0f) return share ? launch_kind<true, 4>(h, k, B, zeroers, cluster, st) : launch_kind<true, 1>(h, k, B, zeroers, cluster, st);
    return share ? launch_kind<false, 4>(h, k, B, zeroers, cluster, st) : launch_kind<false, 1>(h, k, B, zeroers, cluster, st);
}

namespace {

// ranks i and b are interchangeable: equal costs to and from every other rank, both ways between the two, on the diagonal
bool same_class(const float* C, int R, int i, int b, bool symmetric)
{
    auto at = [&](int x, int y) { return C[(size_t)x * R + y]; };
    if (at(i, i) != at(b, b) || at(i, b) != at(b, i)) return false;
    for (int q = 1; q < R; ++q) {                  // from the rank after b: a rank of another node differs at once
        const int j = b + q < R ? b + q : b + q - R;
        if (j == i) continue;
        if (at(i, j) != at(b, j)) return false;
        if (!symmetric && at(j, i) != at(j, b)) return false;
    }
    return true;
}

}  // namespace

// Classes of interchangeable ranks of the handle's cost, and the kernel that holds them: at most 32 classes the dense
// one; more, if the cost between classes has the three tiers of the tree kernel, that one; otherwise none.  `rep` receives for
// every rank the first rank of its class (itself where no kernel applies).
void taot_build_classes(taot_class_plan* out, const float* C, int R)
{
    out->kind = 0;
    out->rep.resize(R);
    for (int i = 0; i < R; ++i) out->rep[i] = i;
    bool symmetric = true;
    for (int i = 0; i < R && symmetric; ++i)
        for (int j = 0; j < i; ++j)
            if (C[(size_t)i * R + j] != C[(size_t)j * R + i]) { symmetric = false; break; }
    // What the ranks of a class have in common at a glance: the entries of their row and column, in whatever order
    std::vector<uint64_t> key(R, 0);
    for (int i = 0; i < R; ++i) {
        uint64_t row = 0;
        for (int j = 0; j < R; ++j) {
            uint32_t bits;
            std::memcpy(&bits, C + (size_t)i * R + j, 4);
            uint64_t x = (bits + 1) * 0x9E3779B97F4A7C15ull;
            x ^= x >> 29;
            row += x * 0xBF58476D1CE4E5B9ull;
            key[j] += x * 0x94D049BB133111EBull;
        }
        key[i] += row;
    }
    std::vector<int> reps, of(R);
    const size_t most = R <= 64 ? 32 : (size_t)R / 2;              // fewer than two ranks a class: nothing to gain
    for (int i = 0; i < R; ++i) {
        int c = -1;
        // neighbours first: the class of the rank before is the likely one
        if (i > 0 && key[i] == key[reps[of[i - 1]]] && same_class(C, R, i, reps[of[i - 1]], symmetric)) c = of[i - 1];
        for (size_t q = 0; q < reps.size() && c < 0; ++q)
            if (key[i] == key[reps[q]] && same_class(C, R, i, reps[q], symmetric)) c = (int)q;
        if (c < 0) {
            if (reps.size() == most) return;
            c = (int)reps.size();
            reps.push_back(i);
        }
        of[i] = c;
    }
    const int n = (int)reps.size();
    std::vector<int> size(n, 0), second(n, -1);                    // a second member of each class
    for (int i = 0; i < R; ++i) { if (size[of[i]]++ == 1) second[of[i]] = i; }
    auto cost = [&](int x, int y) {
        return x != y ? C[(size_t)reps[x] * R + reps[y]] : (second[x] >= 0 ? C[(size_t)reps[x] * R + second[x]] : 0.0f);
    };
    std::vector<int> slot(n);
    int slots;
    if (n <= 32) {
        out->kind = 1;
        out->nc = n <= 2 ? 2 : (n <= 4 ? 4 : (n <= 8 ? 8 : (n <= 16 ? 16 : 32)));
        slots = out->nc;
        for (int c = 0; c < n; ++c) slot[c] = c;
        out->cost.assign((size_t)slots * slots, 0.0f);
        for (int x = 0; x < n; ++x)
            for (int y = 0; y < n; ++y) out->cost[(size_t)x * slots + y] = cost(x, y);
    } else {
        // three tiers?  c1: inside the classes; c2 <= c3: between them
        float c1 = -1.0f, lo = INFINITY, hi = -1.0f;
        for (int x = 0; x < n; ++x) {
            if (second[x] >= 0) {
                if (c1 < 0.0f) c1 = cost(x, x);
                if (cost(x, x) != c1) return;
            }
            for (int y = 0; y < n; ++y)
                if (x != y) { lo = std::min(lo, cost(x, y)); hi = std::max(hi, cost(x, y)); }
        }
        if (c1 < 0.0f) c1 = lo;
        if (c1 > lo) return;
        std::vector<int> group(n, -1);
        std::vector<std::vector<int>> groups;
        for (int x = 0; x < n; ++x) {
            if (group[x] >= 0) continue;
            if (lo == hi && !groups.empty() && groups.back().size() < 4) {       // no group tier: any grouping will do
                group[x] = (int)groups.size() - 1;
                groups.back().push_back(x);
                continue;
            }
            group[x] = (int)groups.size();
            groups.push_back({x});
            for (int y = x + 1; y < n && lo != hi; ++y)
                if (group[y] < 0 && cost(x, y) == lo) { group[y] = group[x]; groups.back().push_back(y); }
        }
        size_t largest = 0;
        for (const auto& g : groups) largest = std::max(largest, g.size());
        for (int x = 0; x < n; ++x)
            for (int y = 0; y < n; ++y)
                if (x != y && cost(x, y) != (group[x] == group[y] ? lo : hi)) return;
        const int ng = (int)groups.size();
        if (largest <= 4 && ng <= 32) { out->gpl = 1; out->npg = 4; }
        else if (largest <= 4 && ng <= 64) { out->gpl = 2; out->npg = 4; }
        else if (largest <= 8 && ng <= 32) { out->gpl = 1; out->npg = 8; }
        else if (largest <= 4 && ng <= 128) { out->gpl = 4; out->npg = 4; }
        else return;
        out->kind = 2;
        out->tier[0] = c1; out->tier[1] = lo; out->tier[2] = hi;
        slots = 32 * out->gpl * out->npg;
        // groups go round the lanes, so that a problem's work is spread evenly
        for (int g = 0; g < ng; ++g)
            for (size_t i = 0; i < groups[g].size(); ++i)
                slot[groups[g][i]] = ((g % 32) * out->gpl + g / 32) * out->npg + (int)i;
        out->cost.assign(1, 0.0f);
    }
    out->slot_rep.assign(slots, -1);
    for (int c = 0; c < n; ++c) out->slot_rep[slot[c]] = reps[c];
    out->cls.resize(R);
    out->off.assign(slots + 1, 0);
    for (int i = 0; i < R; ++i) { out->cls[i] = (uint16_t)slot[of[i]]; out->off[out->cls[i] + 1]++; out->rep[i] = reps[of[i]]; }
    for (int s = 0; s < slots; ++s) out->off[s + 1] += out->off[s];
    out->list.resize(R);
    std::vector<int32_t> at(out->off.begin(), out->off.end() - 1);
    for (int i = 0; i < R; ++i) out->list[at[out->cls[i]]++] = (uint16_t)i;
}
