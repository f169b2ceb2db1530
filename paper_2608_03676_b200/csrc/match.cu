// Phase 2 (Appendix A.3, Algorithm 2: column-priority iterative matching) and Phase 3
// (Appendix A.4, Algorithm 3: Lagrangian auction), one CTA per layer, all round state in shared
// memory.
//
// Both phases are chains of short dependent rounds; a round is "every rank (slot) takes an
// argmax, conflicts are arbitrated by a second argmax, winners are applied".  The argmaxes are
// taken over packed 64-bit keys (score bits high, inverted index low) so that a single integer
// max gives "highest score, lowest index on ties", independent of thread order.  Scores are fp32
// with one rounding per operation (__fmul_rn / __fadd_rn / __fsub_rn / __fdiv_rn: no FMA
// contraction), which keeps every integer decision reproducible bit for bit on a CPU.
//
// Phase 2: the two score terms that do not change between rounds (alpha*B and 0.1*alpha*T_norm)
// are computed once per layer for the experts that spill, and the scores once per slot index.  It is
// bound by that chain of rounds.  A rank has several lanes and its state in their registers: they
// re-form its entries of the experts served in the last round, and scan its row again only if its
// best pair was among them; three barriers a round (one warp for up to 64 ranks: 87 -> 55 k cycles at
// 64 ranks, 16 rounds; a fourth barrier and all rows scanned in every round beyond: matching stage of
// 200 ranks with 600 slots 739 -> 688 us, 64 ranks 129 -> 123, 32 ranks 59.4 -> 57.3).
//
// In a plan the kernel is set up (loads, spills, score terms) while Phase 1 still runs and waits for
// it where it first reads the hint: a plan of one 8-rank layer 69 -> 66 us, 32 ranks 141 -> 129 us,
// 24 ranks 173 -> 164 us.
//
// Phase 3: the bonus matrix of a real topology has a handful of distinct values (tiers): the auction of auction.cuh.  A bonus
// matrix with more than TAOT_MAX_TIERS distinct values, a price step that is not positive or more than 1024 slots take a
// dense scan instead.
#include <type_traits>

#include "auction.cuh"
#include "taot_internal.cuh"

namespace {

typedef unsigned long long u64;

struct MatchArgs {
    const int32_t* n;            // [L,R,E]
    const int32_t* expert_load;  // [L,E]
    const int32_t* rank_load;    // [L,R]
    const float* plan;           // [L,R,R]
    const int32_t* e2r;          // [E]
    const float* B;              // [R,R]
    const int32_t* rank_off;     // [R+1]
    const int32_t* rank_list;    // [E]
    const uint32_t* tiermask;    // [ntiers][W][R hosts] bit r of word w: B3[32w + r][host] == tierval[t]
    const float* tierval;        // [ntiers] descending
    const uint32_t* bidlist;     // [nbid] (tier, win count) pairs by decreasing score: tier | win count << 8, bit 31: next has the same score
    const uint32_t* bident;      // [nbid] the same by tier and win count (see auction.cuh)
    const int32_t* hostcls;      // [R] hosts that see every rank at the same bonus share a number
    int32_t* slot_expert;        // [L,R,K]
    int32_t* slot_tokens;        // [L,R,K]
    int32_t* X;                  // [L,R,S]
    int32_t* rounds;             // [L,2] or null
    int32_t* info;               // [L]
    int32_t* nrem_g;             // [L, dmax, R] global fallback for the remaining counts
    float* t12;                  // [L, E, 2, R] scratch: alpha*B and beta*T_norm rows of the spilling experts
    int32_t R, E, K, dmax, ntiers, W, nbid;
    float eps0, price_step;
    int32_t auction_max_rounds;
    int32_t bon_in_smem;         // dense scan: the bonus matrix is in shared memory
    int32_t early;               // launched while Phase 1 runs: the hint is the only input that may not be there yet
    int32_t ablation;            // TAOT_ABLATE_* bits: a term switched off is an exact zero in the score
    int32_t nrem_in_smem;
    int32_t tm_in_smem;
    int32_t big_floats;          // 4-byte words of the shared block that holds the Phase-2 score rows, then nrem
    long long* cyc;              // [L][16] SM cycles per part of the kernel as thread 0 sees them, or null (profiling aid):
                                 // 0 set-up, 1 Phase 2, 2 Phase-3 set-up, 3 Phase-3 rounds of more than 32 classes, 4 of at most
                                 // 32 (one warp), 5 whole kernel, 6 classes, 7 the round the one warp went on with, 8-11 Phase-2
                                 // split, 12 the Phase-3 loop as a whole
};

__device__ __forceinline__ uint32_t ordered_bits(float f)
{
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ u64 warp_max_u64(u64 k)
{
    for (int o = 16; o > 0; o >>= 1) {
        const u64 other = __shfl_xor_sync(0xffffffffu, k, o);
        k = other > k ? other : k;
    }
    return k;
}

template <class T> struct Type { using type = T; };

constexpr size_t kSmemBudget = 224 * 1024;   // dynamic shared memory the kernel plans with (227 KB per CTA less the static part)

// Arbitration "best bidder per target" for one warp's worth of bids.  Many bidders often pick the
// same target (all slots of a tier chase the cheapest rank), so the lanes that bid for the same
// target first agree on their best key with warp-wide reductions and only one of them touches the
// shared-memory arbiter.  key = (score bits << 32) | inverted bidder index; valid bids have key != 0.
__device__ __forceinline__ void arbitrate(u64* arb, int target, u64 key)
{
    // (a hardware match-any on the target was measured several times slower than this loop over distinct targets)
    unsigned todo = __ballot_sync(0xffffffffu, key != 0);
    const uint32_t hi = (uint32_t)(key >> 32), lo = (uint32_t)key;
    const int lane = threadIdx.x & 31;
    while (todo) {                                   // one pass per distinct target among this warp's bids
        const int leader = __ffs(todo) - 1;
        const int tgt = __shfl_sync(0xffffffffu, target, leader);
        const bool mine = key != 0 && target == tgt;
        const unsigned group = __ballot_sync(0xffffffffu, mine);
        const uint32_t hi_max = __reduce_max_sync(0xffffffffu, mine ? hi : 0u);
        const uint32_t lo_max = __reduce_max_sync(0xffffffffu, (mine && hi == hi_max) ? lo : 0u);
        if (lane == leader) atomicMax(arb + tgt, ((u64)hi_max << 32) | (u64)lo_max);
        todo &= ~group;
    }
}

// LEAN: the auction's build for handles with at most four tiers and no equal scores; NSM: what the ranks hold is in shared memory
template <bool TIMED, int MAXT, bool LEAN, bool NSM>
__global__ void __launch_bounds__(MAXT, 1)
match_kernel(MatchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int R = a.R, E = a.E, K = a.K, S = R * K, W = a.W;
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = NT >> 5;
    const int64_t l = blockIdx.x;

    // ---- carve shared memory
    u64* arb_e = reinterpret_cast<u64*>(smem_raw);            // [E]  Phase 2 arbitration per expert
    u64* arb_r = arb_e + E;                                    // [2][R]  Phase 3 arbitration per rank, ping-pong by round
    uint2* tw_s = reinterpret_cast<uint2*>(arb_r + 2 * R);     // [ntiers][S] word and mask of a tier that one word holds, by class (LEAN: elsewhere)
    int32_t* spill = reinterpret_cast<int32_t*>(tw_s + (!LEAN && a.nbid ? a.ntiers * S : 0)); // [E]
    int32_t* hot0 = spill + E;                                 // [E]  experts that spill at the start of Phase 2
    int32_t* hot_home = hot0 + E;                              // [E]  their home ranks
    int32_t* dcol = hot_home + E;                              // [E]  expert -> column of nrem, or -1
    int32_t* spare = dcol + E;                                 // [R]
    int32_t* excess = spare + R;                               // [R]
    int32_t* matched = excess + R;                             // [R]
    int32_t* estar = matched + R;                              // [R]
    int32_t* wins = estar + R;                                 // [R]
    int32_t* slot_e = wins + R;                                // [S]
    int32_t* slot_a0 = slot_e + S;                             // [S]  planned tokens (Phase 2 result)
    int32_t* slot_a = slot_a0 + S;                             // [S+1] still to collect (Phase 3)
    uint32_t* avail = reinterpret_cast<uint32_t*>(slot_a + S + 1); // [W][dmax]  ranks still holding tokens of the expert (word-major: no bank conflicts across slots)
    uint32_t* lvl = avail + a.dmax * W;                        // [W][S+1]   ranks by win count (word-major)
    uint32_t* tm_s = lvl + (S + 1) * W;                                // [ntiers][W][S] tier masks by slot, if they fit
    uint32_t* bid_s = tm_s + (a.tm_in_smem ? a.ntiers * W * S : 0);    // [nbid] (tier, win count) pairs, best score first
    uint32_t* ent_s = bid_s + a.nbid;                                  // [nbid] the pairs by tier and win count
    int32_t* key_s = reinterpret_cast<int32_t*>(ent_s + a.nbid);       // [S] class keys, then the classes' lists
    uint16_t* nxt_s = reinterpret_cast<uint16_t*>(key_s + (a.nbid ? S : 0));            // [S] next slot of the class
    uint16_t* lead_s = nxt_s + (a.nbid ? S + 2 : 0);                   // [S] first slot of each class
    const int RS = R | 1;
    float* bon_s = reinterpret_cast<float*>(lead_s + (a.nbid ? S : 0));                // dense scan, if it fits: [R][RS] bonus of rank r for host h at h * RS + r
    int32_t* nrem_s = reinterpret_cast<int32_t*>(bon_s + (a.bon_in_smem ? R * RS : 0)); // [dmax*R] if it fits
    // LEAN, Phase 3 only, behind the counts in the block that Phase 2 uses for its keys
    uint2* rec_s = reinterpret_cast<uint2*>((reinterpret_cast<uintptr_t>(nrem_s + (a.nrem_in_smem ? a.dmax * (R | 1) : 0)) + 7) & ~(uintptr_t)7);   // [S+1] next slot of the class and its tokens
    uint2* const tw = LEAN ? rec_s + S + 1 : tw_s;
    __shared__ long long s_tot;
    __shared__ int s_cnt, s_any, s_ns;
    __shared__ taot_auction::Control ctl;
    __shared__ int s_wcnt[32];

    const int32_t* n = a.n + l * (int64_t)R * E;
    const int32_t* el = a.expert_load + l * E;
    const int32_t* rl = a.rank_load + l * R;
    const float* plan = a.plan + l * (int64_t)R * R;
    int32_t* nrem = a.nrem_in_smem ? nrem_s : a.nrem_g + l * (int64_t)a.dmax * R;
    const int RC = a.nrem_in_smem ? RS : R;       // stride of its columns
    float* t12 = a.t12 + l * (int64_t)E * 2 * R;      // global scratch; replaced by shared memory below if the rows fit

    // Everything up to the flow hint itself follows from the loads, which are there before Phase 1 starts: in a plan (a.early)
    // this kernel is set up while Phase 1 still runs, and only waits for it where the hint is first read.
    if (!a.early) taot_await();
    const bool timed = TIMED && tid == 0;
    const long long c_start = timed ? clock64() : 0;
    long long c_scan = 0, c_win = 0, c_row = 0, c_build = 0;
    // ---- integer mean, excess, spare (Appendix A.1)
    if (tid == 0) { s_tot = 0; s_cnt = 0; }
    int32_t* const el_s = dcol;                    // (dcol is Phase 3's)
    for (int e = tid; e < E; e += NT) el_s[e] = el[e];
    __syncthreads();
    {
        long long part = 0;
        for (int r = tid; r < R; r += NT) part += rl[r];
        if (part) atomicAdd(reinterpret_cast<u64*>(&s_tot), (u64)part);
    }
    // what Phase 3 starts from: every rank with 0 wins, no tokens in the plan
    for (int i = tid; i < (S + 1) * W; i += NT) {
        const int w = i / (S + 1), left = R - 32 * w;
        lvl[i] = i - w * (S + 1) != 0 ? 0u : (left >= 32 ? 0xFFFFFFFFu : (1u << left) - 1u);
    }
    int32_t* const Xl = a.X + l * (int64_t)R * S;
    if ((R * S) % 4 == 0 && (reinterpret_cast<uintptr_t>(Xl) & 15) == 0) {
        for (int q = tid; q < R * S / 4; q += NT) reinterpret_cast<int4*>(Xl)[q] = make_int4(0, 0, 0, 0);
    } else {
        for (int q = tid; q < R * S; q += NT) Xl[q] = 0;
    }
    for (int q = tid; q < a.nbid; q += NT) { bid_s[q] = a.bidlist[q]; ent_s[q] = a.bident[q]; }
    if (a.bon_in_smem) {
#pragma unroll 4
        for (int r = warp; r < R; r += NW)
            for (int h = lane; h < R; h += 32) bon_s[h * RS + r] = h == r ? 1.0f : a.B[(int64_t)r * R + h];
    }
    __syncthreads();
    const long long mean = s_tot / R;
    for (int r = tid; r < R; r += NT) {
        const long long lr = rl[r];
        excess[r] = (int32_t)(lr > mean ? lr - mean : 0);
        spare[r] = (int32_t)(mean > lr ? mean - lr : 0);
        wins[r] = 0;
        arb_r[r] = 0;
        arb_r[R + r] = 0;
    }
    // ---- spill by cumulative-excess differencing: position of e in its rank's (load, index) order
    for (int e = tid; e < E; e += NT) {
        const int r = a.e2r[e];
        const int32_t mine = el_s[e];
        const int q1 = a.rank_off[r + 1];
        long long cum = 0;
#pragma unroll 4
        for (int q = a.rank_off[r]; q < q1; ++q) {
            const int e2 = a.rank_list[q];
            const int32_t v = el_s[e2];
            cum += v < mine || (v == mine && e2 <= e) ? v : 0;
        }
        const long long hi = cum - mean, lo = cum - mine - mean;
        const int32_t sp = (int32_t)((hi > 0 ? hi : 0) - (lo > 0 ? lo : 0));
        spill[e] = sp;
        arb_e[e] = 0;
    }
    for (int s = tid; s < S; s += NT) { slot_e[s] = -1; slot_a0[s] = 0; }
    __syncthreads();
    // the experts that spill, in ascending index order (position q in this list orders them as the index does, so
    // "lowest expert on ties" is "lowest position on ties")
    int nhot0 = 0;
    for (int base = 0; base < E; base += NT) {
        const int e = base + tid;
        const bool hot = e < E && spill[e] > 0;
        const unsigned bal = __ballot_sync(0xffffffffu, hot);
        if (lane == 0) s_wcnt[warp] = __popc(bal);
        __syncthreads();
        int off = nhot0, tot = 0;
        for (int w = 0; w < NW; ++w) { const int c = s_wcnt[w]; if (w < warp) off += c; tot += c; }
        if (hot) {
            const int q = off + __popc(bal & ((1u << lane) - 1u));
            hot0[q] = e;
            hot_home[q] = a.e2r[e];
        }
        nhot0 += tot;
        __syncthreads();
    }

    const float alpha = __fdiv_rn((float)(mean * (long long)R), (float)E);
    const float beta = __fmul_rn(0.1f, alpha);
    // Phase 2 keeps the current score of every (rank, spilling expert) pair as an integer key, row stride odd so that
    // neither a rank's scan nor an expert's update meets bank conflicts; the keys and the round-invariant rows below
    // are only used in Phase 2 and the remaining counts only exist in Phase 3: they share one block
    const int NHs = nhot0 | 1;
    const bool keyed = nhot0 > 0 && (int64_t)NHs * R <= (int64_t)a.big_floats;
    uint32_t* keyM = reinterpret_cast<uint32_t*>(nrem_s);                       // [R][NHs]
    const int64_t key_words = keyed ? (int64_t)NHs * R : 0;
    if (key_words + (int64_t)nhot0 * 2 * R <= (int64_t)a.big_floats) t12 = reinterpret_cast<float*>(nrem_s) + key_words;

    // ---- round-invariant score terms of the spilling experts: t1 = alpha*B, t2 = beta*T/max(excess, eps0).  Thread tid takes
    // rank tid % RP (RP a power of two) of every (NT / RP)-th expert: no division, consecutive threads on consecutive ranks
    int rsh = 5;
    while ((1 << rsh) < R) ++rsh;
    const int my_r = tid & ((1 << rsh) - 1), my_q = tid >> rsh, q_step = NT >> rsh;
    if (my_r < R) {
#pragma unroll 4
        for (int q = my_q; q < nhot0; q += q_step) {
            const float bp = (a.ablation & TAOT_ABLATE_TOPOLOGY) ? 0.0f : a.B[hot_home[q] * R + my_r];
            t12[(int64_t)(2 * q) * R + my_r] = __fmul_rn(alpha, bp);
        }
    }
    if (a.early) taot_await();
    if (my_r < R) {
#pragma unroll 4
        for (int q = my_q; q < nhot0; q += q_step) {
            const int hr = hot_home[q];
            const float ex = fmaxf((float)excess[hr], a.eps0);
            const float tn = (a.ablation & TAOT_ABLATE_HINT) ? 0.0f : __fdiv_rn(plan[hr * R + my_r], ex);
            t12[(int64_t)(2 * q + 1) * R + my_r] = __fmul_rn(beta, tn);
        }
    }
    __syncthreads();

    // =========================================================== Phase 2
    const long long c_p2 = timed ? clock64() : 0;
    int rounds2 = 0;
    int qsh = 0;                                  // lanes per rank in the scan: QS = 2^qsh, the largest power of two <= min(32, NT / R)
    while ((2 << qsh) <= 32 && (2 << qsh) * R <= NT) ++qsh;
    const int QS = 1 << qsh;
    const int qs = tid & (QS - 1);
    // score of expert position q on rank r as an ordered integer key, 0 if the pair is no candidate (Algorithm 2's mask:
    // the expert still spills, r is not its home, it is not on r already); the rank-side conditions (unmatched, spare
    // left) are tested by the rank's scan
    auto pair_key = [&](int q, int r, int kappa) -> uint32_t {
        const int e = hot0[q];
        const int32_t se = spill[e];
        bool ok = se > 0 && hot_home[q] != r;
        for (int kk = 0; kk < kappa; ++kk) ok = ok && (slot_e[r * K + kk] != e);
        const int32_t sp = spare[r];
        const int32_t gain = se < sp ? se : sp;
        const float sc = __fadd_rn(__fadd_rn((float)gain, t12[((int64_t)q * 2) * R + r]), t12[((int64_t)q * 2 + 1) * R + r]);
        return ok ? ordered_bits(sc) : 0u;
    };
    int32_t* served = dcol;                       // [E] positions of the experts served in a round (dcol is Phase 3's)
    // score of a pair whose key is not 0 after its expert's spill has shrunk to se
    auto shrunk_key = [&](int q, int r, int32_t se, int32_t sp) -> uint32_t {
        const int32_t gain = se < sp ? se : sp;
        return ordered_bits(__fadd_rn(__fadd_rn((float)gain, t12[(int64_t)(2 * q) * R + r]), t12[(int64_t)(2 * q + 1) * R + r]));
    };
    for (int kappa = 0; keyed && kappa < K; ++kappa) {
        // Between rounds a pair's score changes only when its expert was served (its spill shrank): a rank's spare
        // changes only when it is matched, and then it is out for this slot index.  So all keys are formed once per
        // slot index and a round re-forms the rows of the experts it served; a rank's arg-max is one load and one
        // compare per spilling expert.
        const long long c_b0 = timed ? clock64() : 0;
        // arbitration state per expert: best score among this round's bidders, then the lowest rank that has it
        uint32_t* arb_hi = reinterpret_cast<uint32_t*>(arb_e);
        uint32_t* arb_lo = arb_hi + E;
        int smax = 0;                              // largest spare of this slot index: a row changes only below it
        for (int r = tid; r < R; r += NT) { smax = spare[r] > smax ? spare[r] : smax; }
        for (int e = tid; e < E; e += NT) { arb_hi[e] = 0u; arb_lo[e] = 0xFFFFFFFFu; }
        smax = __reduce_max_sync(0xffffffffu, smax);
        if (tid == 0) s_cnt = 0;
        __syncthreads();
        if (lane == 0) atomicMax(&s_cnt, smax);
        if (my_r < R)
#pragma unroll 4
            for (int q = my_q; q < nhot0; q += q_step) keyM[my_r * NHs + q] = pair_key(q, my_r, kappa);
        __syncthreads();
        const int32_t spare_cap = s_cnt;
        if (timed) c_build += clock64() - c_b0;
        // QS adjacent lanes share a rank and its row of keys (QS * R <= NT: one pass covers every rank); the rank's state is in
        // registers, the same in all of them.
        const int r = tid >> qsh;
        const bool lead = qs == 0;
        const unsigned group = (QS == 32 ? 0xFFFFFFFFu : ((1u << QS) - 1u) << (lane & ~(QS - 1)));
        uint32_t* const row = keyM + (r < R ? r : 0) * NHs;
        const int32_t sp = r < R ? spare[r] : 0;
        bool open = sp > 0, scan = open;
        uint32_t bk = 0u;                          // the rank's best candidate: key and position (0: none)
        int bq = 0, ns = 0;
        for (;;) {
            const long long c_s0 = timed ? clock64() : 0;
            // the served experts' entries of the row, which change only where min(spill, spare) does
            if (ns > 0) {                          // uniform over the CTA
                bool hit = false;
                if (open) {
                    for (int i = qs; i < ns; i += QS) {
                        const int q = served[i];
                        const int32_t se = spill[hot0[q]];
                        if (se < sp && row[q]) {
                            row[q] = se > 0 ? shrunk_key(q, r, se, sp) : 0u;
                            hit = hit || q == bq;
                        }
                    }
                }
                scan = (__ballot_sync(0xffffffffu, hit) & group) != 0u;
                __syncwarp();
            }
            const long long c_s1 = timed ? clock64() : 0;
            // Steps 1-2: every unmatched cold rank takes its best candidate expert (ties: lowest position = lowest index); one
            // whose best pair did not change in the last round still has it, since keys only shrink
            if (__any_sync(0xffffffffu, scan)) {
                uint32_t best = 0u;
                int at = 0;
                if (open) {
#pragma unroll 4
                    for (int q = qs; q < nhot0; q += QS) {      // ascending positions: a strict compare keeps the lowest
                        const uint32_t v = row[q];
                        at = v > best ? q : at;
                        best = v > best ? v : best;
                    }
                }
                for (int o = 1; o < QS; o <<= 1) {
                    const uint32_t v = __shfl_xor_sync(0xffffffffu, best, o);
                    const int p = __shfl_xor_sync(0xffffffffu, at, o);
                    const bool better = (v > best) | ((v == best) & (p < at));
                    best = better ? v : best;
                    at = better ? p : at;
                }
                bk = best; bq = at;
                open = open && best != 0u;
                scan = false;
            }
            // Step 3, first half: the best score any rank offers the expert
            const bool bids = lead && open;
            if (bids) atomicMax(&arb_hi[bq], bk);
            if (!__syncthreads_or(bids)) break;
            if (tid == 0) s_ns = 0;
            // Step 3, second half: among the ranks that offer it, the lowest
            if (bids && arb_hi[bq] == bk) atomicMin(&arb_lo[bq], (uint32_t)r);
            __syncthreads();
            const long long c_s2 = timed ? clock64() : 0;
            // Step 4: winners take min(spill, spare), and put the arbitration entries back (a loser compares arb_lo with its own
            // rank: the reset value is nobody's).  Rows whose expert still spills at least the largest spare of this slot index
            // are left as they are.
            const bool win = bids && arb_lo[bq] == (uint32_t)r;
            if (win) {
                const int e = hot0[bq];
                const int32_t se = spill[e], g = se < sp ? se : sp;
                spill[e] = se - g;
                spare[r] = sp - g;
                slot_e[r * K + kappa] = e;
                slot_a0[r * K + kappa] = g;
                arb_hi[bq] = 0u;
                arb_lo[bq] = 0xFFFFFFFFu;
                if (se - g < spare_cap) served[atomicAdd(&s_ns, 1)] = bq;
            }
            if (__ballot_sync(0xffffffffu, win) & group) open = false;
            __syncthreads();
            ns = s_ns;
            ++rounds2;
            if (timed) { const long long c_s3 = clock64(); c_row += c_s1 - c_s0; c_scan += c_s2 - c_s1; c_win += c_s3 - c_s2; }
        }
        __syncthreads();
    }
    for (int kappa = 0; !keyed && kappa < K; ++kappa) {
        for (int r = tid; r < R; r += NT) matched[r] = 0;
        for (;;) {
            if (tid == 0) s_any = 0;
            __syncthreads();
            // Steps 1-2: every unmatched cold rank takes its best candidate expert.  QS adjacent lanes share one rank
            // and split the list of spilling experts between them; their best keys meet by xor-shuffles.
            for (int rb = 0; rb < R; rb += NT >> qsh) {
                const int r = rb + (tid >> qsh);                  // whole warps stay in the loop for the warp-wide steps
                int best_e = -1;
                u64 key = 0;
                const int32_t sp = r < R ? spare[r] : 0;
                if (r < R && !matched[r] && sp > 0) {
                    for (int q = qs; q < nhot0; q += QS) {
                        const int e = hot0[q];
                        const int32_t se = spill[e];
                        if (se <= 0 || hot_home[q] == r) continue;
                        bool placed = false;
                        for (int kk = 0; kk < kappa; ++kk) placed |= (slot_e[r * K + kk] == e);
                        if (placed) continue;
                        const int32_t gain = se < sp ? se : sp;
                        const float t1 = t12[((int64_t)q * 2) * R + r];
                        const float t2 = t12[((int64_t)q * 2 + 1) * R + r];
                        const float sc = __fadd_rn(__fadd_rn((float)gain, t1), t2);
                        const u64 k64 = ((u64)ordered_bits(sc) << 32) | (u64)(0xFFFFFFFFu - (uint32_t)e);   // ordered: a negative preference may give a negative score
                        key = k64 > key ? k64 : key;
                    }
                }
                for (int o = 1; o < QS; o <<= 1) {
                    const u64 other = __shfl_xor_sync(0xffffffffu, key, o);
                    key = other > key ? other : key;
                }
                if (key != 0) best_e = (int)(0xFFFFFFFFu - (uint32_t)key);
                const bool lead = qs == 0 && r < R;
                if (lead) {
                    estar[r] = best_e;
                    if (key != 0) s_any = 1;
                }
                // Step 3: arbitration, best rank per expert (ties: lowest rank)
                arbitrate(arb_e, best_e, (key == 0 || !lead) ? 0ull : ((key & 0xFFFFFFFF00000000ull) | (u64)(0xFFFFFFFFu - (uint32_t)r)));
            }
            __syncthreads();
            if (!s_any) break;
            // Step 4: winners take min(spill, spare)
            for (int r = tid; r < R; r += NT) {
                const int e = estar[r];
                if (e >= 0 && (uint32_t)arb_e[e] == 0xFFFFFFFFu - (uint32_t)r) {
                    const int32_t g = spill[e] < spare[r] ? spill[e] : spare[r];
                    spill[e] -= g;
                    spare[r] -= g;
                    matched[r] = 1;
                    slot_e[r * K + kappa] = e;
                    slot_a0[r * K + kappa] = g;
                }
            }
            __syncthreads();
            for (int q = tid; q < nhot0; q += NT) arb_e[hot0[q]] = 0;
            ++rounds2;
        }
        __syncthreads();
    }

    // =========================================================== Phase 3
    const long long c_p3 = timed ? clock64() : 0;
    long long c_p3loop = c_p3, c_p3warp = c_p3, c_p3end = c_p3, c_classes = 0, c_handed = 0;
    // compact the experts that sit in some slot; keep their per-rank remaining counts transposed [col][r]
    for (int e = tid; e < E; e += NT) dcol[e] = -1;
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    for (int s = tid; s < S; s += NT) {
        slot_a[s] = slot_a0[s];
        if (slot_e[s] >= 0) dcol[slot_e[s]] = -2;
    }
    __syncthreads();
    for (int e = tid; e < E; e += NT)
        if (dcol[e] == -2) dcol[e] = atomicAdd(&s_cnt, 1);
    __syncthreads();
    const int D = s_cnt;
    for (int e = tid; e < E; e += NT)
        if (dcol[e] >= 0) hot0[dcol[e]] = e;                   // column -> expert (the Phase-2 list is no longer needed)
    __syncthreads();
    // a warp per expert and word of 32 ranks: the word of ranks that hold its tokens by a vote (reductions of single bits into
    // one shared word queue up: 55 k cycles at 256 ranks)
#pragma unroll 4
    for (int q = warp; q < D * W; q += NW) {
        const int col = q / W, w = q - col * W, r = 32 * w + lane;
        const int32_t v = r < R ? n[r * E + hot0[col]] : 0;
        if (r < R) nrem[col * RC + r] = v;
        const unsigned word = __ballot_sync(0xffffffffu, v > 0);
        if (lane == 0) avail[w * a.dmax + col] = word;
    }
    __syncthreads();

    int rounds3 = 0;
    const long long cap = (long long)R * S + S;
    const bool tiered = a.nbid > 0 && S <= NT;
    if (tiered && D > 0) {
        // ---- bit-set auction (auction.cuh): bidders are classes of slots that make the same bids
        namespace au = taot_auction;
        uint32_t* const arb = reinterpret_cast<uint32_t*>(arb_r);       // [2][R + W]
        for (int q = tid; q < 2 * (R + W); q += NT) arb[q] = 0u;
        // a live slot's class: expert and the way its host sees the ranks; the lowest slot leads, the others queue behind it
        const int s = tid;
        const bool slive = s < S && slot_e[s] >= 0 && slot_a[s] > 0;
        if (s < S) {
            key_s[s] = slive ? slot_e[s] * R + a.hostcls[s / K] : -1 - s;
            nxt_s[s] = (uint16_t)S;
        }
        if (tid == 0) { nxt_s[S] = (uint16_t)S; slot_a[S] = 0; ctl.event[0] = ctl.event[1] = ctl.dead[0] = ctl.dead[1] = ctl.last = ctl.handed = 0u; }
        __syncthreads();
        bool lead = slive;
        if (slive) {
            const int32_t mine = key_s[s];
            int prev = -1;
#pragma unroll 8
            for (int q = 0; q < s; ++q) prev = key_s[q] == mine ? q : prev;
            if (prev >= 0) { nxt_s[prev] = (uint16_t)s; lead = false; }
        }
        const unsigned lb = __ballot_sync(0xffffffffu, lead);
        if (lane == 0) s_wcnt[warp] = __popc(lb);
        __syncthreads();
        int C = 0;
        {
            int off = 0;
            for (int w = 0; w < NW; ++w) { const int cnt = s_wcnt[w]; if (w < warp) off += cnt; C += cnt; }
            if (lead) lead_s[off + __popc(lb & ((1u << lane) - 1u))] = (uint16_t)s;
        }
        if constexpr (LEAN)
            for (int q = tid; q <= S; q += NT) rec_s[q] = make_uint2(nxt_s[q], (uint32_t)slot_a[nxt_s[q]]);
        __syncthreads();
        // tier masks by class, and for each tier the word that holds all of it
        if (a.tm_in_smem) {
            for (int q = tid; q < a.ntiers * W * C; q += NT) {
                const int tw = q / C, c = q - tw * C;
                tm_s[tw * S + c] = a.tiermask[(int64_t)tw * R + lead_s[c] / K];
            }
        }
        const uint32_t* tm = a.tm_in_smem ? tm_s : a.tiermask;
        const int tms = a.tm_in_smem ? S : R;
        __syncthreads();
        for (int q = tid; q < a.ntiers * C; q += NT) {
            const int t = q / C, c = q - t * C;
            int nz = 0, wd = 0;
            uint32_t val = 0u;
            for (int w = 0; w < W; ++w) {
                const uint32_t mk = tm[(t * W + w) * tms + (a.tm_in_smem ? c : lead_s[c] / K)];
                if (mk) { ++nz; wd = w; val = mk; }
            }
            tw[t * S + c] = make_uint2(nz <= 1 ? (uint32_t)wd : 0xFFFFFFFFu, val);
        }
        __syncthreads();
        long long limit = cap;
        if (a.auction_max_rounds > 0 && a.auction_max_rounds < limit) limit = a.auction_max_rounds;
        const uint32_t round_limit = (uint32_t)limit;                   // at most R * S + S < 2^19
        if (timed) c_p3loop = clock64();
        const au::Tables tab{arb, avail, lvl, bid_s, ent_s, tm, tw, slot_e, slot_a, rec_s, nxt_s, dcol, nrem, Xl,
                             R, S, K, W, a.dmax, a.ntiers, tms, a.tm_in_smem != 0, RC,
                             reinterpret_cast<int32_t*>(a.t12 + l * (int64_t)E * 2 * R)};       // (Phase 2's scratch)
        const int NP = ((C + 31) >> 5) << 5;
        auto run = [&](auto type, auto rounds_block, auto rounds_warp) {
            using B = typename decltype(type)::type;
            uint32_t rd = 1u;
            if (C > 32) {
                if (tid < NP) {
                    B b(tab);
                    if (tid < C) b.start(tid, lead_s[tid]);
                    __syncwarp();
                    rd = rounds_block(b);
                }
                __syncthreads();
            }
            if (timed) { c_p3warp = clock64(); c_classes = C; c_handed = (long long)rd; }
            if (warp == 0) {
                B b(tab);
                if (C > 32) {
                    if (lane < (int)ctl.handed) b.start((int)(ctl.hand[lane] >> 16), (int)(ctl.hand[lane] & 0xFFFFu));
                } else if (lane < C) {
                    b.start(lane, lead_s[lane]);
                }
                __syncwarp();
                const uint32_t last = rounds_warp(b, rd);
                __syncwarp();
                if (lane == 0) ctl.last = last;
            }
        };
        if constexpr (!LEAN) {
            run(Type<au::Bidder>{},
                [&](auto& b) { return au::run_block(b, NP, C, round_limit, &ctl); },
                [&](auto& b, uint32_t rd) { return au::run_warp(b, rd, round_limit, ctl.last); });
        } else {
            const auto lean = [&](auto tiers, auto words) {
                run(Type<au::Lean<decltype(tiers)::value, NSM, decltype(words)::value>>{},
                    [&](auto& b) { return au::run_block_lean(b, NP, C, round_limit, &ctl); },
                    [&](auto& b, uint32_t rd) { return au::run_warp_lean(b, rd, round_limit, ctl.last); });
            };
            const auto lean_w = [&](auto tiers) {
                if (W == 1) lean(tiers, std::integral_constant<int, 1>{});
                else if (W == 2) lean(tiers, std::integral_constant<int, 2>{});
                else if (W <= 4) lean(tiers, std::integral_constant<int, 4>{});
                else lean(tiers, std::integral_constant<int, au::kMaxWords>{});
            };
            if (a.ntiers <= 2) lean_w(std::integral_constant<int, 2>{});
            else lean_w(std::integral_constant<int, 4>{});
        }
        if (timed) c_p3end = clock64();
        __syncthreads();
        rounds3 = (int)ctl.last;                  // rounds in which somebody bid
    } else {
        // Dense scan: LPS lanes per slot (as many as two slots per thread cover) look at every rank that holds tokens of its
        // expert, each slot starting at a rank of its own so that lanes on different rows do not meet in one bank; the rank's
        // best bidder is found by 32-bit maxima in two steps (score, then the lowest slot that offers it).  A round is one
        // chain, so what does not change (addresses: integer divisions) is worked out before the loop and the scan has no branch.
        // (At most 2048 slots, and a CTA of at least half as many threads: two slots per thread always suffice.)
        // Measured: 24 ranks with measured costs, 7 layers, 72 slots, 22 rounds: matching stage 73 -> 51 us (before: a warp per slot,
        // the bonus from global memory, 64-bit maxima; 4500 cycles a round).
        if (timed) c_p3loop = clock64();
        float* const price = reinterpret_cast<float*>(estar);          // [R] step * wins
        uint32_t* const bid_hi = reinterpret_cast<uint32_t*>(arb_r);   // [R] best score offered
        uint32_t* const bid_lo = bid_hi + R;                           // [R] lowest slot that offers it
        int lsh = 0;
        while (lsh < 5 && ((int64_t)S << (lsh + 1)) <= 2 * NT) ++lsh;
        const int LPS = 1 << lsh, sub = tid & (LPS - 1);
        int slot[2], host[2], coff[2], boff[2], r0[2];
        bool own[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int q = (tid >> lsh) + p * (NT >> lsh);
            own[p] = q < S && slot_e[q < S ? q : 0] >= 0;
            slot[p] = own[p] ? q : 0;
            host[p] = slot[p] / K;
            coff[p] = own[p] ? dcol[slot_e[q]] * RC : 0;
            boff[p] = host[p] * RS;
            r0[p] = (sub + slot[p]) % R;
        }
        for (int r = tid; r < R; r += NT) { price[r] = __fmul_rn(a.price_step, 0.0f); bid_hi[r] = 0u; bid_lo[r] = 0xFFFFFFFFu; }
        if (tid == 0) s_any = 0;
        __syncthreads();
        // the best (score, lowest rank) over this lane's ranks; `bon`: the bonus matrix is in shared memory
        auto scan = [&](auto bon, const bool (&live)[2], uint32_t (&bk)[2], int (&br)[2]) {
            int r[2] = {r0[0], r0[1]};
#pragma unroll 4
            for (int i = sub; i < R; i += LPS) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int32_t have = nrem[coff[p] + r[p]];
                    float b3;
                    if constexpr (decltype(bon)::value) b3 = bon_s[boff[p] + r[p]];
                    else b3 = r[p] == host[p] ? 1.0f : __ldg(a.B + (int64_t)r[p] * R + host[p]);
                    const uint32_t bits = ordered_bits(__fsub_rn(b3, price[r[p]]));
                    const uint32_t k = (have > 0) & live[p] ? bits : 0u;
                    const bool better = (k > bk[p]) | ((k == bk[p]) & (r[p] < br[p]));
                    bk[p] = better ? k : bk[p];
                    br[p] = better ? r[p] : br[p];
                    const int next = r[p] + LPS;
                    r[p] = next >= R ? next - R : next;      // (more lanes than ranks: there is no next one)
                }
            }
        };
        for (;;) {
            if (a.auction_max_rounds > 0 && rounds3 >= a.auction_max_rounds) break;
            if (rounds3 >= cap || D == 0) break;
            // Step 1: every unfinished slot bids for the source rank with the best bonus minus price (ties: the lowest rank)
            bool live[2];
            uint32_t bk[2] = {0u, 0u};
            int br[2] = {0x7FFFFFFF, 0x7FFFFFFF};
#pragma unroll
            for (int p = 0; p < 2; ++p) live[p] = own[p] && slot_a[slot[p]] > 0;
            if (__any_sync(0xffffffffu, live[0] | live[1])) {
                if (a.bon_in_smem) scan(std::true_type{}, live, bk, br);
                else scan(std::false_type{}, live, bk, br);
                for (int o = 1; o < LPS; o <<= 1) {
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        const uint32_t k = __shfl_xor_sync(0xffffffffu, bk[p], o);
                        const int r = __shfl_xor_sync(0xffffffffu, br[p], o);
                        const bool better = (k > bk[p]) | ((k == bk[p]) & (r < br[p]));
                        bk[p] = better ? k : bk[p];
                        br[p] = better ? r : br[p];
                    }
                }
            }
            bool bids[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                bids[p] = sub == 0 && bk[p] != 0u;
                if (bids[p]) { atomicMax(&bid_hi[br[p]], bk[p]); s_any = rounds3 + 1; }
            }
            __syncthreads();
            if (s_any != rounds3 + 1) break;
            // Step 2: the rank keeps its best bidder (ties: lowest slot)
#pragma unroll
            for (int p = 0; p < 2; ++p)
                if (bids[p] && bid_hi[br[p]] == bk[p]) atomicMin(&bid_lo[br[p]], (uint32_t)slot[p]);
            __syncthreads();
            // Steps 3-4: allocate, update holdings, plan and price (a loser compares with its own slot: the reset value is nobody's)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (!bids[p] || bid_lo[br[p]] != (uint32_t)slot[p]) continue;
                const int r = br[p], q = slot[p];
                bid_hi[r] = 0u;
                bid_lo[r] = 0xFFFFFFFFu;
                const int32_t have = nrem[coff[p] + r], left = slot_a[q];
                const int32_t x = have < left ? have : left;
                Xl[(int64_t)r * S + q] = x;          // a (rank, slot) pair is served at most once
                nrem[coff[p] + r] = have - x;
                slot_a[q] = left - x;
                if (x > 0) price[r] = __fmul_rn(a.price_step, (float)++wins[r]);
            }
            ++rounds3;
            __syncthreads();
        }
        if (timed) c_p3end = clock64();
    }

    taot_release();
    // ---- outputs
    int residual = 0;
    for (int s = tid; s < S; s += NT) {
        a.slot_expert[l * S + s] = slot_e[s];
        a.slot_tokens[l * S + s] = slot_a0[s];
        if (slot_e[s] >= 0 && slot_a[s] > 0) residual = 1;
    }
    residual = __syncthreads_or(residual);
    if (tid == 0) {
        if (a.rounds) { a.rounds[l * 2] = rounds2; a.rounds[l * 2 + 1] = rounds3; }
        if (residual) atomicOr(a.info + l, TAOT_INFO_AUCTION_RESIDUAL);
        if (timed) {
            long long* c = a.cyc + l * 16;
            c[0] = c_p2 - c_start; c[1] = c_p3 - c_p2; c[2] = c_p3loop - c_p3;
            c[3] = c_p3warp - c_p3loop; c[4] = c_p3end - c_p3warp;
            c[5] = clock64() - c_start; c[6] = c_classes; c[7] = c_handed;
            c[8] = c_scan; c[9] = c_win; c[10] = c_row; c[11] = c_build;
            c[12] = c_p3end - c_p3loop;
            for (int i = 13; i < 16; ++i) c[i] = 0;
        }
    }
}

size_t match_smem_fixed(int R, int E, int K, int dmax, int W)
{
    const size_t S = (size_t)R * K;
    return sizeof(u64) * (E + 2 * (size_t)R) + sizeof(int32_t) * (4 * (size_t)E + 5 * (size_t)R + 3 * S + 1) +
           sizeof(uint32_t) * ((size_t)dmax * W + (S + 1) * W);
}

}  // namespace

int taot_launch_match(taot_handle_t h, const int32_t* d_n, const int32_t* d_expert_load,
                      const int32_t* d_rank_load, const float* d_plan, int32_t* d_slot_expert,
                      int32_t* d_slot_tokens, int32_t* d_X, int32_t* d_rounds, int32_t* d_info,
                      int32_t* d_nrem, float* d_t12, cudaStream_t st, long long* d_cyc, bool early)
{
    const taot_params& p = h->p;
    MatchArgs a;
    a.cyc = d_cyc;
    a.early = early ? 1 : 0;
    a.n = d_n; a.expert_load = d_expert_load; a.rank_load = d_rank_load; a.plan = d_plan;
    a.e2r = h->d_e2r; a.B = h->d_B; a.rank_off = h->d_rank_off; a.rank_list = h->d_rank_list;
    a.tiermask = h->d_tiermask; a.tierval = h->d_tierval; a.bidlist = h->d_bidlist;
    a.bident = h->d_bident; a.hostcls = h->d_hostcls;
    a.slot_expert = d_slot_expert; a.slot_tokens = d_slot_tokens; a.X = d_X; a.rounds = d_rounds;
    a.info = d_info; a.nrem_g = d_nrem; a.t12 = d_t12;
    a.R = p.R; a.E = p.E; a.K = p.K;
    a.dmax = p.E < p.R * p.K ? p.E : p.R * p.K;
    a.W = (p.R + 31) / 32;
    a.nbid = (h->ntiers > 0 && h->nbid > 0 && a.W <= taot_auction::kMaxWords && p.R * p.K <= 1024) ? h->nbid : 0;
    a.ntiers = a.nbid > 0 ? h->ntiers : 0;
    a.eps0 = p.eps0; a.price_step = p.price_step; a.auction_max_rounds = p.auction_max_rounds;
    a.ablation = p.ablation;
    size_t smem = match_smem_fixed(p.R, p.E, p.K, a.dmax, a.W);
    const bool few_tiers = h->ntiers <= 4 && !h->bid_ties;
    const size_t S = (size_t)p.R * p.K;
    const size_t lists = sizeof(uint32_t) * (2 * (size_t)h->nbid + (few_tiers ? 0 : 2 * (size_t)h->ntiers * S) + 2 * S + 1);
    // (few tiers: what only Phase 3 needs lies behind the counts, see below)
    size_t lean_bytes = a.nbid > 0 && few_tiers ? sizeof(uint2) * (S + 1 + (size_t)h->ntiers * S) + 8 : 0;
    if (a.nbid > 0 && smem + lists + lean_bytes > kSmemBudget) { a.nbid = 0; a.ntiers = 0; lean_bytes = 0; }      // (no room for the lists: the dense scan)
    if (a.nbid > 0) smem += lists;
    const size_t nrem_bytes = sizeof(int32_t) * (size_t)a.dmax * (p.R | 1);
    // the bonus matrix of the dense scan, where it fits beside the remaining counts
    const size_t bon_bytes = sizeof(float) * (size_t)p.R * (p.R | 1);
    a.bon_in_smem = (a.nbid == 0 && smem + bon_bytes + nrem_bytes <= kSmemBudget) ? 1 : 0;
    if (a.bon_in_smem) smem += bon_bytes;
    const size_t tm_bytes = sizeof(uint32_t) * (size_t)a.ntiers * a.W * p.R * p.K;
    a.tm_in_smem = (a.ntiers > 0 && smem + tm_bytes <= 96 * 1024) ? 1 : 0;
    if (a.tm_in_smem) smem += tm_bytes;
    a.nrem_in_smem = (smem + nrem_bytes + lean_bytes <= kSmemBudget) ? 1 : 0;
    // one block for Phase 2 (per spilling expert R keys and 2 * R floats of round-invariant score rows) and then the
    // remaining counts and the lists of Phase 3: as large as those need, and as much of what Phase 2 could use as there is
    // room for (a layer whose keys do not fit takes the full scan: 256 ranks, 1024 experts, 1024 slots 1.7 -> 2.1 ms with 8 KB less)
    size_t big = (a.nrem_in_smem ? nrem_bytes : 0) + lean_bytes;
    const size_t want = sizeof(float) * ((size_t)p.R * ((size_t)p.E | 1) + 2 * (size_t)p.R * (size_t)p.E);
    const size_t room = kSmemBudget > smem ? kSmemBudget - smem : 0;
    if (big < want) big = want < room ? want : (room > big ? room : big);
    a.big_floats = (int32_t)(big / 4);
    smem += big;
    // a round of the auction reads the arbiters of all words of its build, and on behind the last rank's: that has to be there for a
    // handful of ranks and experts too
    const size_t reach = sizeof(u64) * (size_t)p.E + sizeof(uint32_t) * ((size_t)p.R + a.W + 33 * (taot_auction::kMaxWords - 1) + 32);
    if (smem < reach) smem = reach;
    if (smem > 227 * 1024) return TAOT_ERR_UNSUPPORTED;
    const int need = p.R * p.K;
    // two threads per slot: Phase 2 splits each rank's scan over more lanes, and the extra warps cost less than that saves
    // (measured: 256 threads for 16 and 64 ranks, 512 for 256 ranks x 1 slot); more than 512 only if there are more slots,
    // since the registers of the auction's builds are cut in half there
    int NT = 2 * (((need + 31) / 32) * 32);
    NT = NT < 256 ? 256 : (NT > 512 && need <= 512 ? 512 : (NT > 1024 ? 1024 : NT));
    auto launch = [&](auto kernel) -> int {
        TAOT_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        TAOT_CUDA_OK(taot_launch_chained(kernel, p.L, NT, smem, st, a));
        return 1;
    };
    const bool lean = a.nbid > 0 && few_tiers, nsm = a.nrem_in_smem != 0;
    auto build = [&](auto timed, auto maxt) -> int {
        constexpr bool TIMED = decltype(timed)::value;
        constexpr int MAXT = decltype(maxt)::value;
        if (!lean) return launch(match_kernel<TIMED, MAXT, false, false>);
        return nsm ? launch(match_kernel<TIMED, MAXT, true, true>) : launch(match_kernel<TIMED, MAXT, true, false>);
    };
    if (d_cyc) return build(std::true_type{}, std::integral_constant<int, 1024>{});
    return NT <= 512 ? build(std::false_type{}, std::integral_constant<int, 512>{}) : build(std::false_type{}, std::integral_constant<int, 1024>{});
}
