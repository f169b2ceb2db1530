// Phase 3 (Appendix A.4, Algorithm 3) as a bit-set auction, for match.cu.
//
// In every round each slot that still collects tokens bids for the source rank that holds tokens of its expert and
// maximises  B3 - step * wins;  every rank serves its best bidder (ties: lowest slot); a rank that served gets dearer.
//
// Bidders.  Slots of the same expert whose hosts see every rank at the same bonus make the same bid in every round, and of
// equal bids the lowest slot wins: only the lowest unfinished slot of such a class can ever win.  So a bidder is a class
// (one thread) with a queue of slots; 216 slots of a 256-rank layer are about 85 classes, 58 of a 64-rank layer about 30 --
// one warp.
//
// A bid.  The bonus of a real topology has few distinct values (tiers), so every score is one of (tier, win count) pairs,
// ordered once per handle by their fp32 score.  A class rests on the best pair that still has candidates: ranks of the
// tier, holding the expert, with that win count.  Win counts only grow and holdings only shrink, so no pair before it can
// regain one, and candidates of the pair itself only go away -- by being won.  Every rank that is bid for is won by somebody
// and leaves its win count, so the ranks bid for in a round, one bit each, are all a class has to know to keep its word of
// candidates (32 ranks, a register) exact.  Only when that word runs empty does it look at the shared sets again (walk).
//
// A round.  Bid: a maximum into the rank's arbiter; the tokens the rank holds are fetched ahead.  Then one barrier (or a warp
// barrier, once at most 32 classes are left), and the arbiters are read back: those that hold a key of this round are the
// ranks that were won (32 of them per load and vote), they leave the word, and the class whose key its arbiter holds books the
// tokens.  Keys grow with the round and the arbiters alternate between two sets, so nothing has to be cleared.  What bounds it
// is the length of that dependent chain, so it has no branch but the loop's (a finished slot and an empty word leave it), and
// the vote that ends the loop is taken while the next round's bids are on their way.
//
// Measured (B200), handles with at most four tiers and no equal scores (Lean, below; the others take Bidder): a round of one warp
// about 310 cycles, of several 510 (Bidder 390 and 650 to 860; one thread per slot and two barriers before that: 1000).  A lone
// warp takes three to five cycles per instruction, so what counts is their number; a reduction into shared memory takes two
// cycles per lane that meets another in its bank, so arbiters and holdings are laid out against that.  Matching stage, 256 ranks,
// 48 layers 967 -> 835 us, 32 ranks 67 -> 60 us, 64 ranks (where half the time is classes that move) 125 us as before.
//
// Equal scores.  Pairs whose fp32 scores are equal form a group and their candidates one set (the lowest rank wins, as in
// a dense scan).  A group with two win counts of one tier (a price step below the scores' last bit) keeps a rank that was
// won, so it is walked anew every round.
#pragma once

#include "taot_internal.cuh"

namespace taot_auction {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void red_max_u32(uint32_t addr, uint32_t v) { asm volatile("red.shared.max.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void red_and_u32(uint32_t addr, uint32_t v) { asm volatile("red.shared.and.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void red_or_u32(uint32_t addr, uint32_t v) { asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void red_add_u32(uint32_t addr, uint32_t v) { asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

// barrier over the first `nthreads` threads of the CTA (a multiple of 32): the warps that hold classes
__device__ __forceinline__ void bar_part(int nthreads) { asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory"); }

constexpr int kMaxWords = 8;  // words of 32 ranks of a rank set: R <= 256

// what the auction works on, in shared memory (nrem may be global)
struct Tables {
    uint32_t* arb;            // [2][R + W] best bid per rank, by parity of the round while there are several warps; a word's 32 begin a
                              // bank further on than the word's before, since bids go to the lowest ranks of their words
    uint32_t* avail;          // [W][dmax] ranks still holding tokens of the expert in column col
    uint32_t* lvl;            // [W][S + 1] ranks by win count
    const uint32_t* list;     // [nbid] pairs, best score first: tier | win count << 8, bit 31: the next one scores the same
    const uint32_t* ent;      // [ntiers][S + 1] the same by pair: list position << 16 | tie << 14 | class << 11 | win count,
                              // class = tiers that score strictly higher at this win count (orders the bids of a rank)
    const uint32_t* tm;       // [ntiers][W][tms] tier masks: by class, or by host if there is no room in shared memory
    const uint2* tw;          // [ntiers][S] by class: the word that holds the whole tier (-1: no one does) and its mask there
    const int32_t* slot_e;    // [S]
    int32_t* slot_a;          // [S + 1] tokens a slot still collects (S: 0)
    const uint2* rec;         // [S + 1] (lean) next slot of the class and the tokens it collects
    const uint16_t* nxt;      // [S + 1] next slot of the class, S: none (and S: S)
    const int32_t* dcol;      // [E] column of an expert
    int32_t* nrem;            // [D][RC] what each rank still holds of the expert in the column
    int32_t* X;               // [R][S] the plan of this layer (global)
    int32_t R, S, K, W, dmax, ntiers, tms;
    bool by_class;            // how tm goes (with a slot per rank both strides are the same)
    int32_t RC;               // odd in shared memory: bids for the same rank by different experts meet in no bank
    int32_t* idle;            // a word in global memory that nobody reads
};


// A bidder: one class, its state in registers, some pairs of which may have equal scores.
struct Bidder {
    static constexpr int NT = TAOT_MAX_TIERS, WM = kMaxWords;
    const Tables& t;
    int c = 0;                // class
    int ci = 0;               // its column of tm
    int s;                    // its lowest unfinished slot (S: none)
    int col = 0;
    bool live = false;
    int32_t A = 0;            // tokens slot s still collects
    uint32_t cw = 0u;         // candidates: word pw of the pair (or group) the class rests on
    int pw = 0;
    uint32_t low = 0u;        // key: class of the score, slot (inverted)
    uint32_t a_lv;            // shared address of lvl[pw][win count]
    uint32_t next[NT];        // by tier: the entry of its first pair not yet looked at; ~0: no member holds tokens any more
    uint32_t any = 0u;        // members of the tier that hold tokens, over the words seen at this pair
    int et = -1;              // the pair's tier; -1: not started
    uint32_t ev = 0u;         // its entry
    int gend = 0;             // a group: the list position after it; 0: a pair of its own
    bool one = true;          // no other word to look at
    bool again = false;       // a group with two win counts of one tier: no word survives a round

    __device__ __forceinline__ explicit Bidder(const Tables& tt) : t(tt), s(tt.S), a_lv(smem_u32(tt.lvl))
    {
#pragma unroll
        for (int k = 0; k < NT; ++k) next[k] = 0xFFFFFFFFu;
    }

    __device__ __forceinline__ void start(int cc, int ss)
    {
        c = cc; s = ss;
        ci = t.by_class ? cc : ss / t.K;
        live = true;
        col = t.dcol[t.slot_e[ss]];
        A = t.slot_a[ss];
        et = -1; cw = 0u; one = true; gend = 0; again = false;
#pragma unroll
        for (int k = 0; k < NT; ++k) next[k] = k < t.ntiers ? t.ent[k * (t.S + 1)] : 0xFFFFFFFFu;
    }

    __device__ __forceinline__ uint32_t after(uint32_t tier, uint32_t w) const
    {
        return (int)w < t.S ? t.ent[tier * (t.S + 1) + w + 1] : 0xFFFFFFFFu;
    }
    __device__ __forceinline__ void set_next(int tier, uint32_t v)
    {
#pragma unroll
        for (int k = 0; k < NT; ++k) next[k] = k == tier ? v : next[k];
    }

    // to the next word with candidates; cw == 0: there is none, ever
    __device__ __forceinline__ void walk()
    {
        const int S = t.S, W = t.W, LS = t.S + 1;
        uint32_t m_tw = 0u;                       // the tier's mask, if one word holds all of it
#pragma unroll 1
        for (;;) {
            if (!one && pw + 1 < W) {
                ++pw;
            } else {
                if (et >= 0 && any == 0u && gend == 0) set_next(et, 0xFFFFFFFFu);
                uint32_t best = next[0];
                int bt = 0;
#pragma unroll
                for (int k = 1; k < NT; ++k) {
                    bt = next[k] < best ? k : bt;
                    best = next[k] < best ? next[k] : best;
                }
                if (best == 0xFFFFFFFFu) { cw = 0u; return; }
                const uint2 tw = t.tw[bt * S + c];
                et = bt; ev = best;
                any = 0u;
                one = (int)tw.x >= 0;
                pw = one ? (int)tw.x : 0;
                m_tw = tw.y;
                set_next(bt, after((uint32_t)bt, best & 0x7FFu));
                again = false;
                gend = 0;
                if ((best >> 14) & 1u) {     // equal scores: all pairs of the group at once, word by word
                    int g = (int)(best >> 16);
                    uint32_t seen = 1u << bt, pr;
                    do {
                        pr = t.list[++g];
                        const uint32_t k = pr & 0xFFu;
                        again = again || ((seen >> k) & 1u);
                        seen |= 1u << k;
                        set_next((int)k, after(k, (pr >> 8) & 0xFFFu));
                    } while (pr >> 31);
                    gend = g + 1;
                    one = W == 1 && !again;
                    pw = 0;
                }
            }
            const uint32_t av = t.avail[pw * t.dmax + col];
            if (gend == 0) {
                const uint32_t* lv = t.lvl + pw * LS + (ev & 0x7FFu);
                const uint32_t h = (one ? m_tw : t.tm[(et * W + pw) * t.tms + ci]) & av;
                any |= h;
                cw = h & *lv;
                a_lv = smem_u32(lv);
                low = ((7u - ((ev >> 11) & 7u)) << 10) | (1023u - (uint32_t)s);
            } else {
                cw = 0u;
                for (int g = (int)(ev >> 16); g < gend; ++g) {
                    const uint32_t pr = t.list[g];
                    cw |= t.tm[((pr & 0xFFu) * W + pw) * t.tms + ci] & av & t.lvl[pw * LS + ((pr >> 8) & 0xFFFu)];
                }
            }
            if (cw) return;
        }
    }

    // a group: the pair of the rank `bit` of this word belongs to
    __device__ __forceinline__ void settle(int bit)
    {
        const int LS = t.S + 1;
        for (int g = (int)(ev >> 16); g < gend; ++g) {
            const uint32_t pr = t.list[g], w = (pr >> 8) & 0xFFFu;
            if (((t.tm[((pr & 0xFFu) * t.W + pw) * t.tms + ci] >> bit) & 1u) && (!again || ((t.lvl[pw * LS + w] >> bit) & 1u))) {
                a_lv = smem_u32(t.lvl + pw * LS + w);
                low = ((7u - ((t.ent[(pr & 0xFFu) * LS + w] >> 11) & 7u)) << 10) | (1023u - (uint32_t)s);
            }
        }
    }

    // ---- one round, in straight-line code for every lane: one without a bid sends a zero to some arbiter
    uint32_t key = 0u, a_mine = 0u, bitm = 0u;
    int rank = 0;
    int32_t have = 0;

    // the bid: the lowest rank of the word.  rk = round << 13, a_arb: the round's arbiters
    __device__ __forceinline__ void place(uint32_t rk, uint32_t a_arb)
    {
        const uint32_t c2 = A > 0 ? cw : 0u;            // (a finished slot waits for its class to move on)
        const int bit = c2 ? __ffs(c2) - 1 : 0;
        if (c2 && gend) settle(bit);
        const int word = pw < 0 ? 0 : pw;     // (a group that is walked anew stands before its first word)
        bitm = c2 & (0u - c2);
        rank = (word << 5) + bit;
        key = c2 ? rk | low : 0u;
        a_mine = a_arb + ((uint32_t)(rank + word) << 2);
        red_max_u32(a_mine, key);
        have = c2 ? t.nrem[col * t.RC + rank] : 0;
    }

    // Reads the round back.  The class that won its rank collects x = min(n, A); holdings, win count, price and plan follow.  The
    // rank holds tokens of the expert (its availability bit was set) and the slot still wants some, so x > 0 and the rank's bit
    // moves one word up in lvl; a (rank, slot) pair is served at most once.  True if the rank was won.
    __device__ __forceinline__ bool collect(uint32_t rk, uint32_t a_arb)
    {
        const bool mine = key != 0u && lds_u32(a_mine) == key;
        // (beyond the last rank the loads run into other shared data: bits no candidate word has)
        uint32_t gone = 0u;
        const uint32_t a_lane = a_arb + ((threadIdx.x & 31u) << 2);
#pragma unroll
        for (int w = 0; w < WM; ++w) {
            const uint32_t b = __ballot_sync(0xffffffffu, lds_u32(a_lane + 132u * w) >= rk);
            gone = w == pw ? b : gone;
        }
        cw = again ? 0u : cw & ~gone;
        const int32_t x = have < A ? have : A;
        const int32_t rest = have - x;
        // (a reduction or a store under a predicate costs 40 to 60 cycles more than one by every lane: the lanes that have not
        // won reduce with a neutral operand and store where nobody reads)
        const uint32_t on = mine ? bitm : 0u, off = mine && rest == 0 ? bitm : 0u;
        red_and_u32(a_lv, ~on);
        red_or_u32(a_lv + 4u, on);
        red_and_u32(smem_u32(t.avail + (rank >> 5) * t.dmax + col), ~off);
        if (mine) t.nrem[col * t.RC + rank] = rest;
        int32_t* const cell = mine ? t.X + (uint32_t)(rank * t.S + s) : t.idle;
        asm volatile("st.global.u32 [%0], %1;" ::"l"(cell), "r"(x) : "memory");
        A = mine ? A - x : A;
        return mine;
    }

    // Between rounds: a finished slot makes way for the next of its class, an empty word for the next one.
    __device__ __forceinline__ void move_on()
    {
        if (live && A <= 0) {
            t.slot_a[s] = 0;
            s = t.nxt[s];
            if (s == t.S) {
                live = false;
                cw = 0u;
            } else {
                A = t.slot_a[s];
                low = (low & ~1023u) | (1023u - (uint32_t)s);
            }
        }
        if (live && cw == 0u) {
            if (again) pw = -1;
            walk();
            live = cw != 0u;
        }
    }
    __device__ __forceinline__ bool must_move() const { return live && (cw == 0u || A <= 0); }
};

// At most 32 classes, one warp: rounds from `rd` on.  Returns the last round somebody won.
template <class B>
__device__ __forceinline__ uint32_t run_warp(B& b, uint32_t rd, uint32_t round_limit, uint32_t last)
{
    const Tables& t = b.t;
    const uint32_t a_arb = smem_u32(t.arb);
    while (rd <= round_limit) {
        __syncwarp();
        b.move_on();
        __syncwarp();
        if (!__any_sync(0xffffffffu, b.live)) break;
        b.place(rd << 13, a_arb);          // (again, for most: that changes nothing)
        bool stop;
        do {
            __syncwarp();
            b.collect(rd << 13, a_arb);
            ++rd;
            stop = b.must_move() || rd > round_limit;
            __syncwarp();                  // the arbiters have been read
            b.place(rd << 13, a_arb);
            stop = __any_sync(0xffffffffu, stop);
        } while (!stop);
        last = rd - 1u;
    }
    if (b.s != t.S) t.slot_a[b.s] = b.A;      // what is left uncollected
    return last;
}

// More than 32 classes: NP threads (whole warps), one class each, until at most 32 are left; those are listed in `hand` as
// class << 16 | slot and the number of the round they are to go on with is returned.  Every pass of the loop has one barrier.
// A pass in which some class has to walk does only that, between its barrier and the next, when nobody changes a shared
// set; the round's bids are then placed again (which changes nothing) together with the walkers'.
struct Control {
    uint32_t event[2];        // by parity of the pass: the pass, if a class has to walk or has finished
    uint32_t dead[2];         // classes that finished, by parity of the pass
    uint32_t last;            // the last round somebody won
    uint32_t handed;
    uint32_t hand[32];
};
template <class B>
__device__ __forceinline__ uint32_t run_block(B& b, const int NP, const int classes, const uint32_t round_limit, Control* ctl)
{
    const Tables& t = b.t;
    const int tid = threadIdx.x;
    const uint32_t a_arb = smem_u32(t.arb);
    const uint32_t a_ctl = smem_u32(ctl);
    uint32_t rd = 1u, pass = 1u, apar = 4u * (uint32_t)(t.R + t.W);      // round 1 takes the second set of arbiters
    uint32_t dead0 = 0u, dead1 = 0u;
    bool died = false;
    while (rd <= round_limit) {
        b.place(rd << 13, a_arb + apar);
        const uint32_t a_ev = a_ctl + ((pass & 1u) << 2);
        if (b.must_move() || died) {
            if (died) red_add_u32(a_ctl + 8u + ((pass & 1u) << 2), 1u);
            sts_u32(a_ev, pass);
        }
        died = false;
        __syncwarp();
        bar_part(NP);
        if (lds_u32(a_ev) == pass) {               // (the same answer in every thread)
            const uint32_t d = lds_u32(a_ev + 8u); // (its parity is counted again in the pass after next)
            if (pass & 1u) dead1 = d; else dead0 = d;
            ++pass;
            if (classes - (int)(dead0 + dead1) <= 32) break;
            const bool was = b.live;
            b.move_on();
            died = was && !b.live;
            continue;
        }
        ++pass;
        if (b.collect(rd << 13, a_arb + apar)) sts_u32(a_ctl + 16u, rd);
        apar ^= 4u * (uint32_t)(t.R + t.W);
        ++rd;
    }
    if (b.s != t.S) t.slot_a[b.s] = b.A;
    if (b.live && rd <= round_limit) ctl->hand[atomicAdd(&ctl->handed, 1u)] = ((uint32_t)b.c << 16) | (uint32_t)b.s;
    return rd;
}

// ---- Handles with at most four tiers and no equal scores.
//
// The same rounds with fewer instructions: win counts and availability, which nobody reads but a class that walks, follow in one go
// before the next walk; a finished slot makes way for the next of its class in place; the rounds are left only where a class's word
// is empty or its last slot finished.  (Several classes per lane instead of several warps: 200 cycles a round for each, 1000 at
// four; the loads of the next round ahead of the vote that ends the rounds: 60 cycles a round slower.)
// NT: 2 or 4 tiers (walking goes through all of them: 32 ranks 67 -> 60 us with two); NSM: nrem is in shared memory; WM: most words
// of 32 ranks.
__device__ __forceinline__ void red_max_if(bool on, uint32_t addr, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p red.shared.max.u32 [%0], %1; }" ::"r"(addr), "r"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void sts_if(bool on, uint32_t addr, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.shared.u32 [%0], %1; }" ::"r"(addr), "r"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void stg_if(bool on, int32_t* addr, int32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.global.u32 [%0], %1; }" ::"l"(addr), "r"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ uint2 lds_u64(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
    return v;
}

template <int NT, bool NSM, int WM>
struct Lean {
    const Tables& t;
    const uint32_t a_arb, a_rec, a_slot, a_lvl, a_avail, a_ent, a_tw, S, LS, dmax;      // shared addresses of the tables
    // what a round needs
    bool act = false;         // the thread has a class that is not through
    uint32_t cw = 0u;         // its candidates: ranks of word pw; 0 where there is no class
    uint32_t A = 0u;          // tokens the slot in front still collects
    uint32_t s = 0u, low = 0u;
    uint32_t a_word;          // shared address of the word's arbiters
    uint32_t cell = 0u;       // nrem: index (NSM: shared address) of the column's first rank of the word
    uint32_t x0 = 0u;         // X: index of the word's first rank and the slot
    uint32_t on = 0u, off = 0u;       // ranks of the word won by the class since the sets were last brought up to date; those now empty
    // what a walk needs
    uint32_t next[NT], ev = 0u;
    uint32_t a_tw_c = 0u, a_av_c = 0u, cell_c = 0u;   // the class's and its column's places in the tables
    uint32_t a_lv = 0u, a_av = 0u;                     // of the pair and word it rests on
    int et = -1, pw = 0, c = 0;
    bool one = true;

    __device__ __forceinline__ explicit Lean(const Tables& tt)
        : t(tt), a_arb(smem_u32(tt.arb)), a_rec(smem_u32(tt.rec)), a_slot(smem_u32(tt.slot_a)), a_lvl(smem_u32(tt.lvl)),
          a_avail(smem_u32(tt.avail)), a_ent(smem_u32(tt.ent)), a_tw(smem_u32(tt.tw)), S((uint32_t)tt.S),
          LS(4u * (uint32_t)tt.S + 4u), dmax(4u * (uint32_t)tt.dmax), a_word(a_arb)
    {
#pragma unroll
        for (int k = 0; k < NT; ++k) next[k] = 0xFFFFFFFFu;
        if (NSM) cell = smem_u32(tt.nrem);
    }
    __device__ __forceinline__ void start(int cc, int ss)
    {
        c = cc;
        s = (uint32_t)ss;
        low = 1023u - s;
        const uint32_t col = (uint32_t)t.dcol[t.slot_e[ss]];
        a_tw_c = a_tw + 8u * (uint32_t)cc;
        a_av_c = a_avail + 4u * col;
        cell_c = NSM ? smem_u32(t.nrem) + 4u * col * (uint32_t)t.RC : col * (uint32_t)t.RC;
        A = lds_u32(a_slot + 4u * s);
        act = A != 0u;
#pragma unroll
        for (int k = 0; k < NT; ++k) next[k] = k < t.ntiers ? lds_u32(a_ent + (uint32_t)k * LS) : 0xFFFFFFFFu;
    }
    // win counts and availability
    __device__ __forceinline__ void settle()
    {
        if (on) {
            red_and_u32(a_lv, ~on);
            red_or_u32(a_lv + 4u, on);
            if (off) red_and_u32(a_av, ~off);
            on = off = 0u;
        }
    }
    // to the next word with candidates; cw == 0: there is none, ever
    __device__ __forceinline__ void walk()
    {
        int first = pw + 1;                           // first word to look at
        uint32_t held = 1u, m = 0u;                   // held: members of the tier that hold tokens; only 0 matters
#pragma unroll 1
        for (;;) {
            const uint32_t a_wins = a_lvl + 4u * (ev & 0x7FFu);
            if (WM > 1 && et >= 0 && !one) {          // the tier's words from `first` on
                const int ci = t.by_class ? c : (int)(1023u - (low & 1023u)) / t.K;
                const uint32_t* tm = t.tm + et * t.W * t.tms + ci;
#pragma unroll 1
                for (int w = first; w < t.W; ++w) {
                    const uint32_t h = tm[w * t.tms] & lds_u32(a_av_c + (uint32_t)w * dmax);
                    held |= h;
                    cw = h & lds_u32(a_wins + (uint32_t)w * LS);
                    pw = w;
                    if (cw) break;
                }
            } else if (first == 0) {
                held = m & lds_u32(a_av_c + (uint32_t)pw * dmax);
                cw = held & lds_u32(a_wins + (uint32_t)pw * LS);
            }
            if (cw) break;
#pragma unroll
            for (int k = 0; k < NT; ++k) next[k] = k == et && held == 0u ? 0xFFFFFFFFu : next[k];
            uint32_t best = next[0];
            et = 0;
#pragma unroll
            for (int k = 1; k < NT; ++k) {
                et = next[k] < best ? k : et;
                best = next[k] < best ? next[k] : best;
            }
            if (best == 0xFFFFFFFFu) return;
            ev = best;
            const uint32_t w = best & 0x7FFu;
            const uint2 tw = lds_u64(a_tw_c + 8u * S * (uint32_t)et);
            const uint32_t after = w < S ? lds_u32(a_ent + (uint32_t)et * LS + 4u * w + 4u) : 0xFFFFFFFFu;
#pragma unroll
            for (int k = 0; k < NT; ++k) next[k] = k == et ? after : next[k];
            one = WM == 1 || (int)tw.x >= 0;
            pw = WM > 1 && one ? (int)tw.x : 0;
            m = tw.y;
            first = 0;
            held = 0u;
        }
        low = ((7u - ((ev >> 11) & 7u)) << 10) | (low & 1023u);
        a_lv = a_lvl + 4u * (ev & 0x7FFu) + (uint32_t)pw * LS;
        a_av = a_av_c + (uint32_t)pw * dmax;
        a_word = a_arb + 132u * (uint32_t)pw;
        cell = cell_c + (NSM ? 128u : 32u) * (uint32_t)pw;
        x0 = 32u * (uint32_t)pw * S + s;
    }
    // a class without candidates, after settle() of all: on to its next word, or through
    __device__ __forceinline__ void move_on()
    {
        if (A != 0u) walk();
        act = cw != 0u;
        if (!act && A != 0u) {
            sts_u32(a_slot + 4u * s, A);              // (what is left uncollected)
            A = 0u;
        }
    }

    uint32_t bitm = 0u, bit = 0u, key = 0u, have = 0u, a_mine = 0u;

    // the bid: the lowest rank of the word.  rk = round << 13, par: offset of the round's arbiters
    __device__ __forceinline__ void place(uint32_t rk, uint32_t par)
    {
        bitm = cw & (0u - cw);
        asm("bfind.u32 %0, %1;" : "=r"(bit) : "r"(bitm));           // (no candidates: -1, the word before, which is not used)
        key = rk | low;
        a_mine = a_word + par + 4u * bit;
        red_max_if(cw != 0u, a_mine, key);
        if (NSM) have = lds_u32(cell + 4u * bit);
        else have = cw ? (uint32_t)t.nrem[cell + bit] : 0u;
    }
    // Reads the round back.  The class that won its rank collects x = min(n, A) > 0 (the rank holds tokens of the expert, its
    // availability bit was set, and the slot still wants some).
    __device__ __forceinline__ void collect(uint32_t rk, uint32_t par)
    {
        const uint32_t won = lds_u32(a_mine);
        const uint2 then = lds_u64(a_rec + 8u * s);
        const uint32_t a_lane = a_arb + par + ((threadIdx.x & 31u) << 2);
        uint32_t g[WM];
        // (beyond the last rank the loads run into other shared data: bits no candidate word has)
#pragma unroll
        for (int w = 0; w < WM; ++w) g[w] = lds_u32(a_lane + 132u * w);
#pragma unroll
        for (int w = 0; w < WM; ++w) g[w] = __ballot_sync(0xffffffffu, g[w] >= rk);
#pragma unroll
        for (int h = 1; h < WM; h <<= 1)
#pragma unroll
            for (int w = 0; w < WM; w += 2 * h) g[w] = pw & h ? g[w + h] : g[w];
        const bool mine = (won == key) & (cw != 0u);
        const uint32_t x = have < A ? have : A, rest = have - x;
        on |= mine ? bitm : 0u;
        off |= mine & (rest == 0u) ? bitm : 0u;
        if (NSM) sts_if(mine, cell + 4u * bit, rest);
        else stg_if(mine, t.nrem + (cell + bit), (int32_t)rest);
        stg_if(mine, t.X + (x0 + bit * S), (int32_t)x);
        A -= mine ? x : 0u;
        const bool done = mine & (A == 0u);           // the next of the class (S, with nothing to collect, behind the last)
        sts_if(done, a_slot + 4u * s, 0u);
        const uint32_t step = done ? then.x - s : 0u;
        s += step; low -= step; x0 += step;
        A = done ? then.y : A;
        cw = A != 0u ? cw & ~g[0] : 0u;
    }
};

template <class B>
__device__ __forceinline__ uint32_t run_warp_lean(B& b, uint32_t rd, uint32_t round_limit, uint32_t last)
{
    while (rd <= round_limit) {
        __syncwarp();
        b.settle();
        __syncwarp();
        if (b.act && b.cw == 0u) b.move_on();
        __syncwarp();
        if (!__any_sync(0xffffffffu, b.act)) break;
        b.place(rd << 13, 0u);                        // (again, for most: that changes nothing)
        do {
            __syncwarp();
            b.collect(rd << 13, 0u);
            ++rd;
            __syncwarp();                             // the arbiters have been read
            b.place(rd << 13, 0u);
        } while (!__any_sync(0xffffffffu, (b.act & (b.cw == 0u)) | (rd > round_limit)));
        last = rd - 1u;
    }
    if (b.act && b.A != 0u) b.t.slot_a[b.s] = (int32_t)b.A;
    return last;
}

// More than 32 classes, a barrier a pass.  A pass in which some class has none but its next word or its end before it does only that
// (and has one more).
template <class B>
__device__ __forceinline__ uint32_t run_block_lean(B& b, const int NP, const int classes, const uint32_t round_limit, Control* ctl)
{
    const uint32_t a_ctl = smem_u32(ctl), flip = 4u * (uint32_t)(b.t.R + b.t.W);
    uint32_t rd = 1u, pass = 1u, par = flip;          // round 1 takes the second set of arbiters
    bool moved = false;
    while (rd <= round_limit) {
        b.place(rd << 13, par);
        const uint32_t a_ev = a_ctl + ((pass & 1u) << 2);
        if (b.act && b.cw == 0u) sts_u32(a_ev, pass);
        __syncwarp();
        bar_part(NP);
        if (moved && classes - (int)lds_u32(a_ctl + 8u) <= 32) break;         // (the same answer in every thread)
        moved = lds_u32(a_ev) == pass;
        ++pass;
        if (moved) {
            b.settle();
            bar_part(NP);
            if (b.act && b.cw == 0u) {
                b.move_on();
                if (!b.act) red_add_u32(a_ctl + 8u, 1u);
            }
            continue;
        }
        b.collect(rd << 13, par);
        if (threadIdx.x == 0) sts_u32(a_ctl + 16u, rd);
        par ^= flip;
        ++rd;
    }
    if (b.act) {
        b.t.slot_a[b.s] = (int32_t)b.A;
        if (rd <= round_limit) ctl->hand[atomicAdd(&ctl->handed, 1u)] = ((uint32_t)b.c << 16) | b.s;
    }
    return rd;
}

}  // namespace taot_auction
