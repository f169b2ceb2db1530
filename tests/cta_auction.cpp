// The rounds of the auction in one warp (auction.cuh), on tables that the caller has made, on a CPU.
#include "cta.h"

#include "auction.cuh"

using namespace taot_auction;

namespace {

struct Sizes { int32_t R, S, K, W, dmax, ntiers, classes; };
Sizes n;
// what a layer starts from, by name as in Tables; `lead`: the first slot of each class
const uint32_t *avail, *lvl, *list, *ent, *tm, *rec, *tw;
const int32_t *slot_e, *slot_a, *dcol, *nrem, *lead;
const uint16_t* nxt;
int32_t *X, *left, *last;

template <class T>
T* place(unsigned char*& at, const T* from, size_t count)
{
    T* to = reinterpret_cast<T*>(at);
    at += (sizeof(T) * count + 15) & ~(size_t)15;
    for (size_t i = cta::me; from && i < count; i += cta::count) to[i] = from[i];
    return to;
}

template <class B, bool LEAN>
void kernel()
{
    unsigned char* at = cta::dynamic + 64;         // (a class without candidates reads the word before the first)
    Tables t;
    const size_t pairs = (size_t)n.ntiers * (n.S + 1), cols = n.R | 1;
    t.R = n.R; t.S = n.S; t.K = n.K; t.W = n.W; t.dmax = n.dmax; t.ntiers = n.ntiers; t.tms = n.S; t.by_class = true; t.RC = (int32_t)cols;
    t.arb = place<uint32_t>(at, nullptr, 2 * (n.R + n.W) + 33 * kMaxWords);      // (a round reads on behind the last rank's)
    for (int i = cta::me; i < 2 * (n.R + n.W); i += cta::count) t.arb[i] = 0u;
    t.avail = place(at, avail, (size_t)n.W * n.dmax);
    t.lvl = place(at, lvl, (size_t)n.W * (n.S + 1));
    t.list = place(at, list, pairs);
    t.ent = place(at, ent, pairs);
    t.tm = place(at, tm, (size_t)n.ntiers * n.W * n.S);
    t.tw = reinterpret_cast<uint2*>(place(at, tw, 2 * (size_t)n.ntiers * n.S));
    t.slot_e = place(at, slot_e, n.S);
    t.slot_a = place(at, slot_a, n.S + 1);
    t.rec = reinterpret_cast<uint2*>(place(at, rec, 2 * (size_t)(n.S + 1)));
    t.nxt = place(at, nxt, n.S + 1);
    t.dcol = place(at, dcol, n.dmax);
    t.nrem = place(at, nrem, (size_t)n.dmax * cols);
    t.X = X;
    t.idle = left + n.S;
    __syncthreads();
    B b(t);
    if (cta::me < n.classes) b.start(cta::me, lead[cta::me]);
    __syncwarp();
    uint32_t end;
    if constexpr (LEAN) end = run_warp_lean(b, 1u, n.R * n.S + n.S, 0u);
    else end = run_warp(b, 1u, n.R * n.S + n.S, 0u);
    __syncthreads();
    if (cta::me == 0) *last = (int32_t)end;
    for (int i = cta::me; i < n.S; i += cta::count) left[i] = t.slot_a[i];
}

}  // namespace

extern "C" void cta_auction(int lean, const Sizes* sizes, const void* const* in, int32_t* plan, int32_t* slots_left, int32_t* rounds)
{
    n = *sizes;
    int i = 0;
    const auto next = [&](auto& p) { p = static_cast<std::remove_reference_t<decltype(p)>>(in[i++]); };
    next(avail); next(lvl); next(list); next(ent); next(tm); next(tw); next(slot_e); next(slot_a); next(rec); next(nxt); next(dcol); next(nrem); next(lead);
    X = plan; left = slots_left; last = rounds;
    if (lean) cta::launch(0, 32, [] { kernel<Lean<4, true, 2>, true>(); });
    else cta::launch(0, 32, [] { kernel<Bidder, false>(); });
}
