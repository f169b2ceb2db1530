// The threads of cta.h: fibers, meetings, vector clocks.  Compiled without -fsanitize=thread.
#include "cta.h"

#include <stdio.h>
#include <stdlib.h>
#include <ucontext.h>

#include <map>
#include <tuple>
#include <unordered_map>
#include <vector>

namespace cta {

int me, count, block, blocks;
alignas(1024) unsigned char dynamic[227 * 1024];

namespace {

constexpr int kMax = 1024;
constexpr size_t kStack = 256 * 1024;

struct Thread {
    ucontext_t ctx;
    std::vector<uint32_t> clock;
    bool done = false;
};
struct Meeting {
    std::vector<int> in;                 // who has come
    uint64_t round = 0;                  // how often it has taken place
    uint64_t value[2][kMax];             // what they brought, by parity of the round
};
struct At { int thread; uint32_t clock; };
struct Word { At write = {-1, 0}; std::vector<At> read, atomic; };      // the last write, reads and atomic operations since
enum Kind { kRead, kWrite, kAtomic };

char* stacks = static_cast<char*>(aligned_alloc(4096, kMax * kStack));
std::vector<Thread> threads;
std::map<std::tuple<int, int, int>, Meeting> meetings;
std::unordered_map<uintptr_t, Word> words;
ucontext_t host;
void (*body)();
long progress, races, stuck;
char first[256];

void yield() { swapcontext(&threads[me].ctx, &host); }

void run()
{
    body();
    threads[me].done = true;
    ++progress;
    for (;;) yield();
}

void access(uintptr_t p, size_t bytes, Kind kind)
{
    if (me >= count || p - (uintptr_t)stacks < kMax * kStack) return;       // between launches; a thread's own
    const std::vector<uint32_t>& clock = threads[me].clock;
    const auto unordered = [&](const At& x) { return x.thread >= 0 && x.thread != me && x.clock > clock[x.thread]; };
    for (uintptr_t w = p / 4; w <= (p + bytes - 1) / 4; ++w) {
        Word& x = words[w];
        const char* other = nullptr;
        int by = -1;
        // (one store instruction of a warp: one of its threads performs the write)
        if (unordered(x.write) && !(kind == kWrite && x.write.thread / 32 == me / 32)) { by = x.write.thread; other = "writes"; }
        if (kind != kRead)
            for (const At& r : x.read) if (unordered(r)) { by = r.thread; other = "reads"; }
        if (kind != kAtomic)
            for (const At& r : x.atomic) if (unordered(r)) { by = r.thread; other = "updates"; }
        if (other && races++ == 0)
            snprintf(first, sizeof first, "thread %d %s a word that thread %d %s, and no wait lies between", me,
                     kind == kRead ? "reads" : (kind == kWrite ? "writes" : "updates"), by, other);
        if (kind == kWrite) {
            x.write = {me, clock[me]};
            x.read.clear();
            x.atomic.clear();
            continue;
        }
        std::vector<At>& seen = kind == kRead ? x.read : x.atomic;
        size_t q = 0;
        while (q < seen.size() && seen[q].thread != me) ++q;
        if (q < seen.size()) seen[q].clock = clock[me];
        else seen.push_back({me, clock[me]});
    }
}

}  // namespace

void atomic(const void* p) { access((uintptr_t)p, 4, kAtomic); }

const uint64_t* meet(int kind, int id, int n, uint64_t mine, bool orders)
{
    Meeting& m = meetings[{kind, id, n}];
    const uint64_t round = m.round;
    m.value[round & 1][me] = mine;
    m.in.push_back(me);
    ++progress;
    if ((int)m.in.size() == n) {
        if (orders) {
            std::vector<uint32_t> all(count, 0u);
            for (int t : m.in)
                for (int k = 0; k < count; ++k) all[k] = threads[t].clock[k] > all[k] ? threads[t].clock[k] : all[k];
            for (int t : m.in) { threads[t].clock = all; ++threads[t].clock[t]; }
        }
        m.in.clear();
        ++m.round;
    } else {
        while (m.round == round) yield();
    }
    return m.value[round & 1];
}

void launch(int b, int n, void (*f)())
{
    block = b;
    count = n;
    body = f;
    threads.assign(n, Thread());
    meetings.clear();
    words.clear();
    memset(dynamic, 0xa5, sizeof dynamic);
    for (int t = 0; t < n; ++t) {
        Thread& x = threads[t];
        x.clock.assign(n, 0u);
        x.clock[t] = 1u;
        getcontext(&x.ctx);
        x.ctx.uc_stack.ss_sp = stacks + t * kStack;
        x.ctx.uc_stack.ss_size = kStack;
        makecontext(&x.ctx, run, 0);
    }
    for (bool left = true; left;) {
        left = false;
        const long before = progress;
        for (me = 0; me < n; ++me)
            if (!threads[me].done) {
                swapcontext(&host, &threads[me].ctx);
                left |= !threads[me].done;
            }
        if (left && progress == before) { ++stuck; return; }      // (me is `n` here: no thread)
    }
}

}  // namespace cta

extern "C" {

long cta_races() { return cta::races; }
long cta_stuck() { return cta::stuck; }
const char* cta_first() { return cta::first; }
void cta_reset() { cta::races = cta::stuck = 0; cta::first[0] = 0; }

// what the compiler calls before an access
#define CTA_HOOK(N)                                                            \
    void __tsan_read##N(void* p) { cta::access((uintptr_t)p, N, cta::kRead); }      \
    void __tsan_write##N(void* p) { cta::access((uintptr_t)p, N, cta::kWrite); }      \
    void __tsan_unaligned_read##N(void* p) { cta::access((uintptr_t)p, N, cta::kRead); }  \
    void __tsan_unaligned_write##N(void* p) { cta::access((uintptr_t)p, N, cta::kWrite); }
CTA_HOOK(1)
CTA_HOOK(2)
CTA_HOOK(4)
CTA_HOOK(8)
CTA_HOOK(16)
void __tsan_read_range(void* p, size_t n) { cta::access((uintptr_t)p, n, cta::kRead); }
void __tsan_write_range(void* p, size_t n) { cta::access((uintptr_t)p, n, cta::kWrite); }
void __tsan_func_entry(void*) {}
void __tsan_func_exit() {}
void __tsan_init() {}

}  // extern "C"
