// One CTA of a kernel on a CPU, its threads as fibers, and a check of the order of their accesses to memory that they share.
//
// The kernel's source is compiled by g++ as it stands (PTX statements replaced, see cta.py) with -fsanitize=thread, which puts a call
// before each load and store; those calls are answered in cta.cpp, not by a runtime of the compiler's.  Every thread has a vector
// clock.  Barriers and __syncwarp() join the clocks of those that meet; votes and shuffles let their threads meet but order no
// memory.  Two accesses to a 4-byte word, one of them a write, by threads neither of which has the other's behind it are a race,
// whether or not they would meet in time.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

namespace cta {

extern int me, count;                    // the thread that runs, the threads of the CTA
extern int block, blocks;                // its place in the grid, the CTAs of the grid
extern unsigned char dynamic[];          // shared memory whose size the launch gives

// The `n` threads that come to (kind, id) meet; each brings a value and learns where all of them are, by thread of the CTA.
const uint64_t* meet(int kind, int id, int n, uint64_t mine, bool orders);
// An atomic operation on a word: in no race with others of its kind.
void atomic(const void* p);
// Runs f by n threads.  Threads that come to no end (each waits for others) are given up.
void launch(int b, int n, void (*f)());

inline void bar(int id, int n) { meet(0, id, n, 0, true); }
inline bool bar_or(int id, int n, bool p)                        // (by the first n threads)
{
    const uint64_t* v = meet(1, id, n, p, true);
    bool r = false;
    for (int t = 0; t < n; ++t) r |= v[t] != 0;
    return r;
}
inline const uint64_t* warp(uint64_t mine, bool orders = false) { return meet(2, me / 32, 32, mine, orders) + me / 32 * 32; }

// the address that __cvta_generic_to_shared() gave for a place in `dynamic`
inline void* shared(uint32_t a) { return dynamic + (uint32_t)(a - (uint32_t)(uintptr_t)dynamic); }

// two floats in a 64-bit register
inline float low(uint64_t x) { float f; memcpy(&f, &x, 4); return f; }
inline float high(uint64_t x) { x >>= 32; float f; memcpy(&f, &x, 4); return f; }
inline uint64_t pack(float a, float b) { uint32_t l, h; memcpy(&l, &a, 4); memcpy(&h, &b, 4); return (uint64_t)h << 32 | l; }
// not a number, if one of them is
inline float least(float a, float b) { return a != a || a < b ? a : b; }
inline float largest(float a, float b) { return a != a || a > b ? a : b; }
inline float least(float a, float b, float c) { return least(least(a, b), c); }
inline float largest(float a, float b, float c) { return largest(largest(a, b), c); }

struct Now { const int* p; operator unsigned() const { return (unsigned)*p; } };
struct Index { Now x; };

}  // namespace cta

// ---- the device's names
#undef __shared__
#define __shared__ static
#define __launch_bounds__(...)
const cta::Index threadIdx{{&cta::me}}, blockIdx{{&cta::block}}, blockDim{{&cta::count}}, gridDim{{&cta::blocks}};

inline void __syncthreads() { cta::bar(0, cta::count); }
inline int __syncthreads_or(int p) { return cta::bar_or(0, cta::count, p != 0); }
inline void __syncwarp(unsigned = ~0u) { cta::warp(0, true); }
template <class T>
T __shfl_xor_sync(unsigned, T v, int o)
{
    uint64_t x = 0;
    memcpy(&x, &v, sizeof v);
    x = cta::warp(x)[cta::me % 32 ^ o];
    memcpy(&v, &x, sizeof v);
    return v;
}
inline unsigned __ballot_sync(unsigned, bool p)
{
    const uint64_t* v = cta::warp(p);
    unsigned r = 0u;
    for (int k = 0; k < 32; ++k) r |= (unsigned)v[k] << k;
    return r;
}
template <class T>
T __shfl_sync(unsigned, T v, int lane)
{
    uint64_t x = 0;
    memcpy(&x, &v, sizeof v);
    x = cta::warp(x)[lane & 31];
    memcpy(&v, &x, sizeof v);
    return v;
}
inline unsigned __reduce_add_sync(unsigned, unsigned x)
{
    const uint64_t* v = cta::warp(x);
    unsigned r = 0u;
    for (int k = 0; k < 32; ++k) r += (unsigned)v[k];
    return r;
}
inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0u; }
inline bool __all_sync(unsigned m, bool p) { return __ballot_sync(m, p) == ~0u; }
inline int min(int a, int b) { return a < b ? a : b; }
inline unsigned __reduce_or_sync(unsigned, unsigned x)
{
    const uint64_t* v = cta::warp(x);
    unsigned r = 0u;
    for (int k = 0; k < 32; ++k) r |= (unsigned)v[k];
    return r;
}
inline int __reduce_min_sync(unsigned, int x)
{
    const uint64_t* v = cta::warp((uint32_t)x);
    int r = (int)v[0];
    for (int k = 1; k < 32; ++k) r = (int)v[k] < r ? (int)v[k] : r;
    return r;
}
inline unsigned __vcmpeq4(unsigned a, unsigned b)
{
    unsigned r = 0u;
    for (int k = 0; k < 32; k += 8) r |= (a >> k & 255u) == (b >> k & 255u) ? 255u << k : 0u;
    return r;
}
inline uint32_t __cvta_generic_to_shared(const void* p) { return (uint32_t)(uintptr_t)p; }
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __ffs(int x) { return __builtin_ffs(x); }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline uint32_t __float_as_uint(float x) { uint32_t r; memcpy(&r, &x, 4); return r; }
inline int __float_as_int(float x) { return (int)__float_as_uint(x); }
inline float __int_as_float(int x) { float r; memcpy(&r, &x, 4); return r; }
#define CTA_ATOMIC(NAME, NEW)                                                          \
    template <class T, class U>                                                        \
    __attribute__((no_sanitize("thread"))) T NAME(T* p, U v)                           \
    {                                                                                  \
        cta::atomic(p);                                                                \
        const T old = *p;                                                              \
        *p = NEW;                                                                      \
        return old;                                                                    \
    }
CTA_ATOMIC(atomicOr, old | (T)v)
CTA_ATOMIC(atomicAdd, old + (T)v)
CTA_ATOMIC(atomicAnd, old & (T)v)
CTA_ATOMIC(atomicMax, old > (T)v ? old : (T)v)
