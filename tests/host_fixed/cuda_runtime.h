// The part of CUDA's device language that the fixed-point step code uses, for a host build: the
// threads of one block run as fibers of one host thread, and every warp or block operation waits
// until all the threads it names have come to it.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>
#include <ucontext.h>

#include <algorithm>
#include <map>
#include <utility>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __constant__
#define __shared__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))

using std::isfinite;
using std::max;
using std::min;

struct float2 { float x, y; };
struct double2 { double x, y; };
struct int2 { int x, y; };
struct int4 { int x, y, z, w; };
inline float2 make_float2(float x, float y) { return {x, y}; }
inline double2 make_double2(double x, double y) { return {x, y}; }
inline int2 make_int2(int x, int y) { return {x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
struct uint3_ { unsigned x, y, z; };
typedef struct stream_t* cudaStream_t;
enum cudaError_t { cudaSuccess };

template <typename To, typename From>
inline To bits_as(From v)
{
    static_assert(sizeof(To) == sizeof(From), "size");
    To r;
    memcpy(&r, &v, sizeof r);
    return r;
}
inline int __double2hiint(double v) { return (int)(bits_as<uint64_t>(v) >> 32); }
inline int __double2loint(double v) { return (int)bits_as<uint64_t>(v); }
inline double __hiloint2double(int h, int l)
{
    return bits_as<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l);
}
inline double __longlong_as_double(long long v) { return bits_as<double>(v); }
inline long long __double_as_longlong(double v) { return bits_as<long long>(v); }
inline float __int_as_float(int v) { return bits_as<float>(v); }
inline unsigned __float_as_uint(float v) { return bits_as<unsigned>(v); }
inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s)
{
    return (unsigned)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32);
}
inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s)
{
    return (unsigned)((((uint64_t)hi << 32) | lo) >> (s & 31));
}
template <typename V> inline V __ldg(const V* p) { return *p; }
template <typename V> inline void __stcs(V* p, V v) { *p = v; }
inline size_t __cvta_generic_to_shared(const void*) { return 0; }
inline size_t __cvta_generic_to_global(const void* p) { return (size_t)p; }

// ---- fibers -----------------------------------------------------------------------------
namespace host {

struct Meeting {          // one operation of a set of threads
    int arrived = 0;
    long long turn = 0;
    unsigned in[32] = {}, out[32] = {};
    unsigned any = 0, any_out = 0;
};
struct Fiber {
    ucontext_t ctx;
    std::vector<char> stack;
    bool done = false;
};
inline std::vector<Fiber> fibers;
inline ucontext_t scheduler;
inline int current = 0;
inline std::map<std::pair<int, unsigned>, Meeting> meetings;   // (warp, lanes) or (-1, 0): the block

inline void yield() { swapcontext(&fibers[current].ctx, &scheduler); }
// wait for the `count` threads of a meeting; v: this thread's value
inline Meeting& meet(int warp, unsigned lanes, int count, unsigned v)
{
    Meeting& m = meetings[{warp, lanes}];
    const long long turn = m.turn;
    m.in[current & 31] = v;
    m.any |= v;
    if (++m.arrived == count) {
        memcpy(m.out, m.in, sizeof m.out);
        m.any_out = m.any;
        m.any = 0;
        m.arrived = 0;
        ++m.turn;
    } else {
        while (m.turn == turn)
            yield();
    }
    return m;
}
inline Meeting& meet_warp(unsigned lanes, unsigned v)
{
    return meet(current / 32, lanes, __builtin_popcount(lanes), v);
}
template <typename F>
void trampoline(unsigned lo, unsigned hi)
{
    (*(F*)((uintptr_t)hi << 32 | lo))();
    fibers[current].done = true;
    yield();
}
// f() on every thread of a block
template <typename F>
void run_block(int threads, F f)
{
    if ((int)fibers.size() < threads)
        fibers.resize(threads);
    meetings.clear();
    for (int i = 0; i < threads; ++i) {
        Fiber& b = fibers[i];
        b.done = false;
        if (b.stack.empty())
            b.stack.resize(256 << 10);
        getcontext(&b.ctx);
        b.ctx.uc_stack.ss_sp = b.stack.data();
        b.ctx.uc_stack.ss_size = b.stack.size();
        b.ctx.uc_link = nullptr;
        const uintptr_t p = (uintptr_t)&f;
        makecontext(&b.ctx, (void (*)())trampoline<F>, 2, (unsigned)p, (unsigned)(p >> 32));
    }
    for (bool left = true; left;) {
        left = false;
        for (current = 0; current < threads; ++current)
            if (!fibers[current].done) {
                left = true;
                swapcontext(&scheduler, &fibers[current].ctx);
            }
    }
}
struct ThreadIdx {
    struct X {
        operator int() const { return current; }
    } x;
};

}  // namespace host

inline host::ThreadIdx threadIdx;
inline uint3_ blockIdx, blockDim, gridDim;

inline int host_threads();
inline void __syncthreads() { host::meet(-1, 0, host_threads(), 0); }
inline int __syncthreads_or(int v) { return host::meet(-1, 0, host_threads(), v != 0).any_out != 0; }
inline void __syncwarp() { host::meet_warp(0xffffffffu, 0); }
inline unsigned __shfl_xor_sync(unsigned m, unsigned v, int o)
{
    return host::meet_warp(m, v).out[(host::current & 31) ^ o];
}
inline unsigned __reduce_max_sync(unsigned m, unsigned v)
{
    const auto& r = host::meet_warp(m, v).out;
    return *std::max_element(r, r + 32);
}
inline unsigned __reduce_add_sync(unsigned m, unsigned v)
{
    unsigned s = 0;
    for (unsigned x : host::meet_warp(m, v).out)
        s += x;
    return s;
}
inline int __any_sync(unsigned m, int v) { return host::meet_warp(m, v != 0).any_out != 0; }
