// A CUDA block on the host: every thread is a fiber that runs until it meets a barrier or a warp
// collective, so a test picks the order in which the threads go on from one. A barrier that
// threads of a block reach from different source lines is reported. Enough of the language for
// kernels that use block barriers, warp shuffles and atomics.
#pragma once
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <functional>
#include <vector>
#include <ucontext.h>
#include <cuda_runtime.h>

#undef __global__
#undef __device__
#undef __host__
#undef __shared__
#undef __constant__
#undef __forceinline__
#undef __launch_bounds__
#define __global__ static
#define __device__
#define __host__
#define __shared__ static
#define __constant__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define asm                    // device assembly is left out: `asm volatile(...)` becomes nothing
#define volatile(...)

namespace emu {

constexpr size_t STACK = 64 << 10;
struct Fiber {
    ucontext_t ctx;
    std::vector<char> stack = std::vector<char>(STACK);
    int at = 0;                // 0 running, 1 at a block barrier, 2 at a warp collective, 3 done
    int line = 0;
    uint64_t value = 0;
};
inline std::vector<Fiber> fibers;
inline ucontext_t scheduler;
inline int self;
inline int mixed;              // barriers met from more than one line
inline uint64_t reduced;
inline std::function<void()> body;

inline uint3 threadIdx, blockIdx;
inline dim3 blockDim, gridDim;

inline void wait_at(int kind, int line, uint64_t v) {
    Fiber& f = fibers[self];
    f.at = kind;
    f.line = line;
    f.value = v;
    swapcontext(&f.ctx, &scheduler);
}

inline void entry() {
    body();
    fibers[self].at = 3;
    swapcontext(&fibers[self].ctx, &scheduler);
}

inline void release(int first, int last, int kind) {
    uint64_t any = 0;
    int line = 0;
    for (int t = first; t < last; ++t)
        if (fibers[t].at == kind) {
            any |= fibers[t].value;
            if (kind == 1 && line && line != fibers[t].line) ++mixed;
            line = fibers[t].line;
        }
    reduced = any;
    for (int t = first; t < last; ++t)
        if (fibers[t].at == kind) fibers[t].at = 0;
}

// One block: `order` 0 runs its threads upwards, 1 downwards, more a shuffle of its own.
inline void run_block(unsigned block, unsigned grid, unsigned threads, int order, std::function<void()> kernel) {
    body = kernel;
    blockIdx.x = block;
    blockDim.x = threads;
    gridDim.x = grid;
    fibers.resize(threads);
    std::vector<int> turn(threads);
    for (unsigned t = 0; t < threads; ++t) {
        Fiber& f = fibers[t];
        f.at = 0;
        getcontext(&f.ctx);
        f.ctx.uc_stack.ss_sp = f.stack.data();
        f.ctx.uc_stack.ss_size = STACK;
        f.ctx.uc_link = nullptr;
        makecontext(&f.ctx, entry, 0);
        turn[t] = order == 1 ? int(threads - 1 - t) : int(t);
    }
    uint32_t seed = 12345u * unsigned(order) + block;
    if (order > 1)
        for (unsigned t = threads - 1; t > 0; --t) {
            seed = seed * 1664525u + 1013904223u;
            std::swap(turn[t], turn[(seed >> 8) % (t + 1)]);
        }
    for (;;) {
        bool ran = false;
        for (int t : turn)
            if (fibers[t].at == 0) {
                self = t;
                threadIdx.x = unsigned(t);
                ran = true;
                swapcontext(&scheduler, &fibers[t].ctx);
            }
        if (ran) continue;
        // all stopped: a warp whose live threads are at a collective goes on, else the block's barrier
        bool warp = false, live = false;
        for (unsigned w = 0; w < threads; w += 32) {
            bool all = true, some = false;
            for (unsigned t = w; t < w + 32; ++t) {
                all = all && (fibers[t].at == 2 || fibers[t].at == 3);
                some = some || fibers[t].at == 2;
                live = live || fibers[t].at != 3;
            }
            if (all && some) {
                release(int(w), int(w + 32), 2);
                warp = true;
            }
        }
        if (!live) return;
        if (!warp) release(0, int(threads), 1);
    }
}

template <class T>
T shfl_up(T v, int d) {
    static_assert(sizeof(T) <= 8, "one word");
    uint64_t w = 0;
    memcpy(&w, &v, sizeof v);
    wait_at(2, 0, w);
    const int lane = self & 31;
    T r = v;
    if (lane >= d) memcpy(&r, &fibers[self - d].value, sizeof r);
    wait_at(2, 0, w);          // everyone has read
    return r;
}

}  // namespace emu

using emu::blockDim;
using emu::blockIdx;
using emu::gridDim;
using emu::threadIdx;
using std::max;
using std::min;

#define __syncthreads() emu::wait_at(1, __LINE__, 0)
#define __syncthreads_or(p) (emu::wait_at(1, __LINE__, (p) ? 1 : 0), int(emu::reduced))
inline void __threadfence() {}
inline void __syncwarp(unsigned = ~0u) {}
inline size_t __cvta_generic_to_shared(const void*) { return 0; }
template <class T> T __ldg(const T* p) { return *p; }
template <class T> T atomicMin(T* p, T v) { const T o = *p; *p = std::min(o, v); return o; }
template <class T> T atomicAdd(T* p, T v) { const T o = *p; *p = o + v; return o; }
template <class T> T __shfl_up_sync(unsigned, T v, int d) { return emu::shfl_up(v, d); }
template <class T> T __shfl_xor_sync(unsigned, T v, int) { return v; }       // not reached
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __int_as_float(int v) { float f; memcpy(&f, &v, 4); return f; }
