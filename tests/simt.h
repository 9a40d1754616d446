// simt.h -- one block of device code on the CPU: every thread is a fiber that
// runs to its next warp or block operation.  Enough of CUDA's device functions
// for the kernels that the tests include (see test_deferred_sums.py).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <ucontext.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#define __CUDACC__ 1     // (after the headers: the device parts of the library's own)
#undef __shared__
#undef __launch_bounds__
#undef __global__
#undef __device__
#undef __constant__
#undef __forceinline__
#undef __noinline__
#undef __host__
#undef __align__
#define __shared__ static
#define __launch_bounds__(...)
#define __global__ static
#define __device__
#define __constant__
#define __forceinline__ inline
#define __noinline__
#define __host__
#define __align__(n)

using std::max;
using std::min;

struct Simt {
    struct Fiber {
        ucontext_t at;
        std::vector<char> stack;
        bool done = false;
        int waits = 0;      // 1: for its warp, 2: for its block
        int turn = 0;
    };
    std::vector<Fiber> f;
    ucontext_t home;
    std::function<void()> fn;
    int cur = 0, threads = 0;
    unsigned long long lane[32][2][32];      // what a warp's lanes have put up, two operations in turn
};
static Simt S;
static uint32_t* simt_smem;

struct SimtIndex {
    int x;
};
#define threadIdx (SimtIndex{S.cur})
#define blockIdx (SimtIndex{0})
#define blockDim (SimtIndex{S.threads})
#define gridDim (SimtIndex{1})

static void simt_wait(int kind) {
    Simt::Fiber& f = S.f[S.cur];
    f.waits = kind;
    swapcontext(&f.at, &S.home);
}
static unsigned long long* simt_put(unsigned long long v) {
    const int w = S.cur >> 5, turn = S.f[S.cur].turn;
    S.f[S.cur].turn ^= 1;
    S.lane[w][turn][S.cur & 31] = v;
    simt_wait(1);
    return S.lane[w][turn];
}
static void simt_entry() {
    S.fn();
    S.f[S.cur].done = true;
    swapcontext(&S.f[S.cur].at, &S.home);
}

// fn by one block of `threads` threads with `words` words of shared memory
static void simt_run(int threads, size_t words, std::function<void()> fn) {
    const size_t guard = 1 << 14;      // words watched on either side
    std::vector<uint32_t> smem(words + 2 * guard, 0xdeadbeefu);
    simt_smem = smem.data() + guard;
    S.fn = fn;
    S.threads = threads;
    S.f.clear();
    S.f.resize(threads);
    for (auto& f : S.f) {
        f.stack.resize(256 * 1024);
        getcontext(&f.at);
        f.at.uc_stack.ss_sp = f.stack.data();
        f.at.uc_stack.ss_size = f.stack.size();
        f.at.uc_link = &S.home;
        makecontext(&f.at, simt_entry, 0);
    }
    for (bool progress = true; progress;) {
        progress = false;
        int live = 0, at_block = 0;
        for (int w = 0; w < threads / 32; w++) {
            int there = 0, running = 0;
            for (int t = 32 * w; t < 32 * w + 32; t++) {
                if (!S.f[t].done && !S.f[t].waits) {
                    S.cur = t;
                    swapcontext(&S.home, &S.f[t].at);
                    progress = true;
                }
                running += !S.f[t].done;
                there += S.f[t].waits == 1 && !S.f[t].done;
                at_block += S.f[t].waits == 2 && !S.f[t].done;
            }
            live += running;
            if (there && there == running) {
                for (int t = 32 * w; t < 32 * w + 32; t++) S.f[t].waits = 0;
                progress = true;
            }
        }
        if (live && at_block == live) {
            for (auto& f : S.f) f.waits = 0;
            progress = true;
        }
        if (!progress && live) {
            fprintf(stderr, "threads wait for one another\n");
            abort();
        }
    }
    for (size_t i = 0; i < smem.size(); i++)
        if ((i < guard || i >= words + guard) && smem[i] != 0xdeadbeefu) {
            fprintf(stderr, "write outside of shared memory\n");
            abort();
        }
}

static inline void __syncwarp(unsigned = ~0u) { simt_wait(1); }
static inline void __syncthreads() { simt_wait(2); }
template <class F>
static inline unsigned simt_fold(unsigned v, unsigned r, F f) {
    const unsigned long long* b = simt_put(v);
    for (int i = 0; i < 32; i++) r = f(r, (unsigned)b[i]);
    return r;
}
static inline unsigned __ballot_sync(unsigned, int p) {
    const unsigned long long* b = simt_put(p != 0);
    unsigned r = 0;
    for (int i = 0; i < 32; i++) r |= (unsigned)b[i] << i;
    return r;
}
static inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0; }
static inline unsigned __reduce_add_sync(unsigned, unsigned v) { return simt_fold(v, 0, [](unsigned a, unsigned b) { return a + b; }); }
static inline unsigned __reduce_or_sync(unsigned, unsigned v) { return simt_fold(v, 0, [](unsigned a, unsigned b) { return a | b; }); }
static inline unsigned __reduce_max_sync(unsigned, unsigned v) { return simt_fold(v, 0, [](unsigned a, unsigned b) { return max(a, b); }); }
template <class V>
static inline V simt_from(V v, int src) {
    unsigned long long u = 0;
    memcpy(&u, &v, sizeof v);
    u = simt_put(u)[src & 31];
    memcpy(&v, &u, sizeof v);
    return v;
}
template <class V>
static inline V __shfl_sync(unsigned, V v, int src) { return simt_from(v, src); }
template <class V>
static inline V __shfl_xor_sync(unsigned, V v, int o) { return simt_from(v, (S.cur & 31) ^ o); }
static inline void __threadfence() {}
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline int __ffs(int x) { return __builtin_ffs(x); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
template <class V, class U>
static inline V atomicAdd(V* p, U v) { V o = *p; *p = (V)(o + v); return o; }
template <class V, class U>
static inline V atomicSub(V* p, U v) { V o = *p; *p = (V)(o - v); return o; }
template <class V, class U>
static inline V atomicOr(V* p, U v) { V o = *p; *p = (V)(o | v); return o; }
template <class V, class U>
static inline V atomicExch(V* p, U v) { V o = *p; *p = (V)v; return o; }
template <class V>
static inline V __ldcg(const V* p) { return *p; }
