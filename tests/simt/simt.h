// CUDA threads as fibers on the CPU, for tests of device code that depends on its barriers: a thread runs
// until its next barrier or shuffle, and which of the ready threads runs next is the test's choice.  What a
// barrier does not order, some choice will show.  Shared memory is an array per CTA.
#pragma once
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <ucontext.h>

#include <functional>
#include <map>
#include <vector>

#define __device__
#define __forceinline__ inline

struct Dim {
    unsigned x;
};
static Dim threadIdx, blockIdx, blockDim, gridDim;

namespace simt {

struct Barrier {
    int arrived = 0, phase = 0;
};
struct Thread {
    ucontext_t ctx;
    std::vector<char> stack;
    int cta, tid;
    bool done = false;
    Barrier* at = nullptr;  // waiting for its phase to pass
    int phase = 0;
};

static std::vector<Thread> threads;
static std::vector<std::vector<char>> shared;
static std::map<std::pair<int, int>, Barrier> barriers;  // (CTA, id); CTA -1: the cluster's
static std::map<std::pair<int, int>, std::vector<double>> lanes;  // of the shuffles, by (CTA, warp)
static ucontext_t scheduler;
static Thread* self;
static std::function<void()> body;

inline char* shared_of(int cta) { return shared[cta].data(); }

inline void meet(int cta, int id, int count) {
    Barrier& b = barriers[{cta, id}];
    if (++b.arrived == count) {
        b.arrived = 0;
        ++b.phase;
        return;
    }
    self->at = &b;
    self->phase = b.phase;
    swapcontext(&self->ctx, &scheduler);
}

inline void entry() {
    body();
    self->done = true;
    swapcontext(&self->ctx, &scheduler);
}

// Runs f in every thread; order: 0 the lowest ready thread first, 1 the highest, else a random one (the seed).
// False if the threads end up waiting for one another.
inline bool run(int ctas, int per_cta, size_t shared_bytes, unsigned order, std::function<void()> f) {
    body = f;
    threads.assign((size_t)ctas * per_cta, Thread());
    barriers.clear();
    lanes.clear();
    if (shared.size() != (size_t)ctas || shared[0].size() != shared_bytes)
        shared.assign(ctas, std::vector<char>(shared_bytes, 0));
    blockDim.x = per_cta;
    gridDim.x = ctas;
    for (size_t k = 0; k < threads.size(); ++k) {
        Thread& t = threads[k];
        t.cta = (int)k / per_cta;
        t.tid = (int)k % per_cta;
        t.stack.resize(64 << 10);
        getcontext(&t.ctx);
        t.ctx.uc_stack.ss_sp = t.stack.data();
        t.ctx.uc_stack.ss_size = t.stack.size();
        t.ctx.uc_link = &scheduler;
        makecontext(&t.ctx, entry, 0);
    }
    unsigned rnd = order * 2654435761u + 12345u;
    for (;;) {
        std::vector<Thread*> ready;
        bool all_done = true;
        for (Thread& t : threads) {
            if (t.done) continue;
            all_done = false;
            if (!t.at || t.at->phase != t.phase) ready.push_back(&t);
        }
        if (all_done) return true;
        if (ready.empty()) return false;
        rnd = rnd * 1664525u + 1013904223u;
        Thread* t = order == 0 ? ready.front() : (order == 1 ? ready.back() : ready[(rnd >> 8) % ready.size()]);
        t->at = nullptr;
        self = t;
        threadIdx.x = t->tid;
        blockIdx.x = t->cta;
        swapcontext(&scheduler, &t->ctx);
    }
}

// A thread goes on after a wait with its own indices (the scheduler set them).
inline double exchange(double v, int from) {
    const int cta = self->cta, warp = self->tid / 32, lane = self->tid % 32;
    std::vector<double>& l = lanes[{cta, warp}];
    l.resize(32);
    l[lane] = v;
    meet(cta, 100 + warp, 32);
    const double r = l[from & 31];
    meet(cta, 100 + warp, 32);
    return r;
}

}  // namespace simt

inline void __syncthreads() { simt::meet((int)blockIdx.x, 0, (int)blockDim.x); }
inline float __shfl_sync(unsigned, float v, int from) { return (float)simt::exchange(v, from); }
inline double __shfl_xor_sync(unsigned, double v, int mask) { return simt::exchange(v, (simt::self->tid ^ mask) & 31); }
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
