// The sweeps on the coarsest level of the V-cycle's coarse end (riesz.cu), which one CTA holds whole.
// The including file provides lds, sts (a float of shared memory), node_byte and sweep_barrier (the
// first `threads` threads of the CTA meet).
#pragma once

__device__ __forceinline__ int ends_of(unsigned d) { return __popc(d & 63u); }

// The first sweep's result from zero, omega b / diag K.
__device__ __forceinline__ float first_sweep(const CoarseLevel& l, float omega, unsigned d, float b) {
    return d & 64u ? 0.f : omega * l.cB * (float)(1 << ends_of(d)) * b;
}

// The coarsest level's sweeps: one node per thread of the warps that hold nodes (up to 1024 nodes).
__device__ __forceinline__ void coarsest_sweeps(const CoarseLevel l, float omega, int sweeps) {
    const int threads = (l.np + 31) & ~31;
    if ((int)threadIdx.x >= threads) return;
    const bool here = (int)threadIdx.x < l.np;
    const int i = here ? (int)threadIdx.x : 0;
    const unsigned d = node_byte(l, i), sy = 4u * (unsigned)l.sx, sz = 4u * (unsigned)l.sxy;
    const unsigned x = l.x + 4u * (unsigned)i, flip = l.r - l.x;
    const bool dir = (d & 64u) != 0u, d3 = l.dim == 3;
    const unsigned a0 = x + (d & 1u ? 4u : -4u), a1 = x + (d & 2u ? -4u : 4u);
    const unsigned a2 = x + (d & 4u ? sy : -sy), a3 = x + (d & 8u ? -sy : sy);
    const unsigned a4 = x + (d3 ? (d & 16u ? sz : -sz) : 0u), a5 = x + (d3 ? (d & 32u ? -sz : sz) : 0u);
    const float bj = lds(l.b + 4u * (unsigned)i);
    const float w = __fmul_rn(l.cB, (float)(1 << ends_of(d))), inv2d = l.inv2d, dd = d3 ? 6.f : 4.f;
    float xj = first_sweep(l, omega, d, bj);
    if (threads == 32) {  // one warp: the neighbours' values by shuffle
        const unsigned all = 0xffffffffu;
        const int n0 = (int)(a0 - l.x) >> 2, n1 = (int)(a1 - l.x) >> 2, n2 = (int)(a2 - l.x) >> 2, n3 = (int)(a3 - l.x) >> 2;
        const int n4 = (int)(a4 - l.x) >> 2, n5 = (int)(a5 - l.x) >> 2;
        for (int s = 1; s < sweeps; ++s) {
            const float v0 = __shfl_sync(all, xj, n0), v1 = __shfl_sync(all, xj, n1);
            const float v2 = __shfl_sync(all, xj, n2), v3 = __shfl_sync(all, xj, n3);
            float acc = v0 + v1;
            acc += v2 + v3;
            if (d3) acc += __shfl_sync(all, xj, n4) + __shfl_sync(all, xj, n5);
            const float L = __fsub_rn(__fmul_rn(dd, xj), acc);
            const float v = __fmaf_rn(omega, __fmaf_rn(w, bj, -__fmul_rn(inv2d, L)), xj);
            xj = dir ? 0.f : v;
        }
        if (here) sts(x, xj);
        return;
    }
    // the sweeps alternate between x and r and end in x: a copy at the end would have to wait for the
    // last sweep's readers
    unsigned o = sweeps & 1 ? 0u : flip;
    if (here) sts(x + o, xj);
    for (int s = 1; s < sweeps; ++s) {
        sweep_barrier(threads);
        float acc = lds(a0 + o) + lds(a1 + o);
        acc += lds(a2 + o) + lds(a3 + o);
        if (d3) acc += lds(a4 + o) + lds(a5 + o);
        const float L = __fsub_rn(__fmul_rn(dd, xj), acc);
        const float v = __fmaf_rn(omega, __fmaf_rn(w, bj, -__fmul_rn(inv2d, L)), xj);
        xj = dir ? 0.f : v;
        o = flip - o;
        if (here) sts(x + o, xj);
    }
}
