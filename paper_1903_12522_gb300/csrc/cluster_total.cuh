// Sums over a thread-block cluster of kClusterCtas CTAs of kClusterThreads threads.  The including file
// provides the two constants, store_to_cta (a store into another CTA's copy of a shared array) and
// pcg_cluster_sync (all threads of the cluster meet).
#pragma once

// The cluster's totals of v in every thread.  slots: the CTAs' sums and the total, not used by another
// call of the same kernel.  part is free again after the cluster barrier within: the last to read it, the
// first warp, has done so by then.
template <int NV>
__device__ __forceinline__ void cluster_total(double (&v)[NV], double (*part)[kClusterThreads],
                                              double (*slots)[kClusterCtas + 1]) {
    const int tid = (int)threadIdx.x;
#pragma unroll
    for (int k = 0; k < NV; ++k) part[k][tid] = v[k];
    __syncthreads();
    if (tid < 32) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = 0.0;
#pragma unroll
            for (int q = 0; q < kClusterThreads / 32; ++q) x += part[k][tid + 32 * q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (tid < kClusterCtas) store_to_cta(&slots[k][blockIdx.x], tid, x);
        }
    }
    pcg_cluster_sync();
    if (tid < 32) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = slots[k][tid & (kClusterCtas - 1)];
#pragma unroll
            for (int o = kClusterCtas / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (tid == 0) slots[k][kClusterCtas] = x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = slots[k][kClusterCtas];
}
