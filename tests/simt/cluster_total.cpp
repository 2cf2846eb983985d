// cluster_total (csrc/cluster_total.cuh): three sums in a row as k_pcg_cluster takes them, in every thread of
// every CTA, under several orders of the threads.  Prints the number of wrong values per order.
#include "simt.h"

constexpr int kClusterThreads = 96, kClusterCtas = 4;
struct Shared {
    double part[2][kClusterThreads];
    double slots[3][2][kClusterCtas + 1];
};
static void store_to_cta(double* slot, int cta, double v) {
    const size_t at = (char*)slot - simt::shared_of((int)blockIdx.x);
    memcpy(simt::shared_of(cta) + at, &v, sizeof(v));
}
static void pcg_cluster_sync() { simt::meet(-1, 0, kClusterThreads * kClusterCtas); }
#include "cluster_total.cuh"

static double value(int call, int k, int cta, int tid) { return (double)((call * 7 + k * 3 + cta * 5 + tid) % 23 - 9); }

int main() {
    double want[3][2] = {};
    for (int call = 0; call < 3; ++call)
        for (int k = 0; k < 2; ++k)
            for (int cta = 0; cta < kClusterCtas; ++cta)
                for (int tid = 0; tid < kClusterThreads; ++tid) want[call][k] += value(call, k, cta, tid);
    for (unsigned order = 0; order < 20; ++order) {
        int bad = 0;
        const bool ends = simt::run(kClusterCtas, kClusterThreads, sizeof(Shared), order, [&] {
            Shared& sh = *reinterpret_cast<Shared*>(simt::shared_of((int)blockIdx.x));
            const int cta = (int)blockIdx.x, tid = (int)threadIdx.x;
            double two[2] = {value(0, 0, cta, tid), value(0, 1, cta, tid)};
            cluster_total<2>(two, sh.part, sh.slots[0]);
            bad += (two[0] != want[0][0]) + (two[1] != want[0][1]);
            pcg_cluster_sync();
            for (int call = 1; call < 3; ++call) {
                double one[1] = {value(call, 0, cta, tid)};
                cluster_total<1>(one, sh.part, sh.slots[call]);
                bad += one[0] != want[call][0];
            }
        });
        printf("order %u: %d\n", order, ends ? bad : -1);
    }
}
