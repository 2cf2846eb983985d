// The coarsest level's sweeps (csrc/coarsest.cuh) against the same sweeps one after the other, under
// several orders of the threads.  Prints the number of differing values per case.
#include "simt.h"

#include "coarse_level.h"

using cmcg::CoarseLevel;
static float& word(unsigned a) { return *reinterpret_cast<float*>(simt::shared_of((int)blockIdx.x) + a); }
static float lds(unsigned a) { return word(a); }
static void sts(unsigned a, float v) { word(a) = v; }
static unsigned node_byte(const CoarseLevel& l, int k) { return (unsigned char)simt::shared_of((int)blockIdx.x)[l.node + k]; }
static void sweep_barrier(int threads) { simt::meet((int)blockIdx.x, 1, threads); }
#include "coarsest.cuh"

static int differing(int nx, int ny, int nz, int sweeps, unsigned order) {
    CoarseLevel l{};
    l.nx = nx, l.ny = ny, l.nz = nz, l.dim = nz ? 3 : 2;
    l.sx = nx + 1, l.sy = ny + 1, l.sxy = l.sx * l.sy;
    l.np = l.cnt = l.sxy * (nz + 1);
    l.cB = 0.7f, l.cK = 1.f, l.inv2d = 1.f / (float)(2 * l.dim);
    l.x = 0, l.r = 4 * l.np, l.b = 8 * l.np, l.node = 12 * l.np;
    const size_t bytes = 13 * (size_t)l.np;
    const float omega = 0.8f;
    simt::shared.assign(1, std::vector<char>(bytes, 0));
    char* sm = simt::shared_of(0);
    std::vector<float> b(l.np);
    std::vector<unsigned> node(l.np);
    for (int k = 0; k < l.np; ++k) {
        const int ix = k % l.sx, iy = k / l.sx % l.sy, iz = k / l.sxy;
        unsigned d = (ix == 0 ? 1u : 0u) | (ix == nx ? 2u : 0u) | (iy == 0 ? 4u : 0u) | (iy == ny ? 8u : 0u);
        if (nz) d |= (iz == 0 ? 16u : 0u) | (iz == nz ? 32u : 0u);
        if (k % 11 == 5) d |= 64u;  // some Dirichlet nodes
        b[k] = d & 64u ? 0.f : sinf(1.3f * k);
        node[k] = d;
        memcpy(sm + l.b + 4 * k, &b[k], 4);
        sm[l.node + k] = (char)d;
    }
    // one sweep after the other
    std::vector<float> x(l.np), y(l.np);
    for (int k = 0; k < l.np; ++k) x[k] = first_sweep(l, omega, node[k], b[k]);
    for (int s = 1; s < sweeps; ++s) {
        for (int k = 0; k < l.np; ++k) {
            const unsigned d = node[k];
            float acc = x[k + (d & 1u ? 1 : -1)] + x[k + (d & 2u ? -1 : 1)];
            acc += x[k + (d & 4u ? l.sx : -l.sx)] + x[k + (d & 8u ? -l.sx : l.sx)];
            if (nz) acc += x[k + (d & 16u ? l.sxy : -l.sxy)] + x[k + (d & 32u ? -l.sxy : l.sxy)];
            const float dd = nz ? 6.f : 4.f, L = dd * x[k] - acc, w = l.cB * (float)(1 << ends_of(d));
            y[k] = d & 64u ? 0.f : fmaf(omega, fmaf(w, b[k], -(l.inv2d * L)), x[k]);
        }
        x.swap(y);
    }
    if (!simt::run(1, 1024, bytes, order, [&] { coarsest_sweeps(l, omega, sweeps); })) return -1;
    int bad = 0;
    for (int k = 0; k < l.np; ++k) {
        float v;
        memcpy(&v, simt::shared_of(0) + l.x + 4 * k, 4);
        bad += memcmp(&v, &x[k], 4) != 0;
    }
    return bad;
}

int main() {
    // one warp (shuffles), two, and up to 17; even and odd numbers of sweeps
    const int size[][3] = {{4, 4, 0}, {2, 2, 2}, {6, 6, 0}, {7, 5, 0}, {3, 3, 3}, {4, 5, 3}, {130, 3, 0}, {5, 5, 3}, {12, 3, 9}};
    for (auto& n : size)
        for (int sweeps : {2, 5, 32, 33})
            for (unsigned order : {0u, 1u, 2u, 3u})
                printf("%d %d %d sweeps %d order %u: %d\n", n[0], n[1], n[2], sweeps, order,
                       differing(n[0], n[1], n[2], sweeps, order));
}
