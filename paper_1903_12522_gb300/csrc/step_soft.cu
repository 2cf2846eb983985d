// FP64 leapfrog steps and period endpoints with the stencil sum in integer arithmetic
// (soft64.cuh), for handles in FP64.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "soft64.cuh"

namespace cmcg {

namespace {

using soft64::Term;

constexpr int kST = 256;

struct Values {
    const double* __restrict__ p;
    __device__ __forceinline__ double operator()(int i) const { return p[i]; }
};

struct Difference {  // a - b, formed in FP64 before the stencil sums it
    const double* __restrict__ a;
    const double* __restrict__ b;
    __device__ __forceinline__ double operator()(int i) const { return a[i] - b[i]; }
};

// The rare cases stay out of line: inlined, their FP64 instructions would be predicated into
// every update, and a predicated-off FP64 instruction costs as much as an executed one.

// The negated unscaled Laplacian of f at a node in plain FP64, for the values the fixed-point
// sum does not take.
template <int ORDER, typename F>
__device__ __noinline__ double neg_lap_plain(F f, const Geom& g, int j, int ix, int iy, int iz) {
    auto at = [f](long long i) { return f((int)i); };
    return -lap_t<ORDER, double>(g, at, (long long)j, ix, iy, iz);
}

// The update on an absorbing face, w = 1 / (1 + beta): out = w rhs - (1 - beta) w yp with
// (1 - beta) w = 2 w - 1, and the adjoint's first and last variants (the previous term already
// scaled; no division).
template <int FLAGS>
__device__ __noinline__ double face_update(double rhs, double yp, double w) {
    if (FLAGS & kStepNoDiv) {
        if (FLAGS & kStepPrevScaled) return rhs - yp;
        return rhs - (2.0 - 1.0 / w) * yp;
    }
    if (FLAGS & kStepPrevScaled) return (rhs - yp) * w;
    return fma(rhs, w, -(fma(2.0, w, -1.0) * yp));
}

// (1 - beta) x and x / (1 + beta) on an absorbing face.
__device__ __noinline__ double face_minus(double x, double w) { return (2.0 - 1.0 / w) * x; }
__device__ __noinline__ double face_over(double x, double w) { return x * w; }

__device__ __noinline__ double add_source(double d, const double* __restrict__ S, int j, double cs, double sn) {
    const double2 s = reinterpret_cast<const double2*>(S)[j];
    return d + fma(s.x, cs, s.y * sn);
}

// The period's start takes the real part only: an imaginary part that is not finite acts from the first
// step on, not here through a product with zero.
__device__ __noinline__ double add_half_re(double d, const double* __restrict__ S, int j) { return fma(0.5, S[2 * j], d); }

// One thread's column of a launch: its (x, y), its planes, its faces.
template <int DIM>
struct Column {
    int ix, iy, z0, z1, j;  // j: node of plane z0
    bool valid, fxy;        // fxy: on an absorbing x or y face
    unsigned abc;
    int nz;
    __device__ __forceinline__ Column(const Geom& g, int zc, int radius, bool reverse) {
        const int plane = g.sx * g.sy;
        const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
        const int by = reverse ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
        const int p = bx * kST + (int)threadIdx.x;
        valid = p < plane;
        const int pp = valid ? p : 0;
        iy = (int)((unsigned)pp / (unsigned)g.sx);
        ix = pp - iy * g.sx;
        z0 = DIM == 3 ? by * zc : 0;
        z1 = DIM == 3 ? min(z0 + zc, g.sz) : 1;
        j = pp + plane * z0;
        abc = g.abc;
        nz = g.nz;
        fxy = (ix == 0 && (abc & 1u)) || (ix == g.nx && (abc & 2u)) || (iy == 0 && (abc & 4u)) ||
              (iy == g.ny && (abc & 8u));
        if (valid && !column_in_range(g, ix, iy, z0, z1, radius, kSiteColumn)) valid = false;
    }
    // is the node of plane iz on an absorbing face?
    __device__ __forceinline__ bool face(int iz) const {
        return fxy || (DIM == 3 && ((iz == 0 && (abc & 16u)) || (iz == nz && (abc & 32u))));
    }
};

// -Lt(f) along a column, the z-neighbours' terms carried in registers.  For the 4th order the
// integer sum is 3/4 of it, a1 - a2 / 16 - (15/8) DIM y, whose weights are shifts.
template <int DIM, int ORDER, typename F>
struct SoftLap {
    F f;
    const Geom& g;
    int ix, iy, sZ, oxm, oxp, oym, oyp, ox2m, ox2p, oy2m, oy2p;
    double yc, yz;  // f at the current plane, and (4th order) at the next one
    Term c, zm, zp, zm2;
    __device__ __forceinline__ SoftLap(F f_, const Geom& g_, int ix_, int iy_)
        : f(f_), g(g_), ix(ix_), iy(iy_), sZ(g_.sx * g_.sy), yc(0.0), yz(0.0), c{}, zm{}, zp{}, zm2{} {
        oxm = (int)off_m1(ix, 1), oxp = (int)off_p1(ix, g.nx, 1);
        oym = (int)off_m1(iy, g.sx), oyp = (int)off_p1(iy, g.ny, g.sx);
        ox2m = ox2p = oy2m = oy2p = 0;
        if (ORDER == 4) {
            ox2m = (int)off_m2(ix, 1), ox2p = (int)off_p2(ix, g.nx, 1);
            oy2m = (int)off_m2(iy, g.sx), oy2p = (int)off_p2(iy, g.ny, g.sx);
        }
    }
    __device__ __forceinline__ void start(int j, int iz) {
        yc = f(j);
        c = soft64::term(yc);
        if (DIM == 3) {
            zm = soft64::term(f(j + (iz > 0 ? -sZ : sZ)));
            if (ORDER == 4) {
                zm2 = soft64::term(f(j + (int)off_m2(iz, sZ)));
                yz = f(j + (iz < g.nz ? sZ : -sZ));
                zp = soft64::term(yz);
            }
        }
    }
    // -Lt(f) at plane iz (node j), then on to plane iz + 1; y receives f there.
    __device__ __forceinline__ double next(int j, int iz, double* y) {
        double zn = 0.0;
        if (DIM == 3) zn = f(j + (ORDER == 2 ? (iz < g.nz ? sZ : -sZ) : (int)off_p2(iz, g.nz, sZ)));
        const double x0 = f(j + oxm), x1 = f(j + oxp), y0 = f(j + oym), y1 = f(j + oyp);
        double u0 = 0.0, u1 = 0.0, v0 = 0.0, v1 = 0.0;
        if (ORDER == 4) u0 = f(j + ox2m), u1 = f(j + ox2p), v0 = f(j + oy2m), v1 = f(j + oy2p);
        const Term a0 = soft64::term(x0), a1 = soft64::term(x1), b0 = soft64::term(y0), b1 = soft64::term(y1);
        unsigned e = soft64::max3(soft64::max3(c.e, a0.e, a1.e), b0.e, b1.e);
        Term zp2{};
        if (DIM == 3) {
            if (ORDER == 2) zp = soft64::term(zn);
            else zp2 = soft64::term(zn);
            e = soft64::max3(e, zm.e, zp.e);
        }
        Term c0{}, c1{}, d0{}, d1{};
        if (ORDER == 4) {
            c0 = soft64::term(u0), c1 = soft64::term(u1), d0 = soft64::term(v0), d1 = soft64::term(v1);
            e = soft64::max3(soft64::max3(e, c0.e, c1.e), d0.e, d1.e);
            if (DIM == 3) e = soft64::max3(e, zm2.e, zp2.e);
        }
        const long long C = soft64::align(c, e);
        long long s1 = (soft64::align(a0, e) + soft64::align(a1, e)) + (soft64::align(b0, e) + soft64::align(b1, e));
        if (DIM == 3) s1 += soft64::align(zm, e) + soft64::align(zp, e);
        double L;
        bool ok;
        if (ORDER == 2) {
            L = soft64::to_double(s1 - (DIM == 3 ? 4 * C + 2 * C : 4 * C), e, &ok);
        } else {
            long long s2 = (soft64::align(c0, e) + soft64::align(c1, e)) + (soft64::align(d0, e) + soft64::align(d1, e));
            if (DIM == 3) s2 += soft64::align(zm2, e) + soft64::align(zp2, e);
            const long long q = DIM == 3 ? 6 * C - (3 * C >> 3) : 4 * C - (C >> 2);
            L = soft64::four_thirds(s1 - (s2 >> 4) - q, e, &ok);
        }
        if (!(ok && soft64::in_range(e))) L = neg_lap_plain<ORDER, F>(f, g, j, ix, iy, iz);
        *y = yc;
        if (DIM == 3) {
            if (ORDER == 2) {
                zm = c;
                c = zp;
                yc = zn;
            } else {
                zm2 = zm;
                zm = c;
                c = zp;
                zp = zp2;
                yc = yz;
                yz = zn;
            }
        }
        return L;
    }
};

// One leapfrog step, one thread per (x, y) column of zc planes (2D: one node).
//
// Bound: latency; the FP64 and ALU pipes and the issue slots are each busy 43 to 44 % of the time at
// half of the warp slots (FP64 work left per update: 2 y - y_prev and the fused multiply-add with kappa,
// against nine operations and, on the faces, a square root and a division).  193^3, with a source on the faces: 246 us a step in FP64 arithmetic, 87 us
// now, 73 without one (230 MB of algorithmic bytes, 34 us at the copy bandwidth).
//
// B: resident blocks per SM.  Whole backward periods of 57 steps: 7-point 193^3 4.66 ms with four, 4.47
// with five, 4.19 with six (40 registers, a few spills); 177x171x151 2.98, 2.93, 2.80; 129^3 1.67, 1.62,
// 1.68.  13-point 151x141x131 2.83 ms with three, 2.70 with four, 2.93 with five.
template <int DIM, int ORDER, int FLAGS, bool SRC_FACES, int B>
__global__ void __launch_bounds__(kST, B)
    k_step_soft(const double* __restrict__ cur, double* __restrict__ prev_out, const double* __restrict__ kap,
                const double* __restrict__ wface, const double* __restrict__ S, double cs, double sn, Geom g, int zc,
                int reverse) {
    const Column<DIM> m(g, zc, ORDER / 2, reverse != 0);
    if (!m.valid) return;
    SoftLap<DIM, ORDER, Values> lap(Values{cur}, g, m.ix, m.iy);
    int j = m.j;
    lap.start(j, m.z0);
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const double k = kap[j], yp = prev_out[j];
        double yc;
        const double L = lap.next(j, iz, &yc);
        double out;
        if (m.face(iz)) {
            double rhs = fma(k, L, 2.0 * yc);
            if (FLAGS & kStepSrc) rhs = add_source(rhs, S, j, cs, sn);
            out = face_update<FLAGS>(rhs, yp, wface[j]);
        } else {
            out = fma(k, L, fma(2.0, yc, -yp));
            if ((FLAGS & kStepSrc) && !SRC_FACES) out = add_source(out, S, j, cs, sn);
        }
        prev_out[j] = out;
        j += lap.sZ;
    }
}

// The period's endpoint kernels in FP64 (the formulas are those of k_start, k_end, k_adj_* in
// wave.cu) with the same stencil sum, the face factors and 1 / dt, 1 / M precomputed: the plain
// kernels spend 30 to 50 FP64 operations per node, most of them in divisions.
template <int DIM, int ORDER, bool SRC>
__global__ void __launch_bounds__(kST, 3)
    k_start_soft(const double* __restrict__ w0, const double* __restrict__ w1, double* __restrict__ y0,
                 double* __restrict__ y1, const double* __restrict__ kap, const double* __restrict__ wface,
                 const double* __restrict__ S, Geom g, double dt, int zc, int src_faces) {
    const Column<DIM> m(g, zc, ORDER / 2, false);
    if (!m.valid) return;
    SoftLap<DIM, ORDER, Values> lap(Values{w0}, g, m.ix, m.iy);
    int j = m.j;
    lap.start(j, m.z0);
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const double k = kap[j];
        double vj = w1[j], yc;
        const double L = lap.next(j, iz, &yc);
        const bool face = m.face(iz);
        if (face) vj = face_minus(vj, wface[j]);
        double v = fma(0.5 * k, L, fma(dt, vj, yc));
        if (SRC && (face || !src_faces)) v = add_half_re(v, S, j);
        const bool dir = soft64::is_zero(k);  // Dirichlet
        y0[j] = dir ? 0.0 : yc;
        y1[j] = dir ? 0.0 : v;
        j += lap.sZ;
    }
}

// MODE 0: z = E (Pi(w) - w) and J; MODE 1: (y(T), y_t(T)).  hs, hc: half the source factors.
template <int DIM, int ORDER, bool SRC, int MODE>
__global__ void __launch_bounds__(kST, MODE == 0 ? 2 : 3)
    k_end_soft(const double* __restrict__ yN, const double* __restrict__ yNm1, const double* __restrict__ w0,
               const double* __restrict__ w1, const double* __restrict__ kap, const double* __restrict__ mass,
               const double* __restrict__ wface, const double* __restrict__ S, double hc, double hs,
               double* __restrict__ out0, double* __restrict__ out1, Red red, Geom g, double inv_dt, double ck, int zc,
               int src_faces) {
    const Column<DIM> m(g, zc, ORDER / 2, false);
    double acc[1] = {0.0};
    if (m.valid) {
        SoftLap<DIM, ORDER, Values> lap(Values{yN}, g, m.ix, m.iy);
        SoftLap<DIM, ORDER, Difference> lape(Difference{yN, w0}, g, m.ix, m.iy);
        int j = m.j;
        lap.start(j, m.z0);
        if (MODE == 0) lape.start(j, m.z0);
        for (int iz = m.z0; iz < m.z1; ++iz) {
            const double k = kap[j], ym = yNm1[j];
            double yn;
            const double L = lap.next(j, iz, &yn);
            const bool face = m.face(iz), dir = soft64::is_zero(k);
            double t = fma(0.5 * k, L, yn - ym);
            if (SRC && (face || !src_faces)) t = add_source(t, S, j, hc, hs);
            double vN = t * inv_dt;
            if (face) vN = face_over(vN, wface[j]);
            if (MODE == 1) {
                out0[j] = dir ? 0.0 : yn;
                out1[j] = dir ? 0.0 : vN;
            } else {
                double e0;
                const double Le = lape.next(j, iz, &e0);
                const double e1 = vN - w1[j];
                int ends = (m.ix == 0 || m.ix == g.nx) + (m.iy == 0 || m.iy == g.ny);
                if (DIM == 3) ends += (iz == 0 || iz == g.nz);
                const double z0 = -(ck * Le) * __hiloint2double((1023 - ends) << 20, 0);
                const double z1 = mass[j] * e1;
                out0[j] = dir ? 0.0 : z0;
                out1[j] = dir ? 0.0 : z1;
                if (!dir) acc[0] += fma(e0, z0, e1 * z1);
            }
            j += lap.sZ;
        }
    }
    if (MODE == 0) {
        acc[0] *= 0.5;
        if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[SC_J] = acc[0];
    }
}

// t = D^-1 b = b / (M (1 + beta)).
template <int DIM>
__global__ void __launch_bounds__(kST) k_adj_prep_soft(const double* __restrict__ b, const double* __restrict__ minv,
                                                       const double* __restrict__ wface, double* __restrict__ t, Geom g,
                                                       int zc) {
    const Column<DIM> m(g, zc, 1, false);
    if (!m.valid) return;
    int j = m.j;
    for (int iz = m.z0; iz < m.z1; ++iz, j += g.sx * g.sy) {
        const double mi = minv[j];
        double v = b[j] * mi;
        if (m.face(iz)) v = face_over(v, wface[j]);
        t[j] = soft64::is_zero(mi) ? 0.0 : v;  // Dirichlet: 1/M is stored as 0
    }
}

template <int DIM, int ORDER>
__global__ void __launch_bounds__(kST, 3)
    k_adj_start_soft(const double* __restrict__ a, const double* __restrict__ t, const double* __restrict__ minv,
                     const double* __restrict__ kap, const double* __restrict__ wface, double* __restrict__ cur,
                     double* __restrict__ prev, Geom g, double inv_dt, int zc) {
    const Column<DIM> m(g, zc, ORDER / 2, false);
    if (!m.valid) return;
    SoftLap<DIM, ORDER, Values> lap(Values{t}, g, m.ix, m.iy);
    int j = m.j;
    lap.start(j, m.z0);
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const double k = kap[j], aj = a[j], mi = minv[j];
        double tj;
        const double L = lap.next(j, iz, &tj);
        double u = fma(aj, mi, inv_dt * fma(0.5 * k, L, tj));
        if (m.face(iz)) u = face_over(u, wface[j]);
        const bool dir = soft64::is_zero(k);
        cur[j] = dir ? 0.0 : u;
        prev[j] = dir ? 0.0 : tj * inv_dt;
        j += lap.sZ;
    }
}

// MODE 0: ghat = q - z, g~1 = ghat1 / M (gt1 nullable), (ghat . d, sum ghat0); MODE 1: q.
// cq = dt^2 / 2 h^d / h^2.
template <int DIM, int ORDER, int MODE>
__global__ void __launch_bounds__(kST, 3)
    k_adj_final_soft(const double* __restrict__ s, const double* __restrict__ u1, const double* __restrict__ mass,
                     const double* __restrict__ kap, const double* __restrict__ wface, const double* __restrict__ minv,
                     const double* __restrict__ z0, const double* __restrict__ z1, const double* __restrict__ d0,
                     const double* __restrict__ d1, double* __restrict__ o0, double* __restrict__ o1,
                     double* __restrict__ gt1, Red red, Geom g, double dt, double cq, int zc) {
    const Column<DIM> m(g, zc, ORDER / 2, false);
    double acc[2] = {0.0, 0.0};
    if (m.valid) {
        SoftLap<DIM, ORDER, Values> lap(Values{s}, g, m.ix, m.iy);
        int j = m.j;
        lap.start(j, m.z0);
        for (int iz = m.z0; iz < m.z1; ++iz) {
            const double k = kap[j], M = mass[j];
            double u = u1[j], sj;
            const double L = lap.next(j, iz, &sj);
            double sb = sj;
            if (m.face(iz)) {
                const double w = wface[j];
                u = face_minus(u, w);
                sb = face_minus(sj, w);
            }
            int ends = (m.ix == 0 || m.ix == g.nx) + (m.iy == 0 || m.iy == g.ny);
            if (DIM == 3) ends += (iz == 0 || iz == g.nz);
            const double c = cq * __hiloint2double((1023 - ends) << 20, 0);
            const double q0 = fma(c, L, M * (sj - u));
            const double q1 = (dt * M) * sb;
            const bool dir = soft64::is_zero(k);
            if (MODE == 1) {
                o0[j] = dir ? 0.0 : q0;
                o1[j] = dir ? 0.0 : q1;
            } else {
                const double g0 = q0 - z0[j], g1 = q1 - z1[j];
                o0[j] = dir ? 0.0 : g0;
                o1[j] = dir ? 0.0 : g1;
                if (gt1) gt1[j] = dir ? 0.0 : g1 * minv[j];
                if (!dir) {
                    acc[0] += fma(g0, d0[j], g1 * d1[j]);
                    acc[1] += g0;
                }
            }
            j += lap.sZ;
        }
    }
    if (MODE == 0 && grid_sum<2>(acc, red.partials, red.ticket) && threadIdx.x == 0) {
        red.sc[SC_GD] = acc[0];
        red.sc[SC_GSUM] = acc[1];
    }
}

// ---- the Riesz PCG's FP64 vector passes ----------------------------------------------------
// Bound: the FP64 pipe and latency.  Each pass keeps the operations it cannot do without (Ap 3, x
// and r 3, dots 2, p 1 per node), reads two nodes per access, and sums its block's partials in one
// warp: reduced in every warp by shuffles, five more FP64 instructions per warp would be a third of
// the pass.
constexpr int kPcgBlocks = 152 * 8;

// grid_sum (common.cuh) with fewer FP64 instructions: the block's values meet in shared memory and
// one warp adds them up.
template <int NV>
__device__ __forceinline__ bool pcg_sum(double (&v)[NV], double* partials, unsigned* ticket) {
    __shared__ double part[NV][kST];
    __shared__ bool last;
    const int tid = (int)threadIdx.x;
    const unsigned nb = gridDim.x * gridDim.y, bid = blockIdx.x + gridDim.x * blockIdx.y;
#pragma unroll
    for (int k = 0; k < NV; ++k) part[k][tid] = v[k];
    __syncthreads();
    auto warp_total = [&](double (&t)[NV]) {  // of part, in lane 0 of the first warp
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = 0.0;
#pragma unroll
            for (int q = 0; q < kST / 32; ++q) x += part[k][tid + 32 * q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            t[k] = x;
        }
    };
    if (tid < 32) {
        double t[NV];
        warp_total(t);
        if (tid == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) partials[(size_t)k * nb + bid] = t[k];
            __threadfence();
            last = atomicAdd(ticket, 1u) == nb - 1;
        }
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = 0.0;
        for (unsigned q = tid; q < nb; q += kST) x += __ldcg(&partials[(size_t)k * nb + q]);
        part[k][tid] = x;
    }
    __syncthreads();
    if (tid < 32) {
        warp_total(v);
        if (tid == 0) *ticket = 0u;
    }
    return tid == 0;
}

// f(j, two): the nodes 2 q and 2 q + 1 (two) or the last node alone, q over the grid.
template <typename F>
__device__ __forceinline__ void for_pairs(long long n, F f) {
    const long long pairs = n >> 1, stride = (long long)gridDim.x * kST;
    const long long t = (long long)blockIdx.x * kST + threadIdx.x;
#pragma unroll 2
    for (long long q = t; q < pairs; q += stride) f(2 * q, true);
    if ((n & 1) && t == 0) f(n - 1, false);
}

// Ap = K p and p . Ap; alpha = (r . z) / (p . Ap).
template <int DIM, int ORDER>
__global__ void __launch_bounds__(kST, 3)
    k_pcg_applyK(const double* __restrict__ p, double* __restrict__ Ap, const unsigned char* __restrict__ mask, Red red,
                 Geom g, double ck, int zc) {
    const Column<DIM> m(g, zc, ORDER / 2, false);
    double acc[1] = {0.0};
    if (m.valid) {
        SoftLap<DIM, ORDER, Values> lap(Values{p}, g, m.ix, m.iy);
        int j = m.j;
        lap.start(j, m.z0);
        for (int iz = m.z0; iz < m.z1; ++iz) {
            const bool dir = mask && mask[j];
            double pj;
            const double L = lap.next(j, iz, &pj);
            int ends = (m.ix == 0 || m.ix == g.nx) + (m.iy == 0 || m.iy == g.ny);
            if (DIM == 3) ends += (iz == 0 || iz == g.nz);
            // the weight's power of two goes into the constant's exponent
            const double c = __hiloint2double(__double2hiint(ck) - (ends << 20), __double2loint(ck));
            const double v = dir ? 0.0 : c * L;
            Ap[j] = v;
            acc[0] = fma(pj, v, acc[0]);
            j += lap.sZ;
        }
    }
    if (pcg_sum<1>(acc, red.partials, red.ticket)) {
        red.sc[SC_P_PAP] = acc[0];
        red.sc[SC_P_ALPHA] = acc[0] != 0.0 ? red.sc[SC_P_RZ] / acc[0] : 0.0;  // p = 0 only for a zero residual
    }
}

// XV: x is 16-byte aligned (it is the caller's; the other arrays are the workspace's).
template <bool XV>
__global__ void __launch_bounds__(kST, 4) k_pcg_xr(long long n, double* __restrict__ x, double* __restrict__ r,
                                                   const double* __restrict__ p, const double* __restrict__ Ap,
                                                   float* __restrict__ bf, Red red, int first) {
    const double alpha = red.sc[SC_P_ALPHA];
    double acc[1] = {0.0};
    for_pairs(n, [&](long long j, bool two) {
        if (two) {
            const double2 pv = *reinterpret_cast<const double2*>(p + j), av = *reinterpret_cast<const double2*>(Ap + j);
            double2 rv = *reinterpret_cast<const double2*>(r + j);
            double2 xv = make_double2(0.0, 0.0);
            if (!first) {
                if (XV) xv = *reinterpret_cast<const double2*>(x + j);
                else xv = make_double2(x[j], x[j + 1]);
            }
            xv.x = fma(alpha, pv.x, xv.x), xv.y = fma(alpha, pv.y, xv.y);
            rv.x = fma(-alpha, av.x, rv.x), rv.y = fma(-alpha, av.y, rv.y);
            if (XV) {
                *reinterpret_cast<double2*>(x + j) = xv;
            } else {
                x[j] = xv.x;
                x[j + 1] = xv.y;
            }
            *reinterpret_cast<double2*>(r + j) = rv;
            *reinterpret_cast<float2*>(bf + j) = make_float2(soft64::to_f32(rv.x), soft64::to_f32(rv.y));
            acc[0] = fma(rv.x, rv.x, fma(rv.y, rv.y, acc[0]));
        } else {
            x[j] = fma(alpha, p[j], first ? 0.0 : x[j]);
            const double v = fma(-alpha, Ap[j], r[j]);
            r[j] = v;
            bf[j] = soft64::to_f32(v);
            acc[0] = fma(v, v, acc[0]);
        }
    });
    if (pcg_sum<1>(acc, red.partials, red.ticket)) red.sc[SC_P_RR] = acc[0];
}

// r . z and z . Ap; flexible (Polak-Ribiere) beta = -alpha (z . Ap) / (r . z)_old.
__global__ void __launch_bounds__(kST, 4) k_pcg_dots(long long n, const double* __restrict__ r, const float* __restrict__ z,
                                                     const double* __restrict__ Ap, Red red) {
    double acc[2] = {0.0, 0.0};
    for_pairs(n, [&](long long j, bool two) {
        if (two) {
            const double2 rv = *reinterpret_cast<const double2*>(r + j);
            const float2 zv = *reinterpret_cast<const float2*>(z + j);
            const double z0 = soft64::to_f64(zv.x), z1 = soft64::to_f64(zv.y);
            acc[0] = fma(rv.x, z0, fma(rv.y, z1, acc[0]));
            if (Ap) {
                const double2 av = *reinterpret_cast<const double2*>(Ap + j);
                acc[1] = fma(av.x, z0, fma(av.y, z1, acc[1]));
            }
        } else {
            const double zz = soft64::to_f64(z[j]);
            acc[0] = fma(r[j], zz, acc[0]);
            if (Ap) acc[1] = fma(zz, Ap[j], acc[1]);
        }
    });
    if (pcg_sum<2>(acc, red.partials, red.ticket)) {
        const double rz_old = red.sc[SC_P_RZ];
        red.sc[SC_P_BETA] = (!Ap || rz_old == 0.0) ? 0.0 : -red.sc[SC_P_ALPHA] * acc[1] / rz_old;
        red.sc[SC_P_RZ] = acc[0];
    }
}

__global__ void __launch_bounds__(kST, 4) k_pcg_p(long long n, double* __restrict__ p, const float* __restrict__ z,
                                                  const double* __restrict__ sc, int first) {
    const double beta = first ? 0.0 : sc[SC_P_BETA];
    for_pairs(n, [&](long long j, bool two) {
        if (two) {
            const float2 zv = *reinterpret_cast<const float2*>(z + j);
            double2 v = make_double2(soft64::to_f64(zv.x), soft64::to_f64(zv.y));
            if (!first) {
                const double2 o = *reinterpret_cast<const double2*>(p + j);
                v.x = fma(beta, o.x, v.x), v.y = fma(beta, o.y, v.y);
            }
            *reinterpret_cast<double2*>(p + j) = v;
        } else {
            const double zz = soft64::to_f64(z[j]);
            p[j] = first ? zz : fma(beta, p[j], zz);
        }
    });
}

// One PCG iteration's vector part in one launch of one thread-block cluster, for grids of up to
// kPcgClusterNodes nodes: beta from r . z and z . Ap, p, Ap, alpha, x and r, with cluster barriers in
// place of launches.  The sums are those of the passes above in another order.
//
// Bound: latency and the FP64 pipe of 16 SMs.  Neighbours' p comes from L2 (__ldcg: another CTA wrote
// it).  As four launches the part costs 22 us whatever the size, here 14 at 129^2.  Whole Riesz maps:
// 65^2 680 and 568 us, 129^2 740 and 672, 191^2 1036 and 981, 33^3 1084 and 958; with four to six
// nodes per thread, past 36864 nodes, no gain (226x241 1103 and 1102).
constexpr int kClusterThreads = 768;  // 85 registers, which the stencil sum needs
constexpr int kClusterCtas = 16;

struct Latest {  // values that other CTAs may have written in this launch
    const double* p;
    __device__ __forceinline__ double operator()(int i) const { return __ldcg(p + i); }
};

__device__ __forceinline__ void pcg_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void store_to_cta(double* slot, int cta, double v) {
    unsigned there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"((unsigned)__cvta_generic_to_shared(slot)), "r"(cta));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(there), "d"(v) : "memory");
}
#include "cluster_total.cuh"

// NPT nodes per thread at most, whose values stay in registers.
template <int DIM, int ORDER, int NPT>
__global__ void __launch_bounds__(kClusterThreads, 1)
    k_pcg_cluster(double* __restrict__ x, double* __restrict__ r, double* p, double* __restrict__ Ap,
                  const float* __restrict__ z, float* __restrict__ bf, const unsigned char* __restrict__ mask,
                  double* __restrict__ sc, Geom g, double ck, int first) {
    __shared__ double part[2][kClusterThreads];
    __shared__ double slots[3][2][kClusterCtas + 1];
    const int n = (int)g.np, chunk = (n + kClusterCtas - 1) / kClusterCtas;
    const int lo = min((int)blockIdx.x * chunk, n), hi = min(lo + chunk, n), t0 = lo + (int)threadIdx.x;
    const double rz_old = sc[SC_P_RZ], alpha_old = sc[SC_P_ALPHA];
    double zv[NPT], rv[NPT], pv[NPT], av[NPT], xv[NPT], rz[2] = {0.0, 0.0};
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        const int j = t0 + q * kClusterThreads;
        zv[q] = rv[q] = pv[q] = av[q] = xv[q] = 0.0;
        if (j < hi) {
            zv[q] = soft64::to_f64(z[j]);
            rv[q] = r[j];
            if (!first) av[q] = Ap[j], pv[q] = p[j], xv[q] = x[j];
        }
    }
    pcg_cluster_sync();  // every CTA has started
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        rz[0] = fma(rv[q], zv[q], rz[0]);
        if (!first) rz[1] = fma(av[q], zv[q], rz[1]);
    }
    cluster_total<2>(rz, part, slots[0]);
    const double beta = first || rz_old == 0.0 ? 0.0 : -alpha_old * rz[1] / rz_old;
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        const int j = t0 + q * kClusterThreads;
        pv[q] = first ? zv[q] : fma(beta, pv[q], zv[q]);
        if (j < hi) p[j] = pv[q];
    }
    pcg_cluster_sync();
    double pap[1] = {0.0};
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        const int j = t0 + q * kClusterThreads;
        if (j >= hi) continue;
        const unsigned t = (unsigned)j / (unsigned)g.sx;
        const int ix = j - (int)t * g.sx, iz = DIM == 3 ? (int)(t / (unsigned)g.sy) : 0, iy = (int)t - iz * g.sy;
        if (!column_in_range(g, ix, iy, iz, iz + 1, ORDER / 2, kSitePcgCluster)) continue;
        SoftLap<DIM, ORDER, Latest> lap(Latest{p}, g, ix, iy);
        double pj;
        lap.start(j, iz);
        const double L = lap.next(j, iz, &pj);
        int ends = (ix == 0 || ix == g.nx) + (iy == 0 || iy == g.ny);
        if (DIM == 3) ends += (iz == 0 || iz == g.nz);
        const double c = __hiloint2double(__double2hiint(ck) - (ends << 20), __double2loint(ck));
        av[q] = mask && mask[j] ? 0.0 : c * L;
        Ap[j] = av[q];
        pap[0] = fma(pv[q], av[q], pap[0]);
    }
    cluster_total<1>(pap, part, slots[1]);
    const double alpha = pap[0] != 0.0 ? rz[0] / pap[0] : 0.0;  // p = 0 only for a zero residual
    double rr[1] = {0.0};
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        const int j = t0 + q * kClusterThreads;
        if (j >= hi) continue;
        x[j] = fma(alpha, pv[q], xv[q]);
        const double v = fma(-alpha, av[q], rv[q]);
        r[j] = v;
        bf[j] = soft64::to_f32(v);
        rr[0] = fma(v, v, rr[0]);
    }
    cluster_total<1>(rr, part, slots[2]);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc[SC_P_BETA] = beta;
        sc[SC_P_RZ] = rz[0];
        sc[SC_P_PAP] = pap[0];
        sc[SC_P_ALPHA] = alpha;
        sc[SC_P_RR] = rr[0];
    }
}

// w = 1 / (1 + beta) on the nodes of absorbing faces (other entries are not read).
__global__ void __launch_bounds__(kST) k_face_weights(Geom g, const double* __restrict__ kap, double* __restrict__ w) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < g.np; j += stride) {
        const unsigned t = (unsigned)j / (unsigned)g.sx;
        const int ix = (int)((unsigned)j - t * (unsigned)g.sx);
        const int iz = (int)(t / (unsigned)g.sy);
        const int iy = (int)(t - (unsigned)iz * (unsigned)g.sy);
        const int nb = num_abc(g, ix, iy, iz);
        if (nb) w[j] = 1.0 / (1.0 + nb * sqrt(kap[j]));
    }
}

// z-planes per thread: eight amortise a chunk's two extra planes; fewer where eight would leave
// the grid short of one wave of resident blocks.
int soft_zc(const Geom& g, int per_sm) {
    if (g.dim != 3) return 1;
    const long long bxy = ((long long)g.sx * g.sy + kST - 1) / kST;
    int zc = 8;
    while (zc > 2 && bxy * ((g.sz + zc - 1) / zc) < 152ll * per_sm) zc >>= 1;
    return zc;
}

template <int DIM, int ORDER, int FLAGS, int B>
void soft_launch_b(const Geom& g, const double* cur, double* prev, const double* kap, const double* wface,
                   const double* S, double cs, double sn, bool src_faces, bool reverse, cudaStream_t st) {
    const int zc = soft_zc(g, B);
    const dim3 grid((unsigned)(((long long)g.sx * g.sy + kST - 1) / kST), (unsigned)((g.sz + zc - 1) / zc));
    if ((FLAGS & kStepSrc) && src_faces)
        k_step_soft<DIM, ORDER, FLAGS, true, B><<<grid, kST, 0, st>>>(cur, prev, kap, wface, S, cs, sn, g, zc, reverse);
    else
        k_step_soft<DIM, ORDER, FLAGS, false, B><<<grid, kST, 0, st>>>(cur, prev, kap, wface, S, cs, sn, g, zc, reverse);
}

// Six blocks per SM on 7-point grids of two such waves and more, five on smaller ones; four of the
// 13-point kernel (see k_step_soft).
template <int DIM, int ORDER, int FLAGS>
void soft_launch(const Geom& g, const double* cur, double* prev, const double* kap, const double* wface,
                 const double* S, double cs, double sn, bool src_faces, bool reverse, cudaStream_t st) {
    if constexpr (DIM == 3 && ORDER == 2) {
        const long long blocks = ((long long)g.sx * g.sy + kST - 1) / kST * ((g.sz + 7) / 8);
        if (blocks >= 2ll * 152 * 6)
            soft_launch_b<DIM, ORDER, FLAGS, 6>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st);
        else
            soft_launch_b<DIM, ORDER, FLAGS, 5>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st);
    } else {
        soft_launch_b<DIM, ORDER, FLAGS, 4>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st);
    }
}

template <int DIM, int ORDER>
void soft_flags(const Geom& g, const double* cur, double* prev, const double* kap, const double* wface,
                const double* S, double cs, double sn, int flags, bool src_faces, bool reverse, cudaStream_t st) {
    switch (flags) {
        case 0: soft_launch<DIM, ORDER, 0>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st); break;
        case kStepSrc:
            soft_launch<DIM, ORDER, kStepSrc>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st);
            break;
        case kStepPrevScaled:
            soft_launch<DIM, ORDER, kStepPrevScaled>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st);
            break;
        case kStepNoDiv:
            soft_launch<DIM, ORDER, kStepNoDiv>(g, cur, prev, kap, wface, S, cs, sn, src_faces, reverse, st);
            break;
        default:
            soft_launch<DIM, ORDER, kStepPrevScaled | kStepNoDiv>(g, cur, prev, kap, wface, S, cs, sn, src_faces,
                                                                  reverse, st);
            break;
    }
}

}  // namespace

void launch_face_weights(const Geom& g, const double* kap, double* w, cudaStream_t st) {
    note_launch(1);
    const long long b = std::min<long long>((g.np + kST - 1) / kST, 152 * 8);
    k_face_weights<<<(unsigned)b, kST, 0, st>>>(g, kap, w);
}

void launch_step_soft(const Geom& g, int order, const double* cur, double* prev, const double* kap,
                      const double* wface, const double* S, double cs, double sn, int flags, bool src_faces,
                      bool reverse, cudaStream_t st) {
    note_launch(1);
    if (g.dim == 3) {
        if (order == 2) soft_flags<3, 2>(g, cur, prev, kap, wface, S, cs, sn, flags, src_faces, reverse, st);
        else soft_flags<3, 4>(g, cur, prev, kap, wface, S, cs, sn, flags, src_faces, reverse, st);
    } else {
        if (order == 2) soft_flags<2, 2>(g, cur, prev, kap, wface, S, cs, sn, flags, src_faces, reverse, st);
        else soft_flags<2, 4>(g, cur, prev, kap, wface, S, cs, sn, flags, src_faces, reverse, st);
    }
}

// The endpoint kernels: `run` is called with the dimension and order as compile-time constants.
template <typename F>
static void by_stencil(const Geom& g, int order, F run) {
    using std::integral_constant;
    note_launch(1);
    if (g.dim == 3) {
        if (order == 2) run(integral_constant<int, 3>(), integral_constant<int, 2>());
        else run(integral_constant<int, 3>(), integral_constant<int, 4>());
    } else {
        if (order == 2) run(integral_constant<int, 2>(), integral_constant<int, 2>());
        else run(integral_constant<int, 2>(), integral_constant<int, 4>());
    }
}

static dim3 column_grid(const Geom& g, int zc) {
    return dim3((unsigned)(((long long)g.sx * g.sy + kST - 1) / kST), (unsigned)((g.sz + zc - 1) / zc));
}

static double h_pow(const Geom& g) { return (g.dim == 3 ? g.h * g.h * g.h : g.h * g.h) / (g.h * g.h); }

void launch_start_soft(const Geom& g, int order, const double* w0, const double* w1, double* y0, double* y1,
                       const double* kap, const double* wface, const double* S, bool src_faces, double dt, int zc,
                       cudaStream_t st) {
    by_stencil(g, order, [&](auto D, auto O) {
        const dim3 grid = column_grid(g, zc);
        if (S)
            k_start_soft<D(), O(), true><<<grid, kST, 0, st>>>(w0, w1, y0, y1, kap, wface, S, g, dt, zc, src_faces);
        else
            k_start_soft<D(), O(), false><<<grid, kST, 0, st>>>(w0, w1, y0, y1, kap, wface, S, g, dt, zc, 0);
    });
}

void launch_end_soft(const Geom& g, int order, int mode, const double* yN, const double* yNm1, const double* w0,
                     const double* w1, const double* kap, const double* mass, const double* wface, const double* S,
                     bool src_faces, double cs, double sn, double* out0, double* out1, Red red, double dt, int zc,
                     cudaStream_t st) {
    by_stencil(g, order, [&](auto D, auto O) {
        const dim3 grid = column_grid(g, zc);
        const double ck = h_pow(g), id = 1.0 / dt, hc = 0.5 * cs, hs = 0.5 * sn;
        const int sf = src_faces ? 1 : 0;
        auto go = [&](auto kernel) {
            kernel<<<grid, kST, 0, st>>>(yN, yNm1, w0, w1, kap, mass, wface, S, hc, hs, out0, out1, red, g, id, ck, zc,
                                         sf);
        };
        if (mode == 0) S ? go(k_end_soft<D(), O(), true, 0>) : go(k_end_soft<D(), O(), false, 0>);
        else S ? go(k_end_soft<D(), O(), true, 1>) : go(k_end_soft<D(), O(), false, 1>);
    });
}

void launch_adj_prep_soft(const Geom& g, const double* b, const double* minv, const double* wface, double* t, int zc,
                          cudaStream_t st) {
    note_launch(1);
    if (g.dim == 3) k_adj_prep_soft<3><<<column_grid(g, zc), kST, 0, st>>>(b, minv, wface, t, g, zc);
    else k_adj_prep_soft<2><<<column_grid(g, zc), kST, 0, st>>>(b, minv, wface, t, g, zc);
}

void launch_adj_start_soft(const Geom& g, int order, const double* a, const double* t, const double* minv,
                           const double* kap, const double* wface, double* cur, double* prev, double dt, int zc,
                           cudaStream_t st) {
    by_stencil(g, order, [&](auto D, auto O) {
        k_adj_start_soft<D(), O()>
            <<<column_grid(g, zc), kST, 0, st>>>(a, t, minv, kap, wface, cur, prev, g, 1.0 / dt, zc);
    });
}

void launch_adj_final_soft(const Geom& g, int order, int mode, const double* s, const double* u1, const double* mass,
                           const double* kap, const double* wface, const double* minv, const double* z0,
                           const double* z1, const double* d0, const double* d1, double* o0, double* o1, double* gt1,
                           Red red, double dt, int zc, cudaStream_t st) {
    by_stencil(g, order, [&](auto D, auto O) {
        const double cq = 0.5 * dt * dt * h_pow(g);
        auto go = [&](auto kernel) {
            kernel<<<column_grid(g, zc), kST, 0, st>>>(s, u1, mass, kap, wface, minv, z0, z1, d0, d1, o0, o1, gt1, red, g,
                                                       dt, cq, zc);
        };
        mode == 0 ? go(k_adj_final_soft<D(), O(), 0>) : go(k_adj_final_soft<D(), O(), 1>);
    });
}

static unsigned pcg_blocks(long long n) {
    return (unsigned)std::max<long long>(1, std::min<long long>((n / 2 + kST - 1) / kST, kPcgBlocks / 2));
}

void launch_pcg_applyK(const Geom& g, int order, const unsigned char* mask, const double* p, double* Ap, Red red, int zc,
                       cudaStream_t st) {
    by_stencil(g, order, [&](auto D, auto O) {
        // K = W (-Lap): -Lt comes from the kernel, so the constant is negative
        k_pcg_applyK<D(), O()><<<column_grid(g, zc), kST, 0, st>>>(p, Ap, mask, red, g, -h_pow(g), zc);
    });
}

void launch_pcg_xr(long long n, double* x, double* r, const double* p, const double* Ap, float* bf, Red red, bool first,
                   cudaStream_t st) {
    note_launch(1);
    if (((uintptr_t)x & 15u) == 0) k_pcg_xr<true><<<pcg_blocks(n), kST, 0, st>>>(n, x, r, p, Ap, bf, red, first);
    else k_pcg_xr<false><<<pcg_blocks(n), kST, 0, st>>>(n, x, r, p, Ap, bf, red, first);
}

// f(kernel, its launch configuration) for the k_pcg_cluster of this grid.
template <typename F>
static void with_pcg_cluster(const Geom& g, int order, cudaStream_t st, F f) {
    auto go = [&](auto kernel) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kClusterCtas);
        cfg.blockDim = dim3(kClusterThreads);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kClusterCtas;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        // (a refusal stays pending, for cuda_status or pcg_cluster_fits)
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) f(kernel, cfg);
    };
    const bool two = g.np <= 2ll * kClusterCtas * kClusterThreads;
    static_assert(3ll * kClusterCtas * kClusterThreads >= kPcgClusterNodes, "nodes per thread");
    by_stencil(g, order, [&](auto D, auto O) {
        if (two) go(k_pcg_cluster<D(), O(), 2>);
        else go(k_pcg_cluster<D(), O(), 3>);
    });
}

// Grids of up to kPcgClusterNodes nodes (see there).
bool pcg_cluster_fits(const Geom& g, int order) {
    if (g.np > kPcgClusterNodes) return false;
    int clusters = 0;
    with_pcg_cluster(g, order, nullptr, [&](auto kernel, cudaLaunchConfig_t& cfg) {
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) clusters = 0;
    });
    note_launch(-1);  // (by_stencil counts a launch)
    if (clusters < 1) cudaGetLastError();
    return clusters > 0;
}

void launch_pcg_cluster(const Geom& g, int order, const unsigned char* mask, double* x, double* r, double* p, double* Ap,
                        const float* z, float* bf, Red red, bool first, cudaStream_t st) {
    const double ck = -h_pow(g);
    with_pcg_cluster(g, order, st, [&](auto kernel, cudaLaunchConfig_t& cfg) {
        cudaLaunchKernelEx(&cfg, kernel, x, r, p, Ap, z, bf, mask, red.sc, g, ck, first ? 1 : 0);
    });
}

void launch_pcg_dots(long long n, const double* r, const float* z, const double* Ap, Red red, cudaStream_t st) {
    note_launch(1);
    k_pcg_dots<<<pcg_blocks(n), kST, 0, st>>>(n, r, z, Ap, red);
}

void launch_pcg_p(long long n, double* p, const float* z, Red red, bool first, cudaStream_t st) {
    note_launch(1);
    k_pcg_p<<<pcg_blocks(n), kST, 0, st>>>(n, p, z, red.sc, first);
}

CMCG_CHECK_TU(soft)

}  // namespace cmcg
