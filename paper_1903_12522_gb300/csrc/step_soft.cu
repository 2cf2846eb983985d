// FP64 leapfrog steps with the stencil sum in integer arithmetic (soft64.cuh).
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "soft64.cuh"

namespace cmcg {

namespace {

using soft64::Term;

constexpr int kST = 256;

// The negated unscaled Laplacian at a node in plain FP64, for the values the fixed-point sum
// does not take.  Out of line: inlined, its additions would be predicated into every update.
template <int ORDER>
__device__ __noinline__ double neg_lap_plain(const double* __restrict__ cur, const Geom& g, int j, int ix, int iy,
                                             int iz) {
    auto f = [cur](long long i) { return cur[i]; };
    return -lap_t<ORDER, double>(g, f, (long long)j, ix, iy, iz);
}

// The update on an absorbing face, w = 1 / (1 + beta): out = w rhs - (1 - beta) w yp with
// (1 - beta) w = 2 w - 1, and the adjoint's first and last variants (the previous term already
// scaled; no division).  Out of line for the same reason.
template <int FLAGS>
__device__ __noinline__ double face_update(double rhs, double yp, double w) {
    if (FLAGS & kStepNoDiv) {
        if (FLAGS & kStepPrevScaled) return rhs - yp;
        return rhs - (2.0 - 1.0 / w) * yp;
    }
    if (FLAGS & kStepPrevScaled) return (rhs - yp) * w;
    return fma(rhs, w, -(fma(2.0, w, -1.0) * yp));
}

__device__ __noinline__ double add_source(double d, const double* __restrict__ S, int j, double cs, double sn) {
    const double2 s = reinterpret_cast<const double2*>(S)[j];
    return d + fma(s.x, cs, s.y * sn);
}

// One leapfrog step, one thread per (x, y) column of zc planes (2D: one node).
//
// Bound: issue slots of the integer pipes and latency (FP64 work left per update: 2 y - y_prev
// and the fused multiply-add with kappa, against nine operations and, on the faces, a square
// root and a division).  The z-neighbours' terms stay in registers.
template <int DIM, int ORDER, int FLAGS, bool SRC_FACES>
__global__ void __launch_bounds__(kST, ORDER == 2 ? 4 : 3)
    k_step_soft(const double* __restrict__ cur, double* __restrict__ prev_out, const double* __restrict__ kap,
                const double* __restrict__ wface, const double* __restrict__ S, double cs, double sn, Geom g, int zc,
                int reverse) {
    const int plane = g.sx * g.sy;
    const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int by = reverse ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    const int p = bx * kST + (int)threadIdx.x;
    if (p >= plane) return;
    const int iy = (int)((unsigned)p / (unsigned)g.sx), ix = p - iy * g.sx;
    const int z0 = DIM == 3 ? by * zc : 0, z1 = DIM == 3 ? min(z0 + zc, g.sz) : 1;
    if (!column_in_range(g, ix, iy, z0, z1, ORDER / 2, kSiteColumn)) return;
    const int sZ = plane;
    const int oxm = (int)off_m1(ix, 1), oxp = (int)off_p1(ix, g.nx, 1);
    const int oym = (int)off_m1(iy, g.sx), oyp = (int)off_p1(iy, g.ny, g.sx);
    bool fxy = (ix == 0 && (g.abc & 1u)) || (ix == g.nx && (g.abc & 2u)) || (iy == 0 && (g.abc & 4u)) ||
               (iy == g.ny && (g.abc & 8u));
    int ox2m = 0, ox2p = 0, oy2m = 0, oy2p = 0;
    if (ORDER == 4) {
        ox2m = (int)off_m2(ix, 1), ox2p = (int)off_p2(ix, g.nx, 1);
        oy2m = (int)off_m2(iy, g.sx), oy2p = (int)off_p2(iy, g.ny, g.sx);
    }
    int j = p + sZ * z0;
    double yc = cur[j];
    Term c = soft64::term(yc), zm{}, zp{}, zm2{}, zp2{};
    double yz = 0.0;  // ORDER 4: the raw value of plane iz + 1
    if (DIM == 3) {
        zm = soft64::term(cur[j + (z0 > 0 ? -sZ : sZ)]);
        if (ORDER == 4) {
            zm2 = soft64::term(cur[j + (int)off_m2(z0, sZ)]);
            yz = cur[j + (z0 < g.nz ? sZ : -sZ)];
            zp = soft64::term(yz);
        }
    }
    for (int iz = z0; iz < z1; ++iz) {
        double znew = 0.0;
        if (DIM == 3) znew = cur[j + (ORDER == 2 ? (iz < g.nz ? sZ : -sZ) : (int)off_p2(iz, g.nz, sZ))];
        const double x0 = cur[j + oxm], x1 = cur[j + oxp], y0 = cur[j + oym], y1 = cur[j + oyp];
        double u0 = 0.0, u1 = 0.0, v0 = 0.0, v1 = 0.0;
        if (ORDER == 4) u0 = cur[j + ox2m], u1 = cur[j + ox2p], v0 = cur[j + oy2m], v1 = cur[j + oy2p];
        const double k = kap[j], yp = prev_out[j];
        const Term a0 = soft64::term(x0), a1 = soft64::term(x1), b0 = soft64::term(y0), b1 = soft64::term(y1);
        unsigned e = soft64::max3(soft64::max3(c.e, a0.e, a1.e), b0.e, b1.e);
        if (DIM == 3) {
            if (ORDER == 2) zp = soft64::term(znew);
            else zp2 = soft64::term(znew);
            e = soft64::max3(e, zm.e, zp.e);
        }
        Term c0{}, c1{}, d0{}, d1{};
        if (ORDER == 4) {
            c0 = soft64::term(u0), c1 = soft64::term(u1), d0 = soft64::term(v0), d1 = soft64::term(v1);
            e = soft64::max3(soft64::max3(e, c0.e, c1.e), d0.e, d1.e);
            if (DIM == 3) e = soft64::max3(e, zm2.e, zp2.e);
        }
        // L = -Lt(y)
        bool ok = soft64::in_range(e);
        const long long C = soft64::align(c, e);
        long long s1 = (soft64::align(a0, e) + soft64::align(a1, e)) + (soft64::align(b0, e) + soft64::align(b1, e));
        if (DIM == 3) s1 += soft64::align(zm, e) + soft64::align(zp, e);
        double L;
        bool big;
        if (ORDER == 2) {
            L = soft64::to_double(s1 - (DIM == 3 ? 4 * C + 2 * C : 4 * C), e, &big);
        } else {
            // 3/4 of the 4th-order sum: a1 - a2 / 16 - (DIM 15/8) y, so that its weights are shifts
            long long s2 = (soft64::align(c0, e) + soft64::align(c1, e)) + (soft64::align(d0, e) + soft64::align(d1, e));
            if (DIM == 3) s2 += soft64::align(zm2, e) + soft64::align(zp2, e);
            const long long q = DIM == 3 ? 6 * C - (3 * C >> 3) : 4 * C - (C >> 2);
            L = soft64::to_double(s1 - (s2 >> 4) - q, e, &big);
        }
        ok = ok && big;
        double kk = k;
        if (ORDER == 4) kk = k * (4.0 / 3.0);
        if (!ok) {
            L = neg_lap_plain<ORDER>(cur, g, j, ix, iy, iz);
            kk = k;
        }
        const bool fz = DIM == 3 && ((iz == 0 && (g.abc & 16u)) || (iz == g.nz && (g.abc & 32u)));
        double out;
        if (fxy || fz) {
            double rhs = fma(kk, L, 2.0 * yc);
            if (FLAGS & kStepSrc) rhs = add_source(rhs, S, j, cs, sn);
            out = face_update<FLAGS>(rhs, yp, wface[j]);
        } else {
            out = fma(kk, L, fma(2.0, yc, -yp));
            if ((FLAGS & kStepSrc) && !SRC_FACES) out = add_source(out, S, j, cs, sn);
        }
        prev_out[j] = out;
        if (DIM == 3) {
            if (ORDER == 2) {
                zm = c;
                c = zp;
                yc = znew;
            } else {
                zm2 = zm;
                zm = c;
                c = zp;
                zp = zp2;
                yc = yz;
                yz = znew;
            }
        }
        j += sZ;
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

template <int DIM, int ORDER, int FLAGS>
void soft_launch(const Geom& g, const double* cur, double* prev, const double* kap, const double* wface,
                 const double* S, double cs, double sn, bool src_faces, bool reverse, cudaStream_t st) {
    const int zc = soft_zc(g, ORDER == 2 ? 4 : 3);
    const dim3 grid((unsigned)(((long long)g.sx * g.sy + kST - 1) / kST), (unsigned)((g.sz + zc - 1) / zc));
    if ((FLAGS & kStepSrc) && src_faces)
        k_step_soft<DIM, ORDER, FLAGS, true><<<grid, kST, 0, st>>>(cur, prev, kap, wface, S, cs, sn, g, zc, reverse);
    else
        k_step_soft<DIM, ORDER, FLAGS, false><<<grid, kST, 0, st>>>(cur, prev, kap, wface, S, cs, sn, g, zc, reverse);
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

CMCG_CHECK_TU(soft)

}  // namespace cmcg
