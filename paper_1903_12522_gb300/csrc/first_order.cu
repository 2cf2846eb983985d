// First-order (mixed) formulation of Sec. 3 on a staggered grid: v = y_t on the nodes,
// p = grad y on the grid links, stepped with the staggered leapfrog
//
//   p_a^{n+1/2} = p_a^{n-1/2} + tau (v_{j+e_a} - v_j)                      tau = dt / h
//   v^{n+1}     = [(1 - beta) v^n - sigma sum_a (p_a(j - e_a) - p_a(j)) / w_a(j_a)
//                  + Re(S e^{-i w t_{n+1/2}}) / dt] / (1 + beta)             sigma = kappa h / dt
//
// which is the semi-discrete Eq. mixWE  M v' + B v = -G^T W_e p + F,  p' = G v  with the lumped
// link mass W_e = h^d prod_{b != a} w(j_b) (so G^T W_e G = K of the second-order scheme),
// beta = (dt/2) M^-1 B = nb sqrt(kappa), S = dt^2 M^-1 F^ (the handle's source array) and
// w_a = 1/2 on the two end nodes of axis a.  Missing links (j_a = n_a) hold 0; Dirichlet nodes
// (kappa = 0) hold v = 0.
//
// State layout: p_x | p_y | (p_z) | v, each N_p long; p_a[j] is the link (j, j + e_a).
//
// Adjoint.  With E = diag(W_e, M) the E-adjoint of the homogeneous step, run on the
// variables (q, u) = (E^-1 pbar, (1 + beta)^-1 E^-1 vbar), is the same update with tau and
// sigma negated; so one kernel runs both the forward period and the backward period of
// Eq. mixJ_deriative_2, and the gradient's E-representer P* e - e needs no elliptic solve.
#include <math.h>

#include <algorithm>

#include "soft64.cuh"
#include "solver.h"

namespace cmcg {

namespace {

constexpr int kFT = 256;

inline dim3 fo_grid(const Geom& g, int zc) {
    const long long plane = (long long)g.sx * g.sy;
    return dim3((unsigned)((plane + kFT - 1) / kFT), (unsigned)((g.sz + zc - 1) / zc));
}

inline unsigned fo_vec_blocks(long long n) {
    long long b = (n + kFT - 1) / kFT;
    return (unsigned)std::max<long long>(1, std::min<long long>(b, kMaxBlocksReduce));
}

__device__ __forceinline__ double inv_w(int i, int n) { return (i == 0 || i == n) ? 2.0 : 1.0; }

// Link mass W_e of link (j, j + e_a), 0 where the link does not exist.
__device__ __forceinline__ double link_mass(const Geom& g, int a, int ix, int iy, int iz) {
    const int i[3] = {ix, iy, iz};
    const int n[3] = {g.nx, g.ny, g.nz};
    if (i[a] >= n[a]) return 0.0;
    double w = g.dim == 3 ? g.h * g.h * g.h : g.h * g.h;
    for (int b = 0; b < g.dim; ++b)
        if (b != a && (i[b] == 0 || i[b] == n[b])) w *= 0.5;
    return w;
}

// Component c of element e of a (dim + 1) N_p state, and the node's coordinates.
struct Elem {
    int comp, ix, iy, iz;
    long long j;
};

__device__ __forceinline__ Elem elem(const Geom& g, long long e) {
    Elem r;
    if (e >> 32 == 0 && g.np >> 32 == 0) {  // (the 64-bit divisions cost more than the rest of an element)
        const unsigned c = (unsigned)e / (unsigned)g.np, j = (unsigned)e - c * (unsigned)g.np;
        const unsigned t = j / (unsigned)g.sx, z = t / (unsigned)g.sy;
        r.comp = (int)c;
        r.j = j;
        r.ix = (int)(j - t * (unsigned)g.sx);
        r.iz = (int)z;
        r.iy = (int)(t - z * (unsigned)g.sy);
        return r;
    }
    r.comp = (int)(e / g.np);
    r.j = e - (long long)r.comp * g.np;
    const long long t = r.j / g.sx;
    r.ix = (int)(r.j - t * g.sx);
    r.iz = (int)(t / g.sy);
    r.iy = (int)(t - (long long)r.iz * g.sy);
    return r;
}

// The element's place in a stepping state whose rows have pitch px.
__device__ __forceinline__ long long place(const Geom& g, const Elem& r, int px) {
    return r.ix + px * (r.iy + g.sy * (r.iz + (long long)g.sz * r.comp));
}

// Energy weight of element e: W_e for a link component, M for the velocity.
__device__ __forceinline__ double e_weight(const Geom& g, const double* mass, const Elem& r) {
    return r.comp < g.dim ? link_mass(g, r.comp, r.ix, r.iy, r.iz) : mass[r.j];
}

// The face terms of k_fo_step.  The FP64 ones are out of line: inlined, the compiler makes their
// instructions conditional, and an FP64 instruction holds the pipe even where no lane executes it.
__device__ __forceinline__ bool is_zero(float k) { return k == 0.f; }
__device__ __forceinline__ bool is_zero(double k) { return soft64::is_zero(k); }
__device__ __forceinline__ float rounded_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rounded_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float face_beta(float k, int nb) { return __fmul_rn((float)nb, sqrtf(k)); }
__device__ __noinline__ double face_beta(double k, int nb) { return nb * sqrt(k); }
__device__ __forceinline__ float face_rhs(float v, float beta, float t) { return __fmaf_rn(1.f - beta, v, -t); }
__device__ __noinline__ double face_rhs(double v, double beta, double t) { return __fma_rn(1.0 - beta, v, -t); }
__device__ __forceinline__ float face_over(float x, float beta) { return x / (1.f + beta); }
__device__ __noinline__ double face_over(double x, double beta) { return x / (1.0 + beta); }

// One staggered leapfrog step for a column of z-planes (3D) or one node (2D).  SRC adds the
// source at t_{n+1/2} (cs, sn already divided by dt); ACC accumulates v^n e^{i w t_n} into acc.
// Consecutive lanes hold consecutive nodes of a row, so v_{j-1}, v_{j+1} and the old value of
// the link (j - 1, j) come from the neighbouring lanes (lane 0 and lane 31 load them); lanes
// past the last column take part in the shuffles but touch no memory.
template <typename T, int DIM, bool SRC, bool ACC>
__global__ void __launch_bounds__(kFT) k_fo_step(const T* __restrict__ sin_, T* __restrict__ sout,
                                                 const T* __restrict__ kap, const double* __restrict__ S, double cs,
                                                 double sn, T tau, T sig, Geom g, int zc, double* __restrict__ acc,
                                                 double ca, double sa, const unsigned char* __restrict__ scol) {
    const long long plane = (long long)g.sx * g.sy;
    const long long pidx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = pidx < plane;
    const long long pc = valid ? pidx : plane - 1;  // in-range stand-in for idle lanes
    const int iy = (int)(pc / g.sx);
    const int ix = (int)(pc - (long long)iy * g.sx);
    const int lane = threadIdx.x & 31;
    const int z0 = DIM == 3 ? (int)blockIdx.y * zc : 0;
    const int z1 = DIM == 3 ? min(z0 + zc, g.sz) : 1;
    if (z0 >= z1) return;  // uniform over the block
    const long long np = g.np;
    const long long sZ = plane;
    const T* px = sin_;
    const T* py = sin_ + np;
    const T* pz = sin_ + 2 * np;
    const T* v = sin_ + (long long)DIM * np;
    T* qx = sout;
    T* qy = sout + np;
    T* qz = sout + 2 * np;
    T* w = sout + (long long)DIM * np;
    const T rx = (T)inv_w(ix, g.nx), ry = (T)inv_w(iy, g.ny);
    const bool hx0 = ix > 0, hx1 = ix < g.nx, hy0 = iy > 0, hy1 = iy < g.ny;
    const bool vol = !SRC || !scol || scol[pc];  // a source in the column inside the grid
    int nbxy = 0;
    nbxy += (ix == 0) & (int)(g.abc & 1u);
    nbxy += (ix == g.nx) & (int)((g.abc >> 1) & 1u);
    nbxy += (iy == 0) & (int)((g.abc >> 2) & 1u);
    nbxy += (iy == g.ny) & (int)((g.abc >> 3) & 1u);
    constexpr unsigned kAll = 0xffffffffu;
    long long j = pc + sZ * z0;
    T vc = v[j];
    T pzl = T(0);  // new value of the z-link below (j - sZ, j)
    if (DIM == 3 && z0 > 0) pzl = pz[j - sZ] + tau * (vc - v[j - sZ]);
    for (int iz = z0; iz < z1; ++iz) {
        T vz = T(0), pzr = T(0);
        if (DIM == 3 && iz < g.nz) {
            vz = v[j + sZ];
            pzr = pz[j] + tau * (vz - vc);
        }
        const T pxo = px[j];  // old value of the link (j, j + 1) (0 in the slot j_x = n_x)
        const T vl = __shfl_up_sync(kAll, vc, 1), vr = __shfl_down_sync(kAll, vc, 1);
        const T pl = __shfl_up_sync(kAll, pxo, 1);
        const T vxm = hx0 ? (lane > 0 ? vl : v[j - 1]) : T(0);
        const T vxp = hx1 ? (lane < 31 ? vr : v[j + 1]) : T(0);
        const T pxlo = hx0 ? (lane > 0 ? pl : px[j - 1]) : T(0);
        const T pxr = hx1 ? pxo + tau * (vxp - vc) : T(0);
        const T pxl = hx0 ? pxlo + tau * (vc - vxm) : T(0);
        const T pyr = hy1 ? py[j] + tau * (v[j + g.sx] - vc) : T(0);
        const T pyl = hy0 ? py[j - g.sx] + tau * (vc - v[j - g.sx]) : T(0);
        T div = (pxl - pxr) * rx + (pyl - pyr) * ry;
        int nb = nbxy;
        if (DIM == 3) {
            div += (pzl - pzr) * (T)inv_w(iz, g.nz);
            nb += ((iz == 0) & (int)((g.abc >> 4) & 1u)) + ((iz == g.nz) & (int)((g.abc >> 5) & 1u));
        }
        const T k = __ldcs(kap + j);  // streamed: the fields are what the next step re-reads
        T out = T(0);
        if (!is_zero(k)) {
            // (beta only on the faces: an FP64 square root for every node is most of the FP64 step)
            T rhs = rounded_mul(sig * k, div), beta = T(0);
            if (nb == 0) {
                rhs = vc - rhs;
            } else {
                beta = face_beta(k, nb);
                rhs = face_rhs(vc, beta, rhs);
            }
            if (SRC && (vol || iz == 0 || iz == g.nz)) {
                const double2 s = reinterpret_cast<const double2*>(S)[j];
                if (!(soft64::is_zero(s.x) && soft64::is_zero(s.y))) rhs += (T)__fma_rn(s.x, cs, __dmul_rn(s.y, sn));
            }
            out = nb == 0 ? rhs : face_over(rhs, beta);
        }
        if (valid) {
            if (ACC) {
                acc[2 * j] += (double)vc * ca;
                acc[2 * j + 1] += (double)vc * sa;
            }
            qx[j] = pxr;
            qy[j] = pyr;
            if (DIM == 3) qz[j] = pzr;
            w[j] = out;
        }
        if (DIM == 3) {
            pzl = pzr;
            vc = vz;
            j += sZ;
        }
    }
}

// The same step in FP32 on a 3D grid.  The stepping state's rows are padded to whole float4s (pitch
// px; the padding holds zeros), and so is kappa: a thread owns four consecutive nodes of a row and
// marches z.  Per four nodes nine 16-byte loads and four stores; the x neighbours come by shuffles.
// scol: the columns with sources inside the grid; elsewhere S (FP64, and its sum FP64 arithmetic) is
// read on the lowest and highest plane only.
//
// Bound: L2 and latency.  At 129^3 (36 B per node, 78 MB of state and kappa, which stay in L2) 41.6 us
// a step with one node per thread, of which 11 us are the source's FP64 arithmetic on every node and
// the rest 4-byte accesses; now 16 us backward, 19 us with a source on the faces.  Whole backward
// periods of 46 steps, before and after: 33^3 855 and 241 us, 97^3 1071 and 454, 129^3 1445 and 758,
// 257^3 8493 and 4761.
//
// The roundings are those of k_fo_step<float>, written out: same bits.
constexpr int kFR = 128;

struct F4 {
    float e[4];
};
__device__ __forceinline__ F4 get4(const float* p) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    return F4{{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ void put4(float* p, const F4& v) {
    *reinterpret_cast<float4*>(p) = make_float4(v.e[0], v.e[1], v.e[2], v.e[3]);
}
// p + tau (b - a): a link's update
__device__ __forceinline__ float link(float p, float tau, float b, float a) { return __fmaf_rn(tau, b - a, p); }
__device__ __forceinline__ F4 link4(const F4& p, float tau, const F4& b, const F4& a) {
    F4 r;
#pragma unroll
    for (int e = 0; e < 4; ++e) r.e[e] = link(p.e[e], tau, b.e[e], a.e[e]);
    return r;
}

template <bool SRC>
__global__ void __launch_bounds__(kFR, 8) k_fo_row(const float* __restrict__ in, float* __restrict__ out,
                                                   const float* __restrict__ kap, const double* __restrict__ S,
                                                   const unsigned char* __restrict__ scol, double cs, double sn,
                                                   float tau, float sig, Geom g, int px, int zc, int reverse) {
    const int cx = px >> 2, plane4 = cx * g.sy;
    const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int by = reverse ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    const int p = bx * kFR + (int)threadIdx.x;
    const int z0 = by * zc, z1 = min(z0 + zc, g.sz);
    if (!CMCG_RANGE_OK(z0, z1 - 1, g.sz, kSiteRow)) return;  // uniform over the block
    bool valid = p < plane4;
    int pc = valid ? p : plane4 - 1;  // (idle lanes take part in the shuffles)
    int iy = (int)((unsigned)pc / (unsigned)cx), ic = pc - iy * cx;
    if (!chunk_in_range(g, 4 * ic, iy, z0, z1, 1, kSiteRow)) {
        valid = false;
        pc = iy = ic = 0;
    }
    const int x0 = 4 * ic;
    const int lane = (int)threadIdx.x & 31;
    const bool first = ic == 0;
    const int xe = g.nx - x0;  // element of the node x = nx (0 .. 3 in a row's last chunk)
    const int m = min(4, g.sx - x0);
    const int sZ = px * g.sy;
    const long long field = (long long)sZ * g.sz;
    const float *qx = in, *qy = in + field, *qz = in + 2 * field, *v = in + 3 * field;
    float *ox = out, *oy = out + field, *oz = out + 2 * field, *ov = out + 3 * field;
    const bool hy0 = iy > 0, hy1 = iy < g.ny;
    const bool needl = lane == 0 && !first, needr = lane == 31 && xe >= 4;
    const float ry = hy0 && hy1 ? 1.f : 2.f;
    const int nby = (!hy0 ? (int)((g.abc >> 2) & 1u) : 0) + (!hy1 ? (int)((g.abc >> 3) & 1u) : 0);
    const int nbl = first ? (int)(g.abc & 1u) : 0, nbr = xe < 4 ? (int)((g.abc >> 1) & 1u) : 0;
    // the chunk's columns with sources: none, one (the x faces' nodes: with the FP64 sum for one node,
    // not for each of the four, a step with a source on the faces takes 13 instead of 17 us at 129^3),
    // several
    int cols = 0, col = 0;
    if (SRC) {
        for (int e = 0; e < m; ++e) {
            if (scol[x0 + e + g.sx * iy]) {
                ++cols;
                col = e;
            }
        }
    }
    int j = 4 * pc + sZ * z0;
    F4 c = get4(v + j), zl{};  // zl: the new value of the z-link below
    if (z0 > 0) zl = link4(get4(qz + j - sZ), tau, c, get4(v + j - sZ));
    for (int iz = z0; iz < z1; ++iz) {
        const bool top = iz == g.nz;
        const F4 up = get4(v + (top ? j : j + sZ)), zo = get4(qz + j);
        const F4 ya = get4(v + (hy0 ? j - px : j)), yb = get4(v + (hy1 ? j + px : j));
        const F4 yo = get4(qy + j), yl = get4(qy + (hy0 ? j - px : j));
        const F4 xo = get4(qx + j), k = get4(kap + j);
        float el = 0.f, er = 0.f, ep = 0.f;
        if (needl) {
            el = v[j - 1];
            ep = qx[j - 1];
        }
        if (needr) er = v[j + 4];
        float vl = __shfl_up_sync(0xffffffffu, c.e[3], 1), vr = __shfl_down_sync(0xffffffffu, c.e[0], 1);
        float pl = __shfl_up_sync(0xffffffffu, xo.e[3], 1);
        if (lane == 0) {
            vl = el;
            pl = ep;
        }
        if (lane == 31) vr = er;
        F4 zr{}, yr{}, yd{}, xr, div;
        if (!top) zr = link4(zo, tau, up, c);
        if (hy1) yr = link4(yo, tau, yb, c);
        if (hy0) yd = link4(yl, tau, c, ya);
        const float nx[4] = {c.e[1], c.e[2], c.e[3], vr};
#pragma unroll
        for (int e = 0; e < 4; ++e) xr.e[e] = e < xe ? link(xo.e[e], tau, nx[e], c.e[e]) : 0.f;
        const float xl[4] = {first ? 0.f : link(pl, tau, c.e[0], vl), xr.e[0], xr.e[1], xr.e[2]};
        const float rz = iz > 0 && !top ? 1.f : 2.f;
        F4 w;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            // (the products with 1 / w, 1 or 2, are exact)
            const float rx = (e == 0 && first) || e == xe ? 2.f : 1.f;
            div.e[e] = __fmaf_rn(xl[e] - xr.e[e], rx, (yd.e[e] - yr.e[e]) * ry);
            div.e[e] = __fmaf_rn(zl.e[e] - zr.e[e], rz, div.e[e]);
            w.e[e] = __fsub_rn(c.e[e], __fmul_rn(__fmul_rn(sig, k.e[e]), div.e[e]));
        }
        const int nbz = (iz == 0 ? (int)((g.abc >> 4) & 1u) : 0) + (top ? (int)((g.abc >> 5) & 1u) : 0);
        const bool face = (nby | nbl | nbr | nbz) != 0;
        float beta[4];
        if (face) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int nb = nby + nbz + (e == 0 ? nbl : 0) + (e == xe ? nbr : 0);
                beta[e] = __fmul_rn((float)nb, sqrtf(k.e[e]));
                w.e[e] = __fmaf_rn(1.f - beta[e], c.e[e], -__fmul_rn(__fmul_rn(sig, k.e[e]), div.e[e]));
            }
        }
        if (SRC && (cols || iz == 0 || top)) {
            const double2* sp = reinterpret_cast<const double2*>(S) + x0 + (long long)g.sx * (iy + (long long)g.sy * iz);
            if (cols == 1 && iz > 0 && !top) {
                const double2 s = sp[col];
                const float t = (float)__fma_rn(s.x, cs, __dmul_rn(s.y, sn));
#pragma unroll
                for (int e = 0; e < 4; ++e) w.e[e] += e == col ? t : 0.f;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (e >= m) continue;
                    const double2 s = sp[e];
                    if (soft64::is_zero(s.x) && soft64::is_zero(s.y)) continue;
                    w.e[e] += (float)__fma_rn(s.x, cs, __dmul_rn(s.y, sn));
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (face && beta[e] != 0.f) w.e[e] = w.e[e] / (1.f + beta[e]);
            if (k.e[e] == 0.f) w.e[e] = 0.f;  // Dirichlet nodes (and the padding)
        }
        if (valid) {
            put4(ox + j, xr);
            put4(oy + j, yr);
            put4(oz + j, zr);
            put4(ov + j, w);
        }
        zl = zr;
        c = up;
        j += sZ;
    }
}

// FP64 state -> stepping precision; MODE 0 a copy (0 on missing links and Dirichlet nodes),
// MODE 1 the adjoint's entry variables
// (q, u) = (p, v / (1 + beta)) (the input already E-scaled), MODE 2 the same from an unscaled
// cotangent: (pbar / W_e, vbar / (M (1 + beta))).
template <typename T, int MODE>
__global__ void __launch_bounds__(kFT) k_fo_load(const double* __restrict__ src, T* __restrict__ dst,
                                                 const double* __restrict__ kap64, const double* __restrict__ mass,
                                                 Geom g) {
    const long long n = (long long)(g.dim + 1) * g.np;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) {
        const Elem r = elem(g, e);
        double x = src[e];
        if (MODE == 0) {
            const int i = r.comp == 0 ? r.ix : (r.comp == 1 ? r.iy : r.iz), n = r.comp == 0 ? g.nx : (r.comp == 1 ? g.ny : g.nz);
            const bool keep = r.comp < g.dim ? i < n : !soft64::is_zero(kap64[r.j]);
            dst[e] = keep ? (T)x : T(0);
            continue;
        }
        if (r.comp < g.dim) {
            if (MODE == 2) {
                const double we = link_mass(g, r.comp, r.ix, r.iy, r.iz);
                x = we > 0.0 ? x / we : 0.0;
            }
        } else {
            const double k = kap64[r.j];
            if (k == 0.0) {
                x = 0.0;
            } else {
                const double beta = num_abc(g, r.ix, r.iy, r.iz) * sqrt(k);
                if (MODE == 2) x /= mass[r.j];
                x /= 1.0 + beta;
            }
        }
        dst[e] = (T)x;
    }
}

// End of a forward period.  MODE 0: e = s_N - s_0 and J = (e, e)_E / 2 into sc[SC_J], with s_0
// rounded to the stepping precision (the state the period started from).
// MODE 1: out = s_N (FP64).
template <typename T, int MODE>
__global__ void __launch_bounds__(kFT) k_fo_end(const T* __restrict__ sN, const double* __restrict__ s0,
                                                double* __restrict__ out, const double* __restrict__ mass, Geom g,
                                                Red red, int px) {
    const long long n = (long long)(g.dim + 1) * g.np;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) {
        if (MODE == 1) {
            out[e] = (double)sN[e];  // (px == sx here)
            continue;
        }
        const Elem r = elem(g, e);
        const double d = (double)sN[place(g, r, px)] - (double)(T)s0[e];  // against the copy the period started from
        out[e] = d;
        acc[0] += e_weight(g, mass, r) * d * d;
    }
    if (MODE == 0 && grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[SC_J] = 0.5 * acc[0];
}

// End of the backward period.  MODE 0 (CG): g = P* e - e from the final (q, u) and
// (g, d)_E into sc[SC_GD].  MODE 1 (plain transpose): out = E (q, (1 + beta) u).
template <typename T, int MODE>
__global__ void __launch_bounds__(kFT) k_fo_adj_end(const T* __restrict__ s, const double* __restrict__ e_in,
                                                    const double* __restrict__ d, double* __restrict__ out,
                                                    const double* __restrict__ kap64, const double* __restrict__ mass,
                                                    Geom g, Red red, int px) {
    const long long n = (long long)(g.dim + 1) * g.np;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) {
        const Elem r = elem(g, e);
        double x = (double)s[place(g, r, px)];
        double wgt;
        if (r.comp < g.dim) {
            wgt = link_mass(g, r.comp, r.ix, r.iy, r.iz);
        } else {
            const double k = kap64[r.j];
            x = k == 0.0 ? 0.0 : x * (1.0 + num_abc(g, r.ix, r.iy, r.iz) * sqrt(k));
            wgt = mass[r.j];
        }
        if (MODE == 1) {
            out[e] = wgt * x;
            continue;
        }
        const double gv = wgt > 0.0 ? x - e_in[e] : 0.0;
        out[e] = gv;
        acc[0] += wgt * gv * d[e];
    }
    if (MODE == 0 && grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[SC_GD] = acc[0];
}

// k_fo_load, k_fo_end<1> and k_fo_adj_end<1> for the padded FP32 state: one padded node per thread
// and turn, all four components.  Bound: HBM (129^3: 103 MB).  On the elements of the flat state, with
// three 64-bit divisions, FP64 conversions and, in the loads, FP64 divisions each, the FP64 pipe and
// the index arithmetic took 89 us for MODE 0 at 129^3; now 27 us.
struct RowNode {
    int x, iy, iz;
    long long j;  // in a flat field
    bool in, live[3];  // a node (not padding), its links
};
__device__ __forceinline__ RowNode row_node(const Geom& g, int px, unsigned i) {
    RowNode r;
    const unsigned t = i / (unsigned)px, z = t / (unsigned)g.sy;
    r.x = (int)(i - t * (unsigned)px);
    r.iy = (int)(t - z * (unsigned)g.sy);
    r.iz = (int)z;
    r.j = r.x + (long long)g.sx * t;
    r.in = r.x < g.sx;
    r.live[0] = r.x < g.nx;
    r.live[1] = r.iy < g.ny;
    r.live[2] = r.iz < g.nz;
    return r;
}
// link_mass of an existing link: h^3 halved for each of the other axes whose end the node is at
__device__ __forceinline__ double row_link_mass(const Geom& g, const RowNode& r, int a, double h3) {
    const int ends[3] = {r.x == 0 || r.x == g.nx, r.iy == 0 || r.iy == g.ny, r.iz == 0 || r.iz == g.nz};
    const int halvings = (a != 0 ? ends[0] : 0) + (a != 1 ? ends[1] : 0) + (a != 2 ? ends[2] : 0);
    return __hiloint2double(__double2hiint(h3) - (halvings << 20), __double2loint(h3));
}
__device__ __noinline__ double over_one_plus(double x, double nb, double k) { return x / (1.0 + nb * sqrt(k)); }
__device__ __noinline__ double times_one_plus(double x, double nb, double k) { return x * (1.0 + nb * sqrt(k)); }
__device__ __noinline__ float quotient_f32(double x, double d) { return (float)(x / d); }

// (float)(x / d), the division rounded to FP64 first, with r = 1 / d: x r is within two units in the
// last place of the quotient, so unless the 29 bits that the float drops are that close to one half,
// both round to the same float.
__device__ __forceinline__ float div_f32(double x, double d, double r) {
    const double q = x * r;
    const unsigned hi = (unsigned)__double2hiint(q) & 0x7fffffffu, lo = (unsigned)__double2loint(q) & 0x1fffffffu;
    if (hi - 0x38100000u < 0x0fc00000u && lo - 0x0ffffffcu > 8u) return soft64::to_f32(q);
    return quotient_f32(x, d);
}

template <int MODE>
__global__ void __launch_bounds__(kFT) k_fo_row_load(const double* __restrict__ src, float* __restrict__ dst,
                                                     const double* __restrict__ kap64, const double* __restrict__ mass,
                                                     Geom g, int px) {
    const unsigned field = (unsigned)px * (unsigned)(g.sy * g.sz), stride = gridDim.x * blockDim.x;
    const double h3 = g.h * g.h * g.h;
    double rw[3];  // the reciprocals of h^3, h^3 / 2, h^3 / 4
    if (MODE == 2) {
        rw[0] = 1.0 / h3;
        rw[1] = 2.0 * rw[0];
        rw[2] = 4.0 * rw[0];
    }
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < field; i += stride) {
        const RowNode r = row_node(g, px, i);
        if (r.in && !CMCG_RANGE_OK(r.j, r.j, g.np, kSiteRow)) continue;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float x = 0.f;
            if (r.in && (MODE == 1 || r.live[a])) {
                const double y = src[r.j + a * g.np];
                if (MODE != 2) {
                    x = soft64::to_f32(y);
                } else {
                    const double we = row_link_mass(g, r, a, h3);
                    const int halvings = (__double2hiint(h3) - __double2hiint(we)) >> 20;
                    x = div_f32(y, we, halvings == 0 ? rw[0] : (halvings == 1 ? rw[1] : rw[2]));
                }
            }
            dst[i + (size_t)a * field] = x;
        }
        float x = 0.f;
        if (r.in) {
            const double k = kap64[r.j];
            if (!soft64::is_zero(k)) {
                double y = src[r.j + 3 * g.np];
                if (MODE == 2) y /= mass[r.j];
                const int nb = MODE == 0 ? 0 : num_abc(g, r.x, r.iy, r.iz);
                if (nb) y = over_one_plus(y, nb, k);
                x = soft64::to_f32(y);
            }
        }
        dst[i + (size_t)3 * field] = x;
    }
}

// ADJ: out = E (q, (1 + beta) u), else the state itself
template <bool ADJ>
__global__ void __launch_bounds__(kFT) k_fo_row_end(const float* __restrict__ s, double* __restrict__ out,
                                                    const double* __restrict__ kap64, const double* __restrict__ mass,
                                                    Geom g, int px) {
    const unsigned field = (unsigned)px * (unsigned)(g.sy * g.sz), stride = gridDim.x * blockDim.x;
    const double h3 = g.h * g.h * g.h;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < field; i += stride) {
        const RowNode r = row_node(g, px, i);
        if (!r.in || !CMCG_RANGE_OK(r.j, r.j, g.np, kSiteRow)) continue;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double x = soft64::to_f64(s[i + (size_t)a * field]);
            if (ADJ) x = r.live[a] ? row_link_mass(g, r, a, h3) * x : 0.0;
            out[r.j + a * g.np] = x;
        }
        double x = soft64::to_f64(s[i + (size_t)3 * field]);
        if (ADJ) {
            const double k = kap64[r.j];
            const int nb = num_abc(g, r.x, r.iy, r.iz);
            if (soft64::is_zero(k)) x = 0.0;
            else if (nb) x = times_one_plus(x, nb, k);
            x *= mass[r.j];
        }
        out[r.j + 3 * g.np] = x;
    }
}

// (4) r = d = g; gamma = gamma0 = (g, g)_E.
__global__ void __launch_bounds__(kFT) k_fo_cg_init(const double* __restrict__ gr, double* __restrict__ r,
                                                    double* __restrict__ d, const double* __restrict__ mass, Geom g,
                                                    Red red) {
    const long long n = (long long)(g.dim + 1) * g.np;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) {
        const double x = gr[e];
        r[e] = x;
        d[e] = x;
        acc[0] += e_weight(g, mass, elem(g, e)) * x * x;
    }
    if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) {
        red.sc[SC_GAMMA] = acc[0];
        red.sc[SC_GAMMA0] = acc[0];
        red.sc[SC_REL] = acc[0] > 0.0 ? 1.0 : 0.0;
        red.sc[SC_STATUS] = isfinite(acc[0]) ? 0.0 : 1.0;
    }
}

// 5.3-5.6: alpha = gamma / (g, d)_E, s -= alpha d, r -= alpha g, gamma_new = (r, r)_E.  A
// non-positive or non-finite (g, d)_E (rounding of the FP32 periods at their precision floor)
// leaves s and r unchanged and sets the status.
__global__ void __launch_bounds__(kFT) k_fo_cg_update(double* __restrict__ s, double* __restrict__ r,
                                                      const double* __restrict__ d, const double* __restrict__ gr,
                                                      const double* __restrict__ mass, Geom g, Red red) {
    const double gamma = red.sc[SC_GAMMA];
    const double gd = red.sc[SC_GD];
    const bool breakdown = !(gd > 0.0) || !isfinite(gd);
    const double alpha = breakdown ? 0.0 : gamma / gd;
    const long long n = (long long)(g.dim + 1) * g.np;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) {
        s[e] -= alpha * d[e];
        const double x = r[e] - alpha * gr[e];
        r[e] = x;
        acc[0] += e_weight(g, mass, elem(g, e)) * x * x;
    }
    if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) {
        const double gnew = acc[0];
        red.sc[SC_ALPHA] = alpha;
        red.sc[SC_GAMMA_NEW] = gnew;
        red.sc[SC_BETA] = gamma > 0.0 ? gnew / gamma : 0.0;
        const double g0 = red.sc[SC_GAMMA0];
        red.sc[SC_REL] = g0 > 0.0 ? sqrt(fmax(gnew, 0.0) / g0) : 0.0;
        if (breakdown) red.sc[SC_STATUS] = 1.0;
        if (!isfinite(gnew)) red.sc[SC_STATUS] = 2.0;
    }
}

// 5.7: d = r + beta d; gamma = gamma_new.
__global__ void __launch_bounds__(kFT) k_fo_cg_direction(const double* __restrict__ r, double* __restrict__ d,
                                                         long long n, double* __restrict__ sc) {
    const double beta = sc[SC_BETA];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) d[e] = r[e] + beta * d[e];
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) sc[SC_GAMMA] = sc[SC_GAMMA_NEW];
}

// Step (6) by Eq. mix_solution, discrete-exact: Im U = v / wt, Re P = (2 p + dt G v) / (2 cos(w dt/2)),
// Re U = [(kappa h / dt^2) sum_a (ReP_a(j - e_a) - ReP_a(j)) / w_a + wh (2 beta / dt) Im U - S_re / dt^2] / wt^2.
__global__ void __launch_bounds__(kFT) k_fo_recover(const double* __restrict__ s, const double* __restrict__ kap64,
                                                    const double* __restrict__ S, double* __restrict__ u, Geom g,
                                                    double dt, double wt, double wh, double c_half) {
    const long long np = g.np;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const double* v = s + (long long)g.dim * np;
    const double gdt = dt / g.h;
    const double inv2c = 1.0 / (2.0 * c_half);
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const double k = kap64[j];
        if (k == 0.0) {
            u[2 * j] = 0.0;
            u[2 * j + 1] = 0.0;
            continue;
        }
        const long long t = j / g.sx;
        const int ix = (int)(j - t * g.sx);
        const int iz = (int)(t / g.sy);
        const int iy = (int)(t - (long long)iz * g.sy);
        const int i[3] = {ix, iy, iz};
        const int nn[3] = {g.nx, g.ny, g.nz};
        const long long str[3] = {1, g.sx, (long long)g.sx * g.sy};
        const double vc = v[j];
        double div = 0.0;
        for (int a = 0; a < g.dim; ++a) {
            const double* p = s + (long long)a * np;
            double rr = 0.0, rl = 0.0;
            if (i[a] < nn[a]) rr = (2.0 * p[j] + gdt * (v[j + str[a]] - vc)) * inv2c;
            if (i[a] > 0) rl = (2.0 * p[j - str[a]] + gdt * (vc - v[j - str[a]])) * inv2c;
            div += (rl - rr) * inv_w(i[a], nn[a]);
        }
        const double im = vc / wt;
        const double beta = num_abc(g, ix, iy, iz) * sqrt(k);
        const double re = (k * g.h / (dt * dt) * div + wh * (2.0 * beta / dt) * im - S[2 * j] / (dt * dt)) / (wt * wt);
        u[2 * j] = re;
        u[2 * j + 1] = im;
    }
}

// Step (6) by Eq. TH_FILTERED_MIXED_SOLUTION: U = (2 i / (N wt)) acc, acc = sum v^n e^{i w t_n}.
__global__ void k_fo_filter_final(long long np, double* __restrict__ u, double scale) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += stride) {
        const double re = u[2 * j], im = u[2 * j + 1];
        u[2 * j] = -scale * im;
        u[2 * j + 1] = scale * re;
    }
}

template <typename T, int DIM>
void step_launch(const Geom& g, const T* a, T* b, const T* kap, const double* S, double cs, double sn, double tau,
                 double sig, int zc, double* acc, double ca, double sa, const unsigned char* scol, cudaStream_t st) {
    note_launch(1);
    const dim3 grid = fo_grid(g, DIM == 3 ? zc : 1);
    auto go = [&](auto kernel) {
        kernel<<<grid, kFT, 0, st>>>(a, b, kap, S, cs, sn, (T)tau, (T)sig, g, zc, acc, ca, sa, scol);
    };
    if constexpr (std::is_same<T, double>::value) {
        if (S && acc) return go(k_fo_step<T, DIM, true, true>);
    }
    if (S) go(k_fo_step<T, DIM, true, false>);
    else go(k_fo_step<T, DIM, false, false>);
}

void row_launch(const Geom& g, const float* a, float* b, const float* kap, const double* S, const unsigned char* scol,
                double cs, double sn, double tau, double sig, int reverse, cudaStream_t st) {
    note_launch(1);
    const int px = row_pitch(g), plane4 = (px >> 2) * g.sy;
    const unsigned bxy = (unsigned)((plane4 + kFR - 1) / kFR);
    // planes per thread: one while that makes one wave of blocks at most (65^3, backward period: 338
    // us with one, 424 with four), else two (129^3: 771, 811 with one; 201^3: 2438, 2516 with four)
    const int zc = planes_per_thread((long long)bxy * g.sz <= 152ll * 8 ? 1 : 2, g.sz);
    const dim3 grid(bxy, (unsigned)((g.sz + zc - 1) / zc));
    auto go = [&](auto kernel) {
        kernel<<<grid, kFR, 0, st>>>(a, b, kap, S, scol, cs, sn, (float)tau, (float)sig, g, px, zc, reverse);
    };
    if (S) go(k_fo_row<true>);
    else go(k_fo_row<false>);
}

}  // namespace

namespace detail {

// z-planes per thread of k_fo_step: as many (16 at most) as leave a wave of blocks; each start of a
// column works the z-link below out again.  With 16 planes always, an FP64 backward period of 46
// steps took 2263 us at 33^3 (487 now) and 3908 at 97^3 (2513): too few warps for FP64 latencies.
int fo_zc(const Geom& g) {
    const long long plane = ((long long)g.sx * g.sy + kFT - 1) / kFT;
    int zc = 16;
    while (zc > 1 && plane * ((g.sz + zc - 1) / zc) < 152ll * 8) zc /= 2;
    return zc;
}

template <typename T>
const T* fo_kap(const cmcg_handle* H) {
    return std::is_same<T, float>::value ? (const T*)H->kap32 : (const T*)H->kap64;
}

// Row pitch of the stepping state: FP32 states on 3D grids are padded.
template <typename T>
int fo_pitch(const Geom& g) {
    return std::is_same<T, float>::value && g.dim == 3 ? row_pitch(g) : g.sx;
}

template <typename T>
void fo_step(cmcg_handle* H, const T* a, T* b, bool src, int n, bool backward, double* acc, double theta = 1.0) {
    const Geom& g = H->g;
    const double t = (n + 0.5) * H->dt;  // the source is T-periodic: n may count past one period
    const double cs = src ? theta * cos(H->omega * t) / H->dt : 0.0;
    const double sn = src ? theta * sin(H->omega * t) / H->dt : 0.0;
    const double tn = n * H->dt;
    const double ca = acc ? cos(H->omega * tn) : 0.0, sa = acc ? sin(H->omega * tn) : 0.0;
    const double tau = (backward ? -1.0 : 1.0) * H->dt / g.h;
    const double sig = (backward ? -1.0 : 1.0) * g.h / H->dt;
    const double* S = src ? H->S : nullptr;
    if (g.dim == 3) {
        if constexpr (std::is_same<T, float>::value)
            row_launch(g, a, b, H->row_kap, S, H->scol, cs, sn, tau, sig, a == (const float*)H->fo_b, H->st);
        else
            step_launch<T, 3>(g, a, b, fo_kap<T>(H), S, cs, sn, tau, sig, fo_zc(g), acc, ca, sa, H->scol, H->st);
    } else {
        step_launch<T, 2>(g, a, b, fo_kap<T>(H), S, cs, sn, tau, sig, 1, acc, ca, sa, nullptr, H->st);
    }
}

// FP64 state -> stepping state (MODE of k_fo_load), and back at the end of a period.
template <typename T, int MODE>
void fo_load(cmcg_handle* H, const double* src, T* dst) {
    const Geom& g = H->g;
    note_launch(1);
    if constexpr (std::is_same<T, float>::value) {
        if (g.dim == 3) {
            const int px = row_pitch(g);
            k_fo_row_load<MODE><<<fo_vec_blocks((long long)px * g.sy * g.sz), kFT, 0, H->st>>>(src, dst, H->kap64, H->mass, g, px);
            return;
        }
    }
    k_fo_load<T, MODE><<<fo_vec_blocks((long long)(g.dim + 1) * g.np), kFT, 0, H->st>>>(src, dst, H->kap64, H->mass, g);
}

template <typename T>
void fo_state_end(cmcg_handle* H, const T* s, double* out) {
    const Geom& g = H->g;
    note_launch(1);
    if constexpr (std::is_same<T, float>::value) {
        if (g.dim == 3) {
            const int px = row_pitch(g);
            k_fo_row_end<false><<<fo_vec_blocks((long long)px * g.sy * g.sz), kFT, 0, H->st>>>(s, out, H->kap64, H->mass, g, px);
            return;
        }
    }
    k_fo_end<T, 1><<<fo_vec_blocks((long long)(g.dim + 1) * g.np), kFT, 0, H->st>>>(s, out, out, H->mass, g, H->red(), g.sx);
}

// Forward period from the FP64 state s0.  mode 0: out = Pi(s0) - s0 and J; mode 1: out = Pi(s0).
// acc (optional, forced FP64 periods only) accumulates v^n e^{i w t_n}.
template <typename T>
void fo_forward(cmcg_handle* H, const double* s0, bool src, int mode, double* out, double* acc) {
    const Geom& g = H->g;
    const long long n = (long long)(g.dim + 1) * g.np;
    T* a = (T*)H->fo_a;
    T* b = (T*)H->fo_b;
    fo_load<T, 0>(H, s0, a);
    const int slot = timing_begin(H, std::is_same<T, float>::value, H->N);
    for (int k = 0; k < H->N; ++k) {
        fo_step<T>(H, a, b, src, k, false, acc);
        std::swap(a, b);
    }
    timing_end(H, slot);
    if (mode == 0) {
        note_launch(1);
        k_fo_end<T, 0><<<fo_vec_blocks(n), kFT, 0, H->st>>>(a, s0, out, H->mass, g, H->red(), fo_pitch<T>(g));
    } else {
        fo_state_end<T>(H, a, out);
    }
    H->periods += 1;
}

// Backward (adjoint) period.  mode 0: from the mismatch e (an E-scaled cotangent),
// out = P* e - e and (out, d)_E into sc[SC_GD]; mode 1: out = P^T y (plain transpose) for an
// unscaled cotangent y.
template <typename T>
void fo_backward(cmcg_handle* H, const double* y, const double* d, int mode, double* out) {
    const Geom& g = H->g;
    const long long n = (long long)(g.dim + 1) * g.np;
    T* a = (T*)H->fo_a;
    T* b = (T*)H->fo_b;
    if (mode == 0)
        fo_load<T, 1>(H, y, a);
    else
        fo_load<T, 2>(H, y, a);
    const int slot = timing_begin(H, std::is_same<T, float>::value, H->N);
    for (int k = 0; k < H->N; ++k) {
        fo_step<T>(H, a, b, false, k, true, nullptr);
        std::swap(a, b);
    }
    timing_end(H, slot);
    note_launch(1);
    H->periods += 1;
    if constexpr (std::is_same<T, float>::value) {
        if (mode == 1 && g.dim == 3) {
            const int px = row_pitch(g);
            k_fo_row_end<true><<<fo_vec_blocks((long long)px * g.sy * g.sz), kFT, 0, H->st>>>(a, out, H->kap64, H->mass, g, px);
            return;
        }
    }
    auto go = [&](auto kernel) {
        kernel<<<fo_vec_blocks(n), kFT, 0, H->st>>>(a, y, d, out, H->kap64, H->mass, g, H->red(), fo_pitch<T>(g));
    };
    if (mode == 0) go(k_fo_adj_end<T, 0>);
    else go(k_fo_adj_end<T, 1>);
}

// Steps 5.1-5.8 of the CMCG Algorithm on the first-order state, from r = d = g already set
// (k_fo_cg_init): J^' by a forward and a backward period (Eq. mixJ_deriative_2), no Riesz
// solve.  Updates the iterate x.  Stops at rel <= tol, after max_iter iterations, when
// (g, d)_E stops being positive (status 1: the FP32 periods' rounding floor), or when the
// residual has grown a hundredfold above its smallest value (FP32 periods only).  Returns a
// CMCG status (CMCG_ERR_DIVERGED on a non-finite residual); *it, *rel report the run.
template <typename T>
int fo_cg_iterate(cmcg_handle* H, double* x, double tol, int max_iter, int* it_out, double* rel_out) {
    const Geom& g = H->g;
    const long long n = (long long)(g.dim + 1) * g.np;
    // relative to the reference in SC_GAMMA0 (the start gradient's, or the zero guess's after a run-up)
    double rel = H->hsc[SC_GAMMA0] > 0.0 ? sqrt(std::max(H->hsc[SC_GAMMA], 0.0) / H->hsc[SC_GAMMA0]) : 0.0;
    double best = rel;
    int it = 0;
    if (rel > tol) {
        for (it = 1; it <= max_iter; ++it) {
            // 5.1 homogeneous forward and backward period from d
            fo_forward<T>(H, H->fo_d, false, 0, H->fo_e, nullptr);
            fo_backward<T>(H, H->fo_e, H->fo_d, 0, H->fo_g);
            // 5.3-5.6
            note_launch(1);
            k_fo_cg_update<<<fo_vec_blocks(n), kFT, 0, H->st>>>(x, H->fo_r, H->fo_d, H->fo_g, H->mass, g, H->red());
            // 5.7
            note_launch(1);
            k_fo_cg_direction<<<fo_vec_blocks(n), kFT, 0, H->st>>>(H->fo_r, H->fo_d, n, H->sc);
            if (sync_read(H) != CMCG_OK) return CMCG_ERR_CUDA;
            if (H->hsc[SC_STATUS] == 2.0) {
                *it_out = it;
                *rel_out = rel;
                return CMCG_ERR_DIVERGED;
            }
            if (H->hsc[SC_STATUS] != 0.0) break;  // (g, d)_E <= 0: x is the last good iterate
            rel = H->hsc[SC_REL];
            best = std::min(best, rel);
            if (rel <= tol) break;  // 5.8
            if (std::is_same<T, float>::value && rel > 100.0 * best) break;
        }
        if (it > max_iter) it = max_iter;
    }
    *it_out = it;
    *rel_out = rel;
    return rel <= tol ? CMCG_OK : CMCG_NOT_CONVERGED;
}

// (1)-(4): x = 0, the gradient with the sources at x in stepping precision T, r = d = g.
template <typename T>
int fo_cg_start(cmcg_handle* H, double* x) {
    const Geom& g = H->g;
    const long long n = (long long)(g.dim + 1) * g.np;
    cudaMemsetAsync(x, 0, sizeof(double) * n, H->st);
    fo_forward<T>(H, x, true, 0, H->fo_e, nullptr);
    fo_backward<T>(H, H->fo_e, H->fo_e, 0, H->fo_g);
    note_launch(1);
    k_fo_cg_init<<<fo_vec_blocks(n), kFT, 0, H->st>>>(H->fo_g, H->fo_r, H->fo_d, H->mass, g, H->red());
    return sync_read(H) == CMCG_OK ? CMCG_OK : CMCG_ERR_CUDA;
}

// Initial run-up (Sec. 4.2.3) on the first-order state: the forced staggered leapfrog from rest for
// `periods` periods with the sources ramped in by theta_tr over [0, periods T]; the state at
// t = periods T goes to out (FP64).
template <typename T>
void fo_runup(cmcg_handle* H, int periods, double* out) {
    const Geom& g = H->g;
    T* a = (T*)H->fo_a;
    T* b = (T*)H->fo_b;
    cudaMemsetAsync(a, 0, sizeof(T) * (size_t)(g.dim + 1) * fo_pitch<T>(g) * g.sy * g.sz, H->st);
    const long long total = (long long)periods * H->N;
    const double ttr = total * H->dt;
    for (long long k = 0; k < total; ++k) {
        fo_step<T>(H, a, b, true, (int)(k % H->N), false, nullptr, ramp((k + 0.5) * H->dt, ttr));
        std::swap(a, b);
    }
    fo_state_end<T>(H, a, out);
    H->periods += periods;
}

// With a run-up: the zero-guess gradient's gamma (the tolerance reference, and J0), then the
// run-up state into x and its gradient with r = d = g, and SC_GAMMA0 set to the reference.
// Without: x = 0 and its gradient.  Returns the number of run-up periods (or a negative status).
template <typename T>
int fo_start_with_runup(cmcg_handle* H, double* x, cmcg_stats* st) {
    const Geom& g = H->g;
    const long long n = (long long)(g.dim + 1) * g.np;
    if (fo_cg_start<T>(H, x) != CMCG_OK) return CMCG_ERR_CUDA;
    st->J0 = H->hsc[SC_J];
    const int ell = runup_count(H);
    if (ell <= 0) return 0;
    const double gamma_zero = H->hsc[SC_GAMMA0];
    fo_runup<T>(H, ell, x);
    fo_forward<T>(H, x, true, 0, H->fo_e, nullptr);
    fo_backward<T>(H, H->fo_e, H->fo_e, 0, H->fo_g);
    note_launch(1);
    k_fo_cg_init<<<fo_vec_blocks(n), kFT, 0, H->st>>>(H->fo_g, H->fo_r, H->fo_d, H->mass, g, H->red());
    cudaMemcpyAsync(H->sc + SC_GAMMA0, &gamma_zero, sizeof(double), cudaMemcpyHostToDevice, H->st);
    if (sync_read(H) != CMCG_OK) return CMCG_ERR_CUDA;
    return ell;
}

template <typename T>
int fo_cg(cmcg_handle* H, double tol, cmcg_stats* st) {
    const int ell = fo_start_with_runup<T>(H, H->fo_s, st);
    if (ell < 0) return ell;
    st->runup_periods = ell;
    int it = 0;
    double rel = 1.0;
    const int rc = fo_cg_iterate<T>(H, H->fo_s, tol, H->opt.max_iter, &it, &rel);
    st->iterations = it;
    st->outer_iterations = 1;
    st->rel_residual = rel;
    return rc;
}

// CMCG_MIXED: FP64 defect correction around FP32 CG.  Each outer step evaluates the gradient
// with the sources at s in FP64 (the true residual), then solves for the correction with FP32
// periods from zero to the relative tolerance inner_tol (tightened so as not to stop the outer
// loop short of tol) and adds it to s.  rel is relative to the first outer gradient (s = 0).
int fo_mixed(cmcg_handle* H, double tol, cmcg_stats* st) {
    const Geom& g = H->g;
    const long long n = (long long)(g.dim + 1) * g.np;
    cudaMemsetAsync(H->fo_s, 0, sizeof(double) * n, H->st);
    double gamma_ref = -1.0, rel = 1.0;
    int total = 0, outer = 0;
    const int max_outer = 50;
    const int ell = runup_count(H);
    if (ell > 0) {
        // the tolerance reference is the FP64 gradient of the zero guess; then an FP32 run-up
        fo_forward<double>(H, H->fo_s, true, 0, H->fo_e, nullptr);
        fo_backward<double>(H, H->fo_e, H->fo_e, 0, H->fo_g);
        note_launch(1);
        k_fo_cg_init<<<fo_vec_blocks(n), kFT, 0, H->st>>>(H->fo_g, H->fo_r, H->fo_d, H->mass, g, H->red());
        if (sync_read(H) != CMCG_OK) return CMCG_ERR_CUDA;
        gamma_ref = H->hsc[SC_GAMMA0];
        st->J0 = H->hsc[SC_J];
        fo_runup<float>(H, ell, H->fo_s);
        st->runup_periods = ell;
    }
    for (outer = 0; outer < max_outer; ++outer) {
        fo_forward<double>(H, H->fo_s, true, 0, H->fo_e, nullptr);
        fo_backward<double>(H, H->fo_e, H->fo_e, 0, H->fo_g);
        note_launch(1);
        k_fo_cg_init<<<fo_vec_blocks(n), kFT, 0, H->st>>>(H->fo_g, H->fo_r, H->fo_d, H->mass, g, H->red());
        if (sync_read(H) != CMCG_OK) return CMCG_ERR_CUDA;
        const double gam = H->hsc[SC_GAMMA0];
        if (!(gam == gam) || gam < 0) return CMCG_ERR_DIVERGED;
        if (gamma_ref < 0) {
            gamma_ref = gam;
            st->J0 = H->hsc[SC_J];
        }
        rel = gamma_ref > 0 ? sqrt(gam / gamma_ref) : 0.0;
        if (rel <= tol || total >= H->opt.max_iter) break;
        const double inner = std::min(0.5, std::max(H->opt.inner_tol, 0.5 * tol / std::max(rel, 1e-300)));
        int it = 0;
        double irel = 1.0;
        cudaMemsetAsync(H->fo_x, 0, sizeof(double) * n, H->st);
        const int rc = fo_cg_iterate<float>(H, H->fo_x, inner, H->opt.max_iter - total, &it, &irel);
        if (rc < 0) return rc;
        total += it;
        launch_axpy(n, 1.0, H->fo_x, H->fo_s, H->st);
        if (it == 0) break;  // no progress possible
    }
    st->iterations = total;
    st->outer_iterations = outer;
    st->rel_residual = rel;
    if (cuda_status() != CMCG_OK) return CMCG_ERR_CUDA;
    return rel <= tol ? CMCG_OK : CMCG_NOT_CONVERGED;
}

int fo_recover(cmcg_handle* H, double* u) {
    const Geom& g = H->g;
    if (H->opt.flags & CMCG_FLAG_FILTER) {
        // one forced FP64 period from s, accumulating v^n e^{i w t_n}
        cudaMemsetAsync(u, 0, sizeof(double) * 2 * g.np, H->st);
        fo_forward<double>(H, H->fo_s, true, 1, H->fo_e, u);
        note_launch(1);
        k_fo_filter_final<<<fo_vec_blocks(g.np), kFT, 0, H->st>>>(g.np, u, 2.0 / (H->N * H->wt));
    } else {
        note_launch(1);
        k_fo_recover<<<fo_vec_blocks(g.np), kFT, 0, H->st>>>(H->fo_s, H->kap64, H->S, u, g, H->dt, H->wt, H->wh,
                                                             cos(0.5 * H->omega * H->dt));
    }
    if (cudaStreamSynchronize(H->st) != cudaSuccess) return CMCG_ERR_CUDA;
    return cuda_status();
}

void fo_J(cmcg_handle* H) { fo_forward<double>(H, H->fo_s, true, 0, H->fo_e, nullptr); }

int fo_solve(cmcg_handle* H, double tol, cmcg_stats* st) {
    if (H->opt.precision == CMCG_FP64) return fo_cg<double>(H, tol, st);
    if (H->opt.precision == CMCG_FP32) return fo_cg<float>(H, tol, st);
    return fo_mixed(H, tol, st);
}

int fo_period(cmcg_handle* H, const double* s0, bool src, double* out) {
    if (H->opt.precision == CMCG_FP64)
        fo_forward<double>(H, s0, src, 1, out, nullptr);
    else
        fo_forward<float>(H, s0, src, 1, out, nullptr);
    return cuda_status();
}

int fo_adjoint(cmcg_handle* H, const double* y, double* out) {
    if (H->opt.precision == CMCG_FP64)
        fo_backward<double>(H, y, y, 1, out);
    else
        fo_backward<float>(H, y, y, 1, out);
    return cuda_status();
}

}  // namespace detail

CMCG_CHECK_TU(first_order)

}  // namespace cmcg
