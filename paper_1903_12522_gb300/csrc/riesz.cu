// Riesz map of Eq. CMCG_PRECONDITIONIER: K s = rhs with K = W (-Lap_h) (the discrete
// (grad s, grad phi)), solved matrix-free on the GPU.  The paper solves this SPD,
// omega-independent problem with a two-level Schwarz method (Sec. 4.3); here it is FP64
// flexible PCG whose preconditioner is one geometric multigrid V-cycle in FP32:
//   - vertex-centred coarsening n -> ceil(n/2) per axis (nested 2:1 for even n, general
//     linear interpolation for odd n), rediscretised K on each level, Dirichlet mask taken
//     from the nearest fine node;
//   - damped Jacobi smoothing, residual restriction by the transpose of (bi/tri)linear
//     interpolation, prolongation by that interpolation;
//   - the levels below kSpreadMaxNodes nodes run as one V-cycle inside one thread-block cluster in
//     shared memory; its coarsest level is solved by Jacobi sweeps.
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "soft64.cuh"

namespace cmcg {

namespace {

constexpr int kT = 256;

inline unsigned vec_blocks(long long n) {
    long long b = (n + kT - 1) / kT;
    if (b > kMaxBlocksReduce) b = kMaxBlocksReduce;
    if (b < 1) b = 1;
    return (unsigned)b;
}

inline unsigned node_blocks(long long n) { return (unsigned)((n + kT - 1) / kT); }

inline dim3 mg_grid(const Geom& g, int zc) {
    const long long plane = (long long)g.sx * g.sy;
    return dim3((unsigned)((plane + kT - 1) / kT), (unsigned)((g.sz + zc - 1) / zc), 1);
}

template <typename R>
struct Ld {
    const R* __restrict__ p;
    __device__ __forceinline__ R operator()(long long i) const { return p[i]; }
};

// Node coordinates (node counts stay below 2^31, so 32-bit division suffices).
__device__ __forceinline__ void coords(const Geom& g, long long j, int& ix, int& iy, int& iz) {
    const unsigned u = (unsigned)j;
    const unsigned t = u / (unsigned)g.sx;
    ix = (int)(u - t * (unsigned)g.sx);
    iz = (int)(t / (unsigned)g.sy);
    iy = (int)(t - (unsigned)iz * (unsigned)g.sy);
}

template <typename R>
struct LdM {  // masked load: Dirichlet nodes read as 0
    const R* __restrict__ p;
    const unsigned char* __restrict__ m;
    __device__ __forceinline__ R operator()(long long i) const { return (m && m[i]) ? R(0) : p[i]; }
};

// ---- multigrid (FP32) ---------------------------------------------------------------------
// K-form on every level: K = (h^d / h^2) s Lt with s = prod_a w(j_a) in {1, 1/2, 1/4, 1/8};
// diag K = (h^d / h^2) s 2d.  Damped Jacobi: x += omega (b - K x) / diag K.
// Iterates are kept exactly 0 on Dirichlet nodes, so neighbour loads need no mask.
__device__ __forceinline__ int axis_ends(const Geom& g, int ix, int iy, int iz) {
    int e = (ix == 0 || ix == g.nx) + (iy == 0 || iy == g.ny);
    if (g.dim == 3) e += (iz == 0 || iz == g.nz);
    return e;
}

struct MGConst {
    float cK;     // h^d / h^2
    float cB;     // h^2 / (2d h^d)
    float inv2d;  // 1 / (2d)
};

__device__ __forceinline__ MGConst mg_const(const Geom& g) {
    MGConst c;
    const float h = (float)g.h;
    const float hd = g.dim == 3 ? h * h * h : h * h;
    c.cK = hd / (h * h);
    c.inv2d = 1.f / (float)(2 * g.dim);
    c.cB = (h * h) / (hd * (float)(2 * g.dim));
    return c;
}

// One damped Jacobi update at node j (xin == nullptr: from x = 0).
__device__ __forceinline__ float jacobi_zero(const MGConst& c, float bj, float omega, int ends) {
    const float inv_s = (float)(1 << ends);
    return omega * c.cB * inv_s * bj;
}

// f: the values of x by node index (global memory, or a cluster's shared memory).
template <typename F>
__device__ __forceinline__ float jacobi_from(const Geom& g, const MGConst& c, F f, float bj, float omega, long long j,
                                             int ix, int iy, int iz) {
    const float inv_s = (float)(1 << axis_ends(g, ix, iy, iz));
    const float L = lap_t<2, float>(g, f, j, ix, iy, iz);
    return f(j) + omega * (c.cB * inv_s * bj - c.inv2d * L);
}

__device__ __forceinline__ float jacobi_node(const Geom& g, const MGConst& c, const float* xin, float bj, float omega,
                                             long long j, int ix, int iy, int iz) {
    if (!xin) return jacobi_zero(c, bj, omega, axis_ends(g, ix, iy, iz));
    return jacobi_from(g, c, Ld<float>{xin}, bj, omega, j, ix, iy, iz);
}

template <typename F>
__device__ __forceinline__ float residual_node(const Geom& g, const MGConst& c, F f, float bj, long long j, int ix, int iy,
                                               int iz) {
    const float s = 1.f / (float)(1 << axis_ends(g, ix, iy, iz));
    return bj - c.cK * s * lap_t<2, float>(g, f, j, ix, iy, iz);
}

// Coarsening n_f -> n_c = ceil(n_f / 2) per axis: fine node i sits at coarse coordinate
// xi = i n_c / n_f; it interpolates from coarse nodes J0 = floor(xi) (weight 1 - t) and
// J0 + 1 (weight t), t = xi - J0.  For even n_f this is the nested 2:1 scheme (t in {0, 1/2}).
// Restriction is the exact transpose of this interpolation.
struct Interp1 {
    int j0;
    float t;
};

// floor(a b / d); 32-bit division (a fraction of the 64-bit one's instructions) where the product fits
__device__ __forceinline__ int scaled(int a, int b, int d, bool small) {
    return small ? (int)((unsigned)a * (unsigned)b / (unsigned)d) : (int)((long long)a * b / d);
}

__device__ __forceinline__ Interp1 interp1(int i, int nf, int nc) {
    Interp1 r;
    r.j0 = scaled(i, nc, nf, nf < 46000);
    r.t = (float)(int)((long long)i * nc - (long long)r.j0 * nf) / (float)nf;
    if (r.j0 >= nc) {
        r.j0 = nc;
        r.t = 0.f;
    }
    return r;
}

// weight with which fine node i contributes to coarse node J along one axis
__device__ __forceinline__ float interp_weight(int i, int J, int nf, int nc) {
    const Interp1 p = interp1(i, nf, nc);
    if (p.j0 == J) return 1.f - p.t;
    if (p.j0 + 1 == J) return p.t;
    return 0.f;
}

// The fine nodes that contribute to coarse node J along one axis, first .. first + 3 at most (those
// with J - 1 < xi < J + 1; xi steps by n_c / n_f >= 1/2), and their weights (0: none).
struct AxisWeights {
    int first;
    float w[4];
};

__device__ __forceinline__ AxisWeights axis_weights(int J, int nf, int nc) {
    AxisWeights r;
    r.first = J > 0 ? scaled(J - 1, nf, nc, nf < 46000) + 1 : 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) r.w[e] = r.first + e <= nf ? interp_weight(r.first + e, J, nf, nc) : 0.f;
    return r;
}

// Restriction with general weights: the sum over z, y, x in this order, one fused multiply-add per
// contributing fine node.  All of a plane's reads are issued before the sum.  (With the weights, two
// 64-bit divisions each, worked out in the innermost loop, a coarse plane's launch took 179 us on a
// 102x88x94 grid; now 14.)
template <typename F>
__device__ __forceinline__ float restrict_weighted(const Geom& gf, F rf, const AxisWeights& X, const AxisWeights& Y,
                                                   const AxisWeights& Z) {
    const int last = gf.nx - X.first;  // (reads without a weight stay in the row)
    float acc = 0.f;
#pragma unroll 1
    for (int z = 0; z < (gf.dim == 3 ? 4 : 1); ++z) {
        const float wz = Z.w[0] * (z == 0 ? 1.f : 0.f) + Z.w[1] * (z == 1 ? 1.f : 0.f) + Z.w[2] * (z == 2 ? 1.f : 0.f) +
                         Z.w[3] * (z == 3 ? 1.f : 0.f);  // Z.w[z]
        if (wz == 0.f) continue;
        float r[4][4];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const long long row = node(gf, X.first, Y.w[y] != 0.f ? Y.first + y : Y.first, Z.first + z);
#pragma unroll
            for (int x = 0; x < 4; ++x) r[y][x] = rf(row + min(x, last));
        }
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (Y.w[y] != 0.f && X.w[x] != 0.f)
                    acc = __fmaf_rn(__fmul_rn(__fmul_rn(X.w[x], Y.w[y]), wz), r[y][x], acc);
    }
    return acc;
}

__device__ __forceinline__ bool nested(const Geom& gf, const Geom& gc) {
    return gf.nx == 2 * gc.nx && gf.ny == 2 * gc.ny && (gf.dim == 2 || gf.nz == 2 * gc.nz);
}

// nested 2:1 case: weights 1 at 2J and 1/2 at 2J +- 1 per axis
template <typename F>
__device__ __forceinline__ float restrict_nested(const Geom& gf, F rf, int jx, int jy, int jz) {
    const int cx = 2 * jx, cy = 2 * jy, cz = 2 * jz;
    float acc = 0.f;
    const int zlo = gf.dim == 3 ? -1 : 0, zhi = gf.dim == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        const int fz = cz + dz;
        if (fz < 0 || fz > gf.nz) continue;
        const float wz = dz == 0 ? 1.f : 0.5f;
        for (int dy = -1; dy <= 1; ++dy) {
            const int fy = cy + dy;
            if (fy < 0 || fy > gf.ny) continue;
            const float wy = dy == 0 ? 1.f : 0.5f;
            const long long row = node(gf, 0, fy, fz);
            float racc = rf(row + cx);
            if (cx > 0) racc += 0.5f * rf(row + cx - 1);
            if (cx < gf.nx) racc += 0.5f * rf(row + cx + 1);
            acc += wy * wz * racc;
        }
    }
    return acc;
}

__device__ __forceinline__ AxisWeights axis_weights_z(const Geom& gf, const Geom& gc, int jz) {
    if (gf.dim == 3) return axis_weights(jz, gf.nz, gc.nz);
    return AxisWeights{0, {1.f, 0.f, 0.f, 0.f}};
}

__device__ __forceinline__ Interp1 interp1_fast(int i, int nf, int nc) {
    if (nf == 2 * nc) {
        Interp1 r;
        r.j0 = i >> 1;
        r.t = (i & 1) ? 0.5f : 0.f;
        return r;
    }
    return interp1(i, nf, nc);
}

template <typename F>
__device__ __forceinline__ float prolong_node(const Geom& gc, F xc, const Geom& gf, int ix, int iy, int iz) {
    const Interp1 px = interp1_fast(ix, gf.nx, gc.nx), py = interp1_fast(iy, gf.ny, gc.ny);
    const int x1 = px.t > 0.f ? px.j0 + 1 : px.j0, y1 = py.t > 0.f ? py.j0 + 1 : py.j0;
    const float ax = 1.f - px.t, ay = 1.f - py.t;
    if (gf.dim != 3)
        return ay * (ax * xc(node(gc, px.j0, py.j0, 0)) + px.t * xc(node(gc, x1, py.j0, 0))) +
               py.t * (ax * xc(node(gc, px.j0, y1, 0)) + px.t * xc(node(gc, x1, y1, 0)));
    const Interp1 pz = interp1_fast(iz, gf.nz, gc.nz);
    const int z1 = pz.t > 0.f ? pz.j0 + 1 : pz.j0;
    const long long offz0 = (long long)pz.j0 * gc.sx * gc.sy, offz1 = (long long)z1 * gc.sx * gc.sy;
    const float v0 = ay * (ax * xc(offz0 + node(gc, px.j0, py.j0, 0)) + px.t * xc(offz0 + node(gc, x1, py.j0, 0))) +
                     py.t * (ax * xc(offz0 + node(gc, px.j0, y1, 0)) + px.t * xc(offz0 + node(gc, x1, y1, 0)));
    const float v1 = ay * (ax * xc(offz1 + node(gc, px.j0, py.j0, 0)) + px.t * xc(offz1 + node(gc, x1, py.j0, 0))) +
                     py.t * (ax * xc(offz1 + node(gc, px.j0, y1, 0)) + px.t * xc(offz1 + node(gc, x1, y1, 0)));
    return (1.f - pz.t) * v0 + pz.t * v1;
}

struct PlaneIt {
    int ix, iy, z0, z1;
    bool valid;
};

__device__ __forceinline__ PlaneIt plane_it(const Geom& g, int zc) {
    PlaneIt m;
    const unsigned plane = (unsigned)g.sx * (unsigned)g.sy;
    const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
    m.valid = p < plane;
    const unsigned pp = m.valid ? p : 0u;
    m.iy = (int)(pp / (unsigned)g.sx);
    m.ix = (int)(pp - (unsigned)m.iy * (unsigned)g.sx);
    m.z0 = blockIdx.y * zc;
    m.z1 = min(m.z0 + zc, g.sz);
    if (m.valid && !column_in_range(g, m.ix, m.iy, m.z0, m.z1, 1, kSiteMultigrid)) m.valid = false;
    return m;
}

__global__ void __launch_bounds__(kT) k_jacobi(Geom g, const unsigned char* __restrict__ mask,
                                               const float* __restrict__ xin, float* __restrict__ xout,
                                               const float* __restrict__ b, float omega, int zc) {
    const PlaneIt m = plane_it(g, zc);
    if (!m.valid) return;
    const MGConst c = mg_const(g);
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const long long j = node(g, m.ix, m.iy, iz);
        // the mask, b and the stencil are loaded together and the mask selects at the end: a
        // branch on the mask byte would put its load's latency before every other load
        const bool dir = mask && mask[j];
        const float v = jacobi_node(g, c, xin, b[j], omega, j, m.ix, m.iy, iz);
        xout[j] = dir ? 0.f : v;
    }
}

__global__ void __launch_bounds__(kT) k_residual(Geom g, const unsigned char* __restrict__ mask,
                                                 const float* __restrict__ x, const float* __restrict__ b,
                                                 float* __restrict__ r, int zc) {
    const PlaneIt m = plane_it(g, zc);
    if (!m.valid) return;
    const MGConst c = mg_const(g);
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const long long j = node(g, m.ix, m.iy, iz);
        const bool dir = mask && mask[j];  // selected at the end (see k_jacobi)
        const float v = residual_node(g, c, Ld<float>{x}, b[j], j, m.ix, m.iy, iz);
        r[j] = dir ? 0.f : v;
    }
}

// 3D Jacobi sweep (from a given x) and residual, two z-planes per loop trip: both planes' loads
// (x with its x/y neighbours, b, the mask byte) are issued before either update, and the
// z-neighbours come from registers.  The expressions are those of jacobi_node / residual_node
// with the 7-point Laplacian summed in lap_t's order, so the results are bitwise equal to
// k_jacobi / k_residual.
struct Col3 {
    long long sZ, oxm, oxp, oym, oyp;
    int exy;  // axis ends of the column in x and y
};

__device__ __forceinline__ Col3 col3(const Geom& g, int ix, int iy) {
    Col3 c;
    c.sZ = (long long)g.sx * g.sy;
    c.oxm = off_m1(ix, 1);
    c.oxp = off_p1(ix, g.nx, 1);
    c.oym = off_m1(iy, g.sx);
    c.oyp = off_p1(iy, g.ny, g.sx);
    c.exy = (ix == 0 || ix == g.nx) + (iy == 0 || iy == g.ny);
    return c;
}

// MODE 0: Jacobi x_out = x + omega (cB s^-1 b - L / 6); MODE 1: residual r = b - cK s L.
template <int MODE>
__global__ void __launch_bounds__(kT) k_mg3_z2(Geom g, const unsigned char* __restrict__ mask,
                                               const float* __restrict__ x, const float* __restrict__ b,
                                               float* __restrict__ out, float omega, int zc) {
    const PlaneIt m = plane_it(g, zc);
    if (!m.valid || m.z0 >= m.z1) return;
    const MGConst c = mg_const(g);
    const Col3 o = col3(g, m.ix, m.iy);
    const long long sZ = o.sZ;
    auto update = [&](float xc, float xm, float xp, float sx, float sy, long long jj, int iz, float bj, bool dir) {
        float acc = sx;
        acc += sy;
        acc += xm + xp;
        const float L = 6.f * xc - acc;
        const int e = o.exy + (iz == 0 || iz == g.nz);
        float v;
        if (MODE == 0) {
            const float inv_s = (float)(1 << e);
            v = xc + omega * (c.cB * inv_s * bj - c.inv2d * L);
        } else {
            const float s = 1.f / (float)(1 << e);
            v = bj - c.cK * s * L;
        }
        out[jj] = dir ? 0.f : v;
    };
    long long j = node(g, m.ix, m.iy, m.z0);
    float xm = x[j + (m.z0 > 0 ? -sZ : sZ)];
    float xc = x[j];
    int iz = m.z0;
    for (; iz + 1 < m.z1; iz += 2) {
        const long long j1 = j + sZ;
        const float x1 = x[j1];                               // plane iz+1 (exists: iz+1 < z1 <= sz)
        const float x2 = x[j1 + (iz + 1 < g.nz ? sZ : -sZ)];  // plane iz+2 (mirrored at the top)
        const float sx0 = x[j + o.oxm] + x[j + o.oxp], sy0 = x[j + o.oym] + x[j + o.oyp];
        const float sx1 = x[j1 + o.oxm] + x[j1 + o.oxp], sy1 = x[j1 + o.oym] + x[j1 + o.oyp];
        const float b0 = b[j], b1 = b[j1];
        const bool d0 = mask && mask[j], d1 = mask && mask[j1];
        update(xc, xm, x1, sx0, sy0, j, iz, b0, d0);
        update(x1, xc, x2, sx1, sy1, j1, iz + 1, b1, d1);
        xm = x1;
        xc = x2;
        j += 2 * sZ;
    }
    if (iz < m.z1) {
        const float xp = x[j + (iz < g.nz ? sZ : -sZ)];
        const float sx0 = x[j + o.oxm] + x[j + o.oxp], sy0 = x[j + o.oym] + x[j + o.oyp];
        update(xc, xm, xp, sx0, sy0, j, iz, b[j], mask && mask[j]);
    }
}

// The first two sweeps of a cycle, x = J(J(0)), in one pass over b: the first sweep from zero is
// omega b / diag K at each node, formed for a node's neighbours from their b (zero on Dirichlet
// nodes) instead of being stored and read back.  Bits as k_jacobi then k_mg3_z2.  At 129^3 the
// two took 7.1 + 10.5 us.
__global__ void __launch_bounds__(kT) k_mg3_first(Geom g, const unsigned char* __restrict__ mask,
                                                  const float* __restrict__ b, float* __restrict__ out, float omega,
                                                  int zc) {
    const PlaneIt m = plane_it(g, zc);
    if (!m.valid || m.z0 >= m.z1) return;
    const MGConst c = mg_const(g);
    const Col3 o = col3(g, m.ix, m.iy);
    const long long sZ = o.sZ;
    const float wcb = omega * c.cB;
    // powers of two: a node on e grid ends has 2^e times the factor
    auto ends = [](int i, int n) { return i == 0 || i == n ? 2.f : 1.f; };
    const float fx = ends(m.ix, g.nx), fy = ends(m.iy, g.ny);
    const float wc = wcb * (fx * fy);
    const float wxm = wcb * (ends(m.ix > 0 ? m.ix - 1 : 1, g.nx) * fy), wxp = wcb * (ends(m.ix < g.nx ? m.ix + 1 : g.nx - 1, g.nx) * fy);
    const float wym = wcb * (fx * ends(m.iy > 0 ? m.iy - 1 : 1, g.ny)), wyp = wcb * (fx * ends(m.iy < g.ny ? m.iy + 1 : g.ny - 1, g.ny));
    const float wj = c.cB * (fx * fy);
    auto update = [&](float bc, float bm, float bp, float b0, float b1v, float b2v, float b3v, long long jj, int iz,
                      bool dir) {
        const float fz = ends(iz, g.nz);
        const float xc = wc * fz * bc;
        float acc = __fadd_rn(wxm * fz * b0, wxp * fz * b1v);
        acc = __fadd_rn(acc, __fadd_rn(wym * fz * b2v, wyp * fz * b3v));
        acc = __fadd_rn(acc, __fadd_rn(wc * ends(iz > 0 ? iz - 1 : 1, g.nz) * bm, wc * ends(iz < g.nz ? iz + 1 : g.nz - 1, g.nz) * bp));
        const float L = __fmaf_rn(6.f, xc, -acc);
        const float v = __fmaf_rn(omega, __fmaf_rn(wj * fz, bc, -__fmul_rn(c.inv2d, L)), xc);
        out[jj] = dir ? 0.f : v;
    };
    long long j = node(g, m.ix, m.iy, m.z0);
    float bm = b[j + (m.z0 > 0 ? -sZ : sZ)];
    float bc = b[j];
    int iz = m.z0;
    for (; iz + 1 < m.z1; iz += 2) {
        const long long j1 = j + sZ;
        const float b1 = b[j1];
        const float b2 = b[j1 + (iz + 1 < g.nz ? sZ : -sZ)];
        const float a0 = b[j + o.oxm], a1 = b[j + o.oxp], a2 = b[j + o.oym], a3 = b[j + o.oyp];
        const float c0 = b[j1 + o.oxm], c1 = b[j1 + o.oxp], c2 = b[j1 + o.oym], c3 = b[j1 + o.oyp];
        const bool d0 = mask && mask[j], d1 = mask && mask[j1];
        update(bc, bm, b1, a0, a1, a2, a3, j, iz, d0);
        update(b1, bc, b2, c0, c1, c2, c3, j1, iz + 1, d1);
        bm = b1;
        bc = b2;
        j += 2 * sZ;
    }
    if (iz < m.z1) {
        const float bp = b[j + (iz < g.nz ? sZ : -sZ)];
        update(bc, bm, bp, b[j + o.oxm], b[j + o.oxp], b[j + o.oym], b[j + o.oyp], j, iz, mask && mask[j]);
    }
}

__global__ void __launch_bounds__(kT) k_mg2_first(Geom g, const unsigned char* __restrict__ mask,
                                                  const float* __restrict__ b, float* __restrict__ out, float omega) {
    const PlaneIt m = plane_it(g, 1);
    if (!m.valid) return;
    const MGConst c = mg_const(g);
    const float wcb = omega * c.cB;
    auto ends = [](int i, int n) { return i == 0 || i == n ? 2.f : 1.f; };
    const int xm = m.ix > 0 ? m.ix - 1 : 1, xp = m.ix < g.nx ? m.ix + 1 : g.nx - 1;
    const int ym = m.iy > 0 ? m.iy - 1 : 1, yp = m.iy < g.ny ? m.iy + 1 : g.ny - 1;
    const float fx = ends(m.ix, g.nx), fy = ends(m.iy, g.ny);
    const long long j = m.ix + (long long)g.sx * m.iy, row = j - m.ix;
    const float bc = b[j];
    const float xc = wcb * (fx * fy) * bc;
    float acc = __fadd_rn(wcb * (ends(xm, g.nx) * fy) * b[row + xm], wcb * (ends(xp, g.nx) * fy) * b[row + xp]);
    acc = __fadd_rn(acc, __fadd_rn(wcb * (fx * ends(ym, g.ny)) * b[m.ix + (long long)g.sx * ym],
                                   wcb * (fx * ends(yp, g.ny)) * b[m.ix + (long long)g.sx * yp]));
    const float L = __fmaf_rn(4.f, xc, -acc);
    const float v = __fmaf_rn(omega, __fmaf_rn(c.cB * (fx * fy), bc, -__fmul_rn(c.inv2d, L)), xc);
    out[j] = mask && mask[j] ? 0.f : v;
}

// 3D prolongation x_f += P x_c along a thread's fine z-column.  Every fine plane blends the
// xy-interpolated values of at most two coarse planes; those are kept in registers and
// reused by the next fine plane (for 2:1 coarsening, one new coarse plane per two fine
// planes).  Same expressions as prolong_node: bitwise equal to k_prolong_add.
__global__ void __launch_bounds__(kT) k_prolong_add3(Geom gc, const float* __restrict__ xc, Geom gf,
                                                     const unsigned char* __restrict__ maskf, float* __restrict__ xf,
                                                     int zc) {
    const PlaneIt m = plane_it(gf, zc);
    if (!m.valid || m.z0 >= m.z1) return;
    const Interp1 px = interp1_fast(m.ix, gf.nx, gc.nx), py = interp1_fast(m.iy, gf.ny, gc.ny);
    const int x1 = px.t > 0.f ? px.j0 + 1 : px.j0, y1 = py.t > 0.f ? py.j0 + 1 : py.j0;
    const float ax = 1.f - px.t, ay = 1.f - py.t;
    const long long o00 = node(gc, px.j0, py.j0, 0), o10 = node(gc, x1, py.j0, 0);
    const long long o01 = node(gc, px.j0, y1, 0), o11 = node(gc, x1, y1, 0);
    const long long planeC = (long long)gc.sx * gc.sy;
    auto pxy = [&](int J) {
        const float* cp = xc + (long long)J * planeC;
        return ay * (ax * cp[o00] + px.t * cp[o10]) + py.t * (ax * cp[o01] + px.t * cp[o11]);
    };
    int ja = -1, jb = -1;  // coarse planes held in va, vb
    float va = 0.f, vb = 0.f;
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const long long i = node(gf, m.ix, m.iy, iz);
        const bool dir = maskf && maskf[i];  // tested at the store (see k_jacobi)
        const float x0 = xf[i];
        const Interp1 pz = interp1_fast(iz, gf.nz, gc.nz);  // the same for every thread of the block
        const int z1 = pz.t > 0.f ? pz.j0 + 1 : pz.j0;
        const float v0 = pz.j0 == jb ? vb : (pz.j0 == ja ? va : pxy(pz.j0));
        const float v1 = z1 == pz.j0 ? v0 : (z1 == jb ? vb : pxy(z1));
        ja = pz.j0;
        va = v0;
        jb = z1;
        vb = v1;
        const float v = (1.f - pz.t) * v0 + pz.t * v1;
        if (!dir) xf[i] = x0 + v;
    }
}

// 3D restriction for 2:1 coarsening along a thread's coarse z-column.  Coarse plane J gathers
// fine planes 2J-1, 2J, 2J+1; the x-weighted row sums of plane 2J+1 are kept in registers
// for plane J+1, so each coarse plane loads two fine planes.  Rows outside the grid are read
// at a clamped address and left out of the sum, so every load is issued before the sums.  The
// terms and their order are those of restrict_nested: bitwise equal to k_restrict.
__global__ void __launch_bounds__(kT) k_restrict3_nested(Geom gf, const float* __restrict__ rf, Geom gc,
                                                         const unsigned char* __restrict__ maskc,
                                                         float* __restrict__ bc, int zc) {
    const PlaneIt m = plane_it(gc, zc);
    if (!m.valid || m.z0 >= m.z1) return;
    const int cx = 2 * m.ix, cy = 2 * m.iy;
    const bool xm = cx > 0, xp = cx < gf.nx;
    const int xl = xm ? cx - 1 : cx, xr = xp ? cx + 1 : cx;
    bool yok[3];
    long long yoff[3];
    for (int d = 0; d < 3; ++d) {
        const int fy = cy + d - 1;
        yok[d] = fy >= 0 && fy <= gf.ny;
        yoff[d] = (long long)(yok[d] ? fy : cy) * gf.sx;
    }
    const long long sZ = (long long)gf.sx * gf.sy;
    auto rows = [&](int fz, float* r) {  // row sums of fine plane fz (0 <= fz <= nz)
        const float* pl = rf + (long long)fz * sZ;
        float a[3], l[3], q[3];
        for (int d = 0; d < 3; ++d) {
            a[d] = pl[yoff[d] + cx];
            l[d] = pl[yoff[d] + xl];
            q[d] = pl[yoff[d] + xr];
        }
        for (int d = 0; d < 3; ++d) {
            float racc = a[d];
            if (xm) racc += 0.5f * l[d];
            if (xp) racc += 0.5f * q[d];
            r[d] = racc;
        }
    };
    float lo[3] = {0.f, 0.f, 0.f};  // row sums of fine plane 2J - 1
    bool have_lo = false;
    for (int jz = m.z0; jz < m.z1; ++jz) {
        const long long J = node(gc, m.ix, m.iy, jz);
        const bool dir = maskc && maskc[J];
        const int cz = 2 * jz;
        const bool zlo = cz - 1 >= 0, zhi = cz + 1 <= gf.nz;
        if (zlo && !have_lo) rows(cz - 1, lo);
        float mid[3], hi[3] = {0.f, 0.f, 0.f};
        rows(cz, mid);
        if (zhi) rows(cz + 1, hi);
        float acc = 0.f;
        if (zlo)
            for (int d = 0; d < 3; ++d)
                if (yok[d]) acc += (d == 1 ? 1.f : 0.5f) * 0.5f * lo[d];
        for (int d = 0; d < 3; ++d)
            if (yok[d]) acc += (d == 1 ? 1.f : 0.5f) * 1.f * mid[d];
        if (zhi)
            for (int d = 0; d < 3; ++d)
                if (yok[d]) acc += (d == 1 ? 1.f : 0.5f) * 0.5f * hi[d];
        bc[J] = dir ? 0.f : acc;
        for (int d = 0; d < 3; ++d) lo[d] = hi[d];
        have_lo = zhi;
    }
}

// b_c[J] = sum over fine nodes i of the interpolation weights times r_f[i].
__global__ void __launch_bounds__(kT) k_restrict(Geom gf, const float* __restrict__ rf, Geom gc,
                                                 const unsigned char* __restrict__ maskc, float* __restrict__ bc,
                                                 int zc) {
    const PlaneIt m = plane_it(gc, zc);
    if (!m.valid) return;
    const bool two = nested(gf, gc);
    AxisWeights X{}, Y{};
    if (!two) {
        X = axis_weights(m.ix, gf.nx, gc.nx);
        Y = axis_weights(m.iy, gf.ny, gc.ny);
    }
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const long long J = node(gc, m.ix, m.iy, iz);
        const bool dir = maskc && maskc[J];  // selected at the end (see k_jacobi)
        const float v = two ? restrict_nested(gf, Ld<float>{rf}, m.ix, m.iy, iz)
                            : restrict_weighted(gf, Ld<float>{rf}, X, Y, axis_weights_z(gf, gc, iz));
        bc[J] = dir ? 0.f : v;
    }
}

// x_f[i] += interpolated x_c.
__global__ void __launch_bounds__(kT) k_prolong_add(Geom gc, const float* __restrict__ xc, Geom gf,
                                                    const unsigned char* __restrict__ maskf, float* __restrict__ xf,
                                                    int zc) {
    const PlaneIt m = plane_it(gf, zc);
    if (!m.valid) return;
    for (int iz = m.z0; iz < m.z1; ++iz) {
        const long long i = node(gf, m.ix, m.iy, iz);
        const bool dir = maskf && maskf[i];  // tested at the store (see k_jacobi)
        const float v = prolong_node(gc, Ld<float>{xc}, gf, m.ix, m.iy, iz);
        const float x0 = xf[i];
        if (!dir) xf[i] = x0 + v;
    }
}

__global__ void k_coarsen_mask(Geom gf, const unsigned char* __restrict__ mf, Geom gc, unsigned char* __restrict__ mc) {
    const long long J = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (J >= gc.np) return;
    int jx, jy, jz;
    coords(gc, J, jx, jy, jz);
    // the fine node nearest to the coarse node's position
    const int fx = (int)(((long long)jx * gf.nx * 2 + gc.nx) / (2 * gc.nx));
    const int fy = (int)(((long long)jy * gf.ny * 2 + gc.ny) / (2 * gc.ny));
    const int fz = gf.dim == 3 ? (int)(((long long)jz * gf.nz * 2 + gc.nz) / (2 * gc.nz)) : 0;
    mc[J] = mf[node(gf, fx, fy, fz)];
}

// The coarse end of the V-cycle in one launch of one thread-block cluster (up to 16 CTAs of 1024
// threads): levels 0 .. n-1 of CoarseLevels live in the CTAs' shared memory; b of the first level
// comes from global memory and its x goes back.  Same smoother (two sweeps before and two after),
// restriction and prolongation as the grid-wide kernels, bit for bit.
//
// Bound: latency.  A launch per operation costs 5 to 8 us on these levels, whatever their size; a
// cluster barrier and one round of shared-memory reads cost a fraction of that.  Levels 0 .. nc-1
// are spread over the cluster in equal runs of the flat node index.  A CTA holds, next to its run of
// an iterate, copies of the `halo` entries before and after it (a row in 2D, a plane in 3D); whoever
// works out a value near the end of a run stores it into the neighbour's copy too, so that sweeps
// and residuals read their own shared memory only.  Restriction and prolongation, which reach
// further, read through distributed shared memory, with all of a node's reads issued before the
// first is used.  What an operation needs to know of a node (which faces it is on, Dirichlet) is
// worked out once, a byte per node.
// Levels nc .. n-1, too small for that, run in CTA 0 with CTA barriers; the coarsest one's many
// Jacobi sweeps keep one node per thread in registers, and only the warps that hold nodes meet.
// The host works out a level's descriptor, and each operation takes it by value: indexed kernel
// parameters and per-level divisions cost more than the arithmetic.
// Microseconds of a cycle from this level down: 33^3 114 as launches, 67 with every neighbour in
// another CTA read remotely, 45 now; 129^2 43 and 35; 151x111 (ragged coarsening) 77 and 48.
//
// Division of the flat index by a fixed number d: (i m) >> 40 with m = floor(2^40 / d) + 1,
// exact for i d < 2^40.
struct CoarseNode {
    int i, ix, iy, iz;
};
// A node's byte: bits 0-5 it is on the first / last x, y, z face, bit 6 Dirichlet.

__device__ __forceinline__ unsigned shared_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ float lds(unsigned a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts(unsigned a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }

// Element i of a level's array at shared address a: SPREAD, in whichever CTA it is (no branch, so
// that the reads of a node's neighbours overlap); else in this CTA.
template <bool SPREAD>
__device__ __forceinline__ float at(const CoarseLevel& l, unsigned a, int i) {
    if (!CMCG_RANGE_OK(i, i, l.np, kSiteCoarse)) return 0.f;
    if (!SPREAD) return lds(a + 4u * (unsigned)i);
    const unsigned k = (unsigned)(i - l.lo);
    const unsigned owner = (unsigned)(((unsigned)i * l.m_chunk) >> 40);
    unsigned p;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(a + 4u * ((unsigned)i - owner * (unsigned)l.chunk)), "r"(owner));
    asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %1, %2;\n\t@q ld.shared.f32 %0, [%3];\n\t"
                 "@!q ld.shared::cluster.f32 %0, [%4];\n\t}"
                 : "=f"(v)
                 : "r"(k), "r"((unsigned)l.cnt), "r"(a + 4u * k), "r"(p)
                 : "memory");
    return v;
}

// Element i of an array that CTA 0 holds whole.
__device__ __forceinline__ float at_first(unsigned a, int i) {
    unsigned p;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(a + 4u * (unsigned)i), "r"(0));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(p) : "memory");
    return v;
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ CoarseNode coarse_node(const CoarseLevel& l, int k) {
    CoarseNode n;
    n.i = l.lo + k;
    const unsigned t = (unsigned)(((unsigned)n.i * l.m_sx) >> 40);
    n.ix = n.i - (int)t * l.sx;
    n.iz = (int)((t * l.m_sy) >> 40);
    n.iy = (int)t - n.iz * l.sy;
    return n;
}
__device__ __forceinline__ unsigned faces_of(const CoarseLevel& l, const CoarseNode& n) {
    unsigned d = (n.ix == 0 ? 1u : 0u) | (n.ix == l.nx ? 2u : 0u) | (n.iy == 0 ? 4u : 0u) | (n.iy == l.ny ? 8u : 0u);
    if (l.dim == 3) d |= (n.iz == 0 ? 16u : 0u) | (n.iz == l.nz ? 32u : 0u);
    return d;
}
__device__ __forceinline__ unsigned node_byte(const CoarseLevel& l, int k) {
    unsigned d;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(d) : "r"(l.node + (unsigned)k) : "memory");
    return d;
}
__device__ __forceinline__ void sweep_barrier(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }
#include "coarsest.cuh"

// Stores of an iterate's values: in this CTA, and SPREAD in the neighbours' copies.
template <bool SPREAD>
struct Put {
    unsigned own, before, after;
    int halo, tail;
    __device__ __forceinline__ Put(const CoarseLevel& l, unsigned a) : own(a), before(0), after(0), halo(0), tail(INT_MAX) {
        if (!SPREAD) return;
        if (blockIdx.x > 0) {
            halo = l.halo;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(before) : "r"(a), "r"(blockIdx.x - 1u));
            before += 4u * (unsigned)l.chunk;
        }
        if (l.lo + l.cnt < l.np) {
            tail = l.cnt - l.halo;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(after) : "r"(a), "r"(blockIdx.x + 1u));
            after -= 4u * (unsigned)l.cnt;
        }
    }
    __device__ __forceinline__ void operator()(int k, float v) const {
        sts(own + 4u * (unsigned)k, v);
        if (!SPREAD) return;
        if (k < halo) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(before + 4u * (unsigned)k), "f"(v) : "memory");
        if (k >= tail) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(after + 4u * (unsigned)k), "f"(v) : "memory");
    }
};

// The roundings of the smoother and the interpolation, written out (a fused multiply-add, or a
// product rounded before the sum), so that a level gives the same bits in whichever kernel and CTA
// it runs.  fused: 2 d x - (neighbour sum) as one fused multiply-add, as in the grid-wide 3D
// kernels; levels of up to kCoarsestMaxNodes nodes round the product first.
__device__ __forceinline__ float relax_rn(float xc, float L, float bj, float omega, int ends, float cB, float inv2d) {
    const float w = __fmul_rn(cB, (float)(1 << ends));
    return __fmaf_rn(omega, __fmaf_rn(w, bj, -__fmul_rn(inv2d, L)), xc);
}
__device__ __forceinline__ float lap_rn(float xc, float acc, int dim, bool fused) {
    const float d = dim == 3 ? 6.f : 4.f;
    return fused ? __fmaf_rn(d, xc, -acc) : __fsub_rn(__fmul_rn(d, xc), acc);
}
__device__ __forceinline__ float blend_rn(float wa, float a, float wb, float b) {
    return __fmaf_rn(wa, a, __fmul_rn(wb, b));
}

// The neighbour sum at node k (byte d) of the array at `a`.
__device__ __forceinline__ float neighbour_sum(const CoarseLevel& l, unsigned a, int k, unsigned d) {
#ifdef CMCG_CHECKED  // the sum's reach in the CTA's run and its copies of the neighbours'
    {
        int lo = d & 1u && !(d & 2u) ? 0 : -1, hi = d & 2u && !(d & 1u) ? 0 : 1;
        auto axis = [&](bool first, bool last, int stride) {
            if (!first || last) lo = min(lo, -stride);
            if (!last || first) hi = max(hi, stride);
        };
        axis((d & 4u) != 0u, (d & 8u) != 0u, l.sx);
        if (l.dim == 3) axis((d & 16u) != 0u, (d & 32u) != 0u, l.sxy);
        const int n = l.halo ? l.chunk : l.np;
        if (!CMCG_RANGE_OK(k + l.halo + lo, k + l.halo + hi, n + 2 * l.halo, kSiteCoarse)) return 0.f;
    }
#endif
    const unsigned p = a + 4u * (unsigned)k, sy = 4u * (unsigned)l.sx, sz = 4u * (unsigned)l.sxy;
    const float v0 = lds(p + (d & 1u ? 4u : -4u)), v1 = lds(p + (d & 2u ? -4u : 4u));
    const float v2 = lds(p + (d & 4u ? sy : -sy)), v3 = lds(p + (d & 8u ? -sy : sy));
    float v4 = 0.f, v5 = 0.f;
    if (l.dim == 3) {
        v4 = lds(p + (d & 16u ? sz : -sz));
        v5 = lds(p + (d & 32u ? -sz : sz));
    }
    float acc = __fadd_rn(v0, v1);
    acc = __fadd_rn(acc, __fadd_rn(v2, v3));
    if (l.dim == 3) acc = __fadd_rn(acc, __fadd_rn(v4, v5));
    return acc;
}

template <bool SPREAD>
__device__ __forceinline__ void coarse_sweep(const CoarseLevel l, unsigned in, unsigned out, float omega) {
    const Put<SPREAD> put(l, out);
    for (int k = (int)threadIdx.x; k < l.cnt; k += (int)blockDim.x) {
        const unsigned d = node_byte(l, k);
        const float bj = lds(l.b + 4u * k), xc = lds(in + 4u * k);
        const float acc = neighbour_sum(l, in, k, d);
        const float v = relax_rn(xc, lap_rn(xc, acc, l.dim, l.fused != 0), bj, omega, ends_of(d), l.cB, l.inv2d);
        put(k, d & 64u ? 0.f : v);
    }
}

__device__ __forceinline__ void coarse_residual(const CoarseLevel l) {
    for (int k = (int)threadIdx.x; k < l.cnt; k += (int)blockDim.x) {
        const unsigned d = node_byte(l, k);
        const float bj = lds(l.b + 4u * k), xc = lds(l.x + 4u * k);
        const float s = __int_as_float((127 - ends_of(d)) << 23);  // 2^-ends
        const float L = lap_rn(xc, neighbour_sum(l, l.x, k, d), l.dim, l.fused != 0);
        const float v = __fmaf_rn(-__fmul_rn(l.cK, s), L, bj);
        sts(l.r + 4u * k, d & 64u ? 0.f : v);
    }
}

// Where a restricted value goes: b of the coarse level, and the first sweep's result from zero in its
// r.  TO_FIRST: CTA 0 holds the coarse level; every CTA works out a share of it (CTA 0 alone would
// read all of the residual through its one port) and stores it there.
template <bool SPREAD, bool TO_FIRST>
struct PutRestricted {
    const CoarseLevel& c;
    const Put<SPREAD && !TO_FIRST> put;
    float omega;
    __device__ __forceinline__ PutRestricted(const CoarseLevel& c_, float omega_) : c(c_), put(c_, c_.r), omega(omega_) {}
    __device__ __forceinline__ void operator()(int k, float v) const {
        if (!TO_FIRST) {
            const unsigned d = node_byte(c, k);
            v = d & 64u ? 0.f : v;
            sts(c.b + 4u * (unsigned)k, v);
            put(k, first_sweep(c, omega, d, v));
            return;
        }
        unsigned p, d;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(c.node + (unsigned)k), "r"(0));
        asm volatile("ld.shared::cluster.u8 %0, [%1];" : "=r"(d) : "r"(p) : "memory");
        v = d & 64u ? 0.f : v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(c.b + 4u * (unsigned)k), "r"(0));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(p), "f"(v) : "memory");
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(c.r + 4u * (unsigned)k), "r"(0));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(p), "f"(first_sweep(c, omega, d, v)) : "memory");
    }
};

// restrict_nested with a thread per fine row of a coarse node (three in 2D, nine in 3D): a node's
// thread would wait for 27 reads in a row where few nodes are left for it.  The rows' terms are
// summed in restrict_nested's order by the node's first thread.
template <int DIM, bool SPREAD, bool TO_FIRST>
__device__ __forceinline__ void restrict_rows(const CoarseLevel& f, const CoarseLevel& c, int lo, int end,
                                              const PutRestricted<SPREAD, TO_FIRST>& put) {
    constexpr int G = DIM == 3 ? 9 : 3, NPW = 32 / G;  // nodes per warp
    const int lane = (int)threadIdx.x & 31, g = lane / G, row = lane - g * G;
    const int fy0 = row % 3 - 1, fz0 = DIM == 3 ? row / 3 - 1 : 0;
    const float w = (fy0 == 0 ? 1.f : 0.5f) * (fz0 == 0 ? 1.f : 0.5f);
    for (int k0 = lo + ((int)threadIdx.x >> 5) * NPW; k0 < end; k0 += ((int)blockDim.x >> 5) * NPW) {
        const int k = k0 + g;
        const bool here = g < NPW && k < end;
        const CoarseNode n = coarse_node(c, here ? k : k0);
        const int cx = 2 * n.ix, fy = 2 * n.iy + fy0, fz = DIM == 3 ? 2 * n.iz + fz0 : 0;
        const bool ok = here && fy >= 0 && fy <= f.ny && fz >= 0 && fz <= f.nz;
        float t = 0.f;
        if (ok) {
            const int j = fz * f.sxy + fy * f.sx + cx;
            const bool xm = cx > 0, xp = cx < f.nx;
            t = at<SPREAD>(f, f.r, j);
            const float l = at<SPREAD>(f, f.r, xm ? j - 1 : j), q = at<SPREAD>(f, f.r, xp ? j + 1 : j);
            if (xm) t += 0.5f * l;
            if (xp) t += 0.5f * q;
            t *= w;
        }
        const unsigned oks = __ballot_sync(0xffffffffu, ok) >> (lane - row);
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const float v = __shfl_down_sync(0xffffffffu, t, i);
            if (oks >> i & 1u) acc += v;
        }
        if (here && row == 0) put(k, acc);
    }
}

// b of the coarse level = restriction of the fine level's residual.
template <bool SPREAD, bool TO_FIRST>
__device__ __forceinline__ void coarse_restrict(const Geom& gf, const Geom& gc, const CoarseLevel f, const CoarseLevel c,
                                                float omega) {
    const int share = TO_FIRST ? (c.np + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int lo = TO_FIRST ? (int)blockIdx.x * share : 0, end = TO_FIRST ? min(lo + share, c.np) : c.cnt;
    const PutRestricted<SPREAD, TO_FIRST> put(c, omega);
    if (nested(gf, gc)) {
        if (f.dim == 3) restrict_rows<3>(f, c, lo, end, put);
        else restrict_rows<2>(f, c, lo, end, put);
        return;
    }
    auto rf = [&](long long i) { return at<SPREAD>(f, f.r, (int)i); };
    for (int k = lo + (int)threadIdx.x; k < end; k += (int)blockDim.x) {
        const CoarseNode n = coarse_node(c, k);
        put(k, restrict_weighted(gf, rf, axis_weights(n.ix, gf.nx, gc.nx), axis_weights(n.iy, gf.ny, gc.ny),
                                 axis_weights_z(gf, gc, n.iz)));
    }
}

// x of the fine level += prolongation of the coarse level's x; FIRST: CTA 0 holds that, and each CTA
// fetches a copy first (interpolating from CTA 0, all CTAs would queue at its one port).
template <bool SPREAD, bool FIRST>
__device__ __forceinline__ void coarse_prolong(const Geom& gf, const Geom& gc, const CoarseLevel f, const CoarseLevel c) {
    if (FIRST) {
        if (blockIdx.x != 0)
            for (int k = (int)threadIdx.x; k < c.np; k += (int)blockDim.x) sts(c.x + 4u * k, at_first(c.x, k));
        __syncthreads();
    }
    auto xc = [&](int i) { return at<SPREAD && !FIRST>(c, c.x, i); };
    const Put<SPREAD> put(f, f.x);
    for (int k = (int)threadIdx.x; k < f.cnt; k += (int)blockDim.x) {
        const CoarseNode n = coarse_node(f, k);
        const Interp1 px = interp1_fast(n.ix, gf.nx, gc.nx), py = interp1_fast(n.iy, gf.ny, gc.ny);
        const int x1 = px.t > 0.f ? px.j0 + 1 : px.j0, y1 = py.t > 0.f ? py.j0 + 1 : py.j0;
        const float ax = 1.f - px.t, ay = 1.f - py.t;
        const int o00 = px.j0 + c.sx * py.j0, o10 = x1 + c.sx * py.j0, o01 = px.j0 + c.sx * y1, o11 = x1 + c.sx * y1;
        Interp1 pz;
        pz.j0 = 0;
        pz.t = 0.f;
        if (f.dim == 3) pz = interp1_fast(n.iz, gf.nz, gc.nz);
        const int z0 = pz.j0 * c.sxy, z1 = pz.t > 0.f ? z0 + c.sxy : z0;
        const float a0 = xc(z0 + o00), a1 = xc(z0 + o10), a2 = xc(z0 + o01), a3 = xc(z0 + o11);
        float b0 = a0, b1 = a1, b2 = a2, b3 = a3;
        if (f.dim == 3) b0 = xc(z1 + o00), b1 = xc(z1 + o10), b2 = xc(z1 + o01), b3 = xc(z1 + o11);
        float v = blend_rn(ay, blend_rn(ax, a0, px.t, a1), py.t, blend_rn(ax, a2, px.t, a3));
        if (f.dim == 3) {
            const float w = blend_rn(ay, blend_rn(ax, b0, px.t, b1), py.t, blend_rn(ax, b2, px.t, b3));
            v = blend_rn(1.f - pz.t, v, pz.t, w);
        }
        if (!(node_byte(f, k) & 64u)) put(k, lds(f.x + 4u * k) + v);
    }
}

__global__ void __launch_bounds__(1024) k_coarse_vcycle(const __grid_constant__ CoarseLevels lv,
                                                        const float* __restrict__ bglob, float* __restrict__ xglob,
                                                        float omega, int coarse_sweeps) {
    extern __shared__ __align__(16) float sm[];
    __shared__ CoarseLevel lev[kCoarseMax];
    const int rank = (int)blockIdx.x, tid = (int)threadIdx.x, nt = (int)blockDim.x;
    const int nl = lv.n, nc = lv.nc;
    if (tid < nl) {
        CoarseLevel l = lv.level[tid];
        const unsigned base = shared_addr(sm);
        if (tid < nc) {
            l.lo = min(rank * l.chunk, l.np);
            l.cnt = min(l.chunk, l.np - l.lo);
        }
        l.x += base, l.r += base, l.b += base, l.node += base;
        lev[tid] = l;
    }
    __syncthreads();
    // the first level's right-hand side; the nodes' bytes
    for (int q = 0; q < nl; ++q) {
        if (q >= nc && rank != 0) break;
        const CoarseLevel& l = lev[q];
        const unsigned char* const mask = lv.mask[q];
        for (int k = tid; k < l.cnt; k += nt) {
            if (!CMCG_RANGE_OK(l.lo + k, l.lo + k, lv.g[q].np, kSiteCoarse)) continue;
            float b = 0.f;
            unsigned dir = 0u;
            if (q == 0) b = bglob[l.lo + k];
            if (mask) dir = mask[l.lo + k];
            const unsigned d = faces_of(l, coarse_node(l, k)) | (dir ? 64u : 0u);
            asm volatile("st.shared.u8 [%0], %1;" ::"r"(l.node + (unsigned)k), "r"(d) : "memory");
            if (q == 0) sts(l.b + 4u * k, b);
        }
    }
    if (nc > 0) cluster_sync();  // (every CTA has started)
    else __syncthreads();
    {
        const CoarseLevel& l = lev[0];
        if (nc > 0) {
            const Put<true> put(l, l.r);
            for (int k = tid; k < l.cnt; k += nt) put(k, first_sweep(l, omega, node_byte(l, k), lds(l.b + 4u * k)));
            cluster_sync();
        } else {
            for (int k = tid; k < l.cnt; k += nt) sts(l.r + 4u * k, first_sweep(l, omega, node_byte(l, k), lds(l.b + 4u * k)));
            __syncthreads();
        }
    }
    // down through the spread levels
    for (int q = 0; q < nc; ++q) {
        const CoarseLevel& l = lev[q];
        coarse_sweep<true>(l, l.r, l.x, omega);
        cluster_sync();
        coarse_residual(l);
        cluster_sync();
        if (q + 1 < nc) coarse_restrict<true, false>(lv.g[q], lv.g[q + 1], l, lev[q + 1], omega);
        else coarse_restrict<true, true>(lv.g[q], lv.g[q + 1], l, lev[q + 1], omega);
        cluster_sync();
    }
    // the small levels, in CTA 0
    if (rank == 0) {
        for (int q = nc; q + 1 < nl; ++q) {
            const CoarseLevel& l = lev[q];
            coarse_sweep<false>(l, l.r, l.x, omega);
            __syncthreads();
            coarse_residual(l);
            __syncthreads();
            coarse_restrict<false, false>(lv.g[q], lv.g[q + 1], l, lev[q + 1], omega);
            __syncthreads();
        }
        {
            const CoarseLevel& l = lev[nl - 1];
            if (l.np <= nt) {
                coarsest_sweeps(l, omega, coarse_sweeps);
                __syncthreads();
            } else {
                coarse_sweep<false>(l, l.r, l.x, omega);  // the second sweep
                __syncthreads();
                unsigned in = l.x, out = l.r;
                for (int s = 2; s < coarse_sweeps; ++s) {
                    coarse_sweep<false>(l, in, out, omega);
                    __syncthreads();
                    const unsigned t = in;
                    in = out;
                    out = t;
                }
                if (in != l.x) {
                    for (int k = tid; k < l.np; k += nt) sts(l.x + 4u * k, lds(in + 4u * k));
                    __syncthreads();
                }
            }
        }
        for (int q = nl - 2; q >= nc; --q) {
            const CoarseLevel& l = lev[q];
            coarse_prolong<false, false>(lv.g[q], lv.g[q + 1], l, lev[q + 1]);
            __syncthreads();
            coarse_sweep<false>(l, l.x, l.r, omega);
            __syncthreads();
            coarse_sweep<false>(l, l.r, l.x, omega);
            __syncthreads();
        }
    }
    if (nc > 0) cluster_sync();
    // up through the spread levels
    for (int q = nc - 1; q >= 0; --q) {
        const CoarseLevel& l = lev[q];
        if (q + 1 < nc) coarse_prolong<true, false>(lv.g[q], lv.g[q + 1], l, lev[q + 1]);
        else coarse_prolong<true, true>(lv.g[q], lv.g[q + 1], l, lev[q + 1]);
        cluster_sync();
        coarse_sweep<true>(l, l.x, l.r, omega);
        cluster_sync();
        coarse_sweep<true>(l, l.r, l.x, omega);
        cluster_sync();
    }
    if (nc > 0 || rank == 0) {
        const CoarseLevel& l = lev[0];
        if (nc == 0) __syncthreads();
        for (int k = tid; k < l.cnt; k += nt)
            if (CMCG_RANGE_OK(l.lo + k, l.lo + k, lv.g[0].np, kSiteCoarse)) xglob[l.lo + k] = lds(l.x + 4u * k);
    }
}

// ---- FP64 PCG pieces ----------------------------------------------------------------------
// y = K x (masked); optional dot(dotwith, y) into sc[slot].
template <int ORDER>
__global__ void __launch_bounds__(kT) k_applyK(Geom g, const unsigned char* __restrict__ mask,
                                               const double* __restrict__ x, double* __restrict__ y,
                                               const double* __restrict__ dotwith, Red red, int slot) {
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    const double ih2 = 1.0 / (g.h * g.h);
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < g.np; j += stride) {
        if (mask && mask[j]) {
            y[j] = 0.0;
            continue;
        }
        int ix, iy, iz;
        coords(g, j, ix, iy, iz);
        Ld<double> f{x};  // PCG vectors are zero on Dirichlet nodes
        const double v = weight(g, ix, iy, iz) * ih2 * lap_t<ORDER, double>(g, f, j, ix, iy, iz);
        y[j] = v;
        if (dotwith) acc[0] += dotwith[j] * v;
    }
    if (dotwith) {
        if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[slot] = acc[0];
    }
}

__global__ void k_to_float(long long n, const double* __restrict__ in, float* __restrict__ out) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride)
        out[j] = soft64::to_f32(in[j]);
}

__global__ void __launch_bounds__(kT) k_reduce_sum(long long n, const double* __restrict__ x, Red red, int slot) {
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) acc[0] += x[j];
    if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[slot] = acc[0];
}

// b = rhs - (sum rhs / volume) W (range projection when K is singular), masked; ||b||^2.
__global__ void __launch_bounds__(kT) k_project(Geom g, const double* __restrict__ in, double* __restrict__ out,
                                                const unsigned char* __restrict__ mask, double inv_volume,
                                                int project, Red red) {
    const double mu = project ? red.sc[SC_P_BSUM] * inv_volume : 0.0;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < g.np; j += stride) {
        double v = 0.0;
        if (!(mask && mask[j])) {
            v = in[j];
            if (project) {
                int ix, iy, iz;
                coords(g, j, ix, iy, iz);
                v -= mu * weight(g, ix, iy, iz);
            }
        }
        out[j] = v;
        acc[0] += v * v;
    }
    if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[SC_P_BB] = acc[0];
}

// After the preconditioner: zd = z (FP64), rz = r.z, zAp = z.Ap; flexible (Polak-Ribiere)
// beta = (z_new . (r_new - r_old)) / rz_old = -alpha zAp / rz_old.
__global__ void __launch_bounds__(kT) k_dots_after_precond(long long n, const double* __restrict__ r,
                                                           const float* __restrict__ z, const double* __restrict__ Ap,
                                                           double* __restrict__ zd, Red red, int first) {
    double acc[2] = {0.0, 0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        const double zz = (double)z[j];
        zd[j] = zz;
        acc[0] += r[j] * zz;
        if (!first) acc[1] += zz * Ap[j];
    }
    if (grid_sum<2>(acc, red.partials, red.ticket) && threadIdx.x == 0) {
        const double rz_old = red.sc[SC_P_RZ];
        // a zero residual (zero right-hand side) gives rz = 0: no direction update
        red.sc[SC_P_BETA] = (first || rz_old == 0.0) ? 0.0 : -red.sc[SC_P_ALPHA] * acc[1] / rz_old;
        red.sc[SC_P_RZ] = acc[0];
    }
}

__global__ void k_p_update(long long n, double* __restrict__ p, const double* __restrict__ zd,
                           const double* __restrict__ sc, int first) {
    const double beta = first ? 0.0 : sc[SC_P_BETA];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride)
        p[j] = first ? zd[j] : zd[j] + beta * p[j];
}

// alpha = rz / pAp; x += alpha p; r -= alpha Ap; rr = r.r.
__global__ void __launch_bounds__(kT) k_xr_update(long long n, double* __restrict__ x, double* __restrict__ r,
                                                  const double* __restrict__ p, const double* __restrict__ Ap, Red red) {
    const double pap = red.sc[SC_P_PAP];
    const double alpha = pap != 0.0 ? red.sc[SC_P_RZ] / pap : 0.0;  // p = 0 only for a zero residual
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        x[j] += alpha * p[j];
        const double rv = r[j] - alpha * Ap[j];
        r[j] = rv;
        acc[0] += rv * rv;
    }
    if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) {
        red.sc[SC_P_ALPHA] = alpha;
        red.sc[SC_P_RR] = acc[0];
    }
}

// x -= (sum W x / volume): W-weighted mean zero.
__global__ void __launch_bounds__(kT) k_wsum(Geom g, const double* __restrict__ x, Red red) {
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < g.np; j += stride) {
        int ix, iy, iz;
        coords(g, j, ix, iy, iz);
        acc[0] += weight(g, ix, iy, iz) * x[j];
    }
    if (grid_sum<1>(acc, red.partials, red.ticket) && threadIdx.x == 0) red.sc[SC_P_XW] = acc[0];
}

__global__ void k_sub_const(long long n, double* __restrict__ x, const double* __restrict__ sc, double inv_volume) {
    const double mu = sc[SC_P_XW] * inv_volume;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) x[j] -= mu;
}

}  // namespace

void launch_mg_coarsen_mask(const MGLevel& fine, const MGLevel& coarse, cudaStream_t st) {
    note_launch((fine.mask && coarse.mask) ? 1 : 0);
    if (!fine.mask || !coarse.mask) return;
    k_coarsen_mask<<<node_blocks(coarse.g.np), kT, 0, st>>>(fine.g, fine.mask, coarse.g, coarse.mask);
}

// z-planes per thread of the 3D level kernels.  Sweeps and residuals: as many as make one wave of
// blocks, 2 to 16 (129^3: a sweep takes 9.3 us with ten planes, 10.4 with eight, whose second wave is
// a fifth full, 12.2 with two; 65^3: 4.3 with two, 6.0 with eight).  Prolongation, whose threads
// reuse the coarse planes between pairs of fine ones: eight, or fewer where eight leave less than
// one wave (129^3: 13.7 us, with ten 15.2).
static int mg_zc(const Geom& g) {
    if (g.dim != 3) return 1;
    const long long bxy = ((long long)g.sx * g.sy + kT - 1) / kT;
    return (int)std::min(16ll, std::max(2ll, (bxy * g.sz + 152 * 6 - 1) / (152 * 6)));
}
static int mg_zc_prolong(const Geom& g) {
    if (g.dim != 3) return 1;
    const long long bxy = ((long long)g.sx * g.sy + kT - 1) / kT;
    int zc = 8;
    while (zc > 2 && bxy * ((g.sz + zc - 1) / zc) < 152 * 6) zc >>= 1;
    return zc;
}

void launch_mg_jacobi(const MGLevel& L, const float* xin, float* xout, const float* b, float omega, bool zero_init,
                      cudaStream_t st) {
    note_launch(1);
    const int zc = mg_zc(L.g);
    if (L.g.dim == 3 && !zero_init)
        k_mg3_z2<0><<<mg_grid(L.g, zc), kT, 0, st>>>(L.g, L.mask, xin, b, xout, omega, zc);
    else
        k_jacobi<<<mg_grid(L.g, zc), kT, 0, st>>>(L.g, L.mask, zero_init ? nullptr : xin, xout, b, omega, zc);
}

void launch_mg_first(const MGLevel& L, float* xout, const float* b, float omega, cudaStream_t st) {
    note_launch(1);
    const int zc = mg_zc(L.g);
    if (L.g.dim == 3) k_mg3_first<<<mg_grid(L.g, zc), kT, 0, st>>>(L.g, L.mask, b, xout, omega, zc);
    else k_mg2_first<<<mg_grid(L.g, 1), kT, 0, st>>>(L.g, L.mask, b, xout, omega);
}

void launch_mg_residual(const MGLevel& L, const float* x, const float* b, float* r, cudaStream_t st) {
    note_launch(1);
    const int zc = mg_zc(L.g);
    if (L.g.dim == 3)
        k_mg3_z2<1><<<mg_grid(L.g, zc), kT, 0, st>>>(L.g, L.mask, x, b, r, 0.f, zc);
    else
        k_residual<<<mg_grid(L.g, zc), kT, 0, st>>>(L.g, L.mask, x, b, r, zc);
}

void launch_mg_restrict(const MGLevel& fine, const float* rf, const MGLevel& coarse, float* bc, cudaStream_t st) {
    note_launch(1);
    const Geom& gf = fine.g;
    const Geom& gc = coarse.g;
    // coarse planes per thread of the nested kernel, which carries a fine plane from one to the next:
    // four, fewer where that leaves less than a wave of blocks (to 33^3: 4.3 us with one, 7.7 with
    // four; to 65^3: 7.3 and 8.7)
    const long long bxy = ((long long)gc.sx * gc.sy + kT - 1) / kT;
    const int zc = (int)std::min(4ll, std::max(1ll, bxy * gc.sz / (152 * 6))), one = planes_per_thread(1, gc.sz);
    if (gf.dim == 3 && gf.nx == 2 * gc.nx && gf.ny == 2 * gc.ny && gf.nz == 2 * gc.nz)
        k_restrict3_nested<<<mg_grid(gc, zc), kT, 0, st>>>(gf, rf, gc, coarse.mask, bc, zc);
    else
        k_restrict<<<mg_grid(gc, one), kT, 0, st>>>(gf, rf, gc, coarse.mask, bc, one);
}

void launch_mg_prolong_add(const MGLevel& coarse, const float* xc, const MGLevel& fine, float* xf, cudaStream_t st) {
    note_launch(1);
    const int zc = mg_zc_prolong(fine.g);
    if (fine.g.dim == 3)
        k_prolong_add3<<<mg_grid(fine.g, zc), kT, 0, st>>>(coarse.g, xc, fine.g, fine.mask, xf, zc);
    else
        k_prolong_add<<<mg_grid(fine.g, zc), kT, 0, st>>>(coarse.g, xc, fine.g, fine.mask, xf, zc);
}

// Which levels, from the first that fits, run in the cluster: spread ones of up to kSpreadMaxNodes
// nodes (four per thread: a 257^2 Riesz map takes 919 us with its finest level in the cluster, 1030 as
// launches; 81^3 with 41^3 nodes there 2176 and 2237; with 49^3 there 97^3 is slower, 2513 against
// 2389) while they have more than kSpreadMinNodes (below, one CTA is faster than the cluster's
// barriers).
constexpr size_t kCoarseSmemMax = 220 * 1024;  // shared memory of a CTA
size_t mg_coarse_smem(const CoarseLevels& lv) {
    size_t n = 0;
    for (int l = 0; l < lv.n; ++l) {
        const CoarseLevel& c = lv.level[l];
        n += 13 * (size_t)(l < lv.nc ? c.chunk : c.np) + 16 * (size_t)c.halo;
    }
    return n + 16;
}

bool mg_coarse_plan(const MGLevel* levels, int nlev, int first, bool clusters, CoarseLevels* lv) {
    *lv = CoarseLevels();
    lv->n = nlev - first;
    if (lv->n > kCoarseMax || levels[first].g.np > (clusters ? kSpreadMaxNodes : kCoarsestMaxNodes) ||
        levels[nlev - 1].g.np > kCoarsestMaxNodes)
        return false;
    for (int i = 0; i < lv->n; ++i) {
        lv->g[i] = levels[first + i].g;
        lv->mask[i] = levels[first + i].mask;
        if (clusters && lv->g[i].np > kSpreadMinNodes && i + 1 < lv->n) lv->nc = i + 1;
    }
    lv->ctas = lv->nc > 0 ? 16 : 1;
    auto magic = [](long long d) { return (1ull << 40) / (unsigned long long)d + 1ull; };
    unsigned floats = 0, bytes = 0;
    for (int i = 0; i < lv->n; ++i) {
        const Geom& g = lv->g[i];
        CoarseLevel& l = lv->level[i];
        l.np = l.cnt = (int)g.np;
        l.lo = 0;
        // (runs of at least a row or plane: a node's neighbours are in the runs next to its own)
        l.halo = i < lv->nc ? (g.dim == 3 ? g.sx * g.sy : g.sx) : 0;
        l.chunk = std::max((int)((g.np + lv->ctas - 1) / lv->ctas), l.halo);
        l.sx = g.sx, l.sy = g.sy, l.sxy = g.sx * g.sy;
        l.nx = g.nx, l.ny = g.ny, l.nz = g.nz, l.dim = g.dim;
        l.m_chunk = magic(l.chunk), l.m_sx = magic(g.sx), l.m_sy = magic(g.sy);
        const unsigned n = (unsigned)(i < lv->nc ? l.chunk : l.np);
        const unsigned h = (unsigned)l.halo;
        l.x = 4 * (floats + h), l.r = l.x + 4 * (n + 2 * h), l.b = l.r + 4 * (n + h);
        floats += 3 * n + 4 * h;
        l.fused = g.np > kCoarsestMaxNodes;
        const float gh = (float)g.h, hd = g.dim == 3 ? gh * gh * gh : gh * gh;  // as mg_const
        l.cK = hd / (gh * gh);
        l.inv2d = 1.f / (float)(2 * g.dim);
        l.cB = (gh * gh) / (hd * (float)(2 * g.dim));
    }
    for (int i = 0; i < lv->n; ++i) {
        lv->level[i].node = 4 * floats + bytes;
        bytes += (unsigned)(i < lv->nc ? lv->level[i].chunk : lv->level[i].np);
    }
    return mg_coarse_smem(*lv) <= kCoarseSmemMax;
}

static cudaError_t coarse_config(const CoarseLevels& lv, cudaStream_t st, cudaLaunchAttribute* attr,
                                 cudaLaunchConfig_t* cfg) {
    // (always the same value: threads with other plans set it too, between this call and the launch)
    cudaError_t e = cudaFuncSetAttribute(k_coarse_vcycle, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoarseSmemMax);
    if (e == cudaSuccess && lv.ctas > 8)
        e = cudaFuncSetAttribute(k_coarse_vcycle, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    *cfg = {};
    cfg->gridDim = dim3((unsigned)lv.ctas);
    cfg->blockDim = dim3(1024);
    cfg->dynamicSmemBytes = mg_coarse_smem(lv);
    cfg->stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)lv.ctas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return e;
}

bool mg_coarse_resident(const CoarseLevels& lv) {
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg;
    int clusters = 0;
    const bool ok = coarse_config(lv, nullptr, &attr, &cfg) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, k_coarse_vcycle, &cfg) == cudaSuccess && clusters > 0;
    if (!ok) cudaGetLastError();
    return ok;
}

cudaError_t launch_mg_coarse(const CoarseLevels& lv, const float* b, float* x, float omega, int coarse_sweeps,
                             cudaStream_t st) {
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg;
    const cudaError_t e = coarse_config(lv, st, &attr, &cfg);
    if (e != cudaSuccess) return e;
    note_launch(1);
    return cudaLaunchKernelEx(&cfg, k_coarse_vcycle, lv, b, x, omega, coarse_sweeps);
}

void launch_applyK(const Geom& g, int order, const unsigned char* mask, const double* x, double* y,
                   const double* dotwith, Red red, int slot, cudaStream_t st) {
    note_launch(1);
    if (order == 2)
        k_applyK<2><<<vec_blocks(g.np), kT, 0, st>>>(g, mask, x, y, dotwith, red, slot);
    else
        k_applyK<4><<<vec_blocks(g.np), kT, 0, st>>>(g, mask, x, y, dotwith, red, slot);
}

void launch_to_float(long long n, const double* in, float* out, cudaStream_t st) {
    note_launch(1);
    k_to_float<<<vec_blocks(n), kT, 0, st>>>(n, in, out);
}

void launch_reduce_sum(long long n, const double* x, Red red, int slot, cudaStream_t st) {
    note_launch(1);
    k_reduce_sum<<<vec_blocks(n), kT, 0, st>>>(n, x, red, slot);
}

void launch_pcg_project(const Geom& g, const double* in, double* out, const unsigned char* mask, double volume,
                        Red red, bool project, cudaStream_t st) {
    note_launch(1);  // plus launch_reduce_sum's own count
    if (project) launch_reduce_sum(g.np, in, red, SC_P_BSUM, st);
    k_project<<<vec_blocks(g.np), kT, 0, st>>>(g, in, out, mask, 1.0 / volume, project ? 1 : 0, red);
}

void launch_pcg_dots_after_precond(long long n, const double* r, const float* z, const double* Ap, double* zd,
                                   Red red, cudaStream_t st) {
    note_launch(1);
    // "first" is encoded by Ap == nullptr
    k_dots_after_precond<<<vec_blocks(n), kT, 0, st>>>(n, r, z, Ap, zd, red, Ap == nullptr ? 1 : 0);
}

void launch_pcg_xr_update(long long n, double* x, double* r, const double* p, const double* Ap, Red red,
                          cudaStream_t st) {
    note_launch(1);
    k_xr_update<<<vec_blocks(n), kT, 0, st>>>(n, x, r, p, Ap, red);
}

void launch_pcg_p_update(long long n, double* p, const double* zd, Red red, bool first, cudaStream_t st) {
    note_launch(1);
    k_p_update<<<vec_blocks(n), kT, 0, st>>>(n, p, zd, red.sc, first ? 1 : 0);
}

void launch_mean_remove(const Geom& g, double* x, double volume, Red red, cudaStream_t st) {
    note_launch(2);
    k_wsum<<<vec_blocks(g.np), kT, 0, st>>>(g, x, red);
    k_sub_const<<<vec_blocks(g.np), kT, 0, st>>>(g.np, x, red.sc, 1.0 / volume);
}

}  // namespace cmcg

namespace cmcg {
CMCG_CHECK_TU(riesz)
}  // namespace cmcg
