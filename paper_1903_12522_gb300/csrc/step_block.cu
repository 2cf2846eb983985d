// FP32 3D 7-point step loops in one launch, the grid held on chip: the 3D counterpart of
// step_band.cu for grids of up to about 2.3 million nodes (129^3).
//
// Such a grid's wave fields and kappa fit the registers and shared memory of the chip (73 MB), but a
// step at a time costs 8 to 11 us, most of it launch, ramp and drain.  One CTA per SM owns a block
// of whole x rows, ty by tz of them, for the whole loop: y^n in shared memory (two buffers),
// y^{n-1} and kappa in registers, eight float4 chunks of a row per thread at most.  Only the
// block's outermost rows travel, as the self-flagged 8-byte words of step_band.cu, to its four
// neighbours; the rows that travel are computed first.  The rows' ends, which may be on absorbing
// faces, are dealt to warps of their own (with them in every warp: 11 us a step at 129^3).  The
// endpoint kernels' flat fields are read at the start and written at the end.
//
// Bound: shared memory (32 wavefronts per warp of chunks: five 16-byte reads, two 4-byte ones, one
// write; 2.0 us at 129^3) and then one trip through L2 for the exchange, about 1 us.
// Microseconds per step, slope over the step count (backward loop / source on the faces / source
// in a sphere's volume), against the kernels of step_row.cu and wave.cu step by step:
//   33^3 1.5 / 1.7 / 1.6 (8.3 / 9.4 / 9.5), 65^3 1.9 / 2.0 / 2.2 (8.3 / 10.3 / 10.4),
//   97^3 2.8 / 3.1 / 3.7 (8.2 / 10.3 / 10.3), 129^3 4.9 / 6.4 / 7.8 (10.3 / 12.4 / 12.4).
//
// The roundings are those of k_step3d7_z2, written out: same bits.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace cmcg {

namespace {

constexpr int kBT = 512;                 // 128 registers: 64 of them hold y^{n-1} and kappa
constexpr int kMaxBlocks3 = kBandStop;   // one per SM of a GB300
constexpr int kSmemMax3 = 226 * 1024;
constexpr int kHalo = 4;                 // halo chunks per thread

struct BlockArgs {
    float* buf0;  // y^n of the first step; buf1 y^{n-1}; they swap roles every step
    float* buf1;
    const float* kap;
    const float* S;
    const unsigned char* sflag;  // where there are sources (launch_source_flags)
    unsigned long long* words;
    unsigned* count;  // per block: steps done in all launches so far; [kBandStop]: stop word
    double* err;
    Geom g;
    int ny_blocks;              // blocks along y
    int ty, ey, tz, ez;         // rows of a block: ty + 1 for the first ey along y, ty for the others; same for z
    int side;                   // words of one side (4 per chunk, rows in the buffer's pitch)
    int nsteps, adj_first, adj_last;
    int polls;                  // the longest wait
    float cs[kBandSteps], sn[kBandSteps];
};

typedef unsigned long long u64;
__device__ __forceinline__ u64 pack(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack(u64 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
struct V4 {
    u64 a, b;
};
__device__ __forceinline__ V4 load4(const float* p) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    return V4{t.x, t.y};
}
__device__ __forceinline__ void store4(float* p, V4 v) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.a, v.b); }

__device__ __forceinline__ void put4(u64* p, V4 v, unsigned tag) {
    float f[4];
    unpack(v.a, f[0], f[1]);
    unpack(v.b, f[2], f[3]);
    const u64 t = (u64)tag << 32;
    const u64 w0 = t | __float_as_uint(f[0]), w1 = t | __float_as_uint(f[1]), w2 = t | __float_as_uint(f[2]),
              w3 = t | __float_as_uint(f[3]);
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p + 2), "l"(w2), "l"(w3) : "memory");
}
__device__ __forceinline__ void get4(const u64* p, u64 (&w)[4]) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(p));
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[2]), "=l"(w[3]) : "l"(p + 2));
}

__device__ __noinline__ float plain_div3(float v, float d) { return v / d; }

// v / d, correctly rounded, with r = 1 / d correctly rounded (see div_known in step_band.cu).
__device__ __forceinline__ float div_by(float v, float d, float r) {
    const float q0 = __fmul_rn(v, r);
    const float q = __fmaf_rn(__fmaf_rn(-q0, d, v), r, q0);
    const unsigned a = __float_as_uint(v) & 0x7fffffffu;
    if (a - 0x0d800000u < 0x6e000000u || a == 0u) return q;
    return plain_div3(v, d);
}

// Four nodes of which some are on absorbing faces: q = sqrt(kappa) (0 elsewhere) and 1 / (1 + beta),
// beta = nb q with nb faces through the node.
struct Face {
    float4 q, r;
};

// flag bits of a chunk
constexpr unsigned kHere = 1u, kFirst = 2u, kSource = 32u;  // 2-4: element of x = nx (7: none)
constexpr unsigned kSend = 64u, kGhost = 1024u;             // << side (0 -y, 1 +y, 2 -z, 3 +z)
constexpr int kFacesShift = 14;                             // absorbing y and z faces through the row (0 .. 2)
constexpr unsigned kLeft = 1u << 16, kRight = 1u << 17;     // the nodes x = 0, x = nx are on absorbing faces
constexpr int kSlotShift = 18;                              // face slot + 1

// SRC: 0 none, 1 on absorbing faces only, 2 anywhere.  They are read from L2 each step.
template <int NPC, int SRC>
__global__ void __launch_bounds__(kBT, 1) k_block3(const __grid_constant__ BlockArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned short row_of[512];  // (lz << 8 | ly) of the block's rows, those that travel first
    const Geom& g = a.g;
    const int blk = (int)blockIdx.x, tid = (int)threadIdx.x;
    const int by = blk % a.ny_blocks, bz = blk / a.ny_blocks;
    const int nyb = a.ny_blocks, nzb = (int)gridDim.x / nyb;
    const int y0 = by * a.ty + min(by, a.ey), ry = a.ty + (by < a.ey ? 1 : 0);
    const int z0 = bz * a.tz + min(bz, a.ez), rz = a.tz + (bz < a.ez ? 1 : 0);
    const int sx = g.sx, cx = (sx + 3) >> 2, P = 4 * cx + 8;  // node x at column x + 4
    const int my = a.ty + (a.ey ? 1 : 0) + 2, mz = a.tz + (a.ez ? 1 : 0) + 2;
    const int Y = P, Z = P * my;  // strides of a buffer's rows
    const int Y4 = Y >> 2, Z4 = Z >> 2;
    const int bufsz = Z * mz;
    float* const buf = reinterpret_cast<float*>(smem_raw);
    Face* const faces = reinterpret_cast<Face*>(buf + 2 * bufsz);
    const int nc = ry * rz * cx;
    const bool has[4] = {by > 0, by + 1 < nyb, bz > 0, bz + 1 < nzb};
    const int nbr[4] = {blk - 1, blk + 1, blk - nyb, blk + nyb};
    const unsigned base = a.count[blk];

    if (tid == 0) {  // rows that travel first
        int n = 0;
        for (int pass = 0; pass < 2; ++pass)
            for (int lz = 0; lz < rz; ++lz)
                for (int ly = 0; ly < ry; ++ly) {
                    const bool edge = ly == 0 || ly == ry - 1 || lz == 0 || lz == rz - 1;
                    if (edge == (pass == 0)) row_of[n++] = (unsigned short)(lz << 8 | ly);
                }
    }
    // the block and its halo rows of y^n (mirrored at the grid's faces)
    for (int i = tid; i < P * (ry + 2) * (rz + 2); i += kBT) {
        const int r = i / P, x = i - r * P - 4;
        const int lz = r / (ry + 2), ly = r - lz * (ry + 2);
        int y = y0 - 1 + ly, z = z0 - 1 + lz;
        y = y < 0 ? -y : (y > g.ny ? 2 * g.ny - y : y);
        z = z < 0 ? -z : (z > g.nz ? 2 * g.nz - z : z);
        const int o = lz * Z + ly * Y + x + 4;
        buf[o] = x >= 0 && x <= g.nx ? a.buf0[(long long)sx * (y + (long long)g.sy * z) + x] : 0.f;
        buf[bufsz + o] = 0.f;
    }
    __syncthreads();
    V4 prev[NPC], kap[NPC];
    unsigned crd[NPC];  // place in a buffer / 4 | lz << 13 | ly << 21
    unsigned fl[NPC];
#pragma unroll
    for (int q = 0; q < NPC; ++q) {
        const int i = tid + q * kBT;
        crd[q] = (unsigned)(Z4 + Y4 + 1);
        fl[q] = 0;
        prev[q] = kap[q] = V4{0ull, 0ull};
        if (i < nc) {
            // first the rows' ends, which may be on faces: warps of their own take the faces' path
            const int rows = ry * rz, k = i - 2 * rows;
            const int rr = k >= 0 ? k / (cx - 2) : (i < rows ? i : i - rows);
            const int ic = k >= 0 ? 1 + k - rr * (cx - 2) : (i < rows ? 0 : cx - 1);
            const int ly = row_of[rr] & 255, lz = row_of[rr] >> 8;
            const int y = y0 + ly, z = z0 + lz, x0 = 4 * ic, m = min(4, sx - x0);
            const long long j = (long long)sx * (y + (long long)g.sy * z) + x0;
            if (!CMCG_RANGE_OK(j, j + m - 1, g.np, kSiteColumn)) continue;
            crd[q] = (unsigned)((lz + 1) * Z4 + (ly + 1) * Y4 + ic + 1) | (unsigned)lz << 13 | (unsigned)ly << 21;
            float pv[4] = {0.f, 0.f, 0.f, 0.f}, kv[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e < m) {
                    pv[e] = a.buf1[j + e];
                    kv[e] = a.kap[j + e];
                }
            prev[q] = V4{pack(pv[0], pv[1]), pack(pv[2], pv[3])};
            kap[q] = V4{pack(kv[0], kv[1]), pack(kv[2], kv[3])};
            const bool last = g.nx - x0 < 4;
            unsigned f = kHere | (ic == 0 ? kFirst : 0u) | (unsigned)(last ? g.nx - x0 : 7) << 2;
            if (ly == 0 && has[0]) f |= kSend;
            if (ly == ry - 1 && has[1]) f |= kSend << 1;
            if (lz == 0 && has[2]) f |= kSend << 2;
            if (lz == rz - 1 && has[3]) f |= kSend << 3;
            if (y == 1) f |= kGhost;
            if (y == g.ny - 1) f |= kGhost << 1;
            if (z == 1) f |= kGhost << 2;
            if (z == g.nz - 1) f |= kGhost << 3;
            const int nby = (y == 0 && (g.abc & 4u) ? 1 : 0) + (y == g.ny && (g.abc & 8u) ? 1 : 0) +
                            (z == 0 && (g.abc & 16u) ? 1 : 0) + (z == g.nz && (g.abc & 32u) ? 1 : 0);
            const bool left = ic == 0 && (g.abc & 1u), right = last && (g.abc & 2u);
            if (nby || left || right) {
                // slots: the two ends of every row, then whole rows of the first / last y and z
                int slot;
                if (!nby) {
                    slot = 2 * (lz * ry + ly) + (left ? 0 : 1);
                } else {
                    slot = 2 * ry * rz;
                    const bool yl = y == 0 && (g.abc & 4u), yh = y == g.ny && (g.abc & 8u), zl = z == 0 && (g.abc & 16u);
                    // (one of the faces the row is on names its place; face areas in the order -y, +y, -z, +z)
                    const int ny_rows = (y0 == 0 && (g.abc & 4u) ? rz : 0);
                    const int py_rows = (y0 + ry - 1 == g.ny && (g.abc & 8u) ? rz : 0);
                    const int nz_rows = (z0 == 0 && (g.abc & 16u) ? ry : 0);
                    if (yl) slot += lz * cx;
                    else if (yh) slot += (ny_rows + lz) * cx;
                    else if (zl) slot += (ny_rows + py_rows + ly) * cx;
                    else slot += (ny_rows + py_rows + nz_rows + ly) * cx;
                    slot += ic;
                }
                float qe[4], rc[4];
                bool on[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int nb = nby + (left && e == 0 ? 1 : 0) + (right && e == g.nx - x0 ? 1 : 0);
                    on[e] = e < m && nb;
                    qe[e] = on[e] ? sqrtf(kv[e]) : 0.f;
                    rc[e] = __frcp_rn(__fmaf_rn((float)nb, qe[e], 1.f));
                }
                Face& fc = faces[slot];
                fc.q = make_float4(qe[0], qe[1], qe[2], qe[3]);
                fc.r = make_float4(rc[0], rc[1], rc[2], rc[3]);
                f |= (unsigned)(slot + 1) << kSlotShift | (unsigned)nby << kFacesShift | (left ? kLeft : 0u) | (right ? kRight : 0u);
            }
            bool source = SRC == 1 && (f >> kSlotShift);
            if (SRC == 2) source = a.sflag[((long long)(z >> 2) * g.sy + y) * cx + ic] != 0;
            fl[q] = f | (source ? kSource : 0u);
        }
    }
    // this thread's halo chunks: where their words arrive, and where they go in a buffer
    int hword[kHalo], hoff[kHalo];
    {
        const int n[4] = {has[0] ? rz * cx : 0, has[1] ? rz * cx : 0, has[2] ? ry * cx : 0, has[3] ? ry * cx : 0};
#pragma unroll
        for (int h = 0; h < kHalo; ++h) {
            int i = tid + h * kBT, side = 0;
            while (side < 4 && i >= n[side]) i -= n[side], ++side;
            hword[h] = -1;
            hoff[h] = 0;
            if (side < 4) {
                const int row = i / cx, ic = i - row * cx;
                hword[h] = side * a.side + 4 * (row * Y4 + ic);
                const int ly = side == 0 ? 0 : (side == 1 ? ry + 1 : row + 1);
                const int lz = side == 2 ? 0 : (side == 3 ? rz + 1 : row + 1);
                hoff[h] = lz * Z + ly * Y + 4 + 4 * ic;
            }
        }
    }
    __syncthreads();

    u64* const mine = a.words + (long long)blk * 8 * a.side;
    bool failed = false;
    for (int s = 0; s < a.nsteps; ++s) {
        const float* in = buf + (s & 1) * bufsz;
        float* out = buf + ((s + 1) & 1) * bufsz;
        int flags = 0;
        if (a.adj_first && s == 0) flags |= kStepPrevScaled;
        if (a.adj_last && s == a.nsteps - 1) flags |= kStepNoDiv;
        const float cs = SRC ? a.cs[s] : 0.f, sn = SRC ? a.sn[s] : 0.f;
        const bool more = s + 1 < a.nsteps;
        const unsigned tag = base + (unsigned)s + 1u;
        const int slot_off = (int)(tag & 1u) * 4 * a.side;
#pragma unroll
        for (int q = 0; q < NPC; ++q) {
            // (opaque: what follows from them is worked out each step, not kept in registers)
            asm volatile("" : "+r"(crd[q]), "+r"(fl[q]));
            const unsigned f = fl[q];
            if (!(f & kHere)) continue;
            const int o = (int)(crd[q] & 8191u) << 2, xe = (int)(f >> 2) & 7;
            const V4 c = load4(in + o);
            const V4 ym = load4(in + o - Y), yp = load4(in + o + Y), zm = load4(in + o - Z), zp = load4(in + o + Z);
            float xl = in[o - 1], xr = in[o + 4], v[4];
            float t[4] = {0.f, 0.f, 0.f, 0.f};
            if (SRC && (f & kSource)) {
                const int lz = (int)(crd[q] >> 13) & 255, ly = (int)(crd[q] >> 21), x0 = o - (lz + 1) * Z - (ly + 1) * Y - 4;
                const float2* sp = reinterpret_cast<const float2*>(a.S) +
                                   ((long long)sx * (y0 + ly + (long long)g.sy * (z0 + lz)) + x0);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 w = sp[x0 + e < sx ? e : 0];
                    t[e] = __fmaf_rn(w.x, cs, __fmul_rn(w.y, sn));
                }
            }
            unpack(c.a, v[0], v[1]);
            unpack(c.b, v[2], v[3]);
            if (f & kFirst) xl = v[1];
            const float xm[4] = {xl, v[0], v[1], v[2]}, xq[4] = {v[1], v[2], v[3], xr};
            float sx1[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) sx1[e] = xm[e] + (e == xe ? xm[e] : xq[e]);
            const u64 m6 = pack(-6.f, -6.f), m1 = pack(-1.f, -1.f);
            const u64 La = fma2(m6, c.a, add2(add2(pack(sx1[0], sx1[1]), add2(ym.a, yp.a)), add2(zm.a, zp.a)));
            const u64 Lb = fma2(m6, c.b, add2(add2(pack(sx1[2], sx1[3]), add2(ym.b, yp.b)), add2(zm.b, zp.b)));
            u64 ra = fma2(kap[q].a, La, add2(c.a, c.a)), rb = fma2(kap[q].b, Lb, add2(c.b, c.b));
            if (SRC == 2 && (f & kSource)) {
                ra = add2(ra, pack(t[0], t[1]));
                rb = add2(rb, pack(t[2], t[3]));
            }
            V4 w{fma2(m1, prev[q].a, ra), fma2(m1, prev[q].b, rb)};
            if (f >> kSlotShift) {
                const Face fc = faces[(f >> kSlotShift) - 1];
                const float nbx = (float)((f >> kFacesShift) & 3u);
                const float qe[4] = {fc.q.x, fc.q.y, fc.q.z, fc.q.w}, rc[4] = {fc.r.x, fc.r.y, fc.r.z, fc.r.w};
                float r[4], p[4], ov[4];
                unpack(ra, r[0], r[1]);
                unpack(rb, r[2], r[3]);
                unpack(prev[q].a, p[0], p[1]);
                unpack(prev[q].b, p[2], p[3]);
                if (SRC == 1) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) r[e] += t[e];
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float nb = nbx + ((e == 0 && (f & kLeft)) || (e == xe && (f & kRight)) ? 1.f : 0.f);
                    const float c1 = __fmaf_rn(-nb, qe[e], 1.f), d = __fmaf_rn(nb, qe[e], 1.f);
                    const float u = (flags & kStepPrevScaled) ? r[e] - p[e]
                                    : (flags & kStepNoDiv)    ? __fsub_rn(r[e], __fmul_rn(c1, p[e]))
                                                              : __fmaf_rn(-c1, p[e], r[e]);
                    ov[e] = (flags & kStepNoDiv) ? u : div_by(u, d, rc[e]);
                }
                w.a = pack(ov[0], ov[1]);
                w.b = pack(ov[2], ov[3]);
            }
            prev[q] = c;
            store4(out + o, w);
            if (f & (0xfu * kGhost)) {
                if (f & kGhost) store4(out + o - 2 * Y, w);
                if (f & kGhost << 1) store4(out + o + 2 * Y, w);
                if (f & kGhost << 2) store4(out + o - 2 * Z, w);
                if (f & kGhost << 3) store4(out + o + 2 * Z, w);
            }
            if (more && (f & (0xfu * kSend))) {
                // a side's words: chunks in the buffer's pitch, from its first row on
                const int lz = (int)(crd[q] >> 13) & 255;
                const int c0 = (o >> 2) - (lz + 1) * Z4 - 1, wz = 4 * (c0 - Y4);  // (ly + 1) Y4 + ic; z sides' word
                const int ly = (int)(crd[q] >> 21), wy = 4 * (c0 - (ly + 1 - lz) * Y4);
#pragma unroll
                for (int side = 0; side < 4; ++side)
                    if (f & (kSend << side))  // it arrives there from the opposite side
                        put4(a.words + (long long)nbr[side] * 8 * a.side + slot_off + (side ^ 1) * a.side + (side < 2 ? wy : wz), w,
                             tag);
            }
        }
        if (more) {
#pragma unroll
            for (int h = 0; h < kHalo; h += 2) {
                u64 w0[4] = {0ull, 0ull, 0ull, 0ull}, w1[4] = {0ull, 0ull, 0ull, 0ull};
                bool m0 = hword[h] >= 0 && !failed, m1 = hword[h + 1] >= 0 && !failed;
                int polls = 0;
                while (m0 || m1) {
                    if (m0) get4(mine + slot_off + hword[h], w0);
                    if (m1) get4(mine + slot_off + hword[h + 1], w1);
                    auto here = [&](const u64 (&w)[4]) {
                        return (unsigned)(w[0] >> 32) == tag && (unsigned)(w[1] >> 32) == tag && (unsigned)(w[2] >> 32) == tag &&
                               (unsigned)(w[3] >> 32) == tag;
                    };
                    auto place = [&](const u64 (&w)[4], int o) {
                        *reinterpret_cast<float4*>(out + o) =
                            make_float4(__uint_as_float((unsigned)w[0]), __uint_as_float((unsigned)w[1]),
                                        __uint_as_float((unsigned)w[2]), __uint_as_float((unsigned)w[3]));
                    };
                    if (m0 && here(w0)) {
                        place(w0, hoff[h]);
                        m0 = false;
                    }
                    if (m1 && here(w1)) {
                        place(w1, hoff[h + 1]);
                        m1 = false;
                    }
                    if ((m0 || m1) && (!(++polls & 1023) || polls >= a.polls)) {
                        if (polls >= a.polls) {
                            *(volatile unsigned*)(a.count + kBandStop) = 1u;
                            *(volatile double*)a.err = (double)CMCG_ERR_DEVICE_TIMEOUT;
                        }
                        if (*(volatile unsigned*)(a.count + kBandStop)) {
                            failed = true;
                            break;
                        }
                    }
                }
            }
        }
        failed = __syncthreads_or(failed) != 0;
        if (failed) return;
    }
    float* gc = (a.nsteps & 1) ? a.buf1 : a.buf0;
    float* gp = (a.nsteps & 1) ? a.buf0 : a.buf1;
    const float* in = buf + (a.nsteps & 1) * bufsz;
#pragma unroll
    for (int q = 0; q < NPC; ++q) {
        if (!(fl[q] & kHere)) continue;
        const int o = (int)(crd[q] & 8191u) << 2, lz = (int)(crd[q] >> 13) & 255, ly = (int)(crd[q] >> 21);
        const int x0 = o - (lz + 1) * Z - (ly + 1) * Y - 4;
        const long long j = (long long)sx * (y0 + ly + (long long)g.sy * (z0 + lz)) + x0;
        float pv[4];
        unpack(prev[q].a, pv[0], pv[1]);
        unpack(prev[q].b, pv[2], pv[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (x0 + e < sx) {
                gc[j + e] = in[o + e];
                gp[j + e] = pv[e];
            }
    }
    if (tid == 0) a.count[blk] = base + (unsigned)a.nsteps;
}

template <int NPC, int SRC>
cudaError_t block_go(const BlockArgs& a, const BlockPlan& p, cudaStream_t st) {
    auto kernel = k_block3<NPC, SRC>;
    // (always the same value: threads with other plans set it too, between this call and the launch)
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax3);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.ny_blocks * p.nz_blocks));
    cfg.blockDim = dim3(kBT);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

template <int SRC>
cudaError_t block_npc(const BlockArgs& a, const BlockPlan& p, cudaStream_t st) {
    if (p.npc <= 1) return block_go<1, SRC>(a, p, st);
    if (p.npc <= 2) return block_go<2, SRC>(a, p, st);
    if (p.npc <= 4) return block_go<4, SRC>(a, p, st);
    return block_go<8, SRC>(a, p, st);
}

}  // namespace

// Blocks of ty by tz rows: the split along y and z, of at most one block per SM and at least two
// rows each way (a block holds the row that its mirror row repeats), whose fullest block has the
// least chunks to update and, at two thirds of the weight, to receive.
bool block_plan(const Geom& g, int sms, BlockPlan* p) {
    *p = BlockPlan();
    if (g.dim != 3 || g.nx < 4) return false;
    const long long cx = (g.sx + 3) / 4, P = 4 * cx + 8;
    const int most = std::min(sms, kMaxBlocks3);
    double best = 1e30;
    for (int by = 1; by <= std::min(most, g.sy / 2); ++by) {
        const int bz = std::min(most / by, g.sz / 2);
        if (bz < 1) continue;
        const long long ry = (g.sy + by - 1) / by, rz = (g.sz + bz - 1) / bz;
        const long long halo = (by > 1 ? 2 * rz : 0) + (bz > 1 ? 2 * ry : 0);
        if (ry > 255 || rz > 255 || ry * rz > 512 || ry * rz * cx > 8 * kBT || halo * cx > kHalo * kBT) continue;
        const long long bytes = 8 * P * (ry + 2) * (rz + 2);
        // faces: the two ends of every row, and whole rows of the outer blocks' faces
        const long long slots = 2 * ry * rz + cx * ((by > 1 ? 1 : 2) * rz + (bz > 1 ? 1 : 2) * ry);
        const long long smem = bytes + slots * (long long)sizeof(Face);
        if (smem > kSmemMax3 || slots >= (1 << 14) - 1) continue;
        const double cost = (double)(ry * rz * cx) + 0.67 * (double)(halo * cx);
        if (cost >= best) continue;
        best = cost;
        p->ny_blocks = by;
        p->nz_blocks = bz;
        p->npc = (int)((ry * rz * cx + kBT - 1) / kBT);
        p->side = (int)(P * std::max(ry, rz));
        p->smem = (size_t)smem;
        p->words = (size_t)8 * p->side * by * bz;
    }
    return p->ny_blocks > 0;
}

cudaError_t launch_step_block(const Geom& g, const BlockPlan& p, float* cur, float* prev, const float* kap, const float* S,
                              const unsigned char* sflag, bool src_faces, unsigned long long* words, unsigned* count,
                              double* err, int polls, int nsteps, const double* cs, const double* sn, bool adj_first,
                              bool adj_last, cudaStream_t st) {
    BlockArgs a;
    a.polls = polls;
    a.buf0 = cur;
    a.buf1 = prev;
    a.kap = kap;
    a.S = S;
    a.sflag = sflag;
    a.words = words;
    a.count = count;
    a.err = err;
    a.g = g;
    a.ny_blocks = p.ny_blocks;
    a.ty = g.sy / p.ny_blocks;
    a.ey = g.sy % p.ny_blocks;
    a.tz = g.sz / p.nz_blocks;
    a.ez = g.sz % p.nz_blocks;
    a.side = p.side;
    a.nsteps = nsteps;
    a.adj_first = adj_first;
    a.adj_last = adj_last;
    for (int s = 0; s < nsteps && S; ++s) {
        a.cs[s] = (float)cs[s];
        a.sn[s] = (float)sn[s];
    }
    const cudaError_t e = !S ? block_npc<0>(a, p, st) : (src_faces ? block_npc<1>(a, p, st) : block_npc<2>(a, p, st));
    if (e == cudaSuccess) note_launch(1);
    return e;
}

CMCG_CHECK_TU(block)

}  // namespace cmcg
