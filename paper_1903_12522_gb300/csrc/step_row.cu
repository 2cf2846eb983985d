// FP32 3D leapfrog steps (7- and 13-point) on rows padded to whole float4s.
//
// With rows of n + 1 floats a row starts anywhere within a 16-byte word, so the z-pair kernels of
// wave.cu move 4 bytes per access and spend 67 instructions per node and warp.  Here the two wave
// fields and kappa have a row pitch that is a multiple of four; a thread owns four consecutive
// nodes of a row and marches z.  Per four nodes: five 16-byte loads (y^n above, the two y
// neighbours, y^{n-1}, kappa; 13-point: seven), one store, the x neighbours by shuffles, and the
// arithmetic in packed pairs (f32x2).
//
// The endpoint kernels keep the flat layout: the first step of a loop reads it and writes both
// fields padded, the last one reads padded and writes flat, so that the conversion costs two
// extra stores per node and period, not extra passes.
//
// Bound: HBM at 257^3 (16 B per update; the two wave fields and kappa are 204 MB, more than L2):
// 44 us a step, 6.1 TB/s of algorithmic bytes, against 57 us for the z-pair kernel; at 193^3,
// where they fit L2, 18.5 against 22.5 us.  13-point, whole backward periods per step: 68 against
// 85 us.  Successive steps run their blocks in opposite orders: a step starts on the planes that
// the previous one touched last, which are still in L2 (47.4 us in one order).  Ten blocks of 128
// threads per SM and one plane's loads at a time beat two planes at a time (49 us, 80 registers)
// and loads one plane ahead (50 us).
//
// The roundings are those of k_step3d7_z2 / k_step3d13_z2, written out: same bits.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace cmcg {

namespace {

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
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

struct V4 {  // four floats as two packed pairs
    u64 a, b;
};
__device__ __forceinline__ V4 load4(const float* p) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    return V4{t.x, t.y};
}
__device__ __forceinline__ void store4(float* p, V4 v) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.a, v.b); }

constexpr int kRT = 128;

// FLAT: the fields' layout: 0 both padded, 1 cur and prev flat in, both padded out (pout receives
// y^{n+1}, pcopy y^n), 2 padded in, flat out (likewise).
template <int ORDER, int FLAGS, bool SRC_FACES, int FLAT>
__global__ void __launch_bounds__(kRT, ORDER == 2 ? 10 : 7)
    k_step_row(const float* __restrict__ cur, const float* prev, float* pout, float* pcopy,  // pout may be prev
               const float* __restrict__ kap, const float* __restrict__ S, float cs, float sn,
               Geom g, int px, int zc, int reverse, const unsigned char* __restrict__ sflag) {
    const int cx = px >> 2, plane4 = cx * g.sy;
    const int bx = reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int by = reverse ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    const int p = bx * kRT + (int)threadIdx.x;
    const int z0 = by * zc, z1 = min(z0 + zc, g.sz);
    if (!CMCG_RANGE_OK(z0, z1 - 1, g.sz, kSiteRow)) return;  // uniform over the block
    bool valid = p < plane4;
    int pp = valid ? p : plane4 - 1;  // (idle lanes take part in the shuffles)
    int iy = (int)((unsigned)pp / (unsigned)cx), ic = pp - iy * cx;
    if (!chunk_in_range(g, 4 * ic, iy, z0, z1, ORDER / 2, kSiteRow)) {
        valid = false;
        pp = iy = ic = 0;
    }
    const int x0 = 4 * ic;
    const int lane = (int)threadIdx.x & 31;
    const bool first = ic == 0;
    const int xe = g.nx - x0;  // element of the node x = nx (0 .. 3 in a row's last chunk)
    const int m = min(4, g.sx - x0);
    const int fsZ = g.sx * g.sy, psZ = px * g.sy;                  // plane strides: flat, padded
    const int isY = FLAT == 1 ? g.sx : px, isZ = FLAT == 1 ? fsZ : psZ;  // of the fields read
    int ji = FLAT == 1 ? x0 + g.sx * iy + fsZ * z0 : 4 * pp + psZ * z0;  // this thread's nodes in them
    int jp = 4 * pp + psZ * z0;                                    // in a padded field
    int jf = x0 + g.sx * iy + fsZ * z0;                            // in a flat one
    const int oym = (int)off_m1(iy, isY), oyp = (int)off_p1(iy, g.ny, isY);
    const int oym2 = ORDER == 4 ? (int)off_m2(iy, isY) : 0, oyp2 = ORDER == 4 ? (int)off_p2(iy, g.ny, isY) : 0;
    // lanes 0 and 31 load the x neighbours that the shuffles do not bring (not past a row's ends)
    const bool needl = lane == 0 && !first, needr = lane == 31 && xe >= 4;
    const int nby = (iy == 0 ? (int)((g.abc >> 2) & 1u) : 0) + (iy == g.ny ? (int)((g.abc >> 3) & 1u) : 0);
    const int nbl = first ? (int)(g.abc & 1u) : 0, nbr = xe < 4 ? (int)((g.abc >> 1) & 1u) : 0;
    bool vol = false;  // a source in one of the four columns in these four planes
    auto get = [&](const float* f, int j) -> V4 {
        if constexpr (FLAT != 1) {
            return load4(f + j);
        } else {
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = f[j + (e < m ? e : 0)];
            return V4{pack(v[0], v[1]), pack(v[2], v[3])};
        }
    };
    auto put = [&](float* f, V4 v) {
        if (FLAT != 2) {
            store4(f + jp, v);
        } else {
            float o[4];
            unpack(v.a, o[0], o[1]);
            unpack(v.b, o[2], o[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e < m) f[jf + e] = o[e];
        }
    };
    // the z neighbours carried from plane to plane
    V4 c = get(cur, ji), zm = get(cur, ji + (int)off_m1(z0, isZ)), zm2{}, zp{};
    if (ORDER == 4) {
        zm2 = get(cur, ji + (int)off_m2(z0, isZ));
        zp = get(cur, ji + (int)off_p1(z0, g.nz, isZ));
    }
    for (int iz = z0; iz < z1; ++iz) {
        if ((FLAGS & kStepSrc) && !SRC_FACES && (iz == z0 || (iz & 3) == 0)) vol = sflag[(iz >> 2) * plane4 + pp] != 0;
        V4 zp2{};
        if (ORDER == 2) zp = get(cur, ji + (int)off_p1(iz, g.nz, isZ));
        else zp2 = get(cur, ji + (int)off_p2(iz, g.nz, isZ));
        const V4 ym = get(cur, ji + oym), yp = get(cur, ji + oyp);
        V4 ym2{}, yp2{};
        if (ORDER == 4) {
            ym2 = get(cur, ji + oym2);
            yp2 = get(cur, ji + oyp2);
        }
        const V4 k = load4(kap + jp), q = get(prev, ji);
        float el = 0.f, er = 0.f, el2 = 0.f, er2 = 0.f;
        if (needl) {
            el = cur[ji - 1];
            if (ORDER == 4) el2 = cur[ji - 2];
        }
        if (needr) {
            er = cur[ji + 4];
            if (ORDER == 4) er2 = xe >= 5 ? cur[ji + 5] : 0.f;
        }
        float v[4];
        unpack(c.a, v[0], v[1]);
        unpack(c.b, v[2], v[3]);
        float xl = __shfl_up_sync(0xffffffffu, v[3], 1), xr = __shfl_down_sync(0xffffffffu, v[0], 1);
        if (lane == 0) xl = el;
        if (lane == 31) xr = er;
        if (first) xl = v[1];
        const float xm[4] = {xl, v[0], v[1], v[2]}, xq[4] = {v[1], v[2], v[3], xr};
        float sx1[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) sx1[e] = xm[e] + (e == xe ? xm[e] : xq[e]);
        u64 ra, rb;  // 2 y - kappa Lt(y)
        {
            const u64 A = add2(add2(pack(sx1[0], sx1[1]), add2(ym.a, yp.a)), add2(zm.a, zp.a));
            const u64 B = add2(add2(pack(sx1[2], sx1[3]), add2(ym.b, yp.b)), add2(zm.b, zp.b));
            u64 La, Lb;  // -Lt(y)
            if (ORDER == 2) {
                const u64 m6 = pack(-6.f, -6.f);
                La = fma2(m6, c.a, A);
                Lb = fma2(m6, c.b, B);
            } else {
                float xl2 = __shfl_up_sync(0xffffffffu, v[2], 1), xr2 = __shfl_down_sync(0xffffffffu, v[1], 1);
                if (lane == 0) xl2 = el2;
                if (lane == 31) xr2 = er2;
                // two nodes to the left of x = 0, 1 and to the right of x = nx - 1, nx: mirrored
                const float a2[4] = {first ? v[2] : xl2, first ? v[1] : xl, v[0], v[1]};
                const float b2[4] = {v[2], v[3], xr, xr2};
                float sx2[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) sx2[e] = a2[e] + (e == xe ? a2[e] : (e + 1 == xe ? v[e] : b2[e]));
                const u64 C = add2(add2(pack(sx2[0], sx2[1]), add2(ym2.a, yp2.a)), add2(zm2.a, zp2.a));
                const u64 D = add2(add2(pack(sx2[2], sx2[3]), add2(ym2.b, yp2.b)), add2(zm2.b, zp2.b));
                const u64 c1 = pack(4.f / 3.f, 4.f / 3.f), c2 = pack(-1.f / 12.f, -1.f / 12.f), d = pack(-7.5f, -7.5f);
                La = fma2(c2, C, fma2(d, c.a, mul2(c1, A)));
                Lb = fma2(c2, D, fma2(d, c.b, mul2(c1, B)));
            }
            ra = fma2(k.a, La, add2(c.a, c.a));
            rb = fma2(k.b, Lb, add2(c.b, c.b));
        }
        const int nbz = (iz == 0 ? (int)((g.abc >> 4) & 1u) : 0) + (iz == g.nz ? (int)((g.abc >> 5) & 1u) : 0);
        if ((FLAGS & kStepSrc) && !SRC_FACES && vol) {
            float t[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 s = reinterpret_cast<const float2*>(S)[jf + (e < m ? e : 0)];
                t[e] = __fmaf_rn(s.x, cs, __fmul_rn(s.y, sn));
            }
            ra = add2(ra, pack(t[0], t[1]));
            rb = add2(rb, pack(t[2], t[3]));
        }
        const u64 m1 = pack(-1.f, -1.f);
        V4 o{fma2(m1, q.a, ra), fma2(m1, q.b, rb)};
        if (nby | nbl | nbr | nbz) {
            float w[4], r[4], kk[4], qq[4];
            unpack(o.a, w[0], w[1]);
            unpack(o.b, w[2], w[3]);
            unpack(ra, r[0], r[1]);
            unpack(rb, r[2], r[3]);
            unpack(k.a, kk[0], kk[1]);
            unpack(k.b, kk[2], kk[3]);
            unpack(q.a, qq[0], qq[1]);
            unpack(q.b, qq[2], qq[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int nb = nby + nbz + (e == 0 ? nbl : 0) + (e == xe ? nbr : 0);
                if (nb && e < m) {
                    float h = r[e];
                    if ((FLAGS & kStepSrc) && SRC_FACES) {
                        const float2 s = reinterpret_cast<const float2*>(S)[jf + e];
                        h += __fmaf_rn(s.x, cs, __fmul_rn(s.y, sn));
                    }
                    const float beta = (float)nb * sqrtf(kk[e]);
                    const float b1 = 1.f - beta;
                    // (without the division the product is rounded before the difference)
                    const float u = (FLAGS & kStepPrevScaled) ? h - qq[e]
                                    : (FLAGS & kStepNoDiv)    ? __fsub_rn(h, __fmul_rn(b1, qq[e]))
                                                              : __fmaf_rn(-b1, qq[e], h);
                    w[e] = (FLAGS & kStepNoDiv) ? u : u / (1.f + beta);
                }
            }
            o.a = pack(w[0], w[1]);
            o.b = pack(w[2], w[3]);
        }
        if (valid) {
            put(pout, o);
            if (FLAT != 0) put(pcopy, c);
        }
        if (ORDER == 2) {
            zm = c;
            c = zp;
        } else {
            zm2 = zm;
            zm = c;
            c = zp;
            zp = zp2;
        }
        ji += isZ;
        jp += psZ;
        jf += fsZ;
    }
}

__global__ void k_row_pad(Geom g, int px, const float* __restrict__ a, float* __restrict__ b) {
    const long long n = (long long)px * g.sy * g.sz, stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        const long long r = j / px;
        const int x = (int)(j - r * px);
        b[j] = x < g.sx ? a[r * g.sx + x] : 0.f;
    }
}

template <int ORDER, int FLAGS, bool SRC_FACES>
void row_launch(const RowStep& a, cudaStream_t st) {
    const Geom& g = a.g;
    const int plane4 = (a.px >> 2) * g.sy;
    const unsigned bxy = (unsigned)((plane4 + kRT - 1) / kRT);
    // planes per thread: four where that makes at least four waves of blocks, else two (us a step of a
    // backward period with two and with four: 151^3 12.2 and 14.3, 193^3 21.7 and 21.6, 225^3 35.3 and 33.6,
    // 257^3 51.3 and 49.4; 13-point 129^3 12.0 and 14.0, 193^3 28.3 and 28.3, 257^3 66.4 and 62.5)
    const int per_sm = ORDER == 2 ? 10 : 7;
    const int zc = planes_per_thread((long long)bxy * ((g.sz + 3) / 4) >= 4ll * 152 * per_sm ? 4 : 2, g.sz);
    const dim3 grid(bxy, (unsigned)((g.sz + zc - 1) / zc));
    const float cs = (float)a.cs, sn = (float)a.sn;
    auto go = [&](auto kernel) {
        kernel<<<grid, kRT, 0, st>>>(a.cur, a.prev, a.out, a.copy, a.kap, a.S, cs, sn, g, a.px, zc, a.reverse, a.sflag);
    };
    if (a.flat == 0) go(k_step_row<ORDER, FLAGS, SRC_FACES, 0>);
    else if (a.flat == 1) go(k_step_row<ORDER, FLAGS, SRC_FACES, 1>);
    else go(k_step_row<ORDER, FLAGS, SRC_FACES, 2>);
}

template <int ORDER>
void row_flags(const RowStep& a, cudaStream_t st) {
    switch (a.flags) {
        case kStepSrc: a.src_faces ? row_launch<ORDER, kStepSrc, true>(a, st) : row_launch<ORDER, kStepSrc, false>(a, st); break;
        case kStepPrevScaled: row_launch<ORDER, kStepPrevScaled, false>(a, st); break;
        case kStepNoDiv: row_launch<ORDER, kStepNoDiv, false>(a, st); break;
        default: row_launch<ORDER, 0, false>(a, st); break;
    }
}

}  // namespace

int row_pitch(const Geom& g) { return (g.sx + 3) & ~3; }

bool row_fits(const Geom& g) {
    // 32-bit indices; a row of one or two chunks would waste most of a warp's accesses on padding
    return g.dim == 3 && g.nx >= 8 && (long long)row_pitch(g) * g.sy * g.sz < (1ll << 30);
}

void launch_row_pad(const Geom& g, const float* flat, float* padded, cudaStream_t st) {
    note_launch(1);
    k_row_pad<<<152 * 8, 256, 0, st>>>(g, row_pitch(g), flat, padded);
}

void launch_step_row(const RowStep& a, int order, cudaStream_t st) {
    note_launch(1);
    if (order == 2) row_flags<2>(a, st);
    else row_flags<4>(a, st);
}

CMCG_CHECK_TU(row)

}  // namespace cmcg
