// 2D leapfrog step loops in one launch: a persistent kernel that keeps the whole problem on chip.
//
// A 2D step of a grid up to about 1100^2 moves a few megabytes that stay in L2 and is over in two
// microseconds; launched one by one, steps come 6 to 10 microseconds apart (host launch rate and
// kernel-to-kernel latency).  Here one CTA per SM owns a band of grid rows for the whole loop:
// y^n sits in shared memory (two buffers), y^{n-1} and kappa in registers, the source in shared
// memory, and the CTAs exchange only the outermost rows of their bands.
//
// The exchange carries its own flags: a row element travels as one 8-byte word, 32 data bits and
// the 32-bit number of the step it belongs to (a double as two such words).  Eight-byte accesses
// are single, so a reader that sees the step number has the data; there is no fence, no separate
// flag and no grid barrier, and a CTA waits for its two neighbours only.  A band's boundary
// rows are computed and sent first and the first look at the neighbours' words is taken before
// the rest of the band, so that their flight overlaps it.  Words of step s and s + 1 use
// different slots; a slot is overwritten two steps later, which needs the neighbour's rows of
// the step in between, which it computes after it has read the slot.
//
// Up to 16 bands run as one thread-block cluster and write the words straight into the
// neighbour's shared memory; more bands exchange through global memory (L2) in a cooperative
// launch.  In global memory the step numbers run on from launch to launch (each CTA has a count of
// its own; all counts are equal between launches), so no slot has to be cleared, and loops of
// different precision, whose bands and words lie differently, can share them.
//
// Bound: one trip of the exchange (DSMEM or L2) and, in bands of more than a few rows, shared-memory
// reads.  Microseconds per step (slope over the step count; in brackets step by step): FP32 129^2
// 0.93 (5.9), 513^2 1.5 (6), 1025^2 2.3 (9), with a source in the volume 3.1; FP64 437x302 3.0 (7).
//
// Every wait is bounded: on time-out a CTA reports CMCG_ERR_DEVICE_TIMEOUT through *err (host
// memory), sets the stop word that every waiting CTA looks at, and returns.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "soft64.cuh"

namespace cmcg {

namespace {

constexpr int kMaxBands = kBandStop;   // one CTA per SM of a GB300
constexpr int kSmemMax = 227 * 1024;   // shared memory a CTA can have

template <typename T>
constexpr int kBandThreads = std::is_same<T, float>::value ? 1024 : 512;  // FP64 needs the registers

template <typename T>
struct BandArgs {
    T* buf0;  // y^n of the first step; the second buffer y^{n-1}; they swap roles every step
    T* buf1;
    const T* kap;
    const T* S;           // source (complex interleaved), or null
    const double* wface;  // FP64: 1 / (1 + beta)
    unsigned long long* words;
    unsigned* count;      // kMaxBands times: steps done in all launches so far; [kMaxBands]: stop word
    double* err;
    Geom g;
    int rows, extra;      // bands 0 .. extra - 1 own rows + 1 grid rows, the others rows
    int nsteps;
    int face_slots;       // shared-memory slots of face factors
    int adj_first, adj_last;  // step 0 is the adjoint's first, step nsteps - 1 its last
    int polls;            // the longest wait
    T cs[kBandSteps], sn[kBandSteps];
};

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// The exchange of one band: received words live at [slot][from][n], from = 0 the band before
// (its last rows), 1 the band after (its first rows), n words each, in this CTA's shared memory
// (CL) or at its place in global memory.
template <bool CL>
struct Exchange {
    unsigned long long* words;  // of band 0
    unsigned sm;                // CL: shared address of this CTA's words
    int band, n;
    unsigned* stop;
    double* err;
    int limit;  // polls of the longest wait
    __device__ __forceinline__ long long at(unsigned tag, int from) const { return (long long)((tag & 1u) * 2 + from) * n; }
    // where band `to` looks for words of this step that come from side `from`
    __device__ __forceinline__ unsigned long long* global_of(int to, unsigned tag, int from) const {
        return words + (long long)to * 4 * n + at(tag, from);
    }
    __device__ __forceinline__ unsigned remote_of(int to, unsigned tag, int from) const {
        unsigned r;
        const unsigned local = sm + 8u * (unsigned)at(tag, from);
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(to));
        return r;
    }
    // side 0: this band's first rows, to the band before; side 1: its last rows, to the band after
    __device__ __forceinline__ void put(int side, int i, unsigned data, unsigned tag) const {
        const unsigned long long w = ((unsigned long long)tag << 32) | data;
        const int to = side ? band + 1 : band - 1, from = side ? 0 : 1;
        if (CL) {
            const unsigned p = remote_of(to, tag, from) + 8u * i;
            asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(p), "l"(w) : "memory");
        } else {
            unsigned long long* p = global_of(to, tag, from) + i;
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
        }
    }
    // four elements at word 4 i (16-byte aligned: two 8-byte words per store, each valid by itself)
    __device__ __forceinline__ void put4(int side, int i, float4 v, unsigned tag) const {
        const unsigned long long t = (unsigned long long)tag << 32;
        const unsigned long long w0 = t | __float_as_uint(v.x), w1 = t | __float_as_uint(v.y),
                                 w2 = t | __float_as_uint(v.z), w3 = t | __float_as_uint(v.w);
        const int to = side ? band + 1 : band - 1, from = side ? 0 : 1;
        if (CL) {
            const unsigned p = remote_of(to, tag, from) + 32u * i;
            asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(p), "l"(w0), "l"(w1) : "memory");
            asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(p + 16), "l"(w2), "l"(w3)
                         : "memory");
        } else {
            unsigned long long* p = global_of(to, tag, from) + 4 * i;
            asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
            asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p + 2), "l"(w2), "l"(w3) : "memory");
        }
    }
    __device__ __forceinline__ unsigned long long get(int from, int i, unsigned tag) const {
        unsigned long long w;
        if (CL) {
            const unsigned p = sm + 8u * ((unsigned)at(tag, from) + i);
            asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w) : "r"(p) : "memory");
        } else {
            const unsigned long long* p = global_of(band, tag, from) + i;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
        }
        return w;
    }
    __device__ __forceinline__ void get4(int from, int i, unsigned tag, unsigned long long (&w)[4]) const {
        if (CL) {
            const unsigned p = sm + 8u * ((unsigned)at(tag, from) + 4 * i);
            asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "r"(p) : "memory");
            asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];"
                         : "=l"(w[2]), "=l"(w[3])
                         : "r"(p + 16)
                         : "memory");
        } else {
            const unsigned long long* p = global_of(band, tag, from) + 4 * i;
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(p) : "memory");
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[2]), "=l"(w[3]) : "l"(p + 2) : "memory");
        }
    }
    // after an unsuccessful poll: true to give up
    __device__ __forceinline__ bool give_up(int& polls) const {
        if ((++polls & 1023) && polls < limit) return false;
        if (polls >= limit) {
            *(volatile unsigned*)stop = 1u;
            *(volatile double*)err = (double)CMCG_ERR_DEVICE_TIMEOUT;
        }
        return *(volatile unsigned*)stop != 0u;
    }
};

// Zeroes a CTA's word area (CL) and meets the cluster, so that no word arrives before it.
template <bool CL>
__device__ __forceinline__ void open_exchange(unsigned long long* sm_words, int count) {
    if (CL) {
        for (int i = (int)threadIdx.x; i < count; i += (int)blockDim.x) sm_words[i] = 0ull;
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// No CTA of a cluster leaves while another may still write into its shared memory (each gets here:
// every wait on the way is bounded).
template <bool CL>
__device__ __forceinline__ void close_exchange() {
    if (CL) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __noinline__ double plain_lap2(double c, double xm, double xp, double ym, double yp) {
    return ((xm + xp) + (ym + yp)) - 4.0 * c;
}
__device__ __noinline__ double plain_lap4(double c, double a1, double a2) {
    return (4.0 / 3.0) * a1 - (1.0 / 12.0) * a2 - 5.0 * c;
}
__device__ __noinline__ float plain_div(float v, float d) { return v / d; }

// v / d, correctly rounded, with r = 1 / d correctly rounded and computed once: a quotient estimate
// and one correction by its exact remainder (Markstein 1990, IBM J. Res. Dev. 34(1)).  Small and
// huge v, where the remainder may not be exact, take the division.
__device__ __forceinline__ float div_known(float v, float d, float r) {
    const float q0 = __fmul_rn(v, r);
    const float q = __fmaf_rn(__fmaf_rn(-q0, d, v), r, q0);
    const unsigned a = __float_as_uint(v) & 0x7fffffffu;
    if (a - 0x0d800000u < 0x6e000000u || a == 0u) return q;  // 2^-100 <= |v| < 2^120, or 0
    return plain_div(v, d);
}

// What an absorbing face's node needs besides kappa: FP32 1 - beta, 1 + beta and its reciprocal;
// FP64 w = 1 / (1 + beta).  sr, si: its source (SRC == 1).  Worked out once per launch: a square
// root and a division per step would be most of a small band's step.
template <typename T>
struct FaceNode;
template <>
struct FaceNode<float> {
    float c1, d, r, sr, si;
    __device__ __forceinline__ void set(int nb, float k, const double*) {
        const float beta = (float)nb * sqrtf(k);
        c1 = 1.f - beta;
        d = 1.f + beta;
        r = __frcp_rn(d);
    }
};
template <>
struct FaceNode<double> {
    double w, sr, si;
    __device__ __forceinline__ void set(int, double, const double* wf) { w = *wf; }
};

// The face's part of an update.  The FP32 roundings are those of k_step: without the division
// (the adjoint's last step) its product is not fused.
__device__ __forceinline__ float face_out(float rhs, float yq, const FaceNode<float>& f, int flags) {
    const float v = (flags & kStepPrevScaled) ? rhs - yq
                    : (flags & kStepNoDiv)    ? rhs - __fmul_rn(f.c1, yq)
                                              : __fmaf_rn(-f.c1, yq, rhs);
    return (flags & kStepNoDiv) ? v : div_known(v, f.d, f.r);
}
__device__ __noinline__ double face_out(double rhs, double yq, const FaceNode<double>& f, int flags) {
    const double w = f.w;
    if (flags & kStepNoDiv) return rhs - ((flags & kStepPrevScaled) ? yq : (2.0 - 1.0 / w) * yq);
    if (flags & kStepPrevScaled) return (rhs - yq) * w;
    return fma(rhs, w, -(fma(2.0, w, -1.0) * yq));
}
// the source term as the step kernels round it
__device__ __forceinline__ float source_term(float sr, float si, float cs, float sn) {
    return __fmaf_rn(sr, cs, __fmul_rn(si, sn));
}
__device__ __forceinline__ double source_term(double sr, double si, double cs, double sn) {
    return fma(sr, cs, si * sn);
}

// -Lt(y) in FP32 or FP64 at one node; in points at y^n there, P = row pitch.
template <int R>
__device__ __forceinline__ double band_lap(const double* in, int P) {
    using soft64::align;
    using soft64::term;
    const double c = in[0], xm = in[-1], xp = in[1], ym = in[-P], yp = in[P];
    const soft64::Term tc = term(c), a = term(xm), b = term(xp), d = term(ym), e = term(yp);
    unsigned m = soft64::max3(soft64::max3(tc.e, a.e, b.e), d.e, e.e);
    double L;
    bool ok;
    if (R == 1) {
        const long long C = align(tc, m);
        L = soft64::to_double((align(a, m) + align(b, m)) + (align(d, m) + align(e, m)) - 4 * C, m, &ok);
        if (!(ok && soft64::in_range(m))) L = plain_lap2(c, xm, xp, ym, yp);
    } else {
        const double x2 = in[-2], x3 = in[2], y2 = in[-2 * P], y3 = in[2 * P];
        const soft64::Term p = term(x2), q = term(x3), t = term(y2), u = term(y3);
        m = soft64::max3(soft64::max3(m, p.e, q.e), t.e, u.e);
        const long long C = align(tc, m);
        const long long s1 = (align(a, m) + align(b, m)) + (align(d, m) + align(e, m));
        const long long s2 = (align(p, m) + align(q, m)) + (align(t, m) + align(u, m));
        L = soft64::four_thirds(s1 - (s2 >> 4) - (4 * C - (C >> 2)), m, &ok);
        if (!(ok && soft64::in_range(m))) L = plain_lap4(c, (xm + xp) + (ym + yp), (x2 + x3) + (y2 + y3));
    }
    return L;
}
// 2 y - kappa Lt(y), the FP32 expressions in k_step's order: same bits.
template <int R>
__device__ __forceinline__ float rhs_of(const float* in, int P, float k) {
    const float c = in[0];
    float L;
    if (R == 1) {
        float acc = in[-1] + in[1];
        acc += in[-P] + in[P];
        L = 4.f * c - acc;
    } else {
        const float c1 = 4.f / 3.f, c2 = 1.f / 12.f;
        float a1 = in[-1] + in[1];
        float a2 = in[-2] + in[2];
        a1 += in[-P] + in[P];
        a2 += in[-2 * P] + in[2 * P];
        const float diag = 5.f * c;
        L = diag - c1 * a1 + c2 * a2;
    }
    return 2.f * c - k * L;
}

// One node's update; face: its factors on an absorbing face, else null.
template <int R, bool VOLUME>
__device__ __forceinline__ float update(const float* in, int P, float k, float yq, const FaceNode<float>* face, bool src,
                                        int flags, float sr, float si, float cs, float sn) {
    float rhs = rhs_of<R>(in, P, k);
    if (VOLUME) rhs += source_term(sr, si, cs, sn);
    if (!face) return rhs - yq;
    const FaceNode<float> f = *face;
    if (!VOLUME && src) rhs += source_term(f.sr, f.si, cs, sn);
    return face_out(rhs, yq, f, flags);
}
template <int R, bool VOLUME>
__device__ __forceinline__ double update(const double* in, int P, double k, double yq, const FaceNode<double>* face,
                                         bool src, int flags, double sr, double si, double cs, double sn) {
    const double L = band_lap<R>(in, P), c = in[0];
    if (!face) {
        double out = fma(2.0, c, -yq);
        if (VOLUME) out = fma(sr, cs, fma(si, sn, out));
        return fma(k, L, out);
    }
    double rhs = fma(k, L, 2.0 * c);
    if (VOLUME) rhs += source_term(sr, si, cs, sn);
    else if (src) rhs += source_term(face->sr, face->si, cs, sn);
    return face_out(rhs, yq, *face, flags);
}

// A band's face nodes (or chunks) are numbered: left and right face of each row, then the first
// and the last grid row.
__device__ __forceinline__ int face_slot(int lr, int rows, bool right, bool row_face, bool second, int i, int per_row) {
    return row_face ? 2 * rows + (second ? per_row : 0) + i : 2 * lr + (right ? 1 : 0);
}

// SRC: 0 none, 1 on absorbing faces only (read from global memory there), 2 everywhere.
// NPT: nodes per thread.  Thread t owns the band's nodes t, t + threads, ... counted from the
// band's last R rows on, so that the boundary rows come first.  Nodes beside a mirror face also
// write the ghost columns and rows that repeat them.
template <typename T, int R, int NPT, int SRC, bool CL>
__global__ void __launch_bounds__(kBandThreads<T>, 1) k_band(const __grid_constant__ BandArgs<T> a) {
    constexpr int BT = kBandThreads<T>;
    constexpr int kWords = (int)sizeof(T) / 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Geom& g = a.g;
    const int band = (int)blockIdx.x, nbands = (int)gridDim.x;
    const int tid = (int)threadIdx.x;
    const int r0 = band * a.rows + min(band, a.extra);
    const int rows = a.rows + (band < a.extra ? 1 : 0);
    const int sx = g.sx, P = sx + 2 * R;
    const int nn = rows * sx;
    const int bufsz = (a.rows + (a.extra ? 1 : 0) + 2 * R) * P;
    unsigned long long* const sm_words = reinterpret_cast<unsigned long long*>(smem_raw);
    const int side_words = R * sx * kWords;
    T* const buf = reinterpret_cast<T*>(sm_words + (CL ? 4 * side_words : 0));  // two buffers of bufsz
    FaceNode<T>* const faces = reinterpret_cast<FaceNode<T>*>(buf + 2 * bufsz);
    T* const ssrc = reinterpret_cast<T*>(faces + a.face_slots);
    const bool up = band > 0, down = band + 1 < nbands;  // is there a band before / after?
    const unsigned base = CL ? 0u : a.count[band];
    const Exchange<CL> ex{a.words, smem_addr(sm_words), band, side_words, a.count + kBandStop, a.err, a.polls};

    // the band and its halo rows of y^n; rows outside the grid hold their mirror rows
    for (int i = tid; i < (rows + 2 * R) * P; i += BT) {
        const int lr = i / P, lx = i - lr * P;
        int r = r0 - R + lr, x = lx - R;
        r = r < 0 ? -r : (r > g.ny ? 2 * g.ny - r : r);
        x = x < 0 ? -x : (x > g.nx ? 2 * g.nx - x : x);
        buf[i] = a.buf0[(long long)r * sx + x];
    }
    // per node: offset in a buffer, y^{n-1}, kappa, and bits: 0 it is next to a mirror face (its
    // value is also a ghost's), 1 / 2 it is in the first / last R rows and goes to the neighbour
    // band, 3 on it is on an absorbing face (slot + 1)
    T prev[NPT], kap[NPT];
    unsigned short off[NPT], fl[NPT];
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        const int i = tid + q * BT;
        off[q] = 0;
        fl[q] = 0;
        prev[q] = kap[q] = T(0);
        if (i < nn) {
            int f = i - R * sx;
            f += f < 0 ? nn : 0;
            const int lr = f / sx, x = f - lr * sx, r = r0 + lr;
            const long long j = (long long)r * sx + x;
            if (!CMCG_RANGE_OK(j, j, g.np, kSiteColumn)) continue;
            off[q] = (unsigned short)((lr + R) * P + x + R);
            prev[q] = a.buf1[j];
            kap[q] = a.kap[j];
            const bool ghost = (x >= 1 && x <= R) || (x >= g.nx - R && x < g.nx) || (r >= 1 && r <= R) ||
                               (r >= g.ny - R && r < g.ny);
            unsigned bits = (ghost ? 1u : 0u) | (up && lr < R ? 2u : 0u) | (down && lr >= rows - R ? 4u : 0u);
            const int nb = num_abc(g, x, r, 0);
            if (nb) {
                const bool yf = (r == 0 && (g.abc & 4u)) || (r == g.ny && (g.abc & 8u));
                const int slot = face_slot(lr, rows, x == g.nx, yf, r == g.ny && nbands == 1, x, sx);
                faces[slot].set(nb, kap[q], sizeof(T) == 8 ? a.wface + j : nullptr);
                if (SRC == 1) {
                    faces[slot].sr = a.S[2 * j];
                    faces[slot].si = a.S[2 * j + 1];
                }
                bits |= (unsigned)(slot + 1) << 3;
            }
            fl[q] = (unsigned short)bits;
            if (SRC == 2) {
                ssrc[2 * i] = a.S[2 * j];
                ssrc[2 * i + 1] = a.S[2 * j + 1];
            }
        }
    }
    open_exchange<CL>(sm_words, 4 * side_words);
    __syncthreads();

    const int n_up = up ? R * sx : 0, n_all = n_up + (down ? R * sx : 0);  // halo elements
    bool failed = false;
    for (int s = 0; s < a.nsteps; ++s) {
        const T* in = buf + (s & 1) * bufsz;
        T* out = buf + ((s + 1) & 1) * bufsz;
        int flags = 0;
        if (a.adj_first && s == 0) flags |= kStepPrevScaled;
        if (a.adj_last && s == a.nsteps - 1) flags |= kStepNoDiv;
        const T cs = SRC ? a.cs[s] : T(0), sn = SRC ? a.sn[s] : T(0);
        const bool more = s + 1 < a.nsteps;
        const unsigned tag = base + (unsigned)s + 1u;
#pragma unroll
        for (int q = 0; q < NPT; ++q) {
            const int i = tid + q * BT;
            if (i < nn) {
                const int o = off[q], f = fl[q];
                const T c = in[o];
                T sr = T(0), si = T(0);
                if (SRC == 2) {
                    sr = ssrc[2 * i];
                    si = ssrc[2 * i + 1];
                }
                const FaceNode<T>* face = f >> 3 ? faces + ((f >> 3) - 1) : nullptr;
                const T v = update<R, SRC == 2>(in + o, P, kap[q], prev[q], face, SRC == 1, flags, sr, si, cs, sn);
                prev[q] = c;
                out[o] = v;
                if (f & 7) {
                    const int lr = o / P - R, x = o - (lr + R) * P - R, r = r0 + lr;
                    if (f & 1) {
#pragma unroll
                        for (int d = 1; d <= R; ++d) {
                            if (x == d) out[o - 2 * d] = v;
                            if (x == g.nx - d) out[o + 2 * d] = v;
                            if (r == d) out[o - 2 * d * P] = v;
                            if (r == g.ny - d) out[o + 2 * d * P] = v;
                        }
                    }
                    if (more && (f & 6)) {
#pragma unroll
                        for (int side = 0; side < 2; ++side) {
                            if (!(f & (side ? 4 : 2))) continue;
                            const int e = ((side ? lr - (rows - R) : lr) * sx + x) * kWords;
                            if (sizeof(T) == 4) {
                                ex.put(side, e, __float_as_uint((float)v), tag);
                            } else {
                                ex.put(side, e, (unsigned)__double2loint((double)v), tag);
                                ex.put(side, e + 1, (unsigned)__double2hiint((double)v), tag);
                            }
                        }
                    }
                }
            }
        }
        if (more && n_all) {
            // halo rows: the last rows of the band before, the first rows of the band after
            for (int i0 = tid; i0 < n_all; i0 += 4 * BT) {
                unsigned long long w[4][kWords] = {};
                unsigned missing = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (i0 + q * BT < n_all) missing |= 1u << q;
                const unsigned mine = missing;
                int polls = 0;
                while (missing) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (!(missing & (1u << q))) continue;
                        const int i = i0 + q * BT;
                        const int from = i < n_up ? 0 : 1, e = (from ? i - n_up : i) * kWords;
#pragma unroll
                        for (int k = 0; k < kWords; ++k) w[q][k] = ex.get(from, e + k, tag);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        bool here = true;
#pragma unroll
                        for (int k = 0; k < kWords; ++k) here = here && (unsigned)(w[q][k] >> 32) == tag;
                        if ((missing & (1u << q)) && here) missing &= ~(1u << q);
                    }
                    if (missing && ex.give_up(polls)) {
                        failed = true;
                        break;
                    }
                }
                if (failed) break;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (!(mine & (1u << q))) continue;
                    const int i = i0 + q * BT;
                    const bool lo = i < n_up;
                    const int e = lo ? i : i - n_up;
                    const int d = e / sx, x = e - d * sx;
                    T v;
                    if (sizeof(T) == 4) v = (T)__uint_as_float((unsigned)w[q][0]);
                    else v = (T)__hiloint2double((int)(unsigned)w[q][kWords - 1], (int)(unsigned)w[q][0]);
                    out[((lo ? 0 : rows + R) + d) * P + x + R] = v;
                }
            }
        }
        failed = __syncthreads_or(failed) != 0;
        if (failed) break;
    }
    close_exchange<CL>();
    if (failed) return;
    // y^n and y^{n-1} back: after an odd number of steps the buffers have swapped roles
    T* gc = (a.nsteps & 1) ? a.buf1 : a.buf0;
    T* gp = (a.nsteps & 1) ? a.buf0 : a.buf1;
    const T* in = buf + (a.nsteps & 1) * bufsz;
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        const int i = tid + q * BT;
        if (i < nn) {
            int f = i - R * sx;
            f += f < 0 ? nn : 0;
            const long long j = (long long)r0 * sx + f;
            gc[j] = in[off[q]];
            gp[j] = prev[q];
        }
    }
    // (the counts past the last band too: a handle's next loop may have more bands)
    if (!CL && band + tid * nbands < kBandStop) a.count[band + tid * nbands] = base + (unsigned)a.nsteps;
}

// The FP32 2nd-order loop, four consecutive nodes of a row (one aligned float4 of shared memory)
// per thread and NPC such chunks: shared-memory reads and instructions per node are a third of
// k_band's.  Mirror columns are selected when they are read; the rows' pitch is padded to whole
// chunks, whose spare columns hold nothing that is used.
struct FaceChunk {  // FaceNode<float> of four nodes; 1, 1, 1 for those that are on no absorbing face
    float4 c1, d, r;
    float4 s01, s23;  // sources (SRC == 1), pairs
};

template <int SRC>
__device__ __forceinline__ float4 update4(const float* in, int P, float4 k4, float4 p4, bool first, int xe,
                                          const FaceChunk* face, int flags, float4 s01, float4 s23, float cs, float sn) {
    const float4 c = *reinterpret_cast<const float4*>(in);
    const float4 m = *reinterpret_cast<const float4*>(in - P), p = *reinterpret_cast<const float4*>(in + P);
    float xl = in[-1], xr = in[4];
    if (first) xl = c.y;
    const float cc[4] = {c.x, c.y, c.z, c.w};
    const float xm[4] = {xl, c.x, c.y, c.z}, xq[4] = {c.y, c.z, c.w, xr};
    const float ym[4] = {m.x, m.y, m.z, m.w}, yp[4] = {p.x, p.y, p.z, p.w};
    const float kk[4] = {k4.x, k4.y, k4.z, k4.w}, pp[4] = {p4.x, p4.y, p4.z, p4.w};
    float rhs[4], o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float xp = e == xe ? xm[e] : xq[e];
        float acc = xm[e] + xp;
        acc += ym[e] + yp[e];
        const float L = 4.f * cc[e] - acc;
        rhs[e] = 2.f * cc[e] - kk[e] * L;
    }
    if (SRC == 2) {
        const float sr[4] = {s01.x, s01.z, s23.x, s23.z}, si[4] = {s01.y, s01.w, s23.y, s23.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) rhs[e] += source_term(sr[e], si[e], cs, sn);
    }
    if (!face) {
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = rhs[e] - pp[e];
    } else {
        const FaceChunk f = *face;
        const float c1[4] = {f.c1.x, f.c1.y, f.c1.z, f.c1.w}, d[4] = {f.d.x, f.d.y, f.d.z, f.d.w};
        const float r[4] = {f.r.x, f.r.y, f.r.z, f.r.w};
        const float sr[4] = {f.s01.x, f.s01.z, f.s23.x, f.s23.z}, si[4] = {f.s01.y, f.s01.w, f.s23.y, f.s23.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float h = rhs[e];
            if (SRC == 1) h += source_term(sr[e], si[e], cs, sn);
            const FaceNode<float> fn{c1[e], d[e], r[e], 0.f, 0.f};
            o[e] = face_out(h, pp[e], fn, flags);
        }
    }
    return make_float4(o[0], o[1], o[2], o[3]);
}

template <int NPC, int SRC, bool CL>
__global__ void __launch_bounds__(kBandThreads<float>, 1) k_band4(const __grid_constant__ BandArgs<float> a) {
    constexpr int BT = kBandThreads<float>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Geom& g = a.g;
    const int band = (int)blockIdx.x, nbands = (int)gridDim.x;
    const int tid = (int)threadIdx.x;
    const int r0 = band * a.rows + min(band, a.extra);
    const int rows = a.rows + (band < a.extra ? 1 : 0);
    const int sx = g.sx, cx = (sx + 3) >> 2, P = 4 * cx + 8;  // node x at column x + 4
    const int nc = rows * cx;
    const int bufsz = (a.rows + (a.extra ? 1 : 0) + 2) * P;
    unsigned long long* const sm_words = reinterpret_cast<unsigned long long*>(smem_raw);
    const int side_words = 4 * cx;
    float* const buf = reinterpret_cast<float*>(sm_words + (CL ? 4 * side_words : 0));
    FaceChunk* const faces = reinterpret_cast<FaceChunk*>(buf + 2 * bufsz);
    float2* const ssrc = reinterpret_cast<float2*>(faces + a.face_slots);
    const bool up = band > 0, down = band + 1 < nbands;
    const unsigned base = CL ? 0u : a.count[band];
    const Exchange<CL> ex{a.words, smem_addr(sm_words), band, side_words, a.count + kBandStop, a.err, a.polls};

    for (int i = tid; i < (rows + 2) * P; i += BT) {
        const int lr = i / P, x = i - lr * P - 4;
        int r = r0 - 1 + lr;
        r = r < 0 ? -r : (r > g.ny ? 2 * g.ny - r : r);
        buf[i] = x >= 0 && x <= g.nx ? a.buf0[(long long)r * sx + x] : 0.f;
        buf[bufsz + i] = 0.f;
    }
    // per chunk: offset, y^{n-1}, kappa, faces and sides
    float4 prev[NPC], kap[NPC];
    int off[NPC];
    unsigned fl[NPC];  // bit 0 exists, 1 first chunk of a row, 2-5 element of x = nx (15: none), 6 / 7 to the band
                       // before / after, 8 / 9 row 1 / ny - 1, 10 on: touches absorbing faces (slot + 1)
#pragma unroll
    for (int q = 0; q < NPC; ++q) {
        const int i = tid + q * BT;
        off[q] = P + 4;
        fl[q] = 0;
        prev[q] = kap[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < nc) {
            int f = i - cx;
            f += f < 0 ? nc : 0;
            const int lr = f / cx, ic = f - lr * cx, r = r0 + lr, x0 = 4 * ic;
            const int m = min(4, sx - x0);  // nodes of the chunk
            const long long j = (long long)r * sx + x0;
            if (!CMCG_RANGE_OK(j, j + m - 1, g.np, kSiteColumn)) continue;
            off[q] = (lr + 1) * P + x0 + 4;
            float pv[4] = {0.f, 0.f, 0.f, 0.f}, kv[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e < m) {
                    pv[e] = a.buf1[j + e];
                    kv[e] = a.kap[j + e];
                }
            prev[q] = make_float4(pv[0], pv[1], pv[2], pv[3]);
            kap[q] = make_float4(kv[0], kv[1], kv[2], kv[3]);
            const bool last = g.nx - x0 < 4;
            const int nby = ((r == 0) & (int)((g.abc >> 2) & 1u)) + ((r == g.ny) & (int)((g.abc >> 3) & 1u));
            const bool left = ic == 0 && (g.abc & 1u), right = last && (g.abc & 2u);
            unsigned slot = 0;
            if (nby || left || right) {
                // (a row of one chunk has both ends in it: the left end's slot)
                slot = 1u + (unsigned)face_slot(lr, rows, !left, nby != 0, r == g.ny && nbands == 1, ic, cx);
                FaceNode<float> fn[4];
                float sr[4] = {0.f, 0.f, 0.f, 0.f}, si[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int nb = nby + (left && e == 0 ? 1 : 0) + (right && e == g.nx - x0 ? 1 : 0);
                    fn[e].set(e < m ? nb : 0, kv[e], nullptr);
                    if (SRC == 1 && e < m && nb) {
                        sr[e] = a.S[2 * (j + e)];
                        si[e] = a.S[2 * (j + e) + 1];
                    }
                }
                FaceChunk& fc = faces[slot - 1];
                fc.c1 = make_float4(fn[0].c1, fn[1].c1, fn[2].c1, fn[3].c1);
                fc.d = make_float4(fn[0].d, fn[1].d, fn[2].d, fn[3].d);
                fc.r = make_float4(fn[0].r, fn[1].r, fn[2].r, fn[3].r);
                fc.s01 = make_float4(sr[0], si[0], sr[1], si[1]);
                fc.s23 = make_float4(sr[2], si[2], sr[3], si[3]);
            }
            fl[q] = 1u | (ic == 0 ? 2u : 0u) | ((unsigned)(last ? g.nx - x0 : 15) << 2) | (up && lr == 0 ? 64u : 0u) |
                    (down && lr == rows - 1 ? 128u : 0u) | (r == 1 ? 256u : 0u) | (r == g.ny - 1 ? 512u : 0u) | slot << 10;
            if (SRC == 2) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    ssrc[4 * i + e] = e < m ? make_float2(a.S[2 * (j + e)], a.S[2 * (j + e) + 1]) : make_float2(0.f, 0.f);
            }
        }
    }
    open_exchange<CL>(sm_words, 4 * side_words);
    __syncthreads();

    const int n_up = up ? cx : 0, n_all = n_up + (down ? cx : 0);  // halo chunks
    const int from0 = tid < n_up ? 0 : 1, e0 = from0 ? tid - n_up : tid;
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
        unsigned long long w[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int q = 0; q < NPC; ++q) {
            // (opaque: what follows from them is worked out each step, not kept in registers)
            asm volatile("" : "+r"(off[q]), "+r"(fl[q]));
            const unsigned f = fl[q];
            if (f & 1u) {
                const int o = off[q], xe = (int)(f >> 2) & 15;
                float4 s01 = make_float4(0.f, 0.f, 0.f, 0.f), s23 = s01;
                if (SRC == 2) {
                    const float4* sp = reinterpret_cast<const float4*>(ssrc + 4 * (tid + q * BT));
                    s01 = sp[0];
                    s23 = sp[1];
                }
                const float4 c = *reinterpret_cast<const float4*>(in + o);
                const float4 v = update4<SRC>(in + o, P, kap[q], prev[q], (f & 2u) != 0u, xe,
                                              f >> 10 ? faces + ((f >> 10) - 1) : nullptr, flags, s01, s23, cs, sn);
                prev[q] = c;
                *reinterpret_cast<float4*>(out + o) = v;
                if (f & 0x3c0u) {
                    if (f & 256u) *reinterpret_cast<float4*>(out + o - 2 * P) = v;
                    if (f & 512u) *reinterpret_cast<float4*>(out + o + 2 * P) = v;
                    if (more && (f & 0xc0u)) {
                        const int ic = (o - 4 - (o / P) * P) >> 2;
                        if (f & 64u) ex.put4(0, ic, v, tag);
                        if (f & 128u) ex.put4(1, ic, v, tag);
                    }
                }
            }
            // the first look at the neighbours' rows, in flight during the other chunks
            if (q == 0 && more && tid < n_all) ex.get4(from0, e0, tag, w);
        }
        if (more) {
            for (int i = tid; i < n_all; i += BT) {
                const int from = i < n_up ? 0 : 1, e = from ? i - n_up : i;
                int polls = 0;
                while ((unsigned)(w[0] >> 32) != tag || (unsigned)(w[1] >> 32) != tag || (unsigned)(w[2] >> 32) != tag ||
                       (unsigned)(w[3] >> 32) != tag) {
                    ex.get4(from, e, tag, w);
                    if (ex.give_up(polls)) {
                        failed = true;
                        break;
                    }
                }
                if (failed) break;
                *reinterpret_cast<float4*>(out + (from ? rows + 1 : 0) * P + 4 + 4 * e) =
                    make_float4(__uint_as_float((unsigned)w[0]), __uint_as_float((unsigned)w[1]),
                                __uint_as_float((unsigned)w[2]), __uint_as_float((unsigned)w[3]));
                w[0] = 0ull;  // the next chunk of a wide grid starts afresh
            }
        }
        failed = __syncthreads_or(failed) != 0;
        if (failed) break;
    }
    close_exchange<CL>();
    if (failed) return;
    float* gc = (a.nsteps & 1) ? a.buf1 : a.buf0;
    float* gp = (a.nsteps & 1) ? a.buf0 : a.buf1;
    const float* in = buf + (a.nsteps & 1) * bufsz;
#pragma unroll
    for (int q = 0; q < NPC; ++q) {
        if (!(fl[q] & 1u)) continue;
        const int o = off[q], lr = o / P - 1, x0 = o - (lr + 1) * P - 4;
        const long long j = (long long)(r0 + lr) * sx + x0;
        const float pv[4] = {prev[q].x, prev[q].y, prev[q].z, prev[q].w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (x0 + e <= g.nx) {
                gc[j + e] = in[o + e];
                gp[j + e] = pv[e];
            }
    }
    // (the counts past the last band too: a handle's next loop may have more bands)
    if (!CL && band + tid * nbands < kBandStop) a.count[band + tid * nbands] = base + (unsigned)a.nsteps;
}

template <typename T, typename K>
cudaError_t band_go(K kernel, const BandArgs<T>& a, const BandPlan& p, size_t smem, cudaStream_t st) {
    // (always the same value: threads with other plans set it too, between this call and the launch)
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e == cudaSuccess && p.cluster > 8)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.bands);
    cfg.blockDim = dim3((unsigned)kBandThreads<T>);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (p.cluster) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)p.bands;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = p.bands > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

// The kernel that runs a plan: k_band4, or k_band with its reach R, made for npt chunks or nodes per
// thread; npt 0: there is none.
struct BandKernel {
    bool four;
    int reach, npt;
};
BandKernel band_kernel_of(int order, int elem_size, const BandPlan& p) {
    const bool four = elem_size == 4 && order == 2;
    auto made_for = [&](int most) { return p.npt <= most; };
    int npt = 0;
    if (four) npt = made_for(1) ? 1 : (made_for(2) ? 2 : (made_for(3) && p.cluster ? 3 : 0));
    else if (order == 2) npt = made_for(1) ? 1 : (made_for(2) ? 2 : (made_for(4) ? 4 : (made_for(8) ? 8 : 0)));
    else npt = made_for(2) ? 2 : (made_for(8) ? 8 : 0);
    return BandKernel{four, order / 2, npt};
}

template <int SRC, bool CL, typename T>
cudaError_t band_kernel(int order, const BandArgs<T>& a, const BandPlan& p, cudaStream_t st) {
    const size_t smem = p.smem[SRC == 2];
    const BandKernel k = band_kernel_of(order, (int)sizeof(T), p);
    if constexpr (std::is_same<T, float>::value) {
        if (k.four) {
            if (k.npt == 1) return band_go(k_band4<1, SRC, CL>, a, p, smem, st);
            if (k.npt == 2) return band_go(k_band4<2, SRC, CL>, a, p, smem, st);
            if constexpr (CL) {
                if (k.npt == 3) return band_go(k_band4<3, SRC, CL>, a, p, smem, st);
            }
            return cudaErrorInvalidValue;
        }
    } else {
        if (k.reach == 1) {
            if (k.npt == 1) return band_go(k_band<double, 1, 1, SRC, CL>, a, p, smem, st);
            if (k.npt == 2) return band_go(k_band<double, 1, 2, SRC, CL>, a, p, smem, st);
            if (k.npt == 4) return band_go(k_band<double, 1, 4, SRC, CL>, a, p, smem, st);
            if (k.npt == 8) return band_go(k_band<double, 1, 8, SRC, CL>, a, p, smem, st);
            return cudaErrorInvalidValue;
        }
    }
    if (k.npt == 2) return band_go(k_band<T, 2, 2, SRC, CL>, a, p, smem, st);
    if (k.npt == 8) return band_go(k_band<T, 2, 8, SRC, CL>, a, p, smem, st);
    return cudaErrorInvalidValue;
}

}  // namespace

// With sms = 16: a plan for kernels that run side by side, one cluster each (up to 443^2 in FP32).
// Bands: as many as there are SMs, but at least R + 1 rows each (a band holds the rows that its
// mirror rows repeat) and enough nodes to occupy a CTA; a grid of a few nodes per thread runs in
// one CTA, without exchange.
bool band_plan(const Geom& g, int order, int elem_size, int sms, BandPlan* p) {
    *p = BandPlan();
    if (g.dim != 2) return false;
    const bool vec = elem_size == 4 && order == 2;  // k_band4: four nodes per thread and chunk
    const int R = order / 2, bt = elem_size == 4 ? kBandThreads<float> : kBandThreads<double>;
    const long long cx = vec ? (g.sx + 3) / 4 : g.sx;        // items of a row
    const long long pitch = vec ? 4 * cx + 8 : g.sx + 2 * R;
    const long long items = cx * g.sy;
    long long bands = std::min<long long>(std::min(sms, kMaxBands), g.sy / (R + 1));
    // FP32: half a CTA's threads busy are enough; up to 16 bands exchange within a cluster, which
    // costs half of what the exchange through L2 does, so a grid that 16 hold stays there
    bands = std::min(bands, (items + bt / 2 - 1) / (bt / 2));
    long long in_cluster = 16;  // largest cluster of at least R + 1 rows per band, a power of two
    while (in_cluster > std::min<long long>(g.sy / (R + 1), sms)) in_cluster >>= 1;
    if (in_cluster > 1 && ((g.sy + in_cluster - 1) / in_cluster) * cx <= bt && bands > in_cluster)
        bands = in_cluster;
    if (bands <= 16) {
        long long b2 = 1;
        while (b2 < bands) b2 <<= 1;
        bands = std::min(b2, in_cluster);
    }
    if (items <= bt / 2 || bands < 1) bands = 1;
    const long long rows = (g.sy + bands - 1) / bands;
    const long long per_thread = (rows * cx + bt - 1) / bt;
    const long long buf = (rows + 2 * R) * pitch;
    const int cluster = bands > 1 && bands <= 16 ? (int)bands : 0;
    // (three chunks per thread in clusters only: one band of more than two runs step by step)
    if (per_thread > (vec ? (cluster ? 3 : 2) : 8) || buf > 65535) return false;
    const long long side_words = (vec ? 4 * cx : R * g.sx) * (elem_size / 4);
    p->cluster = cluster;
    p->face_slots = (int)(2 * rows + (bands == 1 ? 2 : 1) * cx);
    if (!vec && p->face_slots > 8190) return false;  // slot numbers have 13 bits
    const long long slot_bytes = vec ? sizeof(FaceChunk) : (elem_size == 4 ? sizeof(FaceNode<float>) : sizeof(FaceNode<double>));
    if (!vec && elem_size == 4) p->face_slots = (p->face_slots + 3) & ~3;  // keeps what follows aligned
    p->smem[0] = (size_t)(2 * buf * elem_size + (p->cluster ? 32 * side_words : 0) + slot_bytes * p->face_slots);
    p->smem[1] = p->smem[0] + (size_t)(2 * rows * (vec ? 4 * cx : g.sx) * elem_size);
    if (p->smem[0] > (size_t)kSmemMax) return false;
    p->bands = (int)bands;
    p->rows = (int)(g.sy / bands);
    p->extra = (int)(g.sy % bands);
    p->npt = (int)per_thread;
    p->words = p->cluster ? 0 : (size_t)(4 * side_words * bands);
    return true;
}

void band_plan_query(const Geom& g, int order, int elem_size, int sms, int* out) {
    BandPlan p;
    if (!band_plan(g, order, elem_size, sms, &p)) return (void)(out[0] = 0);
    const BandKernel k = band_kernel_of(order, elem_size, p);
    out[0] = p.bands;
    out[1] = p.rows + (p.extra ? 1 : 0);
    out[2] = p.cluster;
    out[3] = k.four ? 4 : 1;
    out[4] = k.reach;
    out[5] = k.npt;
    out[6] = elem_size == 4 ? kBandThreads<float> : kBandThreads<double>;
    out[7] = (int)p.smem[0];
}

bool band_fits(const BandPlan& p, bool volume_source) {
    return p.bands > 0 && p.smem[volume_source ? 1 : 0] <= (size_t)kSmemMax;
}

template <typename T>
cudaError_t launch_step_band(const Geom& g, int order, const BandPlan& p, T* cur, T* prev, const T* kap, const T* S,
                             bool src_faces, const double* wface, unsigned long long* words, unsigned* count,
                             double* err, int polls, int nsteps, const double* cs, const double* sn, bool adj_first,
                             bool adj_last, cudaStream_t st) {
    BandArgs<T> a;
    a.polls = polls;
    a.face_slots = p.face_slots;
    a.buf0 = cur;
    a.buf1 = prev;
    a.kap = kap;
    a.S = S;
    a.wface = wface;
    a.words = words;
    a.count = count;
    a.err = err;
    a.g = g;
    a.rows = p.rows;
    a.extra = p.extra;
    a.nsteps = nsteps;
    a.adj_first = adj_first;
    a.adj_last = adj_last;
    for (int s = 0; s < nsteps && S; ++s) {
        a.cs[s] = (T)cs[s];
        a.sn[s] = (T)sn[s];
    }
    const int src = S ? (src_faces ? 1 : 2) : 0;
    cudaError_t e;
    if (p.cluster)
        e = src == 0   ? band_kernel<0, true>(order, a, p, st)
            : src == 1 ? band_kernel<1, true>(order, a, p, st)
                       : band_kernel<2, true>(order, a, p, st);
    else
        e = src == 0   ? band_kernel<0, false>(order, a, p, st)
            : src == 1 ? band_kernel<1, false>(order, a, p, st)
                       : band_kernel<2, false>(order, a, p, st);
    if (e == cudaSuccess) note_launch(1);
    return e;
}
template cudaError_t launch_step_band<float>(const Geom&, int, const BandPlan&, float*, float*, const float*,
                                             const float*, bool, const double*, unsigned long long*, unsigned*,
                                             double*, int, int, const double*, const double*, bool, bool,
                                             cudaStream_t);
template cudaError_t launch_step_band<double>(const Geom&, int, const BandPlan&, double*, double*, const double*,
                                              const double*, bool, const double*, unsigned long long*, unsigned*,
                                              double*, int, int, const double*, const double*, bool, bool,
                                             cudaStream_t);

CMCG_CHECK_TU(band)

}  // namespace cmcg
