// FP64 stencil sums on the integer pipes.
//
// GB300 issues FP64 arithmetic at 2 lanes per SM and cycle: one warp instruction holds the pipe
// for 16 cycles, as long as 64 issue slots of the SM.  A leapfrog update is mostly the
// neighbour sum, so the sum runs on integers instead: the stencil's values are aligned to the
// largest exponent among them as 64-bit fixed point with six guard bits, added exactly, and the
// sum goes back to FP64 once.  The rounding error of the sum is then at most the truncation of
// the aligned values, 2^-6 units in the last place of the largest one each, plus one conversion,
// where the chain of FP64 additions rounds every partial sum (up to 6 |y|) to 2^-53 of itself.
// Against a period in extended precision (31x27x25, noise): 7-point 1.2e-15 (the chain 1.2e-15),
// 13-point 1.3e-15 (3.2e-15); smooth fields 0.6e-15 (1.1e-15, 3.6e-15).
//
// The largest exponent field must lie in [kExpLo, kExpLo + kExpSpan) (magnitudes from 2^-895
// to 2^1017): infinities, NaN, overflowing sums and fields that are zero or tiny throughout take
// the plain FP64 sum instead, which is what every value took before.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace cmcg {
namespace soft64 {

constexpr unsigned kExpLo = 128u << 20;
constexpr unsigned kExpSpan = 1912u << 20;

// A finite double as a signed fixed-point mantissa (53 bits and six guard bits) and the exponent
// field of its high word.  A zero or subnormal counts as 2^-1023 (1 + ...): aligned to an
// exponent field of kExpLo or more it is shifted out.
struct Term {
    long long m;
    unsigned e;
};

__device__ __forceinline__ Term term(double y) {
    const unsigned hi = (unsigned)__double2hiint(y), lo = (unsigned)__double2loint(y);
    Term t;
    t.e = hi & 0x7ff00000u;
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 6) << 32) | (lo << 6);
    const long long s = (long long)((int)hi >> 31);
    t.m = ((long long)m ^ s) - s;
    return t;
}

// The term in units of 2^(E - 1081), E << 20 = emax (a shift of 63 or more leaves the sign).
__device__ __forceinline__ long long align(const Term& t, unsigned emax) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(t.m), "r"((emax - t.e) >> 20));
    return r;
}

// Is the fixed-point sum safe for terms with this largest exponent field?
__device__ __forceinline__ bool in_range(unsigned emax) { return emax - kExpLo < kExpSpan; }

// x 2^(E - 1081) as a double, rounded to 53 bits (halves away from zero); *ok turns false when |x| < 2^32 (the sum
// cancelled to nearly nothing, or is zero), which the caller leaves to the FP64 sum.
__device__ __forceinline__ double to_double(long long x, unsigned emax, bool* ok) {
    const long long s = x >> 63;
    const unsigned long long a = (unsigned long long)((x ^ s) - s);
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
    *ok = ah != 0u;
    const int lz = __clz((int)ah);  // 0 .. 31 where ok
    const unsigned nh = __funnelshift_l(al, ah, lz), nl = al << (lz & 31);
    unsigned hi = (nh >> 11) + emax + ((unsigned)(4 - lz) << 20), lo = __funnelshift_r(nl, nh, 11);
    // (a carry runs on into the exponent)
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"((nl >> 10) & 1u));
    return __hiloint2double((int)(hi | ((unsigned)(s >> 32) & 0x80000000u)), (int)lo);
}

// 4/3 of a fixed-point sum as a double: 4/3 rounded to FP64 is (1 - 2^-54) 4/3, an error that all
// steps of a loop share, so it is made good in the sum.
__device__ __forceinline__ double four_thirds(long long x, unsigned emax, bool* ok) {
    return (4.0 / 3.0) * to_double(x + ((int)(x >> 32) >> 22), emax, ok);
}

// Conversions between FP32 and FP64 by bit operations: the hardware's run on the FP64 pipe too.
// Normal values in both formats; zeros, subnormals, infinities, NaN and what rounds past the
// largest float take the hardware conversion, out of line.  Same results, bit for bit.
static __device__ __noinline__ float to_f32_hw(double x) { return (float)x; }
static __device__ __noinline__ double to_f64_hw(float x) { return (double)x; }

__device__ __forceinline__ float to_f32(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned a = hi & 0x7fffffffu;
    if (a - 0x38100000u < 0x0fd00000u) {  // 2^-126 <= |x| < 2^127
        const unsigned u = ((a - 0x38000000u) << 3) | (lo >> 29);
        const unsigned inc = (lo << 3) + (u & 1u) > 0x80000000u ? 1u : 0u;  // round to nearest even
        return __uint_as_float((u + inc) | (hi & 0x80000000u));
    }
    if ((a | lo) == 0u) return __uint_as_float(hi);
    return to_f32_hw(x);
}

__device__ __forceinline__ double to_f64(float x) {
    const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu;
    if (a - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)(((a >> 3) + 0x38000000u) | (u & 0x80000000u)), (int)(u << 29));
    if (a == 0u) return __hiloint2double((int)u, 0);
    return to_f64_hw(x);
}

// x == 0 without a comparison on the FP64 pipe.
__device__ __forceinline__ bool is_zero(double x) {
    return ((unsigned)__double2loint(x) | ((unsigned)__double2hiint(x) & 0x7fffffffu)) == 0u;
}

__device__ __forceinline__ unsigned max3(unsigned a, unsigned b, unsigned c) { return max(max(a, b), c); }

}  // namespace soft64
}  // namespace cmcg
