// Linear contractions of float64 values as 57-bit fixed point on the integer
// pipe.
//
// GB300 issues 2 float64 fmas per SM and clock but 64 integer multiply-adds
// with a 64-bit accumulator (measured: fma.f64 1.9, mad.wide.s32 55
// thread-operations per SM and clock, the second unchanged by the first
// running beside it), so a contraction sum_i c_i x_i costs a tenth on the
// integer pipe.  Every operand is scaled by a power of two that its group
// shares and split into two signed words,
//   x = (x.h 2^28 + x.l) 2^(E - 1022 - 57),  |x.h| < 2^29, |x.l| < 2^28,
// where E is the largest biased exponent of the group; a product is
//   c x ~ c.h x.h 2^56 + (c.h x.l + c.l x.h) 2^28
// (c.l x.l < 2^-58 of the largest product is dropped), accumulated exactly in
// two 64-bit integers.  Each operand is truncated below 2^-57 of its group's
// largest, so a sum is within (terms) 2^-56 of max|c| max|x|, where a chain
// of float64 fmas rounds each partial sum at 2^-54 of itself.  The sums are
// exact in any order, and negating an operand negates its words.
//
// Range: up to 31 terms keep both accumulators below 2^63 (2^58 and 2 x 2^57
// per term); the operator has at most 30 (order 5, 3-D, with diffusion).
// Groups whose E lies outside [kFxMinE, kFxMaxE] are the caller's business:
// below, the values are flushed to zero (2^-823); above (and for infinities
// and NaN, whose biased exponent is 2047) the caller takes the float64 sums.
// The absolute error is the group's, so one huge value costs its whole group
// the bits below 2^-57 of it: the caller draws its own line (fx_limit,
// dg_stage64.cuh) well above any physical value and far below kFxMaxE.
#pragma once

#include <cuda_runtime.h>

namespace dgm {

constexpr int kFxMinE = 200;
constexpr int kFxMaxE = 1900;
constexpr int kFxOutE = 4095;    // marks a group as out of range

// biased exponent of x (0 for zero and subnormals, 2047 for infinities and NaN)
__device__ __forceinline__ int fx_expo(double x) {
    return (int)(((unsigned)__double2hiint(x) << 1) >> 21);
}

// x as fixed point with group exponent E >= fx_expo(x)
__device__ __forceinline__ int2 fx_from(double x, int E) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    // the 53-bit mantissa at bits 60..8 of (wh, wl), shifted right by E - e:
    // the high word is then x.h and the low word's upper 28 bits x.l
    const int d = E - (int)((hi << 1) >> 21);
    const unsigned wh = __funnelshift_l(lo, mh, 8);
    const unsigned wl = __funnelshift_rc(lo << 8, wh, (unsigned)d);       // d >= 32: wh
    const unsigned l = __funnelshift_rc(wl, 0u, (unsigned)max(d - 32, 0));
    const unsigned h = __funnelshift_rc(wh, 0u, (unsigned)d);
    const int sg = ((int)hi >> 31) | 1;
    return make_int2((int)h * sg, (int)(l >> 4) * sg);
}

// (a2, a1) += c x
__device__ __forceinline__ void fx_mac(int2 c, int2 x, long long &a2, long long &a1) {
    a2 += (long long)c.x * x.x;
    a1 += (long long)c.x * x.y;
    a1 += (long long)c.y * x.x;
}

// float64 value (rounded to nearest, ties away from zero) of a sum V that
// counts units of 2^(E - 1080)
__device__ __forceinline__ double fx_round(long long v, int E) {
    const long long sg = v >> 63;
    const unsigned long long m = (unsigned long long)((v ^ sg) - sg);
    const unsigned mh = (unsigned)(m >> 32), ml = (unsigned)m;
    const bool small = mh == 0u;
    unsigned h = small ? ml : mh, l = small ? 0u : ml;
    const int lz = __clz((int)h);                   // 32 only for V = 0
    h = __funnelshift_l(l, h, lz);
    l <<= (lz & 31);
    // top bit at 2^63: biased exponent E + 6 - shift, one less here because
    // the mantissa's leading bit adds it back (and a rounding carry goes on
    // into the exponent)
    const unsigned ex = (unsigned)(E + 5 - lz - (small ? 32 : 0));
    const unsigned long long r =
        (((unsigned long long)((h >> 11) + (ex << 20)) << 32) | __funnelshift_r(l, h, 11)) + ((l >> 10) & 1u);
    const unsigned rh = (unsigned)(r >> 32) | ((unsigned)sg & 0x80000000u);
    return h == 0u ? 0.0 : __hiloint2double((int)rh, (int)(unsigned)r);
}

// float64 value of an accumulator pair whose terms have group exponent E (the
// largest exponent(x) + q over the terms, with |c| < 2^q)
__device__ __forceinline__ double fx_value(long long a2, long long a1, int E) {
    return fx_round(a2 + (a1 >> 28), E);
}

// v 2^-d towards minus infinity, d >= 0
__device__ __forceinline__ long long fx_shift(long long v, int d) {
    return v >> min(d, 63);
}

// s_e[k] = max(s_e[k], e[k] over the CTA) for N <= 32 groups: one warp
// reduction per group, then one shared-memory atomic per warp with a group
// per lane, which enters a group above its limit as out of range.  limit: that
// of group threadIdx.x % 32.  Called by whole warps.
template <int N>
__device__ __forceinline__ void fx_reduce_max(const int *e, int limit, int *s_e) {
    const int lane = threadIdx.x & 31;
    int mine = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int r = __reduce_max_sync(0xffffffffu, e[k]);
        if (lane == k) mine = r;
    }
    if (mine > limit) mine = kFxOutE;
    if (lane < N && mine > 0) atomicMax(s_e + lane, mine);
}

}  // namespace dgm
