// fixed.cuh -- block floating point on the integer multipliers, for FP64 arithmetic that the FP64
// unit would bound (1.67 lanes per clock and SM on GB300, where a 32x32+64-bit multiply-add runs
// at 63).  A real x of a block with biased exponent Eb (|x| < 2^(Eb - 1022)) is the integer
// x 2^59 / 2^(Eb - 1022), rounded toward zero, as two signed words hi 2^30 + lo with |hi| < 2^29
// and |lo| < 2^30 (sums of two still fit).  A product takes three multiply-adds: hi hi, and
// hi lo + lo hi in a second 64-bit sum that is rounded into the first; lo lo is dropped.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace lq {

// (double)f: the conversion instruction runs at a fifth of the FP64 unit's rate (0.35 lanes per clock
// and SM, measured), these few integer ones at full rate.  Zeros, subnormals, infinities and NaNs
// take the instruction.
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f);
    if (((b >> 23) & 0xffu) - 1u >= 254u) return (double)f;
    return __hiloint2double((int)((((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

struct Fix2 {  // hi * 2^30 + lo
    int hi, lo;
};
constexpr uint32_t kFixMask = (1u << 30) - 1;

__device__ __forceinline__ uint64_t shr64(uint64_t v, uint32_t n) {  // 0 for n > 63
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}
__device__ __forceinline__ uint32_t shr32(uint32_t v, uint32_t n) {  // 0 for n > 31
    uint32_t r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}
__device__ __forceinline__ long long sar64(long long v, uint32_t n) {  // the sign for n > 63
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) { return (long long)a * b + c; }

__device__ __forceinline__ double value(uint2 w) { return __hiloint2double((int)w.y, (int)w.x); }
__device__ __forceinline__ uint2 words(double v) {
    return make_uint2((unsigned)__double2loint(v), (unsigned)__double2hiint(v));
}

// The larger of m and the high words of two doubles without their signs, compared as FP32
// numbers (of the same order; a word that is an FP32 NaN, from 2^1017 up, gives a NaN, which is
// above every exponent allowed).
__device__ __forceinline__ float max_hi(float m, uint32_t a, uint32_t b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(__uint_as_float(a))), "f"(fabsf(__uint_as_float(b))));
    return r;
}

// |x| as fixed point below the block exponent (rounded toward zero), and the sign as +-1
struct FixMag {
    int hi, lo, s;
};
// e2 = 2 (Eb 2^20 + 2^20 - 1) + 1 + 5 2^21 with Eb the block's biased exponent: e2 - 2 w
// (w: the high word of x) has Eb - e + 5 in its top 11 bits whatever x's sign and mantissa
// are.  neg = 0, or -1 to negate.  A zero or subnormal x is shifted out, for Eb >= kFixEmin.
__device__ __forceinline__ FixMag fix_mag(uint2 x, uint32_t e2, int neg) {
    const uint32_t w = x.y, l = x.x;
    const uint32_t d = (e2 - 2u * w) >> 21;  // the block exponent above x's, plus 5
    const uint32_t nh = __funnelshift_l(l, w, 11) | 0x80000000u, nl = l << 11;  // mantissa, top bit set
    FixMag f;
    f.lo = (int)((uint32_t)shr64(((uint64_t)nh << 32) | nl, d) & kFixMask);
    f.hi = (int)shr32(nh, d - 2u);
    f.s = (((int)w >> 31) ^ neg) | 1;
    return f;
}
__device__ __forceinline__ Fix2 fix_one(uint2 x, uint32_t e2, int neg) {
    const FixMag f = fix_mag(x, e2, neg);
    return {f.hi * f.s, f.lo * f.s};
}
__device__ __forceinline__ Fix2 fix_pair(uint2 x, uint2 y, uint32_t e2, int nx, int ny) {
    const FixMag f = fix_mag(x, e2, nx), g = fix_mag(y, e2, ny);
    return {f.hi * f.s + g.hi * g.s, f.lo * f.s + g.lo * g.s};
}

// sum_k x_k y_k over six products, rounded to units of 2^60 of the product of the scales
__device__ __forceinline__ long long fix_dot(const Fix2 (&u)[6], const Fix2 (&h)[6]) {
    long long mid = 1LL << 29, top;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        mid = mad_wide(u[k].hi, h[k].lo, mid);
        mid = mad_wide(u[k].lo, h[k].hi, mid);
    }
    top = mid >> 30;
#pragma unroll
    for (int k = 0; k < 6; ++k) top = mad_wide(u[k].hi, h[k].hi, top);
    return top;
}

// v 2^(eb - 1079) rounded to nearest, eb a biased exponent in range; negated for the high bit of flip
__device__ __forceinline__ double fix_to_double(long long v, int eb, uint32_t flip) {
    const uint32_t sign = ((uint32_t)(v >> 32) ^ flip) & 0x80000000u;
    uint64_t m = (uint64_t)(v < 0 ? -v : v);
    const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
    // both counts, without a branch: the unit that counts has nothing else to do
    const int lz = mh ? __clz((int)mh) : 32 + __clz((int)ml);
    m <<= lz & 63;  // 64 for zero
    const uint64_t b = (m >> 11) + ((m >> 10) & 1);  // the leading bit carries into the exponent
    const uint32_t h = (uint32_t)(b >> 32) + ((uint32_t)(eb + 6 - lz) << 20);
    return __hiloint2double((int)((m ? h : 0u) | sign), (int)(uint32_t)b);
}

}  // namespace lq
