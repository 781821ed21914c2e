// Arithmetic on unevaluated float32 pairs x = h + l (|l| below one unit in the
// last place of h), two values per operation: GB300 runs float32 at 64 times
// the rate of float64 (77.6 against 1.06 TFLOP/s of multiply-adds measured),
// so a float64 sum of products costs far less as pairs of float32, which hold
// 48 bits.  Error-free sums and products after Knuth and Dekker (with the
// fused multiply-add for the product's error).  Every operation is an explicit
// round-to-nearest intrinsic, which the compiler neither contracts nor
// reorders.
#pragma once

#include <cuda_runtime.h>

namespace bem {

using P2 = float2;                      // the same quantity of two targets

__device__ __forceinline__ P2 p2(float a) { return make_float2(a, a); }
__device__ __forceinline__ P2 padd(P2 a, P2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ P2 pmul(P2 a, P2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ P2 pfma(P2 a, P2 b, P2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ P2 psub(P2 a, P2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// the sign flipped by integer operations, off the float32 pipe
__device__ __forceinline__ P2 pxneg(P2 a) {
    return make_float2(__int_as_float(__float_as_int(a.x) ^ 0x80000000), __int_as_float(__float_as_int(a.y) ^ 0x80000000));
}
__device__ __forceinline__ P2 pneg(P2 a) { return make_float2(-a.x, -a.y); }

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(P2 a, P2 b, P2 &s, P2 &e) {
    s = padd(a, b);
    const P2 bb = psub(s, a);
    e = padd(psub(a, psub(s, bb)), psub(b, bb));
}
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (h, l) + (bh, bl)
__device__ __forceinline__ void df_add(float &h, float &l, float bh, float bl) {
    float s, e;
    two_sum(h, bh, s, e);
    h = s;
    l = __fadd_rn(__fadd_rn(l, bl), e);
}
// a float64 value as a pair
__device__ __forceinline__ void df_split(double x, float &h, float &l) {
    h = (float)x;
    l = (float)(x - (double)h);
}

// x 2^-(E - 1023) as a pair, for a biased exponent E >= that of x: taken from
// the bits of x (24 leading bits, then the other 29 rounded to 24) with integer
// operations and no float64 arithmetic.  Values below 2^-126 of the scale
// become zero; infinities and NaN become NaN.
__device__ __forceinline__ void df_bits(double x, int E, float &h, float &l) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int ex = (int)(hi >> 20) & 0x7ff, e = ex - E + 127;
    const unsigned sign = hi & 0x80000000u;
    if (ex == 0x7ff) {
        h = __int_as_float(0x7fffffff);
        l = 0.f;
        return;
    }
    const bool on = ex > 0 && e > 0;
    h = on ? __uint_as_float(sign | (unsigned)e << 23 | (hi & 0xfffffu) << 3 | lo >> 29) : 0.f;
    const float r = (float)(lo & 0x1fffffffu);
    const int el = e - 52;
    l = on && el > 0 ? r * __uint_as_float(sign | (unsigned)el << 23) : 0.f;
}

}  // namespace bem
