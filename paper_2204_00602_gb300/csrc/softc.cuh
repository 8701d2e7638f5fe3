// Complex products on the integer pipe.
//
// GB300 issues one FP64 warp instruction per 16 cycles and SM, so a complex
// FP64 product (4 instructions) takes 64; the same product of two 62-bit
// fixed-point numbers is 14 wide integer multiply-adds and some simple integer
// instructions, and takes about 22 (measured over 152 SMs, four chains a thread:
// 447 G against 143 G products/s).  It also keeps more bits: after 16 products the
// rms relative error, the rounding to FP64 included, is 5.4e-17 against 3.0e-16.
//
// A running product is p = (re + i im) 2^e with the larger component kept in
// [2^61, 2^62); a factor y is a fixed-point number of a scale its producer
// knows, components at most 2^61 (and a few units) in magnitude, given as
// balanced halves x = h 2^32 + l, l signed.  A product of components is formed
// without its low x low part: re = hi(ph yh) + (ph yl + pl yh) 2^-32, rounded
// to nearest; the cross terms of one component sum to at most 3 2^61 < 2^63.
// The dropped parts are below 2 units of the unshifted result, which is at
// least 2^54 for a factor within 2^-7 of its scale.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pcv {

struct SoftC {
    long long re, im;
    int e;
};

// a b + c, one wide multiply-add.
__device__ __forceinline__ long long soft_mad(int a, int b, long long c)
{
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

__device__ __forceinline__ long long soft_mul32(int a, int b)
{
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}

// Left shift that brings the larger component's leading bit to bit 61 (at
// most 30 places; |x| by its high word, so -2^61 counts as 2^61).
__device__ __forceinline__ int soft_lead(int re_hi, int im_hi)
{
    return __clz((int)((uint32_t)abs(re_hi) | (uint32_t)abs(im_hi))) - 2;
}

// Balanced halves of a fixed-point complex number: {re.h, re.l, im.h, im.l}.
__device__ __forceinline__ int4 soft_split(long long re, long long im)
{
    int4 y;
    y.y = (int)re;
    y.x = (int)(re >> 32) + (int)((uint32_t)y.y >> 31);
    y.w = (int)im;
    y.z = (int)(im >> 32) + (int)((uint32_t)y.w >> 31);
    return y;
}

// The first factor as a running product, normalised.
__device__ __forceinline__ SoftC soft_first(int4 y)
{
    SoftC p;
    p.re = ((long long)y.x << 32) + y.y;
    p.im = ((long long)y.z << 32) + y.w;
    const int s = soft_lead((int)(p.re >> 32), (int)(p.im >> 32));
    p.re <<= s;
    p.im <<= s;
    p.e = -61 - s;
    return p;
}

// p *= y, y a fixed-point number of scale 2^-61.
__device__ __forceinline__ void soft_mul(SoftC& p, const int4 y)
{
    const int4 q = soft_split(p.re, p.im);
    // -p.im: -l can pass 32 bits, ~l = -l - 1 cannot and is 2^-3 units off at most
    const int nh = -q.z, nl = ~q.w;
    const long long half = 1ll << 31;
    const long long hr = soft_mad(q.x, y.x, soft_mul32(nh, y.z));
    const long long cr = soft_mad(q.x, y.y, soft_mad(q.y, y.x, soft_mad(nh, y.w, soft_mad(nl, y.z, half))));
    const long long hi = soft_mad(q.x, y.z, soft_mul32(q.z, y.x));
    const long long ci = soft_mad(q.x, y.w, soft_mad(q.y, y.z, soft_mad(q.z, y.y, soft_mad(q.w, y.x, half))));
    // the cross terms' high word, sign-extended, added on the multiplier
    const long long re = soft_mad((int)(cr >> 32), 1, hr), im = soft_mad((int)(ci >> 32), 1, hi);
    const int s = soft_lead((int)(re >> 32), (int)(im >> 32));
    p.re = re << s;
    p.im = im << s;
    p.e += 3 - s;
}

// The signed integer x as a double (one rounding): both halves become exact
// doubles by the 2^52 offset, 3 FP64 instructions.
__device__ __forceinline__ double soft_value(long long x)
{
    const double hi = __hiloint2double(0x43300000, (int)((uint32_t)(x >> 32) ^ 0x80000000u)) - 4503601774854144.0;
    const double lo = __hiloint2double(0x43300000, (int)(uint32_t)x) - 4503599627370496.0;
    return fma(hi, 4294967296.0, lo);
}

// acc += (neg ? -p : p); a term below 2^-1022 of the common scale adds nothing.
__device__ __forceinline__ void soft_add(double2& acc, const SoftC& p, bool neg)
{
    const int f = 1023 + p.e;
    const double sc = f < 1 ? 0.0 : __hiloint2double((f << 20) | (neg ? (int)0x80000000 : 0), 0);
    acc.x = fma(soft_value(p.re), sc, acc.x);
    acc.y = fma(soft_value(p.im), sc, acc.y);
}

}  // namespace pcv
