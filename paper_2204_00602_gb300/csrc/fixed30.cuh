// Sums of complex products on the integer pipe, without rounding.
//
// A fixed-point number is h 2^30 + l with |l| <= 2^29.  A sum keeps the products
// of the halves apart, hh 2^60 + hl 2^30 + ll, and is rounded once when it is
// taken out: 16 wide integer multiply-adds per complex term, about 16 cycles of
// an SM per warp where the four FP64 instructions take 64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pcv {

__device__ __forceinline__ void wide_mad(long long& acc, int x, int y)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(x), "r"(y));
}

__device__ __forceinline__ void split30(long long x, int& h, int& l)
{
    l = (int)((uint32_t)x << 2) >> 2;
    h = (int)((x - l) >> 30);
}

// {re.h, re.l, im.h, im.l}
__device__ __forceinline__ int4 split30(long long re, long long im)
{
    int4 y;
    split30(re, y.x, y.y);
    split30(im, y.z, y.w);
    return y;
}

__device__ __forceinline__ long long join30(int h, int l) { return ((long long)h << 30) + l; }

struct Sum30 {                                  // hh 2^60 + hl 2^30 + ll
    long long hh = 0, hl = 0, ll = 0;
    __device__ __forceinline__ void add(int xh, int xl, int yh, int yl)
    {
        wide_mad(hh, xh, yh);
        wide_mad(hl, xh, yl);
        wide_mad(hl, xl, yh);
        wide_mad(ll, xl, yl);
    }
    // the sum / 2^(30 + sh), rounded, 0 < sh <= 30
    __device__ __forceinline__ long long value(int sh) const
    {
        const long long v = hl + (ll >> 30);
        return (hh << (30 - sh)) + ((v + (1ll << (sh - 1))) >> sh);
    }
};

// re + i im += u c
__device__ __forceinline__ void add_term(Sum30& re, Sum30& im, const int4 u, const int4 c)
{
    re.add(u.x, u.y, c.x, c.y);
    re.add(-u.z, -u.w, c.z, c.w);
    im.add(u.x, u.y, c.z, c.w);
    im.add(u.z, u.w, c.x, c.y);
}

}  // namespace pcv
