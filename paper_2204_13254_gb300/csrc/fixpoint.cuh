// Powers of two and 57-bit fixed point, shared by the elimination (ozaki.cu) and the
// FP64 GEMV (fxgemv.cu).
#pragma once

#include <cstdint>

namespace {

// An integer t, |t| <= 2^57, in two words: t = hi 2^kLow + lo, |hi|, |lo| <= 2^28 (lo = 0
// where |hi| = 2^28).  Sums of hi hi' and of hi lo' + lo hi' over 64 products fit 64 bits.
constexpr int kBits = 57, kLow = 29;

// Exponent e with |x| < 2^e from the high word (without sign) of |x|; subnormals count as zero.
__device__ __forceinline__ int exp_of_hi(int hi) {
    const int f = hi >> 20;
    return f == 0 ? 0 : f - 1022;
}
__device__ __forceinline__ double pow2n(int x) { return __hiloint2double((x + 1023) << 20, 0); }   // |x| <= 1022
__device__ __forceinline__ double pow2(int x) {
    if (x > -1023 && x < 1024) return pow2n(x);
    return ldexp(1.0, x);
}
// v 2^x without an intermediate overflow of the factor.
__device__ __forceinline__ double scale2(double v, int x) {
    if (x > -1000 && x < 1000) return v * pow2(x);
    return ldexp(v, x);
}
// The two words of an integer |t| <= 2^57, and of v 2^x.
__device__ __forceinline__ int2 split57(long long t) {
    const int hi = (int)((t + (1ll << (kLow - 1))) >> kLow);
    return make_int2(hi, (int)(t - ((long long)hi << kLow)));
}
__device__ __forceinline__ int2 split57(double v, int x) { return split57(__double2ll_rn(scale2(v, x))); }

// acc += a b, one 32 x 32 + 64 bit multiply-add.
__device__ __forceinline__ void imad(long long& acc, int a, int b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// h += hi hi', x += hi lo' + lo hi'
__device__ __forceinline__ void mac(long long& h, long long& x, int mh, int ml, int vh, int vl) {
    imad(h, mh, vh);
    imad(x, mh, vl);
    imad(x, ml, vh);
}

}  // namespace
