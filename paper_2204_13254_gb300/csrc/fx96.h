// The 96-bit integer sums of the fixed-point GEMV (fxgemv.cu), host and device.
//
// A product of two 57-bit integers is at most 2^114.  It reaches the sums as h 2^29 + x in
// units of 2^29 (fixpoint.cuh), and they hold it in units of 2^37: at most 2^77 a product, so
// sums of 2^17 products fit 95 bits and a sign whatever the products' signs, where the
// shared memory of a CTA ends below 2^13 columns.  (In units of 2^29, 2^10 products of one
// sign would leave them.)  The eight bits dropped are below 2^-76 of the largest product.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

constexpr int kFx96Low = 29;             // bits of the low words
constexpr int kFx96Drop = 8;             // bits dropped from x
constexpr int kFx96Unit = kFx96Low + kFx96Drop;   // the sums are in units of 2^37

// h hi hi' + cross sums of up to 64 products, in units of the 96-bit sums.
FX_HD __int128 fx96_part(int64_t h, int64_t x) {
    return ((__int128)h << (kFx96Low - kFx96Drop)) + (x >> kFx96Drop);
}
// (hi, lo) += v
FX_HD void fx96_add(uint64_t& lo, int32_t& hi, __int128 v) {
    v += ((__int128)hi << 64) + lo;
    lo = (uint64_t)v;
    hi = (int32_t)(v >> 64);
}
// The high 64 bits of a sum (times 2^32) and its low 32 bits.
FX_HD int64_t fx96_high(uint64_t lo, int32_t hi) { return (int64_t)(((uint64_t)(uint32_t)hi << 32) | (lo >> 32)); }
FX_HD uint32_t fx96_low(uint64_t lo) { return (uint32_t)lo; }
