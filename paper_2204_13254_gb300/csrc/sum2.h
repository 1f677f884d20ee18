// FP32 numbers added without loss as two FP32 words (Knuth's two-sum), host and device: how
// the CTAs of the one-kernel GMRES (resident.cu) join the FP32 sums of 128 products that
// their warps form, where the kernels beyond its size (gmres.cu) join them in FP64.  The
// FP64 pipe takes 16 clocks for a warp's addition whatever the lanes hold; these are six
// FP32 additions.
#pragma once

#ifdef __CUDACC__
#define S2_HD __host__ __device__ __forceinline__
#else
#define S2_HD inline
#endif

struct Sum2 {
    float hi, lo;   // hi + lo; |lo| at the level of the rounding of hi
};

S2_HD Sum2 sum2_add(Sum2 a, Sum2 b) {
    const float s = a.hi + b.hi, t = s - a.hi;
    const float e = (a.hi - (s - t)) + (b.hi - t);   // s + e == a.hi + b.hi
    return {s, a.lo + b.lo + e};
}
