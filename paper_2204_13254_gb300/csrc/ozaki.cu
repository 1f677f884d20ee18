// FP64-accurate elimination on the tensor cores (sm_103a): the exchange sweep of
// every symmetric matrix of a batch in 64-wide pivot blocks, its products formed
// from BF16 slices on tcgen05 instead of FP64 FMAs (the Ozaki splitting of a
// product into exact low-precision products).
//
// Splitting.  A vector v is scaled by a power of two 2^-e so that |v_k| 2^-e < 1 and
// rounded to the integers t_k = rint(v_k 2^(56-e)), written in seven balanced
// 8-bit digits, t = sum_p 2^(8 (6-p)) a_p with |a_0| <= 256, |a_p| <= 128 (exact
// in BF16).  For two such vectors and every weight class d = p + q <= 6 the
// products a_p b_q are summed over K = 64 and over the class's d + 1 pairs in one
// FP32 accumulator in tensor memory: every partial sum is an integer below
// 64 (2 2^15 + 6 2^14) < 2^24, so the accumulation is exact.  The classes are
// joined in 64-bit integers (T, exact but for a rounding below 2^-62 of the
// largest product) and scaled back with one conversion and one FP64 FMA.
// Dropping the classes d >= 7 leaves an error below 2^-54 of |A_i||B_j| per term:
// FP64 accuracy in the norm, not of every small element (an element far below the largest of
// its row and column has correspondingly fewer digits; DD_FACTOR_FP64 keeps those).
// The pivot rows k are scaled by powers of two before they are cut, D = diag(2^-s_k) with
// D P D of diagonal 1/4 .. 1, and B' by the inverse: with materials of eight decades contrast
// inside a pivot block the rows of the operator agree with an FP64 elimination to 2e-15 (nine
// in ten), without D to 1.7e-14.  The panel's own product takes eight slices of each operand,
// as B' becomes part of the operator: 1.5 % of a factorisation.
//
// Symmetry.  While a set K of indices has been swept, M_ij = M_ji when both or
// none of i, j are in K and M_ij = -M_ji otherwise, so only the lower triangle is
// kept (k_oz_mirror fills the rest at the end), and the column panel of a pivot
// block p is its row panel B = M[p, :] transposed up to the sign s_i = -1 for
// swept rows, +1 otherwise.  One pivot block is three kernels:
//   k_oz_panel   slices of D B; B' = -P^-1 B as a slice product; slices of D^-1 B'; the
//                row and column panels of M;
//   k_oz_update  M_ij += s_i B_i . B'_j over the lower triangle outside p, and,
//                in its first CTAs (one per matrix), P^-1 and its slices of the next
//                block; k_oz_pivot forms the first block's.
// What bounds it: instruction latency and the path to L2 in the update (two FP64
// operations per element and pivot block at two lanes per clock and SM, 16 bytes of
// HBM traffic); the wide pivot block and the triangle each halve both against 32-wide
// blocks over the full square; with a single matrix the pivots one after another.
// Measured, 40 matrices of up to 2,454 rows with their 1,229-row coarse matrix, per
// 64-wide block (mean over both): panel 0.07, update with the next pivot 0.28 ms, against
// 0.51 + 0.09 (pivot, panels in FP64), 0.22 (slices) and 0.70 ms per 32-wide block over
// the full square; the whole factorisation and a step 25.5 against 177 ms.
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "dd_internal.h"
#include "fixpoint.cuh"
#include "tcgen05.cuh"

namespace {

constexpr int kOzS = 7;                      // slices per operand (8 bits each) of the update
constexpr int kOzPanS = 8;                   // of the panel's product
constexpr int kOzRows = 128;                 // rows of a tile (MMA M)
constexpr int kOzCols = 32;                  // columns of one unit of the update (MMA N)
constexpr int kOzK = kOzNB;                  // pivot block width (MMA K = 4 x 16)
constexpr uint32_t kOzPiece = kOzRows * kOzK * 2;    // 16 KB: one slice of a 128-row block
constexpr uint32_t kOzBlock = kOzS * kOzPiece;       // 112 KB: the slices of a 128-row block
constexpr uint32_t kOzPanBlock = kOzPanS * kOzPiece; // 128 KB: the same in the panel's shared memory
constexpr uint32_t kOzPPiece = kOzK * kOzK * 2;      // 8 KB: one slice of P^-1
constexpr uint32_t kOzPBlock = kOzPanS * kOzPPiece;  // 64 KB
constexpr uint32_t kOzUPiece = kOzCols * kOzK * 2;   // 4 KB: one slice of a 32-column unit
constexpr uint32_t kOzUnit = kOzS * kOzUPiece;       // 28 KB
constexpr unsigned kOzPolls = 1u << 22;
static_assert(kOzK == 64, "the slice layout and the exactness bound assume a 64-wide pivot block");

inline cudaStream_t S(void* s) { return (cudaStream_t)s; }

// An integer |d| <= 256 as FP32 (exact; its upper 16 bits are the BF16 value).
__device__ __forceinline__ uint32_t small_float(int d) {
    return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f);
}

// rint(v 2^(56-e)) of |v| < 2^e (halves away from zero) in integer arithmetic: the multiply and
// the conversion would take 32 clocks of the SM's FP64 pipe for a warp, these about 8 of the
// integer pipe.  Subnormals count as zero.
__device__ __forceinline__ long long to_digits(double v, int e) {
    const int hi = __double2hiint(v), ex = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        ((unsigned long long)(uint32_t)((hi & 0xfffff) | 0x100000) << 32) | (uint32_t)__double2loint(v);
    const unsigned r = min((unsigned)(1022 + e - ex), 63u);   // the value is (m 2^4 >> r) / 2
    const unsigned long long t = ex ? (((m << 4) >> r) + 1) >> 1 : 0ull;
    return hi < 0 ? -(long long)t : (long long)t;
}

// The same with eight bits more: the integer t of to_digits and, in `low` (|low| <= 128), the
// multiples of 2^-8 that it leaves.  Bits below those are dropped.
__device__ __forceinline__ long long to_digits(double v, int e, int& low) {
    const int hi = __double2hiint(v), ex = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        ((unsigned long long)(uint32_t)((hi & 0xfffff) | 0x100000) << 32) | (uint32_t)__double2loint(v);
    const unsigned r = (unsigned)(1022 + e - ex);   // the value is m 2^11 >> r in units of 2^-8
    const unsigned long long t8 = ex && r < 64u ? (m << 11) >> r : 0ull;
    const unsigned long long t = (t8 + 128) >> 8;   // (m 2^11 ends in eleven zeros: no carry out)
    const int l = (int)(t8 - (t << 8));
    low = hi < 0 ? -l : l;
    return hi < 0 ? -(long long)t : (long long)t;
}

// v 2^x, by the exponent field where the result is a normal number.
__device__ __forceinline__ double scale_exp(double v, int x) {
    const int hi = __double2hiint(v), ex = (hi >> 20) & 0x7ff;
    if (ex && (unsigned)(ex + x - 1) < 2046u) return __hiloint2double(hi + (x << 20), __double2loint(v));
    return v * pow2(x);
}

// Slices of eight consecutive elements v[0..7] (K direction) of a vector with
// exponent e, scaled by 2^-x[0..7]: one 16-byte chunk per slice, handed to put(slice, chunk).
template <int kS, typename Put>
__device__ __forceinline__ void cut8(const double* v, int e, const int (&x)[8], Put put) {
    uint32_t w[kS][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t f[2][kS];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            long long t;
            if constexpr (kS == 8) {
                int low;
                t = to_digits(v[2 * q + u], e + x[2 * q + u], low);
                f[u][7] = small_float(low);
            } else {
                t = to_digits(v[2 * q + u], e + x[2 * q + u]);
            }
            const unsigned long long b = (unsigned long long)t + 0x0000808080808080ull;   // balanced digits
            const uint32_t lo = (uint32_t)b, hi = (uint32_t)(b >> 32);
            f[u][6] = small_float((int)(lo & 255u) - 128);
            f[u][5] = small_float((int)((lo >> 8) & 255u) - 128);
            f[u][4] = small_float((int)((lo >> 16) & 255u) - 128);
            f[u][3] = small_float((int)(lo >> 24) - 128);
            f[u][2] = small_float((int)(hi & 255u) - 128);
            f[u][1] = small_float((int)((hi >> 8) & 255u) - 128);
            f[u][0] = small_float((int)hi >> 16);
        }
#pragma unroll
        for (int p = 0; p < kS; ++p) w[p][q] = __byte_perm(f[0][p], f[1][p], 0x7632);
    }
#pragma unroll
    for (int p = 0; p < kS; ++p) put(p, make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]));
}

// The high word of |v| 2^-x, for the largest of several: exponents compare as such (zero and
// subnormal numbers below every other), and the exponent of the largest (0 where all are zero).
constexpr int kOzNone = INT_MIN;
__device__ __forceinline__ int scaled_hi(double v, int x) {
    const int hi = __double2hiint(v) & 0x7fffffff;
    return hi >> 20 ? hi - (x << 20) : kOzNone;
}
__device__ __forceinline__ int scaled_exp(int hi) { return hi == kOzNone ? 0 : (hi >> 20) - 1022; }
// Eight scales of the pivot block's rows (a multiple of four integers).
__device__ __forceinline__ void load_scales(const int32_t* p, int (&x)[8]) {
    const int4 a = __ldg(reinterpret_cast<const int4*>(p)), b = __ldg(reinterpret_cast<const int4*>(p) + 1);
    x[0] = a.x;
    x[1] = a.y;
    x[2] = a.z;
    x[3] = a.w;
    x[4] = b.x;
    x[5] = b.y;
    x[6] = b.z;
    x[7] = b.w;
}

// Eight columns of the panel's eight class accumulators (stride `cls` tensor-memory columns
// apart) of the warp's 32 lanes, all loads in flight together.
__device__ __forceinline__ void ld_classes(uint32_t t, uint32_t cls, uint32_t (&r)[kOzPanS][8]) {
#define OZ_O(d) "=r"(r[d][0]), "=r"(r[d][1]), "=r"(r[d][2]), "=r"(r[d][3]), "=r"(r[d][4]), "=r"(r[d][5]), "=r"(r[d][6]), "=r"(r[d][7])
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%64];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%65];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%66];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%67];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%32,%33,%34,%35,%36,%37,%38,%39}, [%68];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%40,%41,%42,%43,%44,%45,%46,%47}, [%69];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%48,%49,%50,%51,%52,%53,%54,%55}, [%70];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%56,%57,%58,%59,%60,%61,%62,%63}, [%71];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : OZ_O(0), OZ_O(1), OZ_O(2), OZ_O(3), OZ_O(4), OZ_O(5), OZ_O(6), OZ_O(7)
        : "r"(t), "r"(t + cls), "r"(t + 2 * cls), "r"(t + 3 * cls), "r"(t + 4 * cls), "r"(t + 5 * cls), "r"(t + 6 * cls),
          "r"(t + 7 * cls)
        : "memory");
#undef OZ_O
}

// The same for the update: eight columns of 32 lanes in the 16 x 256-bit shape, by which a thread
// gets columns 2 (lane % 4), + 1 of rows lane / 4 + 8 k in r[.][2 k], r[.][2 k + 1]: four lanes
// cover 64 contiguous bytes of a row of doubles.
__device__ __forceinline__ void ld_classes_pairs(uint32_t t, uint32_t cls, uint32_t (&r)[kOzS][8]) {
#pragma unroll
    for (int d = 0; d < kOzS; ++d) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];\n"
                         : "=r"(r[d][4 * h]), "=r"(r[d][4 * h + 1]), "=r"(r[d][4 * h + 2]), "=r"(r[d][4 * h + 3])
                         : "r"(t + d * cls + ((uint32_t)(16 * h) << 16))
                         : "memory");
    }
    // the registers pass through the wait so that no use moves above it
#define OZ_P(d) "+r"(r[d][0]), "+r"(r[d][1]), "+r"(r[d][2]), "+r"(r[d][3]), "+r"(r[d][4]), "+r"(r[d][5]), "+r"(r[d][6]), "+r"(r[d][7])
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" : OZ_P(0), OZ_P(1), OZ_P(2) : : "memory");
    asm volatile("" : OZ_P(3), OZ_P(4), OZ_P(5) : : "memory");
    asm volatile("" : OZ_P(6) : : "memory");
#undef OZ_P
}

// T of one element: sum_d D_d 2^(8 (5-d)) ... in units of 2^-40 of class 0, i.e. the
// product is T 2^(e + f - 56) (|T| < 2^63; classes 6 and 7 rounded in, see the file comment).
template <int kS>
__device__ __forceinline__ double join_classes(const uint32_t (&r)[kS][8], int c) {
    auto I = [&](int d) { return (long long)__float2int_rn(__uint_as_float(r[d][c])); };
    const long long H = (I(0) << 16) + (I(1) << 8) + I(2);
    long long L = (I(3) << 24) + (I(4) << 16) + (I(5) << 8) + I(6);
    if constexpr (kS == 8) L += (I(7) + 128) >> 8;
    return (double)((H << 24) + ((L + 128) >> 8));
}

__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t parity, unsigned polls = kOzPolls) {
    for (unsigned k = 0; k < polls; ++k) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(tc::smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ bool oz_wait_or_abort(uint64_t* bar, uint32_t parity, const volatile int* abort) {
    for (unsigned k = 0; k < kOzPolls; ++k) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(tc::smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((k & 255u) == 255u && *abort) return false;
    }
    return false;
}

// Failure-path test (PcgScalars::wait_first = n > 0): the CTA's first wait is for `never`, which
// nothing completes at that point, n polls long.
__device__ __forceinline__ bool oz_first_wait(int n, uint64_t* never) {
    return n > 0 ? oz_wait(never, 0u, (unsigned)n) : true;
}

__device__ __forceinline__ void oz_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void oz_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void oz_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void oz_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            tc::smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(tc::smem_addr(bar))
        : "memory");
}

// The kS (kS + 1) / 2 slice products of A rows (slices at a0, kOzPiece bytes apart) and `cls` B rows (slices
// at b0, one after the other) into the class accumulators at `acc`, `cls` columns apart.
// For one slice p of A the classes p + q lie side by side, and so do the slices q of B: one
// MMA takes as many q as N = 256 columns allow.  An MMA reads its 128 x 16 A operand from
// shared memory whatever N is, which at N = 32 takes four times the product itself (measured,
// per-block means: update 384 -> 367 us, panel 77 -> 72 us against 112 MMAs of N = 32 per unit).
template <int kS>
__device__ __forceinline__ void oz_products(uint32_t acc, int cls, uint32_t a0, uint32_t b0) {
    const int qmax = 256 / cls;
    const uint32_t sb = (uint32_t)cls * kOzK * 2;
    for (int p = 0; p < kS; ++p)
        for (int q = 0; q < kS - p; q += qmax) {
            const int nq = min(qmax, kS - p - q);
            const uint32_t idesc = tc::idesc_bf16_f32(kOzRows, nq * cls);
            for (int ks = 0; ks < kOzK / 16; ++ks) {
                const uint64_t ad = tc::smem_desc(a0 + p * kOzPiece + ks * 256, 128, (kOzK / 8) * 128);
                const uint64_t bd = tc::smem_desc(b0 + q * sb + ks * 256, 128, (kOzK / 8) * 128);
                tc::mma_bf16(acc + (p + q) * cls, ad, bd, idesc, (p | ks) ? 1u : 0u);
            }
        }
}

// ---- pivot block -------------------------------------------------------------
// P^-1 of the pivot block, one CTA per matrix.
//  * All on D P D, whose inverse D^-1 P^-1 D^-1 is called X here.
//  * A first X by a Gauss-Jordan sweep in FP32 (SPD: no pivoting).
//  * Newton: R = I - P X from exact 57-bit fixed-point sums, X += X R in FP32, twice as a rule (|R| is 2^-20,
//    then 2^-41): X ends at its own FP64 rounding.
//  * A block that FP32 does not serve (a pivot that is not positive, |R| >= 2^-5, or >= 2^-36 at
//    the second look: the contraction is 2^-24 of the condition number) is swept in FP64 and
//    taken as swept, in full: its errors are those of a nearby block, which cancel in the
//    panels, while with growing condition number a rounded symmetric X loses more and more of
//    it (measured, coupled operator, condition number of A_rr 3e3: 3e-13 and 2e-12).  Eight
//    meshes of 5 to 9 cells a side against an extended-precision reference, geometric mean,
//    with time steps that make the condition number 1e3 .. 3e5: 1.8e-13, 2.9e-12, 1.7e-11,
//    6.2e-11; FP64 elimination 1.6e-13, 3.0e-12, 1.6e-11, 5.5e-11.
// With the FP64 sweep for every block, and one correction, 173 us (its FMAs alone 124 us: the
// FP64 pipe), with this 76 us (40 matrices).  The sweep's 64 roundings per element would be the
// largest error of a well-conditioned elimination (the products are exact to 2^-54).  Measured,
// coupled operator against an extended-precision reference, seven meshes (six bisected into
// 139 to 600 uneven subdomains): 1.9e-16 .. 3.5e-16; with the FP64 sweep alone 2.9e-16 ..
// 4.5e-16, with 32-wide pivot blocks in plain FP64 2.5e-16 .. 4.0e-16.
// Writes P^-1 back into M[p, p] (the panel kernel does not read that block), and the slices of
// P^-1 D^-1, their exponents and the exponents of D.
constexpr int kOzPivThreads = 256;
constexpr int kPs = kOzK + 1;   // row stride in shared memory

// The FP32 sweep, the inverse in place: thread (ty, tx) holds elements (ty + 16 u, 4 tx + v) of
// the full square.  Step k publishes row and column k and the pivot d; with p = 1 / d and the
// pivot's own entries published as d + 1 (row) and d - 1 (column), a_ij -= c_i (r_j p) is the
// whole exchange, row and column k included (d < 1 by the scaling, so 1 +- d costs no accuracy).
// buf [2][kSwBuf] by step parity, so that one barrier a step is enough (a step's readers meet
// the next writers of its half one barrier on).  The reciprocal may be approximate, as the
// result is corrected.  One loop body and no selection by register index: the code is run
// once per launch, and with bodies unrolled over the registers its instruction fetches beside
// the update took longer than the steps.  False, in every thread, if a pivot was not positive.
constexpr int kSwBuf = 2 * kOzK + 4;
constexpr size_t kOzPivSmem = kOzK * kPs * (sizeof(double) + 2 * sizeof(int2)) + 2 * kSwBuf * sizeof(float) + 3 * kOzK * sizeof(int);
__device__ __forceinline__ bool sweep32(float (&a)[4][4], float* buf, int nb, int tid) {
    const int tx = tid & 15, ty = tid >> 4;
    bool good = true;
#pragma unroll 1
    for (int k = 0; k < nb; ++k) {
        float* row = buf + (k & 1) * kSwBuf;
        float* col = row + kOzK;
        if (ty == (k & 15)) {
            const int uk = k >> 4;
            float4 w = make_float4(a[0][0], a[0][1], a[0][2], a[0][3]);
#pragma unroll
            for (int u = 1; u < 4; ++u)
                if (uk == u) w = make_float4(a[u][0], a[u][1], a[u][2], a[u][3]);
            *reinterpret_cast<float4*>(row + 4 * tx) = w;
        }
        if (tx == (k >> 2)) {
            const int q = k & 3;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float x = q < 2 ? (q == 0 ? a[u][0] : a[u][1]) : (q == 2 ? a[u][2] : a[u][3]);
                const bool own = ty + 16 * u == k;
                col[ty + 16 * u] = own ? x - 1.0f : x;
                if (own) {
                    row[k] = x + 1.0f;
                    col[kOzK] = x;
                }
            }
        }
        __syncthreads();
        float d = col[kOzK];
        if (!(d > 0.0f) || !isfinite(d)) {
            good = false;
            d = 1.0f;
        }
        const float p = __fdividef(1.0f, d);
        const float4 r = *reinterpret_cast<const float4*>(row + 4 * tx);
        const float rp[4] = {r.x * p, r.y * p, r.z * p, r.w * p};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float c = col[ty + 16 * u];
#pragma unroll
            for (int v = 0; v < 4; ++v) a[u][v] = fmaf(-c, rp[v], a[u][v]);
        }
    }
    __syncthreads();
    return good;
}

// The FP64 sweep, for the blocks that the FP32 one leaves: the same in shared memory, Q [.][kPs].
__device__ __forceinline__ bool sweep64(double* Q, int nb, int tid) {
    const int tx = tid & 15, ty = tid >> 4;
    bool good = true;
    for (int k = 0; k < nb; ++k) {
        double d = Q[k * kPs + k];
        if (!(d > 0.0) || !isfinite(d)) {
            good = false;
            d = 1.0;
        }
        const double p = 1.0 / d;
        double r[4], c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            r[u] = Q[k * kPs + tx + 16 * u] * p;
            c[u] = Q[(ty + 16 * u) * kPs + k];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = ty + 16 * u;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int j = tx + 16 * v;
                double* q = Q + i * kPs + j;
                *q = i == k ? (j == k ? p : r[v]) : (j == k ? -c[u] * p : fma(-c[u], r[v], *q));
            }
        }
        __syncthreads();
    }
    return good;
}

// Threads 0 .. kOzPivThreads - 1 of the CTA (the others have exited); smem kOzPivSmem bytes.
__device__ __forceinline__ void pivot_block(const MatDesc& md, double* __restrict__ M, int m, int k0,
                                            uint16_t* __restrict__ Ps, int32_t* __restrict__ ep,
                                            int32_t* __restrict__ status, unsigned char* smem) {
    const int nb = min(kOzK, md.nr - k0);
    double* Q = reinterpret_cast<double*>(smem);         // [kOzK][kPs] the block in full; then R in FP32
    int2* Pi = reinterpret_cast<int2*>(Q + kOzK * kPs);  // [kOzK][kPs] P, row i in units of 2^(rp_i - 57)
    int2* Xi = Pi + kOzK * kPs;                          // [kOzK][kPs] X, column j in units of 2^(cx_j - 57)
    float* sw = reinterpret_cast<float*>(Xi + kOzK * kPs);   // the sweep's rows and columns
    int* rp = reinterpret_cast<int*>(sw + 2 * kSwBuf);
    int* cx = rp + kOzK;
    int* sd = cx + kOzK;
    double* A = M + md.moff + (int64_t)k0 * md.ld + k0;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int ri = tid >> 2, rq = tid & 3;   // (row, quarter of its 64 columns) for row maxima and slices
    // the k-th column of the quarter, rotated so that a half warp's 16 elements lie in 16 bank pairs
    auto qc = [&](int k) { return 16 * rq + ((k + 4 * rq) & 15); };
    double a[4][4];
    auto load = [&]() {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v) {
                const int i = ty + 16 * u, j = tx + 16 * v;
                a[u][v] = (i < nb && j <= i) ? A[(int64_t)i * md.ld + j] : 0.0;
            }
    };
    auto scale = [&]() {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v) a[u][v] *= pow2n(-sd[ty + 16 * u] - sd[tx + 16 * v]);
    };
    // the lower triangle in registers -> the full symmetric block in Q (zero outside nb)
    auto spread = [&]() {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v) {
                const int i = ty + 16 * u, j = tx + 16 * v;
                if (j > i) continue;
                const double x = i < nb ? a[u][v] : 0.0;
                Q[i * kPs + j] = x;
                Q[j * kPs + i] = x;
            }
        __syncthreads();
    };
    auto row_exp = [&]() {   // exponent of the largest element of row ri (all four lanes of the row)
        int mx = 0;
        for (int k = 0; k < 16; ++k) mx = max(mx, __double2hiint(Q[ri * kPs + qc(k)]) & 0x7fffffff);
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        return exp_of_hi(mx);
    };
    // row ri of Q in 57-bit units of 2^(e - 57), handed to put(column, words)
    auto split_row = [&](int e, auto put) {
        const int x = kBits - e;
        if (x > -1000 && x < 1000) {   // (scale2's range, outside the loop)
            const double f = pow2(x);
#pragma unroll 4
            for (int k = 0; k < 16; ++k) put(qc(k), split57(__double2ll_rn(Q[ri * kPs + qc(k)] * f)));
        } else {
#pragma unroll 1
            for (int k = 0; k < 16; ++k) put(qc(k), split57(Q[ri * kPs + qc(k)], x));
        }
    };
    // P from here on is D P D with D = diag(2^-sd), its diagonal in [1/4, 1) (D = 1 where an exponent
    // is far out), and X its inverse
    load();
    const int dx = tid < nb ? (exp_of_hi(__double2hiint(A[(int64_t)tid * md.ld + tid]) & 0x7fffffff) + 1) >> 1 : 0;
    const int far = __syncthreads_or(abs(dx) > 200);
    if (tid < kOzK) sd[tid] = far ? 0 : dx;
    __syncthreads();
    scale();
    spread();
    {
        const int e = row_exp();
        rp[ri] = e;
        split_row(e, [&](int c, int2 w) { Pi[ri * kPs + c] = w; });
    }
    __syncthreads();
    // X = 0, so that the FP64 sweep follows, where an exponent is far out or a pivot was not positive
    float* F = reinterpret_cast<float*>(Xi);   // [kOzK][kPs]
    if (!far) {
        float f[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int i = ty + 16 * u, j = 4 * tx + v;
                f[u][v] = (float)Q[i * kPs + j];
                if (i == j && i >= nb) f[u][v] = 1.0f;
            }
        const bool ok = sweep32(f, sw, nb, tid);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) F[(ty + 16 * u) * kPs + 4 * tx + v] = ok ? f[u][v] : 0.0f;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v) {
                const int i = ty + 16 * u, j = tx + 16 * v;
                a[u][v] = (double)F[i * kPs + j];
            }
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v) a[u][v] = 0.0;
    }
    bool swept = false;   // in FP64, X in Q
    for (int pass = 0; pass < 2; ++pass) {
        spread();
        {
            const int e = row_exp();   // X is symmetric: also its column exponent
            cx[ri] = e;
            split_row(e, [&](int c, int2 w) { Xi[c * kPs + ri] = w; });
        }
        __syncthreads();
        // R = I - P X: 64 products per element fit the accumulators
        float* R = reinterpret_cast<float*>(Q);
        long long hh[4][4] = {}, xx[4][4] = {};
        for (int k = 0; k < nb; ++k) {
            int2 p[4], x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                p[u] = Pi[(ty + 16 * u) * kPs + k];
                x[u] = Xi[k * kPs + tx + 16 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) mac(hh[u][v], xx[u][v], p[u].x, p[u].y, x[v].x, x[v].y);
        }
        int big = 0;   // 2: |R| >= 2^-5 (or exponents out of range), 1: |R| >= 2^-36
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                // the sums hold P X in units of 2^-sh; the 1 is taken off before the low words join
                const int i = ty + 16 * u, j = tx + 16 * v, sh = 2 * kBits - kLow - rp[i] - cx[j];
                const bool one = u == v && tx == ty && i < nb;
                const bool fit = sh >= 40 && sh <= (one ? kLow + 62 : 120);
                const long long t = (one && fit ? 1ll << (sh - kLow) : 0ll) - hh[u][v] - (xx[u][v] >> kLow);
                const float lo = (float)((int)xx[u][v] & ((1 << kLow) - 1)) * (1.0f / (1 << kLow));
                const float f = fit ? ((float)t - lo) * __int_as_float((127 + kLow - sh) << 23) : 0.0f;
                const float g = fabsf(f);
                if (i < nb && j < nb) big = max(big, !fit || g >= 0x1p-5f ? 2 : g >= 0x1p-36f ? 1 : 0);
                R[i * kPs + j] = f;   // (every thread is done with Q)
            }
        const int any2 = __syncthreads_or(big == 2), any1 = __syncthreads_or(big >= 1);
        if (any2 || (any1 && pass == 1)) {
            load();
            scale();
            spread();
            if (!sweep64(Q, nb, tid) && tid == 0) atomicCAS(status, 0, DD_ERR_NOT_SPD);
            swept = true;
            break;
        }
        float y[4][4] = {};   // (X R) in units of 2^(cx_i - 28) X's
#pragma unroll 8
        for (int k = 0; k < kOzK; ++k) {
            float x[4], r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                x[u] = (float)Xi[k * kPs + ty + 16 * u].x;
                r[u] = R[k * kPs + tx + 16 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v <= u; ++v) y[u][v] = fmaf(x[u], r[v], y[u][v]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v) {
                const int i = ty + 16 * u, j = tx + 16 * v;
                if (i < nb && j <= i) a[u][v] += (double)y[u][v] * pow2(cx[i] - (kBits - kLow));
            }
        __syncthreads();
        if (!any1) break;
    }
    if (!swept) spread();
    for (int p = tid; p < kOzK * kOzK; p += kOzPivThreads) {
        const int i = p >> 6, j = p & 63;
        if (i < nb && j <= i) A[(int64_t)i * md.ld + j] = Q[i * kPs + j] * pow2n(-sd[i] - sd[j]);
    }
    // slices
    const int e = row_exp();
    if (rq == 0) {
        ep[(int64_t)m * 2 * kOzK + ri] = e - sd[ri];
        ep[(int64_t)m * 2 * kOzK + kOzK + ri] = sd[ri];
    }
    unsigned char* out = reinterpret_cast<unsigned char*>(Ps) + (int64_t)m * kOzPBlock;
    for (int g = 0; g < 2; ++g) {
        const int k = 16 * rq + 8 * g;
        double v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = Q[ri * kPs + k + c];
        const int none[8] = {};
        cut8<kOzPanS>(v, e, none, [&](int p, uint4 w) {
            *reinterpret_cast<uint4*>(out + p * kOzPPiece + tc::kmajor_off(ri, k, kOzK)) = w;
        });
    }
}

// The first pivot block, one CTA per matrix; the later ones are formed by k_oz_update.
__global__ void __launch_bounds__(kOzPivThreads, 1) k_oz_pivot(const MatDesc* __restrict__ mats, double* __restrict__ M,
                                                               uint16_t* __restrict__ Ps, int32_t* __restrict__ ep,
                                                               int32_t* __restrict__ status) {
    const MatDesc md = mats[blockIdx.x];
    if (md.nr <= 0) return;
    extern __shared__ __align__(16) unsigned char smem[];
    pivot_block(md, M, (int)blockIdx.x, 0, Ps, ep, status, smem);
}

// ---- panel -------------------------------------------------------------------
// One CTA per (128 indices j, matrix), thread (j, half): 32 of the 64 pivot rows each.
// The panel's values (row-read for swept j, column-read below the block) become slices
// in shared memory (the MMA's A operand) and in global memory (the update's rows); the
// slice product with P^-1 gives B' = -P^-1 B, which is written back to the row panel
// (j < k0) or, negated, to the column panel (j >= k0 + nb), and cut into slices again
// (the update's columns).  192 KB of shared memory, 512 tensor-memory columns.
constexpr int kOzPanThreads = 256;
constexpr size_t kOzPanSmem = kOzPanBlock + kOzPBlock + 64;
__global__ void __launch_bounds__(kOzPanThreads, 1) k_oz_panel(const MatDesc* __restrict__ mats, double* __restrict__ M,
                                                               int k0, int nrb, const uint16_t* __restrict__ Ps,
                                                               const int32_t* __restrict__ ep, uint16_t* __restrict__ Bs,
                                                               int32_t* __restrict__ eb, uint16_t* __restrict__ Cs,
                                                               int32_t* __restrict__ ec, int nmax,
                                                               PcgScalars* __restrict__ sc) {
    const int m = blockIdx.y, rb = blockIdx.x;
    const MatDesc md = mats[m];
    if (k0 >= md.nr || rb * kOzRows >= md.ns) return;
    const int nb = min(kOzK, md.nr - k0);
    extern __shared__ __align__(128) unsigned char sm[];
    unsigned char* sB = sm;
    unsigned char* sP = sm + kOzPanBlock;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sP + kOzPBlock);   // [0] P^-1 slices, [1] products
    uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2);
    __shared__ int xmax[2][kOzRows];
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        oz_init(&bars[0], 1);
        oz_init(&bars[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        oz_expect(&bars[0], kOzPBlock);
        oz_bulk(sP, reinterpret_cast<const unsigned char*>(Ps) + (int64_t)m * kOzPBlock, kOzPBlock, &bars[0]);
    }
    if (warp == 0) tc::tmem_alloc(tslot, 512);
    const int r = tid & (kOzRows - 1), half = tid >> 7, kb = 32 * half;
    const int j = rb * kOzRows + r;
    const bool on = j < md.ns && (j < k0 || j >= k0 + nb);
    const bool row = j < k0;   // stored in the row panel
    double* A = M + md.moff;
    double v[32];
    int mx = kOzNone;
    // below the block a thread's values are contiguous: 16-byte accesses
    double2* const col = reinterpret_cast<double2*>(A + (int64_t)j * md.ld + k0 + kb);
    if (on && !row) {
#pragma unroll
        for (int k = 0; k < 32; k += 2) {
            double2 t = make_double2(0.0, 0.0);
            if (kb + k + 1 < nb) t = col[k / 2];
            else if (kb + k < nb) t.x = col[k / 2].x;
            v[k] = t.x;
            v[k + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = on && kb + k < nb ? A[(int64_t)(k0 + kb + k) * md.ld + j] : 0.0;
    }
    const int32_t* const epm = ep + (int64_t)m * 2 * kOzK;   // exponents of the rows of P^-1 D^-1, then sd
    const int32_t* const sdm = epm + kOzK + kb;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        int x[8];
        load_scales(sdm + 8 * g, x);
#pragma unroll
        for (int c = 0; c < 8; ++c) mx = max(mx, scaled_hi(v[8 * g + c], x[c]));
    }
    xmax[half][r] = mx;
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;
    const int64_t blk = ((int64_t)m * nrb + rb) * kOzBlock;
    const int e = scaled_exp(max(xmax[0][r], xmax[1][r]));
    {   // D B
        unsigned char* gB = reinterpret_cast<unsigned char*>(Bs) + blk;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint32_t o = tc::kmajor_off(r, kb + 8 * g, kOzK);
            int x[8];
            load_scales(sdm + 8 * g, x);
            cut8<kOzPanS>(v + 8 * g, e, x, [&](int p, uint4 w) {
                *reinterpret_cast<uint4*>(sB + p * kOzPiece + o) = w;
                if (p < kOzS) *reinterpret_cast<uint4*>(gB + p * kOzPiece + o) = w;
            });
        }
    }
    if (half == 0 && j < md.ns) eb[(int64_t)m * nmax + j] = e;
    tc::fence_proxy_async();
    __syncthreads();
    bool ok = true;
    if (tid == 0) {
        ok = oz_first_wait(sc->wait_first, &bars[1]) && oz_wait(&bars[0], 0u);
        if (ok) {
            tc::fence_after_sync();
            oz_products<kOzPanS>(tmem, kOzK, tc::smem_addr(sB), tc::smem_addr(sP));
        }
        tc::mma_commit(&bars[1]);
    }
    const bool done = oz_wait(&bars[1], 0u);
    tc::fence_after_sync();
    const bool good = __syncthreads_and(done && ok) != 0;
    if (good) {
        mx = kOzNone;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            int x[8];
            load_scales(sdm + 8 * g, x);
            uint32_t D[kOzPanS][8];
            ld_classes(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + kb + 8 * g, kOzK, D);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int i = kb + 8 * g + c;
                const double y = -scale_exp(join_classes(D, c), e + epm[i] - 56);
                v[8 * g + c] = y;
                mx = max(mx, scaled_hi(y, -x[c]));
            }
        }
        if (on && row) {
#pragma unroll
            for (int k = 0; k < 32; ++k)
                if (kb + k < nb) A[(int64_t)(k0 + kb + k) * md.ld + j] = v[k];
        } else if (on) {
#pragma unroll
            for (int k = 0; k < 32; k += 2) {
                if (kb + k + 1 < nb) col[k / 2] = make_double2(-v[k], -v[k + 1]);
                else if (kb + k < nb) col[k / 2].x = -v[k];
            }
        }
    }
    xmax[half][r] = mx;   // the first exchange was read before the previous barriers
    __syncthreads();
    if (good) {
        const int f = scaled_exp(max(xmax[0][r], xmax[1][r]));   // of D^-1 B'
        if (half == 0 && j < md.ns) ec[(int64_t)m * nmax + j] = f;
        unsigned char* gC = reinterpret_cast<unsigned char*>(Cs) + blk;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint32_t o = tc::kmajor_off(r, kb + 8 * g, kOzK);
            int x[8];
            load_scales(sdm + 8 * g, x);
#pragma unroll
            for (int c = 0; c < 8; ++c) x[c] = -x[c];
            cut8<kOzS>(v + 8 * g, f, x, [&](int p, uint4 w) { *reinterpret_cast<uint4*>(gC + p * kOzPiece + o) = w; });
        }
    } else if (tid == 0) {
        atomicExch(&sc->wait_err, 1);
        oz_wait(&bars[0], 0u);   // the copy lands before the CTA ends (bounded)
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_free(tmem, 512);
}

// ---- trailing update ------------------------------------------------------------
// One CTA per (128-row block, run of kOzRun 32-column units of its lower triangle,
// matrix): the row block's 112 KB of slices are copied once for the run; the units'
// 28 KB come through a ring of four buffers, two units ahead.  Warp 8 issues the copies and
// the MMAs; warps 0..7 (rows 32 (w mod 4) .. + 31, columns 16 (w / 4) .. + 15) combine unit
// n from one tensor-memory half while the MMAs of unit n + 1 run into the other.
// What bounds it: latency and the path to L2 rather than the two FP64 operations per element.
// C is loaded a unit ahead (367 -> 350 us, mean over the blocks of 40 matrices of up to 2,454
// rows and their coarse matrix), and a thread holds column pairs of four rows so that a warp's
// access is whole 64-byte pieces of rows: with a row per lane every 16-byte access was half a
// sector, and the copies leave too little L1 to join them (350 -> 260 us).  Sixteen warps of
// eight columns with warp 0 issuing were slower in both layouts (398, 309 us).
// Every wait is bounded; a CTA whose wait gives up sets the error word, lets its copies land
// and frees its tensor memory.
constexpr int kOzRun = 16;
constexpr int kOzStages = 4;
constexpr int kOzThreads = 288;
constexpr int kOzWCols = 16;   // columns of a unit per warp
constexpr size_t kOzSmem = kOzBlock + kOzStages * kOzUnit + (1 + 2 * kOzStages + 4) * sizeof(uint64_t) + 16;
static_assert(kOzSmem <= 227 * 1024 && kOzPivSmem <= kOzBlock, "shared memory of the update");

__global__ void __launch_bounds__(kOzThreads, 1) k_oz_update(const MatDesc* __restrict__ mats, double* __restrict__ M,
                                                             int k0, int nrb, const uint16_t* __restrict__ Bs,
                                                             const uint16_t* __restrict__ Cs,
                                                             const int32_t* __restrict__ eb,
                                                             const int32_t* __restrict__ ec, int nmax,
                                                             uint16_t* __restrict__ Ps, int32_t* __restrict__ ep,
                                                             int nm, int runs, int32_t* __restrict__ status,
                                                             PcgScalars* __restrict__ pcg) {
    const bool ahead = (int)blockIdx.x < nm;
    const int m = ahead ? (int)blockIdx.x : ((int)blockIdx.x - nm) / runs;
    const MatDesc md = mats[m];
    if (k0 >= md.nr) return;
    const int nb = min(kOzK, md.nr - k0);
    const int k1 = k0 + kOzK, nb1 = max(0, min(kOzK, md.nr - k1));   // the next pivot block
    int rb = 0, u0, u1;
    if (ahead) {
        if (nb1 == 0) return;
        rb = k1 / kOzRows;
        u0 = k1 / kOzCols;
        u1 = u0 + (nb1 + kOzCols - 1) / kOzCols;
    } else {   // (row block, run): row block rb has ceil(4 (rb + 1) / kOzRun) runs
        int run = ((int)blockIdx.x - nm) % runs;
        for (;;) {
            const int nrun = (4 * (rb + 1) + kOzRun - 1) / kOzRun;
            if (run < nrun) break;
            run -= nrun;
            ++rb;
        }
        if (rb * kOzRows >= md.ns) return;
        u0 = run * kOzRun;
        u1 = min(min(u0 + kOzRun, 4 * (rb + 1)), (md.ns + kOzCols - 1) / kOzCols);
    }
    // units inside the pivot block are left out
    const int s0 = k0 / kOzCols, s1 = (k0 + nb) / kOzCols;   // units [s0, s1) lie wholly in it
    auto unit = [&](int n) {   // the n-th unit of the run
        int u = u0 + n;
        if (u >= s0 && u0 < s1) u += u0 >= s0 ? s1 - u0 : s1 - s0;
        return u;
    };
    const int skip = max(0, min(u1, s1) - max(u0, s0));
    const int nu = u1 - u0 - skip;
    if (nu <= 0) return;

    extern __shared__ __align__(128) unsigned char sm[];
    unsigned char* sA = sm;
    unsigned char* sC = sm + kOzBlock;
    uint64_t* abar = reinterpret_cast<uint64_t*>(sC + kOzStages * kOzUnit);
    uint64_t* full = abar + 1;             // [stage] unit copied
    uint64_t* empty = full + kOzStages;    // [stage] its products completed
    uint64_t* tfull = empty + kOzStages;   // [half] products in tensor memory
    uint64_t* tempty = tfull + 2;          // [half] read by the eight warps
    uint32_t* tslot = reinterpret_cast<uint32_t*>(tempty + 2);
    __shared__ int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned char* gC = reinterpret_cast<const unsigned char*>(Cs) + (int64_t)m * nrb * kOzBlock;
    int issued = 0;   // unit copies issued (the issuing lane)
    auto copy_unit = [&](int n) {
        const int u = unit(n), s = n % kOzStages;
        const unsigned char* src = gC + (int64_t)(u >> 2) * kOzBlock + (u & 3) * kOzUPiece;
        oz_expect(&full[s], kOzUnit);
#pragma unroll
        for (int p = 0; p < kOzS; ++p) oz_bulk(sC + s * kOzUnit + p * kOzUPiece, src + p * kOzPiece, kOzUPiece, &full[s]);
        ++issued;
    };
    if (tid == 256) {
        abort_flag = 0;
        oz_init(abar, 1);
        for (int s = 0; s < kOzStages; ++s) {
            oz_init(&full[s], 1);
            oz_init(&empty[s], 1);
        }
        for (int hh = 0; hh < 2; ++hh) {
            oz_init(&tfull[hh], 1);
            oz_init(&tempty[hh], 8);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        oz_expect(abar, kOzBlock);
        oz_bulk(sA, reinterpret_cast<const unsigned char*>(Bs) + ((int64_t)m * nrb + rb) * kOzBlock, kOzBlock, abar);
        for (int n = 0; n < 2 && n < nu; ++n) copy_unit(n);
    }
    if (warp == 0) tc::tmem_alloc(tslot, 512);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;

    // the issuing lane: the copy of unit n + 2 and the MMAs of unit n
    auto issue = [&](int n) {
        const int s = n % kOzStages, hh = n & 1;
        bool ok = true;
        if (n + 2 < nu) {   // unit n + 2 into the stage of unit n - 2
            if (n >= 2) ok = oz_wait_or_abort(&empty[(n - 2) % kOzStages], (uint32_t)((n - 2) / kOzStages) & 1u, &abort_flag);
            if (ok) copy_unit(n + 2);
        }
        if (ok) ok = oz_wait_or_abort(&full[s], (uint32_t)(n / kOzStages) & 1u, &abort_flag);
        if (ok && n >= 2) ok = oz_wait_or_abort(&tempty[hh], (uint32_t)((n >> 1) - 1) & 1u, &abort_flag);
        if (!ok) {
            abort_flag = 1;
            return;
        }
        tc::fence_after_sync();
        oz_products<kOzS>(tmem + 256u * hh, kOzCols, tc::smem_addr(sA), tc::smem_addr(sC + s * kOzUnit));
        tc::mma_commit(&tfull[hh]);
        tc::mma_commit(&empty[s]);
    };
    if (warp == 8) {
        if (lane == 0) {
            if (!oz_first_wait(pcg->wait_first, &tempty[0]) || !oz_wait(abar, 0u)) abort_flag = 1;
            for (int n = 0; n < nu && !abort_flag; ++n) issue(n);
        }
    } else {
        // rows i0 + 8 k, columns j0 .. j0 + 1 of every group of eight
        const int i0 = rb * kOzRows + 32 * (warp & 3) + (lane >> 2);
        const int hcol = kOzWCols * (warp >> 2) + 2 * (lane & 3);
        const int32_t* ecm = ec + (int64_t)m * nmax;
        double* crow = M + md.moff + (int64_t)i0 * md.ld;
        const int64_t step = 8 * (int64_t)md.ld;
        int e[4], jend[4], sg[4];   // exponent, end of the row in the lower triangle, sign bit
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + 8 * k;
            const bool next = i >= k1 && i < k1 + nb1;   // rows of the next pivot block
            const bool row_ok = ahead ? next : i < md.ns && (i < k0 || i >= k0 + nb);
            e[k] = row_ok ? eb[(int64_t)m * nmax + i] : 0;
            jend[k] = row_ok ? (next && !ahead ? k1 : i + 1) : 0;
            sg[k] = i < k0 ? (int)0x80000000 : 0;
        }
        auto in = [&](int k, int j) { return j < jend[k] && (j < k0 || j >= k0 + nb); };
        auto load_c = [&](int n, double (&c)[kOzWCols], int (&f)[kOzWCols / 4]) {
#pragma unroll
            for (int g = 0; g < kOzWCols / 8; ++g) {
                const int j = unit(n) * kOzCols + hcol + 8 * g;
                f[2 * g] = j < md.ns ? ecm[j] : 0;
                f[2 * g + 1] = j + 1 < md.ns ? ecm[j + 1] : 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    double* const p = crow + k * step + j;
                    double2 t = make_double2(0.0, 0.0);
                    if (in(k, j) && in(k, j + 1)) t = *reinterpret_cast<const double2*>(p);
                    else {
                        if (in(k, j)) t.x = p[0];
                        if (in(k, j + 1)) t.y = p[1];
                    }
                    c[8 * g + 2 * k] = t.x;
                    c[8 * g + 2 * k + 1] = t.y;
                }
            }
        };
        double cn[kOzWCols];
        int fn[kOzWCols / 4];
        load_c(0, cn, fn);
        for (int n = 0; n < nu; ++n) {
            const int hh = n & 1, j0 = unit(n) * kOzCols + hcol;
            double c[kOzWCols];
            int f[kOzWCols / 4];
#pragma unroll
            for (int q = 0; q < kOzWCols; ++q) c[q] = cn[q];
#pragma unroll
            for (int q = 0; q < kOzWCols / 4; ++q) f[q] = fn[q];
            if (n + 1 < nu) {
                load_c(n + 1, cn, fn);   // in flight while this unit is combined
            }
            const bool ok = oz_wait_or_abort(&tfull[hh], (uint32_t)(n >> 1) & 1u, &abort_flag);
            if (__any_sync(0xffffffffu, !ok)) {
                abort_flag = 1;
                break;
            }
            tc::fence_after_sync();
#pragma unroll
            for (int g = 0; g < kOzWCols / 8; ++g) {
                uint32_t D[kOzS][8];
                ld_classes_pairs(tmem + 256u * hh + ((uint32_t)(32 * (warp & 3)) << 16) + kOzWCols * (warp >> 2) + 8 * g,
                                 kOzCols, D);
                if (g == kOzWCols / 8 - 1) {   // the half is read: later products may overwrite it
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) oz_arrive(&tempty[hh]);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const double sc = pow2(e[k] + f[2 * g + u] - 56);   // its sign set without an FP64 operation
                        c[8 * g + 2 * k + u] =
                            fma(join_classes(D, 2 * k + u),
                                __hiloint2double(__double2hiint(sc) ^ sg[k], __double2loint(sc)), c[8 * g + 2 * k + u]);
                    }
                    const int j = j0 + 8 * g;
                    double* const p = crow + k * step + j;
                    if (in(k, j) && in(k, j + 1))
                        *reinterpret_cast<double2*>(p) = make_double2(c[8 * g + 2 * k], c[8 * g + 2 * k + 1]);
                    else {
                        if (in(k, j)) p[0] = c[8 * g + 2 * k];
                        if (in(k, j + 1)) p[1] = c[8 * g + 2 * k + 1];
                    }
                }
            }
        }
    }
    __syncthreads();
    if (abort_flag && tid == 256) {   // the copies issued land before the CTA ends (bounded), then report
        oz_wait(abar, 0u);
        for (int n = issued > kOzStages ? issued - kOzStages : 0; n < issued; ++n)
            oz_wait(&full[n % kOzStages], (uint32_t)(n / kOzStages) & 1u);
        atomicExch(&pcg->wait_err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_free(tmem, 512);
    if (!ahead || abort_flag || warp == 8) return;
    pivot_block(md, M, m, k1, Ps, ep, status, sm);   // written by this CTA, before the barrier above
}

// M[i][j] for j > i from the lower triangle: -M[j][i] when exactly one index was swept
// (i < nr <= j), M[j][i] otherwise.  One CTA per 64 x 64 tile pair, through shared memory.
__global__ void __launch_bounds__(256) k_oz_mirror(const MatDesc* __restrict__ mats, double* __restrict__ M) {
    const MatDesc md = mats[blockIdx.y];
    int a = 0, b = (int)blockIdx.x;   // tile (a, b), b <= a
    while (b > a) b -= ++a;
    if (a * 64 >= md.ns) return;
    __shared__ double t[64][65];
    double* A = M + md.moff;
    const int lx = threadIdx.x & 63, ly = threadIdx.x >> 6;
    for (int y = ly; y < 64; y += 4) {
        const int i = a * 64 + y, j = b * 64 + lx;
        if (i < md.ns && j < i) t[y][lx] = (j < md.nr && i >= md.nr) ? -A[(int64_t)i * md.ld + j] : A[(int64_t)i * md.ld + j];
    }
    __syncthreads();
    for (int y = ly; y < 64; y += 4) {
        const int j = b * 64 + y, i = a * 64 + lx;   // element (j, i) of the upper triangle
        if (i < md.ns && j < i) A[(int64_t)j * md.ld + i] = t[lx][y];
    }
}

}  // namespace

// Workspace of one pivot block (bytes): slices of P^-1, B and B' and their exponents.
namespace {
struct OzLayout {
    size_t ps, bs, cs, ep, eb, ec, total;
};
OzLayout oz_layout(int nm, int nmax) {
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t nrb = (size_t)(nmax + kOzRows - 1) / kOzRows;
    OzLayout L;
    L.ps = 0;
    L.bs = L.ps + up((size_t)nm * kOzPBlock);
    L.cs = L.bs + up((size_t)nm * nrb * kOzBlock);
    L.ep = L.cs + up((size_t)nm * nrb * kOzBlock);
    L.eb = L.ep + up((size_t)nm * 2 * kOzK * sizeof(int32_t));
    L.ec = L.eb + up((size_t)nm * nmax * sizeof(int32_t));
    L.total = L.ec + up((size_t)nm * nmax * sizeof(int32_t));
    return L;
}
}  // namespace

size_t oz_bytes(int nm, int nmax) { return oz_layout(nm, std::max(nmax, 1)).total; }

// One pivot block [k0, k0 + 64) of the sweep of nm matrices (of at most nmax rows), and the
// inverse of the next one; called for k0 = 0, 64, ... in turn.
int launch_oz_sweep(const MatDesc* mats, double* M, int nm, int nmax, int k0, unsigned char* ws, int32_t* status,
                    PcgScalars* sc, void* stream) {
    const int nrb = (nmax + kOzRows - 1) / kOzRows;
    const OzLayout L = oz_layout(nm, nmax);
    uint16_t* Ps = reinterpret_cast<uint16_t*>(ws + L.ps);
    uint16_t* Bs = reinterpret_cast<uint16_t*>(ws + L.bs);
    uint16_t* Cs = reinterpret_cast<uint16_t*>(ws + L.cs);
    int32_t* ep = reinterpret_cast<int32_t*>(ws + L.ep);
    int32_t* eb = reinterpret_cast<int32_t*>(ws + L.eb);
    int32_t* ec = reinterpret_cast<int32_t*>(ws + L.ec);
    cudaError_t e = cudaFuncSetAttribute(k_oz_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzPanSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_oz_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_oz_pivot, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzPivSmem);
    if (e != cudaSuccess) return (int)e;
    if (k0 == 0) k_oz_pivot<<<(unsigned)nm, kOzPivThreads, kOzPivSmem, S(stream)>>>(mats, M, Ps, ep, status);
    k_oz_panel<<<dim3((unsigned)nrb, (unsigned)nm), kOzPanThreads, kOzPanSmem, S(stream)>>>(mats, M, k0, nrb, Ps, ep, Bs,
                                                                                            eb, Cs, ec, nmax, sc);
    unsigned runs = 0;
    for (int rb = 0; rb < nrb; ++rb) runs += (unsigned)((4 * (rb + 1) + kOzRun - 1) / kOzRun);
    k_oz_update<<<(unsigned)nm * (1 + runs), kOzThreads, kOzSmem, S(stream)>>>(mats, M, k0, nrb, Bs, Cs, eb, ec, nmax, Ps,
                                                                              ep, nm, (int)runs, status, sc);
    return (int)cudaGetLastError();
}

// The upper triangles after the last pivot block.
int launch_oz_mirror(const MatDesc* mats, double* M, int nm, int nmax, void* stream) {
    const unsigned nt = (unsigned)(nmax + 63) / 64;
    k_oz_mirror<<<dim3(nt * (nt + 1) / 2, (unsigned)nm), 256, 0, S(stream)>>>(mats, M);
    return (int)cudaGetLastError();
}
