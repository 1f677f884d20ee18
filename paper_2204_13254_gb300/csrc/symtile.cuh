// Shared by the packed symmetric GEMVs (symgemv.cu, fxgemv.cu): the mbarrier ring of
// bulk copies and the shapes of the listed tiles.
#pragma once

#include <cstdint>

#include "dd_internal.h"

namespace {

constexpr unsigned kWaitLimit = 1u << 20;   // polls of one mbarrier wait before it gives up (well under a second)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// L2 policies for the tile copies: evict_last keeps a subset of the operator
// resident in L2 across the launches of one Krylov solve, evict_first streams
// the rest past it.
__device__ __forceinline__ uint64_t l2_policy(bool keep) {
    uint64_t pol;
    if (keep) asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    else asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// One tile (bytes: a multiple of 16, at most kTileBytes) global -> shared,
// completing on `bar` (which expects the bytes).
__device__ __forceinline__ void load_tile(float* dst, const float* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// The same without the time that try_wait may take over it.
__device__ __forceinline__ bool mbar_done(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of `bar`; false if it gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned limit = kWaitLimit) {
    for (unsigned k = 0; k < limit; ++k)
        if (mbar_test(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Failure-path test (PcgScalars::wait_first > 0): the CTA's first wait polls
// `never`, an mbarrier no thread or copy ever completes, wait_first times and
// gives up, exercising the give-up / drain / report path with every copy issued.
__device__ __forceinline__ bool first_wait_test(int n, uint64_t* never) {
    return n > 0 ? mbar_wait(never, 0u, (unsigned)n) : true;
}
__device__ __forceinline__ bool first_wait_test(const XSrc& xs, uint64_t* never) {
    return first_wait_test(xs.sc ? xs.sc->wait_first : 0, never);
}

// Shape of a listed tile: rows, padded width (floats per row of a rectangle),
// diagonal (padded triangle), bytes.
struct TileShape {
    int h, wp;
    bool diag, full;
    uint32_t bytes;
};

// Shape of the tile of list entry word e0, from the subdomain's descriptor.
__device__ __forceinline__ TileShape tile_shape(const SymDesc& sd, uint32_t e) {
    const int a = (int)(e >> 16), b = (int)((e >> 3) & 0x1fff);
    const bool diag = (e & 4) != 0;
    TileShape t;
    t.h = sym_h(sd, a);
    const int w = sym_h(sd, b);
    t.wp = (w + 3) & ~3;
    t.diag = diag;
    t.full = !diag && t.h == kSymT && w == kSymT;
    t.bytes = 4u * (uint32_t)sym_tile_floats(t.h, w, diag);
    return t;
}

// First word of list entry k (the tile's rows, columns and roles): from the
// CTA's copy in shared memory (LSM) or, read-only, from the mode's list in
// global memory.
template <bool LSM>
__device__ __forceinline__ uint32_t tl_word(const uint32_t* tl, int k) {
    return LSM ? tl[kTlW * k] : __ldg(tl + kTlW * k);
}

// Issue the bulk copy of list entry k.
template <bool LSM = false>
__device__ __forceinline__ void issue_tile(const uint32_t* tl, int k, const SymDesc& sd, const float* tiles, float* dst,
                                           uint64_t* bar, uint64_t pol) {
    const uint32_t e0 = tl_word<LSM>(tl, k), e1 = LSM ? tl[kTlW * k + 1] : __ldg(tl + kTlW * k + 1);
    load_tile(dst, tiles + e1, tile_shape(sd, e0).bytes, bar, pol);
}

// First padded position a mode touches (the I run only when I is in the mask).
__host__ __device__ inline int mask_lo(const SymDesc& sd, int mask) { return (mask & 1) ? 0 : kSymT * sd.tI; }

}  // namespace
