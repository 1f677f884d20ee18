// The whole interface solve of a small tearing in one kernel, with the operators resident
// in shared memory (sm_103a, one problem): the coupled GMRES of DD_MIXED (k_gm_resident)
// and the Schur CG of both precisions (k_cg_resident, further below).
//
// GMRES.  On small tearings every kernel of an Arnoldi step (operator GEMV, two Gram-Schmidt
// passes, normalisation; gmres.cu) runs for 2 to 11 us of launch, load and reduction
// latency over a few kilobytes per SM.  Here one CTA holds one subdomain: the packed
// FP32 tiles of its [Gamma | c] block are copied to shared memory once per solve, and the
// Krylov vectors at its own interface entries (both sides of a multiplier keep the same
// values) live there too.  What an Arnoldi step still exchanges through global memory is
// w = M_s x at the interface entries and two sets of dot products, with one grid barrier
// after each:
//   1. y = M_s z from shared memory, w published                              barrier
//   2. t = jump of w (corner assembly, or the DP2 combination), h1 = V^T t      barrier
//   3. t -= V h1, h2 = V^T t, ||t||^2                                          barrier
//   then H[:, j] = h1 + h2, H[j+1][j] = sqrt(||t||^2 - ||h2||^2), v_{j+1} = (t - V h2) /
//   H[j+1][j]: every CTA on its own entries, from the same totals.
// A seventeenth warp works on the Givens rotations and the end-of-cycle decision while the
// other sixteen already multiply by the new vector (the last product of a cycle is
// dropped).  Every CTA adds the partial sums in the same fixed order, so all of them
// take the same decisions and the result does not depend on scheduling.  Algorithm,
// precisions and stopping rules are those of gmres.cu: FP32 vectors, dot products in FP32 up
// to 128 entries and beyond as in FP64 (sum2.h, partial_sum), FP64 least-squares problem and
// iterate.
//
// Measured (GB300, FP32 solve of a step): 9.3 us per Arnoldi step on 128 subdomains with up
// to 288 interface entries, 26 us as separate kernels in a graph (GEMV 10, Gram-Schmidt 6.7
// + 6.7, normalisation 2.5).  Whole mixed graph steps, separate / resident: 8 subdomains of
// 448 unknowns 0.80 / 0.40 ms, 64 of 604 0.93 / 0.50, 512 of 98 1.09 / 0.58, 216 of 279
// 0.89 / 0.51; no measured tearing that fits was slower.  The bound is the latency of the
// three barriers and of the loads after them (about 2 us each).
//
// Barriers: up to eight subdomains form one thread-block cluster and use its hardware
// barrier (0.3 us against 1.2); more make a cooperative launch and meet at a counter in
// global memory.  Every wait on memory is bounded: a barrier or copy wait that gives up
// sets the error word and the CTA ends; the others then run into their own limits (a
// cluster barrier does not wait for threads that have ended).
#include <cuda_runtime.h>

#include <algorithm>

#include "cg_rows.h"
#include "dd_internal.h"
#include "sum2.h"
#include "symtile.cuh"

namespace {

constexpr int kM1 = kMaxRestart + 1;
constexpr unsigned kBarLimit = 1u << 19;   // polls of one grid barrier (about half a second)

inline cudaStream_t S(void* s) { return (cudaStream_t)s; }

struct ResArgs {
    UView U;
    const SymDesc* descs;
    const float* Msym;
    const int32_t* slot_mult;
    const int32_t* slot_corner;
    const int32_t* slot_upos;
    float* wf;            // published w, in multiplier / corner-copy order
    float* zuf;           // published z (DP2)
    GmresScalars* gs;
    PcgScalars* sc;
    double* partials;     // [2][kM1 + 1][gridDim.x] of two FP32 words, then [2][gridDim.x] in FP64
    int span, tile_floats, have_q, clustered;
};

// Shared memory of one CTA with W product warps, in bytes.
size_t res_smem(int W, int span, int tile_floats, int m) {
    return sizeof(float) * ((size_t)tile_floats + (size_t)span * (2 + W + m + 1));
}

// What the CTAs meet at: the counter in global memory, or (bar null) the cluster.
struct Meet {
    uint32_t* bar;
    uint32_t target;
    int32_t* err;
    int* failed;   // shared memory
    int first;     // thread 0: PcgScalars::wait_first (> 0: wait, this many polls long, for an arrival nobody makes)
};

// Grid barrier: writes of the product warps (W > 0: only these are waited for before the
// arrival, the last warp joins at the end; W = 0: of all threads) before it are visible to
// every CTA's L2 loads (__ldcg) after it.  False when it gave up.
template <int W>
__device__ bool grid_barrier(Meet& m) {
    if (!m.bar) {
        asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
        return true;
    }
    m.target += gridDim.x;
    if constexpr (W == 0) __syncthreads();
    else if (threadIdx.x < 32 * W) asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(m.bar, 1u);
        const uint32_t target = m.target + (m.first > 0 ? 1u : 0u);
        const unsigned limit = m.first > 0 ? (unsigned)m.first : kBarLimit;
        unsigned k = 0;
        uint32_t v;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(m.bar) : "memory");
        } while (v < target && ++k < limit);
        if (v < target) {
            *m.failed = 1;
            atomicExch(m.err, 1);
        }
        __threadfence();
    }
    __syncthreads();
    return *m.failed == 0;
}

// The wait for the copy of the tiles, by every thread of the CTA (first: thread 0's
// PcgScalars::wait_first).  False, in every thread, when it gave up; the copy has then been
// given a second wait, so that it does not land in a CTA that has ended.
__device__ bool tiles_landed(uint64_t* bar, uint64_t* never, int first, int32_t* err, int* failed) {
    const bool ok = first_wait_test(first, never) && mbar_wait(bar, 0u);
    if (!ok) {
        *failed = 1;
        atomicExch(err, 1);
        mbar_wait(bar, 0u);
    }
    __syncthreads();
    return *failed == 0;
}

// Sum of nb partial sums of two FP32 words each (a warp; lanes take q = lane, lane + 32, ...)
// as an integer in units of 2^(*e - shift): exact down to 2^-53 (up to 512 CTAs; 2^-50
// beyond) of the largest, like an FP64 sum but off the two-lane FP64 pipe.  *e = 255 when
// one is not finite.
__device__ __forceinline__ long long partial_sum(const float2* part, int nb, int lane, int shift, int* e) {
    uint32_t mx = 0;
    for (int q = lane; q < nb; q += 32) mx = max(mx, __float_as_uint(__ldcg(part + q).x) & 0x7fffffffu);
    mx = __reduce_max_sync(0xffffffffu, mx);
    const int em = (int)(mx >> 23);
    *e = em;
    auto units = [&](float f) -> long long {
        const uint32_t w = __float_as_uint(f);
        const int x = (int)((w >> 23) & 255u);
        const long long t = x ? (long long)((w & 0x7fffffu) | 0x800000u) : 0ll;   // subnormals count as zero
        const int sh = shift - (em - x);
        const long long u = sh >= 0 ? t << sh : (sh > -24 ? t >> -sh : 0ll);
        return (int32_t)w < 0 ? -u : u;
    };
    long long v = 0;
    for (int q = lane; q < nb; q += 32) {
        const float2 f = __ldcg(part + q);
        v += units(f.x) + units(f.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Tiles of the [Gamma | c] block (the subdomain's first run): (a, c) and float offsets; returns
// the floats in all.  One thread.
__device__ int tile_table(const SymDesc& sd, int* tile_ab, int* tile_off) {
    int off = 0, q = 0;
    for (int a = 0; a < sd.nt - sd.tI; ++a)
        for (int c = 0; c <= a; ++c, ++q) {
            tile_ab[q] = a | (c << 8);
            tile_off[q] = off;
            off += sym_tile_floats(sym_h(sd, sd.tI + a), sym_h(sd, sd.tI + c), a == c);
        }
    return off;
}

// y = S x over tiles [q0, nT) of a subdomain's [Gamma | c] block in shared memory, by W
// product warps, into one partial y per warp (yw): warp (group, w4) takes rows 16 w4 ..
// + 15 of the group's tiles, lane (rg, cq) rows 8 rg .. + 7 of those and columns 4 cq .. + 3.
template <int W>
__device__ __forceinline__ void tile_product(const SymDesc& sd, const float* tiles, const int* tile_ab,
                                             const int* tile_off, int q0, int nT, const float* xg, float* yw, int span) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= W) return;
    float* yc = yw + warp * span;
    for (int p = lane; p < span; p += 32) yc[p] = 0.0f;
    __syncwarp();
    const int w4 = warp & 3, rg = lane >> 4, cq = lane & 15, row0 = 16 * w4 + 8 * rg;
    for (int q = q0 + (warp >> 2); q < nT; q += W / 4) {
        const int a = tile_ab[q] & 255, c = tile_ab[q] >> 8;
        TileShape ts;
        ts.h = sym_h(sd, sd.tI + a);
        ts.wp = (sym_h(sd, sd.tI + c) + 3) & ~3;
        ts.diag = a == c;
        const float* T = tiles + tile_off[q];
        const float4 xb = *reinterpret_cast<const float4*>(xg + c * kSymT + 4 * cq);
        float acc[8];
        float4 col = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int row = row0 + r;
            float4 mm = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (row < ts.h) {
                if (ts.diag) {
                    if (4 * cq < sym_rowlen(row)) mm = *reinterpret_cast<const float4*>(T + sym_trioff(row) + 4 * cq);
                } else if (4 * cq < ts.wp) {
                    mm = *reinterpret_cast<const float4*>(T + row * ts.wp + 4 * cq);
                }
            }
            const float xa = xg[a * kSymT + row];
            acc[r] = fmaf(mm.x, xb.x, fmaf(mm.y, xb.y, fmaf(mm.z, xb.z, mm.w * xb.w)));
            col.x = fmaf(mm.x, xa, col.x);
            col.y = fmaf(mm.y, xa, col.y);
            col.z = fmaf(mm.z, xa, col.z);
            col.w = fmaf(mm.w, xa, col.w);
        }
        // rows: halving exchanges over the 16 column quads; lane pair (cq / 2) ends with one row
        float v4[4], v2[2];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const bool hi = (cq & 8) != 0;
            v4[r] = (hi ? acc[r + 4] : acc[r]) + __shfl_xor_sync(0xffffffffu, hi ? acc[r] : acc[r + 4], 8);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const bool hi = (cq & 4) != 0;
            v2[r] = (hi ? v4[r + 2] : v4[r]) + __shfl_xor_sync(0xffffffffu, hi ? v4[r] : v4[r + 2], 4);
        }
        const bool hi = (cq & 2) != 0;
        float v = (hi ? v2[1] : v2[0]) + __shfl_xor_sync(0xffffffffu, hi ? v2[0] : v2[1], 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        if (!(cq & 1)) yc[a * kSymT + row0 + ((cq & 8) ? 4 : 0) + ((cq & 4) ? 2 : 0) + ((cq & 2) ? 1 : 0)] += v;
        // columns: the warp's two row groups
        col.x += __shfl_xor_sync(0xffffffffu, col.x, 16);
        col.y += __shfl_xor_sync(0xffffffffu, col.y, 16);
        col.z += __shfl_xor_sync(0xffffffffu, col.z, 16);
        col.w += __shfl_xor_sync(0xffffffffu, col.w, 16);
        __syncwarp();
        if (lane < 16) {
            float4* yp = reinterpret_cast<float4*>(yc + c * kSymT + 4 * cq);
            float4 y = *yp;
            y.x += col.x;
            y.y += col.y;
            y.z += col.z;
            y.w += col.w;
            *yp = y;
        }
        __syncwarp();
    }
}

// W product warps (groups of four taking alternate tiles) and the warp of the small dense
// problem; one interface entry per thread.
template <int W>
__global__ void __launch_bounds__(32 * W + 32, 16 / W) k_gm_resident(ResArgs P) {
    constexpr int kW = W, kT = 32 * W + 32;
    extern __shared__ __align__(128) float sm[];
    float* tiles = sm;
    float* xg = tiles + P.tile_floats;   // [span] operator input
    float* tm = xg + P.span;             // [span] t, zero where another CTA counts the entry
    float* yw = tm + P.span;             // [kW][span] partial products per warp
    float* V = yw + kW * P.span;         // [m + 1][span] Krylov basis at the CTA's entries
    __shared__ double sH[kMaxRestart * kM1];
    __shared__ double scs[kMaxRestart], ssn[kMaxRestart], sg[kM1], sy[kMaxRestart];
    __shared__ double h1[kM1 + 1], h2[kM1 + 1];   // totals of the two passes, and in FP32
    __shared__ float h1f[kM1 + 1], h2f[kM1 + 1], syf[kMaxRestart];
    __shared__ long long isum[kM1 + 1];
    __shared__ int iexp[kM1 + 1];
    __shared__ double red[2][kT / 32];
    __shared__ double shnext, sresid, s_beta, s_bnorm, s_thr;
    __shared__ float sinv;
    __shared__ int s_end, s_final, s_k, s_conv, s_status, s_it, s_fail;
    __shared__ uint64_t bar_tiles, never;
    __shared__ int tile_ab[64], tile_off[64];

    const UView& U = P.U;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = gridDim.x, b = blockIdx.x;
    const SymDesc sd = P.descs[b];
    const int g = sd.n[1] + sd.n[2], nG = sd.nt - sd.tI, nT = nG * (nG + 1) / 2;
    GmresScalars* gs = P.gs;
    const int m = gs->m, max_it = gs->max_it;
    const double tol = gs->tol;
    const int first_polls = tid == 0 ? P.sc->wait_first : 0;
    Meet meet{P.clustered ? nullptr : &gs->bar, 0u, &P.sc->wait_err, &s_fail, first_polls};

    // the tiles of the [Gamma | c] block: the subdomain's first run
    if (tid == 0) {
        s_fail = 0;
        s_it = 0;
        s_status = DD_OK;
        const int off = tile_table(sd, tile_ab, tile_off);
        mbar_init(&bar_tiles, 1);
        mbar_init(&never, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        load_tile(tiles, P.Msym + sd.toff, 4u * (uint32_t)off, &bar_tiles, l2_policy(true));
    }
    for (int p = tid; p < P.span; p += kT) xg[p] = tm[p] = 0.0f;
    // this thread's entry
    const int e = tid;
    const bool on = e < g;
    int64_t ui = 0, k0 = 0, k1 = 0;   // index in u; corner copies, or the M_T row (DP2)
    int up = 0, side = 0;
    bool own = false, corner = false;
    float sgn = 0.0f;
    double dinv = 0.0, rhs = 0.0, xs = 0.0;
    double* xp = nullptr;
    float* xpf = nullptr;
    if (on) {
        const int64_t slot = sd.voff + sd.n[0] + e;
        const int mu = P.slot_mult[slot];
        up = P.slot_upos[slot];
        corner = mu == 0;
        if (!corner) {
            const int64_t k = (mu > 0 ? mu : -mu) - 1;
            side = mu > 0 ? 0 : 1;
            const bool second = U.n2 > 0 && side == 1;   // DP2: the second side has its own unknown
            ui = second ? U.n1 + k : k;
            own = U.n2 > 0 || side == 0;
            sgn = (U.n2 > 0 || side == 0) ? 1.0f : -1.0f;
            if (U.n2 > 0) {
                k0 = U.mtp[k];
                k1 = U.mtp[k + 1];
            }
            dinv = (!second && U.d1) ? U.d1[k] : 1.0;
            rhs = second ? U.b2[k] : U.b1[k];
            xp = (second ? U.x2 : U.x1) + k;
            xpf = (second ? U.x2f : U.x1f) + k;
        } else {
            const int64_t c = P.slot_corner[slot];
            ui = U.n1 + U.n2 + c;
            k0 = U.cp[c];
            k1 = U.cp[c + 1];
            own = U.cs[k0] == slot;
            sgn = U.n2 > 0 ? 1.0f : -1.0f;
            dinv = U.dc ? U.dc[c] : 1.0;
            rhs = U.bc[c];
            xp = U.xc + c;
            xpf = U.xcf + c;
        }
        xs = *xp;
    }
    const float dinvf = (float)dinv;
    const int nw = (g + 31) >> 5;   // warps with entries
    __syncthreads();
    if (!tiles_landed(&bar_tiles, &never, first_polls, &P.sc->wait_err, &s_fail)) return;

    auto product = [&]() { tile_product<kW>(sd, tiles, tile_ab, tile_off, 0, nT, xg, yw, P.span); };
    // this entry's row of M_s x, published (the corner rows of M = J S change sign)
    auto publish = [&]() {
        if (!on) return;
        float y = 0.0f;
#pragma unroll
        for (int w = 0; w < kW; ++w) y += yw[w * P.span + e];
        P.wf[up] = corner ? -y : y;
    };
    // (M u) of this entry from the published w (and, for DP2, the unknowns of both sides); a DP1
    // multiplier's jump is one FP32 subtraction (the FP64 pipe takes 16 clocks per warp instruction)
    float jump = 0.0f;
    auto combined = [&](bool residual) -> double {
        jump = 0.0f;
        const int64_t wc = 2 * U.n1;
        if (corner) {
            double s = 0.0;
            for (int64_t k = k0; k < k1; ++k) s += (double)__ldcg(P.wf + wc + k);
            return U.n2 > 0 ? s : -s;
        }
        const int64_t k = side && U.n2 > 0 ? ui - U.n1 : ui;
        if (U.n2 == 0) {
            const float2 w = __ldcg(reinterpret_cast<const float2*>(P.wf) + k);
            jump = w.x - w.y;
            return 0.0;
        }
        const int other = side == 0 ? 1 : 0;
        double acc = 0.0;
        for (int64_t p = k0; p < k1; ++p) acc += U.mtv[p] * (double)__ldcg(P.wf + 2 * (int64_t)U.mtc[p] + other);
        const double in = residual ? __ldcg(U.x1 + k) + __ldcg(U.x2 + k)
                                   : (double)__ldcg(P.zuf + k) + (double)__ldcg(P.zuf + U.n1 + k);
        return in - U.two_alpha * acc;
    };
    // dots of tm with v_0 .. v_{nv-1}, and with itself as sum nv when `norm`: this CTA's partial
    // sums (set s), then the totals over the grid
    const int shift = nb <= 512 ? 29 : 26;
    auto dots = [&](int s, int nv, bool norm, double* tot, float* totf) -> bool {
        const int nsum = nv + (norm ? 1 : 0);
        float2* part = reinterpret_cast<float2*>(P.partials) + (size_t)s * (kM1 + 1) * nb;
        for (int k = warp; k < nsum; k += kW + 1) {
            const float* v = k < nv ? V + k * P.span : tm;
            Sum2 p{0.0f, 0.0f};
            for (int q0 = 0; q0 < g; q0 += 128) {   // (no more than 128 products in FP32)
                float f = 0.0f;
#pragma unroll
                for (int q = q0 + lane; q < q0 + 128; q += 32)
                    if (q < g) f = fmaf(tm[q], v[q], f);
                p = sum2_add(p, Sum2{f, 0.0f});
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                p = sum2_add(p, Sum2{__shfl_xor_sync(0xffffffffu, p.hi, o), __shfl_xor_sync(0xffffffffu, p.lo, o)});
            if (lane == 0) part[(size_t)k * nb + b] = make_float2(p.hi, p.lo);
        }
        if (!grid_barrier<0>(meet)) return false;
        for (int k = warp; k < nsum; k += kW + 1) {
            int ex;
            const long long v = partial_sum(part + (size_t)k * nb, nb, lane, shift, &ex);
            if (lane == 0) {
                isum[k] = v;
                iexp[k] = ex;
            }
        }
        __syncthreads();
        if (tid < nsum) {   // (one or two warps: the conversions run on the FP64 pipe)
            const int ex = iexp[tid];
            const double v = ex == 255 ? __longlong_as_double(0x7ff8000000000000ll)
                                       : (double)isum[tid] * __longlong_as_double((long long)(ex - 150 - shift + 1023) << 52);
            tot[tid] = v;
            totf[tid] = (float)v;
        }
        __syncthreads();
        return true;
    };

    bool warm = P.have_q != 0;
    for (int cycle = 0;; ++cycle) {
        // residual r = b - M x, its norm and ||b||
        float t = 0.0f;
        if (warm) {
            if (on) xg[e] = sgn * (float)xs;
            __syncthreads();
            product();
            __syncthreads();
            publish();
            if (!grid_barrier<0>(meet)) return;
        }
        if (on) {
            const double mu = warm ? combined(true) : 0.0;
            t = (float)(rhs - (mu + (double)jump));   // (one of the two is zero)
        }
        warm = true;
        {
            const bool mine = on && own;
            if (warp < nw) {
                const double rr = warp_sum(mine ? (double)t * (double)t : 0.0), bb = warp_sum(mine ? rhs * rhs : 0.0);
                if (lane == 0) {
                    red[0][warp] = rr;
                    red[1][warp] = bb;
                }
            }
            __syncthreads();
            double* part = P.partials + (size_t)2 * (kM1 + 1) * nb;   // past the FP32 sets
            if (tid < 2) {
                double v = 0.0;
                for (int w = 0; w < nw; ++w) v += red[tid][w];
                part[(size_t)tid * nb + b] = v;
            }
            if (!grid_barrier<0>(meet)) return;
            if (warp < 2) {
                double v = 0.0;
                for (int q = lane; q < nb; q += 32) v += __ldcg(part + (size_t)warp * nb + q);
                v = warp_sum(v);
                if (lane == 0) red[warp][0] = v;
            }
            __syncthreads();
        }
        if (tid == 0) {
            const double beta = sqrt(red[0][0]), bnorm = sqrt(red[1][0]);
            const bool finite = isfinite(beta) && isfinite(bnorm);
            s_beta = beta;
            s_bnorm = bnorm;
            s_thr = tol * bnorm;
            sg[0] = sresid = shnext = beta;
            sinv = (float)(1.0 / beta);
            s_k = 0;
            s_conv = finite && beta <= s_thr ? 1 : 0;
            s_status = finite ? DD_OK : DD_ERR_NONFINITE;
            s_end = s_final = (!finite || s_conv || s_it >= max_it) ? 1 : 0;
        }
        __syncthreads();
        for (int j = 0; !(j == 0 && s_end); ++j) {
            // v_j = t / H[j][j-1], z = D^-1 v_j, w = M_s z; the rotations of column j - 1 meanwhile
            if (warp < kW) {
                if (on) {
                    const float v = t * sinv, z = dinvf * v;
                    V[j * P.span + e] = v;
                    xg[e] = sgn * z;
                    if (U.n2 > 0) P.zuf[ui] = z;   // (corners: not read back)
                }
                asm volatile("bar.sync 1, %0;" ::"n"(32 * kW) : "memory");
                product();
                asm volatile("bar.sync 1, %0;" ::"n"(32 * kW) : "memory");
                publish();
            } else if (j > 0 && lane == 0) {
                const int c = j - 1;
                double* col = sH + c * kM1;
                for (int i = 0; i <= c; ++i) col[i] = h1[i] + h2[i];
                col[c + 1] = shnext;
                for (int i = 0; i < c; ++i) {
                    const double x = col[i], y = col[i + 1];
                    col[i] = scs[i] * x + ssn[i] * y;
                    col[i + 1] = -ssn[i] * x + scs[i] * y;
                }
                double cs = 1.0, sn = 0.0;
                const double r = hypot(col[c], col[c + 1]);
                if (r != 0.0) {
                    cs = col[c] / r;
                    sn = col[c + 1] / r;
                }
                col[c] = cs * col[c] + sn * col[c + 1];
                col[c + 1] = 0.0;
                scs[c] = cs;
                ssn[c] = sn;
                sg[c + 1] = -sn * sg[c];
                sg[c] = cs * sg[c];
                const int it = ++s_it;
                const double resid = fabs(sg[c + 1]);
                const bool fin = isfinite(resid) && isfinite(shnext) && isfinite(col[c]);
                const bool conv = fin && resid <= s_thr;
                sresid = resid;
                s_conv = conv ? 1 : 0;
                s_final = (!fin || conv || it >= max_it) ? 1 : 0;
                if (!fin) s_status = DD_ERR_NONFINITE;
                s_k = fin ? c + 1 : 0;
                s_end = (s_final || c + 1 == m || shnext == 0.0) ? 1 : 0;
                if (s_end)
                    for (int i = s_k - 1; i >= 0; --i) {
                        double v = sg[i];
                        for (int l = i + 1; l < s_k; ++l) v -= sH[l * kM1 + i] * sy[l];
                        sy[i] = v / sH[i * kM1 + i];
                        syf[i] = (float)sy[i];
                    }
            }
            if (!grid_barrier<W>(meet)) return;
            if (s_end) break;   // (the same decision in every CTA; this product is dropped)
            const int nv = j + 1;
            t = 0.0f;
            if (on) {
                const double mu = combined(false);
                t = corner || U.n2 > 0 ? (float)mu : jump;
            }
            if (on) tm[e] = own ? t : 0.0f;
            __syncthreads();
            if (!dots(0, nv, false, h1, h1f)) return;
            if (on) {
                for (int k = 0; k < nv; ++k) t -= h1f[k] * V[k * P.span + e];
                tm[e] = own ? t : 0.0f;
            }
            __syncthreads();
            if (!dots(1, nv, true, h2, h2f)) return;
            if (warp == kW) {
                const double q = lane < nv ? h2[lane] : 0.0;   // nv <= 32
                const double sq = warp_sum(q * q);
                if (lane == 0) {
                    shnext = sqrt(fmax(h2[nv] - sq, 0.0));
                    sinv = (float)(1.0 / shnext);
                }
            } else if (on) {
                for (int k = 0; k < nv; ++k) t -= h2f[k] * V[k * P.span + e];
            }
            __syncthreads();
        }
        // x += D^-1 V y
        if (on && s_k > 0) {
            float vs = 0.0f;
            for (int q = 0; q < s_k; ++q) vs += syf[q] * V[q * P.span + e];
            xs += (double)vs * dinv;
            if (own) {
                *xp = xs;
                *xpf = (float)xs;
            }
        }
        if (b == 0 && tid == 0) {
            gs->bnorm = s_bnorm;
            gs->thr = s_thr;
            gs->beta = s_beta;
            gs->resid = sresid;
            if (s_final) {
                gs->it = P.sc->it = s_it;
                gs->converged = P.sc->done = s_conv;
                gs->status = P.sc->status = s_status;
                gs->cycles = cycle + 1;
                gs->final = 1;
                P.sc->it_total += s_it;
                P.sc->cycles += cycle + 1;
                P.sc->rr = sresid * sresid;
                P.sc->gg = s_bnorm * s_bnorm;
            }
        }
        __syncthreads();
        if (s_final) return;
        __syncthreads();   // s_final was read; the next cycle rewrites it
    }
}

// ---- Schur CG -------------------------------------------------------------------
// CG on Eq. f1schur (k_pcg_* in kernels.cu: same recurrences, precisions and stopping rule;
// T is the type of the operator and its input, everything else FP64).  One CTA per
// subdomain holds its [Gamma | c] block: packed FP32 tiles, or the dense FP64 rows.  One
// application of the operator is
//   u = corner rows of M_s B_r^T p, published                                   barrier
//   v = K~cc^-1 sum_s u: every CTA assembles sum u and does its share of the rows  barrier
//   w = interface rows of M_s [B_r^T p; -v], published                          barrier
// and an iteration adds the barriers of p.q and of r.r, r.z.  Measured, FP64 step with the
// library's defaults on 8 subdomains of 448 unknowns: 1.15 ms as seven launches per
// iteration polled every eight, 0.45 ms here (21 us per iteration: the five exchanges and
// the FP64 products, 17,000 FMAs per CTA at two per clock).
struct CgArgs {
    const SymDesc* descs;
    const MatDesc* mats;
    const float* Msym;
    const double* M;
    const int32_t* slot_mult;
    const int32_t* slot_corner;
    const int32_t* slot_upos;
    const int64_t* cp;        // corner copies
    const double* g;          // right-hand side
    const double* dinv;       // null: no preconditioner
    double* lam;
    float* lamf;
    const void* K;            // K~cc^-1 in T, row stride ldc
    void* w;                  // published w in T (multiplier / corner-copy order), v
    void* v;
    PcgScalars* sc;
    uint32_t* bar;
    double* partials;         // [kCgRows][gridDim.x]
    double tol, refine_tol;
    int64_t nl;
    int nc, ldc, ld, span, floats, have_q, adaptive, max_it, clustered;
};

// Shared memory of one CTA: the block (FP32 tiles with x and W partial y, or dense FP64 rows with x
// and y) and the assembled corner vector.
size_t cg_smem(bool f32, int W, int span, int floats, int g, int ld, int nc) {
    return f32 ? sizeof(float) * ((size_t)floats + (size_t)span * (1 + W)) + sizeof(double) * (size_t)nc
               : sizeof(double) * ((size_t)g * ld + 2 * (size_t)span + nc);
}

template <typename T, int W>
__global__ void __launch_bounds__(32 * W, W == 16 ? 1 : 2) k_cg_resident(CgArgs P) {
    constexpr bool kF32 = sizeof(T) == 4;
    constexpr int kT = 32 * W;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ double red[3][W];
    __shared__ double s_rz, s_gg, s_rr, s_tol2, s_alpha, s_beta;
    __shared__ int s_done, s_finite;
    __shared__ int s_fail, tile_ab[64], tile_off[64];
    __shared__ uint64_t bar_tiles, never;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = gridDim.x, b = blockIdx.x;
    const SymDesc sd = P.descs[b];
    const MatDesc md = P.mats[b];
    const int nGam = sd.n[1], g = nGam + sd.n[2], nG = sd.nt - sd.tI, nT = nG * (nG + 1) / 2;
    // FP32: tiles | x | y per warp | uc;  FP64: rows | x | y | uc
    float* tiles = reinterpret_cast<float*>(smem);
    double* rows = reinterpret_cast<double*>(smem);
    T* xg = kF32 ? reinterpret_cast<T*>(tiles + P.floats) : reinterpret_cast<T*>(rows + (size_t)P.ld * P.floats);
    T* yg = xg + P.span;
    double* uc = reinterpret_cast<double*>(yg + (kF32 ? W : 1) * P.span);
    T* w = reinterpret_cast<T*>(P.w);
    T* vC = reinterpret_cast<T*>(P.v);
    const T* K = reinterpret_cast<const T*>(P.K);
    const int first_polls = tid == 0 ? P.sc->wait_first : 0;
    Meet meet{P.clustered ? nullptr : P.bar, 0u, &P.sc->wait_err, &s_fail, first_polls};
    if (tid == 0) s_fail = 0;
    if constexpr (kF32) {
        if (tid == 0) {
            const int off = tile_table(sd, tile_ab, tile_off);
            mbar_init(&bar_tiles, 1);
            mbar_init(&never, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            load_tile(tiles, P.Msym + sd.toff, 4u * (uint32_t)off, &bar_tiles, l2_policy(true));
        }
    } else {
        const double* src = P.M + md.moff + (int64_t)sd.n[0] * md.ld + sd.n[0];
        for (int i = warp; i < g; i += W)
            for (int j = lane; j < g; j += 32) rows[(size_t)i * P.ld + j] = src[(int64_t)i * md.ld + j];
    }
    for (int p = tid; p < P.span; p += kT) xg[p] = (T)0;
    // this thread's entry
    const int e = tid;
    const bool gam = e < nGam, cor = e >= nGam && e < g;
    int64_t mi = 0;
    int up = 0, ci = 0;
    bool own = false;
    double sgn = 0.0, dinv = 1.0, rhs = 0.0, lam = 0.0;
    if (gam || cor) {
        const int64_t slot = sd.voff + sd.n[0] + e;
        up = P.slot_upos[slot];
        if (gam) {
            const int mu = P.slot_mult[slot];
            own = mu > 0;
            mi = (mu > 0 ? mu : -mu) - 1;
            sgn = own ? 1.0 : -1.0;
            rhs = P.g[mi];
            if (P.dinv) dinv = P.dinv[mi];
            lam = P.lam[mi];
        } else {
            ci = P.slot_corner[slot];
        }
    }
    double tol = P.tol;
    if (P.adaptive) {   // a later refinement pass only has to cut the current step residual to refine_tol
        const double resid = P.sc->norm_b2 > 0.0 ? sqrt(P.sc->norm_r2 / P.sc->norm_b2) : 0.0;
        if (resid > 0.0) tol = fmin(0.1, fmax(tol, 0.3 * P.refine_tol / resid));
    }
    __syncthreads();
    if constexpr (kF32) {
        if (!tiles_landed(&bar_tiles, &never, first_polls, &P.sc->wait_err, &s_fail)) return;
    }
    // rows [i0, g) of M_s x; the result of entry e in y(e)
    auto product = [&](int i0) {
        if constexpr (kF32) {
            const int a0 = i0 / kSymT;
            tile_product<W>(sd, tiles, tile_ab, tile_off, a0 * (a0 + 1) / 2, nT, xg, yg, P.span);
        } else {   // four threads per row, every fourth column (rows an odd multiple of four banks apart)
            for (int i = i0 + (tid >> 2); i - (tid >> 2) < g; i += kT / 4) {
                double s0 = 0.0, s1 = 0.0;
                if (i < g) {
                    const double* r = rows + (size_t)i * P.ld;
                    int j = tid & 3;
                    for (; j + 4 < g; j += 8) {
                        s0 = fma(r[j], (double)xg[j], s0);
                        s1 = fma(r[j + 4], (double)xg[j + 4], s1);
                    }
                    if (j < g) s0 = fma(r[j], (double)xg[j], s0);
                }
                s0 += s1;
                s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
                s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
                if (i < g && (tid & 3) == 0) yg[i] = (T)s0;
            }
        }
        __syncthreads();
    };
    auto y = [&]() -> T {
        if constexpr (kF32) {
            T v = (T)0;
#pragma unroll
            for (int k = 0; k < W; ++k) v += yg[k * P.span + e];
            return cor ? -v : v;   // the tiles hold S = J M
        } else {
            return yg[e];
        }
    };
    // q = (Schur operator) x at this thread's interface entry, x in T
    auto apply = [&](T x, double& q) -> bool {
        if (gam) xg[e] = x;
        if (cor) xg[e] = (T)0;
        __syncthreads();
        if (P.nc > 0) {
            product(nGam);
            if (cor) w[up] = y();
            if (!grid_barrier<0>(meet)) return false;
            for (int I = tid; I < P.nc; I += kT) {
                double s = 0.0;
                for (int64_t k = P.cp[I]; k < P.cp[I + 1]; ++k) s += (double)__ldcg(w + 2 * P.nl + k);
                uc[I] = kF32 ? (double)(float)s : s;
            }
            __syncthreads();
            for (int I = b + nb * warp; I < P.nc; I += nb * W) {
                const T* r = K + (int64_t)I * P.ldc;
                T s = (T)0;
                for (int J = lane; J < P.nc; J += 32) s += r[J] * (T)uc[J];
                s = warp_sum(s);
                if (lane == 0) vC[I] = s;
            }
            if (!grid_barrier<0>(meet)) return false;
            if (cor) xg[e] = -__ldcg(vC + ci);
            __syncthreads();
        }
        product(0);
        if (gam) w[up] = y();
        if (!grid_barrier<0>(meet)) return false;
        q = 0.0;
        if (gam) q = (double)__ldcg(w + 2 * mi) - (double)__ldcg(w + 2 * mi + 1);
        return true;
    };
    // the sums R over the multipliers (each counted by its first side), in CTA order, left in
    // red[k][0]; through the rows of the exchange buffer that cg_rows.h gives them
    const int nw = (nGam + 31) >> 5;   // warps with interface entries
    auto sums = [&](CgSums R, double a0, double a1, double a2) -> bool {
        const int n = R.n;
        double v[3] = {own ? a0 : 0.0, own ? a1 : 0.0, own ? a2 : 0.0};
        if (warp < nw)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (k >= n) continue;
                v[k] = warp_sum(v[k]);
                if (lane == 0) red[k][warp] = v[k];
            }
        __syncthreads();
        if (tid < n) {
            double s = 0.0;
            for (int k = 0; k < nw; ++k) s += red[tid][k];
            P.partials[(size_t)(R.row + tid) * nb + b] = s;
        }
        if (!grid_barrier<0>(meet)) return false;
        if (warp < n) {
            double s = 0.0;
            for (int k = lane; k < nb; k += 32) s += __ldcg(P.partials + (size_t)(R.row + warp) * nb + k);
            s = warp_sum(s);
            if (lane == 0) red[warp][0] = s;
        }
        __syncthreads();
        return true;
    };
    // the vector updates run in the warps that hold interface entries, quotients in one thread: the
    // FP64 pipe takes 16 clocks per warp instruction, whatever the lanes hold
    double q = 0.0;
    if (P.have_q && !apply((T)(sgn * lam), q)) return;
    double r = 0.0, z = 0.0, p = 0.0;
    if (warp < nw) {
        r = rhs - q;
        z = r * dinv;
    }
    if (!sums(kCgStart, r * z, rhs * rhs, r * r)) return;
    if (tid == 0) {
        const double a = red[0][0], gg = red[1][0], rr = red[2][0];
        const bool finite = isfinite(a) && isfinite(gg) && isfinite(rr);
        s_rz = a;
        s_gg = gg;
        s_rr = rr;
        s_tol2 = tol * tol * gg;
        s_beta = 0.0;
        s_finite = finite;
        s_done = !finite || rr <= s_tol2;
    }
    __syncthreads();
    int it = 0;
    while (!s_done && it < P.max_it) {
        double pn = 0.0;
        T x = (T)0;
        if (warp < nw) {
            const double beta = s_beta;
            pn = z + beta * p;
            if constexpr (kF32) x = (T)sgn * fmaf((float)beta, (float)p, (float)z);
            else x = (T)(sgn * pn);
        }
        if (!apply(x, q)) return;
        if (!sums(kCgPq, warp < nw ? pn * q : 0.0, 0.0, 0.0)) return;
        if (tid == 0) s_alpha = s_rz / red[0][0];
        __syncthreads();
        if (warp < nw) {
            const double alpha = s_alpha;
            lam += alpha * pn;
            r -= alpha * q;
            z = r * dinv;
            p = pn;
        }
        ++it;
        if (!sums(kCgRes, warp < nw ? r * r : 0.0, warp < nw ? r * z : 0.0, 0.0)) return;
        if (tid == 0) {
            const double rr = red[0][0], rz = red[1][0];
            const bool finite = isfinite(rr) && isfinite(rz) && isfinite(s_alpha);
            s_rr = rr;
            s_finite = finite;
            s_done = !finite || rr <= s_tol2;
            s_beta = rz / s_rz;
            s_rz = rz;
        }
        __syncthreads();
    }
    if (own && it > 0) {
        P.lam[mi] = lam;
        if (kF32) P.lamf[mi] = (float)lam;
    }
    if (b == 0 && tid == 0) {
        PcgScalars* sc = P.sc;
        sc->rz = s_rz;
        sc->gg = s_gg;
        sc->rr = s_rr;
        sc->tol2 = s_tol2;
        sc->it = it;
        sc->it_total += it;
        sc->status = s_finite ? DD_OK : DD_ERR_NONFINITE;
        sc->done = s_done ? 1 : 0;
    }
}

}  // namespace

// Host: largest interface block, its padded entries and its tile floats over the subdomains.
void build_res(dd_handle* h) {
    ResSizes z{0, 0, 0};
    for (const SymDesc& sd : h->sym) {
        z.g = std::max(z.g, sd.n[1] + sd.n[2]);
        z.span = std::max(z.span, (sd.nt - sd.tI) * kSymT);
        int f = 0;
        for (int a = sd.tI; a < sd.nt; ++a)
            for (int c = sd.tI; c <= a; ++c) f += sym_tile_floats(sym_h(sd, a), sym_h(sd, c), a == c);
        z.floats = std::max(z.floats, (f + 31) / 32 * 32);
    }
    h->res = z;
}

namespace {

// Launch of a resident kernel with one CTA per subdomain: all of them on the device at once,
// as one cluster (up to eight) or cooperatively.
struct Launch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    bool clustered = false;
    template <typename Kern>
    bool plan(const dd_handle* h, Kern kern, int threads, size_t smem) {
        cudaFuncAttributes fa;
        if (smem > 227 * 1024) return false;
        if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || smem + fa.sharedSizeBytes > 227 * 1024 ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        cfg.gridDim = dim3((unsigned)h->n_sub);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (h->n_sub <= 8) {
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)h->n_sub;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            int n = 0;
            clustered = cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n >= 1;
            if (clustered) return true;
            cudaGetLastError();
        }
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return (int64_t)per_sm * h->n_sm >= h->n_sub;
    }
};

bool res_candidate(const dd_handle* h) {
    return h->members <= 1 && h->sym_ok && !h->mult_dof.empty() && h->n_sm > 0 && h->res.g <= 512;
}

}  // namespace

// Runs the coupled GMRES (after k_gm_init) in its resident form; *ran = false, and nothing
// launched, where it does not apply or the launch is not to be had.  Sixteen product warps first (one CTA per SM), then
// eight, then four, for the first with which every subdomain finds a CTA of its own.
int launch_gm_resident(const dd_handle* h, const UView& U, int have_q, int m, bool probe, bool* ran, void* stream) {
    *ran = false;
    if (!res_candidate(h)) return 0;
    const ResSizes& z = h->res;
    ResArgs P;
    P.U = U;
    P.descs = h->d.symd;
    P.Msym = h->d.Msym;
    P.slot_mult = h->d.slot_mult;
    P.slot_corner = h->d.slot_corner;
    P.slot_upos = h->d.slot_upos;
    P.wf = h->d.wf;
    P.zuf = h->d.zuf;
    P.gs = h->d.gs;
    P.sc = h->d.sc;
    P.partials = h->d.rpart;
    P.span = z.span;
    P.tile_floats = z.floats;
    P.have_q = have_q;
    for (int W = 16; W >= 4; W /= 2) {
        if (z.g > 32 * W) break;
        auto kern = W == 16 ? k_gm_resident<16> : W == 8 ? k_gm_resident<8> : k_gm_resident<4>;
        Launch L;
        if (!L.plan(h, kern, 32 * W + 32, res_smem(W, z.span, z.floats, m))) continue;
        *ran = true;
        if (probe) return 0;
        P.clustered = L.clustered ? 1 : 0;
        L.cfg.stream = S(stream);
        return launch_or_decline((int)cudaLaunchKernelEx(&L.cfg, kern, P), ran);
    }
    return 0;
}

// Runs the Schur CG in its resident form from lambda (have_q: its product is needed); *ran as above.
int launch_cg_resident(const dd_handle* h, int prec, double tol, int have_q, int adaptive, bool* ran, void* stream) {
    *ran = false;
    const bool f32 = prec == DD_MIXED;
    const int nc = (int)h->corner_dof.size();
    if (!res_candidate(h) || nc > 2048 || (f32 && !h->prm.sym_fp32)) return 0;
    const ResSizes& z = h->res;
    CgArgs P;
    P.descs = h->d.symd;
    P.mats = h->d.mats;
    P.Msym = h->d.Msym;
    P.M = h->d.M64;
    P.slot_mult = h->d.slot_mult;
    P.slot_corner = h->d.slot_corner;
    P.slot_upos = h->d.slot_upos;
    P.cp = h->d.corner_ptr;
    P.g = h->d.g;
    P.dinv = h->prm.precond ? h->d.dinv : nullptr;
    P.lam = h->d.lam;
    P.lamf = h->d.lamf;
    P.K = f32 ? (const void*)h->d.K32 : (const void*)h->d.K64;
    P.w = f32 ? (void*)h->d.wf : (void*)h->d.w;
    P.v = f32 ? (void*)h->d.vCf : (void*)h->d.vC;
    P.sc = h->d.sc;
    P.bar = &h->d.gs->bar;
    P.partials = h->d.rpart;
    P.tol = tol;
    P.refine_tol = h->prm.refine_tol;
    P.nl = (int64_t)h->mult_dof.size();
    P.nc = nc;
    P.ldc = h->ldc;
    P.ld = (z.g + 11) / 16 * 16 + 4;   // >= g, 4 mod 16: the rows of a half-warp start four banks apart
    P.span = z.span;
    P.floats = f32 ? z.floats : z.g;
    P.have_q = have_q;
    P.adaptive = adaptive;
    P.max_it = h->prm.max_it;
    for (int W = 16; W >= 8; W /= 2) {
        if (z.g > 32 * W) break;
        auto kern = f32 ? (W == 16 ? k_cg_resident<float, 16> : k_cg_resident<float, 8>)
                        : (W == 16 ? k_cg_resident<double, 16> : k_cg_resident<double, 8>);
        Launch L;
        if (!L.plan(h, kern, 32 * W, cg_smem(f32, W, z.span, z.floats, z.g, P.ld, nc))) continue;
        P.clustered = L.clustered ? 1 : 0;
        if (!P.clustered) {
            const cudaError_t e = cudaMemsetAsync(P.bar, 0, sizeof(uint32_t), S(stream));
            if (e != cudaSuccess) return (int)e;
        }
        L.cfg.stream = S(stream);
        return launch_or_decline((int)cudaLaunchKernelEx(&L.cfg, kern, P), ran);
    }
    return 0;
}
