// The whole coupled GMRES solve in one cooperative kernel, with the operator resident in
// shared memory (sm_103a; DD_MIXED, one problem).
//
// On small tearings every kernel of an Arnoldi step (operator GEMV, two Gram-Schmidt
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
// precisions and stopping rules are those of gmres.cu: FP32 vectors, FP64 dot totals,
// least-squares problem and iterate.
//
// Measured (GB300, FP32 solve of a step): 9.3 us per Arnoldi step on 128 subdomains with up
// to 288 interface entries, 26 us as separate kernels in a graph (GEMV 10, Gram-Schmidt 6.7
// + 6.7, normalisation 2.5).  Whole mixed graph steps, separate / resident: 8 subdomains of
// 448 unknowns 0.80 / 0.40 ms, 64 of 604 0.93 / 0.50, 512 of 98 1.09 / 0.58, 216 of 279
// 0.89 / 0.51; no measured tearing that fits was slower.  The bound is the latency of the
// three barriers and of the loads after them (about 2 us each).
//
// Every wait is bounded: a barrier or copy wait that gives up sets the error word and the
// CTA ends; the others then run into their own limits.
#include <cuda_runtime.h>

#include <algorithm>

#include "dd_internal.h"
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
    double* partials;     // [2][kM1 + 1][gridDim.x]
    int span, tile_floats, have_q;
};

// Shared memory of one CTA with W product warps, in bytes.
size_t res_smem(int W, int span, int tile_floats, int m) {
    return sizeof(float) * ((size_t)tile_floats + (size_t)span * (2 + W + m + 1));
}

// Grid barrier: writes of the product warps (W > 0: only these are waited for, the last
// warp joins at the end; W = 0: of all threads) before it are visible to every CTA's L2
// loads (__ldcg) after it.  False when it gave up.
template <int W>
__device__ bool grid_barrier(uint32_t* bar, uint32_t target, int32_t* err, int* failed) {
    if constexpr (W == 0) __syncthreads();
    else if (threadIdx.x < 32 * W) asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        unsigned k = 0;
        uint32_t v;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        } while (v < target && ++k < kBarLimit);
        if (v < target) {
            *failed = 1;
            atomicExch(err, 1);
        }
        __threadfence();
    }
    __syncthreads();
    return *failed == 0;
}

// Sum of nb FP32 partial sums (a warp; lanes take q = lane, lane + 32, ...) as an integer in
// units of 2^(*e - shift): exact down to 2^-53 (up to 512 CTAs; 2^-50 beyond) of the
// largest, like an FP64 sum but off the two-lane FP64 pipe.  *e = 255 when one is not finite.
__device__ __forceinline__ long long partial_sum(const float* part, int nb, int lane, int shift, int* e) {
    uint32_t mx = 0;
    for (int q = lane; q < nb; q += 32) mx = max(mx, __float_as_uint(__ldcg(part + q)) & 0x7fffffffu);
    mx = __reduce_max_sync(0xffffffffu, mx);
    const int em = (int)(mx >> 23);
    *e = em;
    long long v = 0;
    for (int q = lane; q < nb; q += 32) {
        const uint32_t w = __float_as_uint(__ldcg(part + q));
        const int x = (int)((w >> 23) & 255u);
        const long long t = x ? (long long)((w & 0x7fffffu) | 0x800000u) : 0ll;   // subnormals count as zero
        const int sh = shift - (em - x);
        const long long u = sh >= 0 ? t << sh : (sh > -24 ? t >> -sh : 0ll);
        v += (int32_t)w < 0 ? -u : u;
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
    __shared__ double shnext, sresid;
    __shared__ float sinv;
    __shared__ int s_end, s_final, s_k, s_conv, s_status, s_it, s_fail;
    __shared__ uint64_t bar_tiles;
    __shared__ int tile_ab[64], tile_off[64];

    const UView& U = P.U;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = gridDim.x, b = blockIdx.x;
    const SymDesc sd = P.descs[b];
    const int g = sd.n[1] + sd.n[2], nG = sd.nt - sd.tI, nT = nG * (nG + 1) / 2;
    GmresScalars* gs = P.gs;
    const int m = gs->m, max_it = gs->max_it;
    const double tol = gs->tol;
    uint32_t* bar = &gs->bar;
    uint32_t target = 0;

    // the tiles of the [Gamma | c] block: the subdomain's first run
    if (tid == 0) {
        s_fail = 0;
        s_it = 0;
        s_status = DD_OK;
        int off = 0, q = 0;
        for (int a = 0; a < nG; ++a)
            for (int c = 0; c <= a; ++c, ++q) {
                tile_ab[q] = a | (c << 8);
                tile_off[q] = off;
                off += sym_tile_floats(sym_h(sd, sd.tI + a), sym_h(sd, sd.tI + c), a == c);
            }
        mbar_init(&bar_tiles, 1);
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
    __syncthreads();
    if (!mbar_wait(&bar_tiles, 0u)) {   // (every thread waits itself)
        s_fail = 1;
        atomicExch(&P.sc->wait_err, 1);
    }
    __syncthreads();
    if (s_fail) return;

    // y = S x over the tiles in shared memory (product warps): warp (group, w4) takes rows 16 w4 ..
    // + 15 of the group's tiles, lane (rg, cq) rows 8 rg .. + 7 of those and columns 4 cq .. + 3
    auto product = [&]() {
        if (warp >= kW) return;
        float* yc = yw + warp * P.span;
        for (int p = lane; p < P.span; p += 32) yc[p] = 0.0f;
        __syncwarp();
        const int w4 = warp & 3, rg = lane >> 4, cq = lane & 15, row0 = 16 * w4 + 8 * rg;
        for (int q = warp >> 2; q < nT; q += kW / 4) {
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
    };
    // this entry's row of M_s x, published (the corner rows of M = J S change sign)
    auto publish = [&]() {
        if (!on) return;
        float y = 0.0f;
#pragma unroll
        for (int w = 0; w < kW; ++w) y += yw[w * P.span + e];
        P.wf[up] = corner ? -y : y;
    };
    // (M u) of this entry from the published w (and, for DP2, the unknowns of both sides)
    auto combined = [&](bool residual) -> double {
        const int64_t wc = 2 * U.n1;
        if (corner) {
            double s = 0.0;
            for (int64_t k = k0; k < k1; ++k) s += (double)__ldcg(P.wf + wc + k);
            return U.n2 > 0 ? s : -s;
        }
        const int64_t k = side && U.n2 > 0 ? ui - U.n1 : ui;
        if (U.n2 == 0) {
            const float2 w = __ldcg(reinterpret_cast<const float2*>(P.wf) + k);
            return (double)w.x - (double)w.y;
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
        float* part = reinterpret_cast<float*>(P.partials) + (size_t)s * (kM1 + 1) * nb;
        for (int k = warp; k < nsum; k += kW + 1) {
            const float* v = k < nv ? V + k * P.span : tm;
            float p = 0.0f;
            for (int q = lane; q < g; q += 32) p = fmaf(tm[q], v[q], p);
            p = warp_sum(p);
            if (lane == 0) part[(size_t)k * nb + b] = p;
        }
        if (!grid_barrier<0>(bar, target += nb, &P.sc->wait_err, &s_fail)) return false;
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
            if (!grid_barrier<0>(bar, target += nb, &P.sc->wait_err, &s_fail)) return;
        }
        if (on) t = (float)(rhs - (warm ? combined(true) : 0.0));
        warm = true;
        {
            const bool mine = on && own;
            const double rr = warp_sum(mine ? (double)t * (double)t : 0.0), bb = warp_sum(mine ? rhs * rhs : 0.0);
            if (lane == 0) {
                red[0][warp] = rr;
                red[1][warp] = bb;
            }
            __syncthreads();
            double* part = P.partials + (size_t)(kM1 + 1) * nb;   // past the FP32 sets
            if (tid < 2) {
                double v = 0.0;
                for (int w = 0; w < kT / 32; ++w) v += red[tid][w];
                part[(size_t)tid * nb + b] = v;
            }
            if (!grid_barrier<0>(bar, target += nb, &P.sc->wait_err, &s_fail)) return;
            if (warp < 2) {
                double v = 0.0;
                for (int q = lane; q < nb; q += 32) v += __ldcg(part + (size_t)warp * nb + q);
                v = warp_sum(v);
                if (lane == 0) red[warp][0] = v;
            }
            __syncthreads();
        }
        const double beta = sqrt(red[0][0]), bnorm = sqrt(red[1][0]), thr = tol * bnorm;
        const bool finite = isfinite(beta) && isfinite(bnorm);
        __syncthreads();
        if (tid == 0) {
            sg[0] = sresid = shnext = beta;
            sinv = (float)(1.0 / beta);
            s_k = 0;
            s_conv = finite && beta <= thr ? 1 : 0;
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
                const bool conv = fin && resid <= thr;
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
            if (!grid_barrier<W>(bar, target += nb, &P.sc->wait_err, &s_fail)) return;
            if (s_end) break;   // (the same decision in every CTA; this product is dropped)
            const int nv = j + 1;
            t = on ? (float)combined(false) : 0.0f;
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
            gs->bnorm = bnorm;
            gs->thr = thr;
            gs->beta = beta;
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
                P.sc->gg = bnorm * bnorm;
            }
        }
        __syncthreads();
        if (s_final) return;
        __syncthreads();   // s_final was read; the next cycle rewrites it
    }
}

}  // namespace

// Host: sizes of the resident form, and the number of product warps for which every
// subdomain finds a CTA of its own on the device at once (0: the form does not apply).
// Shapes with sixteen warps first (one CTA per SM), then eight, then four.
int res_warps(dd_handle* h, int m) {
    if (h->members > 1 || !h->sym_ok || h->mult_dof.empty() || h->n_sm == 0) return 0;
    int g = 0, span = 0, floats = 0;
    for (const SymDesc& sd : h->sym) {
        g = std::max(g, sd.n[1] + sd.n[2]);
        span = std::max(span, (sd.nt - sd.tI) * kSymT);
    }
    if (g > 512) return 0;
    for (const SymDesc& sd : h->sym) {
        int f = 0;
        for (int a = sd.tI; a < sd.nt; ++a)
            for (int c = sd.tI; c <= a; ++c) f += sym_tile_floats(sym_h(sd, a), sym_h(sd, c), a == c);
        floats = std::max(floats, f);
    }
    floats = (floats + 31) / 32 * 32;
    h->res_span = span;
    h->res_floats = floats;
    for (int W = 16; W >= 4; W /= 2) {
        const size_t smem = res_smem(W, span, floats, m);
        auto kern = W == 16 ? k_gm_resident<16> : W == 8 ? k_gm_resident<8> : k_gm_resident<4>;
        cudaFuncAttributes fa;
        if (g > 32 * W || cudaFuncGetAttributes(&fa, kern) != cudaSuccess || smem + fa.sharedSizeBytes > 227 * 1024) continue;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * W + 32, smem) != cudaSuccess) return 0;
        if ((int64_t)per_sm * h->n_sm >= h->n_sub) return W;
    }
    return 0;
}

int launch_gm_resident(const dd_handle* h, const UView& U, int W, int have_q, int m, void* stream) {
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
    P.span = h->res_span;
    P.tile_floats = h->res_floats;
    P.have_q = have_q;
    auto kern = W == 16 ? k_gm_resident<16> : W == 8 ? k_gm_resident<8> : k_gm_resident<4>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)h->n_sub);
    cfg.blockDim = dim3(32 * W + 32);
    cfg.dynamicSmemBytes = res_smem(W, P.span, P.tile_floats, m);
    cfg.stream = S(stream);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, kern, P);
}
