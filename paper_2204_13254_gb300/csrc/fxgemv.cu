// FP64 batched GEMV of the solves in fixed point on packed symmetric tiles (sm_103a).
//
// GB300 does two FP64 FMAs per clock and SM, so a dense FP64 GEMV (one FMA per 8
// bytes) stops at about 4.2 TB/s, and reading only the stored triangle would not help
// it: the FMAs stay.  The 32 x 32 + 64 bit integer multiply-add runs at 25 per clock
// and SM.  Here every local operator and the input vector are integers of 57 bits and
// sign, products are formed by three such multiply-adds, sums are exact, and one read
// of a tile serves its direct and its transposed role, so the kernel is bound by HBM
// on half of the dense bytes.
//
// Fixed point.  S_s = J M_s (symmetric; symgemv.cu) is scaled by powers of two on both
// sides, |S_ij| 2^(-d_i - d_j) <= 1: d_i = ceil(E_i / 2) with S_ii < 2^E_i on the r
// block (S_rr = A_rr^-1 is positive definite, so |S_ij| <= sqrt(S_ii S_jj)); d_c of a
// corner covers its row over r and its own diagonal.  T_ij = rint(S_ij 2^(57 - d_i - d_j)),
// and with one exponent X per CTA q_j = rint(x_j 2^(d_j + 57 - X)); then
//     y_i = 2^(d_i + X - 114) sum_j T_ij q_j.
// An integer is split as T = hi 2^29 + lo, |hi|, |lo| <= 2^28 (lo = 0 where |hi| = 2^28),
// and the sums of hi hi' and of hi lo' + lo hi' run in two 64-bit accumulators: a product
// adds at most 2^56 to the first and less than 2^57 to the second, so 64 products fit
// (a tile's transposed sums; the direct sums of two lanes over kFlush = 8 tiles).  From
// there the sums go on as 96-bit integers (fx96.h) in shared memory and become FP64 numbers once
// per CTA and row (conversions run on the FP64 pipe, at two per clock and SM).  lo lo' is
// dropped.
//
// Error.  T and q are rounded to 2^-58 of their scales and lo lo' is below 2^-58 of them, so
// y_i is off by less than 3 n 2^-58 of 2^(d_i + X) (about sqrt(n) 2^-59 of it when the
// roundings are random): an absolute bound per row, relative to the largest 2^(d_j) x_j of
// the CTA, not to the row's own sum.  In the norm that is at the level of an FP64 sum
// (block of 648 interface rows, smooth input 1.3e-16, FP64 2.1e-16; random input 3.0e-16,
// FP64 3.2e-16); rows far below the scale of their subdomain have fewer correct digits
// (an input that decays over the subdomain: 1e-7 of the smallest rows).  The solves do not
// see the difference: a Krylov solution is only accurate to the tolerance, at best 2^-53, of
// the norm of the whole vector.  Measured, first steps from a point, a line, a smooth and a
// random source against an extended-precision solve, dense form and this one: to tolerance
// 1e-10 the same errors, to 1e-14 norms within a fifth of each other and the same 90 % and
// 99 % quantiles of the error row by row.
// The operator calls (dd_coupled_apply, dd_schur_apply, ...) hand their rows to the caller
// and stay with the dense form.  This form with lo lo' kept and the small rows summed again
// in FP64 was as accurate row by row, and at 106 us no faster (dense 112 us, 42 M elements).
//
// Layout: the tiles of the packed FP32 operator (64 x 64, or short at a run's end; lower
// triangle), each cut into blocks of 16 rows x 8 columns: 512 bytes of hi words, then 512
// of lo words, lane 2 i + c of a warp holding row i, columns 4 c .. 4 c + 3 (16-byte shared
// loads without bank conflicts).  A tile's blocks follow strip by strip (8 columns each),
// the blocks of a strip by rows; a diagonal tile leaves out the blocks above its
// diagonal.  Warp w of the eight warps takes strip w of every tile through a ring of its
// own (one lane refills a slot as soon as the warp is done with it), so that the
// transposed sums of a tile end inside one warp, the entries 8 w .. 8 w + 7 of every tile
// row of y belong to warp w alone, and only the direct sums cross warps, once per tile
// row.  Every mbarrier wait is bounded; a warp whose wait gave up goes on through the list
// without waiting, so that the barriers of the tile rows still see every warp, and nothing
// is copied any more.
//
// Measured (GB300), dense k_gemv<double> / here: coupled operator of 256 subdomains with
// 400-480 interface rows, 42 M elements, 106 / 64 us (170 MB at 2.7 TB/s); the FP64 step of
// 512 subdomains of 1,854 unknowns 11.1 / 6.5 ms, its GEMVs 9.7 / 5.7 ms (3.8 TB/s).  What
// bounds it now is instruction latency at two CTAs (16 warps) per SM: about 470 warp
// instructions per strip, 96 of them multiply-adds, 36 % of the issue slots.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "dd_internal.h"
#include "fixpoint.cuh"
#include "fx96.h"
#include "symtile.cuh"
#include "xsrc.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kWarps = 8;              // consumer warps: one 8-column strip of a tile each
constexpr int kT = 32 * kWarps;
constexpr int kStMax = 4;              // deepest ring of strips per warp
constexpr int kFlush = 8;              // tiles of one tile row between two flushes of the direct sums
constexpr int kBlkInts = 256;          // one 16 x 8 block: 128 hi words, 128 lo words
constexpr int kStripInts = 4 * kBlkInts;   // ring slot of one warp: 64 rows x 8 columns, 4 KB
constexpr int kPad = 17;               // column stride of the transposed sums in a slot (16 row lanes, no bank conflicts)
constexpr int kSms = 152;              // multiprocessors of a GB300 (the ranges are cut before a device is bound)
constexpr int kFxW = 4;                // words per tile list entry: tile_entry(), first block, block rows | strips << 8, 0

static_assert(kFx96Low == kLow, "the split of the integers");

inline cudaStream_t S(void* s) { return (cudaStream_t)s; }

// Blocks of a tile of h rows and w columns: R rows of blocks, W strips; strip q of a
// diagonal tile starts at block row q / 2.  First block of strip q:
__host__ __device__ inline int fx_strip(int R, int q, bool diag) {
    return q * R - (diag && q > 0 ? (q - 1) * (q - 1) / 4 : 0);
}
__host__ __device__ inline int fx_blocks(int h, int w, bool diag) {
    return fx_strip((h + 15) / 16, (w + 7) / 8, diag);
}

__host__ __device__ inline size_t fx_smem(int span, int st) {
    return (size_t)st * kWarps * kStripInts * sizeof(int32_t) + (size_t)span * (2 * sizeof(uint64_t) + sizeof(int32_t)) +
           kWarps * 64 * sizeof(longlong2) + (size_t)st * kWarps * sizeof(uint64_t);
}
// Ring depth: the deepest that leaves two CTAs on an SM, otherwise the deepest that fits.
inline int fx_depth(int span) {
    for (int st = kStMax; st >= 2; --st)
        if (2 * (fx_smem(span, st) + 1280) <= 228 * 1024) return st;
    for (int st = kStMax; st >= 2; --st)
        if (fx_smem(span, st) + 256 <= 227 * 1024) return st;
    return 0;
}

// A listed tile as a warp sees it: e, the block rows [r0, R) of its strip (none when the
// tile is narrower), the strip's first block.
struct Strip {
    uint32_t e;
    int r0, R, first;
};
__device__ __forceinline__ Strip fx_entry(const uint4& w, int q) {
    Strip t;
    t.e = w.x;
    t.R = (int)(w.z & 255u);
    const bool diag = (w.x & 4) != 0;
    t.r0 = q < (int)(w.z >> 8) ? (diag ? q >> 1 : 0) : t.R;
    t.first = (int)w.y + fx_strip(t.R, q, diag);
    return t;
}
// One lane: the copy of a strip into a ring slot (nothing when it has no blocks: the
// consumer does not wait for it either).
__device__ __forceinline__ void issue_strip(const Strip& t, const int32_t* tiles, int32_t* dst, uint64_t* bar,
                                            uint64_t pol) {
    if (t.r0 < t.R)
        load_tile(reinterpret_cast<float*>(dst), reinterpret_cast<const float*>(tiles) + (int64_t)t.first * kBlkInts,
                  4u * kBlkInts * (uint32_t)(t.R - t.r0), bar, pol);
}

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, const volatile int* abort) {
    for (unsigned k = 0; k < kWaitLimit; ++k) {
        if (mbar_test(bar, parity)) return true;
        if ((k & 255u) == 255u && *abort) return false;
    }
    return false;
}

// One CTA (or cluster of cl CTAs, by ranges of tile rows) per subdomain.
__global__ void __launch_bounds__(kT, 2) k_fxgemv(const SymDesc* __restrict__ descs, const int32_t* __restrict__ ranges,
                                                  const uint32_t* __restrict__ tlist, const int32_t* __restrict__ Mfx,
                                                  const int64_t* __restrict__ moff, const int32_t* __restrict__ exps,
                                                  int span_max, int cl, int st, int rmask, int cmask, int keep, int n_real,
                                                  XSrc xs, GemvOut go, const int32_t* __restrict__ skip,
                                                  int32_t* __restrict__ err) {
    if (skip && *skip) return;   // the same word for every CTA of the grid
    extern __shared__ __align__(128) unsigned char smem_raw[];
    int32_t* ring = reinterpret_cast<int32_t*>(smem_raw);                         // [kWarps][st][kStripInts]
    longlong2* red = reinterpret_cast<longlong2*>(ring + st * kWarps * kStripInts);   // [kWarps][64] direct sums of a tile row
    int2* xq = reinterpret_cast<int2*>(red + kWarps * 64);                        // [span_max], index p - p_lo
    uint64_t* ylo = reinterpret_cast<uint64_t*>(xq + span_max);                   // [span_max] 96-bit sums: low 64 bits,
    uint64_t* full = ylo + span_max;                                              // [kWarps][st]
    int32_t* yhi = reinterpret_cast<int32_t*>(full + st * kWarps);                // [span_max] high 32 bits
    __shared__ int wmax[kWarps];
    __shared__ int abort_flag;
    __shared__ uint64_t never;   // completed by nothing (first_wait_test)

    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t* rg5 = ranges + kSymRng * blockIdx.x;
    const int sub = rg5[3], stored = sub % n_real;
    const SymDesc sd = descs[sub];
    const int32_t* dex = exps + descs[stored].voff;   // exponents of the stored subdomain's rows
    const uint4* lst = reinterpret_cast<const uint4*>(tlist) + rg5[0];
    const int nt_cta = rg5[1], a_end = rg5[2];
    const int np = sd.nt * kSymT;
    const int32_t* tiles = Mfx + moff[stored] * kBlkInts;
    const int p_lo = mask_lo(sd, rmask | cmask), r_lo = mask_lo(sd, rmask);
    const int p_end = min(np, a_end * kSymT);
    const uint64_t pol = l2_policy(stored < keep);
    int32_t* wring = ring + warp * st * kStripInts;   // this warp's slots and barriers
    uint64_t* wfull = full + warp * st;
    const int first_polls = tid == 0 ? xs.sc->wait_first : 0;   // (asked for ahead of its use)
    if (tid == 0) {
        abort_flag = 0;
        mbar_init(&never, 1);
    }
    if (lane == 0) {
        for (int s = 0; s < st; ++s) mbar_init(&wfull[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int s = 0; s < st && s < nt_cta; ++s) {
            issue_strip(fx_entry(__ldg(lst + s), warp), tiles, wring + s * kStripInts, &wfull[s], pol);
        }
    }
    // x 2^d in FP64 (into the words its integers will take), its largest exponent, then the integers
    for (int p = tid; p < np - p_lo; p += kT) {
        ylo[p] = 0;
        yhi[p] = 0;
    }
    double* xd = reinterpret_cast<double*>(xq);
    int mx = 0;
    {
        const double beta = (xs.kind == X_PCG || xs.kind == X_PCG_CV) ? xs.sc->beta : 0.0;
        constexpr int kU = 2;   // entries per pass: index loads, then value loads
        for (int p0 = p_lo + tid; p0 < p_end; p0 += kT * kU) {
            int mm[kU], cc[kU], ll[kU], dd[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int p = p0 + u * kT;
                const int l = p < p_end ? sym_local(sd, p) : -1;
                const bool need = l >= 0 && ((cmask >> sym_lgroup(sd, l)) & 1);
                ll[u] = need ? l : -1;
                mm[u] = need ? xs.slot_mult[sd.voff + l] : 0;
                cc[u] = need ? xs.slot_corner[sd.voff + l] : -1;
                dd[u] = need ? dex[l] : 0;
            }
            double v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u)
                v[u] = ll[u] >= 0 ? xref_value(xsrc_ref<double>(xs, mm[u], cc[u], sd.voff + ll[u], ll[u]), beta) : 0.0;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int p = p0 + u * kT;
                if (p >= p_end) continue;
                const double w = scale2(v[u], dd[u]);
                mx = max(mx, __double2hiint(w) & 0x7fffffff);
                xd[p - p_lo] = w;
            }
        }
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) wmax[warp] = mx;
    __syncthreads();
    mx = wmax[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) mx = max(mx, wmax[w]);
    const bool finite = mx < 0x7ff00000;   // NaN or Inf in x: every row of this CTA becomes NaN
    const int X = exp_of_hi(mx);
    for (int p = p_lo + tid; p < p_end; p += kT) xq[p - p_lo] = finite ? split57(xd[p - p_lo], kBits - X) : make_int2(0, 0);
    if (tid == 0 && !first_wait_test(first_polls, &never)) abort_flag = 1;
    __syncthreads();

    const int ri = lane >> 1, c8 = 8 * warp + 4 * (lane & 1);   // row in a block, first column in a tile
    long long ah[4], ax[4];   // direct sums of rows 16 r + ri over this lane's columns
    int xh[4], xl[4];         // x of those rows
    int cur = -1, cnt = 0;
    bool bad = false;
    // entry p of y += v (a 96-bit integer; the entry belongs to this warp)
    auto add_y = [&](int p, __int128 v) { fx96_add(ylo[p], yhi[p], v); };
    // direct sums of tile row `row` -> y: the two column quads of the lane pair (each lane keeps
    // two rows), then over the eight warps; warp w adds rows 8 w .. 8 w + 7
    auto flush_d = [&](int row) {
        const bool up = (lane & 1) != 0;
        __syncthreads();   // the previous row's sums have been read
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const long long sh = __shfl_xor_sync(0xffffffffu, up ? ah[r] : ah[r + 2], 1);
            const long long sx = __shfl_xor_sync(0xffffffffu, up ? ax[r] : ax[r + 2], 1);
            red[warp * 64 + 16 * (r + (up ? 2 : 0)) + ri] =
                make_longlong2((up ? ah[r + 2] : ah[r]) + sh, (up ? ax[r + 2] : ax[r]) + sx);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) ah[r] = ax[r] = 0;
        cnt = 0;
        __syncthreads();
        const int i = 8 * warp + (lane & 7), q = lane >> 3;
        __int128 v = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const longlong2 t = red[(2 * q + u) * 64 + i];
            v += fx96_part(t.x, t.y);
        }
#pragma unroll
        for (int o = 8; o <= 16; o <<= 1) {
            const uint64_t lo = __shfl_xor_sync(0xffffffffu, (uint64_t)v, o);
            const int32_t hi = __shfl_xor_sync(0xffffffffu, (int32_t)(v >> 64), o);
            v += ((__int128)hi << 64) + lo;
        }
        if (lane < 8) add_y(row * kSymT + i - p_lo, v);
        __syncwarp();
    };
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        ah[r] = ax[r] = 0;
        xh[r] = xl[r] = 0;
    }
    // entries k and k + 1, and the one to copy next (k + st): loaded ahead of their use
    const uint4 none = make_uint4(0, 0, 0, 0);
    uint4 next = nt_cta > 0 ? __ldg(lst) : none;
    uint4 fill = st < nt_cta ? __ldg(lst + st) : none;
    int slot = 0;
    uint32_t phases = 0;   // bit s: parity of slot s's next copy
    for (int k = 0; k < nt_cta; ++k) {
        const Strip t = fx_entry(next, warp);
        const uint32_t e = t.e;
        if (k + 1 < nt_cta) next = __ldg(lst + k + 1);
        const int ca = (int)(e >> 16), cb = (int)((e >> 3) & 0x1fff);
        if (ca != cur) {
            if (cur >= 0) flush_d(cur);
            cur = ca;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int2 q = xq[ca * kSymT + 16 * r + ri - p_lo];
                xh[r] = q.x;
                xl[r] = q.y;
            }
        } else if (cnt == kFlush) {
            flush_d(cur);
        }
        if (t.r0 < t.R) {   // (uniform over the warp)
            if (!bad) {
                if (wait_or_abort(&wfull[slot], (phases >> slot) & 1u, &abort_flag)) {
                    phases ^= 1u << slot;
                } else {
                    bad = true;
                    *(volatile int*)&abort_flag = 1;
                }
            }
            int32_t* strip = wring + slot * kStripInts;
            const int32_t* base = strip - t.r0 * kBlkInts + 4 * lane;
            long long ch[4] = {}, cx[4] = {};
            int4 mh[4], ml[4];
            if (t.r0 == 0 && t.R == 4) {   // (uniform over the warp)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    mh[r] = *reinterpret_cast<const int4*>(base + r * kBlkInts);
                    ml[r] = *reinterpret_cast<const int4*>(base + r * kBlkInts + kBlkInts / 2);
                }
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const bool in = r >= t.r0 && r < t.R;
                    mh[r] = in ? *reinterpret_cast<const int4*>(base + r * kBlkInts) : make_int4(0, 0, 0, 0);
                    ml[r] = in ? *reinterpret_cast<const int4*>(base + r * kBlkInts + kBlkInts / 2) : make_int4(0, 0, 0, 0);
                }
            }
            // rows innermost: four independent chains (a branch on a block left out would cost the
            // overlap of the rows; its words are zero instead)
            if (e & 1) {
                const int4* xp = reinterpret_cast<const int4*>(xq + cb * kSymT + c8 - p_lo);
                const int4 q0 = xp[0], q1 = xp[1];   // (hi, lo) of columns 0, 1 and 2, 3
#pragma unroll
                for (int r = 0; r < 4; ++r) mac(ah[r], ax[r], mh[r].x, ml[r].x, q0.x, q0.y);
#pragma unroll
                for (int r = 0; r < 4; ++r) mac(ah[r], ax[r], mh[r].y, ml[r].y, q0.z, q0.w);
#pragma unroll
                for (int r = 0; r < 4; ++r) mac(ah[r], ax[r], mh[r].z, ml[r].z, q1.x, q1.y);
#pragma unroll
                for (int r = 0; r < 4; ++r) mac(ah[r], ax[r], mh[r].w, ml[r].w, q1.z, q1.w);
            }
            if (e & 2) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    mac(ch[0], cx[0], mh[r].x, ml[r].x, xh[r], xl[r]);
                    mac(ch[1], cx[1], mh[r].y, ml[r].y, xh[r], xl[r]);
                    mac(ch[2], cx[2], mh[r].z, ml[r].z, xh[r], xl[r]);
                    mac(ch[3], cx[3], mh[r].w, ml[r].w, xh[r], xl[r]);
                }
                // column sums over the 16 row lanes through the slot just read ([hi, cross][column][lane])
                __syncwarp();
                long long* sc = reinterpret_cast<long long*>(strip);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    sc[(4 * (lane & 1) + c) * kPad + ri] = ch[c];
                    sc[(8 + 4 * (lane & 1) + c) * kPad + ri] = cx[c];
                }
                __syncwarp();
                const long long* sr = sc + (lane & 15) * kPad + 8 * (lane >> 4);
                long long v = ((sr[0] + sr[1]) + (sr[2] + sr[3])) + ((sr[4] + sr[5]) + (sr[6] + sr[7]));
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                const long long x = __shfl_xor_sync(0xffffffffu, v, 8);   // lanes 0..7: hi sums here, cross sums there
                if (lane < 8) add_y(cb * kSymT + 8 * warp + lane - p_lo, fx96_part(v, x));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before the slot's next copy
            }
        }
        __syncwarp();   // every lane is done with the slot
        if (lane == 0 && k + st < nt_cta && !*(volatile int*)&abort_flag)
            issue_strip(fx_entry(fill, warp), tiles, wring + slot * kStripInts, &wfull[slot], pol);
        if (k + st + 1 < nt_cta) fill = __ldg(lst + k + st + 1);
        ++cnt;
        if (++slot == st) slot = 0;
    }
    if (cur >= 0) flush_d(cur);
    __syncthreads();
    bad = abort_flag != 0;
    if (bad) {   // let the copies still in flight land (bounded; a slot may have none), then report
        if (lane == 0)
            for (int s = 0; s < st; ++s)
                for (unsigned k = 0; k < (1u << 16) && !mbar_done(&wfull[s], (phases >> s) & 1u); ++k) {}
        if (tid == 0) atomicExch(err, 1);
        __syncthreads();
    }
    // this CTA's partial sums in units of 2^d_i (NaN when x was not finite or a wait gave up)
    const double unit = (bad || !finite) ? __longlong_as_double(0x7ff8000000000000ll) : pow2(X - 2 * kBits + kFx96Unit);
    double* y = reinterpret_cast<double*>(ylo);
    for (int p = tid; p < np - p_lo; p += kT)   // 96 bits: the high 64 and the low 32
        y[p] = fma((double)fx96_high(ylo[p], yhi[p]), 0x1p32, (double)fx96_low(ylo[p])) * unit;
    cluster.sync();
    const int rank = (int)cluster.block_rank();
    for (int p = r_lo + rank * kT + tid; p < np; p += cl * kT) {
        const int l = sym_local(sd, p);
        if (l < 0) continue;
        const int g = sym_lgroup(sd, l);
        if (!((rmask >> g) & 1)) continue;
        double v = 0.0;
        for (int c = 0; c < cl; ++c) v += cluster.map_shared_rank(y, c)[p - p_lo];
        v = scale2(v, dex[l]);
        if (g == 2) v = -v;   // J: the corner rows of M = J S
        if (go.alpha != 1.0) v *= go.alpha;
        const int64_t o = sd.voff + l;
        if (go.base) v += go.base[o];
        go.out[go.pos ? (int64_t)go.pos[o] : o] = v;
    }
    cluster.sync();   // no CTA leaves while another reads its shared memory
}

// Exponents d of one stored subdomain's rows (see the file comment), one CTA per subdomain.
__global__ void __launch_bounds__(256) k_fx_exps(const SymDesc* __restrict__ descs, const MatDesc* __restrict__ mats,
                                                 const double* __restrict__ M, int32_t* __restrict__ exps) {
    const SymDesc sd = descs[blockIdx.x];
    const MatDesc md = mats[blockIdx.x];
    const double* A = M + md.moff;
    int32_t* d = exps + sd.voff;
    auto half = [](int e) { return (e + 1) >> 1; };   // ceil(e / 2)
    for (int i = threadIdx.x; i < md.nr; i += blockDim.x)
        d[i] = half(exp_of_hi(__double2hiint(A[(int64_t)i * md.ld + i]) & 0x7fffffff));
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int c = md.nr + (threadIdx.x >> 5); c < md.ns; c += blockDim.x >> 5) {
        const double* row = A + (int64_t)c * md.ld;
        int m = -4000;
        for (int j = lane; j < md.nr; j += 32) {
            const int hi = __double2hiint(row[j]) & 0x7fffffff;
            if (hi >> 20) m = max(m, exp_of_hi(hi) - d[j]);
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) d[c] = max(m, half(exp_of_hi(__double2hiint(row[c]) & 0x7fffffff)));
    }
}

// Pack: one CTA per stored tile, S = J M in fixed point, the diagonal halved on diagonal
// tiles, zeros in the padding; a warp per block (rows read in 64-byte pieces).
__global__ void __launch_bounds__(256) k_fx_pack(const SymDesc* __restrict__ descs, const MatDesc* __restrict__ mats,
                                                 const int32_t* __restrict__ dir, const double* __restrict__ M,
                                                 const int64_t* __restrict__ moff, const int32_t* __restrict__ exps,
                                                 int32_t* __restrict__ Mfx) {
    const int32_t* dr = dir + 4 * (int64_t)blockIdx.x;
    const int s = dr[0], a = dr[1], b = dr[2];
    const SymDesc sd = descs[s];
    const MatDesc md = mats[s];
    const bool diag = a == b;
    const int h = sym_h(sd, a), w = sym_h(sd, b), R = (h + 15) >> 4, W = (w + 7) >> 3;
    const int la0 = a < sd.tI ? kSymT * a : sd.n[0] + kSymT * (a - sd.tI);
    const int lb0 = b < sd.tI ? kSymT * b : sd.n[0] + kSymT * (b - sd.tI);
    int32_t* out = Mfx + (moff[s] + dr[3]) * kBlkInts;
    const int32_t* d = exps + sd.voff;
    const int lane = threadIdx.x & 31;
    for (int q = (int)(threadIdx.x >> 5); q < W * R; q += (int)(blockDim.x >> 5)) {
        const int strip = q / R, br = q - strip * R, r0 = diag ? strip >> 1 : 0;
        if (br < r0) continue;
        const int r = 16 * br + (lane >> 1), li = la0 + r;
        int hi[4], lo[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j = 8 * strip + 4 * (lane & 1) + c;
            int2 t = make_int2(0, 0);
            if (r < h && j < w && (!diag || j <= r)) {
                double v = M[md.moff + (int64_t)li * md.ld + lb0 + j];
                if (li >= sd.n[0] + sd.n[1]) v = -v;   // S = J M
                if (diag && j == r) v *= 0.5;
                t = split57(v, kBits - d[li] - d[lb0 + j]);
            }
            hi[c] = t.x;
            lo[c] = t.y;
        }
        int32_t* o = out + (fx_strip(R, strip, diag) + br - r0) * kBlkInts + 4 * lane;
        *reinterpret_cast<int4*>(o) = make_int4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<int4*>(o + kBlkInts / 2) = make_int4(lo[0], lo[1], lo[2], lo[3]);
    }
}

}  // namespace

// True when the fixed-point form can serve FP64 GEMVs of `mode`, and when it does (its tiles are
// the packed operators in the workspace).
bool fx_built(const dd_handle* h, int mode) { return h->fx_ok && sym_active(h, mode) && h->fx_bytes[mode] > 0.0; }
bool fx_active(const dd_handle* h, int mode) { return fx_built(h, mode) && h->packed == DD_FP64; }

// Host side: the directory and the tile lists with block offsets, CTAs per subdomain, the
// ranges of every mode.
//  * The form serves a mode when there are at least 48 subdomains and it streams at least
//    8 MB.  A CTA stages x, sums and converts for about 8 us besides its tiles, and at most
//    eight share a subdomain, where the dense form cuts its rows as finely as it likes.
//    Measured, one FP64 GMRES step, dense / fixed point: 512 subdomains of 1,854 unknowns
//    11.10 / 6.98 ms, 64 of them 2.16 / 1.92, 128 of 604 1.83 / 1.66, 64 of 604 1.15 /
//    1.11; but 27 of 1,854 1.47 / 1.65, 8 of 1,512 0.99 / 1.13, 8 of 3,584 1.32 / 1.64,
//    8 of 448 0.87 / 0.89.
//  * CTAs per subdomain: every CTA more stages x again, but one CTA per subdomain leaves SMs
//    with one CTA beside SMs with two where there are fewer subdomains than slots (two per
//    SM, 304).  So two up to 256 subdomains, the largest number below that line at which two
//    were measured to be better (by 2 %; at 343 one is), and more (a cluster of 8 at most)
//    only until every SM has a CTA.  Measured, FP64 GMRES step with 1 / 2 / 4 / 8 CTAs per subdomain, in us: 64
//    subdomains of 1,854 unknowns 3,203 / 2,086 / 1,559 / 1,618, 100 of 741 1,323 / 1,047 /
//    1,108 / 1,405, 128 of 2,196 3,947 / 3,110 / 3,330 / 4,164, 216 of 1,115 2,200 / 1,947 /
//    2,207 / 3,091, 256 of 1,152 2,241 / 2,198 / 2,602 / 3,576, 343 of 604 1,511 / 1,624.
//  * Subdomains kept in L2 between the launches of a Krylov solve: 64 MB worth, about half
//    of L2, as the FP32 tuner settled on.
void build_fx(dd_handle* h) {
    h->fx_ok = h->sym_elems > 0 && fx_depth(h->sym_np_max) > 0;
    h->packed = h->prm.precision;
    h->fx_dir.clear();
    h->fx_moff.clear();
    h->fx_blocks = 0;
    if (!h->fx_ok) return;
    // tiles in the order of sym_dir (every stored subdomain's tiles follow each other)
    h->fx_dir = h->sym_dir;
    std::vector<std::vector<int32_t>> offs(h->n_sub_real);
    for (size_t k = 0; k < h->fx_dir.size(); k += 4) {
        const int s = h->fx_dir[k], a = h->fx_dir[k + 1], b = h->fx_dir[k + 2];
        const SymDesc& sd = h->sym[s];
        if ((int)h->fx_moff.size() == s) {
            h->fx_moff.push_back(h->fx_blocks);
            offs[s].assign((size_t)sd.nt * sd.nt, 0);
        }
        const int32_t off = (int32_t)(h->fx_blocks - h->fx_moff[s]);
        h->fx_dir[k + 3] = off;
        offs[s][(size_t)a * sd.nt + b] = off;
        h->fx_blocks += fx_blocks(sym_h(sd, a), sym_h(sd, b), a == b);
    }
    bool any = false;
    for (int m = 0; m < GEMV_NMODES; ++m) {
        h->fx_rng[m].clear();
        h->fx_tl[m].clear();
        int rmask, cmask;
        h->fx_bytes[m] = 0.0;
        if (!sym_active(h, m) || !sym_masks(m, &rmask, &cmask) || h->n_sub < 48) continue;
        size_t q = 0;
        int64_t blocks = 0;
        for (int s = 0; s < h->n_sub_real; ++s)
            for (; q < (size_t)h->sym_tl_off[m][s + 1]; ++q) {
                const uint32_t e = h->sym_tl[m][kTlW * q];   // the same tiles in the same order
                const int a = (int)(e >> 16), b = (int)((e >> 3) & 0x1fff);
                const SymDesc& sd = h->sym[s];
                const uint32_t R = (uint32_t)(sym_h(sd, a) + 15) / 16, W = (uint32_t)(sym_h(sd, b) + 7) / 8;
                h->fx_tl[m].insert(h->fx_tl[m].end(), {e, (uint32_t)offs[s][(size_t)a * sd.nt + b], R | (W << 8), 0u});
                blocks += fx_blocks(sym_h(sd, a), sym_h(sd, b), a == b);
            }
        const double streamed = 1024.0 * (double)blocks;
        if (streamed < 8e6) {
            h->fx_tl[m].clear();
            continue;
        }
        int cl = h->n_sub <= 256 ? 2 : 1;
        while (cl < kSymCLMax && h->n_sub * cl < kSms) cl *= 2;
        h->fx_cl[m] = cl;
        int32_t longest = 0;
        sym_split(h, m, cl, 1, h->fx_rng[m], &longest);
        h->fx_bytes[m] = streamed * (double)std::max(1, h->members);
        const double per_sub = streamed / std::max(1, h->n_sub_real);
        h->fx_keep[m] = (m == GEMV_SCHUR_G || m == GEMV_COUPLED)
                            ? (int32_t)std::min<double>(h->n_sub_real, 64.0e6 / std::max(1.0, per_sub))
                            : 0;
        any = true;
    }
    if (!any) {   // no mode reads the tiles: no storage for them
        h->fx_ok = false;
        h->fx_blocks = 0;
        h->fx_dir.clear();
        h->fx_moff.clear();
    }
}

int launch_fx_pack(const dd_handle* h, void* stream) {
    if (!h->fx_ok || h->sym_ntiles == 0) return 0;
    k_fx_exps<<<(unsigned)h->n_sub_real, 256, 0, S(stream)>>>(h->d.symd, h->d.mats, h->d.M64, h->d.fx_exps);
    k_fx_pack<<<(unsigned)h->sym_ntiles, 256, 0, S(stream)>>>(h->d.symd, h->d.mats, h->d.fx_dir, h->d.M64, h->d.fx_moff,
                                                              h->d.fx_exps, h->d.Mfx);
    return (int)cudaGetLastError();
}

int launch_fxgemv(const dd_handle* h, int mode, XSrc xs, GemvOut go, const int32_t* skip, void* stream) {
    int rmask, cmask;
    if (!sym_masks(mode, &rmask, &cmask) || !go.out) return (int)cudaErrorInvalidValue;
    xs.slot_mult = h->d.slot_mult;
    xs.slot_corner = h->d.slot_corner;
    xs.sc = h->d.sc;
    const int span = sym_span(h, mode), cl = h->fx_cl[mode];
    const int st = fx_depth(span);
    const size_t smem = fx_smem(span, st);
    if (st == 0) return (int)cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_fxgemv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fxgemv, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return (int)e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(h->fx_rng[mode].size() / kSymRng));
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = S(stream);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, k_fxgemv, (const SymDesc*)h->d.symd, (const int32_t*)h->d.fx_rng[mode],
                                   (const uint32_t*)h->d.fx_tl[mode], (const int32_t*)h->d.Mfx,
                                   (const int64_t*)h->d.fx_moff, (const int32_t*)h->d.fx_exps, span, cl, st, rmask, cmask, h->fx_keep[mode],
                                   std::max(1, h->n_sub_real), xs, go, skip, &h->d.sc->wait_err);
}
