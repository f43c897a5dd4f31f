// Gram-Schmidt of the FP64 flexible GMRES on a block fixed-point basis
// (fix60.cuh): the basis vectors are stored once as integer limbs by
// launch_basis_store, and the projections h = V^H w, the norm ||w||^2 and the
// update w -= V h run on the integer pipe, with FP64 inputs and results.
//
// Bound: HBM.  With FP64 multiply-adds (4 per entry and row, 2 per clock and SM)
// the same sums ran at the FP64 pipe's rate.  Measured on GB300, per FGMRES step:
//   32 sources of 1024 x 512 (two passes): dots 12.6 -> 2.8 ms, updates
//   7.1 -> 3.1 ms (6.6 and 6.4 TB/s); one source at 1024 x 1024: 450 -> 136 us
//   and 262 -> 128 us; 128^3: 1.28 -> 0.32 ms and 0.74 -> 0.33 ms.
// Accuracy against 113-bit sums on the Arnoldi vectors of a point source
// (320 x 200), in the norm: update error 0.2e-16 of |w'| at k = 1 and 1.2e-16 at
// k = 2 (FP64 sums: 0 and 0.7e-16; v_0 has one nonzero entry), 0.7e-16 .. 1.0e-16
// for k = 3 .. 20 (1.1e-16 .. 3.9e-16, growing with k); projections within
// 9e-17 |w| (7e-17).  Per entry there is no such bound (fix60.cuh).
//
// Batched over right-hand sides (blockIdx.z) with the flags and strides of
// k_krylov.cu: pass 1 forms h1 = V^H w together with ||w||^2 and then
// w' = w - V h1 together with ||w'||^2; the pass-2 launches read the
// per-right-hand-side flag and return at once when it is clear.
#include "bah_internal.cuh"
#include "fix60.cuh"
#include "givens.cuh"

#include <algorithm>

namespace bah {

__device__ __forceinline__ bool inactive_gs(const KS& ks, int r) { return ks.active && !ks.active[r]; }

constexpr int kGsThreads = 128;
constexpr int kGsWarps = kGsThreads / 32;
constexpr int kGsRows = 8;           // basis rows of one CTA
constexpr int kGsFew = 64;           // up to so many partial sums a row are added by the dot kernel's last CTA

// true in every thread of the last CTA (of `total`) to come here with this counter; what
// the other CTAs wrote before is then visible.  The counter is zero again afterwards.
__device__ __forceinline__ bool last_cta(int* cnt, int total) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(cnt, 1) == total - 1;
        if (last) *cnt = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// the tile's entries of w from this lane's first one, e0 (zero from `end` on), and its biased exponent
__device__ __forceinline__ int load_tile(const double2* __restrict__ w, size_t e0, size_t end, double2 (&x)[kTileU]) {
    int mx = 0;
#pragma unroll
    for (int u = 0; u < kTileU; ++u) x[u] = e0 + 32 * u < end ? w[e0 + 32 * u] : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < kTileU; ++u) mx = max(mx, max(abs_hi(x[u].x), abs_hi(x[u].y)));
    return tile_exp((int)__reduce_max_sync(0xffffffffu, (unsigned)mx));
}

// ---------------------------------------------------------------------------
// Partial sums of rows 0 .. k of one CTA's tiles: row y < k is conj(V_y) w,
// row k is |w|^2.  One warp per tile: w is converted to limbs once; for each
// group of up to R rows every lane sums its eight entries per row in 64-bit
// integers, the lanes' sums are added as integers (one exponent per tile and
// row), and the lane left with a value adds it to the CTA's FP64 sum.  Rows are
// split into equal groups (k = 10: two groups of R = 5), R a template
// parameter, because a predicated-off multiply-add still costs its issue slot.
// Groups run one after another in the warp (gridDim.y = 1), or, when the tiles
// alone would leave SMs idle, in different CTAs (gridDim.y = groups).
//
// The rows' limbs pass through a ring of kGsStages shared-memory slots per warp
// (cp.async, two rows ahead): each lane copies and reads only its own entries,
// so the ring needs no barrier, and the copies keep running while the warp
// converts w and adds up its lanes.
// ---------------------------------------------------------------------------
constexpr int kGsStages = 3;
// The rings start on 128-byte boundaries: 16 or 48 bytes off, a warp's rows straddle lines and the
// update of eight sources of 1024 x 512 took 636 us instead of 544.
constexpr size_t kGsSmem = (size_t)kGsWarps * kGsStages * kTile * sizeof(int4);

__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

template <int R, bool LAST>
__global__ void __launch_bounds__(kGsThreads, 4) k_gs_dot(const int4* __restrict__ VL, const int* __restrict__ VE, int k,
                                                          int rows, const double2* __restrict__ w, Tiles tl,
                                                          double2* __restrict__ partial, double2* __restrict__ out,
                                                          const int* flag, int* cnt, KS ks) {
    pdl_prologue();
    const int r = blockIdx.z;
    if (inactive_gs(ks, r)) return;
    if (flag && flag[r] == 0) {
        if (LAST && blockIdx.x == 0 && blockIdx.y == 0)
            for (int i = threadIdx.x; i <= k; i += kGsThreads) out[r * ks.so + i] = make_double2(0.0, 0.0);
        return;
    }
    const size_t nt = tl.count, npad = nt * kTile;
    VL += r * ks.sv;
    VE += r * ks.se;
    w += r * ks.sw;
    partial += r * ks.sp;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    constexpr int NV = R <= 1 ? 2 : (R <= 2 ? 4 : (R <= 4 ? 8 : 16));
    const int myval = lane / (32 / NV), myrow = myval >> 1;       // the value this lane ends with
    // this CTA's rows [ya, yb), taken in groups of `rows`
    const int ya = blockIdx.y * rows, yb = gridDim.y > 1 ? min(k, ya + rows) : k;
    const size_t tstep = (size_t)gridDim.x * kGsWarps;
    extern __shared__ __align__(128) int4 ring_all[];
    const int4* ring = ring_all + (size_t)wp * kGsStages * kTile + lane;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    size_t pt = (size_t)blockIdx.x * kGsWarps + wp;             // next row to copy: tile, row, slot
    int py = ya, ps = 0, cs = 0;
    auto prefetch = [&]() {
        if (pt < nt) {
            const int4* src = VL + (size_t)py * npad + pt * kTile + lane;
#pragma unroll
            for (int u = 0; u < kTileU; ++u) copy16(ring_s + (uint32_t)(ps * kTile + 32 * u) * 16u, src + 32 * u);
            if (++py == yb) { py = ya; pt += tstep; }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ps = ps == kGsStages - 1 ? 0 : ps + 1;
    };
#pragma unroll
    for (int i = 0; i < kGsStages - 1; ++i) prefetch();
    __shared__ double sum[kGsWarps][2 * 64 + 1];                  // per warp: row values, |w|^2
    for (int i = lane; i < 2 * 64 + 1; i += 32) sum[wp][i] = 0.0;
    __syncwarp();
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (size_t t = (size_t)blockIdx.x * kGsWarps + wp; t < nt; t += tstep) {
        size_t end;
        const size_t e0 = tl.first((unsigned)t, end) + lane;
        double2 x[kTileU];
        const int ew = load_tile(w, e0, end, x);
        int4 a[kTileU];
#pragma unroll
        for (int u = 0; u < kTileU; ++u) a[u] = limbs2(x[u], ew);
        for (int y0 = ya; y0 < yb; y0 += rows) {
            const int ny = min(rows, yb - y0);
            const int ev = myrow < ny ? VE[(size_t)(y0 + myrow) * nt + t] : 0;
            long long v[NV];
            unsigned lo[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) { v[i] = 0; lo[i] = 0; }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (q >= ny) break;
                asm volatile("cp.async.wait_group %0;" ::"n"(kGsStages - 2) : "memory");
                prefetch();                      // into the slot of the row before this one
                const int4* row = ring + cs * kTile;
                cs = cs == kGsStages - 1 ? 0 : cs + 1;
                long long hr = 0, cr = 0, hi = 0, ci = 0, hn = 0, cn = 0;
#pragma unroll
                for (int u = 0; u < kTileU; ++u) {
                    const int4 b = row[32 * u];
                    // conj(b) a = (bx ax + by ay) + i (bx ay - by ax)
                    mad(hr, b.x, a[u].x); mad(hr, b.z, a[u].z);
                    mad(cr, b.x, a[u].y); mad(cr, b.y, a[u].x);
                    mad(cr, b.z, a[u].w); mad(cr, b.w, a[u].z);
                    mad(hi, b.x, a[u].z); mad(hn, b.z, a[u].x);
                    mad(ci, b.x, a[u].w); mad(ci, b.y, a[u].z);
                    mad(cn, b.z, a[u].y); mad(cn, b.w, a[u].x);
                }
                split65(hr, cr, v[2 * q], lo[2 * q]);
                // the cross sums' difference could overflow: carry their high parts into hh first
                split65(hi - hn + (ci >> 30) - (cn >> 30), (ci & 0x3fffffff) - (cn & 0x3fffffff), v[2 * q + 1],
                        lo[2 * q + 1]);
            }
            const long long sv = warp_sum_values<NV>(v, lane);
            const unsigned sl = warp_sum_values<NV>(lo, lane);
            if (lane % (32 / NV) == 0 && myrow < ny) {
                // integers scaled by 2^(59 - Ev) 2^(59 - Ew)
                const int p = (ev - 1023) + (ew - 1023) - 118;
                double s = fma((double)sv, pow2(p + 65), (double)sl * pow2(p + 39));
                if (ev == kExpBad || ew == kExpBad) s = nan;
                sum[wp][2 * y0 + myval] += s;
            }
        }
        if (blockIdx.y == 0) {
            // |w|^2: both factors are the same number, so the l l products add up and are kept
            long long hr = 0, cr = 0, ll = 0;
#pragma unroll
            for (int u = 0; u < kTileU; ++u) {
                mad(hr, a[u].x, a[u].x); mad(hr, a[u].z, a[u].z);
                mad(cr, a[u].x, a[u].y); mad(cr, a[u].z, a[u].w);
                mad(ll, a[u].y, a[u].y); mad(ll, a[u].w, a[u].w);
            }
            long long v[2];
            unsigned lo[2];
            split65(hr + (cr >> 29), ((cr & 0x1fffffff) << 1) + (ll >> 30), v[0], lo[0]);
            v[1] = 0;
            lo[1] = 0;
            const long long sv = warp_sum_values<2>(v, lane);
            const unsigned sl = warp_sum_values<2>(lo, lane);
            if (lane == 0) {
                const int p = 2 * (ew - 1023) - 118;
                sum[wp][2 * 64] += ew == kExpBad ? nan : fma((double)sv, pow2(p + 65), (double)sl * pow2(p + 39));
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int q = 2 * ya + threadIdx.x; q < 2 * yb; q += kGsThreads) {
        const int y = q >> 1;
        double s = 0.0;
#pragma unroll
        for (int u = 0; u < kGsWarps; ++u) s += sum[u][q];
        reinterpret_cast<double*>(partial + (size_t)y * gridDim.x + blockIdx.x)[q & 1] = s;
    }
    if (threadIdx.x == 0 && blockIdx.y == 0) {
        double s = 0.0;
#pragma unroll
        for (int u = 0; u < kGsWarps; ++u) s += sum[u][2 * 64];
        partial[(size_t)k * gridDim.x + blockIdx.x] = make_double2(s, 0.0);
    }
    if constexpr (LAST) {
        if (!last_cta(cnt + r, gridDim.x * gridDim.y)) return;
        // few partial sums: added here, four lanes to a row
        for (int y = threadIdx.x >> 2; y < ((k + 1 + 7) & ~7); y += kGsThreads / 4) {
            double2 s = make_double2(0.0, 0.0);
            if (y <= k)
                for (int e = threadIdx.x & 3; e < gridDim.x; e += 4) {
                    const double2 a = __ldcg(partial + (size_t)y * gridDim.x + e);
                    s.x += a.x;
                    s.y += a.y;
                }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
            }
            if ((threadIdx.x & 3) == 0 && y <= k) out[r * ks.so + y] = s;
        }
    }
}

__global__ void __launch_bounds__(128) k_gs_reduce(const double2* __restrict__ partial, int np, double2* out,
                                                   const int* flag, KS ks) {
    pdl_prologue();
    const int r = blockIdx.z;
    if (inactive_gs(ks, r)) return;
    partial += r * ks.sp;
    out += r * ks.so;
    if (flag && flag[r] == 0) {
        if (threadIdx.x == 0) out[blockIdx.y] = make_double2(0.0, 0.0);
        return;
    }
    double2 acc = make_double2(0.0, 0.0);
    for (int e = threadIdx.x; e < np; e += 128) {
        const double2 a = partial[(size_t)blockIdx.y * np + e];
        acc.x += a.x;
        acc.y += a.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
    }
    __shared__ double2 sh[4];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0)
        out[blockIdx.y] = make_double2((sh[0].x + sh[1].x) + (sh[2].x + sh[3].x), (sh[0].y + sh[1].y) + (sh[2].y + sh[3].y));
}

// CTAs along the tiles: whole rounds of tiles per warp; at most GS_CTAS, and for
// a batch about two waves in all (a CTA's fixed cost then falls on many tiles)
static int gs_ctas(const Tiles& tl, int nrhs) {
    const size_t nt = tl.count;
    const size_t most = (size_t)std::max(16, std::min(GS_CTAS, 2 * GS_CTAS / nrhs)) * kGsWarps;
    const size_t per = (nt + most - 1) / most;
    return (int)((nt + per * kGsWarps - 1) / (per * kGsWarps));
}

// Rows go to groups in different CTAs while the tiles alone fill less than half the chip;
// then a group is as small as fills it (one or two rows: all its loads are in flight at
// once).  Up to kGsFew partial sums a row, the last CTA adds them (one launch less): one
// source at 64 x 64, k = 20, 7.3 us and 4 us for the sum -> 9.0 us with it.
void launch_dot_norm(const int4* VL, const int* VE, int k, const double2* w, const Tiles& tl, double2* partial, double2* out,
                     const int* flag, int* cnt, int nrhs, const KS& ks, cudaStream_t st) {
    const int nc = gs_ctas(tl, nrhs);
    const bool split = (size_t)nc * nrhs * 2 <= GS_CTAS;
    int rows = split ? std::min(kGsRows, std::max(1, (k * nc * nrhs + GS_CTAS - 1) / GS_CTAS)) : kGsRows;
    const int groups = (k + rows - 1) / rows;
    rows = (k + groups - 1) / groups;
    const bool last = nc <= kGsFew;
    const dim3 g(nc, split ? (k + rows - 1) / rows : 1, nrhs), b(kGsThreads);
    switch (rows) {
#define BAH_GS_DOT(R)                                                                                                   \
    case R:                                                                                                             \
        launch_pdl(last ? k_gs_dot<R, true> : k_gs_dot<R, false>, g, b, kGsSmem, st, VL, VE, k, rows, w, tl, partial, out, \
                   flag, cnt, ks);                                                                                      \
        break;
        BAH_GS_DOT(1) BAH_GS_DOT(2) BAH_GS_DOT(3) BAH_GS_DOT(4) BAH_GS_DOT(5) BAH_GS_DOT(6) BAH_GS_DOT(7) BAH_GS_DOT(8)
#undef BAH_GS_DOT
    }
    if (!last) launch_pdl(k_gs_reduce, dim3(1, k + 1, nrhs), dim3(128), 0, st, (const double2*)partial, nc, out, flag, ks);
}

int dot_ctas(const Tiles& tl, int nrhs) { return gs_ctas(tl, nrhs); }
int dot_launches(const Tiles& tl, int nrhs) { return gs_ctas(tl, nrhs) <= kGsFew ? 1 : 2; }

// ---------------------------------------------------------------------------
// w -= sum_i coef_i V_i, and per-CTA partial sums of |w_new|^2.  One warp per
// tile: the coefficients are scaled so that every row's products share one
// exponent Eo (the largest of row exponent + coefficient exponent), lane i
// converting row i's to limbs in shared memory; the sum over the rows is an
// exact integer, rounded once and subtracted from w in FP64.  The rows, and w
// as the last row of each tile, come through the same ring as in k_gs_dot.
// ---------------------------------------------------------------------------
// ||w'||^2 from the CTAs' sums (thread 0 holds this CTA's), by the last CTA: after pass 1
// the DGKS decision too.  Separate kernels for this cost 4.7 and 4 us per step.
__device__ __forceinline__ void gs_norm(double s, double* npart, const double2* coef, int k, int r, int pass,
                                        const GsNorm& nm) {
    if (threadIdx.x == 0) npart[blockIdx.x] = s;
    if (!last_cta(nm.cnt + r, gridDim.x)) return;
    __shared__ double sh[kGsWarps];
    s = 0.0;
    for (int e = threadIdx.x; e < gridDim.x; e += kGsThreads) s += __ldcg(npart + e);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    s = (sh[0] + sh[1]) + (sh[2] + sh[3]);
    double* sc = nm.sc + r * 8;
    sc[2] = sqrt(s);
    if (pass == 1) {
        const int f = s < nm.eta2 * coef[k].x ? 1 : 0;           // coef[k]: ||w||^2 before pass 1
        nm.flag[r] = f;
        sc[3] += (double)f;
    }
}

// the coefficients' share of the common exponent, for the rows lane and lane + 32
struct GsCoef {
    double2 c[2];
    int ec[2];
    bool bad;
    __device__ __forceinline__ GsCoef(const double2* coef, int k, int lane) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = lane + 32 * q;
            c[q] = i < k ? coef[i] : make_double2(0.0, 0.0);
            ec[q] = max(abs_hi(c[q].x), abs_hi(c[q].y)) >> 20;   // biased exponent field (0: no contribution)
        }
        bad = __any_sync(0xffffffffu, ec[0] == 0x7ff || ec[1] == 0x7ff);
    }
    // limbs of every coefficient scaled to the tile's common exponent; returns the scale of the
    // sums, whose units are 2^(60 - sb) of integers scaled by 2^(59 - Ev) 2^(59 - Ec)
    __device__ __forceinline__ double limbs(const int (&ev)[2], int k, int lane, int head, int sb, int4* out) const {
        int eo = 0;
        bool b = bad;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            b |= ev[q] == kExpBad;
            if (ec[q] > 0) eo = max(eo, ev[q] + ec[q] + 1 + head);
        }
        eo = (int)__reduce_max_sync(0xffffffffu, (unsigned)eo);  // biased twice
        b = __any_sync(0xffffffffu, b);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = lane + 32 * q;
            if (i < k) {
                const int eb = eo - ev[q];                       // exponent the coefficient is scaled to
                out[i] = ec[q] > 0 && eb >= kExpMin ? limbs2(c[q], eb) : make_int4(0, 0, 0, 0);
            }
        }
        __syncwarp();
        return b ? __longlong_as_double(0x7ff8000000000000ll) : pow2((eo - 2 * 1023) - 118 + 60 - sb);
    }
};
// the coefficients keep 58 bits, so hh holds 2k products of 2^56: 32 rows fit 2^62, and
// the shift sb uses the bits left
__device__ __forceinline__ int gs_head(int k) { return k > 32 ? 3 : 2; }
__device__ __forceinline__ int gs_shift(int k) {
    return k > 16 ? 0 : (k > 8 ? 1 : (k > 4 ? 2 : (k > 2 ? 3 : (k > 1 ? 4 : 5))));
}
// hh and cross sums of c b, both parts, over one row's entries
__device__ __forceinline__ void gs_row(const int4* row, const int4& cc, long long (&hr)[kTileU], long long (&cr)[kTileU],
                                       long long (&hi)[kTileU], long long (&ci)[kTileU]) {
    const int nz = -cc.z, nw = -cc.w;
#pragma unroll
    for (int u = 0; u < kTileU; ++u) {
        const int4 b = row[32 * u];
        // c b = (cx bx - cy by) + i (cx by + cy bx)
        mad(hr[u], cc.x, b.x); mad(hr[u], nz, b.z);
        mad(cr[u], cc.x, b.y); mad(cr[u], cc.y, b.x);
        mad(cr[u], nz, b.w); mad(cr[u], nw, b.z);
        mad(hi[u], cc.x, b.z); mad(hi[u], cc.z, b.x);
        mad(ci[u], cc.x, b.w); mad(ci[u], cc.y, b.z);
        mad(ci[u], cc.z, b.y); mad(ci[u], cc.w, b.x);
    }
}
// the cross sums hold 8 rows: carry into hh
__device__ __forceinline__ void gs_carry(long long (&hr)[kTileU], long long (&cr)[kTileU], long long (&hi)[kTileU],
                                         long long (&ci)[kTileU]) {
#pragma unroll
    for (int u = 0; u < kTileU; ++u) {
        hr[u] += cr[u] >> 30; cr[u] &= 0x3fffffff;
        hi[u] += ci[u] >> 30; ci[u] &= 0x3fffffff;
    }
}
// x - the sum, rounded once to 2^(60 - sb)
__device__ __forceinline__ double gs_sub(double x, long long h, long long c, int sb, double sc) {
    return fma(-(double)((h << sb) + ((c + (1ll << (29 - sb))) >> (30 - sb))), sc, x);
}

__global__ void __launch_bounds__(kGsThreads, 4) k_gs_axpy(const int4* __restrict__ VL, const int* __restrict__ VE, int k,
                                                           const double2* __restrict__ coef, double2* __restrict__ w,
                                                           Tiles tl, double* __restrict__ npart, int pass, GsNorm nm, KS ks) {
    pdl_prologue();
    const int r = blockIdx.z;
    if (inactive_gs(ks, r) || (pass == 2 && nm.flag[r] == 0)) return;
    const size_t nt = tl.count, npad = nt * kTile;
    VL += r * ks.sv;
    VE += r * ks.se;
    w += r * ks.sw;
    coef += r * ks.so;
    npart += r * GS_CTAS;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const size_t tstep = (size_t)gridDim.x * kGsWarps;
    size_t t = (size_t)blockIdx.x * kGsWarps + wp;
    extern __shared__ __align__(128) int4 ring_all[];
    const int4* ring = ring_all + (size_t)wp * kGsStages * kTile + lane;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    size_t pt = t;
    int py = 0, ps = 0, cs = 0;
    auto prefetch = [&]() {                                      // row py of tile pt (row k: w)
        if (pt < nt) {
            const uint32_t dst = ring_s + (uint32_t)(ps * kTile) * 16u;
            if (py < k) {
                const int4* src = VL + (size_t)py * npad + pt * kTile + lane;
#pragma unroll
                for (int u = 0; u < kTileU; ++u) copy16(dst + 512u * u, src + 32 * u);
                ++py;
            } else {
                size_t end;
                const size_t e0 = tl.first((unsigned)pt, end) + lane;
#pragma unroll
                for (int u = 0; u < kTileU; ++u)
                    if (e0 + 32 * u < end) copy16(dst + 512u * u, w + e0 + 32 * u);
                py = 0;
                pt += tstep;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ps = ps == kGsStages - 1 ? 0 : ps + 1;
    };
#pragma unroll
    for (int i = 0; i < kGsStages - 1; ++i) prefetch();
    auto next_row = [&]() -> const int4* {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGsStages - 2) : "memory");
        prefetch();                                              // into the slot of the row before this one
        const int4* row = ring + cs * kTile;
        cs = cs == kGsStages - 1 ? 0 : cs + 1;
        return row;
    };
    __shared__ int4 csh[kGsWarps][64];
    const GsCoef gc(coef, k, lane);
    int evn[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) evn[q] = lane + 32 * q < k && t < nt ? VE[(size_t)(lane + 32 * q) * nt + t] : kExpMin;
    const int head = gs_head(k), sb = gs_shift(k);
    double nn = 0.0;
    for (; t < nt; t += tstep) {
        int ev[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = lane + 32 * q;
            ev[q] = evn[q];
            evn[q] = i < k && t + tstep < nt ? VE[(size_t)i * nt + t + tstep] : kExpMin;
        }
        const double sc = gc.limbs(ev, k, lane, head, sb, csh[wp]);
        long long hr[kTileU], cr[kTileU], hi[kTileU], ci[kTileU];
#pragma unroll
        for (int u = 0; u < kTileU; ++u) hr[u] = cr[u] = hi[u] = ci[u] = 0;
        for (int i = 0; i < k; ++i) {
            gs_row(next_row(), csh[wp][i], hr, cr, hi, ci);
            if ((i & 7) == 7) gs_carry(hr, cr, hi, ci);
        }
        const double2* wrow = reinterpret_cast<const double2*>(next_row());
        size_t end;
        const size_t e0 = tl.first((unsigned)t, end) + lane;
#pragma unroll
        for (int u = 0; u < kTileU; ++u) {
            if (e0 + 32 * u < end) {
                double2 x = wrow[32 * u];
                x.x = gs_sub(x.x, hr[u], cr[u], sb, sc);
                x.y = gs_sub(x.y, hi[u], ci[u], sb, sc);
                w[e0 + 32 * u] = x;
                nn = fma(x.x, x.x, nn);
                nn = fma(x.y, x.y, nn);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
    __shared__ double sh[kGsWarps];
    if (lane == 0) sh[wp] = nn;
    __syncthreads();
    gs_norm((sh[0] + sh[1]) + (sh[2] + sh[3]), npart, coef, k, r, pass, nm);
}

// The same with one tile per CTA, its rows split over the four warps: on a small grid a
// warp that takes 20 rows in turn is a chain of load latencies (one source at 64 x 64,
// k = 20, 12 CTAs: 10.7 us; so 48 CTAs, 8.9 us with the norm, of which 4 to 5 was a launch
// of its own).  The warps' sums are integers, so that their total does not
// depend on the split.  ST: ring slots per warp.
template <int ST>
__global__ void __launch_bounds__(kGsThreads, ST > 3 ? 2 : 4) k_gs_axpy_split(const int4* __restrict__ VL, const int* __restrict__ VE,
                                                                 int k, const double2* __restrict__ coef,
                                                                 double2* __restrict__ w, Tiles tl,
                                                                 double* __restrict__ npart, int pass, GsNorm nm, KS ks) {
    pdl_prologue();
    const int r = blockIdx.z;
    if (inactive_gs(ks, r) || (pass == 2 && nm.flag[r] == 0)) return;
    const size_t nt = tl.count, npad = nt * kTile, t = blockIdx.x;
    size_t end;
    const size_t e0 = tl.first((unsigned)t, end);
    VL += r * ks.sv;
    VE += r * ks.se;
    w += r * ks.sw;
    coef += r * ks.so;
    npart += r * GS_CTAS;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int per = (k + kGsWarps - 1) / kGsWarps, i0 = min(k, wp * per), i1 = min(k, i0 + per);
    extern __shared__ __align__(128) int4 ring_all[];
    const int4* ring = ring_all + (size_t)wp * ST * kTile + lane;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    int py = i0, ps = 0, cs = 0;
    auto prefetch = [&]() {
        if (py < i1) {
            const int4* src = VL + (size_t)py * npad + t * kTile + lane;
#pragma unroll
            for (int u = 0; u < kTileU; ++u) copy16(ring_s + (uint32_t)(ps * kTile) * 16u + 512u * u, src + 32 * u);
            ++py;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ps = ps == ST - 1 ? 0 : ps + 1;
    };
#pragma unroll
    for (int i = 0; i < ST - 1; ++i) prefetch();
    // the two entries of w that this thread finishes
    double2 x[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const size_t e = e0 + threadIdx.x + kGsThreads * q;
        x[q] = e < end ? w[e] : make_double2(0.0, 0.0);
    }
    __shared__ int4 csh[kGsWarps][64];
    int ev[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) ev[q] = lane + 32 * q < k ? VE[(size_t)(lane + 32 * q) * nt + t] : kExpMin;
    const GsCoef gc(coef, k, lane);
    const int head = gs_head(k), sb = gs_shift(k);
    const double sc = gc.limbs(ev, k, lane, head, sb, csh[wp]);
    long long hr[kTileU], cr[kTileU], hi[kTileU], ci[kTileU];
#pragma unroll
    for (int u = 0; u < kTileU; ++u) hr[u] = cr[u] = hi[u] = ci[u] = 0;
    for (int i = i0; i < i1; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
        prefetch();                              // into the slot of the row before this one
        gs_row(ring + cs * kTile, csh[wp][i], hr, cr, hi, ci);
        cs = cs == ST - 1 ? 0 : cs + 1;
        if (((i - i0) & 7) == 7) gs_carry(hr, cr, hi, ci);
    }
    gs_carry(hr, cr, hi, ci);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    // the sums of all warps, over the warp's own ring: [sum][entry], 8 KB of its at least 12
    long long* acc = reinterpret_cast<long long*>(ring_all + (size_t)wp * ST * kTile);
#pragma unroll
    for (int u = 0; u < kTileU; ++u) {
        acc[lane + 32 * u] = hr[u];
        acc[kTile + lane + 32 * u] = cr[u];
        acc[2 * kTile + lane + 32 * u] = hi[u];
        acc[3 * kTile + lane + 32 * u] = ci[u];
    }
    __syncthreads();
    double nn = 0.0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = threadIdx.x + kGsThreads * q;
        long long s[4] = {0, 0, 0, 0};
#pragma unroll
        for (int v = 0; v < kGsWarps; ++v) {
            const long long* a = reinterpret_cast<const long long*>(ring_all + (size_t)v * ST * kTile);
#pragma unroll
            for (int z = 0; z < 4; ++z) s[z] += a[z * kTile + e];
        }
        if (e0 + e < end) {
            x[q].x = gs_sub(x[q].x, s[0], s[1], sb, sc);
            x[q].y = gs_sub(x[q].y, s[2], s[3], sb, sc);
            w[e0 + e] = x[q];
            nn = fma(x[q].x, x[q].x, nn);
            nn = fma(x[q].y, x[q].y, nn);
        }
    }
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
    __shared__ double sh[kGsWarps];
    if (lane == 0) sh[wp] = nn;
    __syncthreads();
    gs_norm((sh[0] + sh[1]) + (sh[2] + sh[3]), npart, coef, k, r, pass, nm);
}
constexpr int kGsDeep = 6;
constexpr size_t kGsDeepSmem = (size_t)kGsWarps * kGsDeep * kTile * sizeof(int4);

// one tile per CTA while all of them run at once (four CTAs to an SM; with a CTA or two to
// an SM the deeper ring)
void launch_axpy_norm(const int4* VL, const int* VE, int k, const double2* coef, double2* w, const Tiles& tl, double* npart,
                      int pass, const GsNorm& nm, int nrhs, const KS& ks, cudaStream_t st) {
    const size_t nt = tl.count;
    const dim3 b(kGsThreads);
    if (nt * nrhs <= GS_CTAS / 2)
        launch_pdl(k_gs_axpy_split<kGsDeep>, dim3((unsigned)nt, 1, nrhs), b, kGsDeepSmem, st, VL, VE, k, coef, w, tl, npart, pass,
                   nm, ks);
    else if (nt * nrhs <= GS_CTAS)
        launch_pdl(k_gs_axpy_split<kGsStages>, dim3((unsigned)nt, 1, nrhs), b, kGsSmem, st, VL, VE, k, coef, w, tl, npart, pass,
                   nm, ks);
    else
        launch_pdl(k_gs_axpy, dim3(gs_ctas(tl, nrhs), 1, nrhs), b, kGsSmem, st, VL, VE, k, coef, w, tl, npart, pass, nm, ks);
}

int gs_prepare() {
    const void* fn[] = {
#define BAH_GS_DOT(R) (const void*)k_gs_dot<R, true>, (const void*)k_gs_dot<R, false>,
        BAH_GS_DOT(1) BAH_GS_DOT(2) BAH_GS_DOT(3) BAH_GS_DOT(4) BAH_GS_DOT(5) BAH_GS_DOT(6) BAH_GS_DOT(7) BAH_GS_DOT(8)
#undef BAH_GS_DOT
        (const void*)k_gs_axpy, (const void*)k_gs_axpy_split<kGsStages>};
    for (const void* f : fn)
        BAH_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGsSmem));
    BAH_CUDA_TRY(cudaFuncSetAttribute(k_gs_axpy_split<kGsDeep>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGsDeepSmem));
    return BAH_OK;
}

// ---------------------------------------------------------------------------
// v = w / sc[slot]: the vector as the next preconditioner input (rounded to
// FP32 for an FP32 preconditioner, which then reads half the bytes and converts
// nothing: the distributor of 32 sources of 1024 x 512 493 -> 116 us) and its limbs and tile exponents in the basis
// ---------------------------------------------------------------------------
template <class Vc>
__global__ void __launch_bounds__(kGsThreads) k_gs_store(const double2* w, const double* sc, int slot,
                                                         Vc* vc, size_t svc, int4* __restrict__ vl,
                                                         int* __restrict__ ve, Tiles tl, size_t sw, KS ks, int givens,
                                                         GivensArgs gv) {
    pdl_prologue();
    const int r = blockIdx.y;
    // the first CTA runs the step's Givens update beside the copy (a launch of its own took 11 us)
    if (givens && blockIdx.x == 0) return arnoldi_givens(gv, r, ks);
    if (inactive_gs(ks, r)) return;
    const size_t nt = tl.count;
    w += r * sw;
    if (vc) vc += r * svc;
    vl += r * ks.sv;
    ve += r * ks.se;
    const int lane = threadIdx.x & 31;
    const double s = 1.0 / sc[r * 8 + slot];
    const size_t t = (size_t)(blockIdx.x - givens) * kGsWarps + (threadIdx.x >> 5);
    if (t < nt) {
        size_t end;
        const size_t e0 = tl.first((unsigned)t, end) + lane;
        double2 x[kTileU];
        int mx = 0;
#pragma unroll
        for (int u = 0; u < kTileU; ++u) x[u] = e0 + 32 * u < end ? w[e0 + 32 * u] : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < kTileU; ++u) {
            if (e0 + 32 * u < end) {
                x[u].x *= s;
                x[u].y *= s;
                if (vc) vc[e0 + 32 * u] = cconv<Vc>(x[u]);
            }
            mx = max(mx, max(abs_hi(x[u].x), abs_hi(x[u].y)));
        }
        const int eb = tile_exp((int)__reduce_max_sync(0xffffffffu, (unsigned)mx));
        if (lane == 0) ve[t] = eb;
#pragma unroll
        for (int u = 0; u < kTileU; ++u) vl[t * kTile + lane + 32 * u] = limbs2(x[u], eb);
    }
}
template <class Vc>
void launch_basis_store(const double2* w, const double* sc, int slot, Vc* vc, size_t svc, int4* vl, int* ve, const Tiles& tl,
                        size_t sw, int nrhs, const KS& ks, cudaStream_t st, const GivensArgs* gv) {
    const size_t nt = tl.count;
    const int givens = gv ? 1 : 0;
    launch_pdl(k_gs_store<Vc>, dim3((unsigned)((nt + kGsWarps - 1) / kGsWarps) + givens, nrhs), dim3(kGsThreads), 0, st, w, sc,
               slot, vc, svc, vl, ve, tl, sw, ks, givens, gv ? *gv : GivensArgs());
}
template void launch_basis_store<double2>(const double2*, const double*, int, double2*, size_t, int4*, int*, const Tiles&, size_t, int,
                                          const KS&, cudaStream_t, const GivensArgs*);
template void launch_basis_store<float2>(const double2*, const double*, int, float2*, size_t, int4*, int*, const Tiles&, size_t, int,
                                         const KS&, cudaStream_t, const GivensArgs*);

}  // namespace bah
