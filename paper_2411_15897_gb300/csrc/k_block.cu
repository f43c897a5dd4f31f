// Kernels of block FGMRES: one Krylov space for a block of s right-hand sides
// (the batched form of the outer solve; FGMRES of Sec. 2.2 and Sec. 4 applied
// to a block).  The basis is stored in block fixed point (fix60.cuh): column a
// of basis block i has its limbs at VL + a * sv + i * tiles * 256 and its tile
// exponents at VE + a * se + i * tiles; the newest block also stands as the preconditioner's
// input, in W in FP64 or in its slot of Z in FP32.  W and X hold column b at b * n.
//
//   block dot    C[(i, a), b] = sum_e conj(V_i[a][e]) W[b][e]      ((k s) x s, k blocks)
//   block Gram   C[a, b] = sum_e conj(W[a][e]) W[b][e]
//   block update W[b][e] -= sum_(i, a) V_i[a][e] C[(i, a), b]
//   Cholesky     G = L L^H, R = L^H, T = R^{-1}                    (CholQR, one warp)
//   block scale  V[b][e] = sum_(b' <= b) W[b'][e] T[b', b]         (W R^{-1})
//   solution     X[b][e] += sum_(i, a) Z_i[a][e] Y[(i, a), b]      (Z in the multigrid's precision)
//
// The dots, the Gram matrix, the updates and the scaling sum exact integer
// products; with FP64 multiply-adds (4 per entry, row and column, 2 per clock
// and SM) they were bound by the FP64 pipe.  Now the integer multiply-adds
// bound them (60 % of their rate).  Measured, 8 sources on 256 x 128, 20 block
// steps: 96.1 -> 23.6 ms (dots and updates of 112 rows 195 and 215 us each), of
// which the cycles were a part that has become faster since (20.7 ms).
#include "bah_internal.cuh"
#include "fix60.cuh"

#include <algorithm>

namespace bah {

constexpr int kBlkRows = 64;       // most rows of a dot CTA

__device__ __forceinline__ void bmac(double2& acc, const double2& a, const double2& b) {        // acc += a b
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}

// one warp: a column's entries of tile t as limbs in g[0 .. kTile); the exponent
__device__ __forceinline__ int stage_tile(const double2* __restrict__ w, size_t t, const Tiles& tl, int4* g, int lane) {
    size_t end;
    const size_t e0 = tl.first((unsigned)t, end) + lane;
    double2 x[kTileU];
    int mx = 0;
#pragma unroll
    for (int u = 0; u < kTileU; ++u) x[u] = e0 + 32 * u < end ? w[e0 + 32 * u] : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < kTileU; ++u) mx = max(mx, max(abs_hi(x[u].x), abs_hi(x[u].y)));
    const int eb = tile_exp((int)__reduce_max_sync(0xffffffffu, (unsigned)mx));
#pragma unroll
    for (int u = 0; u < kTileU; ++u) g[32 * u + lane] = limbs2(x[u], eb);
    return eb;
}

// ---------------------------------------------------------------------------
// partial[(row * s + b) * gridDim.x + cta] for the CTA's rpc rows (blockIdx.y)
// and tiles.  The s columns of W are converted to limbs in shared memory once
// per tile and CTA; each warp takes every eighth row, holds its tile in
// registers and meets all columns, so a basis row is read once for s columns.
// SELF: the rows are the columns of W themselves (the l l products, which add
// up where both factors are the same number, are kept).
// ---------------------------------------------------------------------------
template <int S, bool SELF>
__global__ void __launch_bounds__(256, 2) k_bdot(const int4* __restrict__ VL, const int* __restrict__ VE, size_t sv,
                                                 size_t se, int k, int s, int rpc, const double2* __restrict__ W,
                                                 Tiles tl, double2* __restrict__ partial) {
    pdl_prologue();
    extern __shared__ __align__(128) int4 g[];                                   // S x kTile
    constexpr int CG = S < 8 ? S : 8, NV = 2 * CG;                // columns and values of one lane reduction
    __shared__ int ew[S];
    __shared__ double sum[kBlkRows][2 * S];
    const size_t n = tl.n, nt = tl.count, npad = nt * kTile;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int nrow = SELF ? s : k * s, row0 = blockIdx.y * rpc;
    for (int q = threadIdx.x; q < kBlkRows * 2 * S; q += 256) (&sum[0][0])[q] = 0.0;
    const int myval = lane / (32 / NV);
    for (size_t t = blockIdx.x; t < nt; t += gridDim.x) {
        __syncthreads();
        for (int b = wp; b < s; b += 8) {
            const int e = stage_tile(W + (size_t)b * n, t, tl, g + b * kTile, lane);
            if (lane == 0) ew[b] = e;
        }
        __syncthreads();
        for (int rl = wp; rl < rpc && row0 + rl < nrow; rl += 8) {
            const int row = row0 + rl, i = row / s, a = row % s;
            int4 v[kTileU];
            int ev;
            if (SELF) {
                ev = ew[row];
#pragma unroll
                for (int u = 0; u < kTileU; ++u) v[u] = g[row * kTile + 32 * u + lane];
            } else {
                ev = VE[(size_t)a * se + (size_t)i * nt + t];
                const int4* src = VL + (size_t)a * sv + (size_t)i * npad + t * kTile + lane;
#pragma unroll
                for (int u = 0; u < kTileU; ++u) v[u] = __ldg(src + 32 * u);
            }
#pragma unroll 1
            for (int c0 = 0; c0 < s; c0 += CG) {
                long long vh[NV];
                unsigned vl[NV];
#pragma unroll
                for (int q = 0; q < NV; ++q) { vh[q] = 0; vl[q] = 0; }
#pragma unroll
                for (int c = 0; c < CG; ++c) {
                    if (c0 + c >= s) break;
                    const int4* col = g + (c0 + c) * kTile + lane;
                    long long hr = 0, cr = 0, hi = 0, ci = 0, hn = 0, cn = 0, ll = 0, ln = 0;
#pragma unroll
                    for (int u = 0; u < kTileU; ++u) {
                        const int4 w = col[32 * u];
                        // conj(v) w = (vx wx + vy wy) + i (vx wy - vy wx)
                        mad(hr, v[u].x, w.x); mad(hr, v[u].z, w.z);
                        mad(cr, v[u].x, w.y); mad(cr, v[u].y, w.x);
                        mad(cr, v[u].z, w.w); mad(cr, v[u].w, w.z);
                        mad(hi, v[u].x, w.z); mad(hn, v[u].z, w.x);
                        mad(ci, v[u].x, w.w); mad(ci, v[u].y, w.z);
                        mad(cn, v[u].z, w.y); mad(cn, v[u].w, w.x);
                        if (SELF) {
                            mad(ll, v[u].y, w.y); mad(ll, v[u].w, w.w);
                            mad(ln, v[u].y, w.w); mad(ln, -v[u].w, w.y);
                        }
                    }
                    split65(hr + (cr >> 30), (cr & 0x3fffffff) + (ll >> 30), vh[2 * c], vl[2 * c]);
                    split65(hi - hn + (ci >> 30) - (cn >> 30), (ci & 0x3fffffff) - (cn & 0x3fffffff) + (ln >> 30),
                            vh[2 * c + 1], vl[2 * c + 1]);
                }
                const long long th = warp_sum_values<NV>(vh, lane);
                const unsigned tl = warp_sum_values<NV>(vl, lane);
                const int b = c0 + (myval >> 1);
                if (lane % (32 / NV) == 0 && b < s) {
                    const int p = (ev - 1023) + (ew[b] - 1023) - 118;
                    double x = fma((double)th, pow2(p + 65), (double)tl * pow2(p + 39));
                    if (ev == kExpBad || ew[b] == kExpBad) x = __longlong_as_double(0x7ff8000000000000ll);
                    sum[rl][2 * b + (myval & 1)] += x;
                }
            }
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < rpc * s; q += 256) {
        const int rl = q / s, b = q % s;
        if (row0 + rl < nrow)
            partial[((size_t)(row0 + rl) * s + b) * gridDim.x + blockIdx.x] = make_double2(sum[rl][2 * b], sum[rl][2 * b + 1]);
    }
}
// C[row * s + b] = sum over the CTAs' partials (fixed order), one warp each
__global__ void __launch_bounds__(128) k_bdot_reduce(const double2* __restrict__ partial, int np, int count, double2* C) {
    pdl_prologue();
    const int q = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;      // row * s + b
    if (q >= count) return;
    double2 t = make_double2(0.0, 0.0);
    for (int e = lane; e < np; e += 32) {
        const double2 v = partial[(size_t)q * np + e];
        t.x += v.x;
        t.y += v.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
        t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
    if (lane == 0) C[q] = t;
}
template <int S, bool SELF>
static void bdot_t(const int4* VL, const int* VE, size_t sv, size_t se, int k, int s, const double2* W, const Tiles& tl,
                   double2* partial, double2* C, cudaStream_t st) {
    const int rows = SELF ? s : k * s, chunks = (rows + kBlkRows - 1) / kBlkRows;
    const int rpc = ((rows + chunks - 1) / chunks + 7) / 8 * 8;      // equal chunks, whole rounds of the eight warps
    // two CTAs per SM in all, whole rounds of tiles
    const size_t nt = tl.count, most = std::max(1, RED_CTAS / chunks), per = (nt + most - 1) / most;
    const int nc = (int)((nt + per - 1) / per);
    launch_pdl(k_bdot<S, SELF>, dim3(nc, chunks), dim3(256), (size_t)s * kTile * sizeof(int4), st, VL, VE, sv, se, k, s, rpc,
               W, tl, partial);
    launch_pdl(k_bdot_reduce, dim3((rows * s + 3) / 4), dim3(128), 0, st, (const double2*)partial, nc, rows * s, C);
}
void launch_block_dot(const int4* VL, const int* VE, size_t sv, size_t se, int k, int s, const double2* W, const Tiles& tl,
                      double2* partial, double2* C, cudaStream_t st) {
    if (s <= 4) bdot_t<4, false>(VL, VE, sv, se, k, s, W, tl, partial, C, st);
    else if (s <= 8) bdot_t<8, false>(VL, VE, sv, se, k, s, W, tl, partial, C, st);
    else bdot_t<16, false>(VL, VE, sv, se, k, s, W, tl, partial, C, st);
}
void launch_block_gram(int s, const double2* W, const Tiles& tl, double2* partial, double2* C, cudaStream_t st) {
    if (s <= 4) bdot_t<4, true>(nullptr, nullptr, 0, 0, 1, s, W, tl, partial, C, st);
    else if (s <= 8) bdot_t<8, true>(nullptr, nullptr, 0, 0, 1, s, W, tl, partial, C, st);
    else bdot_t<16, true>(nullptr, nullptr, 0, 0, 1, s, W, tl, partial, C, st);
}

// ---------------------------------------------------------------------------
// Sums of one column over rows: a warp's accumulators for the eight entries per
// lane of a tile, sum_row V_row[e] c[row], every row's products sharing the
// exponent eo (biased twice); the coefficients keep 60 - head bits so that the
// rows' products fit 62 bits.  U: entries per lane.
// ---------------------------------------------------------------------------
__host__ __device__ inline int rows_head(int rows) {
    int h = 2;
    while ((8 << h) < rows) ++h;
    return h;
}
template <int U> struct ColSum {
    long long hr[U], cr[U], hi[U], ci[U];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int u = 0; u < U; ++u) hr[u] = cr[u] = hi[u] = ci[u] = 0;
    }
    __device__ __forceinline__ void add(const int4* row, const int4& c) {      // row: this lane's entries at 32 u
        const int nz = -c.z, nw = -c.w;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int4 b = row[32 * u];
            mad(hr[u], c.x, b.x); mad(hr[u], nz, b.z);
            mad(cr[u], c.x, b.y); mad(cr[u], c.y, b.x);
            mad(cr[u], nz, b.w); mad(cr[u], nw, b.z);
            mad(hi[u], c.x, b.z); mad(hi[u], c.z, b.x);
            mad(ci[u], c.x, b.w); mad(ci[u], c.y, b.z);
            mad(ci[u], c.z, b.y); mad(ci[u], c.w, b.x);
        }
    }
    __device__ __forceinline__ void carry() {                                  // at least every 4 rows
#pragma unroll
        for (int u = 0; u < U; ++u) {
            hr[u] += cr[u] >> 30; cr[u] &= 0x3fffffff;
            hi[u] += ci[u] >> 30; ci[u] &= 0x3fffffff;
        }
    }
    // x - sum, with s1 = 2^60 and s2 = 2^30 times the scale of the integers
    __device__ __forceinline__ double2 minus(const double2& x, int u, double s1, double s2) const {
        return make_double2(fma(-(double)hr[u], s1, fma(-(double)cr[u], s2, x.x)),
                            fma(-(double)hi[u], s1, fma(-(double)ci[u], s2, x.y)));
    }
};
__device__ __forceinline__ int coef_exp(const double2& c) { return max(abs_hi(c.x), abs_hi(c.y)) >> 20; }

// W[b][e] -= sum over rows (i, a) < k s of V_i[a][e] C[row, b].  One CTA of S
// warps per half tile (whole tiles left 384 units of work for 304 resident CTAs
// at 256 x 128), warp b on column b; the basis rows pass through a ring of
// shared-memory slots (cp.async, groups of rows, one barrier per group), so a
// row is read once for all columns.
constexpr int kUpG = 8, kUpSlots = 3, kUpU = kTileU / 2, kUpE = 32 * kUpU;
template <int S>
__global__ void __launch_bounds__(32 * S) k_bupdate(const int4* __restrict__ VL, const int* __restrict__ VE, size_t sv,
                                                    size_t se, int k, int s, const double2* __restrict__ C,
                                                    double2* __restrict__ W, Tiles tl) {
    pdl_prologue();
    extern __shared__ __align__(128) int4 ring[];                                // kUpSlots x kUpG x kUpE
    __shared__ int4 csh[S][32];
    const size_t nt = tl.count, npad = nt * kTile;
    const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
    const int rows = k * s, head = rows_head(rows), ngrp = (rows + kUpG - 1) / kUpG;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    for (size_t h = blockIdx.x; h < 2 * nt; h += gridDim.x) {
        const size_t t = h >> 1, eb0 = h * kUpE;                  // tile and its first entry among the padded ones
        auto fetch = [&](int gq) {                                // group gq's rows into its slot
            if (gq < ngrp)
                for (int e = threadIdx.x; e < kUpG * kUpE; e += 32 * S) {
                    const int row = gq * kUpG + e / kUpE;
                    if (row < rows) {
                        const int4* src = VL + (size_t)(row % s) * sv + (size_t)(row / s) * npad + eb0 + e % kUpE;
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                         ring_s + (uint32_t)((gq % kUpSlots) * kUpG * kUpE + e) * 16u),
                                     "l"(src)
                                     : "memory");
                    }
                }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        __syncthreads();                                          // the last tile's slots are free
#pragma unroll
        for (int q = 0; q < kUpSlots - 1; ++q) fetch(q);
        // the common exponent of the column
        int eo = 0;
        bool bad = false;
        if (b < s)
            for (int row = lane; row < rows; row += 32) {
                const int ec = coef_exp(C[(size_t)row * s + b]);
                const int ev = VE[(size_t)(row % s) * se + (size_t)(row / s) * nt + t];
                if (ec > 0) eo = max(eo, ev + ec + 1 + head);
                bad |= ec == 0x7ff || ev == kExpBad;
            }
        eo = (int)__reduce_max_sync(0xffffffffu, (unsigned)eo);
        bad = __any_sync(0xffffffffu, bad);
        ColSum<kUpU> acc;
        acc.clear();
        for (int gq = 0; gq < ngrp; ++gq) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kUpSlots - 2) : "memory");
            __syncthreads();                                      // group gq arrived; every warp is done with gq - 1
            fetch(gq + kUpSlots - 1);
            if (b >= s) continue;
            if ((gq * kUpG) % 32 == 0) {                          // limbs of the next 32 coefficients
                __syncwarp();
                const int row = gq * kUpG + lane;
                if (row < rows) {
                    const double2 c = C[(size_t)row * s + b];
                    const int eb = eo - VE[(size_t)(row % s) * se + (size_t)(row / s) * nt + t];
                    csh[b][lane] = coef_exp(c) > 0 && eb >= kExpMin ? limbs2(c, eb) : make_int4(0, 0, 0, 0);
                }
                __syncwarp();
            }
            const int4* slot = ring + (gq % kUpSlots) * kUpG * kUpE + lane;
            for (int q = 0; q < kUpG && gq * kUpG + q < rows; ++q) {
                acc.add(slot + q * kUpE, csh[b][(gq * kUpG + q) & 31]);
                if ((q & 3) == 3) acc.carry();
            }
            acc.carry();
        }
        if (b < s) {
            // integers scaled by 2^(59 - Ev) 2^(59 - Ec)
            const int p = (eo - 2 * 1023) - 118;
            double s1 = pow2(p + 60), s2 = pow2(p + 30);
            if (bad) s1 = __longlong_as_double(0x7ff8000000000000ll);
            double2* w = W + (size_t)b * tl.n;
            size_t end;
            const size_t e0 = tl.first((unsigned)t, end) + (h & 1) * kUpE + lane;
#pragma unroll
            for (int u = 0; u < kUpU; ++u)
                if (e0 + 32 * u < end) w[e0 + 32 * u] = acc.minus(w[e0 + 32 * u], u, s1, s2);
        }
    }
}
void launch_block_update(const int4* VL, const int* VE, size_t sv, size_t se, int k, int s, const double2* C, double2* W,
                         const Tiles& tl, cudaStream_t st) {
    const size_t smem = (size_t)kUpSlots * kUpG * kUpE * sizeof(int4);
    const unsigned nt = 2 * tl.count;
    if (s <= 4) launch_pdl(k_bupdate<4>, dim3(std::min(nt, 1216u)), dim3(128), smem, st, VL, VE, sv, se, k, s, C, W, tl);
    else if (s <= 8) launch_pdl(k_bupdate<8>, dim3(std::min(nt, 608u)), dim3(256), smem, st, VL, VE, sv, se, k, s, C, W, tl);
    else launch_pdl(k_bupdate<16>, dim3(std::min(nt, 304u)), dim3(512), smem, st, VL, VE, sv, se, k, s, C, W, tl);
}

// ---------------------------------------------------------------------------
// Cholesky factor of the s x s Hermitian G (row-major) and the inverse of
// R = L^H, one warp.  A pivot that is not positive and finite makes R and T NaN
// (the host reads R).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(32) k_bchol(const double2* __restrict__ G, int s, double2* R, double2* T) {
    pdl_prologue();
    __shared__ double2 A[16][17], X[16][17];
    const int lane = threadIdx.x;
    for (int q = lane; q < s * s; q += 32) {
        A[q / s][q % s] = G[q];
        X[q / s][q % s] = make_double2(0.0, 0.0);
    }
    __syncwarp();
    for (int j = 0; j < s; ++j) {
        const double d = A[j][j].x;
        const double l = d > 0.0 && isfinite(d) ? sqrt(d) : __longlong_as_double(0x7ff8000000000000ll);
        const double il = 1.0 / l;
        __syncwarp();
        if (lane == j) A[j][j] = make_double2(l, 0.0);
        else if (lane > j && lane < s) A[lane][j] = cscale(A[lane][j], il);
        __syncwarp();
        // trailing lower triangle: A[i][k] -= L[i][j] conj(L[k][j])
        const int m = s - j - 1;
        for (int q = lane; q < m * m; q += 32) {
            const int i = j + 1 + q / m, k = j + 1 + q % m;
            if (k <= i) bmac(A[i][k], cscale(A[i][j], -1.0), cconj(A[k][j]));
        }
        __syncwarp();
    }
    // X = R^{-1} column by column (lane = column), R[q][k] = conj(L[k][q])
    if (lane < s)
        for (int q = lane; q >= 0; --q) {
            double2 acc = make_double2(q == lane ? 1.0 : 0.0, 0.0);
            for (int k = q + 1; k <= lane; ++k) bmac(acc, cscale(cconj(A[k][q]), -1.0), X[k][lane]);
            X[q][lane] = cscale(acc, 1.0 / A[q][q].x);
        }
    __syncwarp();
    for (int q = lane; q < s * s; q += 32) {
        const int i = q / s, j = q % s;
        R[q] = j >= i ? cconj(A[j][i]) : make_double2(0.0, 0.0);
        T[q] = j >= i ? X[i][j] : make_double2(0.0, 0.0);
    }
}
void launch_block_chol(const double2* G, int s, double2* R, double2* T, cudaStream_t st) {
    launch_pdl(k_bchol, dim3(1), dim3(32), 0, st, G, s, R, T);
}

// V[b] = sum_(b' <= b) W[b'] T[b', b] (T upper triangular, s x s, row-major),
// written to dst (column b at b * sd; may be W itself, or null) and, with vl, as basis
// columns.  One CTA of S warps per tile: warp b converts column b to limbs in
// shared memory, then sums column b of the product.
template <int S, class Vd>
__global__ void __launch_bounds__(32 * S) k_bscale(const double2* W, int s, const double2* __restrict__ T, Vd* dst, size_t sd,
                                                   int4* __restrict__ vl, int* __restrict__ ve, size_t sv, size_t se,
                                                   Tiles tl) {
    pdl_prologue();
    extern __shared__ __align__(128) int4 g[];                                   // S x kTile
    __shared__ int ew[S];
    __shared__ int4 csh[S][16];
    const size_t n = tl.n, nt = tl.count;
    const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
    const double2 c = lane <= b && b < s ? T[lane * s + b] : make_double2(0.0, 0.0);
    const int ec = coef_exp(c), head = 2;
    for (size_t t = blockIdx.x; t < nt; t += gridDim.x) {
        __syncthreads();
        if (b < s) {
            const int e = stage_tile(W + (size_t)b * n, t, tl, g + b * kTile, lane);
            if (lane == 0) ew[b] = e;
        }
        __syncthreads();                                          // all of the tile is in shared memory: dst may be W
        if (b >= s) continue;
        const int ev = lane <= b ? ew[lane] : kExpMin;
        const int eo = (int)__reduce_max_sync(0xffffffffu, ec > 0 ? (unsigned)(ev + ec + 1 + head) : 0u);
        const bool bad = __any_sync(0xffffffffu, ec == 0x7ff || ev == kExpBad);
        __syncwarp();
        if (lane <= b) {
            const int eb = eo - ev;
            csh[b][lane] = ec > 0 && eb >= kExpMin ? limbs2(c, eb) : make_int4(0, 0, 0, 0);
        }
        __syncwarp();
        ColSum<kTileU> acc;
        acc.clear();
        for (int q = 0; q <= b; ++q) {
            acc.add(g + q * kTile + lane, csh[b][q]);
            if ((q & 3) == 3) acc.carry();
        }
        const int p = (eo - 2 * 1023) - 118;
        double s1 = -pow2(p + 60);
        const double s2 = -pow2(p + 30);
        if (bad) s1 = __longlong_as_double(0x7ff8000000000000ll);
        size_t end;
        const size_t e0 = tl.first((unsigned)t, end) + lane;
        double2 x[kTileU];
        int mx = 0;
#pragma unroll
        for (int u = 0; u < kTileU; ++u) {
            x[u] = make_double2(0.0, 0.0);
            if (e0 + 32 * u < end) {
                x[u] = acc.minus(x[u], u, s1, s2);
                if (dst) dst[b * sd + e0 + 32 * u] = cconv<Vd>(x[u]);
            }
            mx = max(mx, max(abs_hi(x[u].x), abs_hi(x[u].y)));
        }
        if (vl) {
            const int eb = tile_exp((int)__reduce_max_sync(0xffffffffu, (unsigned)mx));
            if (lane == 0) ve[(size_t)b * se + t] = eb;
#pragma unroll
            for (int u = 0; u < kTileU; ++u) vl[(size_t)b * sv + t * kTile + lane + 32 * u] = limbs2(x[u], eb);
        }
    }
}
template <class Vd>
void launch_block_scale(const double2* W, int s, const double2* T, Vd* dst, size_t sd, int4* vl, int* ve, size_t sv, size_t se,
                        const Tiles& tl, cudaStream_t st) {
    const size_t smem = (size_t)s * kTile * sizeof(int4);
    const unsigned nt = tl.count;
    if (s <= 4) launch_pdl(k_bscale<4, Vd>, dim3(std::min(nt, 608u)), dim3(128), smem, st, W, s, T, dst, sd, vl, ve, sv, se, tl);
    else if (s <= 8) launch_pdl(k_bscale<8, Vd>, dim3(std::min(nt, 304u)), dim3(256), smem, st, W, s, T, dst, sd, vl, ve, sv, se, tl);
    else launch_pdl(k_bscale<16, Vd>, dim3(std::min(nt, 152u)), dim3(512), smem, st, W, s, T, dst, sd, vl, ve, sv, se, tl);
}

// X[b][e] += sum over rows (i, a) < k s of Z_i[a][e] Y[row, b]  (Z FP32 or FP64 complex)
template <int S, class Vz>
__global__ void __launch_bounds__(256) k_bxupdate(const Vz* __restrict__ Z, size_t sz, int k, int s,
                                                  const double2* __restrict__ Y, double2* __restrict__ X, size_t n) {
    pdl_prologue();
    extern __shared__ double2 ys[];
    for (int q = threadIdx.x; q < k * s * s; q += blockDim.x) ys[q] = Y[q];
    __syncthreads();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        double2 acc[S];
#pragma unroll
        for (int b = 0; b < S; ++b) acc[b] = b < s ? X[(size_t)b * n + e] : make_double2(0.0, 0.0);
        for (int row = 0; row < k * s; ++row) {
            const int i = row / s, a = row % s;
            const Vz zv = Z[(size_t)a * sz + (size_t)i * n + e];
            const double2 z = cconv<double2>(zv);
#pragma unroll
            for (int b = 0; b < S; ++b)
                if (b < s) bmac(acc[b], z, ys[row * s + b]);
        }
#pragma unroll
        for (int b = 0; b < S; ++b)
            if (b < s) X[(size_t)b * n + e] = acc[b];
    }
}
template <class Vz>
void launch_block_xupdate(const Vz* Z, size_t sz, int k, int s, const double2* Y, double2* X, size_t n,
                          cudaStream_t st) {
    const int most = std::max(1, 49152 / (s * s * (int)sizeof(double2)));      // blocks whose coefficients fit 48 KiB
    for (int i = 0; i < k; i += most) {
        const int kk = std::min(most, k - i);
        const size_t smem = (size_t)kk * s * s * sizeof(double2);
        const Vz* z = Z + (size_t)i * n;
        const double2* y = Y + (size_t)i * s * s;
        const dim3 g(RED_CTAS * 2), b(256);
        if (s <= 4) launch_pdl(k_bxupdate<4, Vz>, g, b, smem, st, z, sz, kk, s, y, X, n);
        else if (s <= 8) launch_pdl(k_bxupdate<8, Vz>, g, b, smem, st, z, sz, kk, s, y, X, n);
        else launch_pdl(k_bxupdate<16, Vz>, g, b, smem, st, z, sz, kk, s, y, X, n);
    }
}
int block_prepare() {
    const int ring = (int)(kUpSlots * kUpG * kUpE * sizeof(int4)), cols = (int)(16 * kTile * sizeof(int4));
    const struct { const void* f; int b; } fns[] = {
        {(const void*)k_bdot<16, false>, cols}, {(const void*)k_bdot<16, true>, cols}, {(const void*)k_bscale<16, double2>, cols},
        {(const void*)k_bscale<16, float2>, cols},
        {(const void*)k_bupdate<4>, ring},      {(const void*)k_bupdate<8>, ring},     {(const void*)k_bupdate<16>, ring}};
    for (const auto& q : fns) BAH_CUDA_TRY(cudaFuncSetAttribute(q.f, cudaFuncAttributeMaxDynamicSharedMemorySize, q.b));
    return BAH_OK;
}
template void launch_block_scale<double2>(const double2*, int, const double2*, double2*, size_t, int4*, int*, size_t, size_t,
                                          const Tiles&, cudaStream_t);
template void launch_block_scale<float2>(const double2*, int, const double2*, float2*, size_t, int4*, int*, size_t, size_t,
                                         const Tiles&, cudaStream_t);
template void launch_block_xupdate<float2>(const float2*, size_t, int, int, const double2*, double2*, size_t,
                                           cudaStream_t);
template void launch_block_xupdate<double2>(const double2*, size_t, int, int, const double2*, double2*, size_t,
                                            cudaStream_t);

}  // namespace bah
