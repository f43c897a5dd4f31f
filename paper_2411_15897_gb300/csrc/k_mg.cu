// Multigrid level kernels for the acoustic blocks (Sec. 2.2, Algorithm 1;
// Sec. 4.4.1): damped Jacobi relaxation, residual, restriction (Eq. 4.1, 4.2,
// 4.4), bilinear prolongation and the dense FP64 coarsest solve.  Every kernel
// is batched over the blocks of one set (blockIdx.y = block) so the d
// independent displacement blocks run in one launch.
//
// Level 0 reads the 5-point operator from per-point coefficient arrays
// (Fine5); coarser levels read explicit Galerkin stencils of radius (rx, rz).
#include "bah_internal.cuh"
#include "fix60.cuh"
#include "intergrid.cuh"
#include "mg_device.cuh"

#include <algorithm>
#include <cstdlib>

namespace bah {


template <class LS>
static inline int max_radius(const LS& s) {
    int r = 0;
    for (int z = 0; z < s.nb; ++z) r = std::max(r, std::max(s.blk[z].rx, s.blk[z].rz));
    return r;
}

// threads per CTA: in FP64 one warp instruction takes 16 clocks of the SM's pipe,
// so small CTAs spread a small level over more SMs
template <int MODE> constexpr int kTpb = MODE == BAH_FP64 ? 64 : 256;

// ---------------------------------------------------------------------------
// damped Jacobi:  x_out = x_in + w D^{-1} (b - A x_in)   (zero_init: w D^{-1} b, on level 0;
// below it the restriction writes the first sweep).  FP64 launches it for the first sweep only;
// compiled for that alone (24 registers instead of 42), 20 steps of 512 x 512 took 14.54 ms
// instead of 14.48, so the general path stays beside it.
// ---------------------------------------------------------------------------
template <int MODE, bool L0, int RM>
__global__ void __launch_bounds__(kTpb<MODE>) k_jacobi(LvlSet<typename MGT<MODE>::V, typename MGT<MODE>::CC> s,
                                                Fine5<typename MGT<MODE>::C, typename MGT<MODE>::CC> f5,
                                                typename MGT<MODE>::R w, int zero_init) {
    pdl_prologue();
    using V = typename MGT<MODE>::V;
    const auto& B = s.blk[blockIdx.y];
    const int n1 = s.n1, n2 = s.n2, np = n1 * n2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int rr = blockIdx.z;
    if (t >= np || (s.active && !s.active[rr])) return;
    V* __restrict__ xout = B.xout + rr * B.sxo;
    const int i = t % n1, j = t / n1;
    if (!valid_pt(B.type, i, j)) { xout[t] = czero<V>(); return; }
    const V b = B.b[rr * B.sb + t];
    if (zero_init) {
        if constexpr (MODE == BAH_FP64) {
            xout[t] = cscale(cmul(B.idg[t], b), w);
            return;
        } else if constexpr (L0) {
            xout[t] = cscale(cdiv(b, diag_only<MODE>(&f5, B, np, t)), w);
            return;
        }
    }
    const V* __restrict__ xin = B.xin + rr * B.sxi;
    auto X = [&](int g) { return xin[g]; };
    V ax;
    if (L0) ax = apply_fine5_fn<MODE>(f5, B.type, i, j, t, X);
    else ax = apply_stencil_fn<MODE, RM>(B.S, B.rx, B.rz, n1, n2, i, j, t, X);
    const V dg = diag_only<MODE>(L0 ? &f5 : nullptr, B, np, t);
    const V corr = cdiv(csub(b, ax), dg);
    const V x = xin[t];
    xout[t] = cmk<V>(x.x + w * corr.x, x.y + w * corr.y);
}

// ---------------------------------------------------------------------------
// residual:  r = b - A x
// ---------------------------------------------------------------------------
template <int MODE, bool L0, int RM>
__global__ void __launch_bounds__(kTpb<MODE>) k_residual(LvlSet<typename MGT<MODE>::V, typename MGT<MODE>::CC> s,
                                                  Fine5<typename MGT<MODE>::C, typename MGT<MODE>::CC> f5) {
    pdl_prologue();
    using V = typename MGT<MODE>::V;
    const auto& B = s.blk[blockIdx.y];
    const int n1 = s.n1, n2 = s.n2, np = n1 * n2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int rr = blockIdx.z;
    if (t >= np || (s.active && !s.active[rr])) return;
    V* __restrict__ xout = B.xout + rr * B.sxo;
    const int i = t % n1, j = t / n1;
    if (!valid_pt(B.type, i, j)) { xout[t] = czero<V>(); return; }
    const V* __restrict__ xin = B.xin + rr * B.sxi;
    auto X = [&](int g) { return xin[g]; };
    V ax;
    if (L0) ax = apply_fine5_fn<MODE>(f5, B.type, i, j, t, X);
    else ax = apply_stencil_fn<MODE, RM>(B.S, B.rx, B.rz, n1, n2, i, j, t, X);
    xout[t] = csub(B.b[rr * B.sb + t], ax);
}

// ---------------------------------------------------------------------------
// FP64 sweep on level 0.  The FP64 pipe (2 operations per clock and SM) bounds it,
// so the diagonal is inverted once at setup and the sweep written
// x_out = (1 - w) x + w D^{-1} (b - (A - D) x): 14 operations per point where
// dividing took 46.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(64) k_sweep64_fine(LvlSet<double2, double2> s, Fine5<double, double2> f5, double w) {
    pdl_prologue();
    const auto& B = s.blk[blockIdx.y];
    const int n1 = s.n1, n2 = s.n2;
    const int t = blockIdx.x * 64 + threadIdx.x, rr = blockIdx.z;
    if (t >= n1 * n2 || (s.active && !s.active[rr])) return;
    double2* __restrict__ xout = B.xout + rr * B.sxo;
    const int i = t % n1, j = t / n1;
    if (!valid_pt(B.type, i, j)) { xout[t] = make_double2(0.0, 0.0); return; }
    const double2* __restrict__ x = B.xin + rr * B.sxi;
    const double2 r = csub_off_fine5(f5, B.type, i, j, t, B.b[rr * B.sb + t], [&](int g) { return x[g]; });
    double2 v = cscale(x[t], 1.0 - w);
    cfma(v, cscale(B.idg[t], w), r);
    xout[t] = v;
}

template <int MODE>
void launch_jacobi(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& s,
                   const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC>* f5, double w, int zero_init,
                   cudaStream_t st) {
    const int np = s.n1 * s.n2, tpb = kTpb<MODE>;
    dim3 g((np + tpb - 1) / tpb, s.nb, s.nrhs);
    using R = typename Prec<MODE>::R;
    const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC> nof{};
    const bool level = !f5 && !zero_init && (MODE == BAH_FP64 || s.staged);
    if (level) return launch_galerkin_level<MODE>(s, w, false, st);
    if constexpr (MODE == BAH_FP64) {
        if (zero_init) launch_pdl(k_jacobi<MODE, false, 1>, dim3(g), dim3(tpb), 0, st, s, nof, w, 1);
        else launch_pdl(k_sweep64_fine, dim3(g), dim3(tpb), 0, st, s, *f5, w);
    } else {
        const int rm = f5 ? 1 : max_radius(s);
        if (f5) launch_pdl(k_jacobi<MODE, true, 1>, dim3(g), dim3(tpb), 0, st, s, *f5, (R)w, zero_init);
        else if (rm <= 1) launch_pdl(k_jacobi<MODE, false, 1>, dim3(g), dim3(tpb), 0, st, s, nof, (R)w, zero_init);
        else launch_pdl(k_jacobi<MODE, false, 2>, dim3(g), dim3(tpb), 0, st, s, nof, (R)w, zero_init);
    }
}
template <int MODE>
void launch_residual(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& s,
                     const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC>* f5, cudaStream_t st) {
    const int np = s.n1 * s.n2, tpb = kTpb<MODE>;
    dim3 g((np + tpb - 1) / tpb, s.nb, s.nrhs);
    const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC> nof{};
    if (!f5 && (MODE == BAH_FP64 || s.staged)) return launch_galerkin_level<MODE>(s, 0.0, true, st);
    if (f5) launch_pdl(k_residual<MODE, true, 1>, dim3(g), dim3(tpb), 0, st, s, *f5);
    else if constexpr (MODE == BAH_MIXED) {
        if (max_radius(s) <= 1) launch_pdl(k_residual<MODE, false, 1>, dim3(g), dim3(tpb), 0, st, s, nof);
        else launch_pdl(k_residual<MODE, false, 2>, dim3(g), dim3(tpb), 0, st, s, nof);
    }
}

// ---------------------------------------------------------------------------
// restriction: b_c = R r_f  (r_f in blk.xout of the fine set)
// ---------------------------------------------------------------------------

// It also writes the coarse level's first sweep from zero (fs), a launch of its own before:
// 3.4 us on 50 x 16, 10.7 us on two FP64 blocks of 256 x 256.  Small CTAs, for the small levels.
constexpr int kTpbR = 64;
template <int MODE>
__global__ void __launch_bounds__(kTpbR) k_restrict(LvlSet<typename MGT<MODE>::V, typename MGT<MODE>::CC> fine,
                                                   PtrSet<typename MGT<MODE>::V> cb, int intergrid,
                                                   FirstSweep<typename MGT<MODE>::V, typename MGT<MODE>::CC> fs) {
    pdl_prologue();
    using V = typename MGT<MODE>::V;
    using R = typename MGT<MODE>::R;
    const auto& B = fine.blk[blockIdx.y];
    const int n1 = fine.n1, n2 = fine.n2, n1c = n1 / 2, n2c = n2 / 2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int rr = blockIdx.z;
    if (t >= n1c * n2c || (fine.active && !fine.active[rr])) return;
    const int I = t % n1c, J = t / n1c;
    V acc = czero<V>();
    if (valid_pt(B.type, I, J)) {
        const bool nodx = B.type == 0, nodz = B.type == 1;
        const V* r = B.xout + rr * B.sxo;
        const int bx = rbase(nodx, intergrid, I), bz = rbase(nodz, intergrid, J);
        R wxs[4], wzs[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            wxs[q] = rw_axis_t<R>(nodx, intergrid, n1, I, bx + q);
            wzs[q] = rw_axis_t<R>(nodz, intergrid, n2, J, bz + q);
        }
        V v[16];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool ok = wzs[a] != R(0) && wxs[q] != R(0);
                v[a * 4 + q] = r[ok ? (bz + a) * n1 + (bx + q) : 0];
            }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const R wgt = wzs[a] * wxs[q];
                acc.x += wgt * v[a * 4 + q].x;
                acc.y += wgt * v[a * 4 + q].y;
            }
    }
    const int y = blockIdx.y;
    pick(cb, y)[rr * cb.s + t] = acc;
    V* x = y == 0 ? fs.x[0] : (y == 1 ? fs.x[1] : fs.x[2]);
    if (!x) return;
    const auto* d = y == 0 ? fs.d[0] : (y == 1 ? fs.d[1] : fs.d[2]);
    x[rr * fs.sx + t] = valid_pt(B.type, I, J) ? first_sweep<MODE>(d, t, acc, fs.w) : czero<V>();
}

template <int MODE>
void launch_restrict(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& fine,
                     typename Prec<MODE>::V* const* coarse_b, int intergrid, cudaStream_t st, size_t coarse_stride,
                     const FirstSweep<typename Prec<MODE>::V, typename Prec<MODE>::CC>& fs) {
    PtrSet<typename Prec<MODE>::V> cb;
    for (int z = 0; z < 3; ++z) cb.p[z] = z < fine.nb ? coarse_b[z] : nullptr;
    cb.s = coarse_stride;
    const int npc = (fine.n1 / 2) * (fine.n2 / 2);
    dim3 g((npc + kTpbR - 1) / kTpbR, fine.nb, fine.nrhs);
    launch_pdl(k_restrict<MODE>, dim3(g), dim3(kTpbR), 0, st, fine, cb, intergrid, fs);
}

// ---------------------------------------------------------------------------
// prolongation and correction: x_f += P e_c  (x_f = blk.xout of the fine set)
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(kTpb<MODE>) k_prolong_add(LvlSet<typename MGT<MODE>::V, typename MGT<MODE>::CC> fine,
                                                     PtrSet<typename MGT<MODE>::V> ce) {
    pdl_prologue();
    using V = typename MGT<MODE>::V;
    using R = typename MGT<MODE>::R;
    const auto& B = fine.blk[blockIdx.y];
    const int n1 = fine.n1, n2 = fine.n2, n1c = n1 / 2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int rr = blockIdx.z;
    if (t >= n1 * n2 || (fine.active && !fine.active[rr])) return;
    const int i = t % n1, j = t / n1;
    if (!valid_pt(B.type, i, j)) return;
    const bool nodx = B.type == 0, nodz = B.type == 1;
    const V* e = pick(ce, (int)blockIdx.y) + rr * ce.s;
    V* xo = B.xout + rr * B.sxo;
    int cx[2], cz[2];
    R wx[2], wz[2];
    pw_pair<R>(nodx, n1, i, cx, wx);
    pw_pair<R>(nodz, n2, j, cz, wz);
    V v[4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int q = 0; q < 2; ++q) v[a * 2 + q] = e[cz[a] * n1c + cx[q]];
    V acc = xo[t];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const R wgt = wz[a] * wx[q];
            acc.x += wgt * v[a * 2 + q].x;
            acc.y += wgt * v[a * 2 + q].y;
        }
    xo[t] = acc;
}

template <int MODE>
void launch_prolong_add(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& fine,
                        const typename Prec<MODE>::V* const* coarse_x, cudaStream_t st, size_t coarse_stride) {
    PtrSet<typename Prec<MODE>::V> ce;
    for (int z = 0; z < 3; ++z) ce.p[z] = z < fine.nb ? const_cast<typename Prec<MODE>::V*>(coarse_x[z]) : nullptr;
    ce.s = coarse_stride;
    const int np = fine.n1 * fine.n2;
    const int tpb = kTpb<MODE>;
    dim3 g((np + tpb - 1) / tpb, fine.nb, fine.nrhs);
    launch_pdl(k_prolong_add<MODE>, dim3(g), dim3(tpb), 0, st, fine, ce);
}

// ---------------------------------------------------------------------------
// coarsest level: x = A_c^{-1} b with the stored FP64 inverse (one warp per
// row).  The inverse and the right-hand side are in block fixed point and the
// products are exact integers (fix60.cuh; rounding relative to the largest entry of
// a row and of the right-hand side, each block's own), at the integer pipe's rate
// instead of 2 FP64 multiply-adds per clock and SM.
// Each CTA converts the right-hand side once; the result is rounded once to
// the cycle's precision.
// ---------------------------------------------------------------------------
template <class V>
__global__ void __launch_bounds__(256) k_coarse_apply(int npts, int rows, PtrSet<const int4> inv, PtrSet<const int> inve,
                                                      PtrSet<const V> b, PtrSet<V> x, const int* active) {
    pdl_prologue();
    const int z = blockIdx.y;
    const int rr = blockIdx.z;
    if (active && !active[rr]) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    extern __shared__ __align__(128) int4 g[];
    __shared__ int red[32];
    const V* bb = pick(b, z) + rr * b.s;
    const int eg = dense_load<V, typename VecTraits<V>::R>(g, npts, red, [&](int c) { return bb[c]; });
    const int r1 = min(npts, (int)(blockIdx.x + 1) * rows);
    for (int row = blockIdx.x * rows + warp; row < r1; row += 8) {
        const double2 s = dense_row(pick(inv, z) + (size_t)row * npts, pick(inve, z)[row], g, eg, npts, lane);
        if (lane == 0) pick(x, z)[rr * x.s + row] = cconv<V>(s);
    }
}
int coarse_prepare() {
    BAH_CUDA_TRY(cudaFuncSetAttribute((const void*)k_coarse_apply<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      4096 * (int)sizeof(int4)));
    BAH_CUDA_TRY(cudaFuncSetAttribute((const void*)k_coarse_apply<double2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      4096 * (int)sizeof(int4)));
    return BAH_OK;
}

template <int MODE>
void launch_coarse_apply(int nb, int npts, const int4* const* inv, const int* const* inve,
                         const typename Prec<MODE>::V* const* b, typename Prec<MODE>::V* const* x, cudaStream_t st,
                         int nrhs, RhsStride rs) {
    using V = typename Prec<MODE>::V;
    PtrSet<const int4> pi;
    PtrSet<const int> pe;
    PtrSet<const V> pb;
    PtrSet<V> px;
    for (int z = 0; z < 3; ++z) {
        pi.p[z] = z < nb ? inv[z] : nullptr;
        pe.p[z] = z < nb ? inve[z] : nullptr;
        pb.p[z] = z < nb ? b[z] : nullptr;
        px.p[z] = z < nb ? x[z] : nullptr;
    }
    pb.s = rs.s0;
    px.s = rs.s1;
    // rows per CTA: eight (one per warp) while all CTAs are resident at once, more for a batch
    int rows = 8;
    while (rows < 64 && (npts + rows - 1) / rows * nb * nrhs > 1216) rows *= 2;
    dim3 g((npts + rows - 1) / rows, nb, nrhs);
    launch_pdl(k_coarse_apply<V>, dim3(g), dim3(256), (size_t)npts * sizeof(int4), st, npts, rows, pi, pe, pb, px,
               rs.active);
}

// ---------------------------------------------------------------------------
// one acoustic block's fine operator in FP64 (the 5-point stencil of Eq. 2.6 /
// 3.4 with the diagonals given in f5): y = A x, or y = b - A x.  The operator
// of the inner block solves of the exact-block preconditioner.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_block_apply64(Fine5<double, double2> f5, int type,
                                                       const double2* __restrict__ x, double2* __restrict__ y,
                                                       const double2* __restrict__ b) {
    pdl_prologue();
    const int n1 = f5.n1, n2 = f5.n2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n1 * n2) return;
    const int i = t % n1, j = t / n1;
    if (!valid_pt(type, i, j)) { y[t] = make_double2(0.0, 0.0); return; }
    const double2 ax = apply_fine5_fn<BAH_FP64>(f5, type, i, j, t, [&](int g) { return x[g]; });
    y[t] = b ? csub(b[t], ax) : ax;
}
void launch_block_apply64(const Fine5<double, double2>& f5, int type, const double2* x, double2* y, const double2* b,
                          cudaStream_t st) {
    const int np = f5.n1 * f5.n2;
    launch_pdl(k_block_apply64, dim3((np + 255) / 256), dim3(256), 0, st, f5, type, x, y, b);
}

#define INST(MODE)                                                                                                 \
    template void launch_jacobi<MODE>(const LvlSet<Prec<MODE>::V, Prec<MODE>::CC>&,                                \
                                      const Fine5<Prec<MODE>::C, Prec<MODE>::CC>*, double, int, cudaStream_t);     \
    template void launch_residual<MODE>(const LvlSet<Prec<MODE>::V, Prec<MODE>::CC>&,                              \
                                        const Fine5<Prec<MODE>::C, Prec<MODE>::CC>*, cudaStream_t);                \
    template void launch_restrict<MODE>(const LvlSet<Prec<MODE>::V, Prec<MODE>::CC>&, Prec<MODE>::V* const*, int,  \
                                        cudaStream_t, size_t, const FirstSweep<Prec<MODE>::V, Prec<MODE>::CC>&);                                                     \
    template void launch_prolong_add<MODE>(const LvlSet<Prec<MODE>::V, Prec<MODE>::CC>&,                           \
                                           const Prec<MODE>::V* const*, cudaStream_t, size_t);                     \
    template void launch_coarse_apply<MODE>(int, int, const int4* const*, const int* const*,                       \
                                            const Prec<MODE>::V* const*, Prec<MODE>::V* const*, cudaStream_t, int, \
                                            RhsStride);
INST(BAH_FP64)
INST(BAH_MIXED)

}  // namespace bah
