// Fused visits of multigrid level 0 (the 5-point operator read from per-point
// coefficients): one launch down (first damped-Jacobi sweep from zero, residual,
// restriction) and one launch up (prolongation, correction and up to three
// sweeps), with the iterate of a 64 x 32-point region in shared memory and each
// thread's right-hand side, coefficients and iterate of four points in
// registers.  The regions of neighbouring CTAs overlap by the halo that the
// sweeps consume and recompute it.
//
// With the separate kernels a V(1,3) visit moves 176 bytes per point in 7
// launches (FP32); these two move 44, and the halo costs 1.2 to 1.4 times the
// arithmetic.  At 512 x 512 the separate launches were bound by latency (4 to 5
// us each; now 8 us down and 8 us up for one block), in batches by DRAM and L2
// traffic.  Bound now: instruction issue.  20 steps: 512 x 512 6.94 -> 6.50 ms,
// 1024 x 1024 18.3 -> 15.7 ms, 32 sources of 1024 x 512 240 -> 214 ms.
//
// Algebra: with g = w / d, the sweep x + w (b - A x) / d is
// (1 - w) x + g (b + sum of k x_neighbour), and the residual after the sweep
// from zero, x = g b, is (1 - w) b + sum of k x_neighbour; the diagonal itself
// does not appear.  A point outside the grid or without an unknown loads b and k at a
// clamped index but has g = 0, so that it starts and stays at x = 0 and the taps need no
// tests; its residual is written as zero.
#include "bah_internal.cuh"
#include "intergrid.cuh"
#include "mg_device.cuh"

namespace bah {

namespace {

constexpr int kW = 64, kH = 32, kThreads = 512, kQ = 4;     // region, threads, points (rows) per thread
constexpr int kP = kW + 2;                                  // shared-memory pitch (zero border)
// CTAs per SM asked of the compiler: two in FP32 (64 registers; with 66 one CTA fits, and
// the 180 CTAs of a 512 x 512 block then take two waves)
template <int MODE> constexpr int kMinCtas = MODE == BAH_MIXED ? 2 : 1;

// one thread's points: one column, rows j0 .. j0 + 3
template <int MODE, int TYPE> struct Points {
    using V = typename Prec<MODE>::V;
    using R = typename Prec<MODE>::R;
    using C = typename Prec<MODE>::C;
    using CC = typename Prec<MODE>::CC;
    V b[kQ], g[kQ], x[kQ];
    C kw[kQ], ke[kQ], kz[kQ + (TYPE == 2 ? 2 : 1)];         // kz: the column's vertical coefficients, shared by rows
    bool in[kQ];

    // Every load is at an index clamped into the grid; a point without an unknown
    // gets g = 0.  f5's diagonals: FP64 their inverses, mixed the diagonals.
    __device__ __forceinline__ void load(const Fine5<C, CC>& f, const V* __restrict__ bp, int i, int j0, R w) {
        const int n1 = f.n1, n2 = f.n2;
        const int ic = min(max(i, 0), n1 - 1), iw = max(ic - 1, 0), ie = min(ic + 1, n1 - 1);
        const CC* __restrict__ dg = TYPE == 0 ? f.dg0 : (TYPE == 1 ? f.dg1 : f.dg2);
        // horizontal neighbours: u1 mu at cells (i - 1, i), u2 at nodes (i, i + 1), p at cells (i - 1, i + 1)
        const C* __restrict__ ax = TYPE == 0 ? f.cx : (TYPE == 1 ? f.nx : f.wx);
        const C* __restrict__ az = TYPE == 0 ? f.nz : (TYPE == 1 ? f.cz : f.wz);
        const int cw = TYPE == 1 ? ic : iw, ce = TYPE == 0 ? ic : ie;
        auto row = [&](int j) { return min(max(j, 0), n2 - 1) * n1; };
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int t = row(j0 + q);
            in[q] = i >= (TYPE == 0 ? 1 : 0) && i < n1 && j0 + q >= (TYPE == 1 ? 1 : 0) && j0 + q < n2;
            kw[q] = ax[t + cw];
            ke[q] = ax[t + ce];
            b[q] = bp[t + ic];
            const V d = ldc(dg[t + ic]);
            V v;
            if constexpr (MODE == BAH_FP64) v = cscale(d, w);
            else v = cdiv1(cmk<V>(w, 0), d);
            g[q] = in[q] ? v : czero<V>();
        }
        // vertical: u1 nodes j, j + 1; u2 cells j - 1, j; p cells j - 1, j + 1
#pragma unroll
        for (int q = 0; q < kQ + (TYPE == 2 ? 2 : 1); ++q) kz[q] = az[row(j0 + q - (TYPE == 0 ? 0 : 1)) + ic];
    }
    // acc + sum of k x_neighbour at row q; c: the point in shared memory (W, E and the rows
    // above and below the thread's own are read there)
    __device__ __forceinline__ V neighbours(int q, const V* c, V acc) const {
        auto add = [&](C k, const V& v) {
            const R kr = ldr(k);
            acc.x = fma(kr, v.x, acc.x);
            acc.y = fma(kr, v.y, acc.y);
        };
        c += q * kP;
        add(kw[q], c[-1]);
        add(ke[q], c[1]);
        add(kz[q], q > 0 ? x[q > 0 ? q - 1 : 0] : c[-kP]);
        add(kz[q + (TYPE == 2 ? 2 : 1)], q < kQ - 1 ? x[q < kQ - 1 ? q + 1 : 0] : c[kP]);
        return acc;
    }
};

template <class V> __device__ __forceinline__ void clear_border(V* xs) {
    for (int e = threadIdx.x; e < 2 * kP + 2 * kH; e += kThreads) {
        const int o = e < kP ? e : (e < 2 * kP ? (kH + 1) * kP + e - kP
                                               : (e < 2 * kP + kH ? (e - 2 * kP + 1) * kP : (e - 2 * kP - kH + 1) * kP + kW + 1));
        xs[o] = czero<V>();
    }
}

// coarse points of a down region: (I0 .. I0 + 29) x (J0 .. J0 + 13) need fine residuals
// 2 I0 - 1 .. 2 I0 + 60 and 2 J0 - 1 .. 2 J0 + 28
constexpr int kCw = kW / 2 - 2, kCh = kH / 2 - 2;

template <int MODE, int TYPE>
__device__ __forceinline__ void fine_down(const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC>& f,
                                          const typename Prec<MODE>::V* __restrict__ b, typename Prec<MODE>::R w,
                                          typename Prec<MODE>::V* __restrict__ bc, int intergrid,
                                          typename Prec<MODE>::V* __restrict__ x1, const typename Prec<MODE>::CC* d1, double w1c,
                                          typename Prec<MODE>::V* xs) {
    using V = typename Prec<MODE>::V;
    using R = typename Prec<MODE>::R;
    const int n1 = f.n1, n2 = f.n2, n1c = n1 / 2, n2c = n2 / 2;
    const int nbx = (n1c + kCw - 1) / kCw;
    const int I0 = (int)(blockIdx.x % nbx) * kCw, J0 = (int)(blockIdx.x / nbx) * kCh;
    const int ox = 2 * I0 - 2, oy = 2 * J0 - 2;
    V* rs = xs + (kH + 2) * kP;                         // kH x kW residuals
    const int col = threadIdx.x % kW, row0 = threadIdx.x / kW * kQ;
    Points<MODE, TYPE> p;
    p.load(f, b, ox + col, oy + row0, w);
    clear_border(xs);
    V* own = xs + (row0 + 1) * kP + col + 1;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        p.x[q] = cmul(p.g[q], p.b[q]);
        own[q * kP] = p.x[q];
    }
    __syncthreads();
    const R w1 = R(1) - w;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const V r = p.neighbours(q, own, cscale(p.b[q], w1));
        rs[(row0 + q) * kW + col] = p.in[q] ? r : czero<V>();
    }
    __syncthreads();
    constexpr bool nodx = TYPE == 0, nodz = TYPE == 1;
    for (int e = threadIdx.x; e < kCw * kCh; e += kThreads) {
        const int I = I0 + e % kCw, J = J0 + e / kCw;
        if (I >= n1c || J >= n2c) continue;
        V acc = czero<V>();
        if (valid_pt(TYPE, I, J)) {
            const int bx = rbase(nodx, intergrid, I), bz = rbase(nodz, intergrid, J);
            const V* r = rs + (bz - oy) * kW + (bx - ox);
            R wx[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) wx[u] = rw_axis_t<R>(nodx, intergrid, n1, I, bx + u);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const R wz = rw_axis_t<R>(nodz, intergrid, n2, J, bz + v);
                V t = czero<V>();
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const V rv = r[v * kW + u];
                    t.x = fma(wx[u], rv.x, t.x);
                    t.y = fma(wx[u], rv.y, t.y);
                }
                acc.x = fma(wz, t.x, acc.x);
                acc.y = fma(wz, t.y, acc.y);
            }
        }
        bc[(size_t)J * n1c + I] = acc;
        if (x1) x1[(size_t)J * n1c + I] = valid_pt(TYPE, I, J) ? first_sweep<MODE>(d1, J * n1c + I, acc, w1c) : czero<V>();
    }
}

// The correction at the thread's four rows: horizontal interpolation on the coarse rows they
// use (three if the first row is odd, which it is exactly when NS is odd; else four), then
// vertical.  Nodal axes: coarse rows outside 1 .. nc - 1 are the zero boundary; cell-centred
// axes: the nearest row in the grid.
template <class V, class R, int TYPE, bool ODD>
__device__ __forceinline__ void correction(const V* __restrict__ e, int n1, int n2, int i, int j0, V (&x)[kQ]) {
    const int n1c = n1 / 2, n2c = n2 / 2, jb = ODD ? (j0 - 1) >> 1 : (j0 >> 1) - 1;
    int cx[2];
    R wx[2];
    pw_pair<R>(TYPE == 0, n1, min(max(i, 0), n1 - 1), cx, wx);
    V h[4];
#pragma unroll
    for (int v = 0; v < (ODD ? 3 : 4); ++v) {
        const int jc = jb + v, t = min(max(jc, 0), n2c - 1) * n1c;
        const V a = e[t + cx[0]], c = e[t + cx[1]];
        h[v] = cmk<V>(fma(wx[0], a.x, wx[1] * c.x), fma(wx[0], a.y, wx[1] * c.y));
        if (TYPE == 1 && (jc < 1 || jc > n2c - 1)) h[v] = czero<V>();
    }
    auto add = [&](V& a, R k, const V& v) {
        a.x = fma(k, v.x, a.x);
        a.y = fma(k, v.y, a.y);
    };
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        // fine row j0 + q: its coarse row h[m]; an odd row's second one is h[m + 1], an even row's h[m - 1]
        const bool odd = ODD == (q % 2 == 0);
        const int m = ODD ? (q + 1) / 2 : 1 + q / 2;
        if (TYPE == 1) {
            add(x[q], odd ? R(0.5) : R(1), h[m]);
            if (odd) add(x[q], R(0.5), h[m + 1 < 4 ? m + 1 : 3]);
        } else {
            add(x[q], R(0.75), h[m]);
            add(x[q], R(0.25), h[odd ? (m + 1 < 4 ? m + 1 : 3) : (m > 0 ? m - 1 : 0)]);
        }
    }
}

template <int MODE, int TYPE, int NS, bool FROMB>
__device__ __forceinline__ void fine_up(const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC>& f,
                                        const typename Prec<MODE>::V* __restrict__ b, typename Prec<MODE>::R w,
                                        const typename Prec<MODE>::V* __restrict__ e,
                                        const typename Prec<MODE>::V* __restrict__ xin,
                                        typename Prec<MODE>::V* __restrict__ xo, typename Prec<MODE>::V* xs) {
    using V = typename Prec<MODE>::V;
    using R = typename Prec<MODE>::R;
    const int n1 = f.n1, n2 = f.n2;
    constexpr int ow = kW - 2 * NS, oh = kH - 2 * NS;
    static_assert(oh % 2 == 0, "the parity of a thread's first row is that of NS");
    const int nbx = (n1 + ow - 1) / ow;
    const int ox = (int)(blockIdx.x % nbx) * ow - NS, oy = (int)(blockIdx.x / nbx) * oh - NS;
    const int col = threadIdx.x % kW, row0 = threadIdx.x / kW * kQ;
    const int i = ox + col;
    Points<MODE, TYPE> p;
    p.load(f, b, i, oy + row0, w);
    clear_border(xs);
    clear_border(xs + (kH + 2) * kP);
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        if (FROMB) p.x[q] = cmul(p.g[q], p.b[q]);
        else p.x[q] = p.in[q] ? xin[(size_t)(oy + row0 + q) * n1 + i] : czero<V>();
    }
    correction<V, R, TYPE, NS % 2 == 1>(e, n1, n2, i, oy + row0, p.x);
    V* own = xs + (row0 + 1) * kP + col + 1;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        if (!p.in[q]) p.x[q] = czero<V>();
        own[q * kP] = p.x[q];
    }
    __syncthreads();
    const R w1 = R(1) - w;
#pragma unroll
    for (int it = 0; it < NS; ++it) {
        V nx[kQ];
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const V t = p.neighbours(q, own, p.b[q]);
            V v = cscale(p.x[q], w1);
            cfma(v, p.g[q], t);
            nx[q] = v;
        }
        own = it & 1 ? own - (kH + 2) * kP : own + (kH + 2) * kP;
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            p.x[q] = nx[q];
            if (it + 1 < NS) own[q * kP] = nx[q];
        }
        if (it + 1 < NS) __syncthreads();
    }
    if (col < NS || col >= kW - NS || i >= n1) return;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const int row = row0 + q, j = oy + row;
        if (row >= NS && row < kH - NS && j < n2) xo[(size_t)j * n1 + i] = p.x[q];
    }
}

}  // namespace

// b_c = R (b - A x), x = w D^{-1} b, and (fs) the coarse level's first sweep
template <int MODE>
__global__ void __launch_bounds__(kThreads, kMinCtas<MODE>)
    k_fine_down(LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC> s,
                Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC> f, typename Prec<MODE>::R w,
                PtrSet<typename Prec<MODE>::V> cb, int intergrid,
                FirstSweep<typename Prec<MODE>::V, typename Prec<MODE>::CC> fs) {
    pdl_prologue();
    using V = typename Prec<MODE>::V;
    const int rr = blockIdx.z;
    if (s.active && !s.active[rr]) return;
    const auto& B = s.blk[blockIdx.y];
    extern __shared__ __align__(128) unsigned char fine_raw[];
    V* xs = reinterpret_cast<V*>(fine_raw);             // (kH + 2) x kP, then kH x kW
    const V* b = B.b + rr * B.sb;
    V* bc = pick(cb, (int)blockIdx.y) + rr * cb.s;
    const int y = blockIdx.y;
    V* x1 = y == 0 ? fs.x[0] : (y == 1 ? fs.x[1] : fs.x[2]);
    const auto* d1 = y == 0 ? fs.d[0] : (y == 1 ? fs.d[1] : fs.d[2]);
    if (x1) x1 += rr * fs.sx;
    if (B.type == 0) fine_down<MODE, 0>(f, b, w, bc, intergrid, x1, d1, fs.w, xs);
    else if (B.type == 1) fine_down<MODE, 1>(f, b, w, bc, intergrid, x1, d1, fs.w, xs);
    else fine_down<MODE, 2>(f, b, w, bc, intergrid, x1, d1, fs.w, xs);
}

// x_out = NS Jacobi sweeps from x + P e_c; x is w D^{-1} b (FROMB: the state after
// k_fine_down) or read from xin.  The halo is NS points.
template <int MODE, int NS, bool FROMB>
__global__ void __launch_bounds__(kThreads, kMinCtas<MODE>)
    k_fine_up(LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC> s,
              Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC> f, typename Prec<MODE>::R w,
              PtrSet<const typename Prec<MODE>::V> ce) {
    pdl_prologue();
    using V = typename Prec<MODE>::V;
    const int rr = blockIdx.z;
    if (s.active && !s.active[rr]) return;
    const auto& B = s.blk[blockIdx.y];
    extern __shared__ __align__(128) unsigned char fine_raw[];
    V* xs = reinterpret_cast<V*>(fine_raw);             // two buffers of (kH + 2) x kP
    const V* b = B.b + rr * B.sb;
    const V* e = pick(ce, (int)blockIdx.y) + rr * ce.s;
    const V* xin = B.xin + rr * B.sxi;
    V* xo = B.xout + rr * B.sxo;
    if (B.type == 0) fine_up<MODE, 0, NS, FROMB>(f, b, w, e, xin, xo, xs);
    else if (B.type == 1) fine_up<MODE, 1, NS, FROMB>(f, b, w, e, xin, xo, xs);
    else fine_up<MODE, 2, NS, FROMB>(f, b, w, e, xin, xo, xs);
}

template <int MODE> static constexpr size_t fine_smem() {
    return 2 * (size_t)(kH + 2) * kP * sizeof(typename Prec<MODE>::V);
}

template <int MODE>
void launch_fine_down(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& s,
                      const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC>& f5, double w,
                      typename Prec<MODE>::V* const* coarse_b, int intergrid, size_t coarse_stride,
                      const FirstSweep<typename Prec<MODE>::V, typename Prec<MODE>::CC>& fs, cudaStream_t st) {
    PtrSet<typename Prec<MODE>::V> cb;
    for (int z = 0; z < 3; ++z) cb.p[z] = z < s.nb ? coarse_b[z] : nullptr;
    cb.s = coarse_stride;
    const int n1c = s.n1 / 2, n2c = s.n2 / 2;
    const dim3 g(((n1c + kCw - 1) / kCw) * ((n2c + kCh - 1) / kCh), s.nb, s.nrhs);
    launch_pdl(k_fine_down<MODE>, g, dim3(kThreads), fine_smem<MODE>(), st, s, f5, (typename Prec<MODE>::R)w, cb, intergrid, fs);
}
template <int MODE>
void launch_fine_up(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& s,
                    const Fine5<typename Prec<MODE>::C, typename Prec<MODE>::CC>& f5, double w, int sweeps, bool from_b,
                    const typename Prec<MODE>::V* const* coarse_x, size_t coarse_stride, cudaStream_t st) {
    PtrSet<const typename Prec<MODE>::V> ce;
    for (int z = 0; z < 3; ++z) ce.p[z] = z < s.nb ? coarse_x[z] : nullptr;
    ce.s = coarse_stride;
    const int ow = kW - 2 * sweeps, oh = kH - 2 * sweeps;
    const dim3 g(((s.n1 + ow - 1) / ow) * ((s.n2 + oh - 1) / oh), s.nb, s.nrhs);
    const auto r = (typename Prec<MODE>::R)w;
    const size_t sm = fine_smem<MODE>();
#define BAH_UP(N)                                                                                    \
    case N:                                                                                          \
        if (from_b) launch_pdl(k_fine_up<MODE, N, true>, g, dim3(kThreads), sm, st, s, f5, r, ce);   \
        else launch_pdl(k_fine_up<MODE, N, false>, g, dim3(kThreads), sm, st, s, f5, r, ce);         \
        break;
    switch (sweeps) { BAH_UP(1) BAH_UP(2) BAH_UP(3) }
#undef BAH_UP
}

// y = 1 / x
__global__ void k_inverse_diag(const double2* __restrict__ x, double2* __restrict__ y, size_t n) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e < n) y[e] = cdiv(make_double2(1.0, 0.0), x[e]);
}
void launch_inverse_diag(const double2* x, double2* y, size_t n, cudaStream_t st) {
    k_inverse_diag<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, y, n);
}

int fine_prepare() {
    const struct { const void* f; size_t b; } fns[] = {
#define BAH_FN(M)                                                                                                   \
    {(const void*)k_fine_down<M>, fine_smem<M>()},         {(const void*)k_fine_up<M, 1, true>, fine_smem<M>()},    \
        {(const void*)k_fine_up<M, 2, true>, fine_smem<M>()},  {(const void*)k_fine_up<M, 3, true>, fine_smem<M>()},  \
        {(const void*)k_fine_up<M, 1, false>, fine_smem<M>()}, {(const void*)k_fine_up<M, 2, false>, fine_smem<M>()}, \
        {(const void*)k_fine_up<M, 3, false>, fine_smem<M>()}
        BAH_FN(BAH_FP64), BAH_FN(BAH_MIXED)};
#undef BAH_FN
    for (const auto& q : fns) BAH_CUDA_TRY(cudaFuncSetAttribute(q.f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)q.b));
    return BAH_OK;
}

#define INST(M)                                                                                                     \
    template void launch_fine_down<M>(const LvlSet<Prec<M>::V, Prec<M>::CC>&, const Fine5<Prec<M>::C, Prec<M>::CC>&, \
                                      double, Prec<M>::V* const*, int, size_t,                                        \
                                      const FirstSweep<Prec<M>::V, Prec<M>::CC>&, cudaStream_t);                      \
    template void launch_fine_up<M>(const LvlSet<Prec<M>::V, Prec<M>::CC>&, const Fine5<Prec<M>::C, Prec<M>::CC>&,   \
                                    double, int, bool, const Prec<M>::V* const*, size_t, cudaStream_t);
INST(BAH_FP64)
INST(BAH_MIXED)

}  // namespace bah
