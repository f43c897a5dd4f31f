// Jacobi sweeps and residuals on a Galerkin level (levels >= 1), batched over
// blocks (blockIdx.y) and right-hand sides.
//
// One thread per grid point holds the point's stencil in registers (up to 25
// complex entries, bf16 unpacked to FP32 in mixed mode) and applies it to the
// right-hand sides of its CTA one after another; the iterate's rows around the
// CTA's points are copied to shared memory (cp.async, one right-hand side ahead),
// rows outside the grid as zeros.  So every load of a launch is in flight at
// once (a loop over the taps waits for memory at each of them: 15 us for a 32 x 32
// level in FP64), a batch reads the stencils once instead of once per source, and
// a tap is one shared-memory load and four multiply-adds.  Radii are compile-time;
// entries that would reach across the left or right edge are zeroed once.
//
// The sweep is written x_out = (1 - w) x + w D^{-1} (b - (A - D) x).
// Bound: FP64 the FP64 pipe (4 operations per tap), mixed instruction issue.
// Measured per sweep: two displacement blocks of 512 x 256 with 8 sources 83 -> 30
// us; one 256 x 256 pressure block, one source, 7.8 -> 5.6 us, FP64 16.6 -> 8.5 us
// (32 x 32 FP64 15 -> 7.7 us).  20 steps: 512 x 512 6.50 -> 5.96 ms, 32 sources of
// 1024 x 512 214 -> 193 ms.
#include "bah_internal.cuh"

#include <algorithm>

namespace bah {

namespace {

// points per CTA: in FP64 a warp instruction takes 16 clocks of the SM's pipe, so small
// CTAs spread a small level over more SMs
template <int MODE> constexpr int kPts = MODE == BAH_FP64 ? 64 : 128;

__device__ __forceinline__ double2 ld_entry(const double2* p) {        // issued here, wherever it is used
    double2 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned ld_entry(const __nv_bfloat162* p) {
    unsigned v;
    asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 entry(double2 v) { return v; }
__device__ __forceinline__ float2 entry(unsigned v) { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }

template <int BYTES> __device__ __forceinline__ void copy_or_zero(void* dst, const void* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES), "r"(in ? BYTES : 0)
                 : "memory");
}

template <int MODE, int RX, int RZ, bool RES>
__device__ __forceinline__ void apply(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& s,
                                      const LvlBlk<typename Prec<MODE>::V, typename Prec<MODE>::CC>& B,
                                      typename Prec<MODE>::R w, int per, typename Prec<MODE>::V* xs) {
    using V = typename Prec<MODE>::V;
    using R = typename Prec<MODE>::R;
    constexpr int T = kPts<MODE>, WX = 2 * RX + 1, WZ = 2 * RZ + 1, NT = WX * WZ, P = T + 2 * RX;
    const int n1 = s.n1, n2 = s.n2, np = n1 * n2;
    const int t0 = blockIdx.x * T, t = t0 + threadIdx.x, tc = min(t, np - 1);
    const int i = tc % n1, j = tc / n1;
    const int r0 = blockIdx.z * per, r1 = min(s.nrhs, r0 + per);
    // the rows of right-hand side r: row dz holds points t0 + dz n1 - RX .. t0 + dz n1 + T - 1 + RX
    auto stage = [&](int r, V* buf) {
        const V* x = B.xin + r * B.sxi;
        for (int e = threadIdx.x; e < WZ * P; e += T) {
            const int g = t0 + (e / P - RZ) * n1 + e % P - RX;
            const bool in = g >= 0 && g < np;
            copy_or_zero<sizeof(V)>(buf + e, x + (in ? g : 0), in);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto next = [&](int r) {                                    // first active right-hand side from r on
        while (r < r1 && s.active && !s.active[r]) ++r;
        return r;
    };
    int r = next(r0);
    if (r >= r1) return;
    stage(r, xs);
    decltype(ld_entry(B.S)) raw[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) raw[u] = ld_entry(B.S + (size_t)u * np + tc);
    V b = B.b[r * B.sb + tc];
    V g;
    if constexpr (MODE == BAH_FP64) g = cscale(B.idg[tc], w);
    V c[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        const int dx = u % WX - RX;
        c[u] = entry(raw[u]);
        if (dx != 0 && (i + dx < 0 || i + dx >= n1)) c[u] = czero<V>();
    }
    if constexpr (MODE != BAH_FP64) g = cdiv1(cmk<V>(w, 0), c[NT / 2]);
    const bool valid = valid_pt(B.type, i, j);
    int buf = 0;
    while (r < r1) {
        const int rn = next(r + 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();                                        // r's rows arrived; the other buffer is free
        V bn = b;
        if (rn < r1) {
            stage(rn, xs + (buf ^ 1) * WZ * P);
            bn = B.b[rn * B.sb + tc];
        }
        const V* x = xs + buf * WZ * P + threadIdx.x + RX;
        V acc = czero<V>();
#pragma unroll
        for (int u = 0; u < NT; ++u)
            if (RES || u != NT / 2) cfma(acc, c[u], x[(u / WX) * P + u % WX - RX]);
        V v = csub(b, acc);
        if (!RES) {
            const V d = v;
            v = cscale(x[RZ * P], R(1) - w);
            cfma(v, g, d);
        }
        if (t < np) B.xout[r * B.sxo + t] = valid ? v : czero<V>();
        r = rn;
        b = bn;
        buf ^= 1;
    }
}

}  // namespace

template <int MODE, bool RES>
__global__ void __launch_bounds__(kPts<MODE>) k_galerkin_level(LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC> s,
                                                               typename Prec<MODE>::R w, int per) {
    pdl_prologue();
    using V = typename Prec<MODE>::V;
    __shared__ __align__(16) unsigned char raw[2 * 5 * (kPts<MODE> + 4) * sizeof(V)];
    V* xs = reinterpret_cast<V*>(raw);
    const auto& B = s.blk[blockIdx.y];
    if (B.rx == 2 && B.rz == 2) apply<MODE, 2, 2, RES>(s, B, w, per, xs);
    else if (B.rx == 2) apply<MODE, 2, 1, RES>(s, B, w, per, xs);
    else if (B.rz == 2) apply<MODE, 1, 2, RES>(s, B, w, per, xs);
    else apply<MODE, 1, 1, RES>(s, B, w, per, xs);
}

template <int MODE>
void launch_galerkin_level(const LvlSet<typename Prec<MODE>::V, typename Prec<MODE>::CC>& s, double w, bool residual,
                           cudaStream_t st) {
    const int np = s.n1 * s.n2, tiles = (np + kPts<MODE> - 1) / kPts<MODE>;
    // right-hand sides per CTA: as many as leave about four CTAs per SM
    const int per = std::max(1, std::min(s.nrhs, tiles * s.nb * s.nrhs / 608));
    const dim3 g(tiles, s.nb, (s.nrhs + per - 1) / per), b(kPts<MODE>);
    const auto r = (typename Prec<MODE>::R)w;
    if (residual) launch_pdl(k_galerkin_level<MODE, true>, g, b, 0, st, s, r, per);
    else launch_pdl(k_galerkin_level<MODE, false>, g, b, 0, st, s, r, per);
}
template void launch_galerkin_level<BAH_FP64>(const LvlSet<double2, double2>&, double, bool, cudaStream_t);
template void launch_galerkin_level<BAH_MIXED>(const LvlSet<float2, __nv_bfloat162>&, double, bool, cudaStream_t);

}  // namespace bah
