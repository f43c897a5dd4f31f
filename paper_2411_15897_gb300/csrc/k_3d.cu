// Three-dimensional grids: the mixed elastic operator (Eq. 2.6), the
// distributor and back-substitution of the block-acoustic preconditioner
// (Eq. 3.3 - 3.5), and the multigrid of its four acoustic blocks (Sec. 2.2;
// Galerkin coarsening, Eq. 4.3, with the mixed intergrid of Eq. 4.4, the
// transfer the paper takes for its 3-D experiments, Sec. 4.5).
//
// Point (i, j, k) of an n1 x n2 x n3 grid sits at (k*n2 + j)*n1 + i.  Every
// block lives on the padded index space of its level: block type a < 3
// (u_{a+1}, nodal along x_{a+1}) has unknowns where that coordinate is >= 1,
// type 3 (p) at every point; the other points hold structural zeros, which
// every kernel writes as zero and none reads as an unknown.
//
// One thread per point, per column of four planes (level 0) or per pair of points
// (prolongation); a neighbour outside the grid is loaded at a clamped index and does
// not count.  The kernels of the solve's step begin with pdl_prologue() and are
// launched with programmatic dependent launch; the level kernels run the three
// displacement blocks of a level in one launch.
#include "bah_internal.cuh"
#include "op_rows.cuh"

#include <type_traits>

namespace bah {

// pointers of up to three blocks of one level, one per blockIdx.y of a launch;
// pick() selects without indexing the parameter array at a run-time index
// (which would copy it to the stack)
template <class T> struct Set3 { T* p[3]; };
template <class T> __device__ __forceinline__ T* pick(const Set3<T>& s, int y) {
    return y == 0 ? s.p[0] : (y == 1 ? s.p[1] : s.p[2]);
}

__host__ __device__ __forceinline__ bool valid3(int type, const int* c) { return type >= 3 || c[type] >= 1; }

__device__ __forceinline__ void coords3(int p, int n1, int n2, int* c) {
    c[0] = p % n1;
    const int t = p / n1;
    c[1] = t % n2;
    c[2] = t / n2;
}

// stencil entry s -> offset: 7-point (0 centre, 1 + 2a at -e_a, 2 + 2a at +e_a)
// or 27-point ((dz+1)*9 + (dy+1)*3 + (dx+1))
template <int NS> __host__ __device__ __forceinline__ void soff(int s, int* o) {
    if (NS == 7) {
        o[0] = o[1] = o[2] = 0;
        if (s > 0) o[(s - 1) >> 1] = ((s - 1) & 1) ? 1 : -1;
    } else {
        o[0] = s % 3 - 1;
        o[1] = (s / 3) % 3 - 1;
        o[2] = s / 9 - 1;
    }
}
template <int NS> __host__ __device__ constexpr int scentre() { return NS == 7 ? 0 : 13; }

// ---------------------------------------------------------------------------
// medium: 1/(lambda+mu), omega^2 rho~ (rho~ = rho (1 - i gamma/omega)) and
// the edge means of mu.  mue[e] belongs to the pair of axes other than e; at a
// point whose coordinates along that pair are (a, b) it is the mean of mu over
// the four cells around the edge at nodes (a, b), zero on boundary edges
// (where the tangential derivative is dropped with the zero normal
// displacement), the same averaging as the 2-D operator's nodes.
// ---------------------------------------------------------------------------
__global__ void k_prep3_cells(int n1, int n2, int n3, double omega, const double* __restrict__ lam,
                              const double* __restrict__ mu, const double* __restrict__ rho,
                              const double* __restrict__ gam, double* cinv, double2* mrt, double* mue0, double* mue1,
                              double* mue2) {
    const int np = n1 * n2 * n3;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    int c[3];
    coords3(p, n1, n2, c);
    const int st[3] = {1, n1, n1 * n2};
    cinv[p] = 1.0 / (lam[p] + mu[p]);
    mrt[p] = make_double2(omega * omega * rho[p], -omega * rho[p] * gam[p]);
    double* mue[3] = {mue0, mue1, mue2};
    for (int e = 0; e < 3; ++e) {
        const int a = e == 0 ? 1 : 0, b = e == 2 ? 1 : 2;
        double v = 0.0;
        if (c[a] >= 1 && c[b] >= 1)
            v = 0.25 * (mu[p] + mu[p - st[a]] + mu[p - st[b]] + mu[p - st[a] - st[b]]);
        mue[e][p] = v;
    }
}

// diagonals of A_a (unshifted) and the FP64 7-point fine stencils of the four
// shifted blocks A_{a,s} (Eq. 2.6 with the shift of Eq. 2.8) and H_{p,s}
// (Eq. 3.4: B B^T diag((lambda+2mu)/(lambda+mu)) - omega^2 diag(rho~/(lambda+mu)),
// shifted by i alpha omega^2 rho/(lambda+mu))
__global__ void k_prep3_blocks(Op3 op, double alpha, double omega, const double* __restrict__ rho,
                               const double* __restrict__ mu, const double* mue0, const double* mue1,
                               const double* mue2, double2* dg0, double2* dg1, double2* dg2,
                               double2* S0, double2* S1, double2* S2, double2* S3) {
    const int n1 = op.n[0], n2 = op.n[1], n3 = op.n[2];
    const int np = n1 * n2 * n3;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    int c[3];
    coords3(p, n1, n2, c);
    const int st[3] = {1, n1, n1 * n2};
    const double* mue[3] = {mue0, mue1, mue2};
    double2* dg[3] = {dg0, dg1, dg2};
    double2* S[4] = {S0, S1, S2, S3};
    const double aw2 = alpha * omega * omega;
    for (int a = 0; a < 3; ++a) {
        double2 e[7];
        for (int s = 0; s < 7; ++s) e[s] = make_double2(0.0, 0.0);
        double2 d = make_double2(0.0, 0.0);
        if (c[a] >= 1) {
            const int pm = p - st[a];
            double dr = op.ih2[a] * (mu[pm] + mu[p]);
            if (c[a] >= 2) e[1 + 2 * a].x = -op.ih2[a] * mu[pm];
            if (c[a] + 1 <= op.n[a] - 1) e[2 + 2 * a].x = -op.ih2[a] * mu[p];
            for (int b = 0; b < 3; ++b) {
                if (b == a) continue;
                const double* me = mue[3 - a - b];
                const double lo = c[b] >= 1 ? me[p] : 0.0;
                const double hi = c[b] + 1 <= op.n[b] - 1 ? me[p + st[b]] : 0.0;
                dr += op.ih2[b] * (lo + hi);
                e[1 + 2 * b].x = -op.ih2[b] * lo;
                e[2 + 2 * b].x = -op.ih2[b] * hi;
            }
            const double2 m = make_double2(0.5 * (op.mrt[pm].x + op.mrt[p].x), 0.5 * (op.mrt[pm].y + op.mrt[p].y));
            d = make_double2(dr - m.x, -m.y);
            e[0] = make_double2(d.x, d.y + aw2 * 0.5 * (rho[pm] + rho[p]));
        }
        dg[a][p] = d;
        for (int s = 0; s < 7; ++s) S[a][(size_t)s * np + p] = e[s];
    }
    // H_p,s
    {
        double2 e[7];
        for (int s = 0; s < 7; ++s) e[s] = make_double2(0.0, 0.0);
        const double wp = 1.0 + mu[p] * op.cinv[p];
        double cen = 0.0;
        for (int a = 0; a < 3; ++a) {
            if (c[a] >= 1) {
                const int q = p - st[a];
                cen += op.ih2[a] * wp;
                e[1 + 2 * a].x = -op.ih2[a] * (1.0 + mu[q] * op.cinv[q]);
            }
            if (c[a] + 1 <= op.n[a] - 1) {
                const int q = p + st[a];
                cen += op.ih2[a] * wp;
                e[2 + 2 * a].x = -op.ih2[a] * (1.0 + mu[q] * op.cinv[q]);
            }
        }
        e[0] = make_double2(cen - op.mrt[p].x * op.cinv[p], -op.mrt[p].y * op.cinv[p] + aw2 * rho[p] * op.cinv[p]);
        for (int s = 0; s < 7; ++s) S[3][(size_t)s * np + p] = e[s];
    }
}

void launch_prep3(const Op3& op, double omega, double alpha, const double* lam, const double* mu, const double* rho,
                  const double* gam, double* cinv, double2* mrt, double* const* mue, double2* const* dg,
                  double2* const* S, cudaStream_t st) {
    const int np = op.n[0] * op.n[1] * op.n[2];
    const int nb = (np + 255) / 256;
    k_prep3_cells<<<nb, 256, 0, st>>>(op.n[0], op.n[1], op.n[2], omega, lam, mu, rho, gam, cinv, mrt, mue[0], mue[1],
                                      mue[2]);
    k_prep3_blocks<<<nb, 256, 0, st>>>(op, alpha, omega, rho, mu, mue[0], mue[1], mue[2], dg[0], dg[1], dg[2], S[0], S[1], S[2], S[3]);
}

__global__ void k_scale_real(const double* __restrict__ src, double f, double* __restrict__ dst, size_t n) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e < n) dst[e] = f * src[e];
}
void launch_scale_real(const double* src, double f, double* dst, size_t n, cudaStream_t st) {
    k_scale_real<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(src, f, dst, n);
}

// ---------------------------------------------------------------------------
// y = H x (Eq. 2.6), y = b - H x with b, or y = H^H x = conj(H) x (H is complex
// symmetric; only the mass diagonals are complex).  Right-hand side r of the
// launch is blockIdx.y, at element strides sx, sy, sb.
// ---------------------------------------------------------------------------
template <class Vin>
__global__ void __launch_bounds__(256) k_apply3(Op3 op, const Vin* __restrict__ x, double2* __restrict__ y,
                                                const double2* __restrict__ b, int conj, size_t sx, size_t sy,
                                                size_t sb) {
    pdl_prologue();
    const int n1 = op.n[0], n2 = op.n[1];
    const int np = n1 * n2 * op.n[2];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    x += blockIdx.y * sx;
    y += blockIdx.y * sy;
    if (b) b += blockIdx.y * sb;
    int c[3];
    coords3(p, n1, n2, c);
    const int st[3] = {1, n1, n1 * n2};
    auto ld = [&](int comp, int q) { return cconv<double2>(x[(size_t)comp * np + q]); };
    // 74 FP64 operations per cell, all fused, from coefficients divided by h^2 at
    // setup; the FP64 pipe (2 per clock and SM) bounds the kernel.  With FP32 input at
    // 128^3: 643 us when every load was converted by the FP64 pipe and every
    // coefficient formed in the kernel, 308 us now
    auto add = [](double2& acc, double k, const double2& v) {
        acc.x = fma(k, v.x, acc.x);
        acc.y = fma(k, v.y, acc.y);
    };
    auto sub = [](double2& acc, double k, const double2& v) {         // negated inside the fma: no instruction of its own
        acc.x = fma(-k, v.x, acc.x);
        acc.y = fma(-k, v.y, acc.y);
    };
    // every neighbour is loaded (at a clamped index) so that the loads issue together, and
    // replaced by 0 where there is no unknown: what stands in a boundary-normal entry does not count
    const double2 pc = ld(3, p), zero = make_double2(0.0, 0.0);
    double2 out[4];
    double2 div = cscale(pc, -op.cinv[p]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool lo = c[a] >= 1, hi = c[a] + 1 <= op.n[a] - 1;
        const int pm = lo ? p - st[a] : p, pe = hi ? p + st[a] : p;
        const double2 uc = lo ? ld(a, p) : zero, ue = hi ? ld(a, pe) : zero;
        add(div, op.ih[a], csub(uc, ue));
        const double2 uw = ld(a, pm);
        const double kw = op.cmu[a][pm], ke = op.cmu[a][p];
        double2 acc = cscale(c[a] >= 2 ? uw : zero, kw);
        add(acc, ke, ue);
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
            if (bb == a) continue;
            const double* me = op.cme[3 - a - bb][bb];               // zero on boundary edges
            const bool bl = c[bb] >= 1, bh = c[bb] + 1 <= op.n[bb] - 1;
            const int qm = bl ? p - st[bb] : p, qe = bh ? p + st[bb] : p;
            const double km = me[p], kp = me[qe];
            const double2 um = ld(a, qm), up = ld(a, qe);
            add(acc, km, bl ? um : zero);
            add(acc, kp, bh ? up : zero);
        }
        sub(acc, op.ih[a], csub(pc, ld(3, pm)));
        out[a] = lo ? diag_minus(op.dg[a][p], uc, conj, acc) : zero;
    }
    out[3] = div;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool v = k == 3 || c[k] >= 1;
        double2 o = out[k];
        if (b && v) o = csub(b[(size_t)k * np + p], o);
        y[(size_t)k * np + p] = v ? o : make_double2(0.0, 0.0);
    }
}

template <class Vin>
void launch_apply3(const Op3& op, const Vin* x, double2* y, const double2* b, int conj, int nrhs, size_t sx, size_t sy,
                   size_t sb, cudaStream_t st) {
    const int np = op.n[0] * op.n[1] * op.n[2];
    if (nrhs < 1) return;
    launch_pdl(k_apply3<Vin>, dim3((np + 255) / 256, nrhs), dim3(256), 0, st, op, x, y, b, conj, sx, sy, sb);
}
template void launch_apply3<double2>(const Op3&, const double2*, double2*, const double2*, int, int, size_t, size_t,
                                     size_t, cudaStream_t);
template void launch_apply3<float2>(const Op3&, const float2*, double2*, const double2*, int, int, size_t, size_t,
                                    size_t, cudaStream_t);

// zero the boundary-normal entries of nvec padded vectors
__global__ void k_sanitize3(double2* v, int n1, int n2, int n3, int nvec) {
    const int np = n1 * n2 * n3;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    int c[3];
    coords3(p, n1, n2, c);
    for (int r = 0; r < nvec; ++r)
        for (int a = 0; a < 3; ++a)
            if (c[a] == 0) v[((size_t)r * 4 + a) * np + p] = make_double2(0.0, 0.0);
}
void launch_sanitize3(double2* v, int n1, int n2, int n3, int nvec, cudaStream_t st) {
    const int np = n1 * n2 * n3;
    k_sanitize3<<<(np + 255) / 256, 256, 0, st>>>(v, n1, n2, n3, nvec);
}

// ---------------------------------------------------------------------------
// distributor (Eq. 3.3, second row): t_p = B r_u - A_p r_p with
// A_p = B B^T diag(mu) - omega^2 diag(rho~) (Eq. 3.2); FP64 arithmetic,
// result in the cycle's vector type
// ---------------------------------------------------------------------------
template <class V>
__global__ void __launch_bounds__(256) k_distrib3(Op3 op, const double2* __restrict__ r, V* __restrict__ tp) {
    pdl_prologue();
    const int n1 = op.n[0], n2 = op.n[1];
    const int np = n1 * n2 * op.n[2];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    int c[3];
    coords3(p, n1, n2, c);
    const int st[3] = {1, n1, n1 * n2};
    const double2* rp = r + (size_t)3 * np;
    const double2 r0 = rp[p];
    const double2 m = op.mrt[p];
    double2 acc = make_double2(fma(m.x, r0.x, -(m.y * r0.y)), fma(m.x, r0.y, m.y * r0.x));   // + omega^2 rho~ r_p
    double k0 = 0.0;                             // mu_p times the number of neighbours along each axis / h^2
    auto add = [&](double k, const double2& v) {
        acc.x = fma(k, v.x, acc.x);
        acc.y = fma(k, v.y, acc.y);
    };
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double2* ra = r + (size_t)a * np;
        const bool lo = c[a] >= 1, hi = c[a] + 1 <= op.n[a] - 1;
        const int qm = lo ? p - st[a] : p, qe = hi ? p + st[a] : p;
        const double2 gl = ra[p], gh = ra[qe], rl = rp[qm], rh = rp[qe];
        const double kl = op.cmu[a][qm], kh = op.cmu[a][qe], kp = op.cmu[a][p];
        const double2 zero = make_double2(0.0, 0.0);
        add(kl, lo ? rl : zero);
        add(kh, hi ? rh : zero);
        add(op.ih[a], csub(lo ? gl : zero, hi ? gh : zero));
        k0 += lo && hi ? 2.0 * kp : (lo || hi ? kp : 0.0);
    }
    add(-k0, r0);
    tp[p] = cconv<V>(acc);
}

// back-substitution (Eq. 3.5): s_a = r_a - (B^T e_p)_a for the three u blocks
template <class V>
__global__ void __launch_bounds__(256) k_urhs3(Op3 op, const double2* __restrict__ r, const V* __restrict__ ep,
                                               V* __restrict__ s0, V* __restrict__ s1, V* __restrict__ s2) {
    pdl_prologue();
    const int n1 = op.n[0], n2 = op.n[1];
    const int np = n1 * n2 * op.n[2];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    int c[3];
    coords3(p, n1, n2, c);
    const int st[3] = {1, n1, n1 * n2};
    V* s[3] = {s0, s1, s2};
    const double2 e0 = cconv<double2>(ep[p]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool lo = c[a] >= 1;
        const double2 em = cconv<double2>(ep[lo ? p - st[a] : p]), v = r[(size_t)a * np + p];
        const double2 o = make_double2(fma(-op.ih[a], e0.x - em.x, v.x), fma(-op.ih[a], e0.y - em.y, v.y));
        s[a][p] = cconv<V>(lo ? o : make_double2(0.0, 0.0));
    }
}

template <class V>
void launch_distrib3(const Op3& op, const double2* r, V* tp, cudaStream_t st) {
    const int np = op.n[0] * op.n[1] * op.n[2];
    launch_pdl(k_distrib3<V>, dim3((np + 255) / 256), dim3(256), 0, st, op, r, tp);
}
template <class V>
void launch_urhs3(const Op3& op, const double2* r, const V* ep, V* const* su, cudaStream_t st) {
    const int np = op.n[0] * op.n[1] * op.n[2];
    launch_pdl(k_urhs3<V>, dim3((np + 255) / 256), dim3(256), 0, st, op, r, ep, su[0], su[1], su[2]);
}
template void launch_distrib3<double2>(const Op3&, const double2*, double2*, cudaStream_t);
template void launch_distrib3<float2>(const Op3&, const double2*, float2*, cudaStream_t);
template void launch_urhs3<double2>(const Op3&, const double2*, const double2*, double2* const*, cudaStream_t);
template void launch_urhs3<float2>(const Op3&, const double2*, const float2*, float2* const*, cudaStream_t);

// ---------------------------------------------------------------------------
// multigrid level kernels.  Stencils are stored entry-major: entry s of
// point p at S[s * points + p].
// ---------------------------------------------------------------------------
// A launch runs up to three blocks of one level: blockIdx.y = y runs block type
// type0 + y on the y-th pointers.  Sweeps are written
// x_out = (1 - w) x + w D^{-1} (b - (A - D) x) with D^{-1} formed at setup (a complex
// reciprocal is some 40 instructions, in FP64 mode 10 of them on a pipe of two
// operations per clock and SM).
template <class T>
static Set3<T> set3(T* const* v, int nq) {
    Set3<T> s;
    for (int y = 0; y < 3; ++y) s.p[y] = y < nq ? v[y] : nullptr;
    return s;
}
// loads issued here, wherever their results are used; stencil entries (constant) through the non-coherent path
__device__ __forceinline__ double2 ld_now3(const double2* p) {
    double2 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ldv_now3(const double2* p) {
    double2 v;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ldv_now3(const float2* p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned ld_now3(const __nv_bfloat162* p) {
    unsigned v;
    asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 entry3(double2 v) { return v; }
__device__ __forceinline__ float2 entry3(unsigned v) { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }
// base[i] through a 32-bit byte offset: a vector of one block is at most 4 GB (bah_create refuses
// more than 2^28 cells in FP64 and 2^29 in mixed mode)
template <class T> __device__ __forceinline__ T at3(const T* base, unsigned i) {
    return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + (size_t)(i * (unsigned)sizeof(T)));
}

// first sweep from zero: x = w D^{-1} b (any level; below the first, k_restrict3 writes it)
template <class V>
__global__ void __launch_bounds__(128) k_zero3(int type0, int n1, int n2, int n3, Set3<const V> idgset, Set3<const V> bset,
                                               Set3<V> xoset, typename VecTraits<V>::R w) {
    pdl_prologue();
    const int y = blockIdx.y, np = n1 * n2 * n3, p = blockIdx.x * 128 + threadIdx.x;
    if (p >= np) return;
    int c[3];
    coords3(p, n1, n2, c);
    pick(xoset, y)[p] = valid3(type0 + y, c) ? cmul(cscale(pick(idgset, y)[p], w), pick(bset, y)[p]) : czero<V>();
}

// Sweep or residual on a 27-point level.  The small levels of a W-cycle, visited most
// often, are bound by the chain of memory latencies: every load is issued before the
// first multiply-add, and CTAs are small, so that 16^3 points spread over 64 SMs
// (16^3 points, mixed mode: 9.4 us with 256-thread CTAs and the loads left to the
// compiler, 3.7 us).  Entries that would couple to a point outside the grid are zero
// (the Galerkin product clamps at the ends), so such a neighbour's load is redirected
// to the point itself and needs no test.
constexpr int kT27 = 64;
template <class V, class SC, bool RES>
__global__ void __launch_bounds__(kT27) k_level27(int type0, int n1, int n2, int n3, Set3<const SC> Sset, Set3<const V> idgset,
                                                  Set3<const V> bset, Set3<const V> xiset, Set3<V> xoset,
                                                  typename VecTraits<V>::R w) {
    pdl_prologue();
    const int y = blockIdx.y, type = type0 + y;
    const int np = n1 * n2 * n3;
    const int p = blockIdx.x * kT27 + threadIdx.x;
    if (p >= np) return;
    const SC* S = pick(Sset, y) + p;
    const V* xin = pick(xiset, y);
    int c[3];
    coords3(p, n1, n2, c);
    if (!valid3(type, c)) { pick(xoset, y)[p] = czero<V>(); return; }
    const int dx[3] = {c[0] >= 1 ? -1 : 0, 0, c[0] + 1 < n1 ? 1 : 0};
    const int dy[3] = {c[1] >= 1 ? -n1 : 0, 0, c[1] + 1 < n2 ? n1 : 0};
    const int dz[3] = {c[2] >= 1 ? -n1 * n2 : 0, 0, c[2] + 1 < n3 ? n1 * n2 : 0};
    decltype(ld_now3(S)) raw[27];
    V xv[27];
#pragma unroll
    for (int s = 0; s < 27; ++s) {
        if (RES || s != 13) raw[s] = ld_now3(S);
        S += np;
        xv[s] = ldv_now3(reinterpret_cast<const V*>(reinterpret_cast<const char*>(xin) +
                                                    (size_t)((unsigned)(p + dx[s % 3] + dy[s / 3 % 3] + dz[s / 9]) * (unsigned)sizeof(V))));
    }
    const V b = pick(bset, y)[p];
    V g = b;
    if (!RES) g = pick(idgset, y)[p];
    V acc = czero<V>();
#pragma unroll
    for (int s = 0; s < 27; ++s)
        if (RES || s != 13) cfma(acc, entry3(raw[s]), xv[s]);
    V v = csub(b, acc);
    if (!RES) {
        const V d = v;
        v = cscale(xv[13], 1 - w);
        cfma(v, cscale(g, w), d);
    }
    pick(xoset, y)[p] = v;
}

// Level 0, the 7-point operators from per-point coefficients (mu at cells and edges
// over h^2, (lambda + 2 mu) / (lambda + mu) over h^2): 6 to 10 bytes per point in
// mixed mode where seven stored complex entries take 28, with the same values.
// FROMB: the input iterate is the first sweep from zero, x = w D^{-1} b, formed here.
// A thread takes kZ3 points of one column: the block type is a compile-time constant
// of its loop, the column's tests and clamped offsets are formed once, and values and
// coefficients along axis 2 pass from plane to plane in registers.  With a thread per
// point of the flattened grid the kernel was bound by its 280 instructions per point
// (three blocks of 128^3, mixed mode: 64 us a sweep, 100 us with FROMB; now 40 and 48,
// against 79 us from the stored 7-point entries).
constexpr int kZ3 = 4;
template <class V, class C, class SC, bool RES, bool FROMB, int TYPE>
__device__ __forceinline__ void fine3_column(const Fine3<C, SC, V>& f, const V* b, const V* xin, V* xout,
                                             typename VecTraits<V>::R w, int cx, int cy, int z0) {
    using R = typename VecTraits<V>::R;
    const int n1 = f.n[0], n2 = f.n[1], n3 = f.n[2];
    const unsigned pl = (unsigned)(n1 * n2);
    unsigned p = (unsigned)((z0 * n2 + cy) * n1 + cx);
    const int nz = min(kZ3, n3 - z0);
    V out[kZ3];
    if ((TYPE == 0 && cx == 0) || (TYPE == 1 && cy == 0)) {
        for (int k = 0; k < nz; ++k) xout[p + k * pl] = czero<V>();
        return;
    }
    const V* __restrict__ idg = f.idg[TYPE];
    auto X = [&](unsigned q) {
        if constexpr (FROMB) return cmul(cscale(at3(idg, q), w), at3(b, q));
        else return at3(xin, q);
    };
    auto add = [](V& acc, R k, const V& v) {
        acc.x = fma(k, v.x, acc.x);
        acc.y = fma(k, v.y, acc.y);
    };
    const int cc[2] = {cx, cy};
    const unsigned st[2] = {1u, (unsigned)n1};
    bool lo[2], hi[2];
    unsigned ql[2], qh[2];                       // offsets of the neighbours in the plane, zero where there is none
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        lo[a] = cc[a] >= (a == TYPE ? 2 : 1);
        hi[a] = cc[a] + 1 < f.n[a];
        ql[a] = lo[a] ? 0u - st[a] : 0u;
        qh[a] = hi[a] ? st[a] : 0u;
    }
    constexpr int e2 = TYPE < 2 ? 1 - TYPE : 0;
    const C* __restrict__ kz = TYPE == 3 ? f.wv[2] : (TYPE == 2 ? f.cmu[2] : f.cme[e2][2]);
    // neighbours below and at the point along axis 2 and the couplings to the lower one and (TYPE 3) of the point
    V xm = z0 >= (TYPE == 2 ? 2 : 1) ? X(p - pl) : czero<V>();
    V xc = TYPE == 2 && z0 == 0 ? czero<V>() : X(p);
    R kl = TYPE < 2 ? ldr(at3(kz, p)) : (z0 >= 1 ? ldr(at3(kz, p - pl)) : R(0));
    R kc = TYPE == 3 ? ldr(at3(kz, p)) : R(0);
#pragma unroll
    for (int k = 0; k < kZ3; ++k) {
        if (k >= nz) break;
        const int z = z0 + k;
        const bool up = z + 1 < n3;
        const unsigned pu = up ? p + pl : p;
        const V xu = up ? X(pu) : czero<V>();
        const R kh = TYPE == 2 ? ldr(at3(kz, p)) : (up ? ldr(at3(kz, pu)) : R(0));
        V acc = at3(b, p);
        add(acc, kl, xm);
        add(acc, kh, xu);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int e = TYPE == 3 || a == TYPE ? 0 : 3 - TYPE - a;
            const C* __restrict__ ka = TYPE == 3 ? f.wv[a] : (a == TYPE ? f.cmu[a] : f.cme[e][a]);
            const bool below = TYPE == 3 || a == TYPE;                   // the lower coupling is the lower point's coefficient
            const R vl = ldr(at3(ka, below ? p + ql[a] : p)), vh = ldr(at3(ka, a == TYPE ? p : p + qh[a]));
            add(acc, lo[a] ? vl : R(0), X(p + ql[a]));
            add(acc, hi[a] ? vh : R(0), X(p + qh[a]));
        }
        // acc = b - (A - D) x
        if constexpr (RES) {
            out[k] = csub(acc, cmul(ldc(at3(f.dg[TYPE], p)), xc));
        } else {
            out[k] = cscale(xc, 1 - w);
            cfma(out[k], cscale(at3(idg, p), w), acc);
        }
        if (TYPE == 2 && z == 0) out[k] = czero<V>();
        xm = xc;
        xc = xu;
        kl = TYPE == 3 ? kc : kh;
        kc = kh;
        p += pl;
    }
    // stored after the last load: the loads of all planes can be in flight together
    p = (unsigned)((z0 * n2 + cy) * n1 + cx);
#pragma unroll
    for (int k = 0; k < kZ3; ++k)
        if (k < nz) xout[p + k * pl] = out[k];
}
template <class V, class C, class SC, bool RES, bool FROMB>
__global__ void __launch_bounds__(256, sizeof(V) == 16 ? 3 : 5) k_fine3(int type0, int tx, Fine3<C, SC, V> f, Set3<const V> bset, Set3<const V> xiset,
                                               Set3<V> xoset, typename VecTraits<V>::R w) {
    pdl_prologue();
    const int y = blockIdx.y;
    const int ty = blockIdx.x / tx;
    const int cx = (blockIdx.x - ty * tx) * blockDim.x + threadIdx.x, cy = ty * blockDim.y + threadIdx.y;
    if (cx >= f.n[0] || cy >= f.n[1]) return;
    const V *b = pick(bset, y), *xin = pick(xiset, y);
    V* xout = pick(xoset, y);
    const int z0 = blockIdx.z * kZ3;
    switch (type0 + y) {
        case 0: return fine3_column<V, C, SC, RES, FROMB, 0>(f, b, xin, xout, w, cx, cy, z0);
        case 1: return fine3_column<V, C, SC, RES, FROMB, 1>(f, b, xin, xout, w, cx, cy, z0);
        case 2: return fine3_column<V, C, SC, RES, FROMB, 2>(f, b, xin, xout, w, cx, cy, z0);
        default: return fine3_column<V, C, SC, RES, FROMB, 3>(f, b, xin, xout, w, cx, cy, z0);
    }
}

template <class V>
void launch_zero3(int type0, int nq, const int* n, const V* const* idg, const V* const* b, V* const* xout, double w,
                  cudaStream_t st) {
    const int np = n[0] * n[1] * n[2];
    launch_pdl(k_zero3<V>, dim3((np + 127) / 128, nq), dim3(128), 0, st, type0, n[0], n[1], n[2], set3<const V>(idg, nq),
               set3<const V>(b, nq), set3<V>(xout, nq), (typename VecTraits<V>::R)w);
}
template <class V>
void launch_level27(int type0, int nq, const int* n, const void* const* S, const V* const* idg, const V* const* b,
                    const V* const* xin, V* const* xout, double w, bool res, cudaStream_t st) {
    using SC = typename std::conditional<std::is_same<V, double2>::value, double2, __nv_bfloat162>::type;
    const int np = n[0] * n[1] * n[2];
    const SC* s[3];
    for (int y = 0; y < nq; ++y) s[y] = (const SC*)S[y];
    auto fn = res ? k_level27<V, SC, true> : k_level27<V, SC, false>;
    launch_pdl(fn, dim3((np + kT27 - 1) / kT27, nq), dim3(kT27), 0, st, type0, n[0], n[1], n[2], set3<const SC>(s, nq),
               set3<const V>(idg, nq), set3<const V>(b, nq), set3<const V>(xin, nq), set3<V>(xout, nq),
               (typename VecTraits<V>::R)w);
}
template <class V, class C, class SC>
void launch_fine3(const Fine3<C, SC, V>& f, int type0, int nq, const V* const* b, const V* const* xin, V* const* xout, double w,
                  bool res, bool from_b, cudaStream_t st) {
    auto fn = res ? k_fine3<V, C, SC, true, false> : k_fine3<V, C, SC, false, false>;
    if constexpr (std::is_same<V, float2>::value)
        if (from_b) fn = k_fine3<V, C, SC, false, true>;
    // 32 x 8 columns, or 16 x 16 where that leaves fewer threads without a column
    auto up = [](int n, int b) { return (n + b - 1) / b; };
    const int bx = up(f.n[0], 16) * up(f.n[1], 16) < up(f.n[0], 32) * up(f.n[1], 8) ? 16 : 32, by = 256 / bx;
    const int tx = up(f.n[0], bx);
    launch_pdl(fn, dim3(tx * up(f.n[1], by), nq, up(f.n[2], kZ3)), dim3(bx, by), 0, st, type0, tx, f, set3<const V>(b, nq),
               set3<const V>(xin, nq), set3<V>(xout, nq), (typename VecTraits<V>::R)w);
}
#define INST3(V, C, SC)                                                                                                   \
    template void launch_zero3<V>(int, int, const int*, const V* const*, const V* const*, V* const*, double,              \
                                  cudaStream_t);                                                                          \
    template void launch_level27<V>(int, int, const int*, const void* const*, const V* const*, const V* const*,           \
                                    const V* const*, V* const*, double, bool, cudaStream_t);                              \
    template void launch_fine3<V, C, SC>(const Fine3<C, SC, V>&, int, int, const V* const*, const V* const*, V* const*,   \
                                         double, bool, bool, cudaStream_t);
INST3(double2, double, double2)
INST3(float2, __nv_bfloat16, __nv_bfloat162)
#undef INST3

// 1 / x of the stored diagonals, in FP64, rounded to the cycle's type
template <class V, class SC>
__global__ void k_inverse3(const SC* __restrict__ x, V* __restrict__ y, size_t n) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const auto d = ldc(x[e]);
    y[e] = cconv<V>(cdiv(make_double2(1.0, 0.0), make_double2(d.x, d.y)));
}
void launch_inverse3(const void* x, void* y, size_t n, int mode, cudaStream_t st) {
    const unsigned g = (unsigned)((n + 255) / 256);
    if (mode == BAH_MIXED) k_inverse3<float2, __nv_bfloat162><<<g, 256, 0, st>>>((const __nv_bfloat162*)x, (float2*)y, n);
    else k_inverse3<double2, double2><<<g, 256, 0, st>>>((const double2*)x, (double2*)y, n);
}

// (lambda + 2 mu) / (lambda + mu) at cells
__global__ void k_wp3(const double* __restrict__ mu, const double* __restrict__ cinv, double* __restrict__ w, size_t n) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e < n) w[e] = 1.0 + mu[e] * cinv[e];
}
void launch_wp3(const double* mu, const double* cinv, double* w, size_t n, cudaStream_t st) {
    k_wp3<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(mu, cinv, w, n);
}

// 1-D transfer weights.  Restriction (Eq. 4.1 / 4.4, mixed intergrid): along
// the block's nodal axis 1/4 [1 2 1] around fine face 2K; along a cell-centred
// axis 1/2 [1 1] over fine cells 2J, 2J+1.  Prolongation: linear interpolation
// along the nodal axis (missing coarse faces are the zero boundary) and
// bilinear cell-centred interpolation with constant extrapolation at the ends.
__host__ __device__ __forceinline__ int rlist3(bool nodal, int J, int* f, double* w) {
    if (nodal) {
        f[0] = 2 * J - 1; w[0] = 0.25;
        f[1] = 2 * J;     w[1] = 0.5;
        f[2] = 2 * J + 1; w[2] = 0.25;
        return 3;
    }
    f[0] = 2 * J;     w[0] = 0.5;
    f[1] = 2 * J + 1; w[1] = 0.5;
    return 2;
}
__host__ __device__ __forceinline__ int plist3(bool nodal, int m, int nc, int* K, double* w) {
    if (nodal) {
        if ((m & 1) == 0) {
            K[0] = m >> 1; w[0] = 1.0;
            return (K[0] >= 1 && K[0] <= nc - 1) ? 1 : 0;
        }
        int cnt = 0;
        if (((m - 1) >> 1) >= 1) { K[cnt] = (m - 1) >> 1; w[cnt++] = 0.5; }
        if (((m + 1) >> 1) <= nc - 1) { K[cnt] = (m + 1) >> 1; w[cnt++] = 0.5; }
        return cnt;
    }
    const int J = m >> 1;
    int Jn = (m & 1) ? J + 1 : J - 1;
    if (Jn < 0 || Jn > nc - 1) Jn = J;
    K[0] = J;  w[0] = 0.75;
    K[1] = Jn; w[1] = 0.25;
    return 2;
}

// The transfers run with the block type as a compile-time constant, so that every tap
// is an unconditional load: 12 of a coarse point (8 on the pressure block), 12 of a
// pair of fine points along axis 0.  With run-time lists of up to 27 and 8 predicated
// taps, three blocks of 128^3 took 18.8 us down and 58 us up, now 12 and 27; the fine
// array's bandwidth would allow 7 and 15.
constexpr int kTr3 = 128;
// b_c = R r on the coarse grid (fine grid f, coarse f / 2); with x, also the coarse
// level's first sweep from zero, x = w D^{-1} b_c
template <class V, int TYPE>
__device__ __forceinline__ V restrict3_point(const V* r, int f1, int f2, const int* J) {
    using R = typename VecTraits<V>::R;
    V acc = czero<V>();
#pragma unroll
    for (int z = 0; z < (TYPE == 2 ? 3 : 2); ++z)
#pragma unroll
        for (int y = 0; y < (TYPE == 1 ? 3 : 2); ++y)
#pragma unroll
            for (int x = 0; x < (TYPE == 0 ? 3 : 2); ++x) {
                // nodal axis: 1/4, 1/2, 1/4 at 2J - 1, 2J, 2J + 1; the others 1/2 at 2J, 2J + 1
                const int tap = TYPE == 0 ? x : (TYPE == 1 ? y : z);
                const R ww = TYPE == 3 ? R(0.125) : (tap == 1 ? R(0.125) : R(0.0625));
                const int fx = 2 * J[0] + x - (TYPE == 0), fy = 2 * J[1] + y - (TYPE == 1), fz = 2 * J[2] + z - (TYPE == 2);
                const V v = at3(r, (unsigned)((fz * f2 + fy) * f1 + fx));
                acc.x = fma(ww, v.x, acc.x);
                acc.y = fma(ww, v.y, acc.y);
            }
    return acc;
}
template <class V>
__global__ void __launch_bounds__(kTr3) k_restrict3(int type0, int f1, int f2, int f3, Set3<const V> rset, Set3<V> bcset,
                                                    Set3<const V> idgset, Set3<V> xset, typename VecTraits<V>::R w) {
    pdl_prologue();
    const int type = type0 + (int)blockIdx.y;
    const V* r = pick(rset, (int)blockIdx.y);
    V* x = pick(xset, (int)blockIdx.y);
    const int c1 = f1 / 2, c2 = f2 / 2, c3 = f3 / 2;
    const int p = blockIdx.x * kTr3 + threadIdx.x;
    if (p >= c1 * c2 * c3) return;
    int J[3];
    coords3(p, c1, c2, J);
    V acc = czero<V>(), x1 = czero<V>();
    if (valid3(type, J)) {
        V g = acc;
        if (x) g = pick(idgset, (int)blockIdx.y)[p];
        switch (type) {
            case 0: acc = restrict3_point<V, 0>(r, f1, f2, J); break;
            case 1: acc = restrict3_point<V, 1>(r, f1, f2, J); break;
            case 2: acc = restrict3_point<V, 2>(r, f1, f2, J); break;
            default: acc = restrict3_point<V, 3>(r, f1, f2, J);
        }
        x1 = cmul(cscale(g, w), acc);
    }
    pick(bcset, (int)blockIdx.y)[p] = acc;
    if (x) x[p] = x1;
}

// taps of fine index m along one axis: two coarse indices, an unused one with weight 0 at an in-range index
template <class R, bool NODAL>
__device__ __forceinline__ void paxis3(int m, int nc, int* K, R* w) {
    const int J = m >> 1, odd = m & 1;
    if (NODAL) {                                 // even: J; odd: the mean of J and J + 1 (coarse index 0 is no unknown)
        K[0] = J;                  w[0] = J >= 1 ? (odd ? R(0.5) : R(1)) : R(0);
        K[1] = min(J + odd, nc - 1); w[1] = odd && J + 1 < nc ? R(0.5) : R(0);
    } else {                                     // 3/4 of the own cell, 1/4 of the nearer neighbour (constant beyond the ends)
        K[0] = J;                                        w[0] = R(0.75);
        K[1] = odd ? min(J + 1, nc - 1) : max(J - 1, 0); w[1] = R(0.25);
    }
}
// x += P e_c at the fine points 2J, 2J + 1 of a row
template <class V, int TYPE>
__device__ __forceinline__ void prolong3_pair(const V* ec, V* x, int f1, int f2, int c1, int c2, int c3, int J, int fy, int fz) {
    using R = typename VecTraits<V>::R;
    if ((TYPE == 1 && fy == 0) || (TYPE == 2 && fz == 0)) return;
    int ky[2], kz[2];
    R wy[2], wz[2];
    paxis3<R, TYPE == 1>(fy, c2, ky, wy);
    paxis3<R, TYPE == 2>(fz, c3, kz, wz);
    constexpr int NX = TYPE == 0 ? 2 : 3;
    const int kx[3] = {TYPE == 0 ? J : max(J - 1, 0), TYPE == 0 ? min(J + 1, c1 - 1) : J, min(J + 1, c1 - 1)};
    V t[NX];
#pragma unroll
    for (int k = 0; k < NX; ++k) t[k] = czero<V>();
    V* xr = x + (fz * f2 + fy) * f1 + 2 * J;
    V x0 = xr[0], x1 = xr[1];
#pragma unroll
    for (int z = 0; z < 2; ++z)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const R ww = wz[z] * wy[y];
            const unsigned row = (unsigned)((kz[z] * c2 + ky[y]) * c1);
#pragma unroll
            for (int k = 0; k < NX; ++k) {
                const V v = at3(ec, row + kx[k]);
                t[k].x = fma(ww, v.x, t[k].x);
                t[k].y = fma(ww, v.y, t[k].y);
            }
        }
    if constexpr (TYPE == 0) {
        const R we = J >= 1 ? R(1) : R(0), w0 = J >= 1 ? R(0.5) : R(0), w1 = J + 1 < c1 ? R(0.5) : R(0);
        x0 = cmk<V>(fma(we, t[0].x, x0.x), fma(we, t[0].y, x0.y));
        x1 = cmk<V>(x1.x + fma(w0, t[0].x, w1 * t[1].x), x1.y + fma(w0, t[0].y, w1 * t[1].y));
    } else {
        x0 = cmk<V>(x0.x + fma(R(0.75), t[1].x, R(0.25) * t[0].x), x0.y + fma(R(0.75), t[1].y, R(0.25) * t[0].y));
        x1 = cmk<V>(x1.x + fma(R(0.75), t[1].x, R(0.25) * t[2].x), x1.y + fma(R(0.75), t[1].y, R(0.25) * t[2].y));
    }
    if (TYPE != 0 || J >= 1) xr[0] = x0;
    xr[1] = x1;
}
template <class V>
__global__ void __launch_bounds__(kTr3) k_prolong3(int type0, int f1, int f2, int f3, Set3<const V> ecset, Set3<V> xset) {
    pdl_prologue();
    const V* ec = pick(ecset, (int)blockIdx.y);
    V* x = pick(xset, (int)blockIdx.y);
    const int c1 = f1 / 2, c2 = f2 / 2, c3 = f3 / 2;
    const int p = blockIdx.x * kTr3 + threadIdx.x;
    if (p >= c1 * f2 * f3) return;
    int F[3];
    coords3(p, c1, f2, F);
    switch (type0 + (int)blockIdx.y) {
        case 0: return prolong3_pair<V, 0>(ec, x, f1, f2, c1, c2, c3, F[0], F[1], F[2]);
        case 1: return prolong3_pair<V, 1>(ec, x, f1, f2, c1, c2, c3, F[0], F[1], F[2]);
        case 2: return prolong3_pair<V, 2>(ec, x, f1, f2, c1, c2, c3, F[0], F[1], F[2]);
        default: return prolong3_pair<V, 3>(ec, x, f1, f2, c1, c2, c3, F[0], F[1], F[2]);
    }
}

template <class V>
void launch_restrict3(int type0, int nq, const int* nf, const V* const* r, V* const* bc, const V* const* idg, V* const* x,
                      double w, cudaStream_t st) {
    const int npc = (nf[0] / 2) * (nf[1] / 2) * (nf[2] / 2);
    launch_pdl(k_restrict3<V>, dim3((npc + kTr3 - 1) / kTr3, nq), dim3(kTr3), 0, st, type0, nf[0], nf[1], nf[2],
               set3<const V>(r, nq), set3<V>(bc, nq), set3<const V>(idg, nq), set3<V>(x, nq), (typename VecTraits<V>::R)w);
}
template <class V>
void launch_prolong3(int type0, int nq, const int* nf, const V* const* ec, V* const* x, cudaStream_t st) {
    const int pairs = (nf[0] / 2) * nf[1] * nf[2];
    launch_pdl(k_prolong3<V>, dim3((pairs + kTr3 - 1) / kTr3, nq), dim3(kTr3), 0, st, type0, nf[0], nf[1], nf[2],
               set3<const V>(ec, nq), set3<V>(x, nq));
}
template void launch_restrict3<double2>(int, int, const int*, const double2* const*, double2* const*, const double2* const*,
                                       double2* const*, double, cudaStream_t);
template void launch_restrict3<float2>(int, int, const int*, const float2* const*, float2* const*, const float2* const*,
                                       float2* const*, double, cudaStream_t);
template void launch_prolong3<double2>(int, int, const int*, const double2* const*, double2* const*, cudaStream_t);
template void launch_prolong3<float2>(int, int, const int*, const float2* const*, float2* const*, cudaStream_t);

// ---------------------------------------------------------------------------
// Galerkin coarse operator A_c = R A P (Eq. 4.3) in FP64, one thread per
// coarse point, from a 7- or 27-point fine stencil to a 27-point coarse one.
// With the mixed intergrid every coarse coupling stays within one point per
// axis; a coupling outside sets *err (it would mean a wrong transfer).
// ---------------------------------------------------------------------------
template <int NSF>
__global__ void k_galerkin3(int type, int f1, int f2, int f3, const double2* __restrict__ Sf, double2* __restrict__ Sc,
                            int* err) {
    const int nc[3] = {f1 / 2, f2 / 2, f3 / 2};
    const int nf[3] = {f1, f2, f3};
    const int npc = nc[0] * nc[1] * nc[2];
    const int npf = f1 * f2 * f3;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npc) return;
    int J[3];
    coords3(p, nc[0], nc[1], J);
    double2 acc[27];
    for (int s = 0; s < 27; ++s) acc[s] = make_double2(0.0, 0.0);
    if (valid3(type, J)) {
        int f[3][3], cnt[3];
        double wr[3][3];
        for (int a = 0; a < 3; ++a) cnt[a] = rlist3(a == type, J[a], f[a], wr[a]);
        for (int z = 0; z < cnt[2]; ++z)
            for (int y = 0; y < cnt[1]; ++y)
                for (int x = 0; x < cnt[0]; ++x) {
                    const int A[3] = {f[0][x], f[1][y], f[2][z]};
                    const double w0 = wr[0][x] * wr[1][y] * wr[2][z];
                    const size_t pa = ((size_t)A[2] * f2 + A[1]) * f1 + A[0];
                    for (int s = 0; s < NSF; ++s) {
                        int o[3];
                        soff<NSF>(s, o);
                        int B[3];
                        bool in = true;
                        for (int a = 0; a < 3; ++a) {
                            B[a] = A[a] + o[a];
                            if (B[a] < 0 || B[a] >= nf[a]) in = false;
                        }
                        if (!in) continue;
                        const double2 v = Sf[(size_t)s * npf + pa];
                        if (v.x == 0.0 && v.y == 0.0) continue;
                        int K[3][2], pc[3];
                        double wp[3][2];
                        for (int a = 0; a < 3; ++a) pc[a] = plist3(a == type, B[a], nc[a], K[a], wp[a]);
                        for (int kz = 0; kz < pc[2]; ++kz)
                            for (int ky = 0; ky < pc[1]; ++ky)
                                for (int kx = 0; kx < pc[0]; ++kx) {
                                    const int d0 = K[0][kx] - J[0], d1 = K[1][ky] - J[1], d2 = K[2][kz] - J[2];
                                    if (d0 < -1 || d0 > 1 || d1 < -1 || d1 > 1 || d2 < -1 || d2 > 1) {
                                        *err = 1;
                                        continue;
                                    }
                                    const double ww = w0 * wp[0][kx] * wp[1][ky] * wp[2][kz];
                                    double2& t = acc[(d2 + 1) * 9 + (d1 + 1) * 3 + (d0 + 1)];
                                    t.x += ww * v.x;
                                    t.y += ww * v.y;
                                }
                    }
                }
    }
    for (int s = 0; s < 27; ++s) Sc[(size_t)s * npc + p] = acc[s];
}

void launch_galerkin3(int type, const int* nf, int nsf, const double2* Sf, double2* Sc, int* err, cudaStream_t st) {
    const int npc = (nf[0] / 2) * (nf[1] / 2) * (nf[2] / 2);
    if (nsf == 7)
        k_galerkin3<7><<<(npc + 127) / 128, 128, 0, st>>>(type, nf[0], nf[1], nf[2], Sf, Sc, err);
    else
        k_galerkin3<27><<<(npc + 127) / 128, 128, 0, st>>>(type, nf[0], nf[1], nf[2], Sf, Sc, err);
}

// dense matrix of the coarsest 27-point stencil over all points (identity
// rows at structural zeros) and X = I, for the Gauss-Jordan inverse
__global__ void k_dense_assemble3(int type, const double2* __restrict__ S, int n1, int n2, int n3, double2* A,
                                  double2* X) {
    const int np = n1 * n2 * n3;
    const int r = blockIdx.y;
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= np || r >= np) return;
    int cr[3], cc[3];
    coords3(r, n1, n2, cr);
    coords3(col, n1, n2, cc);
    double2 v = make_double2(0.0, 0.0);
    if (valid3(type, cr)) {
        const int o0 = cc[0] - cr[0], o1 = cc[1] - cr[1], o2 = cc[2] - cr[2];
        if (o0 >= -1 && o0 <= 1 && o1 >= -1 && o1 <= 1 && o2 >= -1 && o2 <= 1)
            v = S[(size_t)((o2 + 1) * 9 + (o1 + 1) * 3 + (o0 + 1)) * np + r];
    } else if (col == r) {
        v = make_double2(1.0, 0.0);
    }
    A[(size_t)r * np + col] = v;
    X[(size_t)r * np + col] = make_double2(col == r ? 1.0 : 0.0, 0.0);
}

int coarse_invert3(int type, const int* n, const double2* S, double2* inv, double2* work, int* flag, cudaStream_t st) {
    const int np = n[0] * n[1] * n[2];
    if (np > 65535) {
        set_error("coarsest 3-D level too large for the dense inverse");
        return BAH_ERR_ARG;
    }
    dim3 g((np + 127) / 128, np);
    k_dense_assemble3<<<g, 128, 0, st>>>(type, S, n[0], n[1], n[2], work, inv);
    return gauss_jordan(np, work, inv, work + (size_t)np * np, flag, st);
}

}  // namespace bah
