// Kernels of the adjoint gradient of a receiver misfit
// J = 1/2 sum_s ||Q x_s - d_s||^2 with respect to lambda, mu, rho:
//   * adjoint source Q^H (Q x_s - d_s) and the per-source misfit;
//   * element-wise conjugation (H^H = conj(H) for the complex-symmetric H of
//     Eq. 2.6, so H^H y = b is solved as H conj(y) = conj(b));
//   * the pointwise gradient  dJ/dm_k = -Re sum_s y_s^H (dH/dm_k) x_s, written
//     out per cell from the structure of H: lambda enters through
//     -C = -diag(1/(lambda+mu)), mu through A_e(mu) (own-direction
//     derivatives at the cell, cross derivatives at the 4 nodes around it
//     with weight 1/4) and through C, rho through the face mass
//     A_f(rho (1 - i gamma/omega)) of the faces around the cell.
#include "bah_internal.cuh"

namespace bah {

__global__ void k_conj(double2* v, size_t n) {
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        v[e].y = -v[e].y;
}
void launch_conj(double2* v, size_t n, cudaStream_t st) {
    k_conj<<<RED_CTAS * 2, 256, 0, st>>>(v, n);
}

// adj_s = Q^H (Q x_s - d_s) (adj zeroed beforehand): adj[s][rec[q]] gathers
// x[s][rec[q]] - d[s][q] of every q naming that entry, so a receiver listed
// twice is counted twice, as in J.  Every q marks its entry of the zeroed adj;
// where no entry is marked twice, each thread writes its receivers.  Otherwise
// one thread adds them in the order of q, so the result does not depend on
// scheduling (always doing that, a chain of dependent global reads and writes,
// took 300 us for 1024 receivers).  misfit[s] = 1/2 sum_q |x - d|^2 (one CTA
// per source, fixed-order block reduction).
__global__ void __launch_bounds__(256) k_misfit(const double2* __restrict__ x, const double2* __restrict__ d,
                                                const int* __restrict__ rec, int nrec, size_t vlen, double2* adj,
                                                double* misfit) {
    const int s = blockIdx.x;
    const double2* xs = x + (size_t)s * vlen;
    const double2* ds = d + (size_t)s * nrec;
    double2* as = adj + (size_t)s * vlen;
    double acc = 0.0;
    int twice = 0;
    for (int q = threadIdx.x; q < nrec; q += blockDim.x) {
        const double2 r = csub(xs[rec[q]], ds[q]);
        acc += r.x * r.x + r.y * r.y;
        twice |= atomicExch(reinterpret_cast<int*>(as + rec[q]), 1);
    }
    if (!__syncthreads_or(twice)) {
        for (int q = threadIdx.x; q < nrec; q += blockDim.x) as[rec[q]] = csub(xs[rec[q]], ds[q]);
    } else {
        for (int q = threadIdx.x; q < nrec; q += blockDim.x) as[rec[q]] = make_double2(0.0, 0.0);
        __syncthreads();
        if (threadIdx.x == 0)
            for (int q = 0; q < nrec; ++q) {
                const int i = rec[q];
                as[i] = cadd(as[i], csub(xs[i], ds[q]));
            }
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) misfit[s] = 0.5 * sh[0];
}
void launch_misfit(const double2* x, const double2* d, const int* rec, int nrec, int nrhs, size_t vlen, double2* adj,
                   double* misfit, cudaStream_t st) {
    k_misfit<<<nrhs, 256, 0, st>>>(x, d, rec, nrec, vlen, adj, misfit);
}

struct GradArgs {
    int n1, n2;
    double ih1, ih2, omega;
    const double* cinv;     // 1/(lambda+mu)
    const double* gamma;
    size_t vlen;
    int nrhs;
};

// One grid point per thread: over the nrhs (forward, adjoint) pairs it sums the
// terms that live at its cell (C, the own-direction derivatives), at the node
// and at the two faces on its lower sides.  A cell's gradient then needs the
// node and face sums of its upper neighbours, which pass through shared memory:
// each CTA's last column and row of points only feed their neighbours
// (31 x 15 of 32 x 16 points write a cell).
// Bound: the FP64 pipe, 34 FP64 operations per point and pair; forming every
// node and face term at each cell that uses it takes 130.  Measured with 32
// sources of 1024 x 512: 4.61 -> 1.23 ms.
constexpr int kGx = 32, kGy = 16;
__global__ void __launch_bounds__(kGx * kGy) k_gradient(GradArgs a, const double2* __restrict__ X,
                                                        const double2* __restrict__ Y, double* g_lambda, double* g_mu,
                                                        double* g_rho) {
    const int n1 = a.n1, n2 = a.n2;
    const size_t np = (size_t)n1 * n2;
    const int i = blockIdx.x * (kGx - 1) + threadIdx.x, j = blockIdx.y * (kGy - 1) + threadIdx.y;
    const bool in = i < n1 && j < n2;
    const size_t t = in ? (size_t)j * n1 + i : 0;
    // which of the neighbouring unknowns exist (u1: i >= 1, u2: j >= 1)
    const bool f1 = in && i >= 1, f1e = in && i + 1 < n1, f1s = f1 && j >= 1;
    const bool f2 = in && j >= 1, f2n = in && j + 1 < n2, f2w = f2 && i >= 1;
    const bool node = in && i >= 1 && j >= 1;
    const double2 z = make_double2(0.0, 0.0);
    double cp = 0.0, own1 = 0.0, own2 = 0.0, na = 0.0, nb = 0.0, fr = 0.0, fi = 0.0, gr = 0.0, gi = 0.0;
    auto rdot = [](double& acc, double2 y, double2 x) {                  // acc += Re(conj(y) x)
        acc = fma(y.x, x.x, acc);
        acc = fma(y.y, x.y, acc);
    };
    auto idot = [](double& acc, double2 y, double2 x) {                  // acc += Im(conj(y) x)
        acc = fma(y.x, x.y, acc);
        acc = fma(-y.y, x.x, acc);
    };
    if (in)
#pragma unroll 2
        for (int s = 0; s < a.nrhs; ++s) {
            const double2* x1 = X + (size_t)s * a.vlen + t;
            const double2* y1 = Y + (size_t)s * a.vlen + t;
            const double2 *x2 = x1 + np, *y2 = y1 + np;
            const double2 xc = f1 ? x1[0] : z, yc = f1 ? y1[0] : z;
            const double2 xe = f1e ? x1[1] : z, ye = f1e ? y1[1] : z;
            const double2 xs = f1s ? x1[-n1] : z, ys = f1s ? y1[-n1] : z;
            const double2 uc = f2 ? x2[0] : z, vc = f2 ? y2[0] : z;
            const double2 un = f2n ? x2[n1] : z, vn = f2n ? y2[n1] : z;
            const double2 uw = f2w ? x2[-1] : z, vw = f2w ? y2[-1] : z;
            rdot(cp, y1[2 * np], x1[2 * np]);
            rdot(own1, csub(ye, yc), csub(xe, xc));
            rdot(own2, csub(vn, vc), csub(un, uc));
            if (node) {                                                  // d2 u1 and d1 u2 at the lower node
                rdot(na, csub(yc, ys), csub(xc, xs));
                rdot(nb, csub(vc, vw), csub(uc, uw));
            }
            rdot(fr, yc, xc);
            idot(fi, yc, xc);
            rdot(gr, vc, uc);
            idot(gi, vc, uc);
        }
    const double q1 = a.ih1 * a.ih1, q2 = a.ih2 * a.ih2;
    __shared__ double sn[kGy][kGx], s1r[kGy][kGx], s1i[kGy][kGx], s2r[kGy][kGx], s2i[kGy][kGx];
    const int tx = threadIdx.x, ty = threadIdx.y;
    sn[ty][tx] = fma(q2, na, q1 * nb);
    s1r[ty][tx] = fr; s1i[ty][tx] = fi;
    s2r[ty][tx] = gr; s2i[ty][tx] = gi;
    __syncthreads();
    if (!in || tx == kGx - 1 || ty == kGy - 1) return;
    // own-direction derivatives at the cell, cross derivatives at its four nodes with weight 1/4
    const double ci = a.cinv[t], cterm = cp * ci * ci;
    const double gm = cterm + fma(q1, own1, q2 * own2) +
                      0.25 * ((sn[ty][tx] + sn[ty][tx + 1]) + (sn[ty + 1][tx] + sn[ty + 1][tx + 1]));
    // rho: -Re[ y^H (-omega^2 1/2 (1 - i gamma/omega)) x ] over the cell's four faces
    const double re = (s1r[ty][tx] + s1r[ty][tx + 1]) + (s2r[ty][tx] + s2r[ty + 1][tx]);
    const double im = (s1i[ty][tx] + s1i[ty][tx + 1]) + (s2i[ty][tx] + s2i[ty + 1][tx]);
    g_lambda[t] += -cterm;
    g_mu[t] += -gm;
    g_rho[t] += 0.5 * a.omega * a.omega * (re + a.gamma[t] / a.omega * im);
}
void launch_gradient(int n1, int n2, double h1, double h2, double omega, const double* cinv, const double* gamma,
                     size_t vlen, int nrhs, const double2* X, const double2* Y, double* gl, double* gm, double* gr,
                     cudaStream_t st) {
    GradArgs a{n1, n2, 1.0 / h1, 1.0 / h2, omega, cinv, gamma, vlen, nrhs};
    const dim3 g((n1 + kGx - 2) / (kGx - 1), (n2 + kGy - 2) / (kGy - 1));
    k_gradient<<<g, dim3(kGx, kGy), 0, st>>>(a, X, Y, gl, gm, gr);
}

}  // namespace bah
