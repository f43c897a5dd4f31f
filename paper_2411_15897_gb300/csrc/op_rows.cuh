// The three rows of y = H x at one cell of a 2-D grid (Eq. 2.6), in FP64:
//   u1 row:  (diag A_1) u1 - sum of the four mu-weighted neighbours + (grad_h p)_1
//   u2 row:  the same along x_2
//   p row:   (B u - C p) = -div_h u - p / (lambda + mu)
// The entries of x are read through accessors U1(i, j), U2(i, j) (zero
// outside the unknowns of the component) and P(flat index), so every kernel
// that needs H x (the operator launches and the allocation-free residual)
// shares one definition of the stencil.  conj != 0 applies H^H = conj(H).
// Written as fused multiply-adds: 42 FP64 operations per cell, whose pipe (2 per
// clock and SM) bounds the operator (1024 x 1024: 93 -> 81 us).
#pragma once
#include "bah_internal.cuh"

namespace bah {

__device__ __forceinline__ void add_kv(double2& a, double k, const double2& v) {      // a += k v, k real
    a.x = fma(k, v.x, a.x);
    a.y = fma(k, v.y, a.y);
}
// d u - s for the complex diagonal d (conj(d) u - s): the largest product enters
// last, when the sum of the neighbours is complete (the smallest rounding)
__device__ __forceinline__ double2 diag_minus(const double2& d, const double2& u, int conj, const double2& s) {
    const double di = flip_sign(d.y, conj);
    return make_double2(fma(d.x, u.x, fma(-di, u.y, -s.x)), fma(d.x, u.y, fma(di, u.x, -s.y)));
}

template <class FU1, class FU2, class FP>
__device__ __forceinline__ void elastic_rows(const OpCoef& c, int i, int j, int t, int conj, FU1 U1, FU2 U2, FP P,
                                             double2& y1, double2& y2, double2& yp) {
    const int n1 = c.n1, n2 = c.n2;
    const double2 z = make_double2(0.0, 0.0);
    const double2 p = P(t);
    y1 = z;
    y2 = z;
    if (i >= 1) {
        double2 a = cscale(U1(i - 1, j), c.cx[t - 1]);
        add_kv(a, c.cx[t], U1(i + 1, j));
        add_kv(a, c.nz[t], U1(i, j - 1));
        add_kv(a, (j + 1 < n2) ? c.nz[t + n1] : 0.0, U1(i, j + 1));
        const double2 pw = P(t - 1);
        a.x = fma(-c.ihx, p.x - pw.x, a.x);
        a.y = fma(-c.ihx, p.y - pw.y, a.y);
        y1 = diag_minus(c.d1[t], U1(i, j), conj, a);
    }
    if (j >= 1) {
        double2 a = cscale(U2(i, j - 1), c.cz[t - n1]);
        add_kv(a, c.cz[t], U2(i, j + 1));
        add_kv(a, c.nx[t], U2(i - 1, j));
        add_kv(a, (i + 1 < n1) ? c.nx[t + 1] : 0.0, U2(i + 1, j));
        const double2 ps = P(t - n1);
        a.x = fma(-c.ihz, p.x - ps.x, a.x);
        a.y = fma(-c.ihz, p.y - ps.y, a.y);
        y2 = diag_minus(c.d2[t], U2(i, j), conj, a);
    }
    const double2 u1c = U1(i, j), u1e = U1(i + 1, j), u2c = U2(i, j), u2n = U2(i, j + 1);
    const double ci = c.cinv[t];
    yp.x = fma(-ci, p.x, fma(c.ihx, u1c.x - u1e.x, c.ihz * (u2c.x - u2n.x)));
    yp.y = fma(-ci, p.y, fma(c.ihx, u1c.y - u1e.y, c.ihz * (u2c.y - u2n.y)));
}

}  // namespace bah
