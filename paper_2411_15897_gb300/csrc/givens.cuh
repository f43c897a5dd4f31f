// One column of the Arnoldi relation: h = h1 + h2 with the previous Givens
// rotations applied, the new rotation, the rotated right-hand side and the step's
// status (residual estimate, ||w||, a non-finite value was seen).
#pragma once
#include "bah_internal.cuh"

namespace bah {

struct GivensArgs {
    double2* Hm;                 // Hessenberg columns, leading dimension ldh
    int ldh, j;
    const double2 *h1, *h2;
    const double* sc;            // scalars, 8 per right-hand side; [2] is ||w||
    double2 *cs, *sn, *g;
    double* status;              // 4 per right-hand side
    double* host;                // pinned copy of status, or null
};

// right-hand side r, by the first warp of a CTA.  An FP64 instruction holds the pipe for
// 16 cycles however few lanes use it, so only the recurrence p' = c b - conj(s) p down the
// column stays serial (4 instructions a rotation); the products with b before it, the
// entries c p + s b after it, and pairs of square roots and quotients use the lanes.
__device__ __forceinline__ void arnoldi_givens(const GivensArgs& a, int r, const KS& ks) {
    __shared__ double2 h[66], sb[65], cb[65], pv[66], ssn[65];
    __shared__ double scs[65];
    const int lane = threadIdx.x, j = a.j;
    if (lane >= 32) return;
    double* status = a.status + r * 4;
    if (ks.active && !ks.active[r]) {
        if (a.host && lane < 3) a.host[r * 4 + lane] = status[lane];
        return;
    }
    double2* Hcol = a.Hm + r * ks.sh + (size_t)j * a.ldh;
    const double2 *h1 = a.h1 + r * ks.so, *h2 = a.h2 + r * ks.so;
    double2 *cs = a.cs + r * ks.so, *sn = a.sn + r * ks.so, *g = a.g + r * ks.so;
    const double wn = a.sc[r * 8 + 2];
    const double2 gj = g[j];
    bool bad = !isfinite(wn);
    for (int i = lane; i <= j; i += 32) {
        const double2 v = cadd(h1[i], h2[i]);
        h[i] = v;
        bad |= !isfinite(v.x) || !isfinite(v.y);
    }
    bad = __any_sync(0xffffffffu, bad);
    __syncwarp();
    for (int i = lane; i < j; i += 32) {         // rotation i and the entry below its row
        const double c = cs[i].x;
        const double2 s = sn[i], b = h[i + 1];
        scs[i] = c;
        ssn[i] = s;
        sb[i] = cmul(s, b);
        cb[i] = cscale(b, c);
    }
    __syncwarp();
    double2 p = h[0];                            // the entry carried down the column (every lane)
    for (int i = 0; i < j; ++i) {
        if (lane == 0) pv[i] = p;
        const double2 s = ssn[i], t = cb[i];
        p = make_double2(fma(-s.y, p.y, fma(-s.x, p.x, t.x)), fma(s.y, p.x, fma(-s.x, p.y, t.y)));
    }
    __syncwarp();
    for (int i = lane; i < j; i += 32) Hcol[i] = cadd(cscale(pv[i], scs[i]), sb[i]);
    const double na2 = p.x * p.x + p.y * p.y, nb2 = wn * wn;
    double c;
    double2 s;
    if (nb2 == 0.0) {
        c = 1.0; s = make_double2(0.0, 0.0);
    } else if (na2 == 0.0) {
        c = 0.0; s = make_double2(wn * (1.0 / sqrt(nb2)), 0.0);
    } else {
        const double q = sqrt(lane == 0 ? na2 : na2 + nb2);
        const double na = __shfl_sync(0xffffffffu, q, 0), rr = __shfl_sync(0xffffffffu, q, 1);
        const double d = lane == 0 ? na / rr : 1.0 / (na * rr);
        c = __shfl_sync(0xffffffffu, d, 0);
        s = cscale(p, wn * __shfl_sync(0xffffffffu, d, 1));
    }
    if (lane != 0) return;
    cs[j] = make_double2(c, 0.0);
    sn[j] = s;
    Hcol[j] = make_double2(fma(s.x, wn, p.x * c), fma(s.y, wn, p.y * c));
    Hcol[j + 1] = make_double2(0.0, 0.0);
    g[j] = cscale(gj, c);
    const double2 gn = cscale(cmul(cconj(s), gj), -1.0);
    g[j + 1] = gn;
    const double st[3] = {sqrt(gn.x * gn.x + gn.y * gn.y), wn, bad ? 1.0 : 0.0};
    for (int i = 0; i < 3; ++i) {
        status[i] = st[i];
        if (a.host) a.host[r * 4 + i] = st[i];
    }
}

}  // namespace bah
