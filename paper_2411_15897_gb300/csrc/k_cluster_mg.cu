// Shared-memory-resident multigrid on a thread-block cluster (mixed mode).
//
// The small levels of a block's hierarchy (here: every level from l0 down to
// the coarsest) are held entirely in the shared memory of one cluster of up
// to 16 CTAs, one CTA per SM.  Each level's grid rows are split into equal
// slabs, one per CTA; a CTA stores, for the points of its slab, the level's
// Galerkin stencil (bfloat16 complex, slot-major), the iterate, a work
// vector and the right-hand side.  The coarsest level is solved with the
// dense FP64 inverse, held in block fixed point (fix60.cuh), read from global
// memory (it stays in L2) and applied to the gathered FP32 right-hand side with
// exact integer sums.  A stencil, restriction or prolongation tap
// that falls into another CTA's slab is read from that CTA's shared memory
// through the cluster's distributed shared memory (mapa + ld.shared::cluster).
//
// The cycle walks the same phases as the separate kernels -- zero-guess
// damped Jacobi, Jacobi, residual, restriction, the coarsest solve,
// prolongation and correction -- with the same per-point arithmetic, and the
// W-cycle's second coarse visits (Sec. 2.2), separated by the hardware
// cluster barrier.  Global memory is touched only to load the stencils and
// the level-l0 right-hand side (and iterate, on a warm start) at the start,
// to read the rows of the coarsest inverse, and to store the level-l0 result
// at the end.
//
// Deadlock freedom: the hardware co-schedules all CTAs of a cluster, every
// thread of every CTA executes the same sequence of barriers (the control
// flow depends only on kernel arguments; the only early exit is taken by a
// whole cluster at once), and a final barrier keeps every CTA's shared
// memory alive until no CTA of the cluster can still read it.
#include "bah_internal.cuh"
#include "fix60.cuh"
#include "intergrid.cuh"

#include <algorithm>
#include <cstring>
#include <type_traits>

namespace bah {

constexpr int kSmThreads = 512;   // threads per CTA (one CTA per SM)

namespace {

__device__ __forceinline__ uint32_t mapa_rank(uint32_t local_addr, unsigned rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 ld_cluster_at(uint32_t cluster_addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(cluster_addr));
    return v;
}
template <int BYTES> __device__ __forceinline__ void cp_async(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}

}  // namespace

template <int RM>
__global__ void __launch_bounds__(kSmThreads, 1) k_cluster_mg(SmArgs a) {
    constexpr int MODE = BAH_MIXED;
    using V = typename Prec<MODE>::V;
    using CC = typename Prec<MODE>::CC;
    using R = typename Prec<MODE>::R;
    constexpr unsigned kV = sizeof(V);
    constexpr int G = RM;                               // ghost columns on each side of a row
    const unsigned cid = cluster_index();
    const int z = (int)(cid % (unsigned)a.nb), rr = (int)(cid / (unsigned)a.nb);
    const unsigned q = cluster_rank();
    const int tid = threadIdx.x, nth = blockDim.x;
    const int type = a.b0 + z;
    const bool nodx = type == 0, nodz = type == 1;
    extern __shared__ __align__(128) unsigned char sm[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);
    const int nlev = a.nlev, kc = nlev - 1;

    auto p0 = [&](const SmLevel& L) { return (int)q * L.rp * L.n1; };
    auto nrow = [&](const SmLevel& L) { return max(0, min(L.n2 - (int)q * L.rp, L.rp)); };   // own rows
    auto nown = [&](const SmLevel& L) { return nrow(L) * L.n1; };
    // own points: b unpadded, x and t with G zero columns before and after each row
    auto vec = [&](unsigned off) { return reinterpret_cast<V*>(sm + off); };
    auto at = [&](const SmLevel& L, int r, int i) { return r * (L.n1 + 2 * G) + G + i; };
    // cluster address of column 0 of grid row `row` of x or t of level L (one owner
    // lookup and one mapa per row; the columns follow at kV bytes), and of b
    auto row_addr = [&](const SmLevel& L, unsigned off, int row) -> uint32_t {
        const int owner = (int)(((float)row + 0.5f) * L.inv_rp);
        return mapa_rank(sbase + off + (uint32_t)at(L, row - owner * L.rp, 0) * kV, (unsigned)owner);
    };
    auto row_addr_b = [&](const SmLevel& L, int row) -> uint32_t {
        const int owner = (int)(((float)row + 0.5f) * L.inv_rp);
        return mapa_rank(sbase + L.off_b + (uint32_t)((row - owner * L.rp) * L.n1) * kV, (unsigned)owner);
    };
    // own row and column of own point lt of level L
    auto own_rc = [&](const SmLevel& L, int lt, int& r, int& col) {
        r = (int)(((float)lt + 0.5f) * L.inv_n1);
        col = lt - r * L.n1;
    };
    auto coef = [&](int k) { return reinterpret_cast<const CC*>(sm + a.lv[k].off_c); };

    // ---- load ----
    // The stencils never change after setup, so they are copied (cp.async: many
    // copies in flight per thread) before this launch waits for the kernel in front
    // of it; the level-l0 vectors follow after the wait.
    for (int k = 0; k < kc; ++k) {
        const SmLevel& L = a.lv[k];
        const int np = L.n1 * L.n2, own = nown(L), g0 = p0(L), cap = L.rp * L.n1;
        const int nsl = (2 * a.rx[z][k] + 1) * (2 * a.rz[z][k] + 1);
        const CC* S = (const CC*)a.S[z][k];
        // 16 bytes per copy where every slot's slab starts and ends on 16 bytes
        constexpr int E = 16 / (int)sizeof(CC);
        if (E == 1 || (np % E == 0 && cap % E == 0 && own % E == 0)) {
            const int own4 = own / E, cnt4 = nsl * own4;
            const float inv = 1.0f / (float)max(own4, 1);
            for (int e = tid; e < cnt4; e += nth) {
                const int s = (int)(((float)e + 0.5f) * inv), t = (e - s * own4) * E;
                cp_async<16>(sbase + L.off_c + (uint32_t)(s * cap + t) * (uint32_t)sizeof(CC), S + (size_t)s * np + g0 + t);
            }
        } else {
            for (int s = 0; s < nsl; ++s)
                for (int t = tid; t < own; t += nth)
                    cp_async<sizeof(CC)>(sbase + L.off_c + (uint32_t)(s * cap + t) * (uint32_t)sizeof(CC),
                                         S + (size_t)s * np + g0 + t);
        }
        // zero iterates, so that the ghost columns are zero
        const int cnt = L.rp * (L.n1 + 2 * G);
        for (int t = tid; t < cnt; t += nth) { vec(L.off_x)[t] = czero<V>(); vec(L.off_t)[t] = czero<V>(); }
    }
    for (int t = tid; t < a.lv[kc].rp * (a.lv[kc].n1 + 2 * G); t += nth) vec(a.lv[kc].off_x)[t] = czero<V>();
    pdl_prologue();
    if (a.active && !a.active[rr]) {                    // uniform over the cluster
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    __syncthreads();
    {
        const SmLevel& L = a.lv[0];
        const int own = nown(L), g0 = p0(L);
        const size_t roff = (size_t)rr * L.n1 * L.n2 + g0;
        for (int t = tid; t < own; t += nth) {
            cp_async<sizeof(V)>(sbase + L.off_b + (uint32_t)t * kV, (const V*)a.gb[z] + roff + t);
            if (a.warm) {
                int r, i;
                own_rc(L, t, r, i);
                cp_async<sizeof(V)>(sbase + L.off_x + (uint32_t)at(L, r, i) * kV, (const V*)a.gx[z] + roff + t);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    cluster_barrier();

    // ---- phases (own points only) ----
    // Jacobi sweep (res: residual) of level k with stencil radii RX, RZ: the RZ rows
    // above and below the slab are first copied from the neighbours' shared memory,
    // zero outside the grid, so that every tap is an unconditional local load (rows
    // read through the cluster with a test per tap cost 860 instructions per point,
    // this 250)
    V* halo = reinterpret_cast<V*>(sm + a.off_g);       // 2 RZ rows of the input's pitch
    auto sweep = [&](auto rx_, auto rz_, int k, unsigned xin, unsigned xout, bool res) {
        constexpr int RX = decltype(rx_)::value, RZ = decltype(rz_)::value;
        const SmLevel& L = a.lv[k];
        const int rows = nrow(L), r0 = (int)q * L.rp, P = L.n1 + 2 * G, cap = L.rp * L.n1;
        for (int e = tid; e < 2 * RZ * P; e += nth) {
            const int h = (int)(((float)e + 0.5f) * L.inv_p), col = e - h * P - G;
            const int row = h < RZ ? r0 - RZ + h : r0 + rows + h - RZ;
            const bool in = row >= 0 && row < L.n2 && col >= 0 && col < L.n1;
            halo[e] = in ? ld_cluster_at(row_addr(L, xin, row) + (uint32_t)col * kV) : czero<V>();
        }
        __syncthreads();
        const V* b = vec(L.off_b);
        const V* x = vec(xin);
        V* xo = vec(xout);
        const int own = rows * L.n1;
        for (int lt = tid; lt < own; lt += nth) {
            int r, i;
            own_rc(L, lt, r, i);
            const int o = at(L, r, i);
            if (!valid_pt(type, i, r0 + r)) { xo[o] = czero<V>(); continue; }
            const CC* cs = coef(k) + lt;
            V ax = czero<V>();
#pragma unroll
            for (int dz = -RZ; dz <= RZ; ++dz) {
                const int t = r + dz;
                const V* xr = (t < 0 ? halo + (RZ + t) * P : (t >= rows ? halo + (RZ + t - rows) * P : x + t * P)) + G + i;
#pragma unroll
                for (int dx = -RX; dx <= RX; ++dx) cfma(ax, ldc(cs[((dz + RZ) * (2 * RX + 1) + dx + RX) * cap]), xr[dx]);
            }
            const V d = csub(b[lt], ax);
            if (res) { xo[o] = d; continue; }
            const V dg = ldc(cs[(RZ * (2 * RX + 1) + RX) * cap]);
            const V c = cdiv1(d, dg), xv = x[o];
            xo[o] = cmk<V>(xv.x + (R)L.w * c.x, xv.y + (R)L.w * c.y);
        }
    };
    auto stencil_phase = [&](int k, unsigned xin, unsigned xout, bool res) {
        std::integral_constant<int, 1> one;
        std::integral_constant<int, RM> rm;
        if (a.rx[z][k] == RM && a.rz[z][k] == RM) sweep(rm, rm, k, xin, xout, res);
        else if (a.rx[z][k] == RM) sweep(rm, one, k, xin, xout, res);
        else if (a.rz[z][k] == RM) sweep(one, rm, k, xin, xout, res);
        else sweep(one, one, k, xin, xout, res);
    };
    auto jacobi_zero = [&](int k, unsigned xout) {
        const SmLevel& L = a.lv[k];
        const int own = nown(L);
        const V* b = vec(L.off_b);
        V* xo = vec(xout);
        const CC* cs = coef(k) + (size_t)(a.rz[z][k] * (2 * a.rx[z][k] + 1) + a.rx[z][k]) * (L.rp * L.n1);
        for (int lt = tid; lt < own; lt += nth) {
            int r, i;
            own_rc(L, lt, r, i);
            xo[at(L, r, i)] = valid_pt(type, i, (int)q * L.rp + r) ? cscale(cdiv1(b[lt], ldc(cs[lt])), (R)L.w) : czero<V>();
        }
    };
    auto restrict_ = [&](int k, unsigned rin) {          // b_{k+1} = R r_k on own coarse points
        const SmLevel& L = a.lv[k];
        const SmLevel& Lc = a.lv[k + 1];
        const int own = nown(Lc);
        V* bc = vec(Lc.off_b);
        for (int lt = tid; lt < own; lt += nth) {
            int J, I;
            own_rc(Lc, lt, J, I);
            J += (int)q * Lc.rp;
            V acc = czero<V>();
            if (valid_pt(type, I, J)) {
                const int bx = rbase(nodx, a.intergrid, I), bz = rbase(nodz, a.intergrid, J);
                R wxs[4], wzs[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    wxs[e] = rw_axis_t<R>(nodx, a.intergrid, L.n1, I, bx + e);
                    wzs[e] = rw_axis_t<R>(nodz, a.intergrid, L.n2, J, bz + e);
                }
                V v[16];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool rok = wzs[e] != R(0);
                    const uint32_t ra = row_addr(L, rin, rok ? bz + e : 0);
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        const bool ok = rok && wxs[f] != R(0);
                        v[e * 4 + f] = ld_cluster_at(ra + (uint32_t)(ok ? bx + f : 0) * kV);
                    }
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        const R wgt = wzs[e] * wxs[f];
                        acc.x += wgt * v[e * 4 + f].x;
                        acc.y += wgt * v[e * 4 + f].y;
                    }
            }
            bc[lt] = acc;
        }
    };
    auto prolong = [&](int k, unsigned xoff) {             // x_k += P x_{k+1} on own fine points
        const SmLevel& L = a.lv[k];
        const SmLevel& Lc = a.lv[k + 1];
        const int own = nown(L);
        V* x = vec(xoff);
        for (int lt = tid; lt < own; lt += nth) {
            int r, i;
            own_rc(L, lt, r, i);
            const int j = (int)q * L.rp + r;
            if (!valid_pt(type, i, j)) continue;
            int cx[2], cz[2];
            R wx[2], wz[2];
            pw_pair<R>(nodx, L.n1, i, cx, wx);
            pw_pair<R>(nodz, L.n2, j, cz, wz);
            V v[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t ra = row_addr(Lc, Lc.off_x, cz[e]);
#pragma unroll
                for (int f = 0; f < 2; ++f) v[e * 2 + f] = ld_cluster_at(ra + (uint32_t)cx[f] * kV);
            }
            const int o = at(L, r, i);
            V acc = x[o];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const R wgt = wz[e] * wx[f];
                    acc.x += wgt * v[e * 2 + f].x;
                    acc.y += wgt * v[e * 2 + f].y;
                }
            x[o] = acc;
        }
    };
    auto coarse = [&]() {                                   // x_c = A_c^{-1} b_c on own rows, exact integer sums
        const SmLevel& L = a.lv[kc];
        const int npc = L.n1 * L.n2, own = nown(L), g0 = p0(L);
        int4* gath = reinterpret_cast<int4*>(sm + a.off_g);
        const int eg = dense_load<V, R>(gath, npc, reinterpret_cast<int*>(sm + a.off_r), [&](int g) {
            return ld_cluster_at(row_addr_b(L, g / L.n1) + (uint32_t)(g % L.n1) * kV);
        });
        V* x = vec(L.off_x);
        const int lane = tid & 31;
        for (int row = tid >> 5; row < own; row += nth >> 5) {
            // the inverse's row from global memory (L2-resident)
            const double2 s = dense_row(a.inv[z] + (size_t)(g0 + row) * npc, a.inve[z][g0 + row], gath, eg, npc, lane);
            if (lane == 0) x[at(L, row / L.n1, row % L.n1)] = cconv<V>(s);
        }
    };
    auto zero_vec = [&](int k, unsigned off) {
        const int cnt = a.lv[k].rp * (a.lv[k].n1 + 2 * G);
        for (int t = tid; t < cnt; t += nth) vec(off)[t] = czero<V>();
    };
    auto copy_vec = [&](int k, unsigned from, unsigned to) {
        const int cnt = a.lv[k].rp * (a.lv[k].n1 + 2 * G);
        for (int t = tid; t < cnt; t += nth) vec(to)[t] = vec(from)[t];
    };

    // ---- the cycle: an explicit walk over the recursion of Algorithm 1 ----
    // Each pass of the loop picks the next phase from the per-level state and
    // runs it through one switch, so every phase's code exists once in the
    // kernel (fewer instructions to fetch after other kernels ran on the SM).
    enum { kJacobi, kZero, kResidual, kRestrict, kCoarse, kProlong, kCopy };
    unsigned xs[kMaxLevels], ts[kMaxLevels];
    int pc[kMaxLevels], nsw[kMaxLevels];
    bool warm[kMaxLevels];
    int k = 0;
    pc[0] = 0;
    warm[0] = a.warm != 0;
    while (true) {
        int op = -1, kk = k;
        unsigned u = 0, v = 0;
        bool zero = false;
        if (k == kc) {
            op = kCoarse;
            --k;
        } else {
            const SmLevel& L = a.lv[k];
            switch (pc[k]) {
            case 0: {                                       // entering the visit
                unsigned x = L.off_x, t = L.off_t;
                nsw[k] = 0;
                if (!warm[k]) {
                    // with a zero initial guess, start in the buffer from which the visit's
                    // buffer swaps (the pre-sweeps after the first, and the post-sweeps)
                    // end in off_x, where the parent level and the final store read the
                    // result: no copy phase
                    if (((a.nu_pre >= 1 ? a.nu_pre - 1 : 0) + a.nu_post) & 1) {
                        x = L.off_t;
                        t = L.off_x;
                    }
                    if (a.nu_pre >= 1) {
                        op = kJacobi;
                        zero = true;
                        v = x;
                        nsw[k] = 1;
                    } else {
                        op = kZero;
                        u = x;
                    }
                }
                xs[k] = x;
                ts[k] = t;
                pc[k] = 1;
                break;
            }
            case 1:                                         // pre-sweeps, then the residual
                if (nsw[k] < a.nu_pre) {
                    op = kJacobi;
                    u = xs[k];
                    v = ts[k];
                    ts[k] = u;
                    xs[k] = v;
                    ++nsw[k];
                } else {
                    op = kResidual;
                    u = xs[k];
                    v = ts[k];
                    pc[k] = 2;
                }
                break;
            case 2:
                op = kRestrict;
                u = ts[k];
                pc[k] = 3;
                break;
            case 3:                                         // the coarse visit(s)
                pc[k] = (a.wcycle && k + 1 < kc) ? 4 : 5;
                ++k;
                pc[k] = 0;
                warm[k] = false;
                break;
            case 4:                                         // the W-cycle's second coarse visit
                pc[k] = 5;
                ++k;
                pc[k] = 0;
                warm[k] = true;
                break;
            case 5:
                op = kProlong;
                u = xs[k];
                nsw[k] = 0;
                pc[k] = 6;
                break;
            case 6:                                         // post-sweeps, then the copy to off_x
                if (nsw[k] < a.nu_post) {
                    op = kJacobi;
                    u = xs[k];
                    v = ts[k];
                    ts[k] = u;
                    xs[k] = v;
                    ++nsw[k];
                    break;
                }
                pc[k] = 7;
                if (xs[k] != L.off_x) {
                    op = kCopy;
                    u = xs[k];
                    v = L.off_x;
                    xs[k] = L.off_x;
                }
                break;
            default:                                        // visit done
                break;
            }
            if (op < 0 && pc[kk] == 7) {
                if (kk == 0) break;
                k = kk - 1;
            }
        }
        if (op < 0) continue;
        switch (op) {
        case kJacobi:
        case kResidual:
            if (zero) jacobi_zero(kk, v);
            else stencil_phase(kk, u, v, op == kResidual);
            break;
        case kZero: zero_vec(kk, u); break;
        case kRestrict: restrict_(kk, u); break;
        case kCoarse: coarse(); break;
        case kProlong: prolong(kk, u); break;
        default: copy_vec(kk, u, v); break;
        }
        cluster_barrier();
    }

    // ---- store the level-l0 result; keep shared memory alive for remote readers ----
    {
        const SmLevel& L = a.lv[0];
        const int own = nown(L), g0 = p0(L);
        const size_t roff = (size_t)rr * L.n1 * L.n2 + g0;
        const V* x = vec(L.off_x);
        for (int t = tid; t < own; t += nth) {
            int r, i;
            own_rc(L, t, r, i);
            ((V*)a.gx[z])[roff + t] = x[at(L, r, i)];
        }
    }
    cluster_barrier();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static auto smmg_fn(int rm) { return rm <= 1 ? k_cluster_mg<1> : k_cluster_mg<2>; }

size_t smmg_layout(SmArgs& a, const int* n1, const int* n2, const int* nslot_max, int nlev, int cs, int rm) {
    const size_t vb = sizeof(float2), cb = sizeof(__nv_bfloat162);
    size_t off = 0, halo = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 15) & ~size_t(15);
        return (unsigned)o;
    };
    a.nlev = nlev;
    for (int k = 0; k < nlev; ++k) {
        SmLevel& L = a.lv[k];
        L.n1 = n1[k];
        L.n2 = n2[k];
        L.rp = (n2[k] + cs - 1) / cs;
        L.inv_rp = 1.0f / (float)L.rp;
        L.inv_n1 = 1.0f / (float)L.n1;
        L.inv_p = 1.0f / (float)(L.n1 + 2 * rm);
        const size_t cap = (size_t)L.rp * L.n1, padded = (size_t)L.rp * (L.n1 + 2 * rm);
        if (k < nlev - 1) {
            L.off_c = take(cap * nslot_max[k] * cb);
            L.off_t = take(padded * vb);
            halo = std::max(halo, (size_t)2 * rm * (L.n1 + 2 * rm) * vb);
        } else {
            L.off_c = 0;
            L.off_t = 0;
        }
        L.off_x = take(padded * vb);
        L.off_b = take(cap * vb);
    }
    // the sweeps' halo rows and the coarsest solve's right-hand side are never in use together
    const SmLevel& Lc = a.lv[nlev - 1];
    const size_t npc = (size_t)Lc.n1 * Lc.n2;
    a.off_g = take(std::max(npc * 16, halo));
    a.off_r = take(32 * 4);
    return off;
}

int smmg_prepare(int rm, int cs, size_t smem) {
    const void* fn = (const void*)smmg_fn(rm);
    // The attribute is the kernel's, shared by all contexts: it is always set to the most the device
    // gives a CTA, because a context that set it to its own size would take it from one created before.
    int dev = 0, most = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, fn) != cudaSuccess || smem + fa.sharedSizeBytes > (size_t)most ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) != cudaSuccess ||
        (cs > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

int launch_cluster_mg(const SmArgs& a, int rm, int nrhs, int cs, size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs * a.nb * nrhs);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, smmg_fn(rm), a);
    return e == cudaSuccess ? 0 : (int)e;
}

}  // namespace bah
