// FP64 kernels of the flexible GMRES outer iteration, batched over
// right-hand sides (blockIdx.z or .y = right-hand side, strides in KS):
// block dot products and norms (warp-shuffle + shared-memory reductions in two
// deterministic stages), the Gram-Schmidt updates with selective
// reorthogonalisation, the Givens update of the Hessenberg least-squares
// problem, the triangular solve and the solution update x += Z y.
// A right-hand side whose active flag is 0 is skipped by every kernel.
#include "bah_internal.cuh"
#include "givens.cuh"
#include "df.cuh"

namespace bah {

__device__ __forceinline__ double2 warp_sum2(double2 v) {
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// block-wide sum of a double2 (blockDim.x a multiple of 32, at most 1024); result valid in thread 0
__device__ __forceinline__ double2 block_sum2(double2 v) {
    __shared__ double2 sh[32];   // one per warp, up to 1024 threads
    v = warp_sum2(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    double2 r = make_double2(0.0, 0.0);
    if (w == 0) {
        r = l < (int)(blockDim.x >> 5) ? sh[l] : make_double2(0.0, 0.0);
        r = warp_sum2(r);
    }
    __syncthreads();
    return r;
}

__device__ __forceinline__ bool inactive(const KS& ks, int r) { return ks.active && !ks.active[r]; }

// ---------------------------------------------------------------------------
// Gram-Schmidt with selective reorthogonalisation (Daniel-Gragg-Kaufman-Stewart
// criterion): a second pass runs only if ||w'|| < ||w|| / sqrt(2).  The
// projections and updates themselves are in k_gs.cu (FP64 basis) and
// k_krylov_df.cu; npart holds np partial sums of ||w'||^2 per right-hand side.
// ---------------------------------------------------------------------------
// reduce the pass-1 norm, decide on the second pass, set ||w|| for the Givens
// step: sc[2] = ||w_final||, sc[3] counts second passes; flag = 1 when
// ||w'||^2 < ||w||^2 / 2 (with the FP64 basis the last CTA of k_gs_axpy does both)
__global__ void __launch_bounds__(256) k_dgks_decide(const double* npart, int np, const double2* h1norm, int k,
                                                     int* flag, double* sc, double eta2, KS ks) {
    pdl_prologue();
    const int r = blockIdx.x;
    if (inactive(ks, r)) return;
    npart += r * GS_CTAS;
    double acc = 0.0;
    for (int e = threadIdx.x; e < np; e += blockDim.x) acc += npart[e];
    double2 s = block_sum2(make_double2(acc, 0.0));
    if (threadIdx.x == 0) {
        const double w0 = h1norm[r * ks.so + k].x;          // ||w||^2 before pass 1
        const int f = (s.x < eta2 * w0) ? 1 : 0;
        flag[r] = f;
        sc[r * 8 + 2] = sqrt(s.x);
        sc[r * 8 + 3] += (double)f;
    }
}
void launch_dgks_decide(const double* npart, int np, const double2* h1norm, int k, int* flag, double* sc, int nrhs,
                        const KS& ks, cudaStream_t st, double eta2) {
    launch_pdl(k_dgks_decide, dim3(nrhs), dim3(256), 0, st, npart, np, h1norm, k, flag, sc, eta2, ks);
}
// after pass 2: ||w''|| replaces ||w'||
__global__ void __launch_bounds__(256) k_pass2_norm(const double* npart, int np, const int* flag, double* sc, KS ks) {
    pdl_prologue();
    const int r = blockIdx.x;
    if (inactive(ks, r) || flag[r] == 0) return;
    npart += r * GS_CTAS;
    double acc = 0.0;
    for (int e = threadIdx.x; e < np; e += blockDim.x) acc += npart[e];
    double2 s = block_sum2(make_double2(acc, 0.0));
    if (threadIdx.x == 0) sc[r * 8 + 2] = sqrt(s.x);
}
void launch_pass2_norm(const double* npart, int np, const int* flag, double* sc, int nrhs, const KS& ks,
                       cudaStream_t st) {
    launch_pdl(k_pass2_norm, dim3(nrhs), dim3(256), 0, st, npart, np, flag, sc, ks);
}

// ---------------------------------------------------------------------------
// 2-norm of w per right-hand side: sc[r*8 + slot] = ||w_r||
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_norm2_partial(const double2* __restrict__ w, size_t n, double* partial, KS ks) {
    pdl_prologue();
    const int r = blockIdx.y;
    if (inactive(ks, r)) return;
    w += r * ks.sw;
    double acc = 0.0;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double2 b = w[e];
        acc += b.x * b.x + b.y * b.y;
    }
    double2 s = block_sum2(make_double2(acc, 0.0));
    if (threadIdx.x == 0) partial[r * RED_CTAS + blockIdx.x] = s.x;
}
__global__ void __launch_bounds__(256) k_norm2_final(const double* partial, int np, double* sc, int slot, KS ks) {
    pdl_prologue();
    const int r = blockIdx.x;
    if (inactive(ks, r)) return;
    double acc = 0.0;
    for (int e = threadIdx.x; e < np; e += blockDim.x) acc += partial[r * RED_CTAS + e];
    double2 s = block_sum2(make_double2(acc, 0.0));
    if (threadIdx.x == 0) sc[r * 8 + slot] = sqrt(s.x);
}
void launch_norm2(const double2* w, size_t n, double* partial, double* sc, int slot, int nrhs, const KS& ks,
                  cudaStream_t st) {
    launch_pdl(k_norm2_partial, dim3(dim3(RED_CTAS, nrhs)), dim3(256), 0, st, w, n, partial, ks);
    launch_pdl(k_norm2_final, dim3(nrhs), dim3(256), 0, st, partial, RED_CTAS, sc, slot, ks);
}

// x += sum_i y_i Z_i  (Z in the preconditioner's precision, x in FP64), k per right-hand side
template <class Vz>
__global__ void __launch_bounds__(256) k_update_x(const Vz* __restrict__ Z, const int* kk, const double2* __restrict__ y,
                                                  double2* __restrict__ x, size_t n, KS ks) {
    pdl_prologue();
    const int r = blockIdx.y;
    const int k = kk[r];
    if (k <= 0) return;
    Z += r * ks.sz;
    y += r * ks.so;
    x += r * ks.sx;
    __shared__ double2 c[64];
    if (threadIdx.x < k) c[threadIdx.x] = y[threadIdx.x];
    __syncthreads();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        double2 acc = x[e];
        for (int i = 0; i < k; ++i) {
            const Vz zv = Z[(size_t)i * n + e];
            const double zx = (double)zv.x, zy = (double)zv.y;
            acc.x += c[i].x * zx - c[i].y * zy;
            acc.y += c[i].x * zy + c[i].y * zx;
        }
        x[e] = acc;
    }
}
// FP32 Z (mixed mode): the k products in double-float arithmetic (y split
// once per CTA into double-float pairs, every product an error-free FP32
// product, every sum a two-sum), added to the FP64 x once per element; the
// loads of kU rows go out together
template <>
__global__ void __launch_bounds__(256) k_update_x<float2>(const float2* __restrict__ Z, const int* kk,
                                                          const double2* __restrict__ y, double2* __restrict__ x,
                                                          size_t n, KS ks) {
    pdl_prologue();
    const int r = blockIdx.y;
    const int k = kk[r];
    if (k <= 0) return;
    Z += r * ks.sz;
    y += r * ks.so;
    x += r * ks.sx;
    __shared__ float4 c[64];
    if (threadIdx.x < k) c[threadIdx.x] = cdf_from_double2(y[threadIdx.x]);
    __syncthreads();
    constexpr int kU = 8;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        dfacc ar, ai;
        auto mac = [&](const float2& zv, const float4& cc) {
            // (cr + i ci)(zx + i zy) = (cr zx - ci zy) + i (cr zy + ci zx)
            const dfl cr = re_of(cc), ci = im_of(cc);
            ar.add(df_mul_f(cr, zv.x));
            ar.add(df_neg(df_mul_f(ci, zv.y)));
            ai.add(df_mul_f(cr, zv.y));
            ai.add(df_mul_f(ci, zv.x));
        };
        int i = 0;
        for (; i + kU <= k; i += kU) {
            float2 zv[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) zv[u] = __ldg(Z + (size_t)(i + u) * n + e);
#pragma unroll
            for (int u = 0; u < kU; ++u) mac(zv[u], c[i + u]);
        }
        for (; i < k; ++i) mac(__ldg(Z + (size_t)i * n + e), c[i]);
        double2 acc = x[e];
        acc.x += ar.value();
        acc.y += ai.value();
        x[e] = acc;
    }
}
template <class Vz>
void launch_update_x(const Vz* Z, const int* kk, const double2* y, double2* x, size_t n, int nrhs, const KS& ks,
                     cudaStream_t st) {
    launch_pdl(k_update_x<Vz>, dim3(dim3(RED_CTAS * 2, nrhs)), dim3(256), 0, st, Z, kk, y, x, n, ks);
}
template void launch_update_x<double2>(const double2*, const int*, const double2*, double2*, size_t, int, const KS&,
                                       cudaStream_t);
template void launch_update_x<float2>(const float2*, const int*, const double2*, double2*, size_t, int, const KS&,
                                      cudaStream_t);

// v = w / sc[slot]  (per right-hand side)
__global__ void k_scale_copy(const double2* __restrict__ w, const double* sc, int slot, double2* __restrict__ v,
                             size_t n, size_t sw, size_t sv, KS ks) {
    pdl_prologue();
    const int r = blockIdx.y;
    if (inactive(ks, r)) return;
    w += r * sw;
    v += r * sv;
    const double s = 1.0 / sc[r * 8 + slot];
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double2 a = w[e];
        v[e] = make_double2(a.x * s, a.y * s);
    }
}
// c = a - b
__global__ void k_sub(const double2* __restrict__ a, const double2* __restrict__ b, double2* __restrict__ c, size_t n) {
    pdl_prologue();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        c[e] = csub(a[e], b[e]);
}
void launch_sub(const double2* a, const double2* b, double2* c, size_t n, cudaStream_t st) {
    launch_pdl(k_sub, dim3(RED_CTAS * 2), dim3(256), 0, st, a, b, c, n);
}

void launch_scale_copy(const double2* w, const double* sc, int slot, double2* v, size_t n, size_t sw, size_t sv,
                       int nrhs, const KS& ks, cudaStream_t st) {
    launch_pdl(k_scale_copy, dim3(dim3(RED_CTAS * 2, nrhs)), dim3(256), 0, st, w, sc, slot, v, n, sw, sv, ks);
}

// ---------------------------------------------------------------------------
// Hessenberg column j = h1 + h2 (two Gram-Schmidt passes) with subdiagonal
// ||w||; apply the previous Givens rotations, form the new one, update g (givens.cuh;
// with the FP64 basis k_gs_store runs it beside the copy of the new basis vector).
// Rotation [c s; -conj(s) c] with c real.  status[0] = |g_{j+1}|,
// status[1] = h_{j+1,j}, status[2] = 1 if a non-finite value appeared.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(32) k_arnoldi_givens(GivensArgs a, KS ks) {
    pdl_prologue();
    arnoldi_givens(a, blockIdx.x, ks);
}
void launch_arnoldi_givens(const GivensArgs& a, int nrhs, const KS& ks, cudaStream_t st) {
    launch_pdl(k_arnoldi_givens, dim3(nrhs), dim3(32), 0, st, a, ks);
}

// R y = g(0..k-1), R upper triangular stored column-major with leading dimension ldh,
// k <= kMaxTri.  The triangle is copied to shared memory at once; then one warp takes the
// columns from the last, a lane per row (two above 32).  By one thread, with each entry
// loaded when its product was due, k = 20 took 79 us; now 17.
constexpr int kMaxTri = 64;
__global__ void __launch_bounds__(128) k_triangular_solve(const double2* Hm, int ldh, const double2* g, const int* kk,
                                                          double2* y, KS ks) {
    pdl_prologue();
    const int r = blockIdx.x;
    const int k = kk[r];
    if (k <= 0) return;
    Hm += r * ks.sh;
    g += r * ks.so;
    y += r * ks.so;
    __shared__ double2 R[kMaxTri * (kMaxTri + 1) / 2];            // column c at c (c + 1) / 2
    const int lane = threadIdx.x & 31;
    for (int c = threadIdx.x >> 5; c < k; c += 4)
        for (int i = lane; i <= c; i += 32) R[c * (c + 1) / 2 + i] = Hm[(size_t)c * ldh + i];
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double2 acc[2], inv[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = lane + 32 * q;
        acc[q] = i < k ? g[i] : make_double2(0.0, 0.0);
        inv[q] = i < k ? cdiv(make_double2(1.0, 0.0), R[i * (i + 1) / 2 + i]) : make_double2(0.0, 0.0);
    }
    for (int c = k - 1; c >= 0; --c) {
        const bool up = c >= 32;
        const double2 v = cmul(up ? acc[1] : acc[0], up ? inv[1] : inv[0]);
        const double2 yc = make_double2(__shfl_sync(0xffffffffu, v.x, c & 31), __shfl_sync(0xffffffffu, v.y, c & 31));
        if (lane == (c & 31)) y[c] = yc;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = lane + 32 * q;
            if (i < c) acc[q] = csub(acc[q], cmul(R[c * (c + 1) / 2 + i], yc));
        }
    }
}
void launch_triangular_solve(const double2* Hm, int ldh, const double2* g, const int* kk, double2* y, int nrhs,
                             const KS& ks, cudaStream_t st) {
    launch_pdl(k_triangular_solve, dim3(nrhs), dim3(128), 0, st, Hm, ldh, g, kk, y, ks);
}

// g = beta e_1, status = (beta, 0, 0)
__global__ void k_init_arnoldi(const double* sc, double2* g, int m, double* status, KS ks) {
    pdl_prologue();
    const int r = blockIdx.x;
    if (inactive(ks, r)) return;
    g += r * ks.so;
    const double beta = sc[r * 8 + 0];
    for (int i = threadIdx.x; i <= m; i += blockDim.x) g[i] = make_double2(i == 0 ? beta : 0.0, 0.0);
    if (threadIdx.x == 0) { status[r * 4 + 0] = beta; status[r * 4 + 1] = 0.0; status[r * 4 + 2] = 0.0; }
}
void launch_init_arnoldi(const double* sc, double2* g, int m, double* status, int nrhs, const KS& ks, cudaStream_t st) {
    launch_pdl(k_init_arnoldi, dim3(nrhs), dim3(128), 0, st, sc, g, m, status, ks);
}

}  // namespace bah
