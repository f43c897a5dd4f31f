// Single Gram-Schmidt and block products of libbah on given vectors, for test_gpu_exact_sums.py.
// All pointers are device pointers; every function returns a CUDA error code.
#include "bah_internal.cuh"
#include "fix60.cuh"

using namespace bah;

namespace {
struct Dev {
    void* p = nullptr;
    explicit Dev(size_t bytes) {
        if (cudaMalloc(&p, bytes) != cudaSuccess) p = nullptr;
        else cudaMemset(p, 0, bytes);
    }
    ~Dev() { cudaFree(p); }
    template <class T> T* as() const { return (T*)p; }
};
struct Basis {                      // vectors of V (n entries each) as basis vectors
    Tiles tl;
    Dev vl, ve, vc, sc;
    Basis(size_t n, size_t nc, int count)
        : tl(n, nc), vl(tl.padded() * count * sizeof(int4)), ve((size_t)tl.count * count * sizeof(int)),
          vc(n * sizeof(double2)), sc(8 * sizeof(double)) {
        const double one = 1.0;
        cudaMemcpy(sc.p, &one, sizeof(one), cudaMemcpyHostToDevice);
    }
    bool ok() const { return vl.p && ve.p && vc.p && sc.p; }
    void store(const double2* v, int row) {
        launch_basis_store(v, sc.as<double>(), 0, vc.as<double2>(), tl.n, vl.as<int4>() + row * tl.padded(),
                           ve.as<int>() + (size_t)row * tl.count, tl, 0, 1, KS(), 0);
    }
};
int finish() {
    const cudaError_t e = cudaGetLastError(), s = cudaDeviceSynchronize();
    return (int)(e != cudaSuccess ? e : s);
}
}  // namespace

extern "C" {

// out[0 .. k) = V^H w, out[k] = |w|^2; then w -= sum coef_i V_i (coef: k + 1 entries, the last |w|^2)
// and norm[0] = ||w||
int gs_pass(const double2* V, int k, double2* w, long long n, long long nc, double2* out, const double2* coef, double* norm) {
    if (gs_prepare() != BAH_OK) return -1;
    Basis b(n, nc, k);
    Dev partial((size_t)(k + 1) * GS_CTAS * sizeof(double2)), npart(GS_CTAS * sizeof(double)), cnt(sizeof(int)), flag(sizeof(int));
    if (!b.ok() || !partial.p || !npart.p || !cnt.p || !flag.p) return -2;
    for (int i = 0; i < k; ++i) b.store(V + (size_t)i * n, i);
    launch_dot_norm(b.vl.as<int4>(), b.ve.as<int>(), k, w, b.tl, partial.as<double2>(), out, nullptr, cnt.as<int>(), 1, KS(), 0);
    const GsNorm nm{cnt.as<int>(), flag.as<int>(), b.sc.as<double>(), 0.5};
    launch_axpy_norm(b.vl.as<int4>(), b.ve.as<int>(), k, coef, w, b.tl, npart.as<double>(), 1, nm, 1, KS(), 0);
    cudaMemcpy(norm, b.sc.as<double>() + 2, sizeof(double), cudaMemcpyDeviceToDevice);
    return finish();
}

// V: k blocks of s vectors.  C = V^H W, G = W^H W, W2 = W T (T upper triangular), then W -= V Y
int block_products(const double2* V, int k, int s, double2* W, long long n, long long nc, double2* C, double2* G,
                   const double2* T, double2* W2, const double2* Y) {
    if (gs_prepare() != BAH_OK || block_prepare() != BAH_OK) return -1;
    Basis b(n, nc, k * s);
    Dev part((size_t)(k + 1) * s * s * RED_CTAS * sizeof(double2));
    if (!b.ok() || !part.p) return -2;
    const size_t sv = (size_t)k * b.tl.padded(), se = (size_t)k * b.tl.count;
    for (int i = 0; i < k; ++i)
        for (int a = 0; a < s; ++a) b.store(V + ((size_t)i * s + a) * n, a * k + i);
    const int4* vl = b.vl.as<int4>();
    const int* ve = b.ve.as<int>();
    launch_block_dot(vl, ve, sv, se, k, s, W, b.tl, part.as<double2>(), C, 0);
    launch_block_gram(s, W, b.tl, part.as<double2>(), G, 0);
    launch_block_scale(W, s, T, W2, b.tl.n, nullptr, nullptr, 0, 0, b.tl, 0);
    launch_block_update(vl, ve, sv, se, k, s, Y, W, b.tl, 0);
    return finish();
}
}
