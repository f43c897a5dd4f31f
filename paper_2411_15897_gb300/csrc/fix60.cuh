// Sums of products on the integer pipe, with FP64's rounding in the norm.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM, but 28 integer ones of
// 32 x 32 + 64 bits (both measured; a complex product takes 4 of the first or
// 12 of the second).  A vector that meets many others is therefore held as block
// fixed point: the entries of a tile (kTile entries of one component)
// share one exponent E, |x| < 2^E for every real of the tile, and each real is
// the 60-bit integer X = round(x 2^(59 - E)), split into two signed limbs,
// X = h 2^30 + l with |h| <= 2^29, -2^29 <= l < 2^29.  A product of two such
// integers takes three multiply-adds (h h, and h l + l h into a second
// accumulator); l l lies below 2^-60 of the largest product and its mean is
// zero unless both factors are the same number.  Sums of the products are
// exact integers, rounded to FP64 once.
//
// Error: every factor is rounded to 2^-59 of its tile's largest real.  Where one
// factor is a coefficient, it gives up head bits so that all rows' products fit
// (rounding and l l terms: 2^-56 of the largest product with up to 32 rows, 2^-51
// with 1024); a dense row of np points gives up dense_head(np).  An FP64 sum
// rounds every partial sum to 2^-53 of itself.  So the bound is one in the norm
// (a tile's largest real is at most sqrt(512) = 22.6 times its r.m.s.), and none
// per entry: a real 2^-q below its tile's largest keeps 60 - q bits, where FP64
// keeps 53, and from q = 60 on it counts as 0.  Entries of unrelated size (the
// components of a vector, in their own units) therefore never share a tile.
//
// Exponents are stored biased as in an FP64 number (E + 1023), at least
// kExpMin; a tile with an infinity or NaN stores kExpBad, and every sum it
// enters becomes NaN.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace bah {

constexpr int kTileU = 8;                 // entries per lane of a tile
constexpr int kTile = 32 * kTileU;        // entries of a tile: entry u * 32 + lane
constexpr int kExpBad = 0x800;            // exponent of a tile that holds a non-finite entry
constexpr int kExpMin = 64;

// A vector of n entries in components of nc as tiles: a tile belongs to one component (the
// displacements' and the pressure's entries have unrelated units: in one tile, entries 2^-33 of
// its largest would keep 27 bits), the last tile of a component is partial.  Tile t's limbs
// stand at t * kTile.
struct Tiles {
    size_t n, nc;
    unsigned per, count;     // tiles per component and in all
    Tiles() = default;
    Tiles(size_t n_, size_t nc_) : n(n_), nc(nc_), per((unsigned)((nc_ + kTile - 1) / kTile)), count(per * (unsigned)(n_ / nc_)) {}
    size_t padded() const { return (size_t)count * kTile; }
#ifdef __CUDACC__
    // first entry of tile t, and the end of its component
    __device__ __forceinline__ size_t first(unsigned t, size_t& end) const {
        const unsigned c = (t >= per) + (t >= 2 * per) + (t >= 3 * per);      // at most four components
        end = (c + 1) * nc;
        return c * nc + (size_t)(t - c * per) * kTile;
    }
#endif
};

// the exponent field (with the bits below it) of |x|, for the maximum over a tile
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }
// biased tile exponent from the largest abs_hi
__device__ __forceinline__ int tile_exp(int max_hi) {
    const int f = max_hi >> 20;
    return f >= 0x7ff ? kExpBad : (f + 1 < kExpMin ? kExpMin : f + 1);
}
// round(x 2^(59 - (eb - 1023))) for |x| < 2^(eb - 1023), eb >= kExpMin
__device__ __forceinline__ long long fix60(double x, int eb) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    // significand with its leading one at bit 63 (subnormals, e = 0, shift out)
    const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;
    const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 11);
    const int sh = eb - e + 3;
    const long long v = sh > 63 ? 0 : (long long)(((m >> sh) + 1) >> 1);
    const long long sg = (long long)((int)hi >> 31);
    return (v ^ sg) - sg;
}
__device__ __forceinline__ void limbs(long long v, int& h, int& l) {
    h = (int)((v + (1 << 29)) >> 30);
    l = (int)(v - ((long long)h << 30));
}
// the same for an FP32 number (24 bits: exact down to 2^-36 of the largest)
__device__ __forceinline__ long long fix60(float x, int eb) {
    const unsigned b = (unsigned)__float_as_int(x);
    const int e = (int)((b >> 23) & 0xffu);
    const unsigned long long m = (unsigned long long)((b << 8) | 0x80000000u) << 32;
    const int sh = eb - (e - 127 + 1023) + 3;
    const long long v = sh > 63 || e == 0 ? 0 : (long long)(((m >> sh) + 1) >> 1);
    const long long sg = (long long)((int)b >> 31);
    return (v ^ sg) - sg;
}
__device__ __forceinline__ int abs_hi(float x) { return __float_as_int(x) & 0x7fffffff; }
// biased tile exponent from the largest abs_hi of FP64 (double) or FP32 (float) numbers
template <class R> __device__ __forceinline__ int tile_exp_of(int max_hi) {
    if (sizeof(R) == 8) return tile_exp(max_hi);
    const int f = max_hi >> 23;
    return f >= 0xff ? kExpBad : f - 127 + 1023 + 1;
}
// re.h, re.l, im.h, im.l
template <class V> __device__ __forceinline__ int4 limbs2(V z, int eb) {
    int4 r;
    limbs(fix60(z.x, eb), r.x, r.y);
    limbs(fix60(z.y, eb), r.z, r.w);
    return r;
}
// acc += a b, as one instruction (written out: from the C expression the compiler forms
// separate products and 64-bit additions, three instructions)
__device__ __forceinline__ void mad(long long& acc, int a, int b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// 2^p (0 below the normal range, infinity above it)
__device__ __forceinline__ double pow2(int p) {
    return p < -1022 ? 0.0 : __hiloint2double((p > 1023 ? 0x7ff : p + 1023) << 20, 0);
}

// A lane's exact sum hh 2^60 + cr 2^30 (|hh| <= 2^62, |cr| <= 2^63) as
// hi 2^65 + lo 2^39, lo < 2^26: the sums of 32 lanes' parts fit 64 and 32 bits
__device__ __forceinline__ void split65(long long hh, long long cr, long long& hi, unsigned& lo) {
    const long long t = hh + (cr >> 30);
    hi = t >> 5;
    lo = ((unsigned)t & 31u) << 21 | (((unsigned)cr >> 9) & 0x1fffffu);
}

// Sum over the warp's lanes of NV values at once: each step adds half of the
// values across one lane bit, so a lane ends with the sum of value
// lane / (32 / NV) (NV a power of two, 2 to 16)
template <int NV, class T>
__device__ __forceinline__ T warp_sum_values(T* v, int lane) {
    int o = 16;
#pragma unroll
    for (int c = NV / 2; c >= 1; c >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < c; ++i) {
            const T keep = up ? v[i + c] : v[i], give = up ? v[i] : v[i + c];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    for (; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// ---------------------------------------------------------------------------
// Dense product x = A g with A's rows in block fixed point (one exponent per
// row) and g converted once per CTA: the coarsest solve with the FP64 inverse.
// dense_head(np): bits that g gives up so that a lane's np / 32 products of
// 2 x 2^58 fit 2^62 (none up to 256 points, 4 at 4096).
// Bound: the chain of conversion, barriers and L2 reads.  With FP64 multiply-adds the
// solve was bound by the FP64 pipe: 48 x 40 x 28 (840 points, three blocks, all SMs)
// 32 -> 14 us per launch; inside the cluster kernel, on 16 SMs, 64 x 64 (256 points)
// 27.6 -> 21.5 us.
// ---------------------------------------------------------------------------
__host__ __device__ inline int dense_head(int np) {
    int h = 0;
    while ((256 << h) < np) ++h;
    return h;
}
// one warp: sum over c < np of arow[c] g[c], valid in lane 0
__device__ __forceinline__ double2 dense_row(const int4* __restrict__ arow, int ea, const int4* g, int eg, int np,
                                             int lane) {
    long long hr = 0, cr = 0, hi = 0, ci = 0;
    auto mac = [&](const int4& a, const int4& b) {
        // a b = (ax bx - ay by) + i (ax by + ay bx)
        const int nz = -b.z, nw = -b.w;
        mad(hr, a.x, b.x); mad(hr, a.z, nz);
        mad(cr, a.x, b.y); mad(cr, a.y, b.x);
        mad(cr, a.z, nw); mad(cr, a.w, nz);
        mad(hi, a.x, b.z); mad(hi, a.z, b.x);
        mad(ci, a.x, b.w); mad(ci, a.y, b.z);
        mad(ci, a.z, b.y); mad(ci, a.w, b.x);
    };
    auto carry = [&]() {                       // the cross sums hold 8 products
        hr += cr >> 30; cr &= 0x3fffffff;
        hi += ci >> 30; ci &= 0x3fffffff;
    };
    constexpr int kU = 8;
    int c = lane;
    for (; c + 32 * (kU - 1) < np; c += 32 * kU) {
        int4 a[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) a[u] = __ldg(arow + c + 32 * u);
#pragma unroll
        for (int u = 0; u < kU; ++u) mac(a[u], g[c + 32 * u]);
        carry();
    }
    if (c < np) {
        int4 a[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) a[u] = c + 32 * u < np ? __ldg(arow + c + 32 * u) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (c + 32 * u < np) mac(a[u], g[c + 32 * u]);
    }
    long long v[2];
    unsigned lo[2];
    split65(hr, cr, v[0], lo[0]);
    split65(hi, ci, v[1], lo[1]);
    const long long sv = warp_sum_values<2>(v, lane);            // lanes 0-15 the real part, 16-31 the imaginary
    const unsigned sl = warp_sum_values<2>(lo, lane);
    const int p = (ea - 1023) + (eg - 1023) - 118;
    double s = fma((double)sv, pow2(p + 65), (double)sl * pow2(p + 39));
    if (ea == kExpBad || eg >= kExpBad) s = __longlong_as_double(0x7ff8000000000000ll);
    return make_double2(s, __shfl_down_sync(0xffffffffu, s, 16));
}
// one CTA: g[0 .. np) = limbs of the entries get(c), their exponent returned
// (blockDim.x a multiple of 32, at most 1024; red: 32 ints of shared memory;
// ends with a barrier)
template <class V, class R, class F>
__device__ __forceinline__ int dense_load(int4* g, int np, int* red, F get) {
    int mx = 0;
    for (int c = threadIdx.x; c < np; c += blockDim.x) {
        const V v = get(c);
        *reinterpret_cast<V*>(g + c) = v;
        mx = max(mx, max(abs_hi(v.x), abs_hi(v.y)));
    }
    mx = (int)__reduce_max_sync(0xffffffffu, (unsigned)mx);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    mx = (int)__reduce_max_sync(0xffffffffu, lane < nw ? (unsigned)red[lane] : 0u);
    const int eg = tile_exp_of<R>(mx) + dense_head(np);
    for (int c = threadIdx.x; c < np; c += blockDim.x) {
        const V v = *reinterpret_cast<const V*>(g + c);
        g[c] = limbs2(v, eg);
    }
    __syncthreads();
    return eg;
}

}  // namespace bah
