// FP64-accurate sums of products on the integer pipe.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM, but 64 integer ones of
// 32 x 32 + 64 bits (both measured).  A vector that meets many others is
// therefore held as block fixed point: the entries of a tile (kTile entries)
// share one exponent E, |x| < 2^E for every real of the tile, and each real is
// the 60-bit integer X = round(x 2^(59 - E)), split into two signed limbs,
// X = h 2^30 + l with |h| <= 2^29, -2^29 <= l < 2^29.  A product of two such
// integers takes three multiply-adds (h h, and h l + l h into a second
// accumulator); l l lies below 2^-60 of the largest product and its mean is
// zero unless both factors are the same number.  Sums of the products are
// exact integers.  So the error is that of rounding the inputs to 2^-60 of
// the tile's largest entry, where an FP64 sum rounds every partial sum to
// 2^-53 of itself: a tile's largest entry is at most 22 times its r.m.s.
//
// Exponents are stored biased as in an FP64 number (E + 1023), at least
// kExpMin; a tile with an infinity or NaN stores kExpBad, and every sum it
// enters becomes NaN.  Entries below 2^-60 of the tile's largest count as 0.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace bah {

constexpr int kTileU = 8;                 // entries per lane of a tile
constexpr int kTile = 32 * kTileU;        // entries of a tile: entry u * 32 + lane
constexpr int kExpBad = 0x800;            // exponent of a tile that holds a non-finite entry
constexpr int kExpMin = 64;

inline __host__ __device__ size_t tiles_of(size_t n) { return (n + kTile - 1) / kTile; }

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
// re.h, re.l, im.h, im.l
__device__ __forceinline__ int4 limbs2(double2 z, int eb) {
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

}  // namespace bah
