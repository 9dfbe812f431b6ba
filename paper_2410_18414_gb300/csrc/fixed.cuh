// Fixed-point arithmetic of the FP64 path's particle kernels: 128-bit sums, shape weights,
// gather fields.  GB300 issues 2 FP64 operations per clock and SM (0.6 T/s measured) but 32
// 32x32+64-bit multiply-adds (8.9 T/s measured).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "common.cuh"
#include "gpic_internal.h"

namespace gpic {

// hi 2^64 + lo (two's complement over 128 bits) times unscale, rounded to FP64: the
// magnitude is exact below 2^64 before its one rounding, and rounded twice above.
__device__ __forceinline__ double fix128_value(long long hi, unsigned long long lo,
                                               double unscale) {
    const bool neg = hi < 0;
    if (neg) {
        lo = ~lo + 1ull;
        hi = ~hi + (lo == 0ull ? 1ll : 0ll);
    }
    const double m = fma((double)hi, 18446744073709551616.0, (double)lo);
    return (neg ? -m : m) * unscale;
}

// Fixed-point gather fields (FP64 path): `top` is the high word of the largest |f| of a mesh row,
// which gives the row's exponent e with |f| < 2^e (bounded below so that the scales stay
// finite; above 1024 for a row with a value that is not finite, whose gathers are NaN).
__device__ __forceinline__ int row_exponent(unsigned top) {
    return top >= 0x7ff00000u ? 2048 : max((int)(top >> 20) - 1022, -900);
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }
// v in [-2^61, 2^61] as (v.x 2^31 + v.y), |v.y| <= 2^30
__device__ __forceinline__ int2 limbs(long long v) {
    const int lo = (int)((unsigned)v << 1) >> 1;
    return make_int2((int)((v - lo) >> 31), lo);
}
// f 2^(60 - e), rounded: a value keeps its 53 bits down to 2^-7 of its row's bound 2^e, and below
// that the rounding is 2^-61 of the bound
__device__ __forceinline__ int2 field_fix(double f, int e) {
    if (e > 1024) return make_int2(0, 0);
    return limbs(__double2ll_rn(rmul(f, pow2(60 - e))));
}

// FP64 shapes in fixed point: positions X = x/dx 2^sh (one FP64 multiply and conversion),
// weights in units of 2^-62 by 64-bit multiply-highs.  GB300 issues 2 FP64 operations per
// clock and SM but 32 32x32+64-bit multiply-adds, and the rounding of every step is 2^-62 of
// the largest weight, finer than FP64's.
constexpr long long kOne62 = 1ll << 62;
__device__ __forceinline__ long long mul62(long long a, long long b) {  // a, b in [0, 2^62]
    return (long long)__umul64hi((unsigned long long)a << 1, (unsigned long long)b << 1);
}
template <int P>
__device__ __forceinline__ int fix_weights(long long X, int sh, long long* w) {
    if (P % 2 == 0) X += 1ll << (sh - 1);
    const int i = (int)(X >> sh);
    // u: the offset within the cell (odd P) or from the midpoint before it (even P), in [0, 1)
    const long long u = (X & ((1ll << sh) - 1)) << (62 - sh), v = kOne62 - u;
    const long long u2 = mul62(u, u), v2 = mul62(v, v);
    if constexpr (P == 2) {  // ((1-u)^2/2, the rest, u^2/2)
        w[0] = v2 >> 1;
        w[2] = u2 >> 1;
        w[1] = kOne62 - w[0] - w[2];
        return i - 1;
    } else if constexpr (P == 3) {  // ((1-u)^3/6, 2/3 - u^2 + u^3/2, the rest, u^3/6)
        constexpr unsigned long long sixth = 0x2AAAAAAAAAAAAAABull;  // 2^64 / 6
        const long long u3 = mul62(u2, u), v3 = mul62(v2, v);
        w[0] = (long long)__umul64hi((unsigned long long)v3, sixth);
        w[3] = (long long)__umul64hi((unsigned long long)u3, sixth);
        w[1] = 0x2AAAAAAAAAAAAAABll - u2 + (u3 >> 1);  // 2/3 in units of 2^-62
        w[2] = kOne62 - w[0] - w[1] - w[3];
        return i - 1;
    } else {  // ((1-u)^4, 11 - 12u - 6u^2 + 12u^3 - 4u^4, the rest, 1 + 4u + 6u^2 + 4u^3 - 4u^4,
              //  u^4) / 24; the polynomials in units of 2^-58
        constexpr unsigned long long inv24 = 0x0AAAAAAAAAAAAAABull, two3 = 0xAAAAAAAAAAAAAAABull;
        const long long u3 = mul62(u2, u), u4 = mul62(u2, u2), v4 = mul62(v2, v2);
        const long long a = u >> 4, a2 = u2 >> 4, a3 = u3 >> 4, a4 = u4 >> 4, one = kOne62 >> 4;
        const long long n1 = 11 * one - 12 * a - 6 * a2 + 12 * a3 - 4 * a4;
        const long long n3 = one + 4 * (a + a3 - a4) + 6 * a2;
        w[0] = (long long)__umul64hi((unsigned long long)v4, inv24);
        w[1] = (long long)__umul64hi((unsigned long long)n1, two3);  // 16/24
        w[3] = (long long)__umul64hi((unsigned long long)n3, two3);
        w[4] = (long long)__umul64hi((unsigned long long)u4, inv24);
        w[2] = kOne62 - w[0] - w[1] - w[3] - w[4];
        return i - 2;
    }
}
// Fixed-point positions: x/dx 2^sh with nx, ny <= 2^(62 - sh).
struct FixGeom {
    double sx, sy;  // 2^sh / dx, 2^sh / dy
    int sh;
};
inline FixGeom fix_geom(const ParticleGeom& g) {
    int b = 0;
    while ((1 << b) < (g.nx > g.ny ? g.nx : g.ny)) ++b;
    const double s = (double)(1ull << (62 - b));
    return FixGeom{g.inv_dx * s, g.inv_dy * s, 62 - b};
}

// d w / d(x/dx) of fix_weights, in units of 2^-62 (signed; the derivatives add up to 0).
template <int P>
__device__ __forceinline__ void fix_dweights(long long X, int sh, long long* d) {
    if (P % 2 == 0) X += 1ll << (sh - 1);
    const long long u = (X & ((1ll << sh) - 1)) << (62 - sh), v = kOne62 - u;
    const long long u2 = mul62(u, u), v2 = mul62(v, v);
    if constexpr (P == 2) {  // (u - 1, 1 - 2u, u)
        d[0] = -v;
        d[1] = v - u;
        d[2] = u;
    } else if constexpr (P == 3) {  // (-(1-u)^2/2, 3u^2/2 - 2u, the rest, u^2/2)
        d[0] = -(v2 >> 1);
        d[3] = u2 >> 1;
        d[1] = u2 + (u2 >> 1) - 2 * u;
        d[2] = -(d[0] + d[1] + d[3]);
    } else {  // (-(1-u)^3, -3 - 3u + 9u^2 - 4u^3, the rest, 1 + 3u + 3u^2 - 4u^3, u^3) / 6; the
              // polynomials in units of 2^-60, times 4/6 = 1 - 1/3
        constexpr long long third = 0x5555555555555556ll;
        const long long u3 = mul62(u2, u), v3 = mul62(v2, v);
        const long long a = u >> 2, a2 = u2 >> 2, a3 = u3 >> 2, one = kOne62 >> 2;
        // (9 a2 alone passes 2^63 for u > 0.94; 5 a2 + 4 (a2 - a3) stays below 5.6 of the 8 units)
        const long long n0 = -(v3 >> 2), n1 = 5 * a2 + 4 * (a2 - a3) - 3 * (one + a);
        const long long n3 = one + 3 * (a + a2) - 4 * a3, n4 = a3;
        d[0] = n0 - __mul64hi(n0, third);
        d[1] = n1 - __mul64hi(n1, third);
        d[3] = n3 - __mul64hi(n3, third);
        d[4] = n4 - __mul64hi(n4, third);
        d[2] = -(d[0] + d[1] + d[3] + d[4]);
    }
}
// The FP64 deposit's products (RowFix128), each rounded to nearest with v and -v alike: +v and -v
// at one place cancel exactly and the errors of many particles do not add up on one side
// (rounded down, every node's current was half a quantum a contribution too small).
// t = v W_x in units of 2^-3 quanta from v in 2^-2 quanta (|v| <= 2^62): 2^62 2 3/4 < 2^63.
__device__ __forceinline__ long long deposit_row(long long v, long long w) {
    const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const unsigned __int128 t = (unsigned __int128)m * (unsigned long long)w;
    const long long r = (long long)(unsigned long long)((t + ((unsigned __int128)1 << 60)) >> 61);
    return v < 0 ? -r : r;
}
// x = t W_y in quanta.  The weight (units of 2^-62) comes made odd by deposit_col, so that t W_y
// is never halfway between two quanta for |t| < 2^63 (it would need t = 0 mod 2^64) and
// floor((floor(2 x) + 1) / 2) is the nearest for either sign.
__device__ __forceinline__ long long deposit_col(long long w) { return w | 1; }
__device__ __forceinline__ long long deposit_value(long long t, long long w) {
    return (__mul64hi(t, w) + 1) >> 1;
}
// a weight (or derivative) in units of 2^-62 as limbs in units of 2^-61
__device__ __forceinline__ int2 weight_limbs(long long w) { return limbs((w + 1) >> 1); }

// A sum of products of limbs in units of f: 2 h + m 2^-30, the product of the low limbs (at most
// half a unit a term) dropped.  Bounds for the two passes of a gather, with sum |w| <= 1 or, for
// derivatives, 2 (quadratic shapes) and |f| <= 2^60 or, derivatives gathered along the row, 2^61,
// never both doubled: |h| <= 2^60, |m| <= 1.5 2^62.
struct LimbSum {
    long long h = 0, m = 0;
    __device__ __forceinline__ void add(int2 w, int fh, int fl) {
        h += (long long)w.x * fh;
        m += (long long)w.x * fl;
        m += (long long)w.y * fh;
    }
    // rounded to nearest
    __device__ __forceinline__ long long value() const { return 2 * h + ((m + (1ll << 29)) >> 30); }
    // divided by 2^d, d >= 0, rounded to nearest: floor((floor(2 sum / 2^d) + 1) / 2)
    __device__ __forceinline__ long long shifted(int d) const {
        long long t = 4 * h + (m >> 29);
#ifdef __CUDA_ARCH__
        asm("shr.s64 %0, %0, %1;" : "+l"(t) : "r"(d));  // amounts above 63 leave the sign
#else
        t >>= std::min(d, 63);
#endif
        return (t + 1) >> 1;
    }
};

// v 2^(e - 60) rounded to nearest even, by integer operations (an int64 conversion and a
// multiplication would be two of the FP64 pipe's); NaN for the exponent of a row that is not
// finite.
__device__ __forceinline__ double fix_value(long long v, int e) {
    unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)m);
    m <<= lz & 63;  // the leading bit to bit 63
    unsigned long long q = m >> 11;
    const unsigned r = (unsigned)m & 0x7ffu;
    q += r + ((unsigned)q & 1u) > 0x400u ? 1u : 0u;
    // q's leading bit adds 1 to the exponent field (2 when the rounding carried into it)
    const int field = 1025 + e - lz;
    q += (unsigned long long)field << 52;
    if (v < 0) q |= 0x8000000000000000ull;
    if (v == 0) q = 0;
    if (e > 1024) q = 0x7ff8000000000000ull;
    return __longlong_as_double((long long)q);
}

}  // namespace gpic
