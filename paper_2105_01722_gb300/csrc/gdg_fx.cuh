// FP64-accurate dot products on the integer pipe.
//
// GB300 issues one FP64 warp instruction per SM every 16 cycles and one
// 32 x 32 + 64-bit integer multiply-add (IMAD.WIDE) every 1.06 (both measured
// with instruction chains, 4 to 32 warps per SM).  A product of two 58-bit
// integers in two 29-bit limbs each is four of the latter: 4.2 cycles where
// an FP64 FMA costs 16.  The element matrices of the variable-coefficient
// path are fixed after setup, so they are kept as such integers:
//
//   matrix   A_ij = 2^(d_i + d_j) a_ij 2^-57, d_i = half the exponent of A_ii:
//            for a symmetric positive (semi)definite A, |A_ij|^2 <= A_ii A_jj,
//            so |a_ij| <= 2^57 and no row or column is drowned by another;
//   vector   x_j 2^(d_j) = X_j 2^(E - 57), |X_j| <= 2^57, E from the largest
//            entry of the vector at hand (block floating point);
//   sums     of limb products, 2^56 each, over at most 100 terms: below 2^63,
//            exact and the same in any order.
//
// The rounding of a_ij and X_j (half a unit of 2^-57 of the largest) and, once a
// row, of the sum (half a unit of 2^-56) takes the place of the rounding of every
// partial sum in FP64, all of them to nearest: a sum cut off downwards would
// err to one side at every stage, and sums over the mesh that the method conserves
// would drift.  The error of a product with the element matrices and inverses, in
// the 2-norm against extended precision, is on average 0.15 to 0.85 of that of the
// FP64 sum for random and smooth vectors and pulses of a third of the element's
// width (N = 4 to 9, p = 1 to 7); entries far below the largest keep fewer bits than a
// double, so on pulses of a tenth of its width it is 0.3 to 1.1 of it on
// average, and up to 4 times it in one vector.
// A vector with an infinity or NaN gives NaN; entries below 2^-57 of the
// largest, and subnormal ones, count as zero.
#pragma once

#include <cuda_runtime.h>

namespace {

constexpr int FX_LIMB = 29;
constexpr int FX_ONE = 2 * FX_LIMB - 1;   // a full-scale integer is 2^57

// biased exponent of v (0 for zero and subnormals, 2047 for Inf and NaN)
__device__ __forceinline__ int fx_expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

__device__ __forceinline__ int2 fx_split(long long X) {
    const int lo = (int)((unsigned)X << (32 - FX_LIMB)) >> (32 - FX_LIMB);   // balanced low limb
    return make_int2((int)((X - lo) >> FX_LIMB), lo);
}

// v as an integer in units of 2^-57 2^(emax - 1022), rounded to nearest; emax
// >= the biased exponent of v plus `shift` (v counts as v 2^shift)
__device__ __forceinline__ long long fx_int(double v, int emax, int shift = 0) {
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << (FX_ONE - 52);
    const int d = emax - e - shift;   // the implicit one of v sits at bit 57 - d - 1
    unsigned long long s = e == 0 || d > 62 ? 0ull : m >> d;
    s = (s + 1) >> 1;
    return hi < 0 ? -(long long)s : (long long)s;
}

// 2^q (q any; 0 or Inf beyond the range of doubles)
__device__ __forceinline__ double fx_pow2(int q) {
    return q > -1023 ? (q < 1024 ? __hiloint2double((q + 1023) << 20, 0) : __hiloint2double(0x7ff00000, 0)) : 0.0;
}

// T 2^q with one conversion and one product where 2^q is a normal number
__device__ __forceinline__ double fx_scale(long long T, int q) {
    const double v = (double)T;
    return q > -1023 && q < 1024 ? v * fx_pow2(q) : scalbn(v, q);
}

// The sum of limb products, exact until top() or next() rounds it to nearest: m1
// starts at half a unit of the result.
struct FxSum {
    static constexpr int TOP = FX_LIMB - 1, NEXT = FX_LIMB - 2;
    long long hh, m1, m2, ll;
    __device__ explicit FxSum(int half = TOP) : hh(0), m1(1ll << half), m2(0), ll(0) {}
    __device__ __forceinline__ void mad(int2 a, int2 x) {
        hh += (long long)a.x * x.x;
        m1 += (long long)a.x * x.y;
        m2 += (long long)a.y * x.x;
        ll += (long long)a.y * x.y;
    }
    __device__ __forceinline__ void mad(int2 a, int xh, int xl) { mad(a, make_int2(xh, xl)); }
    // the sum in units of 2^58
    __device__ __forceinline__ long long top() const {
        return hh + (((m1 >> 1) + (m2 >> 1) + (ll >> (FX_LIMB + 1))) >> (FX_LIMB - 1));
    }
    // the sum (from FxSum(NEXT)) in units of 2^57, as the next limbs of a chain of contractions
    // whose matrix rows sum to at most 1 (|sum| <= 2^114, few terms: m1 + m2 fits)
    __device__ __forceinline__ int2 next() const {
        return fx_split(hh + hh + ((m1 + m2 + (ll >> FX_LIMB)) >> (FX_LIMB - 1)));
    }
};

// exponent q with sum = top() 2^q for a matrix in units of 2^-57 and a vector
// whose largest biased exponent is emax
__device__ __forceinline__ int fx_top_exp(int emax) { return emax - 1022 - 2 * FX_ONE + 2 * FX_LIMB; }

// Packed lower triangle of a symmetric NA x NA matrix, row by row, padded to
// a whole number of 16-byte copies.
__host__ __device__ constexpr int fx_tri_len(int na) { return (na * (na + 1) / 2 + 1) & ~1; }

}  // namespace
