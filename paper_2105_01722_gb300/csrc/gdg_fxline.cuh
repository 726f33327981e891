// Element transforms of the modal route on the integer pipe (gdg_fx.cuh): a
// thread takes a line of N1 entries in registers, its limbs times a table's
// limbs, which the launch carries as a parameter (constant operands of the
// multiply-adds: no shared-memory reads for them).
//
// Between the passes of a transform an entry is the 64-bit integer sum that a
// pass left in the element's tile; the next pass scales it by the element's
// largest one (`bits`, the OR of the magnitudes of all), so every pass works on
// 57 bits against the element's largest entry.  Three multiply-adds a product:
// the product of two low limbs, about half a unit of 2^-57 after a sum, is left
// out.  Error of a pass: about a unit of 2^-57 of the largest entry times the
// table's largest one, where an FP64 sum leaves 2^-53 of its partial sums.  With
// the tables to 58 bits (parity_modes) the round trip of random fields is off by
// 1.2e-16 to 1.1e-15 (2-norm; N = 3 to 9, p = 3 to 7, 2-D and 3-D), in FP64 by
// 6.8e-16 to 2.3e-15, and dV/dt of a polynomial by 0.2 to 1.0 times as much.
#pragma once

#include "gdg_fx.cuh"

// one table as integers a 2^(pe - 57): P = Psi^T M, row q at q NE, its first
// half (even rows first, then odd ones); or Psi, rows i < NE at i N1.  |a| <=
// 2^57 and the absolute sums of whole rows at most 8 2^57 (fx_line_table).
template <int N1, int DIM>
struct FxLines {
    int2 a[DIM][N1 * ((N1 + 1) / 2)];
    int pe[DIM];
};

namespace {

enum { FX_TO_MODES = 1, FX_TO_NODES = 2 };

// one pass's sum: hh 2^58 + mid 2^29 in units of 2^-57: over at most 8 (differences:
// limbs up to 2^30) or 16 products both stay below 2^62
struct FxPair {
    long long hh, mid;
    __device__ FxPair() : hh(0), mid(0) {}
    __device__ __forceinline__ void mad(int2 a, int h, int l) {
        hh += (long long)a.x * h;
        mid += (long long)a.x * l;
        mid += (long long)a.y * h;
    }
};
__device__ __forceinline__ long long fx_pair_value(long long hh, long long mid) {
    return hh + hh + ((mid + (1 << (FX_LIMB - 2))) >> (FX_LIMB - 1));
}

// limbs of X = Z 2^-5, |Z| < 2^62, the low one balanced; X is rounded to nearest, halves
// away from zero: entries of either sign are treated alike, and what is conserved
// does not drift from transform to transform
__device__ __forceinline__ void fx_limbs(long long Z, int &h, int &l) {
    Z += 16 + (Z >> 63);
    const int hi = (int)(Z >> 32);
    h = (hi + 2) >> 2;
    l = (int)__funnelshift_r((unsigned)Z, (unsigned)hi, 2) >> 3;
}
// ... of the double v in units of 2^-57 2^(emax - 1022)
__device__ __forceinline__ void fx_limbs(double v, int emax, int &h, int &l) {
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
    const long long m = (long long)((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << 9;
    const long long Z = e == 0 ? 0 : m >> min(emax - e, 63);
    fx_limbs(hi < 0 ? -Z : Z, h, l);
}

// magnitude bits of Y, to be OR-ed over an element
__device__ __forceinline__ int fx_bits(long long Y) {
    const int hi = (int)(Y >> 32);
    return hi ^ (hi >> 31);
}
// bits an element's sums need at most (its magnitudes' upper words OR-ed)
__device__ __forceinline__ int fx_length(int bits) { return bits ? 64 - __clz(bits) : 32; }

// Y 2^q as a double; `plain`: 2^q Y is normal for every 1 <= |Y| < 2^63
__device__ __forceinline__ bool fx_plain(int q) { return q > -1022 && q < 960; }
__device__ __forceinline__ double fx_double(long long Y, int q, bool plain, bool nan) {
    const double d = (double)Y;
    if (plain) {
        const int hi = __double2hiint(d);
        return __hiloint2double(hi ? hi + (q << 20) : 0, __double2loint(d));   // Y != 0: hi != 0
    }
    return nan ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(d, q);
}

// One line through a table: emit(i, sum i as an integer).  FX_TO_MODES: rows q >
// 0 sum to zero (M 1 is the constant mode) and are applied to differences from a
// middle node, exact here: the rounding of the table then meets the variation
// along the line, not the values, which the high modes (times lambda
// afterwards) would show.  FX_TO_NODES: a pair of nodes from its even and odd
// parts.
template <int N1, int KIND, typename EMIT>
__device__ __forceinline__ void fx_line(const int2 *A, const int (&xh)[N1], const int (&xl)[N1], EMIT emit) {
    constexpr int NE = (N1 + 1) / 2, H = N1 / 2;
    if (KIND == FX_TO_MODES) {
        const int rh = xh[NE - 1], rl = xl[NE - 1];
        int sh[H], sl[H], dh[H], dl[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            sh[i] = xh[i] + xh[N1 - 1 - i];
            sl[i] = xl[i] + xl[N1 - 1 - i];
            dh[i] = xh[i] - xh[N1 - 1 - i];
            dl[i] = xl[i] - xl[N1 - 1 - i];
        }
        FxPair c;   // the constant mode
#pragma unroll
        for (int i = 0; i < H; ++i) c.mad(A[i], sh[i], sl[i]);
        if (N1 & 1) c.mad(A[H], rh, rl);
        emit(0, fx_pair_value(c.hh, c.mid));
#pragma unroll
        for (int i = 0; i < H; ++i) {
            sh[i] -= 2 * rh;
            sl[i] -= 2 * rl;
        }
#pragma unroll
        for (int q = 1; q < N1; ++q) {
            FxPair s;
#pragma unroll
            for (int i = 0; i < H; ++i) s.mad(A[q * NE + i], q < NE ? sh[i] : dh[i], q < NE ? sl[i] : dl[i]);
            emit(q, fx_pair_value(s.hh, s.mid));
        }
    } else {
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            FxPair ev, od;
#pragma unroll
            for (int k = 0; k < NE; ++k) ev.mad(A[i * N1 + k], xh[k], xl[k]);
            if (i < H) {
#pragma unroll
                for (int k = NE; k < N1; ++k) od.mad(A[i * N1 + k], xh[k], xl[k]);
                emit(N1 - 1 - i, fx_pair_value(ev.hh - od.hh, ev.mid - od.mid));
            }
            emit(i, fx_pair_value(ev.hh + od.hh, ev.mid + od.mid));
        }
    }
}

}  // namespace
