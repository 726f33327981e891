// Device code of the constant-coefficient modal stage shared by the
// per-problem kernels (gdg_const.cu) and the batched kernels (gdg_batch.cu).
#pragma once

#include "gdg_checks.cuh"
#include "gdg_internal.h"

namespace {



// trace buffer index: 2-D [e][face 0..3 = xm,xp,ym,yp][field 0 = v, 1 = n.grad u][N1]
// (signed: on a partitioned mesh the ghost row below the first row has e < 0)
template <int N1>
__device__ __forceinline__ long long tix2(int e, int face, int fld, int i) {
    return (((long long)e * 4 + face) * 2 + fld) * N1 + i;
}
// 1-D: [e][face 0..1][field]
__device__ __forceinline__ size_t tix1(int e, int face, int fld) {
    return ((size_t)e * 2 + face) * 2 + fld;
}

// Fluxes of Section 2.2.1 in normal form (alpha = 1/2):
//   v* = (vi + vo)/2 - beta (di + do),  q* = (di - do)/2 - tau (vi - vo)
// returns g = v* - vi and c2 * q*.  Alternating flux (alpha = 1, sides by a
// fixed orientation: side 1 = the left / lower element): on the element's
// minus face (side = 0, it is side 2) v* = vo, q* = di; on its plus face
// (side = 1) v* = vi, q* = -do; on a Dirichlet side (bnd: vo, do are the
// mirror state) v* = 0, q* = di, which is the alpha = 1/2 formula there.
__device__ __forceinline__ void flux(double vi, double di, double vo, double dO, double beta,
                                     double tau, double c2, int alt, int side, bool bnd, double &g, double &q) {
    if (alt && !bnd) {
        g = side == 0 ? vo - vi : 0.0;
        q = c2 * (side == 0 ? di : -dO);
        return;
    }
    g = 0.5 * (vo - vi) - beta * (di + dO);
    q = c2 * (0.5 * (di - dO) - tau * (vi - vo));
}

// The same fluxes doubled, without c^2 (g2 = 2 (v* - vi), q2 = 2 q*), as the
// parity stage bodies use them.
__device__ __forceinline__ void flux2(double vi, double di, double vo, double dO, double b2, double t2,
                                      int alt, int side, bool bnd, double &g2, double &q2) {
    const double d1 = vo - vi;
    if (alt && !bnd) {
        g2 = side == 0 ? 2.0 * d1 : 0.0;
        q2 = side == 0 ? 2.0 * di : -2.0 * dO;
        return;
    }
    g2 = fma(-b2, di + dO, d1);
    q2 = fma(t2, d1, di - dO);
}

// y = A x for one line of an element transform, A row-major in shared memory.
// KIND 0: any matrix.  The modes are even or odd under r -> 1-r where the
// basis has that symmetry (parity contexts; the even ones, NE = ceil(N1/2),
// first), so a line splits in node pairs and each output is a sum of about
// N1/2 products: 41 FMAs and 8 additions instead of 81 at N1 = 9.
// KIND 3: nodes to modes by Psi^T, row q even or odd in i, from the plain sums
// and differences of the pairs.  KIND 2: modes to nodes (column k even or odd in
// i), a pair from its even and odd parts.
// emit(i, y[i]) as each is formed: a store there keeps the loads of the
// matrix from being moved up into a hundred registers.
template <int N1, int KIND, typename EMIT>
__device__ __forceinline__ void line_transform(const double *A, const double (&x)[N1], EMIT emit) {
    constexpr int NE = (N1 + 1) / 2, H = N1 / 2;   // H pairs, and the middle node when N1 is odd
    if (KIND == 3) {
        double sm[NE], df[H > 0 ? H : 1];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            sm[i] = x[i] + x[N1 - 1 - i];
            df[i] = x[i] - x[N1 - 1 - i];
        }
        if (N1 & 1) sm[NE - 1] = x[H];
#pragma unroll
        for (int q = 0; q < N1; ++q) {
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < (q < NE ? NE : H); ++i) s = fma(A[q * N1 + i], q < NE ? sm[i] : df[i < H ? i : 0], s);
            emit(q, s);
        }
    } else if (KIND == 2) {
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            double ev = 0.0, od = 0.0;
#pragma unroll
            for (int k = 0; k < NE; ++k) ev = fma(A[i * N1 + k], x[k], ev);
            if (i < H) {
#pragma unroll
                for (int k = NE; k < N1; ++k) od = fma(A[i * N1 + k], x[k], od);
                emit(N1 - 1 - i, ev - od);
            }
            emit(i, i < H ? ev + od : ev);
        }
    } else {
#pragma unroll
        for (int q = 0; q < N1; ++q) {
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < N1; ++i) s = fma(A[q * N1 + i], x[i], s);
            emit(q, s);
        }
    }
}

// the two face traces of a modal line (values: L, R = eL, eR; outward slopes:
// gL, gR), its entries added in any order
template <int N1, bool PAR>
struct LineTraces {
    const double *L, *R;
    double a = 0.0, b = 0.0;   // parity: even and odd parts; else left and right
    __device__ LineTraces(const double *L_, const double *R_) : L(L_), R(R_) {}
    __device__ __forceinline__ void add(int k, double y) {
        if (PAR) {
            if (k < (N1 + 1) / 2) a = fma(L[k], y, a);
            else b = fma(L[k], y, b);
        } else {
            a = fma(L[k], y, a);
            b = fma(R[k], y, b);
        }
    }
    __device__ __forceinline__ double left() const { return PAR ? a + b : a; }
    __device__ __forceinline__ double right() const { return PAR ? a - b : b; }
};

// One modal entry of a stage (see stage2p_body): the new (u, v) from the stage
// input (Yu, Yv) and y_n (Nu, Nv), or k itself (M_RHS).  L0, P1, P2, cey, xq
// carry the stage's factor sc unless M_RHS.
template <int MODE>
__device__ __forceinline__ void stage_entry(double sc, double L0, double P1, double P2, double cex, double cey,
                                            double xg, double xq, double FG, double FQ, double Yu, double Yv, double Nu,
                                            double Nv, double &Ru, double &Rv) {
    if (MODE == M_RHS) {
        Ru = fma(P1, xg, fma(P2, FG, Yv));
        Rv = fma(L0, Yu, fma(cex, xq, cey * FQ));
    } else {
        Ru = fma(sc, Yv, fma(P1, xg, fma(P2, FG, Nu)));
        Rv = fma(L0, Yu, fma(cex, xq, fma(cey, FQ, Nv)));
    }
}

// Body of the parity stage kernel for element tile `etile` (blockDim.x / N1
// elements per block).  Parity version of the generic stage: the GD element is symmetric under r -> 1-r,
// so every modified-basis vector is even or odd: Psi[N-i][k] = s_k Psi[i][k].
// With the NE = (N1+1)/2 even modes stored first, eR = s eL and gR = s gL:
// both face traces of a line come from one even/odd split dot, and each
// lift is one FMA per entry.  Fluxes carry a factor 2 (g2 = 2(v* - v_in),
// q2 = 2 q*) that is folded into the lift vectors hgL = gL/2, ceL = c^2 eL/2.
// ALT: the flux kind as a compile-time constant (1 alternating, 0 central or
// upwind; must equal mp.alt), so the per-face choice costs nothing.
// The u lifts enter only through k_u = V + Lambda^+ r_u, so they are folded
// with the diagonal solve: P1[l][k] = hgL_x[k] / lambda[l][k] and
// P2[l][k] = hgL_y[l] / lambda[l][k] (lam2 rows 2 and 3; 0 on the constant
// mode), two FMAs per entry.
// RK4 in nested form: the semi-discretisation is linear and autonomous, so one
// classic RK4 step is the Taylor polynomial of degree 4, and with L y = k(y)
//   w1 = y + dt/4 L y,  w2 = y + dt/3 L w1,  w3 = y + dt/2 L w2,  y' = y + dt L w3
// gives it without an accumulator: a stage reads its input and y_n and writes
// its output, three passes over the state instead of five, and keeps 4 N1
// doubles of a line instead of 6 N1.  The stage's factor sc = dt/4 .. dt is
// folded into its copy of the tables (lam2 rows 0, 2, 3) and the fluxes of v,
// so an entry takes 6 FMAs for both fields (10 operations with k formed first).
template <int N1, int MODE, int ALT>
__device__ __forceinline__ void stage2p_body(const ModalParams &mp, const StageBufs &b, double sc, int etile,
                                             double *smem) {
    constexpr int NE = (N1 + 1) / 2;
    const int epb = blockDim.x / N1;
    const int t = threadIdx.x;
    const int le = t / N1, l = t - le * N1;
    const int e = etile * epb + le;
    const bool valid = le < epb && e < mp.ne;
    double *fy = smem + le * (4 * N1);   // per column: GA, GB, QA, QB of the y faces
    double *tile = smem + epb * 4 * N1 + le * (2 * N1 * (N1 + 1));
    const int nx = mp.nx, ny = mp.ny;
    const int ex = valid ? e % nx : 0, ey = valid ? e / nx : 0;
    const double b2 = mp.beta2, t2 = mp.tau2;
    const size_t row = ((size_t)(valid ? e : 0) * N1 + l) * N1;

    // issue every row load of this stage before the barrier so their latency
    // overlaps the flux work (a few warps per SM only at small element counts)
    double Ru[N1], Rv[N1], Nu[N1], Nv[N1];
    if (valid) {
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            Ru[k] = b.yU[row + k];
            Rv[k] = b.yV[row + k];
            if (MODE == M_S23) {
                Nu[k] = b.nU[row + k];
                Nv[k] = b.nV[row + k];
            }
        }
    }

    double GA = 0, GB = 0, QA = 0, QB = 0;
    if (valid) {
        const double *T = b.trin;
        double vi, di, vo, dO, g2m, q2m, g2p, q2p;
        int en, f;
        bool bnd;
        // x faces, transverse mode l
        vi = T[tix2<N1>(e, 0, 0, l)]; di = T[tix2<N1>(e, 0, 1, l)];
        en = ex - 1;
        if (en < 0 && mp.per_x) en += nx;
        bnd = en < 0;
        if (!bnd) { f = ey * nx + en; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2P_NB + 0); vo = T[tix2<N1>(f, 1, 0, l)]; dO = T[tix2<N1>(f, 1, 1, l)]; }
        else { vo = -vi; dO = -di; }
        flux2(vi, di, vo, dO, b2, t2, ALT, 0, bnd, g2m, q2m);
        vi = T[tix2<N1>(e, 1, 0, l)]; di = T[tix2<N1>(e, 1, 1, l)];
        en = ex + 1;
        if (en >= nx && mp.per_x) en -= nx;
        bnd = en >= nx;
        if (!bnd) { f = ey * nx + en; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2P_NB + 1); vo = T[tix2<N1>(f, 0, 0, l)]; dO = T[tix2<N1>(f, 0, 1, l)]; }
        else { vo = -vi; dO = -di; }
        flux2(vi, di, vo, dO, b2, t2, ALT, 1, bnd, g2p, q2p);
        GA = g2m + g2p; GB = g2m - g2p; QA = q2m + q2p; QB = q2m - q2p;
        // y faces, transverse mode k = l (on a halo side the neighbour row's
        // traces sit in the ghost row en = -1 or en = ny of the trace buffer)
        vi = T[tix2<N1>(e, 2, 0, l)]; di = T[tix2<N1>(e, 2, 1, l)];
        en = ey - 1;
        if (en < 0 && mp.per_y) en += ny;
        bnd = en < 0 && !mp.halo_lo;
        if (!bnd) { f = en * nx + ex; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2P_NB + 2); vo = T[tix2<N1>(f, 3, 0, l)]; dO = T[tix2<N1>(f, 3, 1, l)]; }
        else { vo = -vi; dO = -di; }
        flux2(vi, di, vo, dO, b2, t2, ALT, 0, bnd, g2m, q2m);
        vi = T[tix2<N1>(e, 3, 0, l)]; di = T[tix2<N1>(e, 3, 1, l)];
        en = ey + 1;
        if (en >= ny && mp.per_y) en -= ny;
        bnd = en >= ny && !mp.halo_hi;
        if (!bnd) { f = en * nx + ex; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2P_NB + 3); vo = T[tix2<N1>(f, 2, 0, l)]; dO = T[tix2<N1>(f, 2, 1, l)]; }
        else { vo = -vi; dO = -di; }
        flux2(vi, di, vo, dO, b2, t2, ALT, 1, bnd, g2p, q2p);
        fy[l] = g2m + g2p; fy[N1 + l] = g2m - g2p;
        fy[2 * N1 + l] = q2m + q2p; fy[3 * N1 + l] = q2m - q2p;
    }
    __syncthreads();

    if (valid) {
        const double *L0 = b.lam2 + l * N1;
        const double *P1 = b.lam2 + 2 * N1 * N1 + l * N1, *P2 = b.lam2 + 3 * N1 * N1 + l * N1;
        const double cey = MODE == M_RHS ? mp.d[1].ceL[l] : sc * mp.d[1].ceL[l];
        if (MODE != M_RHS) { QA *= sc; QB *= sc; }
        const double *FG = fy + (l < NE ? 0 : N1);
        const double *FQ = fy + (l < NE ? 2 * N1 : 3 * N1);
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            const double Yu = Ru[k], Yv = Rv[k];
            const double xg = k < NE ? GA : GB, xq = k < NE ? QA : QB;
            stage_entry<MODE>(sc, L0[k], P1[k], P2[k], mp.d[0].ceL[k], cey, xg, xq, FG[k], FQ[k], Yu, Yv,
                              MODE == M_S1 ? Yu : Nu[k], MODE == M_S1 ? Yv : Nv[k], Ru[k], Rv[k]);
        }
#pragma unroll
        for (int k = 0; k < N1; ++k) { b.oU[row + k] = Ru[k]; b.oV[row + k] = Rv[k]; }
    }
    if (MODE == M_RHS) return;

    if (valid) {
        double ve = 0, vo_ = 0, de = 0, do_ = 0;
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            if (k < NE) { ve = fma(mp.d[0].eL[k], Rv[k], ve); de = fma(mp.d[0].gL[k], Ru[k], de); }
            else { vo_ = fma(mp.d[0].eL[k], Rv[k], vo_); do_ = fma(mp.d[0].gL[k], Ru[k], do_); }
            tile[l * (N1 + 1) + k] = Ru[k];
            tile[N1 * (N1 + 1) + l * (N1 + 1) + k] = Rv[k];
        }
        b.trout[tix2<N1>(e, 0, 0, l)] = ve + vo_;
        b.trout[tix2<N1>(e, 0, 1, l)] = de + do_;
        b.trout[tix2<N1>(e, 1, 0, l)] = ve - vo_;
        b.trout[tix2<N1>(e, 1, 1, l)] = de - do_;
    }
    __syncthreads();
    if (valid) {
        const int k = l;
        double ve = 0, vo_ = 0, de = 0, do_ = 0;
#pragma unroll
        for (int j = 0; j < N1; ++j) {
            const double u = tile[j * (N1 + 1) + k], v = tile[N1 * (N1 + 1) + j * (N1 + 1) + k];
            if (j < NE) { ve = fma(mp.d[1].eL[j], v, ve); de = fma(mp.d[1].gL[j], u, de); }
            else { vo_ = fma(mp.d[1].eL[j], v, vo_); do_ = fma(mp.d[1].gL[j], u, do_); }
        }
        b.trout[tix2<N1>(e, 2, 0, k)] = ve + vo_;
        b.trout[tix2<N1>(e, 2, 1, k)] = de + do_;
        b.trout[tix2<N1>(e, 3, 0, k)] = ve - vo_;
        b.trout[tix2<N1>(e, 3, 1, k)] = de - do_;
    }
}

// Half-line variant of stage2p_body: two threads per transverse line, lane
// pair (2m, 2m+1), the even one (h = 0) owning the NE even modes k < NE and
// the odd one (h = 1) the odd modes k >= NE.  Every floating-point operation
// is the one stage2p_body performs, in the same order, so the two bodies give
// bit-identical results; a pair swaps face fluxes and trace partial sums by
// one shuffle.  Twice the threads and half the registers per element: more
// warps per SM to hide FP64 and shared-memory latency on small meshes.
// blockDim.x = epb * 2 * N1 (even, so a pair never straddles a warp).
__device__ __forceinline__ unsigned pair_mask() {
    const int lanes = min(32, (int)blockDim.x - (int)(threadIdx.x & ~31u));
    return lanes >= 32 ? 0xffffffffu : ((1u << lanes) - 1u);
}

// LEAN: y_n is read where the update uses it instead of with the stage input
// (same operations and results; 20 fewer live registers, for kernels held to a
// low register count).
template <int N1, int MODE, bool LEAN = false>
__device__ __forceinline__ void stage2h_body(const ModalParams &mp, const StageBufs &b, double sc, int etile,
                                             double *smem) {
    constexpr int NE = (N1 + 1) / 2;   // even modes; the odd half has N1 - NE <= NE entries
    const int epb = blockDim.x / (2 * N1);
    const int t = threadIdx.x;
    const int le = t / (2 * N1), rr = t - le * (2 * N1);
    const int l = rr >> 1, h = rr & 1;
    const int k0 = h ? NE : 0, nk = h ? N1 - NE : NE;
    const int e = etile * epb + le;
    const bool valid = le < epb && e < mp.ne;
    const unsigned mask = pair_mask();
    double *fy = smem + (le < epb ? le : 0) * (4 * N1);
    double *tile = smem + epb * 4 * N1 + (le < epb ? le : 0) * (2 * N1 * (N1 + 1));
    const int nx = mp.nx, ny = mp.ny;
    const int ex = valid ? e % nx : 0, ey = valid ? e / nx : 0;
    const double b2 = mp.beta2, t2 = mp.tau2;
    const size_t row = ((size_t)(valid ? e : 0) * N1 + l) * N1 + k0;

    double Ru[NE], Rv[NE], Nu[NE], Nv[NE];
    if (valid) {
#pragma unroll
        for (int kk = 0; kk < NE; ++kk) {
            if (kk < nk) {
                Ru[kk] = b.yU[row + kk];
                Rv[kk] = b.yV[row + kk];
                if (!LEAN && MODE == M_S23) {
                    Nu[kk] = b.nU[row + kk];
                    Nv[kk] = b.nV[row + kk];
                }
            }
        }
    }

    // fluxes: h = 0 the minus face, h = 1 the plus face of each direction
    double gx = 0, qx = 0, gy = 0, qy = 0;
    if (valid) {
        const double *T = b.trin;
        double vi, di, vo, dO;
        int en, f;
        bool bnd;
        if (h == 0) {   // x-, transverse mode l
            vi = T[tix2<N1>(e, 0, 0, l)]; di = T[tix2<N1>(e, 0, 1, l)];
            en = ex - 1;
            if (en < 0 && mp.per_x) en += nx;
            bnd = en < 0;
            if (!bnd) { f = ey * nx + en; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2H_NB + 0); vo = T[tix2<N1>(f, 1, 0, l)]; dO = T[tix2<N1>(f, 1, 1, l)]; }
            else { vo = -vi; dO = -di; }
        } else {        // x+
            vi = T[tix2<N1>(e, 1, 0, l)]; di = T[tix2<N1>(e, 1, 1, l)];
            en = ex + 1;
            if (en >= nx && mp.per_x) en -= nx;
            bnd = en >= nx;
            if (!bnd) { f = ey * nx + en; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2H_NB + 1); vo = T[tix2<N1>(f, 0, 0, l)]; dO = T[tix2<N1>(f, 0, 1, l)]; }
            else { vo = -vi; dO = -di; }
        }
        flux2(vi, di, vo, dO, b2, t2, mp.alt, h, bnd, gx, qx);
        if (h == 0) {   // y-, transverse mode l
            vi = T[tix2<N1>(e, 2, 0, l)]; di = T[tix2<N1>(e, 2, 1, l)];
            en = ey - 1;
            if (en < 0 && mp.per_y) en += ny;
            bnd = en < 0;
            if (!bnd) { f = en * nx + ex; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2H_NB + 2); vo = T[tix2<N1>(f, 3, 0, l)]; dO = T[tix2<N1>(f, 3, 1, l)]; }
            else { vo = -vi; dO = -di; }
        } else {        // y+
            vi = T[tix2<N1>(e, 3, 0, l)]; di = T[tix2<N1>(e, 3, 1, l)];
            en = ey + 1;
            if (en >= ny && mp.per_y) en -= ny;
            bnd = en >= ny;
            if (!bnd) { f = en * nx + ex; GDG_CHECK_ELEM2(f, mp, GDG_SITE_STAGE2H_NB + 3); vo = T[tix2<N1>(f, 2, 0, l)]; dO = T[tix2<N1>(f, 2, 1, l)]; }
            else { vo = -vi; dO = -di; }
        }
        flux2(vi, di, vo, dO, b2, t2, mp.alt, h, bnd, gy, qy);
    }
    const double ogx = __shfl_xor_sync(mask, gx, 1), oqx = __shfl_xor_sync(mask, qx, 1);
    const double ogy = __shfl_xor_sync(mask, gy, 1), oqy = __shfl_xor_sync(mask, qy, 1);
    // g2m, g2p of each direction in the order of stage2p_body
    const double g2mx = h ? ogx : gx, g2px = h ? gx : ogx, q2mx = h ? oqx : qx, q2px = h ? qx : oqx;
    const double g2my = h ? ogy : gy, g2py = h ? gy : ogy, q2my = h ? oqy : qy, q2py = h ? qy : oqy;
    // x fluxes of this half's parity (GA, QA even; GB, QB odd)
    const double xg = h ? g2mx - g2px : g2mx + g2px;
    const double xq = h ? q2mx - q2px : q2mx + q2px;
    if (valid) {
        if (h == 0) { fy[l] = g2my + g2py; fy[2 * N1 + l] = q2my + q2py; }
        else { fy[N1 + l] = g2my - g2py; fy[3 * N1 + l] = q2my - q2py; }
    }
    __syncthreads();

    if (valid) {
        const double *L0 = b.lam2 + l * N1 + k0;
        const double *P1 = b.lam2 + 2 * N1 * N1 + l * N1 + k0, *P2 = b.lam2 + 3 * N1 * N1 + l * N1 + k0;
        const double cey = MODE == M_RHS ? mp.d[1].ceL[l] : sc * mp.d[1].ceL[l];
        const double sxq = MODE == M_RHS ? xq : xq * sc;
        const double *FG = fy + (l < NE ? 0 : N1) + k0;
        const double *FQ = fy + (l < NE ? 2 * N1 : 3 * N1) + k0;
        const double *cex = mp.d[0].ceL + k0;
#pragma unroll
        for (int kk = 0; kk < NE; ++kk) {
            if (kk < nk) {
                const double Yu = Ru[kk], Yv = Rv[kk];
                if (LEAN && MODE == M_S23) {
                    Nu[kk] = b.nU[row + kk];
                    Nv[kk] = b.nV[row + kk];
                }
                stage_entry<MODE>(sc, L0[kk], P1[kk], P2[kk], cex[kk], cey, xg, sxq, FG[kk], FQ[kk], Yu, Yv,
                                  MODE == M_S1 ? Yu : Nu[kk], MODE == M_S1 ? Yv : Nv[kk], Ru[kk], Rv[kk]);
            }
        }
#pragma unroll
        for (int kk = 0; kk < NE; ++kk)
            if (kk < nk) { b.oU[row + kk] = Ru[kk]; b.oV[row + kk] = Rv[kk]; }
    }
    if (MODE == M_RHS) return;

    // x-face traces: this half's partial dots (even: ve, de; odd: vo, do)
    double pv = 0, pd = 0;
    if (valid) {
        const double *eLx = mp.d[0].eL + k0, *gLx = mp.d[0].gL + k0;
#pragma unroll
        for (int kk = 0; kk < NE; ++kk) {
            if (kk < nk) {
                pv = fma(eLx[kk], Rv[kk], pv);
                pd = fma(gLx[kk], Ru[kk], pd);
                tile[l * (N1 + 1) + k0 + kk] = Ru[kk];
                tile[N1 * (N1 + 1) + l * (N1 + 1) + k0 + kk] = Rv[kk];
            }
        }
    }
    {
        const double opv = __shfl_xor_sync(mask, pv, 1), opd = __shfl_xor_sync(mask, pd, 1);
        const double ve = h ? opv : pv, de = h ? opd : pd, vo_ = h ? pv : opv, do_ = h ? pd : opd;
        if (valid) {
            if (h == 0) {
                b.trout[tix2<N1>(e, 0, 0, l)] = ve + vo_;
                b.trout[tix2<N1>(e, 0, 1, l)] = de + do_;
            } else {
                b.trout[tix2<N1>(e, 1, 0, l)] = ve - vo_;
                b.trout[tix2<N1>(e, 1, 1, l)] = de - do_;
            }
        }
    }
    __syncthreads();
    // y-face traces of column k = l: this half's rows j (even j < NE, odd j >= NE)
    pv = 0;
    pd = 0;
    if (valid) {
        const int k = l;
        const double *eLy = mp.d[1].eL + k0, *gLy = mp.d[1].gL + k0;
#pragma unroll
        for (int jj = 0; jj < NE; ++jj) {
            if (jj < nk) {
                const int j = k0 + jj;
                const double u = tile[j * (N1 + 1) + k], v = tile[N1 * (N1 + 1) + j * (N1 + 1) + k];
                pv = fma(eLy[jj], v, pv);
                pd = fma(gLy[jj], u, pd);
            }
        }
    }
    {
        const double opv = __shfl_xor_sync(mask, pv, 1), opd = __shfl_xor_sync(mask, pd, 1);
        const double ve = h ? opv : pv, de = h ? opd : pd, vo_ = h ? pv : opv, do_ = h ? pd : opd;
        if (valid) {
            const int k = l;
            if (h == 0) {
                b.trout[tix2<N1>(e, 2, 0, k)] = ve + vo_;
                b.trout[tix2<N1>(e, 2, 1, k)] = de + do_;
            } else {
                b.trout[tix2<N1>(e, 3, 0, k)] = ve - vo_;
                b.trout[tix2<N1>(e, 3, 1, k)] = de - do_;
            }
        }
    }
}

}  // namespace
