// 3-D elements on the modal route (the tensor-product construction of
// Sections 2.1.2 and 3 for d = 3; the paper states it and tests d <= 2):
// fused RK stage, traces, separable transforms and the energy partials of
// gdg_step / gdg_rhs / gdg_mass_solve / gdg_energy for dim = 3 contexts.
// Modal layout [e][m3][m2][m1] (m1 along x); one thread per x line (m3, m2)
// of an element, blockDim.x = epb * N1 * N1.
#include <algorithm>

#include "gdg_checks.cuh"
#include "gdg_fxline.cuh"
#include "gdg_internal.h"
#include "gdg_stage_const.cuh"

namespace {

constexpr int MAXB3 = 256;   // threads per block (epb elements x N1^2 lines)

// trace buffer index: [e][face 0..5 = xm,xp,ym,yp,zm,zp][field][N1*N1];
// transverse index: x faces m3*N1+m2, y faces m3*N1+m1, z faces m2*N1+m1
template <int N1>
__device__ __forceinline__ size_t tix3(int e, int face, int fld, int t) {
    return (((size_t)e * 6 + face) * 2 + fld) * (N1 * N1) + t;
}

// neighbour across face f of element (ex, ey, ez); -1 on a Dirichlet side
__device__ __forceinline__ int nbr3(const ModalParams &mp, int ex, int ey, int ez, int f) {
    int x = ex, y = ey, z = ez;
    switch (f) {
    case 0: x -= 1; if (x < 0) { if (!mp.per_x) return -1; x += mp.nx; } break;
    case 1: x += 1; if (x >= mp.nx) { if (!mp.per_x) return -1; x -= mp.nx; } break;
    case 2: y -= 1; if (y < 0) { if (!mp.per_y) return -1; y += mp.ny; } break;
    case 3: y += 1; if (y >= mp.ny) { if (!mp.per_y) return -1; y -= mp.ny; } break;
    case 4: z -= 1; if (z < 0) { if (!mp.per_z) return -1; z += mp.nz; } break;
    default: z += 1; if (z >= mp.nz) { if (!mp.per_z) return -1; z -= mp.nz; } break;
    }
    return (z * mp.ny + y) * mp.nx + x;
}

// traces on the y and z faces from the element tile (tU, tV in shared
// memory, [m3][m2][m1]); thread (a, c): y faces at (m3 = a, m1 = c), z faces
// at (m2 = a, m1 = c)
template <int N1>
__device__ __forceinline__ void traces3_yz(const ModalParams &mp, const double *tU, const double *tV, int e,
                                           int a, int c, double *trout) {
    double vL = 0, vR = 0, dL = 0, dR = 0;
#pragma unroll
    for (int m2 = 0; m2 < N1; ++m2) {
        const double u = tU[(a * N1 + m2) * N1 + c], v = tV[(a * N1 + m2) * N1 + c];
        vL += mp.d[1].eL[m2] * v;
        vR += mp.d[1].eR[m2] * v;
        dL += mp.d[1].gL[m2] * u;
        dR += mp.d[1].gR[m2] * u;
    }
    const int ty = a * N1 + c;
    trout[tix3<N1>(e, 2, 0, ty)] = vL;
    trout[tix3<N1>(e, 2, 1, ty)] = dL;
    trout[tix3<N1>(e, 3, 0, ty)] = vR;
    trout[tix3<N1>(e, 3, 1, ty)] = dR;
    vL = vR = dL = dR = 0;
#pragma unroll
    for (int m3 = 0; m3 < N1; ++m3) {
        const double u = tU[(m3 * N1 + a) * N1 + c], v = tV[(m3 * N1 + a) * N1 + c];
        vL += mp.d[2].eL[m3] * v;
        vR += mp.d[2].eR[m3] * v;
        dL += mp.d[2].gL[m3] * u;
        dR += mp.d[2].gR[m3] * u;
    }
    trout[tix3<N1>(e, 4, 0, ty)] = vL;
    trout[tix3<N1>(e, 4, 1, ty)] = dL;
    trout[tix3<N1>(e, 5, 0, ty)] = vR;
    trout[tix3<N1>(e, 5, 1, ty)] = dR;
}

template <int N1>
__host__ __device__ constexpr int smem3_doubles() { return 12 * N1 * N1 + 2 * N1 * N1 * N1; }

// elements per block of the 3-D kernels (epb3 on the host)
template <int N1>
__host__ __device__ constexpr int epb3c() { return MAXB3 / (N1 * N1) > 1 ? MAXB3 / (N1 * N1) : 1; }

template <int N1, int MODE>
__global__ void __launch_bounds__(MAXB3)
k_stage3(const __grid_constant__ ModalParams mp, const StageBufs b, double sc) {
    constexpr int NT = N1 * N1, NA = N1 * N1 * N1;
    extern __shared__ double smem[];
    const int epb = blockDim.x / NT;
    const int t = threadIdx.x;
    const int le = t / NT, r = t - le * NT;
    const int a = r / N1, c = r - (r / N1) * N1;
    const int e = blockIdx.x * epb + le;
    const bool valid = e < mp.ne;
    double *F = smem + le * smem3_doubles<N1>();      // [12][NT]: g, q of faces 0..5
    double *tU = F + 12 * NT, *tV = tU + NA;
    const int ex = valid ? e % mp.nx : 0, ey = valid ? (e / mp.nx) % mp.ny : 0, ez = valid ? e / (mp.nx * mp.ny) : 0;

    if (valid) {   // fluxes of the six faces at this thread's transverse mode pair
        const double *T = b.trin;
        const int tt = a * N1 + c;
#pragma unroll
        for (int f = 0; f < 6; ++f) {
            const double vi = T[tix3<N1>(e, f, 0, tt)], di = T[tix3<N1>(e, f, 1, tt)];
            int nb = nbr3(mp, ex, ey, ez, f);
            double vo, dO;
            if (nb >= 0) {
                GDG_CHECK_INDEX(nb, 0, mp.ne, GDG_SITE_STAGE3_NB + f, 0);
                vo = T[tix3<N1>(nb, f ^ 1, 0, tt)]; dO = T[tix3<N1>(nb, f ^ 1, 1, tt)];
            }
            else { vo = -vi; dO = -di; }
            double g, q;
            flux(vi, di, vo, dO, mp.beta, mp.tau, mp.c2, mp.alt, f & 1, nb < 0, g, q);
            F[(2 * f) * NT + tt] = g;
            F[(2 * f + 1) * NT + tt] = q;
        }
    }
    __syncthreads();

    double Ru[N1], Rv[N1];   // next stage input (or k) on line (m3 = a, m2 = c)
    if (valid) {
        const int line = a * N1 + c;
        const size_t row = ((size_t)e * NT + line) * N1;
        const double *L0 = b.lam2 + line * N1;
        const double *L1 = b.lam2 + NA + line * N1;
        const double Gxm = F[0 * NT + line], Qxm = F[1 * NT + line];
        const double Gxp = F[2 * NT + line], Qxp = F[3 * NT + line];
        const double gLy = mp.d[1].gL[c], gRy = mp.d[1].gR[c], eLy = mp.d[1].eL[c], eRy = mp.d[1].eR[c];
        const double gLz = mp.d[2].gL[a], gRz = mp.d[2].gR[a], eLz = mp.d[2].eL[a], eRz = mp.d[2].eR[a];
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            const int ty = a * N1 + k, tz = c * N1 + k;
            const double Yu = b.yU[row + k], Yv = b.yV[row + k];
            const double ru = mp.d[0].gL[k] * Gxm + mp.d[0].gR[k] * Gxp + gLy * F[4 * NT + ty] +
                              gRy * F[6 * NT + ty] + gLz * F[8 * NT + tz] + gRz * F[10 * NT + tz];
            const double rv = mp.d[0].eL[k] * Qxm + mp.d[0].eR[k] * Qxp + eLy * F[5 * NT + ty] +
                              eRy * F[7 * NT + ty] + eLz * F[9 * NT + tz] + eRz * F[11 * NT + tz];
            if (MODE == M_RHS) {
                Ru[k] = Yv + L1[k] * ru;
                Rv[k] = L0[k] * Yu + rv;
            } else {   // L0, L1 carry sc
                const double Nu = MODE == M_S1 ? Yu : b.nU[row + k], Nv = MODE == M_S1 ? Yv : b.nV[row + k];
                Ru[k] = fma(sc, Yv, fma(L1[k], ru, Nu));
                Rv[k] = fma(L0[k], Yu, fma(sc, rv, Nv));
            }
        }
#pragma unroll
        for (int k = 0; k < N1; ++k) { b.oU[row + k] = Ru[k]; b.oV[row + k] = Rv[k]; }
    }
    if (MODE == M_RHS) return;   // uniform across the block

    if (valid) {   // x faces from the line; the tile for the y and z faces
        const int line = a * N1 + c;
        double vL = 0, vR = 0, dL = 0, dR = 0;
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            vL += mp.d[0].eL[k] * Rv[k];
            vR += mp.d[0].eR[k] * Rv[k];
            dL += mp.d[0].gL[k] * Ru[k];
            dR += mp.d[0].gR[k] * Ru[k];
            tU[line * N1 + k] = Ru[k];
            tV[line * N1 + k] = Rv[k];
        }
        b.trout[tix3<N1>(e, 0, 0, line)] = vL;
        b.trout[tix3<N1>(e, 0, 1, line)] = dL;
        b.trout[tix3<N1>(e, 1, 0, line)] = vR;
        b.trout[tix3<N1>(e, 1, 1, line)] = dR;
    }
    __syncthreads();
    if (valid) traces3_yz<N1>(mp, tU, tV, e, a, c, b.trout);
}

// The u lifts are folded with the diagonal solve (rows 2-4 of lam2: hgL of
// each direction over lambda) and RK4 runs in nested form with the stage's
// factor folded into the tables, as in the 2-D parity kernels (stage2p_body).
// Parity version of k_stage3 (modes ordered even first in every direction:
// eR = s eL and gR = s gL, s = +1 for the NE = (N1+1)/2 even modes, -1 for
// the odd ones).  Phase 1 keeps, per direction and transverse mode pair, the
// sum and the difference of the doubled minus- and plus-face fluxes
// (flux2), so that each face pair lifts onto an entry with one product
// (hgL = gL/2, ceL = c^2 eL/2 carry the factors): 3 terms for r_u and 4 for
// r_v instead of 6 and 7.  Each trace pair comes from one dot split into its
// even and odd parts (left = even + odd, right = even - odd).
template <int N1>
__device__ __forceinline__ void traces3_yz_p(const ModalParams &mp, const double *tU, const double *tV, int e,
                                             int a, int c, double *trout) {
    constexpr int NE = (N1 + 1) / 2;
    double ve = 0, vo = 0, de = 0, dd = 0;
#pragma unroll
    for (int m2 = 0; m2 < N1; ++m2) {
        const double u = tU[(a * N1 + m2) * N1 + c], v = tV[(a * N1 + m2) * N1 + c];
        if (m2 < NE) { ve = fma(mp.d[1].eL[m2], v, ve); de = fma(mp.d[1].gL[m2], u, de); }
        else { vo = fma(mp.d[1].eL[m2], v, vo); dd = fma(mp.d[1].gL[m2], u, dd); }
    }
    const int ty = a * N1 + c;
    trout[tix3<N1>(e, 2, 0, ty)] = ve + vo;
    trout[tix3<N1>(e, 2, 1, ty)] = de + dd;
    trout[tix3<N1>(e, 3, 0, ty)] = ve - vo;
    trout[tix3<N1>(e, 3, 1, ty)] = de - dd;
    ve = vo = de = dd = 0;
#pragma unroll
    for (int m3 = 0; m3 < N1; ++m3) {
        const double u = tU[(m3 * N1 + a) * N1 + c], v = tV[(m3 * N1 + a) * N1 + c];
        if (m3 < NE) { ve = fma(mp.d[2].eL[m3], v, ve); de = fma(mp.d[2].gL[m3], u, de); }
        else { vo = fma(mp.d[2].eL[m3], v, vo); dd = fma(mp.d[2].gL[m3], u, dd); }
    }
    trout[tix3<N1>(e, 4, 0, ty)] = ve + vo;
    trout[tix3<N1>(e, 4, 1, ty)] = de + dd;
    trout[tix3<N1>(e, 5, 0, ty)] = ve - vo;
    trout[tix3<N1>(e, 5, 1, ty)] = de - dd;
}

template <int N1, int MODE, int ALT>
__global__ void __launch_bounds__(MAXB3, 3)
k_stage3p(const __grid_constant__ ModalParams mp, const StageBufs b, double sc) {
    constexpr int NT = N1 * N1, NA = N1 * N1 * N1, NE = (N1 + 1) / 2;
    constexpr int EPB = epb3c<N1>(), BD = EPB * NT;   // blockDim.x == BD (launch_stage3)
    extern __shared__ double smem[];
    const int t = threadIdx.x;
    const int le = t / NT, r = t - le * NT;
    const int a = r / N1, c = r - (r / N1) * N1;
    const int e = blockIdx.x * EPB + le;
    const bool valid = e < mp.ne;
    // per element [12][NT]: per direction d, at 4d: g-sum, g-difference,
    // q-sum, q-difference; then the tile tU, tV
    double *F = smem + le * smem3_doubles<N1>();
    double *tU = F + 12 * NT, *tV = tU + NA;
    double *ce = smem + EPB * smem3_doubles<N1>();   // [3][N1]: c^2 eL / 2 of x, y, z
    if (t < 3 * N1) {   // c^2 eL / 2 of x, y, z, times the stage's factor
        const double v = t < N1 ? mp.d[0].ceL[t] : t < 2 * N1 ? mp.d[1].ceL[t - N1] : mp.d[2].ceL[t - 2 * N1];
        ce[t] = MODE == M_RHS ? v : sc * v;
    }
    const int ex = valid ? e % mp.nx : 0, ey = valid ? (e / mp.nx) % mp.ny : 0, ez = valid ? e / (mp.nx * mp.ny) : 0;

    if (valid) {   // fluxes of the three face pairs at this thread's transverse mode pair
        const double *T = b.trin;
        const int tt = a * N1 + c;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double g2[2], q2[2];
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int f = 2 * d + side;
                const double vi = T[tix3<N1>(e, f, 0, tt)], di = T[tix3<N1>(e, f, 1, tt)];
                int nb = nbr3(mp, ex, ey, ez, f);
                double vo, dO;
                if (nb >= 0) {
                    GDG_CHECK_INDEX(nb, 0, mp.ne, GDG_SITE_STAGE3_NB + f, 0);
                    vo = T[tix3<N1>(nb, f ^ 1, 0, tt)]; dO = T[tix3<N1>(nb, f ^ 1, 1, tt)];
                }
                else { vo = -vi; dO = -di; }
                flux2(vi, di, vo, dO, mp.beta2, mp.tau2, ALT, side, nb < 0, g2[side], q2[side]);
            }
            F[(4 * d + 0) * NT + tt] = g2[0] + g2[1];
            F[(4 * d + 1) * NT + tt] = g2[0] - g2[1];
            F[(4 * d + 2) * NT + tt] = q2[0] + q2[1];
            F[(4 * d + 3) * NT + tt] = q2[0] - q2[1];
        }
    }
    __syncthreads();

    // The update runs over the block's EPB N1^3 consecutive entries in a
    // coalesced order: thread t takes entries t + s BD (s < N1), so every
    // warp load and store of the state covers 32 consecutive doubles (one x
    // line per thread would stride them by N1).  Entry q = (m3 N1 + m2) N1 +
    // m1 of element le2 finds its line's fluxes in that element's F; each
    // entry's arithmetic is the same sequence of operations in either order.
    // An entry's input and y_n are read before its output is stored, and no
    // other entry reads it: the output may be y_n itself (the last stage).
    const double *pyU = b.yU, *pyV = b.yV, *pnU = b.nU, *pnV = b.nV;
    const double *__restrict__ lam = b.lam2;
    const size_t base = (size_t)blockIdx.x * EPB * NA;
    const long long left = ((long long)mp.ne - (long long)blockIdx.x * EPB) * NA;   // entries of the block's elements
    constexpr int GRP = 3;   // entries whose loads are in flight together
#pragma unroll
    for (int s0 = 0; s0 < N1; s0 += GRP) {
    double Yr[2 * GRP], Nr[2 * GRP];
#pragma unroll
    for (int i = 0; i < GRP; ++i) {
        const bool in = s0 + i < N1 && t + (s0 + i) * BD < left;
        const size_t g = base + t + (s0 + i) * BD;
        Yr[i] = in ? pyU[g] : 0.0;
        Yr[GRP + i] = in ? pyV[g] : 0.0;
        if (MODE == M_S23) {
            Nr[i] = in ? pnU[g] : 0.0;
            Nr[GRP + i] = in ? pnV[g] : 0.0;
        }
    }
#pragma unroll
    for (int i = 0; i < GRP; ++i) {
        const int s = s0 + i;
        if (s >= N1) continue;
        const int idx = t + s * BD;
        const int le2 = idx / NA, q = idx - le2 * NA;
        if (blockIdx.x * EPB + le2 >= mp.ne) continue;
        const int line = q / N1, k = q - line * N1;
        const int m3 = line / N1, m2 = line - m3 * N1;
        double *F2 = smem + le2 * smem3_doubles<N1>();
        const size_t g = base + idx;
        const double Yu = Yr[i], Yv = Yr[GRP + i];
        const double xg = F2[(k < NE ? 0 : 1) * NT + line], xq = F2[(k < NE ? 2 : 3) * NT + line];
        const double FGy = F2[(4 + (m2 < NE ? 0 : 1)) * NT + m3 * N1 + k];   // at ty = m3 N1 + m1
        const double FQy = F2[(6 + (m2 < NE ? 0 : 1)) * NT + m3 * N1 + k];
        const double FGz = F2[(8 + (m3 < NE ? 0 : 1)) * NT + m2 * N1 + k];   // at tz = m2 N1 + m1
        const double FQz = F2[(10 + (m3 < NE ? 0 : 1)) * NT + m2 * N1 + k];
        // k_u = V + Lambda^+ r_u with the three rank-one lifts folded into
        // rows 2-4 of lam2 (hgL / lambda per direction): three FMAs
        if (MODE == M_RHS) {
            b.oU[g] = fma(lam[2 * NA + q], xg, fma(lam[3 * NA + q], FGy, fma(lam[4 * NA + q], FGz, Yv)));
            b.oV[g] = fma(lam[q], Yu, fma(ce[k], xq, fma(ce[N1 + m2], FQy, ce[2 * N1 + m3] * FQz)));
            continue;
        }
        const double Nu = MODE == M_S1 ? Yu : Nr[i], Nv = MODE == M_S1 ? Yv : Nr[GRP + i];
        const double Ru = fma(sc, Yv, fma(lam[2 * NA + q], xg, fma(lam[3 * NA + q], FGy, fma(lam[4 * NA + q], FGz, Nu))));
        const double Rv = fma(lam[q], Yu, fma(ce[k], xq, fma(ce[N1 + m2], FQy, fma(ce[2 * N1 + m3], FQz, Nv))));
        b.oU[g] = Ru;
        b.oV[g] = Rv;
        double *tU2 = F2 + 12 * NT;
        tU2[q] = Ru;
        tU2[NA + q] = Rv;
    }
    }
    if (MODE == M_RHS) return;   // uniform across the block
    __syncthreads();

    if (valid) {   // x faces from this thread's line; the tile for the y and z faces
        const int line = a * N1 + c;
        double ve = 0, vo = 0, de = 0, dd = 0;
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            const double u = tU[line * N1 + k], v = tV[line * N1 + k];
            if (k < NE) { ve = fma(mp.d[0].eL[k], v, ve); de = fma(mp.d[0].gL[k], u, de); }
            else { vo = fma(mp.d[0].eL[k], v, vo); dd = fma(mp.d[0].gL[k], u, dd); }
        }
        b.trout[tix3<N1>(e, 0, 0, line)] = ve + vo;
        b.trout[tix3<N1>(e, 0, 1, line)] = de + dd;
        b.trout[tix3<N1>(e, 1, 0, line)] = ve - vo;
        b.trout[tix3<N1>(e, 1, 1, line)] = de - dd;
        traces3_yz_p<N1>(mp, tU, tV, e, a, c, b.trout);
    }
}

// Nodes to modes or modes to nodes on the integer pipe (gdg_fxline.cuh), one
// line of an element a thread and pass; tr (modal output (U, V)): also its face
// traces.  32^3 elements, N1 = 9, both fields: 585 us in with the traces (FP64
// pipe 65 %, those sums and the conversions to doubles; issue 41 %) and 507 us
// out (issue 45 %), where FP64 lines by node pairs took 2115 and 1641.
template <int N1, int KIND>
__global__ void __launch_bounds__(MAXB3, 4)
k_fx3(const __grid_constant__ ModalParams mp, const __grid_constant__ FxLines<N1, 3> A, const double *in0,
      const double *in1, double *out0, double *out1, double *tr) {
    constexpr int NT = N1 * N1, NA = N1 * N1 * N1, EPB = epb3c<N1>();
    extern __shared__ long long fx_tiles[];
    __shared__ int slot[2][3][EPB];   // per field and element: largest exponent, bits after x, after y
    const int t = threadIdx.x, le = t / NT, r = t - le * NT, a = r / N1, c = r - a * N1;
    const int e = blockIdx.x * EPB + le;
    const bool valid = e < mp.ne;     // blockDim.x == EPB * NT
    const size_t base = (size_t)blockIdx.x * EPB * NA;           // the block's elements are consecutive
    const int count = min(EPB, mp.ne - (int)blockIdx.x * EPB) * NA;
    long long *T = fx_tiles + le * NA;
    for (int i = t; i < 6 * EPB; i += blockDim.x) (&slot[0][0][0])[i] = 0;
    const int nf = in1 ? 2 : 1;
#pragma unroll 1
    for (int f = 0; f < nf; ++f) {
        const double *in = f ? in1 : in0;
        double *out = f ? out1 : out0;
        for (int i = t; i < count; i += blockDim.x) fx_tiles[i] = __double_as_longlong(in[base + i]);
        __syncthreads();
        int h[N1], l[N1];
        // (1) x: thread = line (m3 = a, m2 = c)
        long long *line = T + r * N1;
        if (valid) {
            int m = 0;
#pragma unroll
            for (int i = 0; i < N1; ++i) m = max(m, fx_expo(__longlong_as_double(line[i])));
            atomicMax(&slot[f][0][le], m);
        }
        __syncthreads();
        const int emax = slot[f][0][le];
        if (valid) {
#pragma unroll
            for (int i = 0; i < N1; ++i) fx_limbs(__longlong_as_double(line[i]), emax, h[i], l[i]);
            int m = 0;
            fx_line<N1, KIND>(A.a[0], h, l, [&](int q, long long Y) { line[q] = Y; m |= fx_bits(Y); });
            atomicOr(&slot[f][1][le], m);
        }
        __syncthreads();
        // (2) y: thread = (m3 = a, m1 = c)
        const int len1 = fx_length(slot[f][1][le]);
        line = T + a * NT + c;
        if (valid) {
#pragma unroll
            for (int i = 0; i < N1; ++i) fx_limbs(line[i * N1] << (62 - len1), h[i], l[i]);
            int m = 0;
            fx_line<N1, KIND>(A.a[1], h, l, [&](int q, long long Y) { line[q * N1] = Y; m |= fx_bits(Y); });
            atomicOr(&slot[f][2][le], m);
        }
        __syncthreads();
        // (3) z: thread = (m2 = a, m1 = c)
        const int len2 = fx_length(slot[f][2][le]);
        line = T + r;
        if (valid) {
#pragma unroll
            for (int i = 0; i < N1; ++i) fx_limbs(line[i * NT] << (62 - len2), h[i], l[i]);
            const int q0 = (emax - 1022) + (A.pe[0] + len1 - 57) + (A.pe[1] + len2 - 57) + A.pe[2] - 57;
            const bool nan = emax == 0x7ff, plain = !nan && fx_plain(q0);
            LineTraces<N1, true> tz(f ? mp.d[2].eL : mp.d[2].gL, nullptr);
            fx_line<N1, KIND>(A.a[2], h, l, [&](int q, long long Y) {
                const double v = fx_double(Y, q0, plain, nan);
                line[q * NT] = __double_as_longlong(v);
                if (KIND == FX_TO_MODES && tr) tz.add(q, v);
            });
            if (KIND == FX_TO_MODES && tr) {
                tr[tix3<N1>(e, 4, 1 - f, r)] = tz.left();
                tr[tix3<N1>(e, 5, 1 - f, r)] = tz.right();
            }
        }
        __syncthreads();
        for (int i = t; i < count; i += blockDim.x) out[base + i] = __longlong_as_double(fx_tiles[i]);
        if (KIND == FX_TO_MODES && tr && valid) {   // the traces of the x and y faces
            LineTraces<N1, true> tx(f ? mp.d[0].eL : mp.d[0].gL, nullptr), ty(f ? mp.d[1].eL : mp.d[1].gL, nullptr);
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                tx.add(k, __longlong_as_double(T[r * N1 + k]));
                ty.add(k, __longlong_as_double(T[(a * N1 + k) * N1 + c]));
            }
            tr[tix3<N1>(e, 0, 1 - f, r)] = tx.left();
            tr[tix3<N1>(e, 1, 1 - f, r)] = tx.right();
            tr[tix3<N1>(e, 2, 1 - f, r)] = ty.left();
            tr[tix3<N1>(e, 3, 1 - f, r)] = ty.right();
        }
        if (f + 1 < nf) __syncthreads();
    }
}

// Separable element transform out = (Cz (x) Cy (x) Cx) diag(D) (Bz (x) By (x) Bx) in
// (C, D optional); per field, passes along x, y, z through an element tile.
// tr (modal output (U, V)): also its face traces.  KB: the kind of B
// (line_transform); C is of kind 2 when B is of kind 3.  Bound by the FP64
// pipe; with parity P and Psi alone go through k_fx3.
template <int N1, int KB>
__global__ void __launch_bounds__(MAXB3)
k_sep3(const __grid_constant__ ModalParams mp, const double *in0, const double *in1, double *out0, double *out1,
       const double *Bx, const double *By, const double *Bz, const double *D, const double *Cx, const double *Cy,
       const double *Cz, double *tr) {
    constexpr int NT = N1 * N1, NA = N1 * N1 * N1, KC = KB == 3 ? 2 : 0;
    extern __shared__ double smem[];
    double *sM = smem;            // Bx, By, Bz, Cx, Cy, Cz
    const int t = threadIdx.x;
    for (int i = t; i < NT; i += blockDim.x) {
        sM[i] = Bx[i];
        sM[NT + i] = By[i];
        sM[2 * NT + i] = Bz[i];
        if (Cx) { sM[3 * NT + i] = Cx[i]; sM[4 * NT + i] = Cy[i]; sM[5 * NT + i] = Cz[i]; }
    }
    const int epb = blockDim.x / NT;
    const int le = t / NT, r = t - le * NT;
    const int a = r / N1, c = r - (r / N1) * N1;
    const int e = blockIdx.x * epb + le;
    const bool valid = e < mp.ne;
    double *T = smem + 6 * NT + le * NA;
    const int nf = in1 ? 2 : 1;
    const size_t base = (size_t)blockIdx.x * epb * NA;           // the block's elements are consecutive
    const int count = min(epb, mp.ne - (int)blockIdx.x * epb) * NA;
    double *Tb = smem + 6 * NT;
    for (int f = 0; f < nf; ++f) {
        const double *in = f ? in1 : in0;
        double *out = f ? out1 : out0;
        double x[N1];
        // the tiles, coalesced (a line per thread would stride the loads by N1)
        for (int i = t; i < count; i += blockDim.x) Tb[i] = in[base + i];
        __syncthreads();
        // (1) x: thread = line (k = a, j = c)
        if (valid) {
#pragma unroll
            for (int i = 0; i < N1; ++i) x[i] = T[(a * N1 + c) * N1 + i];
            line_transform<N1, KB>(sM, x, [&](int q, double v) { T[(a * N1 + c) * N1 + q] = v; });
        }
        __syncthreads();
        // (2) y: thread = (k = a, i = c), column over j
        if (valid) {
#pragma unroll
            for (int j = 0; j < N1; ++j) x[j] = T[(a * N1 + j) * N1 + c];
            line_transform<N1, KB>(sM + NT, x, [&](int m, double v) { T[(a * N1 + m) * N1 + c] = v; });
        }
        __syncthreads();
        // (3) z: thread = (j = a, i = c), column over k; then D
        if (valid) {
#pragma unroll
            for (int k = 0; k < N1; ++k) x[k] = T[(k * N1 + a) * N1 + c];
            LineTraces<N1, false> tc(f ? mp.d[2].eL : mp.d[2].gL, f ? mp.d[2].eR : mp.d[2].gR);
            line_transform<N1, KB>(sM + 2 * NT, x, [&](int m, double v) {
                T[(m * N1 + a) * N1 + c] = D ? v * D[(m * N1 + a) * N1 + c] : v;
                if (tr) tc.add(m, v);
            });
            if (tr) {
                tr[tix3<N1>(e, 4, 1 - f, a * N1 + c)] = tc.left();
                tr[tix3<N1>(e, 5, 1 - f, a * N1 + c)] = tc.right();
            }
        }
        if (!Cx) {   // out, coalesced from the tiles, and the traces of the other faces
            __syncthreads();
            for (int i = t; i < count; i += blockDim.x) out[base + i] = Tb[i];
            if (tr && valid) {
                LineTraces<N1, false> tx(f ? mp.d[0].eL : mp.d[0].gL, f ? mp.d[0].eR : mp.d[0].gR);
                LineTraces<N1, false> ty(f ? mp.d[1].eL : mp.d[1].gL, f ? mp.d[1].eR : mp.d[1].gR);
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    tx.add(k, T[(a * N1 + c) * N1 + k]);
                    ty.add(k, T[(a * N1 + k) * N1 + c]);
                }
                tr[tix3<N1>(e, 0, 1 - f, a * N1 + c)] = tx.left();
                tr[tix3<N1>(e, 1, 1 - f, a * N1 + c)] = tx.right();
                tr[tix3<N1>(e, 2, 1 - f, a * N1 + c)] = ty.left();
                tr[tix3<N1>(e, 3, 1 - f, a * N1 + c)] = ty.right();
            }
            __syncthreads();
            continue;
        }
        // (4) Cz along z (same thread layout), in the thread's own column of the tile
        if (valid) {
#pragma unroll
            for (int k = 0; k < N1; ++k) x[k] = T[(k * N1 + a) * N1 + c];
            line_transform<N1, KC>(sM + 5 * NT, x, [&](int m, double v) { T[(m * N1 + a) * N1 + c] = v; });
        }
        __syncthreads();
        // (5) Cy along y: thread = (k = a, i = c)
        if (valid) {
#pragma unroll
            for (int j = 0; j < N1; ++j) x[j] = T[(a * N1 + j) * N1 + c];
            line_transform<N1, KC>(sM + 4 * NT, x, [&](int m, double v) { T[(a * N1 + m) * N1 + c] = v; });
        }
        __syncthreads();
        // (6) Cx along x: thread = line (k = a, j = c)
        if (valid) {
#pragma unroll
            for (int i = 0; i < N1; ++i) x[i] = T[(a * N1 + c) * N1 + i];
            line_transform<N1, KC>(sM + 3 * NT, x, [&](int q, double v) { T[(a * N1 + c) * N1 + q] = v; });
        }
        __syncthreads();
        for (int i = t; i < count; i += blockDim.x) out[base + i] = Tb[i];
        __syncthreads();
    }
}

// energy partials: sum over modes of (|Vbar|^2 - lam2 Ubar^2), lam2 = -c2 lambda
template <int N1>
__global__ void k_energy_partial3(int ne, const double *yU, const double *yV, const double *lam2, double *partial) {
    __shared__ double red[1024];
    const int t = threadIdx.x;
    constexpr int ents = N1 * N1 * N1;
    double s = 0.0;
    const long long total = (long long)ne * ents;
    for (long long i = (long long)blockIdx.x * blockDim.x + t; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int m = (int)(i % ents);
        const double u = yU[i], v = yV[i];
        s += v * v - lam2[m] * u * u;
    }
    red[t] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (t < w) red[t] += red[t + w];
        __syncthreads();
    }
    if (t == 0) partial[blockIdx.x] = red[0];
}

#define GDG_N1_CASES3(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10)

int epb3(int n1) { return std::max(1, MAXB3 / (n1 * n1)); }
// per element the fluxes and the tile; per block the parity kernel's c^2 eL / 2 table
size_t smem_stage3(int n1) { return ((size_t)epb3(n1) * (12 * n1 * n1 + 2 * n1 * n1 * n1) + 3 * n1) * sizeof(double); }
size_t smem_sep3(int n1) { return (size_t)(6 * n1 * n1 + epb3(n1) * n1 * n1 * n1) * sizeof(double); }

template <int N1>
void launch_stage3(int mode, const ModalParams &mp, const StageBufs &b, double sc, cudaStream_t s) {
    const int epb = epb3(N1);
    const dim3 grid((mp.ne + epb - 1) / epb), block(epb * N1 * N1);
    const size_t sm = smem_stage3(N1);
    if (mp.parity) {
        switch (mode) {
#define GDG_K3P(m) (mp.alt ? k_stage3p<N1, m, 1> : k_stage3p<N1, m, 0>)
        case M_RHS: GDG_K3P(M_RHS)<<<grid, block, sm, s>>>(mp, b, sc); break;
        case M_S1: GDG_K3P(M_S1)<<<grid, block, sm, s>>>(mp, b, sc); break;
        default: GDG_K3P(M_S23)<<<grid, block, sm, s>>>(mp, b, sc); break;
#undef GDG_K3P
        }
        return;
    }
    switch (mode) {
    case M_RHS: k_stage3<N1, M_RHS><<<grid, block, sm, s>>>(mp, b, sc); break;
    case M_S1: k_stage3<N1, M_S1><<<grid, block, sm, s>>>(mp, b, sc); break;
    default: k_stage3<N1, M_S23><<<grid, block, sm, s>>>(mp, b, sc); break;
    }
}

}  // namespace

void gdg3_stage(const ModalParams &mp, int n1, int mode, const StageBufs &b, double sc, cudaStream_t s) {
    switch (n1) {
#define X(n) case n: launch_stage3<n>(mode, mp, b, sc, s); break;
        GDG_N1_CASES3(X)
#undef X
    }
}

void gdg3_sep(const ModalParams &mp, int n1, int kind, const double *in0, const double *in1, double *out0, double *out1,
              const double *Bx, const double *By, const double *Bz, const double *D, const double *Cx, const double *Cy,
              const double *Cz, double *tr, cudaStream_t s) {
    const int epb = epb3(n1);
    const dim3 grid((mp.ne + epb - 1) / epb), block(epb * n1 * n1);
    switch (n1) {
#define X(n) case n: (kind == 0 ? k_sep3<n, 0> : k_sep3<n, 3>)<<<grid, block, smem_sep3(n), s>>>(mp, in0, in1, out0, out1, Bx, By, Bz, D, Cx, Cy, Cz, tr); break;
        GDG_N1_CASES3(X)
#undef X
    }
}

template <int N1>
void launch_fx3(const ModalParams &mp, int kind, const FxTables &t, const double *in0, const double *in1, double *out0,
                double *out1, double *tr, cudaStream_t s) {
    constexpr int EPB = epb3c<N1>(), LEN = N1 * ((N1 + 1) / 2);
    FxLines<N1, 3> A;
    for (int d = 0; d < 3; ++d) {
        std::copy(t.a[d][kind - 1], t.a[d][kind - 1] + LEN, A.a[d]);
        A.pe[d] = t.pe[d][kind - 1];
    }
    (kind == FX_TO_MODES ? k_fx3<N1, FX_TO_MODES> : k_fx3<N1, FX_TO_NODES>)<<<(mp.ne + EPB - 1) / EPB, EPB * N1 * N1,
        (size_t)EPB * N1 * N1 * N1 * sizeof(double), s>>>(mp, A, in0, in1, out0, out1, tr);
}

void gdg3_fx(const ModalParams &mp, int n1, int kind, const FxTables &t, const double *in0, const double *in1, double *out0,
             double *out1, double *tr, cudaStream_t s) {
    switch (n1) {
#define X(n) case n: launch_fx3<n>(mp, kind, t, in0, in1, out0, out1, tr, s); break;
        GDG_N1_CASES3(X)
#undef X
    }
}

void gdg3_energy_partial(int n1, int ne, const double *yU, const double *yV, const double *lam2, double *partial,
                         int blocks, cudaStream_t s) {
    switch (n1) {
#define X(n) case n: k_energy_partial3<n><<<blocks, 256, 0, s>>>(ne, yU, yV, lam2, partial); break;
        GDG_N1_CASES3(X)
#undef X
    }
}

void gdg3_set_smem_limits() {
    const int lim = 200 * 1024;
#define X(n)                                                                                    \
    cudaFuncSetAttribute(k_stage3<n, M_RHS>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim); \
    cudaFuncSetAttribute(k_stage3<n, M_S1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);  \
    cudaFuncSetAttribute(k_stage3<n, M_S23>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim); \
    cudaFuncSetAttribute(k_stage3p<n, M_RHS, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim); \
    cudaFuncSetAttribute(k_stage3p<n, M_S1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);  \
    cudaFuncSetAttribute(k_stage3p<n, M_S23, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim); \
    cudaFuncSetAttribute(k_stage3p<n, M_RHS, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim); \
    cudaFuncSetAttribute(k_stage3p<n, M_S1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);  \
    cudaFuncSetAttribute(k_stage3p<n, M_S23, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim); \
    cudaFuncSetAttribute(k_sep3<n, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);       \
    cudaFuncSetAttribute(k_sep3<n, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    GDG_N1_CASES3(X)
#undef X
}

// this translation unit's check slot (gdg_checks.cuh)
GDG_CHECKS_READER(gdg_checks_read_const3)
