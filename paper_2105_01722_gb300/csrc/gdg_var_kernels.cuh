// Device code of the variable-coefficient / mapped-element path shared by
// gdg_var.cu (per-problem launches) and gdg_batch.cu (batched launches).
#pragma once

#include "gdg_checks.cuh"
#include <cmath>

#include "gdg_fx.cuh"
#include "gdg_internal.h"

#define GDG_VAR_MAXN1 10

// element matrices as integers (k_fx_pack)
struct FxMatrix {
    const int2 *A;
    const short *d;   // FX_BAD: the element's matrix is not finite, nor is any product with it
};
constexpr short FX_BAD = 0x7fff;

struct VarParams {
    int nx, ny, ne, Q;
    int per_x, per_y, upwind;
    int alt;              // alternating flux (alpha = 1; side 1 = the element with the smaller index)
    double xi;            // > 0: constant splitting, else local c
    double rtol;
    int maxit, precond;   // GDG_PC_*
    const double *tab;    // B[Q][N1], D[Q][N1], wq[Q], dphiL[N1], dphiR[N1], Psi[N1][N1], lam[N1]
    const double *w, *pre, *face;
    const double *dS;            // [ne][N1*N1] frozen-coefficient preconditioner diagonal (S system)
    // the operators of the stage as integers (gdg_fx.cuh).  Element matrices: packed lower triangles
    // (fx_tri_len entries an element) and the exponents d of their rows [ne][N1*N1]
    FxMatrix Sx, Mx;             // S_c2, M_J
    FxMatrix Ax, Vx;             // inverse of the u_t system (k_var_invert), M_J^-1 (GDG_SOLVE_INVERSE)
    const int2 *FM;              // [ne][4 faces] operators, [6 N1 columns][3 N1 rows]; inverse route [3][3 N1 rows][2 N1] (k_fm_pack)
    const short2 *FMq;           // [ne][4 faces][3 N1] exponents of a row's v columns and u columns
    int staged;                  // FM's layout: lift_lines_staged's (stages of the inverse route outside batches)
    int slope_exp;               // the u slopes along a face normal count as 2^-slope_exp of the u values
    const int2 *Psx;             // Psi in units of 2^(Ps_exp - 57), rows and columns summing to at most 2^57
    int Ps_exp;
    // point source f = src_amp sin(src_omega t) delta(x - x_s) (gdg_set_point_source)
    int src_e;                   // element holding x_s (-1: no source)
    double src_amp, src_omega;
    const double *src_w;         // [NA]: phi_a(x_s)
    double *time;                // source time at the start of the current RK step
    int inverse;                 // GDG_SOLVE_INVERSE: element inverses instead of PCG
    unsigned long long *stats;   // [0] sum it_u, [1] sum it_v, [2] max it_u, [3] max it_v,
                                 // [4] unconverged u, [5] unconverged v, [6] element solves,
                                 // [7] sum sweeps u, [8] sum sweeps v, [9] max sweeps u, [10] max sweeps v
    int mixed;                   // FP32 inner PCG + FP64 refinement
    const unsigned char *affine; // [ne] 1: the element is a parallelogram (J constant), so the
                                 // frozen-coefficient mass preconditioner is M_J^-1 exactly
    int refine_max;              // FP64 refinement sweeps per solve
    float refine_rtol;           // inner FP32 PCG relative tolerance
};

struct VarBufs {
    const double *yU, *yV;   // stage input (nodal)
    double *nU, *nV, *aU, *aV, *oU, *oV;
    const double *trin;
    double *trout;
    // split stage for the learned initial guess: part 0 = whole stage;
    // part 1 = write the residuals r_u, r_v and stop; part 2 = take r_u, r_v
    // and the u_t guess x0u from memory and solve (falling back to x0 = 0 when
    // the guess's residual is not smaller than ||r_u||)
    int part;
    double *ru, *rv;
    const double *x0u;
    double tstage;           // this stage's time offset in the RK step (0, dt/2, dt/2, dt)
};

struct VarData;

// The element kernels of one N1: their own translation unit each (gdg_var_n*.cu),
// so that they compile in parallel.
struct VarOps {
    void (*attrs)(int smem_limit);
    void (*stage)(const VarParams &P, size_t smem, int mode, const VarBufs &b, double cA, double cY, cudaStream_t s);
    void (*pcg)(const VarParams &P, size_t smem, int which, const double *b, double *x, int *iters, double *rel,
                int *sweeps, cudaStream_t s);
    int (*checks)(GdgCheckSlot *out, int reset);   // the unit's check slot (gdg_checks.cuh)
};
extern const VarOps var_ops_2, var_ops_3, var_ops_4, var_ops_5, var_ops_6, var_ops_7, var_ops_8, var_ops_9, var_ops_10;

struct VarData {
    int nq = 0, Q = 0, NA = 0;
    double *d_w = nullptr, *d_pre = nullptr, *d_face = nullptr;
    double *d_dS = nullptr;
    int2 *d_fx = nullptr;                        // packed integer matrices: S, M (, A^-1, M^-1)
    short *d_fxd = nullptr;                      // their row exponents
    double *d_FM = nullptr;                      // face operators (integers after k_fm_pack)
    short2 *d_FMq = nullptr;
    int2 *d_Psx = nullptr;
    double *d_time = nullptr, *d_src = nullptr;  // point source: time, weights [NA]
    double *d_work = nullptr;                    // setup: the element matrices (and inverses) in FP64, a part of the mesh at a time
    double *d_tab = nullptr, *d_nodes = nullptr;
    unsigned char *d_affine = nullptr;           // per element: a parallelogram
    double *d_state = nullptr, *d_tr = nullptr;
    long long tr_len = 0;
    unsigned long long *d_stats = nullptr;
    int *d_iters = nullptr, *d_sweeps = nullptr;
    double *d_rel = nullptr, *d_red = nullptr, *h_red = nullptr;
    VarParams vp{};
    size_t smem_stage = 0, smem_geom = 0, smem_traces = 0, smem_pcg = 0;
    // learned u_t guess
    float *d_c2feat = nullptr;              // [ne][81] c^2 / element mean of c^2
    int learned = 0;
    uint16_t *d_wbf16 = nullptr;            // attached network (copies)
    float *d_mlp = nullptr;
    double *d_ru = nullptr, *d_rv = nullptr, *d_x0u = nullptr;   // split-stage buffers
};

namespace {

constexpr int GEOM_THREADS = 256;

__host__ __device__ constexpr int nthreads_for(int na) { return ((na + 31) / 32) * 32; }

// element kernels are declared for at least this many resident blocks per SM
// (shared memory allows 3-5); without a minimum ptxas keeps them near 64
// registers and spills inside the PCG loops
constexpr int kVarMinBlocks = 3;

struct Tabs {
    const double *B, *D, *wq, *dphiL, *dphiR, *Ps, *lam;
};

__device__ __forceinline__ Tabs tabs_at(const double *base, int Q, int N1) {
    Tabs t;
    t.B = base;
    t.D = t.B + Q * N1;
    t.wq = t.D + Q * N1;
    t.dphiL = t.wq + Q;
    t.dphiR = t.dphiL + N1;
    t.Ps = t.dphiR + N1;
    t.lam = t.Ps + N1 * N1;
    return t;
}
__host__ __device__ constexpr int tab_len(int Q, int N1) { return 2 * Q * N1 + Q + 2 * N1 + N1 * N1 + N1; }
// copy the 1-D tables into shared memory
__device__ void load_tabs(double *dst, const double *src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

__device__ __forceinline__ size_t fix(int e, int f, int q, int k, int Q) {   // face data
    return (((size_t)e * 4 + f) * Q + q) * 4 + k;
}
// face traces are the face lines of face_lines: [e][face][3 N1] (line index
// m N1 + j as in face_lines); 12 N1 doubles per element
template <int N1>
__device__ __forceinline__ size_t lix(int e, int f) { return ((size_t)e * 4 + f) * 3 * N1; }

// neighbour across face f (0 xm, 1 xp, 2 ym, 3 yp) and its facing face; -1 on a Dirichlet side
__device__ __forceinline__ int neighbour(const VarParams &P, int e, int f, int &fo) {
    int ex = e % P.nx, ey = e / P.nx;
    switch (f) {
    case 0: ex -= 1; fo = 1; break;
    case 1: ex += 1; fo = 0; break;
    case 2: ey -= 1; fo = 3; break;
    default: ey += 1; fo = 2; break;
    }
    if (ex < 0 || ex >= P.nx) {
        if (!P.per_x) return -1;
        ex = (ex + P.nx) % P.nx;
    }
    if (ey < 0 || ey >= P.ny) {
        if (!P.per_y) return -1;
        ey = (ey + P.ny) % P.ny;
    }
    int nb = ey * P.nx + ex;
    GDG_CHECK_INDEX(nb, 0, P.ne, GDG_SITE_VAR_NB, e);
    return nb;
}

// deterministic block sum: warp butterflies, then every thread adds the
// warp partials in the same order
// (the partials are stored in the value's own type: no conversions)
template <typename T>
__device__ __forceinline__ T block_sum(T v, double *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T *part = reinterpret_cast<T *>(red);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[w] = v;
    __syncthreads();
    T s = 0;
    for (int i = 0; i < nw; ++i) s += part[i];
    return s;
}

// ---------------------------------------------------- element solves -----
//
// One block works on one element, thread t owns entry t of every vector (in a
// register).  Products with the element matrices and the preconditioner run on
// integers (gdg_fx.cuh), and the FP64 work left is kept to what one thread per
// entry, or warp 0 alone, can do: an FP64 warp instruction takes 16 cycles of
// the SM's pipe whatever its active lanes.  (One warp per element with three
// rows a lane issues a third fewer instructions but leaves 7 warps an SM, too
// few to hide the integer pipe's latency: 12.2 against 9.5 ms a PCG step of 128 x 128 elements at p = 5.)

// one element's matrix and the block's scratch
struct FxSystem {
    const int2 *A;   // packed integers (shared)
    int d;           // exponent of the thread's row (FX_BAD: the matrix is not finite)
    int2 *X, *X2;    // limb vectors (shared, 16-byte aligned)
    int *slot;       // shared: two sets of 8 ints, used in turn
};

constexpr int FX_NAN = 1 << 20;   // block exponent of a vector with an Inf or NaN
constexpr int FX_NOT = 1 << 14;   // exponents from here on (FX_NAN, FX_BAD): the result is NaN
#define FX_QNAN __longlong_as_double(0x7ff8000000000000ll)

// exponent of v 2^shift for the maximum of a vector (zero and subnormals: below every other)
__device__ __forceinline__ int fx_key(double v, int shift = 0) {
    const int e = fx_expo(v);
    return e == 0 ? -FX_NAN : e == 0x7ff ? FX_NAN : e + shift;
}

// largest k of the block (at most 4 warps).  One barrier: consecutive calls use
// the two slot sets in turn (`set` 0 or 1), so a set is rewritten only after
// the barrier that follows its last read.
__device__ __forceinline__ int fx_block_max(int k, int *slot, int set) {
    k = __reduce_max_sync(0xffffffffu, k);
    int *sl = slot + 8 * set;
    if ((threadIdx.x & 31) == 0) sl[threadIdx.x >> 5] = k;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) k = max(k, sl[w]);
    return k;
}

// T 2^q, or NaN where the vector behind T had an Inf or NaN
__device__ __forceinline__ double fx_value(long long T, int q, int emax) {
    return emax >= FX_NOT ? FX_QNAN : fx_scale(T, q);
}

// mad(entry (t, k), k) over row t of the packed matrix: the columns of earlier
// warps' rows lie in row t, those of later warps' rows in the rows below (both
// at fixed strides), and only those of the own warp's rows need a choice
template <int NA, typename MAD>
__device__ __forceinline__ void fx_row(const int2 *A, MAD mad) {
    const int t = threadIdx.x, k0 = t & ~31, k1 = min(k0 + 32, NA);
    const int2 *row = A + t * (t + 1) / 2;             // entry (t, k), k <= t
#pragma unroll 8
    for (int k = 0; k < k0; ++k) mad(row[k], k);
    const int2 *col = A + k0 * (k0 + 1) / 2 + t;       // entry (k, t), moving with k
#pragma unroll 8
    for (int k = k0; k < k1; ++k) {
        mad(*(k <= t ? row + k : col), k);
        col += k + 1;
    }
#pragma unroll 8
    for (int k = k1; k < NA; ++k) {
        mad(*col, k);
        col += k + 1;
    }
}

// The same with V entries of the vector from one 16-byte read: 2 % faster where
// the products stream through (inverse route: four steps on 128^2 elements 7.52
// -> 7.33 ms), 1 to 2 % slower in the iterative routes.
template <int NA, typename ROW>
__device__ __forceinline__ void fx_row_wide(const int2 *A, ROW &r) {
    constexpr int V = ROW::V, TAIL = NA % V;
    const int t = threadIdx.x, k0 = t & ~31, k1 = min(k0 + 32, NA);
    const int2 *row = A + t * (t + 1) / 2;             // entry (t, k), k <= t
#pragma unroll 8 / V
    for (int k = 0; k < k0; k += V) {
        const int4 x = r.read(k);
#pragma unroll
        for (int j = 0; j < V; ++j) r.mad(row[k + j], x, j);
    }
    const int2 *col = A + k0 * (k0 + 1) / 2 + t;       // entry (k, t), moving with k
    auto choose = [&](int k, const int4 &x, int j) {
        r.mad(*(k + j <= t ? row + k + j : col), x, j);
        col += k + j + 1;
    };
    const int whole = k1 == NA ? NA - TAIL : k1;       // (only the last warp's own rows can end within a read)
#pragma unroll 8 / V
    for (int k = k0; k < whole; k += V) {
        const int4 x = r.read(k);
#pragma unroll
        for (int j = 0; j < V; ++j) choose(k, x, j);
    }
    if (k1 == NA) {
        if (TAIL) {
            const int4 x = r.read(NA - TAIL);          // (past the vector's end: not used)
#pragma unroll
            for (int j = 0; j < TAIL; ++j) choose(NA - TAIL, x, j);
        }
        return;
    }
#pragma unroll 8 / V
    for (int k = k1; k < NA - TAIL; k += V) {
        const int4 x = r.read(k);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            r.mad(*col, x, j);
            col += k + j + 1;
        }
    }
    if (TAIL) {
        const int4 x = r.read(NA - TAIL);
#pragma unroll
        for (int j = 0; j < TAIL; ++j) {
            r.mad(*col, x, j);
            col += NA - TAIL + j + 1;
        }
    }
}

struct FxRow {
    static constexpr int V = 2;
    FxSum s;
    const int2 *X;
    __device__ explicit FxRow(const int2 *X_) : X(X_) {}
    __device__ __forceinline__ int4 read(int k) const { return *reinterpret_cast<const int4 *>(X + k); }
    __device__ __forceinline__ void mad(int2 a, const int4 &x, int j) { s.mad(a, j ? x.z : x.x, j ? x.w : x.y); }
};
// The thread's entry of A x for its entry of x.  Two barriers; `set` as in
// fx_block_max.
template <int NA, bool WIDE = false>
__device__ __forceinline__ double fx_matvec(const FxSystem &f, double x, int set) {
    const int t = threadIdx.x;
    const int emax = fx_block_max(t < NA ? fx_key(x, f.d) : -FX_NAN, f.slot, set);
    if (t < NA) f.X[t] = fx_split(fx_int(x, emax, f.d));
    __syncthreads();
    FxRow row(f.X);
    if (t < NA) {
        if (WIDE) fx_row_wide<NA>(f.A, row);
        else fx_row<NA>(f.A, [&](int2 a, int k) { row.s.mad(a, row.X[k]); });
    }
    return fx_value(row.s.top(), fx_top_exp(emax) + f.d, max(emax, f.d));
}

// Psi of the frozen-coefficient preconditioner as integers (shared), and the
// thread's entry of the diagonal; or none
struct FxPrecond {
    const int2 *Ps;
    int pexp;
    double d;
    bool none;
};

// z = Psi2 diag(d) Psi2^T r, Psi2 = Psi (x) Psi (index j*N1+i), on integers:
// four contractions of N1 terms, the vector rescaled to its largest entry
// before the first and, after the diagonal, before the third (two in a row
// keep at least 52 bits: Psi's rows and columns sum to at most 1 in units of
// 2^pexp).  Four FP64 operations a node where the contractions by node pairs
// took 27.  Uses both slot sets; ends without a barrier.
template <int N1>
__device__ __forceinline__ double fx_precondition(const FxSystem &f, const FxPrecond &p, double r) {
    constexpr int NA = N1 * N1;
    const int t = threadIdx.x;
    if (p.none) return r;
    const bool on = t < NA;
    const int a = on ? t / N1 : 0, c = on ? t - a * N1 : 0;
    const int e1 = fx_block_max(on ? fx_key(r) : -FX_NAN, f.slot, 0);
    if (on) f.X[t] = fx_split(fx_int(r, e1));
    __syncthreads();
    if (on) {   // x modes: sum_i r[j][i] Psi[i][k]
        FxSum s(FxSum::NEXT);
#pragma unroll
        for (int q = 0; q < N1; ++q) s.mad(p.Ps[q * N1 + c], f.X[a * N1 + q]);
        f.X2[t] = s.next();
    }
    __syncthreads();
    double v = 0.0;
    if (on) {   // y modes and the diagonal: d[l][k] sum_j Psi[j][l] t[j][k]
        FxSum s;
#pragma unroll
        for (int q = 0; q < N1; ++q) s.mad(p.Ps[q * N1 + a], f.X2[q * N1 + c]);
        v = (double)s.top() * p.d;
    }
    const int e2 = fx_block_max(on ? fx_key(v) : -FX_NAN, f.slot, 1);
    if (on) f.X[t] = fx_split(fx_int(v, e2));
    __syncthreads();
    if (on) {   // back in x: sum_k t[l][k] Psi[i][k]
        FxSum s(FxSum::NEXT);
#pragma unroll
        for (int q = 0; q < N1; ++q) s.mad(p.Ps[c * N1 + q], f.X[a * N1 + q]);
        f.X2[t] = s.next();
    }
    __syncthreads();
    FxSum s;   // back in y: sum_l Psi[j][l] t[l][i]
    if (on) {
#pragma unroll
        for (int q = 0; q < N1; ++q) s.mad(p.Ps[a * N1 + q], f.X2[q * N1 + c]);
    }
    return fx_value(s.top(), 4 * p.pexp + e1 + e2 + 2 * fx_top_exp(0), max(e1, e2));
}

// warp 0: the sums of a[k] b[k] and of c[k] d[k] over the NA entries in shared
// memory, each in every lane.  A lane adds its entries in order, then a
// butterfly whose first level leaves one sum to each half-warp, so the five
// levels cost five FP64 additions, not ten.
template <int NA>
__device__ __forceinline__ void lane_dot2(const double *a, const double *b, const double *c, const double *d,
                                          double &ab, double &cd) {
    double s = 0.0, q = 0.0;
#pragma unroll
    for (int k = threadIdx.x; k < NA; k += 32) {
        s = fma(a[k], b[k], s);
        q = fma(c[k], d[k], q);
    }
    const bool lo = threadIdx.x < 16;
    double v = (lo ? s : q) + __shfl_xor_sync(0xffffffffu, lo ? q : s, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    ab = __shfl_sync(0xffffffffu, v, 0);
    cd = __shfl_sync(0xffffffffu, v, 16);
}

// the same for the whole block (leading barrier: the vectors are written)
template <int NA>
__device__ __forceinline__ void block_dot2(const double *a, const double *b, const double *c, const double *d,
                                           double *red, double &ab, double &cd) {
    __syncthreads();
    if (threadIdx.x < 32) {
        lane_dot2<NA>(a, b, c, d, ab, cd);
        if (threadIdx.x == 0) { red[0] = ab; red[1] = cd; }
    }
    __syncthreads();
    ab = red[0];
    cd = red[1];
}

// sqrt(rr) <= thr, the square root taken only where the squares are too close
// to decide (or out of range)
__device__ __forceinline__ bool norm_below(double rr, double thr) {
    const double t2 = thr * thr;
    if (t2 > 1e-280 && t2 < 1e280) {
        if (rr > t2 * (1.0 + 1e-14)) return false;
        if (rr < t2 * (1.0 - 1e-14)) return true;
    }
    return sqrt(rr) <= thr;
}

// the block's vectors of a solve (shared, NA doubles each) and its scalars
struct SolveBufs {
    double *r, *z, *p, *Ap, *red;   // red: 8 doubles
    const double *w;
};

// x0 and r0 = b - A x0 (- w (w.x0)) of a solve: x0 = 0, or the guess in x,
// dropped (*fell = 1) when `fallback` and its true residual is no smaller than b
template <int NA>
__device__ __forceinline__ double first_residual(const FxSystem &f, const SolveBufs &v, bool W, double w, double b,
                                                 double &x, bool x0_zero, bool fallback, int *fell) {
    const int t = threadIdx.x;
    if (x0_zero) {
        x = 0.0;
        return b;
    }
    double r = b - fx_matvec<NA>(f, x, 0);
    if (t < NA) v.z[t] = x;
    if (W) {
        double wx, same;
        block_dot2<NA>(v.w, v.z, v.w, v.z, v.red, wx, same);
        r -= w * wx;
    }
    if (fallback) {
        double rr, bb;
        if (t < NA) { v.r[t] = r; v.p[t] = b; }
        block_dot2<NA>(v.r, v.r, v.p, v.p, v.red, rr, bb);
        if (rr >= bb) {
            x = 0.0;
            r = b;
            *fell = 1;
        }
        __syncthreads();
    }
    return r;
}

// Preconditioned CG on A (+ w w^T when W) with x0 = x (x0_zero: x0 = 0).
// Stops when ||r|| <= rtol ||b|| (tested before each iteration), after
// maxit iterations, or when r.z = 0.  Returns the iteration count; *relres is
// formed when asked for or when the cap was reached.  b, x, w: the thread's
// entries.
template <int N1>
__device__ __forceinline__ int pcg(const FxSystem &f, const FxPrecond &pre, const SolveBufs &v, bool W, double w,
                                   double b, double &x, double rtol, int maxit, bool x0_zero, double *relres,
                                   bool fallback, int *fell, bool want_rel) {
    constexpr int NA = N1 * N1;
    const int t = threadIdx.x;
    const bool on = t < NA, warp0 = t < 32;
    double r = first_residual<NA>(f, v, W, w, b, x, x0_zero, fallback, fell);
    if (on) { v.r[t] = r; v.p[t] = b; }
    double b2 = 0.0, thr = 0.0;   // warp 0's
    double p = 0.0, rz = 0.0, rr = 0.0;
    int it = -1;   // the first pass only forms z and p
    while (true) {
        const double z = fx_precondition<N1>(f, pre, r);
        if (on) v.z[t] = z;
        __syncthreads();
        ++it;
        if (warp0) {
            double rzn, rrn, beta = 0.0;
            lane_dot2<NA>(v.r, v.z, v.r, v.r, rzn, rrn);
            if (it == 0) {
                double same;
                lane_dot2<NA>(v.p, v.p, v.p, v.p, b2, same);
                thr = rtol * sqrt(b2);
            }
            const bool done = it >= maxit || norm_below(rrn, thr) || rzn == 0.0;
            if (it && !done) beta = rzn / rz;
            if (t == 0) { v.red[0] = beta; v.red[1] = done ? 1.0 : 0.0; v.red[2] = rrn; }
            rz = rzn;
        }
        __syncthreads();
        if (v.red[1] != 0.0) break;
        p = it ? z + v.red[0] * p : z;
        if (on) v.p[t] = p;
        const double Ap = fx_matvec<NA>(f, p, 0);
        if (on) v.Ap[t] = Ap;
        __syncthreads();
        if (warp0) {   // p.(A + w w^T)p = p.Ap + (w.p)^2
            double pAp, wp;
            lane_dot2<NA>(v.p, v.Ap, W ? v.w : v.p, W ? v.p : v.Ap, pAp, wp);
            if (W) pAp += wp * wp;
            const double alpha = rz / pAp;
            if (t == 0) { v.red[4] = alpha; v.red[5] = wp; }
        }
        __syncthreads();
        const double alpha = v.red[4];
        x += alpha * p;
        r -= alpha * (W ? Ap + w * v.red[5] : Ap);
        if (on) v.r[t] = r;
    }
    rr = v.red[2];
    if (want_rel || it >= maxit) {   // the cap, or the caller's statistics
        __syncthreads();
        if (t == 0) v.red[3] = b2 == 0.0 ? 0.0 : sqrt(rr) / sqrt(b2);   // (NaN where b is)
        __syncthreads();
        *relres = v.red[3];
    } else {
        *relres = 0.0;
    }
    __syncthreads();
    return it;
}

// ---- the FP32 inner solves of the mixed form

// the inner system: the thread's row scale 2^d, preconditioner diagonal and w
struct Inner32 {
    float sc, d, w;
    const float *Ps;       // shared
    float *t1, *t2, *red;  // shared scratch: NA floats each; two sets of 8 partial sums
    float rtol;
    int maxit;
    bool none;
};

// The thread's entry of A x in 32 bits: the upper limbs of A (29 bits against
// the largest of the scaled matrix, where a float has 24) and x as an integer
// of 28 bits against its largest entry, summed exactly.
template <int NA>
__device__ __forceinline__ float fx_matvec32(const FxSystem &f, float sc, float x) {
    const int t = threadIdx.x;
    const float v = x * sc;
    const int e = fx_block_max(t < NA ? (__float_as_int(v) >> 23) & 0xff : 0, f.slot, 0);   // |v| < 2^(e - 126)
    int *X = reinterpret_cast<int *>(f.X);
    if (t < NA) X[t] = __float2int_rn(v * __int_as_float(max(1, min(254, 281 - e)) << 23));   // v 2^(154 - e)
    __syncthreads();
    long long s = 0;
    if (t < NA) fx_row<NA>(f.A, [&](int2 a, int k) { s += (long long)a.x * X[k]; });
    // a.x in units of 2^-28: the sum times 2^(e - 182)
    const float down = e == 255 ? __int_as_float(0x7fc00000) : __int_as_float(max(1, min(254, e - 23)) << 23);
    return ((float)(int)(s >> 32) + (float)(unsigned)s * 2.3283064365386963e-10f) * down * sc;
}

// the thread's entry of z = Psi2 diag(d) Psi2^T r in FP32; ends without a barrier
template <int N1>
__device__ __forceinline__ float precondition32(const Inner32 &in, float r) {
    constexpr int NA = N1 * N1;
    const int t = threadIdx.x;
    if (in.none) return r;
    const bool on = t < NA;
    const int a = on ? t / N1 : 0, c = on ? t - a * N1 : 0;
    if (on) in.t1[t] = r;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < N1; ++q) s = fmaf(in.t1[a * N1 + q], in.Ps[q * N1 + c], s);
    if (on) in.t2[t] = s;
    __syncthreads();
    s = 0.f;
#pragma unroll
    for (int q = 0; q < N1; ++q) s = fmaf(in.Ps[q * N1 + a], in.t2[q * N1 + c], s);
    if (on) in.t1[t] = in.d * s;
    __syncthreads();
    s = 0.f;
#pragma unroll
    for (int q = 0; q < N1; ++q) s = fmaf(in.t1[a * N1 + q], in.Ps[c * N1 + q], s);
    if (on) in.t2[t] = s;
    __syncthreads();
    s = 0.f;
#pragma unroll
    for (int q = 0; q < N1; ++q) s = fmaf(in.Ps[a * N1 + q], in.t2[q * N1 + c], s);
    return s;
}

// two block sums with one barrier (the two sets of partial sums in turn)
__device__ __forceinline__ void block_sum2(float &a, float &b, float *red, int set) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    float *part = red + 8 * set;
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { part[w] = a; part[4 + w] = b; }
    __syncthreads();
    a = b = 0.f;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) { a += part[i]; b += part[4 + i]; }
}

// FP32 PCG from x0 = 0 on A + w w^T (w = 0 for the mass system) for a
// right-hand side of unit norm, r its entry: stops when ||r|| <= rtol, after
// maxit iterations or at r.z = 0.  x: the thread's entry of the result.
template <int N1>
__device__ __forceinline__ int pcg32(const FxSystem &f, const Inner32 &in, float r, float &x) {
    constexpr int NA = N1 * N1;
    const bool on = threadIdx.x < NA;
    float p = 0.f, rz = 0.f;
    x = 0.f;
    int it = -1;
    while (true) {
        const float z = precondition32<N1>(in, r);
        float rzn = on ? r * z : 0.f, rr = on ? r * r : 0.f;
        block_sum2(rzn, rr, in.red, 0);
        ++it;
        if (it >= in.maxit || sqrtf(rr) <= in.rtol || rzn == 0.f) break;
        p = it ? z + (rzn / rz) * p : z;
        rz = rzn;
        const float Ap = fx_matvec32<NA>(f, in.sc, p);
        float pAp = on ? p * Ap : 0.f, wp = on ? in.w * p : 0.f;
        block_sum2(pAp, wp, in.red, 1);
        const float alpha = rz / (pAp + wp * wp);   // p.(A + w w^T)p = p.Ap + (w.p)^2
        x += alpha * p;
        r -= alpha * (Ap + in.w * wp);
    }
    return it;
}

// Mixed-precision solve of A x = b (+ w w^T when W): iterative refinement with
// FP64-accurate products with A for every residual and FP32 PCG for every
// correction.
//   r = b - A x (FP64);  while ||r|| > rtol ||b||:  A c ~= r/||r|| (FP32 PCG),
//   x += ||r|| c (FP64);  r = b - A x (FP64)
// The stopping test is the FP64 PCG's (true FP64 residual), so the accuracy
// is that of the FP64 solver at the same rtol.  Returns the sweeps (FP64
// residual evaluations after the first); *inner = FP32 iterations.
// FP64 step: when `step64` is set and x0 = 0, the solve (of the mass system)
// first takes the FP64 preconditioned steepest-descent step x = alpha P^-1 b
// (the first FP64 PCG iterate); where the frozen-coefficient preconditioner is
// exact (the mass matrix of an affine element) that step already meets the
// tolerance and no FP32 sweep runs.
template <int N1>
__device__ __forceinline__ int refine(const FxSystem &f, const FxPrecond &pre, const Inner32 &in, const SolveBufs &v,
                                      bool W, double w, double b, double &x, double rtol, int maxsweep, bool x0_zero,
                                      int *inner, double *relres, bool fallback, int *fell, bool step64) {
    constexpr int NA = N1 * N1;
    const int t = threadIdx.x;
    const bool on = t < NA;
    double r;
    if (x0_zero && step64) {
        const double z = fx_precondition<N1>(f, pre, b), Az = fx_matvec<NA>(f, z, 0);
        if (on) { v.z[t] = z; v.r[t] = Az; v.p[t] = b; }   // (v.Ap holds the inner solves' Psi)
        double bz, zAz;
        block_dot2<NA>(v.p, v.z, v.z, v.r, v.red, bz, zAz);
        const double alpha = zAz > 0.0 ? bz / zAz : 0.0;
        x = alpha * z;
        r = b - alpha * Az;
    } else {
        r = first_residual<NA>(f, v, W, w, b, x, x0_zero, fallback, fell);
    }
    if (on) { v.r[t] = r; v.p[t] = b; }
    double bb, rr;
    block_dot2<NA>(v.p, v.p, v.r, v.r, v.red, bb, rr);
    const double bnorm = sqrt(bb);
    double rn = sqrt(rr);
    int sweeps = 0, its = 0;
    while (sweeps < maxsweep && rn > rtol * bnorm && rn > 0.0) {
        const double inv = 1.0 / rn;
        float c;
        its += pcg32<N1>(f, in, on ? (float)(r * inv) : 0.f, c);
        x += rn * (double)c;
        r = b - fx_matvec<NA>(f, on ? x : 0.0, 0);
        if (W) {
            if (on) v.z[t] = x;
            double wx, same;
            block_dot2<NA>(v.w, v.z, v.w, v.z, v.red, wx, same);
            r -= w * wx;
        }
        if (on) v.r[t] = r;
        double same;
        block_dot2<NA>(v.r, v.r, v.r, v.r, v.red, rr, same);
        rn = sqrt(rr);
        ++sweeps;
    }
    *inner = its;
    *relres = bnorm == 0.0 ? 0.0 : rn / bnorm;
    if (!isfinite(rn)) x = *relres = FX_QNAN;   // no sweep runs on a NaN, and x may still be zero
    return sweeps;
}

// asynchronous global -> shared copies (cp.async): every copy of a matrix is
// in flight at once instead of a register round trip per element
__device__ __forceinline__ void cp_async_16(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// diagonal of the frozen-coefficient preconditioner in the modified basis,
// made once at setup: dS[e][l*N1+k] = 1 / (Gss lam_l + Grr lam_k) (1 on the
// constant mode), and pre[e][3] = 1 / |e| (the mass preconditioner's diagonal)
template <int N1>
__global__ void __launch_bounds__(nthreads_for(N1 * N1), kVarMinBlocks)
k_fdm_diag(const double *__restrict__ lam, double *pre, double *dS) {
    constexpr int NA = N1 * N1;
    const int e = blockIdx.x, t = threadIdx.x;
    const double Grr = pre[(size_t)e * 4 + 0], Gss = pre[(size_t)e * 4 + 1], Jb = pre[(size_t)e * 4 + 2];
    if (t < NA) {
        const int l = t / N1, k = t - (t / N1) * N1;
        dS[(size_t)e * NA + t] = t == 0 ? 1.0 : 1.0 / (Gss * lam[l] + Grr * lam[k]);
    }
    if (t == 0) pre[(size_t)e * 4 + 3] = 1.0 / Jb;
}

// --------------------------------------------------------- assembly -------

// Sout, Mout: of the elements e0, e0 + 1, ..., a block each
template <int N1>
__global__ void __launch_bounds__(GEOM_THREADS)
k_var_geom(VarParams P, int e0, const double *X, const double *Y, const double *C2, double *Sout, double *Mout,
           double *wout, double *pre, double *face) {
    constexpr int NA = N1 * N1;
    extern __shared__ __align__(16) double sm[];
    const int Q = P.Q, e = e0 + blockIdx.x, t = threadIdx.x;
    double *tb = sm;
    double *nx_ = tb + tab_len(Q, N1);
    double *ny_ = nx_ + NA, *nc = ny_ + NA;
    double *XD = nc + NA, *XB = XD + N1 * Q, *YD = XB + N1 * Q, *YB = YD + N1 * Q, *CB = YB + N1 * Q;
    double *Wr = CB + N1 * Q, *Grr = Wr + Q, *Gss = Grr + Q, *Grs = Gss + Q;
    double *CM = Grs + Q, *Crr = CM + NA, *Css = Crr + NA, *Crs = Css + NA;
    double *red = Crs + NA;    // [32] reduction scratch
    load_tabs(tb, P.tab, tab_len(Q, N1));
    const Tabs T = tabs_at(tb, Q, N1);
    for (int i = t; i < NA; i += blockDim.x) {
        nx_[i] = X[(size_t)e * NA + i];
        ny_[i] = Y[(size_t)e * NA + i];
        nc[i] = C2[(size_t)e * NA + i];
    }
    double sGrr = 0.0, sGss = 0.0, sW = 0.0;   // this thread's share of the element means
    __syncthreads();
    // XD[j][a] = sum_i X[j][i] D[a][i], XB[j][a] = sum_i X[j][i] B[a][i] (same for Y; C2 with B)
    for (int task = t; task < N1 * Q; task += blockDim.x) {
        const int j = task / Q, a = task - (task / Q) * Q;
        double xd = 0, xb = 0, yd = 0, yb = 0, cb = 0;
        for (int i = 0; i < N1; ++i) {
            const double Bi = T.B[a * N1 + i], Di = T.D[a * N1 + i];
            xd += nx_[j * N1 + i] * Di; xb += nx_[j * N1 + i] * Bi;
            yd += ny_[j * N1 + i] * Di; yb += ny_[j * N1 + i] * Bi;
            cb += nc[j * N1 + i] * Bi;
        }
        XD[task] = xd; XB[task] = xb; YD[task] = yd; YB[task] = yb; CB[task] = cb;
    }
    __syncthreads();
    constexpr int PER = (NA * NA + GEOM_THREADS - 1) / GEOM_THREADS;
    for (int pass = 0; pass < 2; ++pass) {   // 0: M_J, 1: S_c2
        double accv[PER];
#pragma unroll
        for (int m = 0; m < PER; ++m) accv[m] = 0.0;
        for (int b = 0; b < Q; ++b) {
            for (int a = t; a < Q; a += blockDim.x) {
                double xr = 0, xs = 0, yr = 0, ys = 0, c2 = 0;
                for (int j = 0; j < N1; ++j) {
                    const double Bj = T.B[b * N1 + j], Dj = T.D[b * N1 + j];
                    xr += Bj * XD[j * Q + a]; xs += Dj * XB[j * Q + a];
                    yr += Bj * YD[j * Q + a]; ys += Dj * YB[j * Q + a];
                    c2 += Bj * CB[j * Q + a];
                }
                const double det = xr * ys - xs * yr;
                const double ww = T.wq[a] * T.wq[b];
                Wr[a] = ww * det;
                Grr[a] = ww * c2 * (xs * xs + ys * ys) / det;
                Gss[a] = ww * c2 * (xr * xr + yr * yr) / det;
                Grs[a] = -ww * c2 * (xr * xs + yr * ys) / det;
                if (pass == 0) { sGrr += Grr[a]; sGss += Gss[a]; sW += Wr[a]; }
            }
            __syncthreads();
            for (int task = t; task < NA; task += blockDim.x) {
                const int i = task / N1, i2 = task - (task / N1) * N1;
                if (pass == 0) {
                    double s = 0;
                    for (int a = 0; a < Q; ++a) s += Wr[a] * T.B[a * N1 + i] * T.B[a * N1 + i2];
                    CM[task] = s;
                } else {
                    double srr = 0, sss = 0, srs = 0;
                    for (int a = 0; a < Q; ++a) {
                        const double Bi = T.B[a * N1 + i], Di = T.D[a * N1 + i];
                        const double Bi2 = T.B[a * N1 + i2], Di2 = T.D[a * N1 + i2];
                        srr += Grr[a] * Di * Di2;
                        sss += Gss[a] * Bi * Bi2;
                        srs += Grs[a] * Di * Bi2;
                    }
                    Crr[task] = srr; Css[task] = sss; Crs[task] = srs;
                }
            }
            __syncthreads();
#pragma unroll
            for (int m = 0; m < PER; ++m) {
                const int o = t + m * GEOM_THREADS;
                if (o < NA * NA) {
                    const int al = o / NA, be = o - (o / NA) * NA;
                    const int j = al / N1, i = al - (al / N1) * N1, j2 = be / N1, i2 = be - (be / N1) * N1;
                    const double Bj = T.B[b * N1 + j], Bj2 = T.B[b * N1 + j2];
                    if (pass == 0) {
                        accv[m] += Bj * Bj2 * CM[i * N1 + i2];
                    } else {
                        const double Dj = T.D[b * N1 + j], Dj2 = T.D[b * N1 + j2];
                        accv[m] += Bj * Bj2 * Crr[i * N1 + i2] + Dj * Dj2 * Css[i * N1 + i2] +
                                   Bj * Dj2 * Crs[i * N1 + i2] + Dj * Bj2 * Crs[i2 * N1 + i];
                    }
                }
            }
            __syncthreads();
        }
        double *out = (pass == 0 ? Mout : Sout) + (size_t)blockIdx.x * NA * NA;
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int o = t + m * GEOM_THREADS;
            if (o < NA * NA) out[o] = accv[m];
        }
        __syncthreads();
        // exact symmetry (the two triangles differ by rounding): lower := upper,
        // so that A x can be formed from columns (coalesced) with row-order sums
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int o = t + m * GEOM_THREADS;
            const int al = o / NA, be = o - (o / NA) * NA;
            if (o < NA * NA && al > be) out[o] = out[(size_t)be * NA + al];
        }
        __syncthreads();
    }
    // w = M_J 1 / |e| (row sums of what was just written), frozen-coefficient scalars
    sGrr = block_sum(sGrr, red);
    sGss = block_sum(sGss, red);
    sW = block_sum(sW, red);
    if (t < NA) {
        const double *row = Mout + (size_t)blockIdx.x * NA * NA + (size_t)t * NA;
        double s = 0.0;
        for (int k = 0; k < NA; ++k) s += row[k];
        wout[(size_t)e * NA + t] = s / sW;   // w = M_J 1 / |e|
    }
    if (t == 0) {
        pre[(size_t)e * 4 + 0] = sGrr;
        pre[(size_t)e * 4 + 1] = sGss;
        pre[(size_t)e * 4 + 2] = sW;
        pre[(size_t)e * 4 + 3] = 0.0;
    }
    // face data: fr, fs (J^-1 n), c^2 |T| w, c at every face point
    for (int task = t; task < 4 * Q; task += blockDim.x) {
        const int f = task / Q, q = task - (task / Q) * Q;
        const double *dphi = (f == 0 || f == 2) ? T.dphiL : T.dphiR;
        double xr = 0, xs = 0, yr = 0, ys = 0, c2 = 0;
        if (f < 2) {   // r = 0 / 1, parametrised by s_q
            const int col = f == 0 ? 0 : N1 - 1;
            for (int j = 0; j < N1; ++j) {
                double dx = 0, dy = 0;
                for (int i = 0; i < N1; ++i) { dx += nx_[j * N1 + i] * dphi[i]; dy += ny_[j * N1 + i] * dphi[i]; }
                const double Bj = T.B[q * N1 + j], Dj = T.D[q * N1 + j];
                xr += Bj * dx; yr += Bj * dy;
                xs += Dj * nx_[j * N1 + col]; ys += Dj * ny_[j * N1 + col];
                c2 += Bj * nc[j * N1 + col];
            }
        } else {       // s = 0 / 1, parametrised by r_q
            const int row = f == 2 ? 0 : N1 - 1;
            for (int i = 0; i < N1; ++i) {
                double dx = 0, dy = 0;
                for (int j = 0; j < N1; ++j) { dx += nx_[j * N1 + i] * dphi[j]; dy += ny_[j * N1 + i] * dphi[j]; }
                const double Bi = T.B[q * N1 + i], Di = T.D[q * N1 + i];
                xs += Bi * dx; ys += Bi * dy;
                xr += Di * nx_[row * N1 + i]; yr += Di * ny_[row * N1 + i];
                c2 += Bi * nc[row * N1 + i];
            }
        }
        double tn, nxv, nyv;
        if (f < 2) { tn = sqrt(xs * xs + ys * ys); nxv = ys / tn; nyv = -xs / tn; }
        else { tn = sqrt(xr * xr + yr * yr); nxv = -yr / tn; nyv = xr / tn; }
        if (f == 0 || f == 2) { nxv = -nxv; nyv = -nyv; }
        const double det = xr * ys - xs * yr;
        face[fix(e, f, q, 0, Q)] = (ys * nxv - xs * nyv) / det;
        face[fix(e, f, q, 1, Q)] = (-yr * nxv + xr * nyv) / det;
        face[fix(e, f, q, 2, Q)] = c2 * tn * T.wq[q];
        face[fix(e, f, q, 3, Q)] = sqrt(c2);
    }
}

// ----------------------------------------------------------- traces ------

// line data of the 4 faces from nodal U, V in shared memory:
// L[(f*3 + m)*N1 + j]: m = 0 value line of v, 1 the r-derivative data, 2 the s-derivative data
// by the `nt` threads t = 0.. of a warp or block
template <int N1>
__device__ __forceinline__ void face_lines(const double *U, const double *V, const Tabs &T, double *L, int t, int nt) {
    for (int task = t; task < 12 * N1; task += nt) {
        const int f = task / (3 * N1), m = (task / N1) % 3, j = task % N1;
        const double *dphi = (f == 0 || f == 2) ? T.dphiL : T.dphiR;
        const int edge = (f == 0 || f == 2) ? 0 : N1 - 1;
        // one slope (m = 1 on x faces, 2 on y faces) and two values a line
        const bool slope = f < 2 ? m == 1 : m == 2;
        const double *line = f < 2 ? U + j * N1 : U + j;
        const int step = f < 2 ? 1 : N1;
        double s = 0.0;
        if (slope) { for (int i = 0; i < N1; ++i) s += line[i * step] * dphi[i]; }
        else s = (m == 0 ? (f < 2 ? V + j * N1 : V + j) : line)[edge * step];
        L[task] = s;
    }
}

template <int N1>
__global__ void k_var_traces(VarParams P, const double *u, const double *v, double *trout) {
    constexpr int NA = N1 * N1;
    extern __shared__ __align__(16) double sm[];
    const int Q = P.Q, e = blockIdx.x;
    double *tb = sm, *U = tb + tab_len(Q, N1), *V = U + NA;
    load_tabs(tb, P.tab, tab_len(Q, N1));
    for (int i = threadIdx.x; i < NA; i += blockDim.x) {
        U[i] = u[(size_t)e * NA + i];
        V[i] = v[(size_t)e * NA + i];
    }
    __syncthreads();
    const Tabs T = tabs_at(tb, Q, N1);
    face_lines<N1>(U, V, T, trout + lix<N1>(e, 0), threadIdx.x, blockDim.x);
}

// ------------------------------------------------------------ stage ------



// load of the point source on r_v at this stage: int phi_a f = phi_a(x_s) s(t)
__device__ __forceinline__ double source_amplitude(const VarParams &P, const VarBufs &b) {
    return P.src_amp * sin(P.src_omega * (*P.time + b.tstage));
}

__global__ void k_set_time(double *time, double t0) { *time = t0; }

// Shared memory of one element's block, in doubles: the packed matrix (or, for
// the lifts of the inverse route, face operators), Psi, w and one scratch region
// for the phases of a stage in turn: the lifts (limbs of the face lines, line
// integrals), the solves (vectors and limb vectors; the FP32 vectors in the place
// of p and Ap), the new state whose face lines go out.  INV: the inverse route
// alone, which keeps a limb vector or the line integrals beside the matrix, all
// else in its place: 27.6 KB at N1 = 9, 8 blocks an SM, where the rest needs 31.4
// KB and 7.
template <int N1, bool INV>
struct StageSmem {
    static constexpr int NA = N1 * N1;
    static constexpr int NP = (NA + 1) & ~1;   // limb vectors start on 16 bytes
    static constexpr int SCR = 36 * N1 > 6 * NP ? (36 * N1 + 1) & ~1 : 6 * NP;
    static constexpr int FACE = 18 * NA;       // a face's operator
    static constexpr int LINES = INV ? 24 * N1 : 0;   // limbs of the face lines, beside the face operators
    static constexpr int ARENA = fx_tri_len(NA) > FACE + LINES ? fx_tri_len(NA) : FACE + LINES;
    static constexpr int SLOTS = (ARENA - LINES) / FACE < 2 ? 1 : 2;
    static constexpr int SIDE = NP > 12 * N1 ? NP : 12 * N1;
    static constexpr int LEN = ARENA + (INV ? SIDE : 2 * NP + SCR) + 24;
    int2 *A, *Ps, *lines, *X, *X2;
    int *slot;
    double *L, *U, *V, *w, *r, *z, *p, *Ap, *red;
    float *Ps32, *t1, *t2, *red32;
    __device__ StageSmem(double *base) {
        A = reinterpret_cast<int2 *>(base);
        red = base + LEN - 24;                            // 8 doubles
        slot = reinterpret_cast<int *>(red + 8);          // 16 ints
        red32 = reinterpret_cast<float *>(red + 16);      // 16 floats
        if (INV) {
            lines = A + SLOTS * FACE;
            L = base + ARENA;
            X = A + ARENA;
            U = base;
            V = base + NP;
            return;
        }
        Ps = A + ARENA;
        w = base + ARENA + NP;
        double *scr = w + NP;
        lines = reinterpret_cast<int2 *>(scr);
        L = scr + 24 * N1;
        X = lines;
        X2 = X + NP;
        r = scr + 2 * NP;
        z = r + NP;
        p = z + NP;
        Ap = p + NP;
        t1 = reinterpret_cast<float *>(p);
        t2 = t1 + NP;
        Ps32 = reinterpret_cast<float *>(Ap);
        U = scr;
        V = scr + NP;
    }
    static constexpr size_t bytes() { return sizeof(double) * (size_t)LEN; }
    __device__ __forceinline__ FxSystem system(const FxMatrix &m, int e) const {
        return FxSystem{A, threadIdx.x < NA ? m.d[(size_t)e * NA + threadIdx.x] : 0, X, X2, slot};
    }
    __device__ __forceinline__ SolveBufs bufs() const { return SolveBufs{r, z, p, Ap, red, w}; }
};

// start the copy of an element's packed matrix into shared memory
template <int N1>
__device__ __forceinline__ void load_fx(int2 *A, const FxMatrix &m, int e) {
    constexpr int LEN = fx_tri_len(N1 * N1);
    const int2 *src = m.A + (size_t)e * LEN;
    for (int i = 2 * threadIdx.x; i < LEN; i += 2 * blockDim.x) cp_async_16(A + i, src + i);
}
// wait for it (the whole block)
__device__ __forceinline__ void fx_arrived() {
    cp_async_wait_all();
    __syncthreads();
}

// Face terms.  Per face f of an element the fluxes of Section 2.2.1 at the Q
// face quadrature points, weighted and integrated against the face basis
// (the line integrals L[f][m][j], m = 0..2 the three lifted quantities, j the
// node along the face), are linear in the 3 N1 face lines of the element
// (face_lines) and the 3 N1 face lines of the neighbour's facing face, with
// coefficients fixed in time (geometry, c^2, the flux).  k_var_facemat
// builds that map once per element and face; the stage applies it.

// traces (v, n.grad u) at face point q of face f of element e from a face
// line vector that is zero except entry (m, j) = 1 (the point evaluation of
// face_lines' lines: x faces (B, B, D) of lines (v, normal slope, u), y faces
// (B, D, B) of lines (v, u, normal slope))
template <int N1>
__device__ __forceinline__ void unit_point_trace(const Tabs &T, const double *face, int e, int f, int q, int Q,
                                                 int m, int j, double &v, double &d) {
    const double Bq = T.B[q * N1 + j], Dq = T.D[q * N1 + j];
    v = m == 0 ? Bq : 0.0;
    double ur, us;
    if (f < 2) { ur = m == 1 ? Bq : 0.0; us = m == 2 ? Dq : 0.0; }
    else { ur = m == 1 ? Dq : 0.0; us = m == 2 ? Bq : 0.0; }
    d = face[fix(e, f, q, 0, Q)] * ur + face[fix(e, f, q, 1, Q)] * us;
}

// the three weighted flux values of face point q (nb < 0: Dirichlet side,
// the caller passes the mirror state vo = -vi, do = -di)
__device__ __forceinline__ void point_flux(const VarParams &P, int e, int f, int q, int nb, double vi, double di,
                                           double vo, double dO, double *w3, int Q) {
    double beta = 0.0, tau = 0.0;
    if (P.upwind) {
        const double xi = P.xi > 0.0 ? P.xi : P.face[fix(e, f, q, 3, Q)];
        beta = 0.5 * xi;
        tau = 0.5 / xi;
    }
    double vstar = 0.5 * (vi + vo) - beta * (di + dO);
    double qstar = 0.5 * (di - dO) - tau * (vi - vo);
    if (P.alt && nb >= 0) {   // minus faces (0, 2): this element is side 2
        vstar = (f == 0 || f == 2) ? vo : vi;
        qstar = (f == 0 || f == 2) ? di : -dO;
    }
    const double g = vstar - vi;
    const double cw = P.face[fix(e, f, q, 2, Q)];
    w3[0] = cw * P.face[fix(e, f, q, 0, Q)] * g;
    w3[Q] = cw * P.face[fix(e, f, q, 1, Q)] * g;
    w3[2 * Q] = cw * qstar;
}

// FM[e][f][c][r]: line integral r = m N1 + j of face f per unit face-line
// value c (c < 3 N1: the element's own line entry c; c >= 3 N1: entry
// c - 3 N1 of the neighbour's facing face, zero columns on a Dirichlet
// side).  One CTA per element; shared: 3 Q doubles.
template <int N1>
__global__ void __launch_bounds__(nthreads_for(N1 * N1))
k_var_facemat(VarParams P, double *__restrict__ FM) {
    constexpr int NL = 3 * N1;
    extern __shared__ __align__(16) double fw[];
    const int Q = P.Q, e = blockIdx.x, t = threadIdx.x;
    const Tabs T = tabs_at(P.tab, Q, N1);
    for (int f = 0; f < 4; ++f) {
        int fo;
        const int nb = neighbour(P, e, f, fo);
        for (int c = 0; c < 2 * NL; ++c) {
            double *col = FM + (((size_t)e * 4 + f) * 2 * NL + c) * NL;
            const bool own = c < NL;
            if (!own && nb < 0) {
                for (int r = t; r < NL; r += blockDim.x) col[r] = 0.0;
                continue;
            }
            const int cc = own ? c : c - NL, m = cc / N1, j = cc - (cc / N1) * N1;
            for (int q = t; q < Q; q += blockDim.x) {
                double vi = 0.0, di = 0.0, vo = 0.0, dO = 0.0;
                if (own) unit_point_trace<N1>(T, P.face, e, f, q, Q, m, j, vi, di);
                else unit_point_trace<N1>(T, P.face, nb, fo, q, Q, m, j, vo, dO);
                if (nb < 0) { vo = -vi; dO = -di; }   // u = 0: mirror state
                point_flux(P, e, f, q, nb, vi, di, vo, dO, fw + q, Q);
            }
            __syncthreads();
            for (int r = t; r < NL; r += blockDim.x) {
                const int mr = r / N1, jr = r - (r / N1) * N1;
                // x faces: (B, D, B); y faces: (D, B, B)
                const bool useD = (f < 2) ? (mr == 1) : (mr == 0);
                const double *tab = useD ? T.D : T.B;
                double sum = 0.0;
                for (int q = 0; q < Q; ++q) sum += tab[q * N1 + jr] * fw[mr * Q + q];
                col[r] = sum;
            }
            __syncthreads();
        }
    }
}

// The columns of a face in three parts of 2 N1: the v lines of both sides, the
// element's own u lines, the neighbour's (column c as in k_var_facemat).
template <int N1> __device__ __forceinline__ int line_third(int c) { return c % (3 * N1) < N1 ? 0 : c < 3 * N1 ? 1 : 2; }
template <int N1> __device__ __forceinline__ int line_place(int c) {
    return c % (3 * N1) < N1 ? c / (3 * N1) * N1 + c % N1 : c % (3 * N1) - N1;
}

// The face operators as integers, in place, face by face.  `staged`: [part][row]
// [2 N1] in place of [6 N1][row], so that a row's part is read 16 bytes at a time
// (lift_lines_staged).  A row's columns fall in two groups,
// each in units of 2^(q - 57): the v lines and the u lines, whose vectors get
// a block exponent each (u and v may differ by any factor).  The u group holds
// values along the face and slopes across it; the slopes count as
// 2^-slope_exp of themselves, 2^slope_exp >= sum |phi'|, so that they are no
// larger than the values behind them.
template <int N1>
__device__ __forceinline__ bool slope_line(int f, int m) { return f < 2 ? m == 1 : m == 2; }

template <int N1>
__global__ void __launch_bounds__(nthreads_for(N1 * N1))
k_fm_pack(double *FM, int slope_exp, int staged, short2 *FMq) {
    constexpr int NL = 3 * N1, FACE = 2 * NL * NL;
    __shared__ double in[FACE];
    const int e = blockIdx.x;
    for (int f = 0; f < 4; ++f) {
        double *face = FM + ((size_t)e * 4 + f) * FACE;
        for (int i = threadIdx.x; i < FACE; i += blockDim.x) in[i] = face[i];
        __syncthreads();
        for (int r = threadIdx.x; r < NL; r += blockDim.x) {
            int qv = -FX_NAN, qu = -FX_NAN;
            for (int c = 0; c < 2 * NL; ++c) {
                const int m = (c % NL) / N1;
                const int k = fx_key(in[c * NL + r], slope_line<N1>(f, m) ? slope_exp : 0) - 1022;   // |v| < 2^k
                if (m == 0) qv = max(qv, k); else qu = max(qu, k);
            }
            // Inf and NaN (c^2 interpolated below zero has no square root) mark the row: FX_BAD
            qv = qv > FX_NAN / 2 ? FX_BAD : max(-16000, qv);
            qu = qu > FX_NAN / 2 ? FX_BAD : max(-16000, qu);
            FMq[((size_t)e * 4 + f) * NL + r] = make_short2((short)qv, (short)qu);
            for (int c = 0; c < 2 * NL; ++c) {
                const int m = (c % NL) / N1;
                const int to = staged ? (line_third<N1>(c) * NL + r) * 2 * N1 + line_place<N1>(c) : c * NL + r;
                reinterpret_cast<int2 *>(face)[to] =
                    (m == 0 ? qv : qu) == FX_BAD
                        ? make_int2(0, 0)
                        : fx_split(fx_int(in[c * NL + r], (m == 0 ? qv : qu) + 1022, slope_line<N1>(f, m) ? slope_exp : 0));
            }
        }
        __syncthreads();
    }
}

// a row's sum T as a line integral; q: the exponent of its columns
__device__ __forceinline__ double fx_face_value(long long T, int q, int emax) {
    return fx_value(T, fx_top_exp(emax) + q, max(emax, q));
}

// line integrals L[f][m][j] of the element's four faces from its own face
// lines and its neighbours' (lines: 24 N1 limb pairs of shared scratch).
// A row's 6 N1 coefficients go to two threads, one for the own and one for the
// neighbour's lines, whose sums are then added.  Bound by the 46.7 KB of
// face operators an element reads (N1 = 9).
template <int N1>
__device__ __forceinline__ void lift_lines(const VarParams &P, int e, const double *trin, int2 *lines, int *slot,
                                           double *L) {
    constexpr int NL = 3 * N1, BD = nthreads_for(N1 * N1), PER = (4 * NL + BD - 1) / BD;
    const int t = threadIdx.x;
    double own[PER], nbl[PER];
    int kv = -FX_NAN, ku = -FX_NAN;
#pragma unroll
    for (int s = 0; s < PER; ++s) {
        const int i = t + BD * s;
        own[s] = nbl[s] = 0.0;
        if (i < 4 * NL) {
            const int f = i / NL, c = i - f * NL, m = c / N1;
            int fo;
            const int nb = neighbour(P, e, f, fo);
            own[s] = trin[lix<N1>(e, 0) + i];
            if (nb >= 0) nbl[s] = trin[lix<N1>(nb, fo) + c];
            const int sh = slope_line<N1>(f, m) ? -P.slope_exp : 0;
            const int k = max(fx_key(own[s], sh), fx_key(nbl[s], sh));
            if (m == 0) kv = max(kv, k); else ku = max(ku, k);
        }
    }
    kv = __reduce_max_sync(0xffffffffu, kv);
    ku = __reduce_max_sync(0xffffffffu, ku);
    if ((t & 31) == 0) { slot[8 + (t >> 5)] = kv; slot[12 + (t >> 5)] = ku; }   // set 1
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { kv = max(kv, slot[8 + w]); ku = max(ku, slot[12 + w]); }
#pragma unroll
    for (int s = 0; s < PER; ++s) {
        const int i = t + BD * s;
        if (i < 4 * NL) {
            const int f = i / NL, m = (i - f * NL) / N1;
            const int sh = slope_line<N1>(f, m) ? -P.slope_exp : 0, k = m == 0 ? kv : ku;
            lines[i] = fx_split(fx_int(own[s], k, sh));
            lines[4 * NL + i] = fx_split(fx_int(nbl[s], k, sh));   // zero on a Dirichlet side
        }
    }
    __syncthreads();
    constexpr int PAIRS = BD / 2;
#pragma unroll 1
    for (int task0 = 0; task0 < 4 * NL; task0 += PAIRS) {
        const int task = min(task0 + (t >> 1), 4 * NL - 1), side = t & 1, f = task / NL;
        const int2 *a = P.FM + (((size_t)e * 4 + f) * 2 + side) * NL * NL + (task - f * NL);
        const int2 *x = lines + side * 4 * NL + f * NL;
        FxSum sv, su;
#pragma unroll
        for (int c = 0; c < N1; ++c) sv.mad(__ldg(a + (size_t)c * NL), x[c]);
#pragma unroll
        for (int c = N1; c < NL; ++c) su.mad(__ldg(a + (size_t)c * NL), x[c]);
        long long T = sv.top(), S = su.top();
        T += __shfl_xor_sync(0xffffffffu, T, 1);
        S += __shfl_xor_sync(0xffffffffu, S, 1);
        const short2 q = P.FMq[(size_t)e * 4 * NL + task];
        // one conversion a thread: the even one takes the v sum, the odd one the u sum
        double y = side ? fx_face_value(S, q.y, ku) : fx_face_value(T, q.x, kv);
        y += __shfl_xor_sync(0xffffffffu, y, 1);
        if (side == 0 && task0 + (t >> 1) < 4 * NL) L[task] = y;
    }
    __syncthreads();
}

// start the copy of the operator of face f into its slot of the matrix's place
template <int N1, typename SMEM>
__device__ __forceinline__ void load_face(const VarParams &P, const SMEM &s, int e, int f) {
    constexpr int FACE = SMEM::FACE;
    const int2 *src = P.FM + ((size_t)e * 4 + f) * FACE;
    int2 *dst = s.A + f % SMEM::SLOTS * FACE;
    for (int i = 2 * threadIdx.x; i < FACE; i += 2 * blockDim.x) cp_async_16(dst + i, src + i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// The same in the inverse route, whose operators all stream through: the face
// operators come through the matrix's place in shared memory, as many at a time
// as fit (the first ones on their way when this starts).  A row's three parts go
// to three lanes of a warp, ten rows a warp.  The own and the neighbour's lines are
// rounded apart and then added, as in lift_lines: the same bits.  128^2 elements, four steps with element
// inverses: 8.55 -> 7.50 ms, with the eighth block an SM that the smaller scratch
// allows (staged alone 7.92).  In the iterative
// routes, where S would have to be read again for the solve, the direct form is
// the faster one: a step of 128^2 elements 9.5 against 9.8 ms.
template <int N1, typename SMEM>
__device__ __forceinline__ void lift_lines_staged(const VarParams &P, const SMEM &s, int e, const double *trin) {
    constexpr int NL = 3 * N1, BD = nthreads_for(N1 * N1), PER = (4 * NL + BD - 1) / BD, WARPS = BD / 32;
    constexpr int FACE = SMEM::FACE, SLOTS = SMEM::SLOTS;
    const int t = threadIdx.x;
    int *slot = s.slot;
    double own[PER], nbl[PER];
    int kv = -FX_NAN, ku = -FX_NAN;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = t + BD * i;
        own[i] = nbl[i] = 0.0;
        if (q < 4 * NL) {
            const int f = q / NL, c = q - f * NL;
            int fo;
            const int nb = neighbour(P, e, f, fo);
            own[i] = trin[lix<N1>(e, 0) + q];
            if (nb >= 0) nbl[i] = trin[lix<N1>(nb, fo) + c];
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = t + BD * i, f = q / NL, m = (q - f * NL) / N1;
        if (q < 4 * NL) {
            const int sh = slope_line<N1>(f, m) ? -P.slope_exp : 0;
            const int k = max(fx_key(own[i], sh), fx_key(nbl[i], sh));
            if (m == 0) kv = max(kv, k); else ku = max(ku, k);
        }
    }
    kv = __reduce_max_sync(0xffffffffu, kv);
    ku = __reduce_max_sync(0xffffffffu, ku);
    if ((t & 31) == 0) { slot[8 + (t >> 5)] = kv; slot[12 + (t >> 5)] = ku; }   // set 1
    __syncthreads();
    for (int w = 0; w < WARPS; ++w) { kv = max(kv, slot[8 + w]); ku = max(ku, slot[12 + w]); }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int q = t + BD * i;
        if (q < 4 * NL) {
            const int f = q / NL, c = q - f * NL, m = c / N1;
            const int sh = slope_line<N1>(f, m) ? -P.slope_exp : 0, k = m == 0 ? kv : ku;
            int2 *x = s.lines + f * 6 * N1;
            x[line_third<N1>(c) * 2 * N1 + line_place<N1>(c)] = fx_split(fx_int(own[i], k, sh));
            x[line_third<N1>(c + NL) * 2 * N1 + line_place<N1>(c + NL)] = fx_split(fx_int(nbl[i], k, sh));   // zero on a Dirichlet side
        }
    }
    const int lane = t & 31, part = lane % 3;
#pragma unroll 1
    for (int f = 0; f < 4; ++f) {
        if (f + 1 < SLOTS) asm volatile("cp.async.wait_group %0;\n" ::"n"(SLOTS > 1 ? SLOTS - 1 : 0) : "memory");   // the first of SLOTS
        else cp_async_wait_all();
        __syncthreads();   // face f has arrived, and every thread is past face f - 1
        if (SLOTS > 1 && f >= 1 && f - 1 + SLOTS < 4) load_face<N1>(P, s, e, f - 1 + SLOTS);
#pragma unroll 1
        for (int row0 = 10 * (t >> 5); row0 < NL; row0 += 10 * WARPS) {
            const int row = min(row0 + lane / 3, NL - 1);
            const short2 q = P.FMq[((size_t)e * 4 + f) * NL + row];
            const int4 *a = reinterpret_cast<const int4 *>(s.A + f % SLOTS * FACE + (part * NL + row) * 2 * N1);
            const int4 *x = reinterpret_cast<const int4 *>(s.lines + (f * 3 + part) * 2 * N1);
            FxSum sum;
            long long own = 0;
#pragma unroll
            for (int c = 0; c < 2 * N1; ++c) {
                if (c == N1 && part == 0) {   // the own v lines end here
                    own = sum.top();
                    sum = FxSum();
                }
                const int4 av = a[c / 2], xv = x[c / 2];
                if (c & 1) sum.mad(make_int2(av.z, av.w), xv.z, xv.w);
                else sum.mad(make_int2(av.x, av.y), xv.x, xv.y);
            }
            long long T = own + sum.top();
            const long long nbr = __shfl_down_sync(0xffffffffu, T, 1);
            if (part == 1) T += nbr;
            const double y = fx_face_value(T, part ? q.y : q.x, part ? ku : kv);
            const double u = __shfl_down_sync(0xffffffffu, y, 1);
            if (part == 0 && lane < 30 && row0 + lane / 3 < NL) s.L[f * NL + row] = y + u;
        }
        if (SLOTS == 1 && f < 3) {
            __syncthreads();
            load_face<N1>(P, s, e, f + 1);
        }
    }
    __syncthreads();
}

// r_u, r_v (r_v without the stiffness term) at node t from the face line integrals
template <int N1>
__device__ __forceinline__ void lift_assemble(const double *L, const Tabs &T, int t, double &ru, double &rv) {
    const int j = t / N1, i = t - (t / N1) * N1;
    const double *Lx0 = L, *Lx1 = L + 3 * N1, *Ly0 = L + 6 * N1, *Ly1 = L + 9 * N1;
    double u_ = T.dphiL[i] * Lx0[j] + T.dphiR[i] * Lx1[j] + T.dphiL[j] * Ly0[N1 + i] + T.dphiR[j] * Ly1[N1 + i];
    double v_ = 0.0;
    if (i == 0) { u_ += Lx0[N1 + j]; v_ += Lx0[2 * N1 + j]; }
    if (i == N1 - 1) { u_ += Lx1[N1 + j]; v_ += Lx1[2 * N1 + j]; }
    if (j == 0) { u_ += Ly0[i]; v_ += Ly0[2 * N1 + i]; }
    if (j == N1 - 1) { u_ += Ly1[i]; v_ += Ly1[2 * N1 + i]; }
    ru = u_;
    rv = v_;
}

// Psi into shared memory, as integers or, for the inner solves, in FP32
template <int N1>
__device__ __forceinline__ void load_psi(const VarParams &P, const StageSmem<N1, false> &s) {
    if (threadIdx.x < N1 * N1) s.Ps[threadIdx.x] = P.Psx[threadIdx.x];
}

// The route of a stage.  ROUTE_ANY reads it from the problem (batches; FP64 PCG,
// which is as fast so: 9.52 ms a step of 128^2 elements, alone 9.56); the mixed
// form by itself spills less at 80 registers (128 x 120 elements, p = 3, a step
// 6.41 -> 6.26 ms), the inverse route has its own layout of shared memory.
enum { ROUTE_ANY, ROUTE_MIXED, ROUTE_INVERSE };
template <int ROUTE> __device__ __forceinline__ bool route_inverse(const VarParams &P) {
    return ROUTE == ROUTE_ANY ? P.inverse != 0 : ROUTE == ROUTE_INVERSE;
}
template <int ROUTE> __device__ __forceinline__ bool route_mixed(const VarParams &P) {
    return ROUTE == ROUTE_ANY ? P.mixed != 0 : ROUTE == ROUTE_MIXED;
}

// solve one of the element's systems (W: the u_t system, + w w^T) from the
// right-hand side b; x: the guess (unless zero) and the result
template <int N1, int ROUTE>
__device__ __forceinline__ void solve(const VarParams &P, const StageSmem<N1, false> &s, const Tabs &T, int e, bool W, double w,
                                      double b, double &x, bool zero, bool guess, int *iters, int *sweeps, int *fell,
                                      double *rel, bool want_rel) {
    constexpr int NA = N1 * N1;
    const int t = threadIdx.x;
    const bool on = t < NA;
    const FxSystem f = s.system(W ? P.Sx : P.Mx, e);
    const FxPrecond pre{s.Ps, P.Ps_exp, W ? (on ? P.dS[(size_t)e * NA + t] : 0.0) : P.pre[(size_t)e * 4 + 3],
                        P.precond == GDG_PC_NONE};
    if (route_mixed<ROUTE>(P)) {
        Inner32 in;
        in.sc = __int_as_float(max(1, min(254, 127 + f.d)) << 23);
        in.d = (float)pre.d;
        in.w = W ? (float)w : 0.f;
        in.Ps = s.Ps32;
        in.t1 = s.t1;
        in.t2 = s.t2;
        in.red = s.red32;
        in.rtol = P.refine_rtol;
        in.maxit = P.maxit;
        in.none = pre.none;
        // in the mass system the FP64 preconditioned step first, only where it
        // solves it outright (a parallelogram); elsewhere it would cost an FP64
        // product and still leave two FP32 sweeps
        *sweeps = refine<N1>(f, pre, in, s.bufs(), W, w, b, x, P.rtol, P.refine_max, zero, iters, rel, guess, fell,
                             !W && P.affine[e]);
    } else {
        *sweeps = 0;
        *iters = pcg<N1>(f, pre, s.bufs(), W, w, b, x, P.rtol, P.maxit, zero, rel, guess, fell, want_rel);
    }
}

// One element's RK stage (one block of nthreads_for(N1*N1) threads).
template <int N1, int ROUTE>
__device__ __forceinline__ void var_stage_body(const VarParams &P, const VarBufs &b, int mode, double cA, double cY, int e,
                                               double *smraw) {
    constexpr int NA = N1 * N1;
    const StageSmem<N1, ROUTE == ROUTE_INVERSE> s(smraw);
    const int t = threadIdx.x;
    const bool inverse = route_inverse<ROUTE>(P), mixed = route_mixed<ROUTE>(P);
    const bool on = t < NA;
    const size_t at = (size_t)e * NA + (on ? t : 0);
    const bool guess = b.part == 2;
    constexpr bool staged = ROUTE == ROUTE_INVERSE;   // (a problem of inverses in a batch: P.staged is 0)
    if constexpr (staged) {
#pragma unroll
        for (int f = 0; f < s.SLOTS; ++f) load_face<N1>(P, s, e, f);
    } else {
        load_fx<N1>(s.A, P.Sx, e);
    }
    const Tabs T = tabs_at(P.tab, P.Q, N1);
    const double Yu = on ? b.yU[at] : 0.0, Yv = on ? b.yV[at] : 0.0;
    double ru = 0.0, rv = 0.0, x = 0.0, w = 0.0;
    if constexpr (ROUTE != ROUTE_INVERSE) {
        w = on ? P.w[at] : 0.0;
        if (on) s.w[t] = w;
        if (!inverse) load_psi<N1>(P, s);
    }
    if constexpr (staged) {
        lift_lines_staged<N1>(P, s, e, b.trin);
        load_fx<N1>(s.A, P.Sx, e);
        if (on) lift_assemble<N1>(s.L, T, t, ru, rv);
    }
    fx_arrived();
    if (!guess) {
        const double SU = fx_matvec<NA, staged>(s.system(P.Sx, e), Yu, 0);
        __syncthreads();   // the matrix and the vector are read
        if (inverse && b.part != 1) load_fx<N1>(s.A, P.Ax, e);   // on its way during the lifts
        if constexpr (!staged) {
            lift_lines<N1>(P, e, b.trin, s.lines, s.slot, s.L);
            if (on) lift_assemble<N1>(s.L, T, t, ru, rv);
        }
        if (on) {
            rv -= SU;
            if (e == P.src_e) rv += source_amplitude(P, b) * P.src_w[t];
        }
        if (b.part == 1) {
            if (on) { b.ru[at] = ru; b.rv[at] = rv; }
            return;
        }
        __syncthreads();   // L is read
    } else if (on) {
        ru = b.ru[at];
        rv = b.rv[at];
        x = b.x0u[at];
    }
    if (inverse) {   // dU/dt = V + (S_c2 + sigma w w^T)^-1 r_u (k_var_invert), dV/dt = M_J^-1 r_v
#pragma unroll 1
        for (int sys = 0; sys < 2; ++sys) {
            fx_arrived();
            const double y = fx_matvec<NA, staged>(s.system(sys ? P.Vx : P.Ax, e), ru, 0);
            __syncthreads();
            if (sys == 0) {
                load_fx<N1>(s.A, P.Vx, e);
                ru = rv;
                rv = Yv + y;   // dU/dt
            }
            x = y;             // dV/dt after the second pass
        }
        if (t == 0 && P.stats) atomicAdd(&P.stats[6], 1ull);
    } else if constexpr (ROUTE != ROUTE_INVERSE) {
        int it[2], sw[2], fell = 0;
        bool bad[2];
#pragma unroll 1
        for (int sys = 0; sys < 2; ++sys) {   // the u_t system from r_u, then the v_t system from r_v
            double rel = 0.0;
            if (mixed && on) s.Ps32[t] = (float)T.Ps[t];
            if (sys) fx_arrived();
            solve<N1, ROUTE>(P, s, T, e, sys == 0, w, ru, x, sys || !guess, guess && !sys, &it[sys], &sw[sys], &fell, &rel, false);
            // (rel is formed at the cap and in the mixed form; a NaN is no convergence)
            bad[sys] = !(rel <= P.rtol) && (!mixed || sw[sys] >= P.refine_max || isnan(rel));
            __syncthreads();
            if (sys == 0) {
                load_fx<N1>(s.A, P.Mx, e);
                ru = rv;
                rv = Yv + x;   // dU/dt
            }
        }
        if (t == 0 && P.stats) {
            atomicAdd(&P.stats[0], (unsigned long long)it[0]);
            atomicAdd(&P.stats[1], (unsigned long long)it[1]);
            atomicMax(&P.stats[2], (unsigned long long)it[0]);
            atomicMax(&P.stats[3], (unsigned long long)it[1]);
            if (bad[0]) atomicAdd(&P.stats[4], 1ull);
            if (bad[1]) atomicAdd(&P.stats[5], 1ull);
            atomicAdd(&P.stats[6], 1ull);
            atomicAdd(&P.stats[7], (unsigned long long)sw[0]);
            atomicAdd(&P.stats[8], (unsigned long long)sw[1]);
            atomicMax(&P.stats[9], (unsigned long long)sw[0]);
            atomicMax(&P.stats[10], (unsigned long long)sw[1]);
            if (guess) atomicAdd(&P.stats[11], 1ull);          // solves started from a guess
            if (fell) atomicAdd(&P.stats[12], 1ull);           // ... of which fell back to x0 = 0
        }
    }
    // k = (rv, x); RK combine into the next stage input
    if (on) {
        const double ku = rv, kv = x;
        double nu = 0.0, nv = 0.0;
        if (mode == M_RHS) {
            b.oU[at] = ku;
            b.oV[at] = kv;
        } else if (mode == M_S1) {
            b.aU[at] = cA * ku;
            b.aV[at] = cA * kv;
            nu = Yu + cY * ku;
            nv = Yv + cY * kv;
        } else if (mode == M_S23) {
            b.aU[at] += cA * ku;
            b.aV[at] += cA * kv;
            nu = b.nU[at] + cY * ku;
            nv = b.nV[at] + cY * kv;
        } else {
            nu = b.nU[at] + b.aU[at] + cA * ku;
            nv = b.nV[at] + b.aV[at] + cA * kv;
        }
        if (mode != M_RHS) {
            (mode == M_S4 ? b.nU : b.oU)[at] = nu;
            (mode == M_S4 ? b.nV : b.oV)[at] = nv;
            s.U[t] = nu;
            s.V[t] = nv;
        }
    }
    // the source block (the only reader of the source time) starts the next step
    if (mode == M_S4 && e == P.src_e && t == 0) *P.time += b.tstage;
    if (mode == M_RHS) return;
    __syncthreads();
    face_lines<N1>(s.U, s.V, T, b.trout + lix<N1>(e, 0), t, blockDim.x);
}

// Where a problem's own steps with inverses stage their face operators: where the passes over the
// 3 N1 rows of a face (ten rows a warp) fill the block better than the direct form's over the 12 N1
// rows of all four (a row a pair of threads), N1 = 3, 6 and 9; and in blocks of one warp on
// meshes beyond the 16 blocks an SM that the registers of the any-route kernel leave.
// Eight steps, staged and direct, in ms.  100 x 100 elements: N1 = 9 9.2 and 10.6, 8 8.5 and 6.9, 7 7.0 and
// 6.3, 6 5.56 and 5.45, 10 14.4 and 14.1, 5 2.8 and 3.5, 4 2.6 and 3.0; 40 x 41: 5 0.60 and 0.55, 4
// 0.56 and 0.47, 3 0.42 and 0.44, 2 0.33 and 0.32.
__host__ __device__ constexpr bool staged_lifts(int n1, int ne, int sms) {
    const int bd = nthreads_for(n1 * n1), warps = bd / 32;
    const int staged = (3 * n1 + 10 * warps - 1) / (10 * warps) * 10 * warps;   // places for 3 N1 rows
    const int direct = (12 * n1 + bd / 2 - 1) / (bd / 2) * (bd / 2);            // ... for 12 N1
    return 4 * staged < direct || (warps == 1 && ne > 16 * sms);
}

// Resident blocks promised to ptxas for the stage kernel: the 7 (inverse route 8)
// that the shared memory of a block of at most 3 warps allows, 4 for larger elements.
__host__ __device__ constexpr int var_stage_min_blocks(int n1, int route) {
    return nthreads_for(n1 * n1) <= 96 ? (route == ROUTE_INVERSE ? 8 : 7) : 4;
}

template <int N1, int ROUTE>
__global__ void __launch_bounds__(nthreads_for(N1 * N1), var_stage_min_blocks(N1, ROUTE))
k_var_stage(const __grid_constant__ VarParams P, const __grid_constant__ VarBufs b, int mode, double cA, double cY) {
    extern __shared__ __align__(16) double smraw[];
    var_stage_body<N1, ROUTE>(P, b, mode, cA, cY, blockIdx.x, smraw);
}

// standalone element PCG (gdg_pcg): which = 0 M, 1 S (+ w w^T)
template <int N1, int ROUTE>
__global__ void __launch_bounds__(nthreads_for(N1 * N1), var_stage_min_blocks(N1, ROUTE_ANY))
k_var_pcg(VarParams P, int which, const double *bvec, double *xvec, int *iters, double *rel, int *sweeps) {
    constexpr int NA = N1 * N1;
    extern __shared__ __align__(16) double smraw[];
    const StageSmem<N1, false> s(smraw);
    const int e = blockIdx.x, t = threadIdx.x;
    const bool on = t < NA;
    const size_t at = (size_t)e * NA + (on ? t : 0);
    load_fx<N1>(s.A, which ? P.Sx : P.Mx, e);
    const Tabs T = tabs_at(P.tab, P.Q, N1);
    const double b = on ? bvec[at] : 0.0, w = on ? P.w[at] : 0.0;
    double x = on ? xvec[at] : 0.0, rr;
    int it, sw = 0, fell = 0;
    if (on) {
        s.w[t] = w;
        if (P.mixed) s.Ps32[t] = (float)T.Ps[t];
    }
    load_psi<N1>(P, s);
    fx_arrived();
    solve<N1, ROUTE>(P, s, T, e, which != 0, w, b, x, false, false, &it, &sw, &fell, &rr, true);
    if (on) xvec[at] = x;
    if (t == 0) {
        iters[e] = it;
        rel[e] = rr;
        if (sweeps) sweeps[e] = sw;
    }
}

// Element inverse at setup (GDG_SOLVE_INVERSE; the precomputed-inverse route
// of Section 3.1 applied to the element systems of Section 7.1):
// Dst[e] = (Src[e] + sigma w_e w_e^T)^-1 - (1/sigma) 1 1^T (w != nullptr) or
// Src[e]^-1.  The u_t system's right-hand sides have 1^T r_u = 0 (the constant
// test function has no gradient), so its solution y is the same for every weight
// sigma > 0: (S + sigma w w^T) 1 = sigma w, hence w^T y = 1^T r_u / sigma = 0.
// sigma, the power of two at or below the trace of S, puts the rank-one term among
// the eigenvalues of S: the inverse is as well conditioned as S on the
// functions without a constant part, whatever the size of c^2 (with sigma = 1 its
// error grew with c^2, 1e-4 at c^2 = 1e8, where it is 1e-13 now, and the part
// below could outweigh the rest of it).  Subtracting (1/sigma) 1 1^T takes the rounding of
// 1^T r_u out of w^T y and changes nothing else (still symmetric, and positive
// semidefinite).  By Cholesky
// A = L L^T in shared memory and one forward + back substitution per column
// of the identity (thread j solves column j); the result is made exactly
// symmetric (lower := upper) for the packed form.
template <int N1>
__global__ void __launch_bounds__(nthreads_for(N1 * N1))
k_var_invert(const double *__restrict__ Src, const double *__restrict__ w, double *__restrict__ Dst) {
    constexpr int NA = N1 * N1;
    extern __shared__ __align__(16) double sm[];
    double *A = sm, *B = A + NA * NA, *dinv = B + NA * NA;
    const int e = blockIdx.x, t = threadIdx.x, nt = blockDim.x;
    const double *src = Src + (size_t)e * NA * NA;
    const double *we = w ? w + (size_t)e * NA : nullptr;
    double sigma = 1.0;
    if (we) {
        double trace = 0.0;
        for (int i = 0; i < NA; ++i) trace += src[i * (NA + 1)];
        sigma = scalbn(1.0, ilogb(trace));
    }
    for (int i = t; i < NA * NA; i += nt) {
        const int r = i / NA, c = i - (i / NA) * NA;
        A[i] = src[i] + (we ? sigma * (we[r] * we[c]) : 0.0);
    }
    __syncthreads();
    // right-looking Cholesky, lower triangle in place
    for (int k = 0; k < NA; ++k) {
        if (t == 0) {
            const double d = sqrt(A[k * NA + k]);
            A[k * NA + k] = d;
            dinv[k] = 1.0 / d;
        }
        __syncthreads();
        const double di = dinv[k];
        for (int i = k + 1 + t; i < NA; i += nt) A[i * NA + k] *= di;
        __syncthreads();
        const int m = NA - k - 1;
        for (int idx = t; idx < m * m; idx += nt) {
            const int i = k + 1 + idx / m, j = k + 1 + idx - (idx / m) * m;
            if (j <= i) A[i * NA + j] -= A[i * NA + k] * A[j * NA + k];
        }
        __syncthreads();
    }
    if (t < NA) {
        const int j = t;
        // L z = e_j (z_i = 0 for i < j), then L^T x = z; column j of B
        for (int i = 0; i < j; ++i) B[i * NA + j] = 0.0;
        for (int i = j; i < NA; ++i) {
            double s0 = (i == j) ? 1.0 : 0.0, s1 = 0.0;
            int k = j;
            for (; k + 1 < i; k += 2) {
                s0 -= A[i * NA + k] * B[k * NA + j];
                s1 -= A[i * NA + k + 1] * B[(k + 1) * NA + j];
            }
            if (k < i) s0 -= A[i * NA + k] * B[k * NA + j];
            B[i * NA + j] = (s0 + s1) * dinv[i];
        }
        for (int i = NA - 1; i >= 0; --i) {
            double s0 = B[i * NA + j], s1 = 0.0;
            int k = i + 1;
            for (; k + 1 < NA; k += 2) {
                s0 -= A[k * NA + i] * B[k * NA + j];
                s1 -= A[(k + 1) * NA + i] * B[(k + 1) * NA + j];
            }
            if (k < NA) s0 -= A[k * NA + i] * B[k * NA + j];
            B[i * NA + j] = (s0 + s1) * dinv[i];
        }
    }
    __syncthreads();
    double *dst = Dst + (size_t)e * NA * NA;
    for (int i = t; i < NA * NA; i += nt) {
        const int r = i / NA, c = i - (i / NA) * NA;
        dst[i] = (r > c ? B[c * NA + r] : B[i]) - (we ? 1.0 / sigma : 0.0);
    }
}

// Integer form of ne exactly symmetric NA x NA element matrices (gdg_fx.cuh):
// packed lower triangles and row exponents, one block per element.  The exponents
// of the rows are those of their diagonal entries, which bound every entry of
// a positive semidefinite matrix; a matrix with a larger entry (of a folded
// element, say) takes the exponent of its largest entry for every row.
template <int N1>
__global__ void k_fx_pack(int ne, const double *__restrict__ src, int2 *__restrict__ dst, short *__restrict__ dexp) {
    constexpr int NA = N1 * N1;
    __shared__ int d[NA], largest, beyond;
    for (int e = blockIdx.x; e < ne; e += gridDim.x) {
        const double *A = src + (size_t)e * NA * NA;
        for (int i = threadIdx.x; i < NA; i += blockDim.x)
            d[i] = (fx_expo(A[(size_t)i * NA + i]) - 1022 + 1) >> 1;   // A_ii < 2^k: half of k, rounded up
        if (threadIdx.x == 0) largest = beyond = 0;
        __syncthreads();
        int big = 0, over = 0;
        for (int q = threadIdx.x; q < NA * NA; q += blockDim.x) {
            const int k = fx_expo(A[q]);
            big = max(big, k);
            over |= k - 1022 > d[q / NA] + d[q % NA];
        }
        atomicMax(&largest, big);
        atomicOr(&beyond, over);
        __syncthreads();
        const bool finite = largest != 0x7ff;
        if (beyond)
            for (int i = threadIdx.x; i < NA; i += blockDim.x) d[i] = (largest - 1022 + 1) >> 1;
        __syncthreads();
        for (int i = threadIdx.x; i < NA; i += blockDim.x) dexp[(size_t)e * NA + i] = finite ? (short)d[i] : FX_BAD;
        int2 *L = dst + (size_t)e * fx_tri_len(NA);
        for (int q = threadIdx.x; q < NA * NA; q += blockDim.x) {
            const int i = q / NA, k = q - (q / NA) * NA;
            if (k <= i)
                L[i * (i + 1) / 2 + k] = finite ? fx_split(__double2ll_rn(scalbn(A[q], FX_ONE - d[i] - d[k]))) : make_int2(0, 0);
        }
        if (NA * (NA + 1) / 2 < fx_tri_len(NA) && threadIdx.x == 0) L[NA * (NA + 1) / 2] = make_int2(0, 0);
        __syncthreads();
    }
}

// per-element V^T M V + U^T S U, the products by the packed matrices (a squared FP64 copy of
// both would hold as much memory as everything else)
template <int N1>
__global__ void __launch_bounds__(nthreads_for(N1 * N1), kVarMinBlocks)
k_var_energy(const __grid_constant__ VarParams P, const double *u, const double *v, double *part) {
    constexpr int NA = N1 * N1;
    extern __shared__ __align__(16) double smraw[];
    const StageSmem<N1, true> s(smraw);
    const int e = blockIdx.x, t = threadIdx.x;
    const size_t at = (size_t)e * NA + (t < NA ? t : 0);
    load_fx<N1>(s.A, P.Sx, e);
    const double U = t < NA ? u[at] : 0.0, V = t < NA ? v[at] : 0.0;
    fx_arrived();
    const double SU = fx_matvec<NA>(s.system(P.Sx, e), U, 0);
    __syncthreads();
    load_fx<N1>(s.A, P.Mx, e);
    fx_arrived();
    const double MV = fx_matvec<NA>(s.system(P.Mx, e), V, 0);
    const double sum = block_sum(t < NA ? V * MV + U * SU : 0.0, s.red);
    if (t == 0) part[e] = sum;
}

__global__ void k_var_sum(int n, const double *part, double *out) {
    __shared__ double red[1024];
    const int t = threadIdx.x;
    double s = 0.0;
    for (int i = t; i < n; i += blockDim.x) s += part[i];
    red[t] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (t < w) red[t] += red[t + w];
        __syncthreads();
    }
    if (t == 0) out[0] = 0.5 * red[0];
}

}  // namespace
