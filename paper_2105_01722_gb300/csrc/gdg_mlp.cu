// Learned initial guess for the element u_t solve: a three-layer perceptron
// (162 -> 64 -> 64 -> 81, tanh) with BF16 weights and FP32 accumulation,
// and its training kernels (a pattern layered on the element PCG of
// Section 7.1; the paper has no learned component).
//
// Parameter block (FP32 master copy, in this order):
//   W1 [64][162], b1 [64], W2 [64][64], b2 [64], W3 [81][64], b3 [81]
// BF16 working weights: W1, W2, W3 in the same order (biases stay FP32).
// Features of an element (162 FP32): c^2 / mean(c^2) at the 81 nodes, then
// r_u / ||r_u||; output: a guess of y / ||r_u|| for (S_c2 + w w^T) y = r_u.
//
// Kernels
//   k_mlp_forward   Y = net(X) for B samples
//   k_mlp_samples   forward and backward pass of every sample of a minibatch:
//                   its activations, the errors at its layers, its loss
//   k_mlp_grad      gradients and loss from those, summed in a fixed order
//   k_mlp_adam      Adam update of the master copy, refresh of the BF16 copy
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>

#include "gdg_internal.h"

namespace {

constexpr int IN = GDG_MLP_IN, HID = GDG_MLP_HID, OUT = GDG_MLP_OUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + HID * IN, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID;
constexpr int OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + OUT * HID, NPARAM = OFF_B3 + OUT;
constexpr int WB_W1 = 0, WB_W2 = HID * IN, WB_W3 = WB_W2 + HID * HID, NWEIGHT = WB_W3 + OUT * HID;
static_assert(NPARAM == GDG_MLP_NPARAM, "parameter count");
static_assert(NWEIGHT == GDG_MLP_NWEIGHT, "weight count");

// Weights in shared memory: BF16 rows padded to 16 bytes more than a multiple
// of 128, so that the 16-byte reads of the 8 lanes of a phase (one row each)
// fall on different banks; rows of W1 are padded with zeros to 168 inputs.
constexpr int KP = 168, S1 = KP, S2 = 72, S3 = 72;
constexpr int SW1 = 0, SW2 = SW1 + HID * S1, SW3 = SW2 + HID * S2, SWEND = SW3 + OUT * S3;
static_assert((S1 * 2) % 16 == 0 && (S2 * 2) % 16 == 0, "16-byte rows");
constexpr int MAXOUT = 88;   // OUT rounded up to a multiple of 8

// shared memory of a block with S samples
template <int S>
struct MlpSmem {
    __nv_bfloat16 *w;
    float *b1, *b2, *b3, *x, *h1, *h2, *y;
    __device__ MlpSmem(float *base) {
        w = reinterpret_cast<__nv_bfloat16 *>(base);
        b1 = base + SWEND / 2;
        b2 = b1 + HID;
        b3 = b2 + HID;
        x = b3 + MAXOUT;
        h1 = x + S * KP;
        h2 = h1 + S * HID;
        y = h2 + S * HID;
    }
    __host__ __device__ static constexpr size_t floats() { return SWEND / 2 + 2 * HID + MAXOUT + S * (KP + 2 * HID + MAXOUT); }
};
static_assert(SWEND % 8 == 0, "16-byte aligned floats behind the weights");

__device__ __forceinline__ void copy_async(void *dst, const void *src) {   // 4 bytes
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copies_done() {   // the caller's next barrier shows them to the block
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// weights and biases into shared memory (rows of 2-byte pairs: IN, HID are even);
// the caller waits with copies_done and a barrier
__device__ __forceinline__ void load_net(const __nv_bfloat16 *wb, const float *params, __nv_bfloat16 *w, float *b1,
                                         float *b2, float *b3) {
    if (reinterpret_cast<uintptr_t>(wb) & 3) {   // BF16s that do not start on a word: one at a time
        for (int i = threadIdx.x; i < HID * KP; i += blockDim.x)
            w[i] = i % KP < IN ? wb[i / KP * IN + i % KP] : __float2bfloat16(0.f);
        for (int i = threadIdx.x; i < (HID + OUT) * HID; i += blockDim.x) w[SW2 + i / HID * S2 + i % HID] = wb[WB_W2 + i];
    } else {   // word by word, asynchronously: every copy in flight at once, no register round trip
        const unsigned *src = reinterpret_cast<const unsigned *>(wb);
        unsigned *dst = reinterpret_cast<unsigned *>(w);
        for (int i = threadIdx.x; i < HID * KP / 2; i += blockDim.x) {
            const int j = i / (KP / 2), k = i - j * (KP / 2);
            if (k < IN / 2) copy_async(dst + i, src + j * (IN / 2) + k);
            else dst[i] = 0u;
        }
        for (int i = threadIdx.x; i < (HID + OUT) * (HID / 2); i += blockDim.x) {   // W2 and W3: rows of HID
            const int j = i / (HID / 2), k = i - j * (HID / 2);
            copy_async(dst + SW2 / 2 + j * (S2 / 2) + k, src + WB_W2 / 2 + i);
        }
    }
    for (int i = threadIdx.x; i < HID; i += blockDim.x) {
        b1[i] = params[OFF_B1 + i];
        b2[i] = params[OFF_B2 + i];
    }
    for (int i = threadIdx.x; i < OUT; i += blockDim.x) b3[i] = params[OFF_B3 + i];
}

// acc[n] += sum_k W[k] in[n][k] for the NS samples of a thread: 8 weights a
// read, two partial sums a sample
template <int K, int NS>
__device__ __forceinline__ void dot_rows(const __nv_bfloat16 *W, const float *in, int stride, float (&acc)[NS]) {
    float odd[NS];
#pragma unroll
    for (int n = 0; n < NS; ++n) odd[n] = 0.f;
#pragma unroll 3
    for (int k = 0; k < K; k += 8) {
        const uint4 w4 = *reinterpret_cast<const uint4 *>(W + k);
        const unsigned u[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int n = 0; n < NS; ++n) {
            const float4 p = *reinterpret_cast<const float4 *>(in + n * stride + k);
            const float4 q = *reinterpret_cast<const float4 *>(in + n * stride + k + 4);
            const float v[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {   // a BF16 is the upper half of a float
                acc[n] = fmaf(__uint_as_float(u[i] << 16), v[2 * i], acc[n]);
                odd[n] = fmaf(__uint_as_float(u[i] & 0xffff0000u), v[2 * i + 1], odd[n]);
            }
        }
    }
#pragma unroll
    for (int n = 0; n < NS; ++n) acc[n] += odd[n];
}

// forward pass of the block's S samples in s.x: h1, h2, y.  Thread t: neuron
// t % 64 (and the 17 outputs above 64 in a second turn) of the NS samples of
// group t / 64.
template <int S, int NS>
__device__ __forceinline__ void forward_tile(const MlpSmem<S> &s) {
    const int j = threadIdx.x & 63, n0 = (threadIdx.x >> 6) * NS;
    float a[NS];
#pragma unroll
    for (int n = 0; n < NS; ++n) a[n] = s.b1[j];
    dot_rows<KP, NS>(s.w + SW1 + j * S1, s.x + n0 * KP, KP, a);
#pragma unroll
    for (int n = 0; n < NS; ++n) { s.h1[(n0 + n) * HID + j] = tanhf(a[n]); a[n] = s.b2[j]; }
    __syncthreads();
    dot_rows<HID, NS>(s.w + SW2 + j * S2, s.h1 + n0 * HID, HID, a);
#pragma unroll
    for (int n = 0; n < NS; ++n) s.h2[(n0 + n) * HID + j] = tanhf(a[n]);
    __syncthreads();
    for (int o = j; o < OUT; o += 64) {
#pragma unroll
        for (int n = 0; n < NS; ++n) a[n] = s.b3[o];
        dot_rows<HID, NS>(s.w + SW3 + o * S3, s.h2 + n0 * HID, HID, a);
#pragma unroll
        for (int n = 0; n < NS; ++n) s.y[(n0 + n) * MAXOUT + o] = a[n];
    }
    __syncthreads();
}

// inference: 16 samples a block, 4 a thread, so that a weight read serves 4
constexpr int SPB = 16, THREADS = 256;

__global__ void __launch_bounds__(THREADS)
k_mlp_forward(const __nv_bfloat16 *wb, const float *params, const float *X, int B, float *Y) {
    extern __shared__ __align__(16) float smf[];
    const MlpSmem<SPB> s(smf);
    load_net(wb, params, s.w, s.b1, s.b2, s.b3);
    const int n0 = blockIdx.x * SPB, ns = min(SPB, B - n0);
    for (int i = threadIdx.x; i < SPB * KP; i += blockDim.x) {
        const int n = i / KP, k = i - n * KP;
        s.x[i] = n < ns && k < IN ? X[(size_t)(n0 + n) * IN + k] : 0.f;
    }
    copies_done();
    __syncthreads();
    forward_tile<SPB, 4>(s);
    for (int i = threadIdx.x; i < ns * OUT; i += blockDim.x) Y[(size_t)n0 * OUT + i] = s.y[i / OUT * MAXOUT + i % OUT];
}

// One minibatch: two kernels.  (One block of 32 samples computing its share of
// every gradient left 144 of 152 SMs idle at 256 samples, and its weight reads,
// 64 floats apart, hit one bank: 103 us.  An iteration of 256 samples, both
// kernels and Adam: 100 us then, 36 with plain loads of the weights, 29.6 now.)
//
// k_mlp_samples: 2 samples a block, so that 256 samples use 128 SMs.  Record of
// a sample in `rec`: h1, h2, g1, g2, g3 (the errors before the layers'
// activations), loss.
constexpr int SPT = 2, TTHREADS = 128;
constexpr int R_H1 = 0, R_H2 = HID, R_G1 = 2 * HID, R_G2 = 3 * HID, R_G3 = 4 * HID, R_LOSS = R_G3 + OUT, REC = R_LOSS + 1;
constexpr int PART = 32;     // samples a unit of the caller's buffer is counted in (gdg_mlp_partial_len)
static_assert(PART * REC <= NPARAM + 1, "records fit the caller's buffer");

__global__ void __launch_bounds__(TTHREADS)
k_mlp_samples(const __nv_bfloat16 *wb, const float *params, const float *X, const float *T, const int *idx, int B,
              float *rec) {
    extern __shared__ __align__(16) float smf[];
    const MlpSmem<SPT> s(smf);
    float *g3 = smf + MlpSmem<SPT>::floats(), *g2 = g3 + SPT * MAXOUT;
    load_net(wb, params, s.w, s.b1, s.b2, s.b3);
    const int n0 = blockIdx.x * SPT;
    for (int i = threadIdx.x; i < SPT * KP; i += blockDim.x) {
        const int n = i / KP, k = i - n * KP;
        s.x[i] = n0 + n < B && k < IN ? X[(size_t)(idx ? idx[n0 + n] : n0 + n) * IN + k] : 0.f;
    }
    copies_done();
    __syncthreads();
    forward_tile<SPT, 1>(s);
    const int n = threadIdx.x >> 6, j = threadIdx.x & 63;
    const bool valid = n0 + n < B;
    float *out = rec + (size_t)(n0 + n) * REC;
    // g3 = 2 (yhat - t) / B, and the sample's share of the loss
    for (int o = j; o < OUT; o += 64) {
        const float d = valid ? s.y[n * MAXOUT + o] - T[(size_t)(idx ? idx[n0 + n] : n0 + n) * OUT + o] : 0.f;
        s.y[n * MAXOUT + o] = d * d;
        const float g = 2.f * d / (float)B;
        g3[n * MAXOUT + o] = g;
        if (valid) out[R_G3 + o] = g;
    }
    __syncthreads();
    // g2 = (g3 W3) (1 - h2^2)
    const __nv_bfloat16 *w3 = s.w + SW3 + j;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll 3
    for (int o = 0; o < OUT; o += 3) {
        a0 = fmaf(g3[n * MAXOUT + o], __bfloat162float(w3[o * S3]), a0);
        a1 = fmaf(g3[n * MAXOUT + o + 1], __bfloat162float(w3[(o + 1) * S3]), a1);
        a2 = fmaf(g3[n * MAXOUT + o + 2], __bfloat162float(w3[(o + 2) * S3]), a2);
    }
    const float h2 = s.h2[n * HID + j], h1 = s.h1[n * HID + j];
    const float e2 = (a0 + a1 + a2) * (1.f - h2 * h2);
    g2[n * HID + j] = e2;
    __syncthreads();
    // g1 = (g2 W2) (1 - h1^2)
    const __nv_bfloat16 *w2 = s.w + SW2 + j;
    a0 = a1 = 0.f;
#pragma unroll 4
    for (int k = 0; k < HID; k += 2) {
        a0 = fmaf(g2[n * HID + k], __bfloat162float(w2[k * S2]), a0);
        a1 = fmaf(g2[n * HID + k + 1], __bfloat162float(w2[(k + 1) * S2]), a1);
    }
    if (valid) {
        out[R_H1 + j] = h1;
        out[R_H2 + j] = h2;
        out[R_G1 + j] = (a0 + a1) * (1.f - h1 * h1);
        out[R_G2 + j] = e2;
    }
    if (j < 32) {   // the first warp of the sample's two (OUT <= 96)
        float l = s.y[n * MAXOUT + j] + s.y[n * MAXOUT + 32 + j] + (64 + j < OUT ? s.y[n * MAXOUT + 64 + j] : 0.f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (valid && j == 0) out[R_LOSS] = l / (float)B;
    }
}
static_assert(OUT % 3 == 0 && HID % 2 == 0, "unrolled sums");

// k_mlp_grad: dW = sum over the samples of (error) x (input of the layer), 16 x
// 16 entries a block.  Four groups of 64 threads (4 entries a thread) take the
// samples 32 at a time in turn, the next 32 on their way from L2 meanwhile (a
// single group spent 8 load latencies in a row at 256 samples: 26 us); the
// groups' sums are added in order.  The first input column's blocks also sum
// the bias, the last block the loss.  Fixed order: deterministic.
constexpr int GT = 16, GN = 32, GG = 4;
__host__ __device__ constexpr int tiles(int n) { return (n + GT - 1) / GT; }
constexpr int T1 = tiles(HID) * tiles(IN), T2 = tiles(HID) * tiles(HID), T3 = tiles(OUT) * tiles(HID);

__global__ void __launch_bounds__(64 * GG)
k_mlp_grad(const float *X, const int *idx, const float *rec, int B, float *grad, float *loss) {
    constexpr int LD = GN * GT / 64;   // values of a stage per thread
    __shared__ float E[GG][GN][GT], I[GG][GN][GT];
    __shared__ float part[GG][GT * GT + GT];
    const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
    int tile = blockIdx.x;
    if (tile == T1 + T2 + T3) {   // loss: partial sums, then in order
        float l = 0.f;
        for (int n = threadIdx.x; n < B; n += 64 * GG) l += rec[(size_t)n * REC + R_LOSS];
        part[0][threadIdx.x] = l;
        __syncthreads();
        if (threadIdx.x < 32) {
            float a = 0.f;
            for (int i = 0; i < 64 * GG / 32; ++i) a += part[0][threadIdx.x + 32 * i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (threadIdx.x == 0) *loss = a;
        }
        return;
    }
    int rows, cols, re, ri, ow, ob;   // outputs, inputs, where errors and inputs lie in a record, in grad
    if (tile < T1) { rows = HID; cols = IN; re = R_G1; ri = -1; ow = OFF_W1; ob = OFF_B1; }
    else if (tile < T1 + T2) { tile -= T1; rows = HID; cols = HID; re = R_G2; ri = R_H1; ow = OFF_W2; ob = OFF_B2; }
    else { tile -= T1 + T2; rows = OUT; cols = HID; re = R_G3; ri = R_H2; ow = OFF_W3; ob = OFF_B3; }
    const int tc = tiles(cols), r0 = (tile / tc) * GT, c0 = (tile - (tile / tc) * tc) * GT;
    const int r = (t >> 3) * 2, c = (t & 7) * 2;   // this thread's 2 x 2 entries
    float a[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, bias[2] = {0.f, 0.f};
    float e[LD], in[LD];
    const int k = t % GT, n1 = t / GT;             // this thread's loads: column k of samples n1 + 4 i
    auto load = [&](int b0) {
#pragma unroll
        for (int i = 0; i < LD; ++i) {
            const int n = b0 + n1 + (64 / GT) * i;
            e[i] = n < B && r0 + k < rows ? rec[(size_t)n * REC + re + r0 + k] : 0.f;
            in[i] = n < B && c0 + k < cols
                        ? (ri < 0 ? X[(size_t)(idx ? idx[n] : n) * IN + c0 + k] : rec[(size_t)n * REC + ri + c0 + k])
                        : 0.f;
        }
    };
    load(g * GN);
    for (int b0 = 0; b0 < B; b0 += GG * GN) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < LD; ++i) {
            E[g][n1 + (64 / GT) * i][k] = e[i];
            I[g][n1 + (64 / GT) * i][k] = in[i];
        }
        __syncthreads();
        if (b0 + GG * GN < B) load(b0 + GG * GN + g * GN);
#pragma unroll 8
        for (int n = 0; n < GN; ++n) {
            const float2 ev = *reinterpret_cast<const float2 *>(&E[g][n][r]), iv = *reinterpret_cast<const float2 *>(&I[g][n][c]);
            a[0][0] = fmaf(ev.x, iv.x, a[0][0]);
            a[0][1] = fmaf(ev.x, iv.y, a[0][1]);
            a[1][0] = fmaf(ev.y, iv.x, a[1][0]);
            a[1][1] = fmaf(ev.y, iv.y, a[1][1]);
            bias[0] += ev.x;
            bias[1] += ev.y;
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int q = 0; q < 2; ++q) part[g][(r + i) * GT + c + q] = a[i][q];
        if (c == 0) part[g][GT * GT + r + i] = bias[i];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < GT * GT + GT; q += 64 * GG) {
        float s = part[0][q];
#pragma unroll
        for (int i = 1; i < GG; ++i) s += part[i][q];
        const int row = q < GT * GT ? q / GT : q - GT * GT, col = q % GT;
        if (r0 + row >= rows) continue;
        if (q < GT * GT) {
            if (c0 + col < cols) grad[ow + (r0 + row) * cols + c0 + col] = s;
        } else if (c0 == 0) {
            grad[ob + r0 + row] = s;
        }
    }
}

__global__ void k_mlp_adam(float *params, float *m, float *v, const float *grad, float lr, float b1, float b2,
                           float eps, float c1, float c2, __nv_bfloat16 *wb) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NPARAM) return;
    const float g = grad[p];
    const float mm = b1 * m[p] + (1.f - b1) * g;
    const float vv = b2 * v[p] + (1.f - b2) * g * g;
    m[p] = mm;
    v[p] = vv;
    const float x = params[p] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    params[p] = x;
    // refresh the BF16 working copy of the weights
    int w = -1;
    if (p < OFF_B1) w = WB_W1 + (p - OFF_W1);
    else if (p >= OFF_W2 && p < OFF_B2) w = WB_W2 + (p - OFF_W2);
    else if (p >= OFF_W3 && p < OFF_B3) w = WB_W3 + (p - OFF_W3);
    if (w >= 0) wb[w] = __float2bfloat16_rn(x);
}

__global__ void k_mlp_to_bf16(const float *params, __nv_bfloat16 *wb) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NPARAM) return;
    int w = -1;
    if (p < OFF_B1) w = WB_W1 + (p - OFF_W1);
    else if (p >= OFF_W2 && p < OFF_B2) w = WB_W2 + (p - OFF_W2);
    else if (p >= OFF_W3 && p < OFF_B3) w = WB_W3 + (p - OFF_W3);
    if (w >= 0) wb[w] = __float2bfloat16_rn(params[p]);
}

// Learned u_t guess for every element: x0 = ||r_u|| net([c2feat, r_u/||r_u||]).
__global__ void __launch_bounds__(THREADS)
k_mlp_guess(const __nv_bfloat16 *wb, const float *params, const float *c2feat, const double *ru, int ne,
            double *x0u) {
    extern __shared__ __align__(16) float smf[];
    const MlpSmem<SPB> s(smf);
    float *nrm = smf + MlpSmem<SPB>::floats();     // [SPB]
    load_net(wb, params, s.w, s.b1, s.b2, s.b3);
    const int n0 = blockIdx.x * SPB, ns = min(SPB, ne - n0);
    if (threadIdx.x < SPB) {
        double a = 0.0;
        if ((int)threadIdx.x < ns)
            for (int k = 0; k < OUT; ++k) {
                const double r = ru[(size_t)(n0 + threadIdx.x) * OUT + k];
                a += r * r;
            }
        nrm[threadIdx.x] = (float)sqrt(a);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SPB * KP; i += blockDim.x) {
        const int n = i / KP, k = i - n * KP;
        float x = 0.f;
        if (n < ns && k < IN) {
            if (k < OUT) x = c2feat[(size_t)(n0 + n) * OUT + k];
            else if (nrm[n] > 0.f) x = (float)(ru[(size_t)(n0 + n) * OUT + (k - OUT)] / (double)nrm[n]);
        }
        s.x[i] = x;
    }
    copies_done();
    __syncthreads();
    forward_tile<SPB, 4>(s);
    for (int i = threadIdx.x; i < ns * OUT; i += blockDim.x)
        x0u[(size_t)n0 * OUT + i] = (double)nrm[i / OUT] * s.y[i / OUT * MAXOUT + i % OUT];
}

// training rows: X = [c2feat, r_u/||r_u||] (FP32) and, when y is given,
// T = y/||r_u|| (FP32); one thread per element
__global__ void k_mlp_rows(const float *c2feat, const double *ru, const double *y, int ne, float *X, float *T) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ne) return;
    double a = 0.0;
    for (int k = 0; k < OUT; ++k) {
        const double r = ru[(size_t)e * OUT + k];
        a += r * r;
    }
    const double n = sqrt(a), inv = n > 0.0 ? 1.0 / n : 0.0;
    for (int k = 0; k < OUT; ++k) {
        X[(size_t)e * IN + k] = c2feat[(size_t)e * OUT + k];
        X[(size_t)e * IN + OUT + k] = (float)(ru[(size_t)e * OUT + k] * inv);
        if (y && T) T[(size_t)e * OUT + k] = (float)(y[(size_t)e * OUT + k] * inv);
    }
}

size_t fwd_smem() { return MlpSmem<SPB>::floats() * sizeof(float); }
size_t guess_smem() { return (MlpSmem<SPB>::floats() + SPB) * sizeof(float); }
size_t samples_smem() { return (MlpSmem<SPT>::floats() + SPT * (MAXOUT + HID)) * sizeof(float); }

bool attrs_done = false;
int set_attrs() {
    if (attrs_done) return GDG_OK;
    if (cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd_smem()) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_samples, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)samples_smem()) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_guess, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)guess_smem()) != cudaSuccess)
        return GDG_ECUDA;
    attrs_done = true;
    return GDG_OK;
}

}  // namespace

int gdg_mlp_guess_launch(const uint16_t *w_bf16, const float *params, const float *c2feat, const double *ru,
                         int ne, double *x0u, cudaStream_t s) {
    if (set_attrs()) return GDG_ECUDA;
    k_mlp_guess<<<(ne + SPB - 1) / SPB, THREADS, guess_smem(), s>>>(
        reinterpret_cast<const __nv_bfloat16 *>(w_bf16), params, c2feat, ru, ne, x0u);
    return GDG_OK;
}

int gdg_mlp_rows_launch(const float *c2feat, const double *ru, const double *y, int ne, float *X, float *T,
                        cudaStream_t s) {
    k_mlp_rows<<<(ne + 127) / 128, 128, 0, s>>>(c2feat, ru, y, ne, X, T);
    return GDG_OK;
}

extern "C" int gdg_mlp_forward(const uint16_t *w_bf16, const float *params, const float *X, int B, float *Y,
                               void *stream) {
    if (!w_bf16 || !params || !X || !Y || B < 0) return GDG_EINVAL;
    if (B == 0) return GDG_OK;
    if (set_attrs()) return GDG_ECUDA;
    const int grid = (B + SPB - 1) / SPB;
    k_mlp_forward<<<grid, THREADS, fwd_smem(), (cudaStream_t)stream>>>(
        reinterpret_cast<const __nv_bfloat16 *>(w_bf16), params, X, B, Y);
    return cudaGetLastError() == cudaSuccess ? GDG_OK : GDG_ECUDA;
}

extern "C" long long gdg_mlp_partial_len(int B) {
    return B <= 0 ? 0 : (long long)((B + PART - 1) / PART) * (NPARAM + 1);
}

extern "C" int gdg_mlp_backward(const uint16_t *w_bf16, const float *params, const float *X, const float *T,
                                const int *idx, int B, float *partial, float *grad, float *loss, void *stream) {
    if (!w_bf16 || !params || !X || !T || !partial || !grad || !loss || B <= 0) return GDG_EINVAL;
    if (set_attrs()) return GDG_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    k_mlp_samples<<<(B + SPT - 1) / SPT, TTHREADS, samples_smem(), s>>>(
        reinterpret_cast<const __nv_bfloat16 *>(w_bf16), params, X, T, idx, B, partial);
    k_mlp_grad<<<T1 + T2 + T3 + 1, 64 * GG, 0, s>>>(X, idx, partial, B, grad, loss);
    return cudaGetLastError() == cudaSuccess ? GDG_OK : GDG_ECUDA;
}

extern "C" int gdg_mlp_adam(float *params, float *m, float *v, const float *grad, int step, float lr,
                            uint16_t *w_bf16, void *stream) {
    if (!params || !m || !v || !grad || !w_bf16 || step < 1 || !(lr > 0.f)) return GDG_EINVAL;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
    k_mlp_adam<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
        params, m, v, grad, lr, b1, b2, eps, c1, c2, reinterpret_cast<__nv_bfloat16 *>(w_bf16));
    return cudaGetLastError() == cudaSuccess ? GDG_OK : GDG_ECUDA;
}

extern "C" int gdg_mlp_to_bf16(const float *params, uint16_t *w_bf16, void *stream) {
    if (!params || !w_bf16) return GDG_EINVAL;
    k_mlp_to_bf16<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
        params, reinterpret_cast<__nv_bfloat16 *>(w_bf16));
    return cudaGetLastError() == cudaSuccess ? GDG_OK : GDG_ECUDA;
}
