// Host entry points of the element kernels of one N1 (VarOps): what each
// gdg_var_n*.cu instantiates.
#pragma once

#include "gdg_var_kernels.cuh"

namespace {

template <int N1>
struct VarLaunch {
    static constexpr bool STAGED = staged_lifts(N1, 1 << 30, 1);   // on meshes of some size
    // The dynamic shared-memory limit is a property of the kernel function, shared
    // by every context: always raised to the device's opt-in maximum so that a
    // context with smaller needs cannot lower it under another one.
    static void attrs(int lim) {
        cudaFuncSetAttribute(k_var_stage<N1, ROUTE_ANY>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_var_stage<N1, ROUTE_MIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        if constexpr (STAGED) cudaFuncSetAttribute(k_var_stage<N1, ROUTE_INVERSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_var_pcg<N1, ROUTE_ANY>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_var_pcg<N1, ROUTE_MIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    }
    static void stage(const VarParams &P, size_t sm, int mode, const VarBufs &b, double cA, double cY, cudaStream_t s) {
        const dim3 grid(P.ne), block(nthreads_for(N1 * N1));   // one block per element
        if constexpr (STAGED) {
            if (P.staged) {
                k_var_stage<N1, ROUTE_INVERSE><<<grid, block, sm, s>>>(P, b, mode, cA, cY);
                return;
            }
        }
        (P.mixed ? k_var_stage<N1, ROUTE_MIXED> : k_var_stage<N1, ROUTE_ANY>)<<<grid, block, sm, s>>>(P, b, mode, cA, cY);
    }
    static void pcg(const VarParams &P, size_t sm, int which, const double *b, double *x, int *iters, double *rel,
                    int *sweeps, cudaStream_t s) {
        (P.mixed ? k_var_pcg<N1, ROUTE_MIXED> : k_var_pcg<N1, ROUTE_ANY>)<<<P.ne, nthreads_for(N1 * N1), sm, s>>>(P, which, b, x, iters, rel, sweeps);
    }
};

GDG_CHECKS_READER(var_unit_checks)

}  // namespace

#define GDG_VAR_OPS(n) \
    extern const VarOps var_ops_##n = {VarLaunch<n>::attrs, VarLaunch<n>::stage, VarLaunch<n>::pcg, var_unit_checks};
