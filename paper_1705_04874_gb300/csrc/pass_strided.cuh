// Launch and shared-memory opt-in of the y / z passes with V floats per global
// access (pass_strided<RA, RB, RC, T, V>): one translation unit per V, so that they
// compile beside one another.
#pragma once
#include "fft_pass.cuh"
#include "pass_plans.h"

namespace es {

template <int RA, int RB, int RC, int T, int V>
static cudaError_t launch_strided_plan(int ntiles, const PassParams& p, cudaStream_t st)
{
    constexpr int threads = pass_threads<T>();
    constexpr size_t smem = pass_smem_strided<RA * RB * RC, T>();
    int grid = 0;
    const cudaError_t e = persistent_grid(pass_strided<RA, RB, RC, T, V>, threads, smem, ntiles * p.njobs, &grid);
    if (e != cudaSuccess) return e;
    return launch_pass_kernel(pass_strided<RA, RB, RC, T, V>, dim3((unsigned)grid), threads, smem, st, p, ntiles);
}

template <int V>
static cudaError_t launch_strided_plans(int ra, int rb, int rc, int ntiles, const PassParams& p, cudaStream_t st)
{
#define ES_CASE(n, a, b, c, t)                                                                               \
    if (ra == a && rb == b && rc == c) return launch_strided_plan<a, b, c, t, V>(ntiles, p, st);
    ES_PLANS(ES_CASE)
#undef ES_CASE
    return cudaErrorInvalidValue;
}

template <int V>
static cudaError_t prepare_strided_plans()
{
    cudaError_t e;
#define ES_PREP(n, a, b, c, t)                                                                               \
    if ((e = cudaFuncSetAttribute(pass_strided<a, b, c, t, V>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                  (int)pass_smem_strided<n, t>())) != cudaSuccess)                              \
        return e;
    ES_PLANS(ES_PREP)
#undef ES_PREP
    return cudaSuccess;
}

}  // namespace es
