// Launch and shared-memory opt-in of the y / z passes with V floats per global
// access (pass_strided<RA, RB, RC, T, V>): one translation unit per V, so that they
// compile beside one another.
#pragma once
#include "fft_pass.cuh"
#include "pass_plans.h"

namespace es {

// Whether an axis of n cells with stage radices ra, rb, ... takes one tile per CTA instead of the persistent
// kernel: short pencils are too little work to hide behind (a tile of 16 cells is 2 KB), and the odd lengths
// want many threads and a third shared tile for the near parts, which leaves two CTAs on an SM.  At 64
// cells the wide copies of an nx that is a multiple of four decide.  ps per cell, the four y and z passes of
// a step on batches of 8 M cells, persistent -> one tile per CTA (the kernel before the persistent one), nx =
// 62, 64 and 63: 16 70.5 -> 59.5 (65.8), 69.6 -> 57.6 (64.0), 76.1 -> 62.7 (80.9); 32 63.9 -> 55.3 (63.2), 56.3
// -> 54.3 (61.4), 69.1 -> 59.1 (86.9); 48 56.7 -> 52.2 (59.1), 54.0 -> 50.9 (57.8), 62.8 -> 58.7 (88.9); 64 57.1
// -> 53.5 (59.5), 48.4 and 50.9, 61.0 -> 59.0 (99.6); 75 74.0 -> 66.1 (67.9), 68.3 -> 65.4 (67.5), 76.9 -> 70.0
// (83.5); 125 79.8 -> 61.3 (63.3), 76.1 -> 60.8 (62.1), 77.6 -> 66.0 (75.5).  At 80 cells the persistent one
// wins, 62.0 and 70.7, 53.4 and 69.4, 64.5 and 74.8, and from there on.  A plan whose first radix is the
// smaller (more threads on a tile than it keeps busy) or 25 stays with it too: 48 = 4 x 12 53.4 and 64.5 at
// nx = 64, 125 = 25 x 5 63.2 and 80.4.
constexpr bool one_tile(int n, int ra, int rb, int nx)
{
    return n % 2 ? ra < 25 : ra >= rb && (n < 64 || (n == 64 && nx % 4 != 0));
}

// ... unless all tiles fit on the device at once: then there is nothing to overlap, and the second trip to L2
// for the stencil is what the one-tile kernel waits for.  us a step, one tile per CTA and persistent (tiles x
// jobs of a y or z pass): 32^3 (96) 32.9 and 30.5, eight of them (768) 48.4 and 41.8, 32 (3072, past one round)
// 98.3 and 116.1; 48^3 (288) 48.3 and 45.0, two (576) 53.4 and 47.7, eight (2304, past it) 78.8 and 104.7; 64 x 64
// x 62 (384) 89.9 and 77.0, four (1536) 129.2 and 126.4, eight 234 and 238; 16^3 21.8 and 21.3.  Below 48 cells a
// tile of few columns costs the persistent kernel more than that (32 x 32 x 34, two (384) 55.2 and 56.2, eight
// 67.2 and 72.2), unless there are no more than two tiles per SM (one (192) 53.5 and 47.2).
constexpr bool short_of_tiles(int n, int nx, int units, int sms)
{
    return n % 2 == 0 && (n >= 48 || nx % 32 == 0 || units <= 2 * sms);
}

template <int RA, int RB, int RC, int T, int V>
static cudaError_t launch_strided_plan(int ntiles, const PassParams& p, cudaStream_t st)
{
    constexpr int N = RA * RB * RC;
    const int units = ntiles * p.njobs;
    bool once = one_tile(N, RA, RB, p.nx);
    if constexpr (N % 2 == 0 || !one_tile(N, RA, RB, V)) {
        constexpr int threads = pass_threads<T>();
        constexpr size_t smem = pass_smem_strided<N, T>();
        int grid = 0, dev = 0, sms = 0;
        cudaError_t e = persistent_grid(pass_strided<RA, RB, RC, T, V>, threads, smem, units, &grid);
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (once && grid == units && short_of_tiles(N, p.nx, units, sms)) once = false;
        if (!once)
            return launch_pass_kernel(pass_strided<RA, RB, RC, T, V>, dim3((unsigned)grid), threads, smem, st, p, ntiles);
    }
    if constexpr (one_tile(N, RA, RB, V))
        return launch_pass_kernel(pass_strided_once<RA, RB, RC, V>, dim3((unsigned)ntiles, (unsigned)p.njobs),
                                  once_threads<RA, RB, RC>(), once_smem<RA, RB, RC>(), st, p, ntiles);
    return cudaErrorInvalidValue;
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
    cudaError_t e = cudaSuccess;
#define ES_PREP(n, a, b, c, t)                                                                               \
    if constexpr (n % 2 == 0 || !one_tile(n, a, b, V))                                                        \
        if (e == cudaSuccess)                                                                                 \
            e = cudaFuncSetAttribute(pass_strided<a, b, c, t, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                     (int)pass_smem_strided<n, t>());
    ES_PLANS(ES_PREP)
#undef ES_PREP
    return e;
}

}  // namespace es
