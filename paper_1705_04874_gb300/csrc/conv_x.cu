// Choice of the transform length, the x convolution pass and the launch of all
// convolution passes (conv_pass.cuh).
#include "conv_pass.cuh"

namespace es {

int conv_length(int n, int axis)
{
    if (n < CONV_MIN_N || (axis == 0 && n % 2 && n < CONV_MIN_ODD_X)) return 0;
    // the plans in ascending order: the first with room for the zero padding
#define ES_CASE(len, a, b, c, t, pr) if (2 * n <= len) return len;
    ES_CONV_PLANS(ES_CASE)
#undef ES_CASE
    return 0;
}

template <int RA, int RB, int RC, int T, int PR>
static cudaError_t launch_conv_x(const PassParams& p, cudaStream_t st)
{
    constexpr int W = 2 * PR;
    const int ntiles = (p.ny * p.nz + W - 1) / W * p.nsim;
    return launch_pass_kernel(conv_x<RA, RB, RC, T, PR>, dim3((unsigned)ntiles, (unsigned)p.njobs),
                              conv_threads<T, PR>(), conv_smem_x<RA * RB * RC, PR>(p.n), st, p);
}

cudaError_t prepare_conv_kernels()
{
    cudaError_t e;
#define ES_PREP(len, a, b, c, t, pr)                                                                        \
    if ((e = cudaFuncSetAttribute(conv_x<a, b, c, t, pr>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                                  (int)conv_smem_x<len, pr>(len / 2))) != cudaSuccess)                \
        return e;
    ES_CONV_PLANS(ES_PREP)
#undef ES_PREP
    if ((e = prepare_conv_strided1()) != cudaSuccess) return e;
    return prepare_conv_strided2();
}

cudaError_t launch_conv(const PassParams& p, cudaStream_t st)
{
    if (p.axis != 0) return p.nx % 2 ? launch_conv_strided1(p, st) : launch_conv_strided2(p, st);
#define ES_CASE(len, a, b, c, t, pr) if (p.m == len) return launch_conv_x<a, b, c, t, pr>(p, st);
    ES_CONV_PLANS(ES_CASE)
#undef ES_CASE
    return cudaErrorInvalidValue;
}

}  // namespace es
