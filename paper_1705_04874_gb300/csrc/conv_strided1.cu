// The y and z convolution passes for an odd nx (a translation unit per variant, so
// that they compile beside one another).
#include "conv_pass.cuh"

namespace es {

cudaError_t launch_conv_strided1(const PassParams& p, cudaStream_t st)
{
#define ES_CASE(len, a, b, c, t, pr) if (p.m == len) return launch_conv_strided<a, b, c, t, pr, 1>(p, st);
    ES_CONV_PLANS(ES_CASE)
#undef ES_CASE
    return cudaErrorInvalidValue;
}

cudaError_t prepare_conv_strided1()
{
    cudaError_t e;
#define ES_PREP(len, a, b, c, t, pr) if ((e = prepare_conv_strided<a, b, c, t, pr, 1>()) != cudaSuccess) return e;
    ES_CONV_PLANS(ES_PREP)
#undef ES_PREP
    return cudaSuccess;
}

}  // namespace es
