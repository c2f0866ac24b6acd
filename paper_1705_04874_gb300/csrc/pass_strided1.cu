// The y and z derivative passes for an odd nx.
#include "pass_strided.cuh"

namespace es {

cudaError_t launch_strided1(int ra, int rb, int rc, int ntiles, const PassParams& p, cudaStream_t st)
{
    return launch_strided_plans<1>(ra, rb, rc, ntiles, p, st);
}
cudaError_t prepare_strided1() { return prepare_strided_plans<1>(); }

}  // namespace es
