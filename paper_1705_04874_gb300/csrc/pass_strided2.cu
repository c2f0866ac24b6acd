// The y and z derivative passes for an even nx.
#include "pass_strided.cuh"

namespace es {

cudaError_t launch_strided2(int ra, int rb, int rc, int ntiles, const PassParams& p, cudaStream_t st)
{
    return launch_strided_plans<2>(ra, rb, rc, ntiles, p, st);
}
cudaError_t prepare_strided2() { return prepare_strided_plans<2>(); }

}  // namespace es
