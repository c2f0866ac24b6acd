// Instantiations, plan choice and launch of the fused derivative passes
// (fft_pass.cuh).
#include <mutex>

#include "fft_pass.cuh"
#include "pass_plans.h"

namespace es {

namespace {
struct PlanRow {
    int n, ra, rb, rc;
};
const PlanRow kPlans[] = {
#define ES_ROW(n, a, b, c, t) {n, a, b, c},
    ES_PLANS(ES_ROW)
#undef ES_ROW
};
constexpr int kNumPlans = sizeof(kPlans) / sizeof(kPlans[0]);
// chosen plan index per pass kind (0 = x, 1 = y/z) and axis length
int g_choice[2][257];
std::once_flag g_init;
void init_choice()
{
    for (int k = 0; k < 2; ++k)
        for (int n = 0; n <= 256; ++n) g_choice[k][n] = -1;
    for (int i = kNumPlans - 1; i >= 0; --i) {
        g_choice[0][kPlans[i].n] = i;
        g_choice[1][kPlans[i].n] = i;
    }
}
}  // namespace

int plan_radices(int n, int* ra, int* rb) { return plan_current(1, n, ra, rb); }

int plan_candidates(int n, int* ra, int* rb, int cap)
{
    int k = 0;
    for (int i = 0; i < kNumPlans && k < cap; ++i)
        if (kPlans[i].n == n) {
            ra[k] = kPlans[i].ra;
            rb[k] = kPlans[i].rb * kPlans[i].rc;
            ++k;
        }
    return k;
}

int plan_select(int kind, int n, int ra, int rb)
{
    std::call_once(g_init, init_choice);
    for (int i = 0; i < kNumPlans; ++i)
        if (kPlans[i].n == n && kPlans[i].ra == ra && kPlans[i].rb * kPlans[i].rc == rb) {
            g_choice[kind][n] = i;
            return 1;
        }
    return 0;
}

int plan_current(int kind, int n, int* ra, int* rb)
{
    std::call_once(g_init, init_choice);
    if (kind < 0 || kind > 1 || n < 1 || n > 256 || g_choice[kind][n] < 0) return 0;
    *ra = kPlans[g_choice[kind][n]].ra;
    *rb = kPlans[g_choice[kind][n]].rb * kPlans[g_choice[kind][n]].rc;
    return 1;
}

template <int RA, int RB, int RC, int T>
static cudaError_t launch_one(const PassParams& p, cudaStream_t st)
{
    constexpr int W = 2 * PAIRS;  // pencils per tile
    if (p.axis == 0) {
        const int ntiles = (p.ny * p.nz + W - 1) / W * p.nsim;
        constexpr int threads = pass_threads<T>();
        constexpr size_t smem = pass_smem_x<RA * RB * RC, T>();
        if constexpr (RA * RB * RC % 16 == 0) {
            int grid = 0;
            const cudaError_t e = persistent_grid(pass_x<RA, RB, RC, T>, threads, smem, ntiles * p.njobs, &grid);
            if (e != cudaSuccess) return e;
            return launch_pass_kernel(pass_x<RA, RB, RC, T>, dim3((unsigned)grid), threads, smem, st, p, ntiles);
        } else {
            return launch_pass_kernel(pass_x_any<RA, RB, RC, T>, dim3((unsigned)ntiles, (unsigned)p.njobs), threads, smem,
                                      st, p);
        }
    }
    const int ntx = (p.nx + W - 1) / W;
    const int outer = p.axis == 1 ? p.nz : p.ny;
    const int ntiles = ntx * outer * p.nsim;
    if (p.nx % 2 == 0) return launch_strided2(RA, RB, RC, ntiles, p, st);
    return launch_strided1(RA, RB, RC, ntiles, p, st);
}

template <int RA, int RB, int RC, int T>
static cudaError_t prepare_one()
{
    constexpr int smem = (int)pass_smem_x<RA * RB * RC, T>();
    if constexpr (RA * RB * RC % 16 == 0)
        return cudaFuncSetAttribute(pass_x<RA, RB, RC, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    else
        return cudaFuncSetAttribute(pass_x_any<RA, RB, RC, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t prepare_pass_kernels()
{
    cudaError_t e;
#define ES_PREP(n, a, b, c, t) if ((e = prepare_one<a, b, c, t>()) != cudaSuccess) return e;
    ES_PLANS(ES_PREP)
#undef ES_PREP
    if ((e = prepare_strided2()) != cudaSuccess) return e;
    if ((e = prepare_strided1()) != cudaSuccess) return e;
    if ((e = prepare_conv_kernels()) != cudaSuccess) return e;
    return prepare_circ_kernels();
}

cudaError_t launch_pass(const PassParams& p, cudaStream_t st)
{
    if (p.circ) return p.m > 0 && !circ_tc_eligible(p) ? launch_conv(p, st) : launch_circ(p, st);
    std::call_once(g_init, init_choice);
    const int kind = p.axis == 0 ? 0 : 1;
    if (p.n < 1 || p.n > 256 || g_choice[kind][p.n] < 0) return cudaErrorInvalidValue;
    const PlanRow& r = kPlans[g_choice[kind][p.n]];
#define ES_CASE(n, a, b, c, t) if (r.ra == a && r.rb == b && r.rc == c) return launch_one<a, b, c, t>(p, st);
    ES_PLANS(ES_CASE)
#undef ES_CASE
    return cudaErrorInvalidValue;
}

}  // namespace es
