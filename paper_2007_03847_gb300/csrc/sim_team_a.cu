// Instantiations of the team kernel for 1, 2, 4 machine slot(s).
#include "simulate_team.cuh"

namespace fmc {

cudaError_t launch_team_nm1(int nd, const void* params, const CUtensorMap* maps, const TeamArgs& a, int smooth,
                            cudaStream_t st, int* max_ctas_per_sm)
{
    switch (nd) {
        case 1: return launch_team_t<1, 1>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 2: return launch_team_t<1, 2>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 4: return launch_team_t<1, 4>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 8: return launch_team_t<1, 8>(params, maps, a, smooth, st, max_ctas_per_sm);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_team_nm2(int nd, const void* params, const CUtensorMap* maps, const TeamArgs& a, int smooth,
                            cudaStream_t st, int* max_ctas_per_sm)
{
    switch (nd) {
        case 1: return launch_team_t<2, 1>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 2: return launch_team_t<2, 2>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 4: return launch_team_t<2, 4>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 8: return launch_team_t<2, 8>(params, maps, a, smooth, st, max_ctas_per_sm);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_team_nm4(int nd, const void* params, const CUtensorMap* maps, const TeamArgs& a, int smooth,
                            cudaStream_t st, int* max_ctas_per_sm)
{
    switch (nd) {
        case 1: return launch_team_t<4, 1>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 2: return launch_team_t<4, 2>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 4: return launch_team_t<4, 4>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 8: return launch_team_t<4, 8>(params, maps, a, smooth, st, max_ctas_per_sm);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fmc
