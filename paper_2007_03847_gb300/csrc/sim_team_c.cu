// Instantiations of the team kernel for 10 machine slot(s).
#include "simulate_team.cuh"

namespace fmc {

cudaError_t launch_team_nm10(int nd, const void* params, const CUtensorMap* maps, const TeamArgs& a, int smooth,
                            cudaStream_t st, int* max_ctas_per_sm)
{
    switch (nd) {
        case 1: return launch_team_t<10, 1>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 2: return launch_team_t<10, 2>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 4: return launch_team_t<10, 4>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 8: return launch_team_t<10, 8>(params, maps, a, smooth, st, max_ctas_per_sm);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fmc
