// Instantiations of the team kernel for 16 machine slot(s).
#include "simulate_team.cuh"

namespace fmc {

cudaError_t launch_team_nm16(int nd, const void* params, const CUtensorMap* maps, const TeamArgs& a, int smooth,
                            cudaStream_t st, int* max_ctas_per_sm)
{
    switch (nd) {
        case 1: return launch_team_t<16, 1>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 2: return launch_team_t<16, 2>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 4: return launch_team_t<16, 4>(params, maps, a, smooth, st, max_ctas_per_sm);
        case 8: return launch_team_t<16, 8>(params, maps, a, smooth, st, max_ctas_per_sm);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fmc
