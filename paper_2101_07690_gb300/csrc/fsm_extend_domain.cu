// fsm_extend_domain.cu -- instantiations of the extension kernel for PASS_DOMAIN.
#include "fsm_extend.cuh"

namespace fsm {

cudaError_t launch_extend_domain(int L, int V, const ExtArgs &A, int grid, cudaStream_t st) {
    if (V == FSM_EXPLORE_SV) return launch_extend_sv(PASS_DOMAIN, L, A, grid, st);
    if (V == FSM_EXPLORE_TV_EDGELIST) return launch_extend_edgelist(PASS_DOMAIN, L, A, grid, st);
    if (V == FSM_EXPLORE_TV_QUOTA) return launch_extend_quota(PASS_DOMAIN, L, A, grid, st);
    switch (L) {
    case 6: extend_kernel<6, PASS_DOMAIN><<<grid, 256, 0, st>>>(A); break;
    case 7: return launch_extend_l7(PASS_DOMAIN, A, grid, st);
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t occupancy_extend_domain(int L, int V, int *blocks_per_sm) {
    if (V == FSM_EXPLORE_SV) return occupancy_extend_sv(PASS_DOMAIN, L, blocks_per_sm);
    if (V == FSM_EXPLORE_TV_EDGELIST) return occupancy_extend_edgelist(PASS_DOMAIN, L, blocks_per_sm);
    if (V == FSM_EXPLORE_TV_QUOTA) return occupancy_extend_quota(PASS_DOMAIN, L, blocks_per_sm);
    switch (L) {
    case 6: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, extend_kernel<6, PASS_DOMAIN>, 256, 0);
    case 7: return occupancy_extend_l7(PASS_DOMAIN, blocks_per_sm);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace fsm
