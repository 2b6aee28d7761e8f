// fsm_extend_emit.cu -- instantiations of the extension kernel for PASS_EMIT.
#include "fsm_extend.cuh"

namespace fsm {

cudaError_t launch_extend_emit(int L, int V, const ExtArgs &A, int grid, cudaStream_t st) {
    if (V == FSM_EXPLORE_SV) return launch_extend_sv(PASS_EMIT, L, A, grid, st);
    if (V == FSM_EXPLORE_TV_EDGELIST) return launch_extend_edgelist(PASS_EMIT, L, A, grid, st);
    if (V == FSM_EXPLORE_TV_QUOTA) return launch_extend_quota(PASS_EMIT, L, A, grid, st);
    switch (L) {
    case 6: extend_kernel<6, PASS_EMIT><<<grid, 256, 0, st>>>(A); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t occupancy_extend_emit(int L, int V, int *blocks_per_sm) {
    if (V == FSM_EXPLORE_SV) return occupancy_extend_sv(PASS_EMIT, L, blocks_per_sm);
    if (V == FSM_EXPLORE_TV_EDGELIST) return occupancy_extend_edgelist(PASS_EMIT, L, blocks_per_sm);
    if (V == FSM_EXPLORE_TV_QUOTA) return occupancy_extend_quota(PASS_EMIT, L, blocks_per_sm);
    switch (L) {
    case 6: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, extend_kernel<6, PASS_EMIT>, 256, 0);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace fsm
