// fsm_join_fused.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_FUSED.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_fused(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_FUSED, false>(L, A, grid, st, bps);
}

} // namespace fsm
