// fsm_join_quota_emit.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_EMIT under sampling quotas.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_quota_emit(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_EMIT, true>(L, A, grid, st, bps);
}

} // namespace fsm
