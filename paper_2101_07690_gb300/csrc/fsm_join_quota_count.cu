// fsm_join_quota_count.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_COUNT under sampling quotas.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_quota_count(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_COUNT, true>(L, A, grid, st, bps);
}

} // namespace fsm
