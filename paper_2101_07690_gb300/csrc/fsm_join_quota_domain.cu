// fsm_join_quota_domain.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_DOMAIN under sampling quotas.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_quota_domain(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_DOMAIN, true>(L, A, grid, st, bps);
}

} // namespace fsm
