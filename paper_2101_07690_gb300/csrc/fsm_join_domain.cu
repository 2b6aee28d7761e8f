// fsm_join_domain.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_DOMAIN.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_domain(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_DOMAIN, false>(L, A, grid, st, bps);
}

} // namespace fsm
