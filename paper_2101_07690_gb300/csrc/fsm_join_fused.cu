// fsm_join_fused.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_FUSED.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_fused(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_FUSED, false>(L, A, grid, st, bps);
}

cudaError_t launch_resolve_keys(const ExtArgs &A, int sms, cudaStream_t st) {
    const uint64_t blocks = (A.qp.mask + 256) / 256;
    resolve_keys_kernel<<<(unsigned)(blocks < (uint64_t)sms * 16 ? blocks : (uint64_t)sms * 16), 256, 0, st>>>(A);
    return cudaGetLastError();
}

} // namespace fsm
