// fsm_join_fused.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_FUSED.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_fused(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_FUSED, false>(L, A, grid, st, bps);
}

namespace {
// Publish the record of every key in the table (after a warm pass): one thread per slot, so that
// canonicalising runs with full warps.
__global__ void resolve_keys_kernel(const ExtArgs A) {
    const ResolveArgs R{A.pat_lab, A.pat_adj, A.cls_size, A.code_keys, A.code_off, A.pool_top,
                        A.code_mask, A.pool_words, A.key_rec, A.off_shift, A.err, A.explore, A.level};
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s <= A.qp.mask; s += (uint64_t)gridDim.x * blockDim.x) {
        const unsigned long long key = A.qp.keys[s];
        if (key != FSM_EMPTY_KEY) resolve_slot(R, (int64_t)s, key);
    }
}

} // namespace

cudaError_t launch_resolve_keys(const ExtArgs &A, int sms, cudaStream_t st) {
    const uint64_t blocks = (A.qp.mask + 256) / 256;
    resolve_keys_kernel<<<(unsigned)(blocks < (uint64_t)sms * 16 ? blocks : (uint64_t)sms * 16), 256, 0, st>>>(A);
    return cudaGetLastError();
}

} // namespace fsm
