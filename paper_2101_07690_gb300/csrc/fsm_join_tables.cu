// fsm_join_tables.cu -- the acceptance tables of the join kernel (JoinGeo, fsm_join.cuh) and the
// dispatch of its passes.
#include "fsm_join_tables.cuh"
#include "fsm_kernels.cuh"

namespace fsm {
namespace {

// one entry per thread
template <int L>
__global__ void acc_kernel(uint32_t *acc) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < JoinGeo<L>::ACC_WORDS; x += (int64_t)gridDim.x * blockDim.x)
        acc[x] = acc_word<L>(x);
}
__global__ void dissect7_kernel(uint16_t *code) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < (1 << 21); c += gridDim.x * blockDim.x) code[c] = dissect7_code(c);
}
__global__ void acc5_kernel(const uint16_t *__restrict__ code, uint32_t *acc) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < JoinGeo<5>::ACC_WORDS; i += (int64_t)gridDim.x * blockDim.x)
        acc[i] = acc5_word(code, i);
}
template <int L>
__global__ void any_kernel(const uint32_t *acc, uint16_t *any) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < JoinGeo<L>::ANY_ENTRIES; x += (int64_t)gridDim.x * blockDim.x)
        any[x] = any_entry<L>(acc, x);
}

template <int L>
cudaError_t build_tables(uint32_t *acc, uint16_t *any, void *tmp, cudaStream_t st) {
    auto blocks = [](int64_t n) { return (int)(n + 127 < 128 * 152 * 64 ? (n + 127) / 128 : 152 * 64); };
    if constexpr (L == 5) {
        dissect7_kernel<<<blocks(1 << 21), 128, 0, st>>>((uint16_t *)tmp);
        acc5_kernel<<<blocks(JoinGeo<L>::ACC_WORDS), 128, 0, st>>>((const uint16_t *)tmp, acc);
        note_launches(3);
    } else {
        acc_kernel<L><<<blocks(JoinGeo<L>::ACC_WORDS), 128, 0, st>>>(acc);
        note_launches(2);
    }
    any_kernel<L><<<blocks(JoinGeo<L>::ANY_ENTRIES), 128, 0, st>>>(acc, any);
    return cudaGetLastError();
}

template <int L>
void table_bytes(size_t *acc, size_t *any, size_t *tmp) {
    *acc = (size_t)JoinGeo<L>::ACC_WORDS * sizeof(uint32_t);
    *any = (size_t)JoinGeo<L>::ANY_ENTRIES * sizeof(uint16_t);
    *tmp = L == 5 ? ((size_t)1 << 21) * sizeof(uint16_t) : 16;
}

cudaError_t dispatch(int pass, int L, int V, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    const bool q = V == FSM_EXPLORE_TV_QUOTA;
    switch (pass) {
    case PASS_COUNT: return q ? join_quota_count(L, A, grid, st, bps) : join_count(L, A, grid, st, bps);
    case PASS_DOMAIN: return q ? join_quota_domain(L, A, grid, st, bps) : join_domain(L, A, grid, st, bps);
    case PASS_EMIT: return q ? join_quota_emit(L, A, grid, st, bps) : join_emit(L, A, grid, st, bps);
    case PASS_FUSED: return q ? cudaErrorInvalidValue : join_fused(L, A, grid, st, bps);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace

cudaError_t launch_join(int pass, int L, int V, const ExtArgs &A, int grid, cudaStream_t st) {
    return dispatch(pass, L, V, &A, grid, st, nullptr);
}
cudaError_t occupancy_join(int pass, int L, int V, int *blocks_per_sm) {
    return dispatch(pass, L, V, nullptr, 0, nullptr, blocks_per_sm);
}

void join_table_bytes(int L, size_t *acc, size_t *any, size_t *tmp) {
    switch (L) {
    case 1: table_bytes<1>(acc, any, tmp); break;
    case 2: table_bytes<2>(acc, any, tmp); break;
    case 3: table_bytes<3>(acc, any, tmp); break;
    case 4: table_bytes<4>(acc, any, tmp); break;
    default: table_bytes<5>(acc, any, tmp); break;
    }
}
cudaError_t launch_join_tables(int L, uint32_t *acc, uint16_t *any, void *tmp, cudaStream_t st) {
    switch (L) {
    case 1: return build_tables<1>(acc, any, tmp, st);
    case 2: return build_tables<2>(acc, any, tmp, st);
    case 3: return build_tables<3>(acc, any, tmp, st);
    case 4: return build_tables<4>(acc, any, tmp, st);
    case 5: return build_tables<5>(acc, any, tmp, st);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace fsm
