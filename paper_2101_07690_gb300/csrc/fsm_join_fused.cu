// fsm_join_fused.cu -- the one-pass last level: instantiations of the join kernel (stored sizes 1..5) for
// PASS_FUSED, the bulk resolution of its keys, and the bits of the joins it put aside.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_fused(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_FUSED, false>(L, A, grid, st, bps);
}

namespace {

// Resolve a key of the one-pass last level: canonicalise the graph its key denotes, find or claim its
// pattern's entry in the code table, claim the pattern's orbit bitmaps from the pool unless another
// lane already did (one CAS decides; a loser's pool words stay unused), and publish the key's record.
// On a full table or pool the error word says so and nothing is published.
struct ResolveArgs {
    const uint64_t *pat_lab, *pat_adj;
    const int32_t *cls_size;
    unsigned long long *code_keys, *code_off, *pool_top;
    uint64_t code_mask;
    unsigned long long pool_words;
    uint32_t *key_rec;
    int shift;
    int *err;
    int explore, level;
};

__device__ __forceinline__ void resolve_slot(const ResolveArgs A, int64_t slot, uint64_t key) {
    // K <= 7 here: the compact words of fsm_canon7.cuh
    int K, lab[8], rep[8];
    uint32_t adj[8];
    key_graph7(A.explore, A.level, key, A.pat_lab, A.pat_adj, K, lab, adj);
    unsigned long long clab;
    uint32_t cadj, inv;
    canonicalise7(K, lab, adj, clab, cadj, inv);
    orbit_reps7(K, clab, cadj, rep);
    int64_t pre[8], words = 0;
    for (int c = 0; c < K; ++c) {
        pre[c] = words;
        if (rep[c] == c)
            words += bitmap_words(__ldg(A.cls_size + ((clab >> (8 * (7 - c))) & 0xff)), A.shift);
    }
    const uint64_t pk = pack_code7(K, clab, cadj);
    uint64_t h = mix64(pk) & A.code_mask;
    int64_t ci = -1;
    for (int probe = 0; probe < FSM_MAX_PROBES; ++probe) {
        unsigned long long cur = __ldcg(A.code_keys + h);
        if (cur == FSM_EMPTY_KEY) cur = atomicCAS(A.code_keys + h, FSM_EMPTY_KEY, pk);
        if (cur == FSM_EMPTY_KEY || cur == pk) { ci = (int64_t)h; break; }
        h = (h + 1) & A.code_mask;
    }
    if (ci < 0) { atomicOr(A.err, FSM_ERR_CODE_FULL); return; }
    unsigned long long off = __ldcg(A.code_off + ci);
    if (off == 0ull) {
        // one reservation for the lanes here together: the bulk resolution makes hundreds of thousands
        const unsigned am = __activemask();
        const int lane = threadIdx.x & 31, leader = __ffs(am) - 1;
        unsigned long long before = 0, sum = 0;
        for (unsigned m = am; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const unsigned long long x = __shfl_sync(am, (unsigned long long)words, src);
            if (src < lane) before += x;
            sum += x;
        }
        unsigned long long res = lane == leader ? atomicAdd(A.pool_top, sum) : 0ull;
        res = __shfl_sync(am, res, leader) + before;
        if (res + (unsigned long long)words > A.pool_words) { atomicOr(A.err, FSM_ERR_POOL); return; }
        const unsigned long long old = atomicCAS(A.code_off + ci, 0ull, res + 1ull);
        off = old ? old : res + 1ull;
    }
    uint32_t *kr = A.key_rec + slot * key_rec_words(K);
    for (int hh = 0; hh < K; ++hh)
        *(kr + 2 + hh) = (uint32_t)(((long long)(off - 1ull) + pre[rep[(inv >> (3 * hh)) & 7]]) >> A.shift);
    *(kr) = (uint32_t)key;
    *(kr + 1) = (uint32_t)(key >> 32);
}

// Publish the record of every key in the table that has none (after the warm pass, and again after the
// level): one thread per slot, so that canonicalising runs with full warps.
__global__ void resolve_keys_kernel(const ExtArgs A) {
    const ResolveArgs R{A.pat_lab, A.pat_adj, A.cls_size, A.code_keys, A.code_off, A.pool_top,
                        A.code_mask, A.pool_words, A.key_rec, A.off_shift, A.err, A.explore, A.level};
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s <= A.qp.mask; s += (uint64_t)gridDim.x * blockDim.x) {
        const unsigned long long key = A.qp.keys[s];
        if (key == FSM_EMPTY_KEY) continue;
        if (A.key_rec[s * key_rec_words(A.level + 2) + 2] != FSM_OFF_NONE) continue;   // resolved before
        resolve_slot(R, (int64_t)s, key);
    }
}

// Domain bits of the joins whose keys had no record during the level.
__global__ void deferred_bits_kernel(const ExtArgs A) {
    const unsigned long long n = min(*A.defer_top, A.defer_cap);
    const int K = A.level + 2;
    for (unsigned long long x = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t *d = A.defer + x * FSM_DEFER_WORDS;
        const uint32_t *kr = A.key_rec + (uint64_t)d[0] * key_rec_words(K);
        for (int h = 0; h < K; ++h) {
            const uint32_t off = kr[2 + h];
            if (off == FSM_OFF_NONE) break;   // the pool ran out: the error word says so
            const uint64_t word = ((uint64_t)off << A.off_shift) + (d[1 + h] >> 5);
            if (word >= A.pool_words) { atomicOr(A.err, FSM_ERR_POOL); break; }
            atomicOr(A.pool + word, 1u << (d[1 + h] & 31));
        }
    }
}
} // namespace

cudaError_t launch_deferred_bits(const ExtArgs &A, int sms, cudaStream_t st) {
    deferred_bits_kernel<<<sms * 8, 256, 0, st>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_resolve_keys(const ExtArgs &A, int sms, cudaStream_t st) {
    const uint64_t blocks = (A.qp.mask + 256) / 256;
    resolve_keys_kernel<<<(unsigned)(blocks < (uint64_t)sms * 16 ? blocks : (uint64_t)sms * 16), 256, 0, st>>>(A);
    return cudaGetLastError();
}

} // namespace fsm
