// fsm_join_domain.cu -- instantiations of the join kernel (stored sizes 1..5) for PASS_DOMAIN, and the
// domain bits of joins that the count pass kept.
#include "fsm_join.cuh"

namespace fsm {

cudaError_t join_domain(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    return join_pass<PASS_DOMAIN, false>(L, A, grid, st, bps);
}

namespace {

// Domain bits from the joins a count pass kept, instead of a second enumeration.  A block takes a part
// of one region, a warp a run of consecutive records of it: those come from a few units, so their
// vertices of s, key records and bits of s repeat (the small table as in the join kernel).
//
// What bounds it is the scattered reductions: 16 bytes of record and K bitmap words a join, where the
// domain pass enumerated five pieces for it.  A word is read first here, whatever its label class: the
// joins come faster than in the domain pass, many to a word, and a read that finds the bit spares the
// reduction (37k vertices, vertex-induced, 3 -> 5, 1.6e8 joins: 8.2 ms without, 5.8 with; 3312 vertices,
// 4.8e7: 1.13 and 0.59).  Eight blocks a region against two: 5.8 and 5.7 ms; 370k vertices, 2 -> 4: 3.2
// and 2.9.  Domain pass against this kernel: 4 -> 6, 2.9e8 joins, 13.6 and 3.4 ms; 5 -> 7 under ST 8,
// 1.2e8 joins, 32.7 and 12.7; the one above 11.2 and 5.7; keeping the joins costs the count pass 7 to 20 %
// (4 -> 6: 9.5 and 11.5 ms).
template <int L>
__global__ void __launch_bounds__(256) kept_bits_kernel(const __grid_constant__ ExtArgs A, int parts) {
    constexpr int K = L + 2, RW = key_rec_words(K);
    __shared__ unsigned long long seen[8][FSM_JOIN_SEEN];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int x = lane; x < FSM_JOIN_SEEN; x += 32) seen[w][x] = ~0ull;
    __syncwarp();
    const uint32_t shard = blockIdx.x / parts;
    const uint64_t n = A.keep_n[shard];
    const uint4 *rec = A.keep + (uint64_t)shard * A.keep_cap;
    const uint64_t warps = (uint64_t)parts * 8, wi = (uint64_t)(blockIdx.x % parts) * 8 + w;
    const uint64_t per = ((n + warps - 1) / warps + 31) / 32 * 32;
    const uint64_t end = min(n, (wi + 1) * per);
    for (uint64_t i = wi * per + lane; i < end; i += 32) {
        const uint4 d = __ldcs(rec + i);
        const uint32_t *kr = A.key_rec + (uint64_t)d.x * RW;
        uint32_t wd[K > 6 ? 16 : 8];
        ld_rec8(kr, wd);
        if (K > 6) ld_rec8(kr + 8, wd + (K > 6 ? 8 : 0));
        if (wd[2] == FSM_OFF_NONE) continue;   // pattern without bitmaps
        const unsigned long long tag = ((unsigned long long)d.x << 32) | d.y;
        volatile unsigned long long *sn = &seen[w][(d.x ^ (d.x >> 7) ^ (d.y << 3)) & (FSM_JOIN_SEEN - 1)];
        const bool own = *sn != tag;           // a lost entry only repeats bits
        if (own) *sn = tag;
        uint32_t *wp[K];
        uint32_t bit[K], old[K] = {};
#pragma unroll
        for (int h = 0; h < K; ++h) {
            uint32_t rk = h == L ? d.z : d.w;
            if (h < L) rk = own ? (uint32_t)__ldg(A.g.rank + __ldg(A.fv + (int64_t)(h < L ? h : 0) * A.fN + d.y)) : 0u;
            wp[h] = A.dom + ((uint64_t)wd[2 + h] << A.off_shift) + (rk >> 5);
            bit[h] = 1u << (rk & 31);
        }
#pragma unroll
        for (int h = 0; h < K; ++h)
            if (h >= L || own) old[h] = __ldcg(wp[h]);
#pragma unroll
        for (int h = 0; h < K; ++h)
            if ((h >= L || own) && !(old[h] & bit[h])) atomicOr(wp[h], bit[h]);
    }
}

} // namespace

cudaError_t launch_kept_bits(int L, const ExtArgs &A, int shards, cudaStream_t st) {
    const int parts = 8;
    switch (L) {
    case 1: kept_bits_kernel<1><<<shards * parts, 256, 0, st>>>(A, parts); break;
    case 2: kept_bits_kernel<2><<<shards * parts, 256, 0, st>>>(A, parts); break;
    case 3: kept_bits_kernel<3><<<shards * parts, 256, 0, st>>>(A, parts); break;
    case 4: kept_bits_kernel<4><<<shards * parts, 256, 0, st>>>(A, parts); break;
    case 5: kept_bits_kernel<5><<<shards * parts, 256, 0, st>>>(A, parts); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

} // namespace fsm
