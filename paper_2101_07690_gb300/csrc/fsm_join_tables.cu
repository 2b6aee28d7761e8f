// fsm_join_tables.cu -- the acceptance tables of the join kernel (JoinGeo, fsm_join.cuh) and the
// dispatch of its passes.
#include "fsm_join.cuh"
#include "fsm_kernels.cuh"

namespace fsm {
namespace {

// one 32-subset word of one row per thread
template <int L>
__global__ void acc_kernel(uint32_t *acc) {
    using G = JoinGeo<L>;
    const int64_t n = (int64_t)G::CLS * G::ROWS * G::W;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int wd = (int)(x % G::W);
        int64_t y = x / G::W;
        const int bgt = (int)(y & 1);
        y >>= 1;
        const int sb = (int)(y % G::SL);
        y /= G::SL;
        const int sa = (int)(y % G::SL);
        y /= G::SL;
        const int form = (int)(y % 3), cls = (int)(y / 3);
        uint32_t m = 0;
        const int subs = G::SUBS < 32 ? G::SUBS : 32;
        for (int s = 0; s < subs; ++s)
            if (join_accepted<L>(cls, form, sa, sb, bgt, (uint32_t)(wd * 32 + s))) m |= 1u << s;
        acc[x] = m;
    }
}

// Seven vertices (l = 5) have 283M combinations but only 2^21 graphs on ordered ids: dissect each
// graph once (part mask | join vertex << 7, 0 if disconnected), then look them up.  Bit of pair
// (x, y), x < y: y (y - 1) / 2 + x.
__global__ void dissect7_kernel(uint16_t *code) {
    const int32_t gid[7] = {0, 1, 2, 3, 4, 5, 6};
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < (1 << 21); c += gridDim.x * blockDim.x) {
        uint32_t adj[7] = {0, 0, 0, 0, 0, 0, 0};
        for (int y = 1; y < 7; ++y)
            for (int x = 0; x < y; ++x)
                if ((c >> (y * (y - 1) / 2 + x)) & 1) { adj[x] |= 1u << y; adj[y] |= 1u << x; }
        uint16_t r = 0;
        if (mask_connected(127u, adj, 7)) {
            uint32_t lm = 0;
            int jn = -1;
            dissect3(7, gid, adj, lm, jn);
            r = (uint16_t)(lm | ((uint32_t)jn << 7));
        }
        code[c] = r;
    }
}
__device__ __forceinline__ uint32_t pair_bit(int x, int y) {
    const int a = x < y ? x : y, b = x < y ? y : x;
    return 1u << (b * (b - 1) / 2 + a);
}
__global__ void acc5_kernel(const uint16_t *code, uint32_t *acc) {
    constexpr int L = 5;
    using G = JoinGeo<L>;
    const int64_t n = (int64_t)G::CLS * G::ROWS * G::W;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int wd = (int)(i % G::W);
        int64_t y = i / G::W;
        const int bgt = (int)(y & 1);
        y >>= 1;
        const int sb = (int)(y % G::SL);
        y /= G::SL;
        const int sa = (int)(y % G::SL);
        y /= G::SL;
        const int form = (int)(y % 3), cls = (int)(y / 3), rv = cls >> G::EB;
        uint32_t m = 0;
        const bool order = (sa == sb || (sb > sa) == (bgt != 0)) && (form == FORM_END || bgt);
        uint32_t sadj[5] = {0, 0, 0, 0, 0};
        int bit = 0;
        for (int t = 0; t < L; ++t)
            for (int u = t + 1; u < L; ++u, ++bit)
                if ((cls >> bit) & 1) { sadj[t] |= 1u << u; sadj[u] |= 1u << t; }
        if (order && mask_connected(31u, sadj, L)) {
            int pos[L];
            for (int t = 0; t < L; ++t) pos[t] = t + (sa <= t) + (sb <= t);
            const int pa = sa + (bgt ? 0 : 1), pb = sb + (bgt ? 1 : 0), pv = pos[rv];
            uint32_t base = pair_bit(pv, pa);
            if (form != FORM_END) base |= pair_bit(pv, pb);
            if (form != FORM_CENTRE) base |= pair_bit(pa, pb);
            for (int t = 0; t < L; ++t)
                for (int u = t + 1; u < L; ++u)
                    if ((sadj[t] >> u) & 1u) base |= pair_bit(pos[t], pos[u]);
            uint32_t cb[8];
            for (int r = 0; r < 4; ++r) {
                const int t = r + (r >= rv);
                cb[r] = pair_bit(pos[t], pa);
                cb[4 + r] = pair_bit(pos[t], pb);
            }
            const uint32_t want = (1u << pv) | (1u << pa) | (1u << pb) | ((uint32_t)pv << 7);
            for (int q = 5; q < 8; ++q)
                if ((wd >> (q - 5)) & 1) base |= cb[q];
            for (int s = 0; s < 32; ++s) {
                uint32_t c = base;
                for (int q = 0; q < 5; ++q)
                    if ((s >> q) & 1) c |= cb[q];
                if (__ldg(code + c) == want) m |= 1u << s;
            }
        }
        acc[i] = m;
    }
}

// entry (class, ANY_*, anchor slot): partner slots that some subset and form accept
template <int L>
__global__ void any_kernel(const uint32_t *acc, uint16_t *any) {
    using G = JoinGeo<L>;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < G::ANY_ENTRIES; x += (int64_t)gridDim.x * blockDim.x) {
        const int s = (int)(x % G::SL), kind = (int)(x / G::SL) & 3;
        const int64_t cls = x / (4 * G::SL);
        auto some = [&](int form, int sa, int sb, int bgt) {
            const uint32_t *r = acc + (cls * G::ROWS + ((int64_t)(form * G::SL + sa) * G::SL + sb) * 2 + bgt) * G::W;
            uint32_t m = 0;
            for (int i = 0; i < G::W; ++i) m |= r[i];
            return m != 0;
        };
        uint32_t m = 0;
        for (int p = 0; p < G::SL; ++p) {
            if (kind == ANY_C || kind == ANY_CT) {   // anchor b, partner a < b
                if (some(FORM_CENTRE, p, s, 1) || (kind == ANY_CT && some(FORM_TRI, p, s, 1))) m |= 1u << p;
            } else {                                 // anchor a, partner b
                if (some(FORM_END, s, p, 0)) m |= 1u << p;
                if (some(FORM_END, s, p, 1) || (kind == ANY_ET && some(FORM_TRI, s, p, 1))) m |= 1u << (p + G::SL);
            }
        }
        any[x] = (uint16_t)m;
    }
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
