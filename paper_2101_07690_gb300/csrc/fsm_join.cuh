// fsm_join.cuh -- the two-vertex extension kernel for stored levels of size l <= 5 (l -> l+2,
// k <= 7; two-vertex exploration with index-based quick patterns, exact, rate-sampled or under
// Section 5's quotas).  fsm_extend.cuh states the work of a join and holds the kernel of the other
// forms; this one does the same joins in another order of steps.
//
// What bounds a level is the number of candidate pieces times the instructions each costs (DRAM is
// nearly idle where the bitmaps fit L2), so the steps are ordered by what they reject per instruction,
// and every step runs with full warps:
//
//   tables     Whether smallest-vertex-first dissection (Algorithm 1) returns exactly (t, s) depends
//              only on the relative order of the l + 2 ids and on the edges among them.  With s
//              sorted by id, that is: the class of s (rank of the key vertex, edges of s in id
//              order), the piece's form, the slots of its two new vertices a and b (how many ids of
//              s lie below each), whether b > a, and the cross-edge subset.  `acc` holds one bit per
//              combination (all 2^(2(l-1)) subsets of a row side by side), `any` the OR over
//              subsets and forms for one new vertex's slot against the other's.
//   segments   A unit's pieces are rows of sorted lists: centre row y (anchor b = y-th neighbour of
//              v, partners a = the neighbours before it) and end list a (anchor a, partners b in
//              N(a)).  One lane prepares one row: the slots its anchor allows its partner cut the
//              row to a range, rows of anchors that allow none are not in the unit's row ranges at
//              all, and the anchor's label, cross edges and pruning bits are found once for the row.
//   filter     Lanes then walk the surviving ranges side by side: one coalesced list read (with the
//              labels and ranks, which lie in an array beside the lists), the
//              partner's slot by l comparisons, one bit test.  Survivors go to a per-warp queue.
//   joins      Full warps take 32 survivors: the size-3 frequency of the piece, cross edges (a
//              shared-memory Bloom filter of each list of s, misses are certain, hits are verified
//              by binary search), joining-point pruning (Section 4.5) as cross bits that must or
//              must not be set, then the subsets that are left and accepted by `acc`.
//   accept     One 32-byte record per key slot holds the key and its patterns' bitmap offsets, so
//              a join finds both in one read; counts are single reductions that nothing waits for.
//
// One launch on a GB300 (same graph and output): the extension kernel before, this kernel with a
// key table per block in shared memory (flushed between chunks) and both new vertices' tests made
// per survivor, and as it is:
//   3 -> 5, one pass, 74k vertices, 1.7e9 pieces, 3.3e8 joins:      475 ms,  77.7 ms,  18.8 ms
//   2 -> 4, one pass, 100k vertices, 7.5e9 pieces, 3.2e9 joins:     733 ms, 283 ms,    88 ms
//   4 -> 6, count, 1656 vertices, 1.4e9 pieces, 2.9e8 joins:        265 ms,  18.5 ms,   9.8 ms
//   5 -> 7, count, ST 8 quotas, 6.0e8 pieces, 1.2e8 joins:          248 ms,  60.6 ms,  27.6 ms
//   1 -> 3, count, 3.7M vertices, 6.3e8 pieces, 2.0e8 joins:       14.4 ms,   8.1 ms,   4.3 ms
// The block tables missed 70 to 77 % of the lookups of levels 1 and 2, and their flushes made warps
// wait for each other; a record read at the L2 costs each join one latency and no barrier.  What is
// left is bound by issue and dependent loads (3 -> 5, one pass, 370k vertices: 9.4 warp instructions a
// piece where the extension kernel took 80, 60 % of the issue slots, 21.5 of 32 lanes, DRAM at 3 %), by
// scattered requests (2 -> 4: load-store unit 66 %, L2 58 % busy) and, where the body is large, by
// instruction fetch: one copy of the joins (take) instead of two took 5 -> 7 from 55 to 35 ms.
#pragma once
#include "fsm_extend.cuh"

namespace fsm {

// forms of a piece, by the order (a, b) in which its two non-key vertices are kept
enum { FORM_CENTRE = 0, FORM_END = 1, FORM_TRI = 2 };
// rows of `any`: centre rows that stand for the wedge only / for wedge and triangle, end lists
// for the wedge only / for the wedge and, when b > a, the triangle
enum { ANY_C = 0, ANY_CT = 1, ANY_E = 2, ANY_ET = 3 };

// Geometry of the tables and of a warp's shared storage for stored size L.
template <int L> struct JoinGeo {
    static constexpr int K = L + 2;
    static constexpr int O = L - 1;                  // vertices of s other than the key vertex
    static constexpr int SUBS = 1 << (2 * O);        // cross-edge subsets
    static constexpr int W = SUBS > 32 ? SUBS / 32 : 1;
    static constexpr int EB = L * (L - 1) / 2;       // edge bits of s, pairs (0,1), (0,2), ... in id order
    static constexpr int CLS = L << EB;              // class = rank of v << EB | edge bits
    static constexpr int SL = L + 1;                 // slots of a new vertex
    static constexpr int ROWS = 3 * SL * SL * 2;     // ((form * SL + slot a) * SL + slot b) * 2 + (b > a)
    static constexpr int64_t ACC_WORDS = (int64_t)CLS * ROWS * W;
    static constexpr int64_t ANY_ENTRIES = (int64_t)CLS * 4 * SL;   // (class * 4 + ANY_*) * SL + anchor slot
};

// Is the join accepted (edge-induced graph given by class, form, slots and cross subset)?  Vertices
// are renamed by id order; sub bit r: a next to the r-th other vertex of s (in id order), bit
// O + r: b next to it.
template <int L>
FSM_HD bool join_accepted(int cls, int form, int sa, int sb, int bgt, uint32_t sub) {
    constexpr int K = L + 2, O = L - 1;
    if (sa != sb && (sb > sa) != (bgt != 0)) return false;   // no such order
    if (form != FORM_END && !bgt) return false;              // centre pieces and triangles keep a < b
    if constexpr (L == 1) {
        return sa == 1 && sb == 1;   // size-3 subgraphs are made at their smallest vertex
    } else {
        const int rv = cls >> JoinGeo<L>::EB;
        int pos[L];
        uint32_t adj[K];
        int32_t gid[K];
        for (int h = 0; h < K; ++h) { adj[h] = 0; gid[h] = h; }
        for (int t = 0; t < L; ++t) pos[t] = t + (sa <= t) + (sb <= t);
        const int pa = sa + (bgt ? 0 : 1), pb = sb + (bgt ? 1 : 0);
        auto link = [&](int x, int y) { adj[x] |= 1u << y; adj[y] |= 1u << x; };
        int bit = 0;
        for (int t = 0; t < L; ++t)
            for (int u = t + 1; u < L; ++u, ++bit)
                if ((cls >> bit) & 1) link(pos[t], pos[u]);
        uint32_t ms = 0;
        for (int t = 0; t < L; ++t) ms |= 1u << pos[t];
        if (!mask_connected(ms, adj, K)) return false;       // no stored embedding has this class
        link(pos[rv], pa);
        if (form != FORM_END) link(pos[rv], pb);
        if (form != FORM_CENTRE) link(pa, pb);
        for (int r = 0; r < O; ++r) {
            const int t = r + (r >= rv);
            if ((sub >> r) & 1u) link(pos[t], pa);
            if ((sub >> (O + r)) & 1u) link(pos[t], pb);
        }
        uint32_t lm = 0;
        int jn = -1;
        dissect3(K, gid, adj, lm, jn);
        return jn == pos[rv] && lm == ((1u << pos[rv]) | (1u << pa) | (1u << pb));
    }
}

// survivors of the filter wait here until 32 are there
#define FSM_JOIN_QUEUE 64
// per warp: key slots whose bits of s the batch's units have set (see accept)
#define FSM_JOIN_SEEN 128

// A queued candidate, and a row's part of it, in one word: unit j (4 bits), end list (1), slot of the
// anchor (3) and of the partner (3), and of the anchor its cross edges to the other vertices of s
// (4), and the cross edges pruning asks of it (4) or forbids (4).
#define FSM_M_END 4
#define FSM_M_SA 5
#define FSM_M_SP 8
#define FSM_M_CROSS 11
#define FSM_M_MUST 15
#define FSM_M_NO 19

// A batch's units in shared memory: UW words each.
template <int L, bool QUOTA> struct UnitRec {
    static constexpr int O = L - 1;
    // Units per batch and shared words per warp for their Bloom filters (L lists each).  8 units against
    // 16: 3 -> 5 one pass 25.5 and 26.8 ms, 2 -> 4 one pass 127 and 131 ms, 1 -> 3 count 6.3 and 6.1
    // ms; 4 units against 8: 5 -> 7 count 38.8 and 35.2 ms.  Twice the words cost more L1 than the
    // searches they save (3 -> 5 one pass 28.2 ms).
    static constexpr int U = L == 1 ? 16 : 8;
    static constexpr int BLOOM = L <= 3 ? 256 : 512;
    static constexpr int RP = 0, D = 1, PID = 2, META = 3, CLS = 4, SCN = 5, OPP = 6, SEG = 7, SLO = 8, RLO = 9,
                         RHI = 11, NC = 13, SEO = 15, SS = 16, BND = SS + L, RK = BND + L, OB = RK + L, OE = OB + O, OK = OE + O,
                         VB = OK + 6 * O, VE = VB + 1, EI = VE + 1, QA = EI + 1, END = QA + (QUOTA ? 6 : 0);
    static constexpr int UW = END | 1;               // odd stride: lanes on different units hit different banks
};

template <int L, int PASS, bool QUOTA> struct JoinSmem {
    using R = UnitRec<L, QUOTA>;
    uint32_t unit[8][R::U * R::UW];
    uint32_t bloom[8][R::BLOOM];
    uint32_t q_anchor[8][FSM_JOIN_QUEUE], q_partner[8][FSM_JOIN_QUEUE], q_meta[8][FSM_JOIN_QUEUE];
    uint32_t q_ainfo[8][FSM_JOIN_QUEUE], q_xinfo[8][FSM_JOIN_QUEUE];   // DevGraph::pinfo of anchor, partner
    uint32_t sg_base[8][32], sg_anchor[8][32], sg_slots[8][32], sg_meta[8][32], sg_info[8][32];
    uint32_t seen[8][PASS == PASS_FUSED || PASS == PASS_DOMAIN ? FSM_JOIN_SEEN : 1];
    uint32_t kept;                 // joins the block met (ExtArgs::keep)
};

__device__ __forceinline__ int32_t sorted_has(const int32_t *col, int32_t lo, int32_t end, int32_t x) {
    int32_t hi = end;
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (__ldg(col + mid) < x) lo = mid + 1; else hi = mid;
    }
    return lo < end && __ldg(col + lo) == x;
}

__device__ __forceinline__ int32_t below(const int32_t *a, int32_t n, int32_t x) {
    int32_t lo = 0, hi = n;
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (__ldg(a + mid) < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Option "debug": does index `at` of the piece lists lie in the list a row's partners come from, that of
// the key vertex [rp, rp + d) for a centre row, that of the anchor [al, al + ad) for an end list?
FSM_HD bool partner_in_list(bool centre, int64_t at, int64_t rp, int64_t d, int64_t al, int64_t ad) {
    return centre ? at >= rp && at < rp + d : at >= al && at < al + ad;
}

// Largest u in [lo, hi] with base[u] <= x (base[lo] <= x), by the whole warp: 32 probes per step,
// so a prefix of millions of units takes five dependent reads instead of over twenty.
__device__ __forceinline__ int64_t warp_last_le(const int64_t *base, int64_t lo, int64_t hi, int64_t x) {
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) >> 5;
        const int64_t p = lo + (int64_t)(lane + 1) * step;
        const bool le = p <= hi && __ldg(base + p) <= x;
        const int c = __popc(__ballot_sync(0xffffffffu, le));   // base is nondecreasing: a prefix of the lanes
        lo += (int64_t)c * step;
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

// The next units with pieces, at most `most` (nu of them), from u on: lane's for lane < nu.  uhi >= u has some.
// Units without come alone or in runs of any length (isolated vertices, lists that sampling empties, edges
// outside their quota): 32 are looked at together, and a longer run is passed by one search.
static __device__ __noinline__ int64_t pick_units(const int64_t *base, int64_t u, int64_t uhi, int most, int &nu) {
    const int lane = threadIdx.x & 31;
    unsigned some = __ballot_sync(0xffffffffu, u + lane <= uhi && __ldg(base + u + lane) < __ldg(base + u + lane + 1));
    if (!some) {
        u = warp_last_le(base, u, uhi, __ldg(base + u));
        some = __ballot_sync(0xffffffffu, u + lane <= uhi && __ldg(base + u + lane) < __ldg(base + u + lane + 1));
    }
    nu = min(most, __popc(some));
    for (int x = 0; x < lane && x < nu; ++x) some &= some - 1;
    return u + __ffs(some) - 1;
}

__device__ __forceinline__ unsigned long long rec_u64(const uint32_t *r, int w) {
    return (unsigned long long)r[w] | ((unsigned long long)r[w + 1] << 32);
}
__device__ __forceinline__ void rec_put64(uint32_t *r, int w, unsigned long long x) {
    r[w] = (uint32_t)x;
    r[w + 1] = (uint32_t)(x >> 32);
}

// Row y of the centre pairs that holds pair number q: rows y < c hold y pairs, later rows c
// (c = d when every pair is enumerated).
__device__ __forceinline__ int32_t centre_row(int64_t q, int32_t c, int32_t d) {
    const int64_t nt = (int64_t)c * (c - 1) / 2;
    if (q < nt) {
        int32_t y = (int32_t)((1.0f + sqrtf(1.0f + 8.0f * (float)q)) * 0.5f);
        while ((int64_t)y * (y - 1) / 2 > q) --y;
        while ((int64_t)(y + 1) * y / 2 <= q) ++y;
        return y;
    }
    const int64_t r = q - nt;
    return c + (int32_t)(r <= 0xffffffffll ? (int64_t)((uint32_t)r / (uint32_t)c) : r / c);
}
__device__ __forceinline__ int64_t centre_row_start(int32_t y, int32_t c) {
    return y <= c ? (int64_t)y * (y - 1) / 2 : (int64_t)c * (c - 1) / 2 + (int64_t)(y - c) * c;
}
// the end list of the unit's key vertex that holds end piece number q
__device__ __forceinline__ int32_t end_row(const int32_t *pend, int32_t d, int64_t q) {
    int32_t lo = 0, hi = d - 1;
    while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if ((int64_t)__ldg(pend + mid) <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Eight words of a key record in one request (a join's scattered requests are what the load-store unit
// is busy with).  Records do not change during a pass.
__device__ __forceinline__ void ld_rec8(const uint32_t *p, uint32_t *x) {
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]) : "l"(p));
}

// The rest of a long probe sequence, out of line: a key of a half-full table rarely gets here.  A table that
// overflows is full before its pass stops, and every key would be looked for in FSM_MAX_PROBES slots until
// then: 30k vertices, size 3, from 64 slots up to 2^18, 98.6 ms, 11.9 this way; 37k, size 5, count 3 -> 5, 109 and
// 19.7 ms.  Near probes 8 or 16: 4 -> 6 whole call 18.7 and 18.0 ms, 3 -> 5 one pass 23.4 and 22.3 (18.7 and 22.9
// with all of them inline).  The extension kernel, whose chunks are small, keeps them inline (edge-list quick
// patterns, 100k vertices, size 4: 3.05 s, 3.42 s this way).
#define FSM_NEAR_PROBES 16   // the smallest table has 64 slots
static __device__ __noinline__ int64_t qp_insert_far(unsigned long long *keys, unsigned long long *used, uint64_t mask,
                                                     unsigned long long max_used, uint64_t key, uint64_t h, int *err) {
    QPTab t;
    t.keys = keys;
    t.used = used;
    t.mask = mask;
    t.max_used = max_used;
    for (uint64_t probe = FSM_NEAR_PROBES; probe <= t.mask && probe < FSM_MAX_PROBES; ++probe) {
        if ((probe & 15) == 0 && (*(volatile int *)err & FSM_ERR_QP_OVERFLOW)) return -1;
        if (qp_try(t, key, h, err)) return (int64_t)h;
        h = (h + 1) & t.mask;
    }
    atomicOr(err, FSM_ERR_QP_OVERFLOW);
    return -1;
}

__device__ __forceinline__ int64_t qp_insert_near(const QPTab &t, uint64_t key, int *err) {
    uint64_t h = mix64(key) & t.mask;
    for (int probe = 0; probe < FSM_NEAR_PROBES; ++probe) {
        if (qp_try(t, key, h, err)) return (int64_t)h;
        h = (h + 1) & t.mask;
    }
    return qp_insert_far(t.keys, t.used, t.mask, t.max_used, key, h, err);
}

template <int L, int PASS, bool QUOTA>
struct Joiner {
    using G = JoinGeo<L>;
    using R = UnitRec<L, QUOTA>;
    using SM = JoinSmem<L, PASS, QUOTA>;
    static constexpr int K = L + 2, O = L - 1, SL = L + 1;

    const ExtArgs &A;
    SM &sm;
    const int w, lane;
    int qn = 0;                       // survivors waiting
    int lb = 0;                       // log2 words of one Bloom filter of this batch
    bool tfe;                         // triangles are made from end lists (see take)
    unsigned long long tested = 0, accepted = 0;

    __device__ __forceinline__ Joiner(const ExtArgs &a, SM &s)
        : A(a), sm(s), w(threadIdx.x >> 5), lane(threadIdx.x & 31),
          // An end piece v-a-b with b next to v closes the triangle {v, a, b}; taking it there, once
          // (a < b), costs one Bloom probe on a survivor, where testing every surviving centre pair
          // costs a search.  Kept pieces (sampling) and numbered candidates (quotas) are defined with
          // the triangle at the centre pair, and vertex-induced centre pairs need the test anyway.
          tfe(!QUOTA && a.mode == 0 && !a.sampled) {}

    __device__ __forceinline__ uint32_t *rec(int j) { return sm.unit[w] + j * R::UW; }

    // Two bits of one word stand for a vertex in a Bloom filter: one read tests both (3
    // -> 5 one pass: 23.3 ms with one bit, 22.4 with two).
    __device__ __forceinline__ static uint32_t bloom_mask(uint32_t h) { return (1u << (h & 31)) | (1u << ((h >> 5) & 31)); }
    // x in the list of the t-th smallest vertex of unit j's s?  A clear bit is a certain no.
    __device__ __forceinline__ bool maybe(int j, int t, int32_t x) const {
        const uint32_t h = (uint32_t)x * 0x9E3779B1u, k = bloom_mask(h >> 7);
        return (sm.bloom[w][((j * L + t) << lb) + (lb ? h >> (32 - lb) : 0u)] & k) == k;
    }

    // Slot and bitmap offsets of a key from its record; false where the key has no bitmaps or no record.
    __device__ __forceinline__ bool key_record(uint64_t key, int64_t &slot, uint32_t (&off)[K]) {
        uint64_t h = mix64(key) & A.qp.mask;
        constexpr int RW = key_rec_words(K);
#pragma unroll 1
        for (int p = 0; p < FSM_MAX_PROBES; ++p) {
            const uint32_t *kr = A.key_rec + h * RW;
            uint32_t wd[K > 6 ? 16 : 8];
            ld_rec8(kr, wd);
            if (K > 6) ld_rec8(kr + 8, wd + (K > 6 ? 8 : 0));
            const uint64_t k = (uint64_t)wd[0] | ((uint64_t)wd[1] << 32);
            if (k == key) {
                bool all = true;
#pragma unroll
                for (int x = 0; x < K; ++x) {
                    off[x] = wd[2 + x];
                    all &= off[x] != FSM_OFF_NONE;
                }
                slot = (int64_t)h;
                return all;
            }
            if (k == FSM_EMPTY_KEY) return false;
            h = (h + 1) & A.qp.mask;
        }
        return false;
    }

    // Bits of the join's vertices; those of s (the first L positions) only when `own` is set.
    __device__ __forceinline__ void set_bits(const uint32_t (&off)[K], const uint32_t *r, uint32_t ra, uint32_t rb, bool swap,
                                             bool own) {
        uint32_t *base = PASS == PASS_DOMAIN ? A.dom : A.pool;
        uint32_t *wd[K];
        uint32_t bit[K], old[K];
#pragma unroll
        for (int h = 0; h < K; ++h) {
            const uint32_t rk = h < L ? r[R::RK + (h < L ? h : 0)] : ((h == L) != swap ? ra : rb);
            wd[h] = base + ((uint64_t)off[h] << A.off_shift) + (rk >> 5);
            bit[h] = 1u << (rk & 31);
            old[h] = 0u;
        }
        // A reduction nothing waits for, except on small label classes (ExtArgs::check_bits), whose few
        // words many joins would queue on: there most bits are set already and a read finds that.
        if (A.check_bits) {
#pragma unroll
            for (int h = 0; h < K; ++h)
                if (h >= L || own) old[h] = __ldcg(wd[h]);
        }
#pragma unroll
        for (int h = 0; h < K; ++h)
            if ((h >= L || own) && !(old[h] & bit[h])) atomicOr(wd[h], bit[h]);
    }

    // One-pass level, a key the warm pass did not meet: count the join and leave its bits for after the
    // level, when such keys are resolved in bulk (deferred_bits_kernel).
    __device__ __forceinline__ void defer(const uint32_t *r, uint64_t key, uint32_t r0, uint32_t r1) {
        const int64_t slot = qp_insert_near(A.qp, key, A.err);
        if (slot < 0) return;
        atomicAdd(A.qp.count + slot, 1ull);
        const unsigned long long at = atomicAdd(A.defer_top, 1ull);
        if (at >= A.defer_cap) { atomicOr(A.err, FSM_ERR_CODE_FULL); return; }
        uint32_t *d = A.defer + at * FSM_DEFER_WORDS;
        d[0] = (uint32_t)slot;
#pragma unroll
        for (int h = 0; h < L; ++h) d[1 + h] = r[R::RK + h];
        d[1 + L] = r0;
        d[2 + L] = r1;
    }

    // One more join of key slot `slot`, for the lanes here together: lanes of one key add once.  A few keys
    // that take all of a level's joins (few labels, hubs) queue on their counters otherwise: 30k vertices, 4
    // labels, two hubs of degree 20000, 4e8 joins of 138 keys, 1 -> 3 count 24.6 ms, 6.2 this way; 2 -> 4 one
    // pass, 3.2e9 joins, whole call 114 and 95 ms; 3.7M vertices, 3 -> 5 one pass, 1.6e10 joins, 2410 and 1361 ms.  Where a count pass meets many keys the match only costs
    // (4 -> 6, 2.9e8 joins, whole call 18.5 and 18.9 ms; 1 -> 3, 37 labels, 10.5 and 10.8): ExtArgs::merge.
    __device__ __forceinline__ void count_join(int64_t slot) {
        if (PASS == PASS_FUSED || A.merge) {
            const unsigned same = __match_any_sync(__activemask(), (uint32_t)slot);
            if (lane == __ffs(same) - 1) atomicAdd(A.qp.count + slot, (unsigned long long)__popc(same));
        } else {
            atomicAdd(A.qp.count + slot, 1ull);
        }
    }

    // One accepted join of this lane (not warp-synchronous).
    __device__ __forceinline__ void accept(const uint32_t *r, int j, uint64_t key, bool centre, int32_t anchor, int32_t x,
                                           uint32_t ainfo, uint32_t xinfo, bool swap) {
        if constexpr (PASS == PASS_COUNT) {
            const int64_t slot = qp_insert_near(A.qp, key, A.err);
            if (slot < 0) return;
            count_join(slot);
            if (A.keep) {
                const unsigned act = __activemask();
                const int leader = __ffs(act) - 1;
                uint32_t at = 0;
                if (lane == leader) {
                    at = atomicAdd(&sm.kept, (uint32_t)__popc(act));
                    if (at >> 31) atomicExch(&sm.kept, 1u << 31);   // never wraps round
                }
                at = __shfl_sync(act, at, leader) + __popc(act & ((1u << lane) - 1u));
                if (at < A.keep_cap) {
                    const uint32_t ranchor = A.g.packed ? ainfo >> 6 : (uint32_t)__ldg(A.g.rank + anchor);
                    const uint32_t rx = A.g.packed ? xinfo >> 6 : (uint32_t)__ldg(A.g.rank + x);
                    const bool flip = centre != swap;   // the first new vertex is x
                    __stcs(A.keep + (uint64_t)blockIdx.x * A.keep_cap + at,
                           make_uint4((uint32_t)slot, r[R::EI], flip ? rx : ranchor, flip ? ranchor : rx));
                }
            }
        } else if constexpr (PASS == PASS_FUSED || PASS == PASS_DOMAIN) {
            uint32_t off[K];
            int64_t slot = -1;
            const uint32_t ranchor = A.g.packed ? ainfo >> 6 : (uint32_t)__ldg(A.g.rank + anchor);
            const uint32_t rx = A.g.packed ? xinfo >> 6 : (uint32_t)__ldg(A.g.rank + x);
            const uint32_t ra = centre ? rx : ranchor, rb = centre ? ranchor : rx;
            if (!key_record(key, slot, off)) {
                if (PASS == PASS_FUSED) defer(r, key, swap ? rb : ra, swap ? ra : rb);
                return;   // domain pass: pattern without bitmaps
            }
            if (PASS == PASS_FUSED) count_join(slot);
            // A unit's joins of one key set the same bits of s: a small table of (unit, slot) pairs
            // already seen in this batch keeps most of those reductions away.  A lost entry or a race
            // only repeats them.
            const uint32_t tag = (uint32_t)slot * 16u + (uint32_t)j;
            bool own = slot >= (1 << 28) - 1;      // such slots do not fit the tag
            if (!own) {
                uint32_t *sn = &sm.seen[w][(tag ^ (tag >> 7)) & (FSM_JOIN_SEEN - 1)];
                own = *(volatile uint32_t *)sn != tag;
                if (own) *(volatile uint32_t *)sn = tag;
            }
            set_bits(off, r, ra, rb, swap, own);
        } else {
            const int64_t slot = qp_find(A.qp, key);
            if (slot < 0) { atomicOr(A.err, FSM_ERR_QP_MISSING); return; }
            const int32_t nid = __ldg(A.newid + __ldg(A.qp.pattern + slot));
            if (nid < 0) return;
            const uint64_t perm = __ldg(A.qp.perm + slot);
            const unsigned act = __activemask();
            const int leader = __ffs(act) - 1;
            unsigned long long base = 0;
            if (lane == leader) base = atomicAdd(A.out_cursor, (unsigned long long)__popc(act));
            base = __shfl_sync(act, base, leader);
            const int64_t pos = (int64_t)base + __popc(act & ((1u << lane) - 1u));
            if (pos >= A.out_N) { atomicOr(A.err, FSM_ERR_BOUNDS); return; }
            const uint32_t meta = r[R::META];
            const int32_t a = centre ? x : anchor, b = centre ? anchor : x;
#pragma unroll
            for (int t = 0; t < L; ++t) {
                const int h = (int)(meta >> (12 + 3 * t)) & 7;   // canonical position of the t-th smallest
                A.out_v[(int64_t)nib_get(perm, h) * A.out_N + pos] = (int32_t)r[R::SS + t];
            }
            A.out_v[(int64_t)nib_get(perm, L) * A.out_N + pos] = swap ? b : a;
            A.out_v[(int64_t)nib_get(perm, L + 1) * A.out_N + pos] = swap ? a : b;
            A.out_pid[pos] = nid;
        }
    }

    // Cross edges of a new vertex x to the other vertices of s (bit o: the o-th in id order), and with
    // `key` to the key vertex (bit O).  What the Bloom filters leave is searched, each lane its own
    // list per round, so a warp waits for its longest chain once and not once per list.
    __device__ __forceinline__ uint32_t cross_of(const uint32_t *r, int j, int rv, int32_t x, bool key) const {
        uint32_t c = key && maybe(j, rv, x) ? 1u << O : 0u;
#pragma unroll
        for (int o = 0; o < O; ++o) c |= (uint32_t)maybe(j, o + (o >= rv), x) << o;
        for (uint32_t p = c; p; p &= p - 1) {
            const int o = __ffs(p) - 1;
            if (!sorted_has(A.g.col, (int32_t)r[o == O ? R::VB : R::OB + o], (int32_t)r[o == O ? R::VE : R::OE + o], x))
                c &= ~(1u << o);
        }
        return c;
    }

    // bit o of the result: label lab is in the which-th mask of the o-th other vertex (see load_units)
    __device__ __forceinline__ uint32_t labels_ok(const uint32_t *r, int which, int lab) const {
        uint32_t m = 0;
#pragma unroll
        for (int o = 0; o < O; ++o) m |= ((r[R::OK + 6 * o + 2 * which + (lab >> 5)] >> (lab & 31)) & 1u) << o;
        return m;
    }
    // is label z frequent in row (p, q) of the tab-th size-3 label table?
    __device__ __forceinline__ bool frequent(int tab, int p, int q, int z) const {
        return (__ldg((const uint32_t *)A.lf + 2 * (tab * 4096 + p * 64 + q) + (z >> 5)) >> (z & 31)) & 1u;
    }

    // The anchor's part of a candidate's word.
    __device__ __forceinline__ uint32_t anchor_meta(const uint32_t *r, int j, int32_t anchor, int lab) const {
        const int rv = (r[R::META] >> 3) & 7;
        uint32_t must = 0, no = 0;
        if (A.lf) {   // the anchor is next to the key vertex
            constexpr uint32_t all = (1u << O) - 1u;
            must = ~labels_ok(r, 0, lab) & all;
            no = ~labels_ok(r, 1, lab) & all;
        }
        return (cross_of(r, j, rv, anchor, false) << FSM_M_CROSS) | (must << FSM_M_MUST) | (no << FSM_M_NO);
    }

    // The last n (<= 32) survivors of the queue, one per lane; warp-synchronous.
    __device__ __forceinline__ void take(int n) {
        __syncwarp();
        const bool on = lane < n;
        const int q = qn - n + (on ? lane : 0);
        uint32_t m = sm.q_meta[w][q];
        const int32_t anchor = (int32_t)sm.q_anchor[w][q], x = (int32_t)sm.q_partner[w][q];
        const int j = m & 15;
        const bool centre = !((m >> FSM_M_END) & 1u);
        const uint32_t *r = rec(j);
        const uint32_t meta = r[R::META];
        const int ki = meta & 7, rv = (meta >> 3) & 7, lv = (meta >> 6) & 63;
        const int32_t v = (int32_t)r[R::SS + rv];
        const uint32_t ainfo = sm.q_ainfo[w][q], xinfo = sm.q_xinfo[w][q];
        const int la = ainfo & 63, lx = xinfo & 63;
        if (QUOTA) m |= anchor_meta(r, j, anchor, la);
        // bits of the anchor and of the partner in a cross subset: a's low, b's high
        const int sh_a = centre ? O : 0, sh_x = centre ? 0 : O;
        constexpr uint32_t all = (1u << O) - 1u;
        uint32_t forms = 0;
        if (on) {
            // the piece's own size-3 pattern must be frequent
            if (centre) {
                if (!A.lf || frequent(0, lv, la, lx)) forms |= 1u << FORM_CENTRE;
                if (!tfe && (!A.lf || frequent(2, lv, la, lx))) forms |= 1u << FORM_TRI;
            } else {
                if (!A.lf || frequent(0, la, lv, lx)) forms |= 1u << FORM_END;
                if (tfe && x > anchor && (!A.lf || frequent(2, lv, la, lx))) forms |= 1u << FORM_TRI;
            }
        }
        uint32_t avail = 0, must1 = 0, no1 = 0, no2 = 0;   // 1: partner next to v, 2: not
        const uint32_t mustA = ((m >> FSM_M_MUST) & all) << sh_a, noA = ((m >> FSM_M_NO) & all) << sh_a;
        if (forms) {
            const bool key = tfe ? (forms >> FORM_TRI) & 1u : A.mode == 1 && !centre;
            const uint32_t c = cross_of(r, j, rv, x, key);
            avail = (((m >> FSM_M_CROSS) & all) << sh_a) | ((c & all) << sh_x);
            if (key && !(c >> O)) forms &= tfe ? ~(1u << FORM_TRI) : ~0u;   // no triangle here
            if (key && (c >> O) && !tfe) forms = 0;                         // vertex-induced: only the triangle
            if (A.lf) {
                must1 = (~labels_ok(r, 0, lx) & all) << sh_x;
                no1 = (~labels_ok(r, 1, lx) & all) << sh_x;
                no2 = (~labels_ok(r, 2, lx) & all) << sh_x;
            }
        }
        const int sA = (m >> FSM_M_SA) & 7, sX = (m >> FSM_M_SP) & 7;
        const bool later = x > anchor;   // partner after anchor; b > a for an end list, always for the others
        const uint32_t *rows = A.acc + ((int64_t)r[R::CLS] * G::ROWS + ((centre ? sX : sA) * SL + (centre ? sA : sX)) * 2 +
                                        (centre || later)) * G::W;
        auto row_of = [&](int f) { return rows + (int64_t)f * (SL * SL * 2) * G::W; };
        if (!tfe && centre && forms) {
            // a ~ b decides between wedge and triangle: searched only where the answer matters
            if (A.mode == 1) {
#pragma unroll
                for (int f = FORM_CENTRE; f <= FORM_TRI; f += 2)
                    if ((forms >> f & 1u) && (((mustA | must1) & ~avail) || ((noA | no1) & avail) ||
                                              !((__ldg(row_of(f) + (avail >> 5)) >> (avail & 31)) & 1u)))
                        forms &= ~(1u << f);
            }
            if (A.mode == 1 ? forms != 0 : (forms >> FORM_TRI) & 1u) {
                const int4 ia = __ldg(A.g.vinfo + anchor), ix = __ldg(A.g.vinfo + x);
                const bool shorter = ia.y - ia.x <= ix.y - ix.x;
                const bool tri = shorter ? sorted_has(A.g.col, ia.x, ia.y, x) : sorted_has(A.g.col, ix.x, ix.y, anchor);
                if (!tri) forms &= ~(1u << FORM_TRI);
                else if (A.mode == 1) forms &= ~(1u << FORM_CENTRE);
            }
        }
        const int32_t a = centre ? x : anchor, b = centre ? anchor : x;
        const int la_ = centre ? lx : la, lb_ = centre ? la : lx;
        const bool ab = lab_id_less(la_, a, lb_, b);
        auto piece = [&](int form, int &jpos) -> uint32_t {
            const bool vb = lab_id_less(lv, v, lb_, b);
            if (form == FORM_CENTRE) {
                jpos = 0;
                return piece_index(PIECE_WEDGE, lv, ab ? la_ : lb_, ab ? lb_ : la_);
            }
            if (form == FORM_END) {
                jpos = vb ? 1 : 2;
                return piece_index(PIECE_WEDGE, la_, vb ? lv : lb_, vb ? lb_ : lv);
            }
            jpos = (lab_id_less(lv, v, la_, a) ? 0 : 1) + (vb ? 0 : 1);
            return tri_index(lv, la_, lb_);
        };
        if (A.piece_sel && forms) {
            int jp;
#pragma unroll
            for (int f = 0; f < 3; ++f)
                if ((forms >> f & 1u) && !__ldg(A.piece_sel + piece(f, jp))) forms &= ~(1u << f);
        }
        int form = 0;
        uint32_t must = 0, free_ = 0, cur = 0, sub = 0;
        bool more = false;
        const uint32_t *row = rows;
        uint32_t roww = 0;
        for (;;) {
            bool have = false;
            while (!have) {
                if (!more) {
                    if (!forms) break;
                    form = __ffs(forms) - 1;
                    forms &= forms - 1;
                    const uint32_t no = noA | (form == FORM_END ? no2 : no1);
                    must = mustA | (form == FORM_END ? 0u : must1);
                    if ((must & ~avail) || (must & no)) continue;
                    if (A.mode == 0) {
                        free_ = avail & ~no & ~must;
                    } else {
                        if (avail & no) continue;
                        must = avail;   // vertex-induced: every cross edge
                        free_ = 0;
                    }
                    cur = free_;
                    row = row_of(form);
                    if (G::W == 1) {
                        roww = __ldg(row);
                        if (!roww) continue;
                    }
                    more = true;
                }
                sub = cur | must;
                ++tested;
                have = ((G::W == 1 ? roww : __ldg(row + (sub >> 5))) >> (sub & 31)) & 1u;
                if (cur == 0) more = false; else cur = (cur - 1) & free_;
            }
            if (!__any_sync(0xffffffffu, have)) break;
            if (have) {
                ++accepted;
                int jpos;
                const uint32_t pidx = piece(form, jpos);
                const bool swap = form != FORM_END && !ab;   // the key's first new vertex is b
                uint32_t cross = 0;
                const uint32_t opp = r[R::OPP];
#pragma unroll
                for (int o = 0; o < O; ++o) {
                    const int pp = (opp >> (3 * o)) & 7;
                    cross |= ((sub >> o) & 1u) << (2 * pp + (swap ? 1 : 0));
                    cross |= ((sub >> (O + o)) & 1u) << (2 * pp + (swap ? 0 : 1));
                }
                accept(r, j, make_key(r[R::PID], pidx, ki, jpos, cross, L), centre, anchor, x, ainfo, xinfo, swap);
            }
        }
        qn -= n;
        __syncwarp();
    }

    // warp-synchronous: queue the survivors among the lanes' candidates; join when 32 wait, or what
    // there is when nothing more comes (`drain`)
    __device__ __forceinline__ void push(bool ok, int32_t anchor, int32_t x, uint32_t m, uint32_t ainfo, uint32_t xinfo,
                                         bool drain) {
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        if (ok) {
            const int p = qn + __popc(bal & ((1u << lane) - 1u));
            sm.q_anchor[w][p] = (uint32_t)anchor;
            sm.q_partner[w][p] = (uint32_t)x;
            sm.q_meta[w][p] = m;
            sm.q_ainfo[w][p] = ainfo;
            sm.q_xinfo[w][p] = xinfo;
        }
        qn += __popc(bal);
        if (qn >= 32 || (drain && qn > 0)) take(min(qn, 32));
    }

    // Load units u0 .. u0 + nu - 1 (raw candidate range [q0, q1) of the chunk) into shared memory.
    __device__ __forceinline__ void load_units(int64_t u, int nu, int64_t q0, int64_t q1) {
        const DevGraph &g = A.g;
        uint32_t *r = rec(lane < nu ? lane : 0);
        int nseg = 0;
        if (lane < nu) {
            const int64_t e = A.e0 + u / L;
            const int iu = (int)(u % L);
            r[R::EI] = (uint32_t)e;
            const int32_t pid = __ldg(A.fpid + e);
            const uint64_t srows = L >= 2 ? __ldg(A.pat_adj + pid) : 0ull;
            int32_t id[L];
            int cp[L];
#pragma unroll
            for (int p = 0; p < L; ++p) { id[p] = __ldg(A.fv + (int64_t)p * A.fN + e); cp[p] = p; }
            // sort by id, carrying canonical positions
#pragma unroll
            for (int x = 1; x < L; ++x)
#pragma unroll
                for (int y = L - 1; y >= x; --y)
                    if (id[y] < id[y - 1]) {
                        const int32_t ti = id[y]; id[y] = id[y - 1]; id[y - 1] = ti;
                        const int tc = cp[y]; cp[y] = cp[y - 1]; cp[y - 1] = tc;
                    }
            int rv = 0, lv = 0;
            int32_t v = 0;
            int4 nfo[L];
            uint32_t meta = (uint32_t)iu;
#pragma unroll
            for (int t = 0; t < L; ++t) {
                nfo[t] = __ldg(g.vinfo + id[t]);
                if (cp[t] == iu) {
                    rv = t;
                    v = id[t];
                    lv = nfo[t].z;
                    r[R::VB] = (uint32_t)nfo[t].x;
                    r[R::VE] = (uint32_t)nfo[t].y;
                }
                meta |= (uint32_t)cp[t] << (12 + 3 * t);
                r[R::SS + t] = (uint32_t)id[t];
                r[R::RK + cp[t]] = (uint32_t)nfo[t].w;
            }
            meta |= ((uint32_t)rv << 3) | ((uint32_t)lv << 6);
            uint32_t cls = (uint32_t)rv << G::EB;
            int bit = 0;
#pragma unroll
            for (int t = 0; t < L; ++t)
#pragma unroll
                for (int t2 = t + 1; t2 < L; ++t2, ++bit)
                    cls |= ((uint32_t)(srows >> (8 * cp[t] + cp[t2])) & 1u) << bit;
            const int32_t rp = __ldg(g.prow + v), d = __ldg(g.prow + v + 1) - rp;
            r[R::RP] = (uint32_t)rp;
            r[R::D] = (uint32_t)d;
            r[R::PID] = (uint32_t)pid;
            r[R::META] = meta;
            r[R::CLS] = cls;
            uint32_t opp = 0;
#pragma unroll
            for (int t = 0; t < L; ++t) {
                if (t == rv) continue;
                const int o = t - (t > rv);
                const int lo = nfo[t].z;
                opp |= (uint32_t)(cp[t] < iu ? cp[t] : cp[t] - 1) << (3 * o);
                r[R::OB + o] = (uint32_t)nfo[t].x;
                r[R::OE + o] = (uint32_t)nfo[t].y;
                if (A.lf) {
                    // labels of a new vertex x with which {v, o, x} may be left as it is:
                    // k0 x next to v only, k1 next to v and o, k2 next to o only
                    const bool e1 = (srows >> (8 * iu + cp[t])) & 1ull;
                    const unsigned long long k0 = e1 ? __ldg(A.lf + lv * 64 + lo) : ~0ull;
                    const unsigned long long k1 = __ldg(A.lf + (e1 ? 8192 : 4096) + lv * 64 + lo);
                    const unsigned long long k2 = e1 ? __ldg(A.lf + lo * 64 + lv) : ~0ull;
                    rec_put64(r, R::OK + 6 * o, k0);
                    rec_put64(r, R::OK + 6 * o + 2, k1);
                    rec_put64(r, R::OK + 6 * o + 4, k2);
                }
            }
            r[R::OPP] = opp;
            int32_t cpos = d;
#pragma unroll 1
            for (int t = 0; t < L; ++t) {
                const int32_t bd = below(g.pcol + rp, d, (int32_t)r[R::SS + t]);
                r[R::BND + t] = (uint32_t)bd;
                if (L == 2 && t != rv) cpos = bd;
            }
            const int64_t nc = L == 2 ? centre_pairs(d, cpos) : (int64_t)d * (d - 1) / 2;
            rec_put64(r, R::NC, (unsigned long long)nc);
            const int64_t ub = __ldg(A.unit_base + u), ue = __ldg(A.unit_base + u + 1);
            const int64_t lo = max(q0 - ub, (int64_t)0), hi = min(q1, ue) - ub;
            rec_put64(r, R::RLO, (unsigned long long)lo);
            rec_put64(r, R::RHI, (unsigned long long)hi);
            if constexpr (QUOTA) {
                // the unit's candidates before the quota cut (as the prefix kernel counted)
                const int64_t c = nc + (__ldg(g.ppc + v) - (int64_t)d * (d - 1) / 2);
                unsigned long long qa = 0, qb = 0, qc = 0;
                if (A.quota > 0 && c > A.quota) {
                    uint64_t x, y;
                    quota_affine(quota_unit_hash(A.qseed, id, L, v), (uint64_t)c, x, y);
                    qa = x;
                    qb = y;
                    qc = (unsigned long long)c;
                }
                rec_put64(r, R::QA, qa);
                rec_put64(r, R::QA + 2, qb);
                rec_put64(r, R::QA + 4, qc);
                nseg = (int)(hi > lo ? hi - lo : 0);   // candidates of this unit in the chunk
                r[R::SLO] = 0;
            } else {
                // rows of the chunk: centre rows [c0, c1), end lists [e0, e1)
                int32_t c0 = 0, c1 = 0, e0 = 0, e1 = 0;
                if (hi > lo) {
                    if (lo < nc) {
                        c0 = lo <= 0 ? 0 : centre_row(lo, cpos, d);
                        c1 = hi >= nc ? d : centre_row(hi - 1, cpos, d) + 1;
                    }
                    if (hi > nc) {
                        e0 = lo <= nc ? 0 : end_row(g.pend + rp, d, lo - nc);
                        e1 = hi >= ue - ub ? d : end_row(g.pend + rp, d, hi - 1 - nc) + 1;
                    }
                    // and of those only the anchors in slots that allow some partner (1 -> 3: every row
                    // whose anchor is below the key vertex goes; 3.7M vertices, count 4.56 -> 4.18 ms)
#pragma unroll 1
                    for (int k = 0; k < 2; ++k) {
                        int a0 = SL, a1 = -1;
#pragma unroll 1
                        for (int t = 0; t < SL; ++t) {
                            uint32_t ok = allowed(r, k == 0, t);
                            if (k == 0) ok &= (1u << SL) - 1u;
                            if (ok) { a0 = min(a0, t); a1 = t; }
                        }
                        const int32_t p0 = a1 < 0 ? d : a0 > 0 ? (int32_t)r[R::BND + a0 - 1] : 0;
                        const int32_t p1 = a1 < L ? (a1 < 0 ? 0 : (int32_t)r[R::BND + a1]) : d;
                        if (k == 0) { c0 = max(c0, p0); c1 = min(c1, p1); }
                        else { e0 = max(e0, p0); e1 = min(e1, p1); }
                    }
                }
                c1 = max(c1, c0);
                e1 = max(e1, e0);
                r[R::SLO] = (uint32_t)c0;
                r[R::SCN] = (uint32_t)(c1 - c0);
                r[R::SEO] = (uint32_t)e0;
                nseg = (c1 - c0) + (e1 - e0);
            }
        }
        int inc = nseg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane < nu) r[R::SEG] = (uint32_t)(inc - nseg);
        total_seg = __shfl_sync(0xffffffffu, inc, 31);
        // Bloom filters of the lists of s (of the key vertex only where end pieces are tested for
        // closing a triangle)
        int bw = R::BLOOM / (nu * L);
        lb = 31 - __clz(bw);
        __syncwarp();
        for (int x = lane; x < R::BLOOM; x += 32) sm.bloom[w][x] = 0u;
        if (PASS == PASS_FUSED || PASS == PASS_DOMAIN)
            for (int x = lane; x < FSM_JOIN_SEEN; x += 32) sm.seen[w][x] = 0xFFFFFFFFu;
        __syncwarp();
        for (int j = 0; j < nu; ++j) {
            const uint32_t *rj = rec(j);
            const int rv = (rj[R::META] >> 3) & 7;
#pragma unroll 1
            for (int t = 0; t < L; ++t) {
                int32_t x0, x1;
                if (t == rv) {
                    if (!tfe && A.mode == 0) continue;
                    x0 = (int32_t)rj[R::VB];
                    x1 = (int32_t)rj[R::VE];
                } else {
                    const int o = t - (t > rv);
                    x0 = (int32_t)rj[R::OB + o];
                    x1 = (int32_t)rj[R::OE + o];
                }
                // A list longer than its filter has bits would answer maybe for nearly every vertex, and to read it
                // for each batch that holds a hub costs more than the searches it leaves where quotas draw a
                // few pieces of each unit (30k vertices, two hubs of degree 20000, quota 2, 2 -> 4 count of 2.1e5
                // pieces: 2.7 and 0.16 ms; 20 hubs of degree 2000, 3 -> 5: 221 and 90 ms): all bits are set.
                // Elsewhere units have pieces enough, and the test costs 3 -> 5 one pass 1 %.
                if (QUOTA && x1 - x0 > 32 << lb) {
#pragma unroll 1
                    for (int x = lane; x < 1 << lb; x += 32) sm.bloom[w][((j * L + t) << lb) + x] = 0xFFFFFFFFu;
                    x1 = x0;
                }
                for (int32_t x = x0 + lane; x < x1; x += 32) {
                    const uint32_t h = (uint32_t)__ldg(g.col + x) * 0x9E3779B1u;
                    atomicOr(&sm.bloom[w][((j * L + t) << lb) + (lb ? h >> (32 - lb) : 0u)], bloom_mask(h >> 7));
                }
            }
        }
        __syncwarp();
    }
    int total_seg = 0;

    __device__ __forceinline__ int unit_of(int g, int nu) {
        int lo = 0;
#pragma unroll
        for (int s = R::U / 2; s > 0; s >>= 1)
            if (lo + s < nu && (int)rec(lo + s)[R::SEG] <= g) lo += s;
        return lo;
    }

    // slots of a partner the row's anchor allows: bit (slot + (partner > anchor ? SL : 0))
    __device__ __forceinline__ uint32_t allowed(const uint32_t *r, bool centre, int s) {
        const int kind = centre ? (tfe ? ANY_C : ANY_CT) : (tfe ? ANY_ET : ANY_E);
        return __ldg(A.any + ((int64_t)r[R::CLS] * 4 + kind) * SL + s);
    }

    // The candidates of the loaded units, row by row.
    __device__ __forceinline__ void walk(int nu) {
        const DevGraph &g = A.g;
        for (int g0 = 0;; g0 += 32) {
            const bool drain = g0 >= total_seg;   // one round more joins what is left in the queue
            int len = 0;
            const int gi = g0 + lane;
            if (gi < total_seg) {
                const int j = unit_of(gi, nu);
                const uint32_t *r = rec(j);
                const int row = gi - (int)r[R::SEG], ncr = (int)r[R::SCN];
                const int32_t rp = (int32_t)r[R::RP], d = (int32_t)r[R::D];
                const bool centre = row < ncr;
                const int32_t y = centre ? (int32_t)r[R::SLO] + row : (int32_t)r[R::SEO] + row - ncr;
                if (A.debug && (y < 0 || y >= d)) {
                    atomicOr(A.err, FSM_ERR_BOUNDS);
                } else {
                    const int32_t anchor = __ldg(g.pcol + rp + y);
                    const uint32_t ainfo = __ldg(g.pinfo + rp + y);
                    bool in = false;
                    int s = 0;
#pragma unroll
                    for (int t = 0; t < L; ++t) {
                        const int32_t x = (int32_t)r[R::SS + t];
                        in |= x == anchor;
                        s += x < anchor;
                    }
                    uint32_t ok = in ? 0u : allowed(r, centre, s);
                    if (centre) ok &= (1u << SL) - 1u;
                    uint32_t m = 0;
                    if (ok) {
                        m = anchor_meta(r, j, anchor, ainfo & 63) | (uint32_t)j | ((centre ? 0u : 1u) << FSM_M_END) |
                            ((uint32_t)s << FSM_M_SA);
                        const uint32_t all = (1u << O) - 1u;
                        const uint32_t c = m >> FSM_M_CROSS, must = m >> FSM_M_MUST, no = m >> FSM_M_NO;
                        // pruning rejects the anchor with any partner
                        if (((must & (~c | no)) | (A.mode == 1 ? c & no : 0u)) & all) ok = 0;
                    }
                    if (ok) {
                        const int64_t lo = (int64_t)rec_u64(r, R::RLO), hi = (int64_t)rec_u64(r, R::RHI);
                        const uint32_t slots = (ok | (ok >> SL)) & ((1u << SL) - 1u);
                        const int s0 = __ffs(slots) - 1, s1 = 31 - __clz(slots);
                        int32_t p0, p1;      // partner positions within its list
                        int32_t lb0;         // that list's begin
                        if (centre) {
                            int32_t cpos = d;
                            if (L == 2) cpos = (int32_t)r[R::BND + (((r[R::META] >> 3) & 7) ? 0 : 1)];
                            const int64_t st = centre_row_start(y, cpos);
                            p0 = (int32_t)max(lo - st, (int64_t)0);
                            p1 = (int32_t)min(hi - st, (int64_t)min(y, cpos));
                            if (s0 > 0) p0 = max(p0, (int32_t)r[R::BND + s0 - 1]);
                            if (s1 < L) p1 = min(p1, (int32_t)r[R::BND + s1]);
                            lb0 = rp;
                        } else {
                            const int64_t st = (int64_t)rec_u64(r, R::NC) + __ldg(g.pend + rp + y);
                            lb0 = __ldg(g.prow + anchor);
                            const int32_t da = __ldg(g.prow + anchor + 1) - lb0;
                            p0 = (int32_t)max(lo - st, (int64_t)0);
                            p1 = (int32_t)min(hi - st, (int64_t)da);
                            // cut to the allowed slots (lists of a few entries are walked whole)
                            if (p1 - p0 > 4) {
                                if (s0 > 0) p0 = max(p0, below(g.pcol + lb0, da, (int32_t)r[R::SS + s0 - 1]));
                                if (s1 < L) p1 = min(p1, below(g.pcol + lb0, da, (int32_t)r[R::SS + s1]));
                            }
                        }
                        len = max(p1 - p0, 0);
                        sm.sg_base[w][lane] = (uint32_t)(lb0 + p0);
                        sm.sg_anchor[w][lane] = (uint32_t)anchor;
                        sm.sg_slots[w][lane] = ok;
                        sm.sg_meta[w][lane] = m;
                        sm.sg_info[w][lane] = ainfo;
                    }
                }
            }
            int inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            const int total = __shfl_sync(0xffffffffu, inc, 31);
            __syncwarp();
            sm.sg_base[w][lane] -= (uint32_t)(inc - len);   // list index of candidate t is base + t
            __syncwarp();
            for (int t0 = 0; t0 < total || (drain && t0 == 0); t0 += 32) {
                const int t = t0 + lane;
                int k = 0;
#pragma unroll
                for (int s = 16; s > 0; s >>= 1)
                    if (__shfl_sync(0xffffffffu, inc, k + s - 1) <= t) k += s;
                bool ok = t < total;
                int32_t x = 0, anchor = 0;
                uint32_t m = 0, ainfo = 0, xinfo = 0;
                if (ok) {
                    ainfo = sm.sg_info[w][k];
                    m = sm.sg_meta[w][k];
                    anchor = (int32_t)sm.sg_anchor[w][k];
                    const int64_t at = (int64_t)(int32_t)(sm.sg_base[w][k] + (uint32_t)t);
                    const uint32_t *r = rec(m & 15);
                    bool in = true;
                    if (A.debug) {
                        const int32_t al = __ldg(g.prow + anchor);
                        in = partner_in_list(!((m >> FSM_M_END) & 1u), at, (int32_t)r[R::RP], (int32_t)r[R::D], al,
                                             __ldg(g.prow + anchor + 1) - al);
                    }
                    if (!in) {
                        atomicOr(A.err, FSM_ERR_BOUNDS);
                        ok = false;
                    } else {
                        x = __ldg(g.pcol + at);
                        xinfo = __ldg(g.pinfo + at);
                        int s = 0;
#pragma unroll
                        for (int t2 = 0; t2 < L; ++t2) {
                            const int32_t y = (int32_t)r[R::SS + t2];
                            ok &= y != x;
                            s += y < x;
                        }
                        m |= (uint32_t)s << FSM_M_SP;
                        ok &= (sm.sg_slots[w][k] >> (s + (x > anchor ? SL : 0))) & 1u;
                    }
                }
                push(ok, anchor, x, m, ainfo, xinfo, drain);
            }
            __syncwarp();
            if (drain) break;
        }
    }

    // Quota variant: the drawn candidates of the loaded units, by their numbers.
    __device__ __forceinline__ void walk_quota(int nu) {
        const DevGraph &g = A.g;
        for (int g0 = 0;; g0 += 32) {
            const bool drain = g0 >= total_seg;
            const int gi = g0 + lane;
            bool ok = gi < total_seg;
            int32_t anchor = 0, x = 0;
            uint32_t m = 0, ainfo = 0, xinfo = 0;
            if (ok) {
                const int j = unit_of(gi, nu);
                const uint32_t *r = rec(j);
                int64_t lq = (int64_t)rec_u64(r, R::RLO) + (gi - (int)r[R::SEG]);
                const unsigned long long qc = rec_u64(r, R::QA + 4);
                if (qc) lq = (int64_t)((rec_u64(r, R::QA) * (unsigned long long)lq + rec_u64(r, R::QA + 2)) % qc);
                const int64_t nc = (int64_t)rec_u64(r, R::NC);
                const int32_t rp = (int32_t)r[R::RP], d = (int32_t)r[R::D];
                const bool centre = lq < nc;
                if (centre) {
                    int32_t cpos = d;
                    if (L == 2) cpos = (int32_t)r[R::BND + (((r[R::META] >> 3) & 7) ? 0 : 1)];
                    const int32_t y = centre_row(lq, cpos, d);
                    const int32_t p = (int32_t)(lq - centre_row_start(y, cpos));
                    if (A.debug && (p < 0 || p >= y || y >= d)) { atomicOr(A.err, FSM_ERR_BOUNDS); ok = false; }
                    if (ok) {
                        anchor = __ldg(g.pcol + rp + y);
                        ainfo = __ldg(g.pinfo + rp + y);
                        x = __ldg(g.pcol + rp + p);
                        xinfo = __ldg(g.pinfo + rp + p);
                    }
                } else {
                    const int32_t y = end_row(g.pend + rp, d, lq - nc);
                    const int64_t p = lq - nc - __ldg(g.pend + rp + y);
                    anchor = __ldg(g.pcol + rp + y);
                    ainfo = __ldg(g.pinfo + rp + y);
                    const int32_t lb0 = __ldg(g.prow + anchor);
                    if (A.debug && (p < 0 || p >= __ldg(g.prow + anchor + 1) - lb0)) { atomicOr(A.err, FSM_ERR_BOUNDS); ok = false; }
                    if (ok) {
                        x = __ldg(g.pcol + lb0 + p);
                        xinfo = __ldg(g.pinfo + lb0 + p);
                    }
                }
                int s = 0, sx = 0;
#pragma unroll
                for (int t = 0; t < L; ++t) {
                    const int32_t y = (int32_t)r[R::SS + t];
                    ok &= y != anchor && y != x;
                    s += y < anchor;
                    sx += y < x;
                }
                if (ok) ok = (allowed(r, centre, s) >> (sx + (x > anchor ? SL : 0))) & 1u;
                m = (uint32_t)j | ((centre ? 0u : 1u) << FSM_M_END) | ((uint32_t)s << FSM_M_SA) | ((uint32_t)sx << FSM_M_SP);
            }
            push(ok, anchor, x, m, ainfo, xinfo, drain);
            if (drain) break;
        }
    }

};

// Resident blocks per SM: four (64 registers) hide more latency in the count and emission passes
// (3.7M vertices, 1 -> 3: 5.2 ms against 6.1 ms with three) and in the domain pass and the one-pass
// level up to l = 3 (domain 11.4 and 12.6 ms); those of l = 4 and 5 spill too much at 64 registers
// (4 -> 6 domain pass: 14.5 and 13.7 ms).
template <int L, int PASS> struct JoinBlocks {
    static constexpr int value = (PASS == PASS_FUSED || PASS == PASS_DOMAIN) && L >= 4 ? 3 : 4;
};

template <int L, int PASS, bool QUOTA>
__global__ void __launch_bounds__(256, JoinBlocks<L, PASS>::value) join_kernel(const __grid_constant__ ExtArgs A) {
    extern __shared__ __align__(16) unsigned char join_smem[];
    using J = Joiner<L, PASS, QUOTA>;
    typename J::SM &sm = *reinterpret_cast<typename J::SM *>(join_smem);
    J jn(A, sm);
    const int lane = jn.lane;
    const int64_t nunits = A.ne * L;
    int64_t total = A.total, nchunks = A.nchunks, chunk = A.chunk;
    if (total < 0) {
        // device-resident size: no host round trip between the prefix sum and this launch
        total = __ldg(A.unit_base + nunits);
        if (chunk <= 0) chunk = join_chunk(total, nunits, (int64_t)gridDim.x * (blockDim.x >> 5));
        nchunks = (total + chunk - 1) / chunk;
    }
    int64_t stride = 1;
    if (A.warm) {   // a sample: every stride-th chunk
        stride = warm_stride(total);
        chunk = min(chunk, (int64_t)FSM_WARM_CHUNK);
        nchunks = ((total + chunk - 1) / chunk + stride - 1) / stride;
    }
    if (PASS == PASS_COUNT && A.keep) {
        if (threadIdx.x == 0) sm.kept = 0;
        __syncthreads();
    }
    if (A.stats && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(A.stats + 2, (unsigned long long)total);
    for (;;) {
        unsigned long long c = 0;
        if (lane == 0) {
            // stop early when the call ran out of time, when an overflowing count pass is to be
            // repeated with a larger table, or when a one-pass level is to be redone in two passes
            const int ew = *(volatile int *)A.err;
            bool stop = (ew & FSM_ERR_TIMEOUT) || (PASS == PASS_COUNT && (ew & FSM_ERR_QP_OVERFLOW)) ||
                        (PASS == PASS_FUSED && ew);
            if (!stop && A.time_limit_ns && global_ns() - __ldcg(A.time_start) > A.time_limit_ns) {
                atomicOr(A.err, FSM_ERR_TIMEOUT);
                stop = true;
            }
            c = stop ? ~0ull : atomicAdd(A.chunk_ctr, 1ull);
        }
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= (unsigned long long)nchunks) break;
        const int64_t q0 = (int64_t)c * stride * chunk;
        const int64_t q1 = min(q0 + chunk, total);
        const int64_t ulo = warp_last_le(A.unit_base, 0, nunits - 1, q0);
        const int64_t uhi = warp_last_le(A.unit_base, ulo, nunits - 1, q1 - 1);
        // From the first batch that had fewer rows than units, the chunk's next ones are made of units that
        // have pieces.  Loading whatever comes next made one warp load millions of empty units (8.4M
        // isolated vertices between two halves of a graph, size 4: 3.3 s a mine, now 3.5 ms) and sampled
        // levels load mostly empty ones (370k vertices, size 5, rate 1e-5: 146 ms, now 3; rate 1e-3: 21
        // and 11).  Looking for them before every batch cost 3 -> 5 one pass 9 % where none are empty, as
        // it is 1 % (74k vertices, whole call 22.6 and 22.9 ms).
        bool thin = false;
        for (int64_t u = ulo; u <= uhi; u += J::R::U) {
            int nu = (int)min((int64_t)J::R::U, uhi - u + 1);
            int64_t mu = u + lane;
            if (thin) {
                mu = pick_units(A.unit_base, u, uhi, J::R::U, nu);
                u = __shfl_sync(0xffffffffu, mu, nu - 1) + 1 - J::R::U;
            }
            jn.load_units(mu, nu, q0, q1);
            thin |= jn.total_seg < nu;
            if constexpr (QUOTA) jn.walk_quota(nu); else jn.walk(nu);
        }
    }

    if (PASS == PASS_COUNT && A.keep) {
        __syncthreads();
        if (threadIdx.x == 0) {
            A.keep_n[blockIdx.x] = min(sm.kept, A.keep_cap);
            if (sm.kept > A.keep_cap) atomicAdd(A.keep_over, 1ull);
        }
    }
    // per-warp totals, one atomic per warp
    unsigned long long t0 = jn.tested, t1 = jn.accepted;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t0 += __shfl_xor_sync(0xffffffffu, t0, o);
        t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    }
    if (lane == 0 && A.stats) {
        atomicAdd(A.stats + 0, t0);
        atomicAdd(A.stats + 1, t1);
    }
}

template <int L, int PASS, bool QUOTA>
cudaError_t join_launch(const ExtArgs &A, int grid, cudaStream_t st) {
    join_kernel<L, PASS, QUOTA><<<grid, 256, sizeof(JoinSmem<L, PASS, QUOTA>), st>>>(A);
    return cudaGetLastError();
}

// resident blocks per SM; also opts the kernel into its shared memory on the current device
template <int L, int PASS, bool QUOTA>
cudaError_t join_occupancy(int *bps) {
    const int bytes = (int)sizeof(JoinSmem<L, PASS, QUOTA>);
    cudaError_t e = cudaFuncSetAttribute(join_kernel<L, PASS, QUOTA>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, join_kernel<L, PASS, QUOTA>, 256, bytes);
}

// One pass's instantiations: launch (bps == NULL) or query occupancy.  Defined in one translation
// unit per pass (join_<pass>), so they compile in parallel.
template <int PASS, bool QUOTA>
cudaError_t join_pass(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps) {
    switch (L) {
    case 1: return bps ? join_occupancy<1, PASS, QUOTA>(bps) : join_launch<1, PASS, QUOTA>(*A, grid, st);
    case 2: return bps ? join_occupancy<2, PASS, QUOTA>(bps) : join_launch<2, PASS, QUOTA>(*A, grid, st);
    case 3: return bps ? join_occupancy<3, PASS, QUOTA>(bps) : join_launch<3, PASS, QUOTA>(*A, grid, st);
    case 4: return bps ? join_occupancy<4, PASS, QUOTA>(bps) : join_launch<4, PASS, QUOTA>(*A, grid, st);
    case 5: return bps ? join_occupancy<5, PASS, QUOTA>(bps) : join_launch<5, PASS, QUOTA>(*A, grid, st);
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t join_count(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);
cudaError_t join_domain(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);
cudaError_t join_emit(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);
cudaError_t join_fused(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);
cudaError_t join_quota_count(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);
cudaError_t join_quota_domain(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);
cudaError_t join_quota_emit(int L, const ExtArgs *A, int grid, cudaStream_t st, int *bps);

} // namespace fsm
