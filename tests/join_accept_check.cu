// Host check of the join kernel's acceptance rule (join_accepted, fsm_join.cuh), which sees a join
// only through its class, form, slots and cross subset, against dissect3 (Algorithm 1) on the
// joined graph with its own ids: random connected s of 2..5 vertices in random id order, every
// key position, form and cross subset, new vertices in random slots.  Built and run by
// tests/test_join_accept.py; host code only.
#include "fsm_join.cuh"
#include <cstdio>
using namespace fsm;

static uint64_t state = 12345;
static uint32_t rnd(uint32_t n) { return (uint32_t)(splitmix_step(state++) % n); }
static long checked = 0, kept = 0, bad = 0;

template <int L> static void run(int rounds) {
    constexpr int K = L + 2, O = L - 1;
    for (int it = 0; it < rounds; ++it) {
        int32_t gid[K];                  // s in stored order, then a, b: distinct ids
        for (int h = 0; h < K;) {
            gid[h] = (int32_t)rnd(50);
            bool ok = true;
            for (int x = 0; x < h; ++x) ok &= gid[x] != gid[h];
            h += ok;
        }
        uint32_t sadj[L];
        do {
            for (int h = 0; h < L; ++h) sadj[h] = 0;
            for (int x = 0; x < L; ++x)
                for (int y = x + 1; y < L; ++y)
                    if (rnd(2)) { sadj[x] |= 1u << y; sadj[y] |= 1u << x; }
        } while (!mask_connected((1u << L) - 1u, sadj, L));
        int cp[L];                       // stored position of the t-th smallest id
        for (int t = 0; t < L; ++t) cp[t] = t;
        for (int x = 1; x < L; ++x)
            for (int y = x; y > 0 && gid[cp[y - 1]] > gid[cp[y]]; --y) { int t = cp[y]; cp[y] = cp[y - 1]; cp[y - 1] = t; }
        int sa = 0, sb = 0;
        for (int h = 0; h < L; ++h) { sa += gid[h] < gid[L]; sb += gid[h] < gid[L + 1]; }
        for (int i = 0; i < L; ++i)
            for (int form = 0; form < 3; ++form) {
                if (form != FORM_END && gid[L] > gid[L + 1]) continue;   // those pieces keep a < b
                int rv = 0;
                while (cp[rv] != i) ++rv;
                int cls = rv << JoinGeo<L>::EB, bit = 0;
                for (int t = 0; t < L; ++t)
                    for (int u = t + 1; u < L; ++u, ++bit) cls |= (int)((sadj[cp[t]] >> cp[u]) & 1u) << bit;
                for (uint32_t sub = 0; sub < (1u << (2 * O)); ++sub) {
                    uint32_t adj[K];
                    for (int h = 0; h < L; ++h) adj[h] = sadj[h];
                    adj[L] = adj[L + 1] = 0;
                    auto link = [&](int x, int y) { adj[x] |= 1u << y; adj[y] |= 1u << x; };
                    link(i, L);
                    if (form != FORM_END) link(i, L + 1);
                    if (form != FORM_CENTRE) link(L, L + 1);
                    for (int r = 0; r < O; ++r) {
                        const int h = cp[r + (r >= rv)];
                        if ((sub >> r) & 1u) link(h, L);
                        if ((sub >> (O + r)) & 1u) link(h, L + 1);
                    }
                    uint32_t lm = 0;
                    int jn = -1;
                    dissect3(K, gid, adj, lm, jn);
                    const bool ref = jn == i && lm == ((1u << i) | (1u << L) | (1u << (L + 1)));
                    const bool got = join_accepted<L>(cls, form, sa, sb, gid[L + 1] > gid[L], sub);
                    ++checked;
                    kept += ref;
                    bad += ref != got;
                }
            }
    }
}

int main() {
    run<2>(400);
    run<3>(400);
    run<4>(200);
    run<5>(100);
    printf("checked %ld kept %ld mismatches %ld\n", checked, kept, bad);
    return bad != 0 || kept == 0;
}
