// Host checks of the join kernel's rules.  Built and run by tests/test_join_host.py; host code only.
#include "fsm_join_tables.cuh"
#include <cstdio>
#include <vector>
using namespace fsm;

// Every index of the lists of a small graph against every row: only the entries of the row's own list may
// be read, not those of another vertex's.
static long bounds() {
    const std::vector<int> row = {0, 3, 3, 4, 9, 11};
    const int n = (int)row.size() - 1;
    long bad = 0, foreign = 0;
    for (int v = 0; v < n; ++v)
        for (int a = 0; a < n; ++a)
            for (int centre = 0; centre < 2; ++centre)
                for (int at = -2; at < row[n] + 2; ++at) {
                    const int own = centre ? v : a;
                    const bool want = at >= row[own] && at < row[own + 1];
                    bad += partner_in_list(centre != 0, at, row[v], row[v + 1] - row[v], row[a], row[a + 1] - row[a]) != want;
                    foreign += !want && at >= 0 && at < row[n];
                }
    return bad + (foreign == 0);
}

// The tables as the device fills them (acc5 from the graphs dissected once) against join_accepted: every
// step-th word of `acc`, and `any` of every cstep-th class against all subsets and forms.
template <int L> static void tables(int64_t step, int cstep, long &acc_bad, long &any_bad, long &kept) {
    using G = JoinGeo<L>;
    std::vector<uint32_t> acc((size_t)G::ACC_WORDS);
    if constexpr (L == 5) {
        std::vector<uint16_t> code(1 << 21);
        for (int c = 0; c < 1 << 21; ++c) code[c] = dissect7_code(c);
        for (int64_t x = 0; x < G::ACC_WORDS; ++x) acc[x] = acc5_word(code.data(), x);
    } else {
        for (int64_t x = 0; x < G::ACC_WORDS; ++x) acc[x] = acc_word<L>(x);
    }
    for (int64_t x = 0; x < G::ACC_WORDS; x += step) {
        // the word's place, counted up as JoinGeo lays the rows out
        const int64_t row = x / G::W;
        const int cls = (int)(row / G::ROWS), in = (int)(row % G::ROWS);
        const int form = in / (2 * G::SL * G::SL), sa = in / (2 * G::SL) % G::SL, sb = in / 2 % G::SL;
        for (int s = 0; s < 32 && s < G::SUBS; ++s) {
            const bool want = join_accepted<L>(cls, form, sa, sb, in & 1, (uint32_t)(x % G::W) * 32 + s);
            kept += want;
            acc_bad += want != ((acc[x] >> s) & 1u);
        }
    }
    for (int cls = 0; cls < G::CLS; cls += cstep)
        for (int s = 0; s < G::SL; ++s) {
            uint32_t want[4] = {0, 0, 0, 0};
            for (int p = 0; p < G::SL; ++p)
                for (uint32_t sub = 0; sub < (uint32_t)G::SUBS; ++sub) {
                    if (join_accepted<L>(cls, FORM_CENTRE, p, s, 1, sub)) want[ANY_C] |= 1u << p, want[ANY_CT] |= 1u << p;
                    if (join_accepted<L>(cls, FORM_TRI, p, s, 1, sub)) want[ANY_CT] |= 1u << p;
                    for (int bgt = 0; bgt < 2; ++bgt)
                        if (join_accepted<L>(cls, FORM_END, s, p, bgt, sub))
                            want[ANY_E] |= 1u << (p + bgt * G::SL), want[ANY_ET] |= 1u << (p + bgt * G::SL);
                    if (join_accepted<L>(cls, FORM_TRI, s, p, 1, sub)) want[ANY_ET] |= 1u << (p + G::SL);
                }
            for (int kind = 0; kind < 4; ++kind)
                any_bad += want[kind] != any_entry<L>(acc.data(), ((int64_t)cls * 4 + kind) * G::SL + s);
        }
}

int main() {
    printf("bounds %ld\n", bounds());
    long acc_bad = 0, any_bad = 0, kept = 0;
    tables<1>(1, 1, acc_bad, any_bad, kept);
    tables<2>(1, 1, acc_bad, any_bad, kept);
    tables<3>(1, 1, acc_bad, any_bad, kept);
    tables<4>(7, 5, acc_bad, any_bad, kept);
    tables<5>(499, 211, acc_bad, any_bad, kept);
    printf("acc %ld\nany %ld\nkept %ld\n", acc_bad, any_bad, kept);
    return 0;
}
