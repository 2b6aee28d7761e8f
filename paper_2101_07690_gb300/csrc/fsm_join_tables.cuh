// fsm_join_tables.cuh -- the entries of the join kernel's acceptance tables (JoinGeo, fsm_join.cuh), one at a
// time: fsm_join_tables.cu fills the tables on the device with these, tests/join_host_check.cu compares them
// on the host with join_accepted.
#pragma once
#include "fsm_join.cuh"

namespace fsm {

// entry x of `acc`: a word of 32 subsets of a row, by dissecting each
template <int L> FSM_HD uint32_t acc_word(int64_t x) {
    using G = JoinGeo<L>;
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
    return m;
}

// Seven vertices (l = 5) have 283M combinations but only 2^21 graphs on ordered ids: each graph is dissected
// once (part mask | join vertex << 7, 0 if disconnected), then they are looked up.  Bit of pair (x, y),
// x < y: y (y - 1) / 2 + x.
FSM_HD uint16_t dissect7_code(int c) {
    const int32_t gid[7] = {0, 1, 2, 3, 4, 5, 6};
    uint32_t adj[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int y = 1; y < 7; ++y)
        for (int x = 0; x < y; ++x)
            if ((c >> (y * (y - 1) / 2 + x)) & 1) { adj[x] |= 1u << y; adj[y] |= 1u << x; }
    if (!mask_connected(127u, adj, 7)) return 0;
    uint32_t lm = 0;
    int jn = -1;
    dissect3(7, gid, adj, lm, jn);
    return (uint16_t)(lm | ((uint32_t)jn << 7));
}
FSM_HD uint32_t pair_bit(int x, int y) {
    const int a = x < y ? x : y, b = x < y ? y : x;
    return 1u << (b * (b - 1) / 2 + a);
}
// entry i of `acc` for l = 5
FSM_HD uint32_t acc5_word(const uint16_t *code, int64_t i) {
    constexpr int L = 5;
    using G = JoinGeo<L>;
    const int wd = (int)(i % G::W);
    int64_t y = i / G::W;
    const int bgt = (int)(y & 1);
    y >>= 1;
    const int sb = (int)(y % G::SL);
    y /= G::SL;
    const int sa = (int)(y % G::SL);
    y /= G::SL;
    const int form = (int)(y % 3), cls = (int)(y / 3), rv = cls >> G::EB;
    if (!((sa == sb || (sb > sa) == (bgt != 0)) && (form == FORM_END || bgt))) return 0;   // no such order
    uint32_t sadj[5] = {0, 0, 0, 0, 0};
    int bit = 0;
    for (int t = 0; t < L; ++t)
        for (int u = t + 1; u < L; ++u, ++bit)
            if ((cls >> bit) & 1) { sadj[t] |= 1u << u; sadj[u] |= 1u << t; }
    if (!mask_connected(31u, sadj, L)) return 0;
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
    uint32_t m = 0;
    for (int s = 0; s < 32; ++s) {
        uint32_t c = base;
        for (int q = 0; q < 5; ++q)
            if ((s >> q) & 1) c |= cb[q];
        if (code[c] == want) m |= 1u << s;
    }
    return m;
}

// entry x of `any` (class, ANY_*, anchor slot): partner slots that some subset and form accept
template <int L> FSM_HD uint16_t any_entry(const uint32_t *acc, int64_t x) {
    using G = JoinGeo<L>;
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
    return (uint16_t)m;
}

} // namespace fsm
