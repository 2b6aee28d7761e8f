// Host checks of the join kernel's rules.  Built and run by tests/test_join_host.py; host code only.
#include "fsm_join.cuh"
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

int main() {
    const long b = bounds();
    printf("bounds %ld\n", b);
    return b != 0;
}
