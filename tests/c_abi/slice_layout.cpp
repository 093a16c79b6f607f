// The column slices' row layout of one system, as the first of a handle and
// behind more than 2^27 blocks of other systems (a batch): the same offsets of
// its coefficients, counted from the system's own first block, within it.
#include "../../paper_1002_1202_gb300/csrc/tb_internal.h"

#include <algorithm>
#include <cstdio>

int main() {
    // a ring of 12 sp atoms and 8 s atoms, each with its two neighbours
    const int n = 20;
    std::vector<int32_t> orb(n, 4), bcol;
    for (int i = 12; i < n; ++i) orb[i] = 1;
    std::vector<int64_t> brow(n + 1, 0);
    for (int i = 0; i < n; ++i) {
        int nb[3] = {(i + n - 1) % n, i, (i + 1) % n};
        std::sort(nb, nb + 3);
        bcol.insert(bcol.end(), nb, nb + 3);
        brow[i + 1] = (int64_t)bcol.size();
    }
    const int64_t first = ((int64_t)1 << 27) + 5;
    std::vector<int64_t> moved(brow);
    for (int64_t& b : moved) b += first;
    tb::SliceHost a, b;
    for (int cl : {1, 2, 3}) {
        tb::slice_layout(n, orb.data(), brow.data(), bcol.data(), 0, cl, a);
        tb::slice_layout(n, orb.data(), moved.data(), bcol.data() - first, 0, cl, b);
        int used = 0;
        for (int s : a.src) {
            if (s < -1 || s >= 16 * (int)bcol.size()) return std::printf("offset %d outside the system\n", s), 1;
            used += s >= 0;
        }
        // every stored entry once: 4 x 4, 4 x 1, 1 x 4 and 1 x 1 blocks
        int want = 0;
        for (int i = 0; i < n; ++i)
            for (int64_t k = brow[i]; k < brow[i + 1]; ++k) want += orb[i] * orb[bcol[k]];
        if (used != want) return std::printf("%d coefficients, %d entries\n", used, want), 1;
        if (a.src != b.src || a.idx != b.idx || a.dest != b.dest) return std::printf("moved layout differs\n"), 1;
    }
    std::puts("ok");
    return 0;
}
