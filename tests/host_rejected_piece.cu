// Host harness: which elements' stage the UY launch may run for a piece (csrc/hbi_internal.h,
// piece_elems).  Prints "<rows> <out_off> <nout> <ok> <first element> <elements>" per record.
#include <cstdio>

#include "../paper_2110_12165_gb300/csrc/hbi_internal.h"

using namespace hbi;

int main() {
    const int64_t recs[][3] = {{48, 96, 3}, {64, 0, 1}, {6, 30, 2}, {48, 1 << 30, 3}, {1 << 30, 96, 1}, {0, -3, 3}};
    for (auto &r : recs)
        for (int ok = 0; ok < 2; ++ok) {
            GemvTask t{};
            t.rows = (int)r[0];
            t.out_off = r[1];
            const PieceElems p = piece_elems(t, (int)r[2], ok != 0);
            printf("%d %lld %d %d %d %d\n", t.rows, (long long)t.out_off, (int)r[2], ok, p.e0, p.ne);
        }
    return 0;
}
