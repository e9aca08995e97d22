// Host harness of the UY piece cutter (csrc/hbi_tables.h): for units of many shapes the pieces
// of each unit must tile its rows exactly, in whole elements, with its own gather list and the
// stream offsets of their first row.  Prints "violations <n>" and "pieces <n> units <n>".
#include <cstdio>
#include <map>

#include "../paper_2110_12165_gb300/csrc/hbi_internal.h"

using namespace hbi;

int main() {
    long long bad = 0, npieces = 0, nunits = 0;
    for (int nout = 1; nout <= 3; ++nout)
        for (int count : {1, 2, 7, 64, 475, 3803})
            for (int ne : {1, 2, 7, 8, 20, 47, 64}) {
                std::vector<GemvTask> units;
                int64_t d2 = 0, d3 = 0, out = 0;
                for (int u = 0; u < count; ++u) {
                    GemvTask t{};
                    const int e = std::max(1, ne - u % 3);
                    t.rows = nout * e; t.cpad = 8 * (3 + u % 5); t.cpad_d = 4 * (u % 4);
                    t.data_off = d2; t.data_off_d = d3; t.out_off = out; t.gather_off = 1000 * u; t.model = u % 2;
                    d2 += (int64_t)t.rows * t.cpad; d3 += (int64_t)t.rows * t.cpad_d; out += t.rows;
                    units.push_back(t);
                }
                std::map<int64_t, std::vector<GemvTask>> of;   // pieces by gather list
                for (const GemvTask &c : cut_uy_units(units, nout, 2, 4, 152, 5)) of[c.gather_off].push_back(c);
                for (const GemvTask &t : units) {
                    int64_t row = 0;
                    for (const GemvTask &c : of[t.gather_off]) {
                        const bool ok = c.rows > 0 && c.rows % nout == 0 && c.out_off == t.out_off + row &&
                                        c.data_off == t.data_off + row * t.cpad &&
                                        c.data_off_d == t.data_off_d + row * t.cpad_d && c.cpad == t.cpad &&
                                        c.cpad_d == t.cpad_d && c.model == t.model;
                        bad += !ok;
                        row += c.rows;
                        ++npieces;
                    }
                    bad += row != t.rows;
                    ++nunits;
                }
            }
    printf("violations %lld\npieces %lld units %lld\n", bad, npieces, nunits);
    return 0;
}
