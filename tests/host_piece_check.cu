// Host harness of the check of the UY pieces against their units (csrc/hbi_tables.h): the cutter's pieces
// of ragged units, one of them without columns, must pass in any order; each corruption listed below,
// applied alone, must be reported.  Prints one line per case: "<name> <violations>".
#include <cstdio>
#include <functional>

#include "../paper_2110_12165_gb300/csrc/hbi_internal.h"

using namespace hbi;

int main() {
    using Pieces = std::vector<GemvTask>;
    const int nout = 3;
    std::vector<GemvTask> units;
    int64_t d2 = 0, d3 = 0, out = 0, g = 0;
    for (int u = 0; u < 6; ++u) {
        GemvTask t{};
        t.rows = nout * (40 - 3 * u); t.cpad = u == 4 ? 0 : 8 * (3 + u); t.cpad_d = u == 4 ? 0 : 4 * (1 + u);
        t.data_off = d2; t.data_off_d = d3; t.out_off = out; t.gather_off = g; t.model = u / 3;
        d2 += (int64_t)t.rows * t.cpad; d3 += (int64_t)t.rows * t.cpad_d; out += t.rows; g += t.cpad + t.cpad_d;
        units.push_back(t);
    }
    const Pieces cut = cut_uy_units(units, nout, 2, 4, 4, 5);
    std::vector<std::pair<const char *, std::function<void(Pieces &)>>> cases = {
        {"valid", [](Pieces &) {}},
        {"valid_reversed", [](Pieces &p) { std::reverse(p.begin(), p.end()); }},
        {"missing", [](Pieces &p) { p.erase(p.begin() + 1); }},
        {"missing_last", [](Pieces &p) { p.pop_back(); }},
        {"twice", [](Pieces &p) { p.push_back(p[1]); }},
        {"past_the_end", [](Pieces &p) { GemvTask t = p.back(); t.out_off += t.rows; p.push_back(t); }},
        {"rows_past_unit", [](Pieces &p) { p[p.size() - 1].rows += 3; }},
        {"rows_overlap", [](Pieces &p) { p[0].rows += 3; }},
        {"rows_part_of_element", [](Pieces &p) { p[0].rows -= 1; }},
        {"out_off", [](Pieces &p) { p[1].out_off += 3; }},
        {"u_offset", [](Pieces &p) { p[1].data_off += 8; }},
        {"dense_offset", [](Pieces &p) { p[1].data_off_d -= 4; }},
        {"cpad", [](Pieces &p) { p[1].cpad += 8; }},
        {"cpad_d", [](Pieces &p) { p[1].cpad_d += 4; }},
        {"gather", [](Pieces &p) { p[1].gather_off += 1; }},
        {"model", [](Pieces &p) { p[1].model += 1; }},
    };
    for (auto &c : cases) {
        Pieces p = cut;
        c.second(p);
        std::string first;
        printf("%s %lld\n", c.first, (long long)check_uy_pieces(units, p, nout, &first));
    }
    printf("pieces %zu\nunits %zu\n", cut.size(), units.size());
    return 0;
}
