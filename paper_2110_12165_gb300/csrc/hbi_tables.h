// Bounds checks of the HMVM work tables (the V^T batches and items, the UY tasks and their
// gather indices) against the buffers they index.  Host code without CUDA dependencies: the
// packer runs it on every operator it builds, and the CPU tests compile it into a host harness
// and feed it corrupted tables.  The bounds-checked build of the product kernels
// (HBI_BOUNDS_CHECK) checks the same conditions on the device, launch by launch.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

namespace hbi {

// Sizes the tables must stay inside (elements unless stated otherwise).
struct TableLimits {
    int64_t n_data1 = 0, n_data2 = 0, n_data3 = 0;   // V^T, U and dense streams
    int64_t n_x = 0;        // x entries (n_in N) at the head of [x | t]
    int64_t n_xt = 0;       // entries of [x | t] (without the 16 zero guard entries)
    int64_t n_y = 0;        // outputs (n_out N)
    int64_t n_gather = 0;   // gather indices
    int es_vt = 2, es_u = 2, es_d = 4, acc_bytes = 4;   // element sizes (bytes)
    int smem_uy = 0;        // dynamic shared memory of a UY CTA (bytes)
    int vt_panel_bytes = 0, vt_x_bytes = 0, vt_max_sub = 0, vt_split_rows = 0;
};

namespace tables_detail {
inline void note(int64_t &bad, std::string *first, const std::string &what) {
    if (bad++ == 0 && first) *first = what;
}
}  // namespace tables_detail

// The V^T stage batches (in CTA order) and their items: every bulk copy and shared-memory
// access of the V^T kernel inside its buffers.  Returns the number of violations; *first
// describes the first.
template <typename Batch, typename Item>
int64_t check_vt_tables(const std::vector<Batch> &batches, const std::vector<Item> &items, const TableLimits &L,
                        std::string *first) {
    using tables_detail::note;
    int64_t bad = 0;
    const int64_t vec = 16 / L.es_vt, za = 16 / L.acc_bytes;
    for (size_t bi = 0; bi < batches.size(); ++bi) {
        const Batch &b = batches[bi];
        const std::string where = "V^T batch " + std::to_string(bi) + ": ";
        if (b.nitems < 1 || b.nitems > L.vt_max_sub || b.item0 < 0 || (int64_t)b.item0 + b.nitems > (int64_t)items.size()) {
            note(bad, first, where + "item range");
            continue;
        }
        if (b.pbytes < 0 || b.pbytes > L.vt_panel_bytes || b.xbytes < 0 || b.xbytes > L.vt_x_bytes || b.pbytes % 16 ||
            b.xbytes % 16 || b.data_off < 0 || (b.data_off * L.es_vt) % 16 || b.data_off * L.es_vt + b.pbytes > L.n_data1 * L.es_vt)
            note(bad, first, where + "panel or x bytes");
        int64_t pacc = 0, xacc = 0;
        for (int k = 0; k < b.nitems; ++k) {
            const Item &it = items[b.item0 + k];
            const std::string wi = where + "item " + std::to_string(k) + ": ";
            const bool whole = (it.flags & 3) == 3;
            if (it.rows < 1 || it.cpad <= 0 || it.cpad % vec || it.lo < 0 || it.lo >= it.hi || it.hi > it.cpad)
                note(bad, first, wi + "shape");
            if (it.x_off < 0 || it.x_off % za || it.x_off + it.cpad > L.n_xt + 16) note(bad, first, wi + "x slice");
            if (it.out_off < L.n_x || it.out_off + it.rows > L.n_xt) note(bad, first, wi + "t rows");
            if (it.data_off != b.data_off + pacc || (int64_t)it.poff != pacc ||
                (int64_t)it.zoff * L.acc_bytes != xacc)
                note(bad, first, wi + "offsets inside the batch");
            if (!whole && it.rows > L.vt_split_rows) note(bad, first, wi + "rows of a split row block");
            pacc += (int64_t)it.rows * it.cpad;
            xacc += (int64_t)it.cpad * L.acc_bytes;
        }
        if (pacc * L.es_vt != b.pbytes || xacc != b.xbytes) note(bad, first, where + "bytes of its items");
    }
    return bad;
}

// The UY tasks and their gather indices: stream segments, gather range, output rows and
// shared memory; a gather index is -1 (padding), an entry of [x | t], or -2 - t for the pair
// t, t + 1 of an FP32-accurate leading factor column.
template <typename Task>
int64_t check_uy_tables(const std::vector<Task> &tasks, const std::vector<int> &gidx, const TableLimits &L,
                        std::string *first) {
    using tables_detail::note;
    int64_t bad = 0;
    for (size_t ti = 0; ti < tasks.size(); ++ti) {
        const Task &t = tasks[ti];
        const std::string where = "UY task " + std::to_string(ti) + ": ";
        if (t.rows < 1 || t.cpad < 0 || t.cpad_d < 0 || t.cpad % (16 / L.es_u) || t.cpad_d % (16 / L.es_d)) {
            note(bad, first, where + "shape");
            continue;
        }
        if (t.data_off < 0 || t.data_off + (int64_t)t.rows * t.cpad > L.n_data2) note(bad, first, where + "U segment");
        if (t.data_off_d < 0 || t.data_off_d + (int64_t)t.rows * t.cpad_d > L.n_data3) note(bad, first, where + "dense segment");
        if (t.out_off < 0 || t.out_off + t.rows > L.n_y) note(bad, first, where + "output rows");
        if ((int64_t)(t.cpad + t.cpad_d) * L.acc_bytes > L.smem_uy) note(bad, first, where + "gathered input size");
        const int64_t c = (int64_t)t.cpad + t.cpad_d;
        if (t.gather_off < 0 || t.gather_off + c > L.n_gather || t.gather_off + c > (int64_t)gidx.size()) {
            note(bad, first, where + "gather range");
            continue;
        }
        for (int64_t j = 0; j < c; ++j) {
            const int64_t g = gidx[t.gather_off + j];
            const bool ok = g == -1 || (g >= 0 && g < L.n_xt) || (g <= -2 && -2 - g >= 0 && -2 - g + 1 < L.n_xt);
            if (!ok) note(bad, first, where + "gather index " + std::to_string(g) + " at " + std::to_string(j));
        }
    }
    return bad;
}

// The UY tasks of leaf row units given by decreasing work: each unit cut by rows into pieces of
// whole elements (nout rows each), which share the unit's gather list.  A piece holds at most the
// work left (its own unit's included) / (2 x CTA slots), as in guided self-scheduling: with one unit
// per task the 475 units of a 20,022-element fault leave most of 760 slots idle in one uneven
// wave (UY phase 68 us uncut, 59 us cut on a GB300; 243 units in FP64 190 against 126 us; 124
// units 33.5 against 16.5 us), and at 160,000 elements the small last pieces even out the CTAs'
// ends (475 against 471 us).  A piece gathers its whole input again, so it keeps 24 rows (12
// rows: 63 us at 20,022 elements) and 112 KB (units of 134 KB cut in two: 46.0 against 44.5 us),
// unless the pieces would then not fill the slots once: down to 8 rows (2,048 elements with one
// output each: 12.8 against 16.9 us).
template <typename Task>
std::vector<Task> cut_uy_units(const std::vector<Task> &units, int nout, int es_u, int es_d, int sms, int ctas_per_sm) {
    auto work = [&](const Task &t) { return (int64_t)t.rows * ((int64_t)t.cpad * es_u + (int64_t)t.cpad_d * es_d); };
    int64_t left = 0, rows = 0;
    for (const Task &t : units) {
        left += work(t);
        rows += t.rows;
    }
    const int64_t slots = std::max<int64_t>(1, (int64_t)sms * ctas_per_sm);
    const int64_t min_rows = std::min<int64_t>(24, std::max<int64_t>(8, (rows + slots - 1) / slots));
    const int64_t min_elems = (min_rows + nout - 1) / nout, min_work = std::min<int64_t>(112 << 10, left / slots);
    const int64_t whole = nout % 2 ? 4 : 2;   // elements of whole 4-row blocks: only a unit's last piece ends in a partial one
    std::vector<Task> cut;
    for (const Task &t : units) {
        const int64_t w = work(t), ne = t.rows / nout, target = std::max<int64_t>(1, left / (2 * slots));
        const int64_t most = std::min(ne / min_elems, w / std::max<int64_t>(1, min_work));
        const int64_t np = std::max<int64_t>(1, std::min((w + target - 1) / target, most));
        for (int64_t q = 0; q < np; ++q) {
            const int64_t r0 = ne * q / np / whole * whole * nout;
            const int64_t r1 = q + 1 < np ? ne * (q + 1) / np / whole * whole * nout : t.rows;
            if (r0 == r1) continue;
            Task c = t;
            c.rows = (int)(r1 - r0);
            c.out_off += r0;
            c.data_off += r0 * t.cpad;
            c.data_off_d += r0 * t.cpad_d;
            cut.push_back(c);
        }
        left -= w;
    }
    return cut;
}

// The pieces that the UY kernel is given against the units that check_uy_tables has passed: in output
// order they tile the units' rows, in whole elements, each with its unit's gather list and columns
// and the stream offsets of its first row, so that every access of a piece is one of its unit's.
template <typename Task>
int64_t check_uy_pieces(std::vector<Task> units, std::vector<Task> pieces, int nout, std::string *first) {
    using tables_detail::note;
    auto by_row = [](const Task &a, const Task &b) { return a.out_off < b.out_off; };
    std::sort(units.begin(), units.end(), by_row);
    std::sort(pieces.begin(), pieces.end(), by_row);
    int64_t bad = 0;
    size_t pi = 0;
    for (const Task &t : units) {
        int64_t row = 0;
        for (; row < t.rows && pi < pieces.size(); ++pi) {
            const Task &c = pieces[pi];
            const std::string where = "UY piece at output " + std::to_string(c.out_off) + ": ";
            if (c.out_off != t.out_off + row || c.rows < 1 || c.rows > t.rows - row || c.rows % nout) {
                note(bad, first, where + "rows");
                return bad;
            }
            if (c.data_off != t.data_off + row * t.cpad || c.data_off_d != t.data_off_d + row * t.cpad_d)
                note(bad, first, where + "stream offsets");
            if (c.cpad != t.cpad || c.cpad_d != t.cpad_d || c.gather_off != t.gather_off || c.model != t.model)
                note(bad, first, where + "columns");
            row += c.rows;
        }
        if (row < t.rows) note(bad, first, "UY unit at output " + std::to_string(t.out_off) + ": rows without a piece");
    }
    if (pi < pieces.size()) note(bad, first, "UY pieces of no unit");
    return bad;
}

}  // namespace hbi
