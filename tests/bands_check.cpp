// Host check of the static plan: every row of every panel and every element of
// every vector lies in exactly one piece, and in exactly one tile; a band's
// (panels walked together) pieces lie side by side in one block, of the same
// rows, to the matrix's last panel; a panel's partials are evenly spaced, inside
// the buffer, and overlap no other's.  And the plan that a handle keeps is one
// whose launch was found to fit.  Compiled with g++ against the planner source by
// tests/test_planner_bands.py; prints "OK" or the first violation.
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>

#include "rikfad_planner.hpp"

using namespace rikfad;

static int fail(const char *what, long long a, long long b)
{
    std::printf("FAIL %s (%lld, %lld)\n", what, a, b);
    return 1;
}

// Blocks that a fake device of 152 units runs at once: `few` a unit with a band
// wider than `limit`, 2 otherwise.
static int check_resident(const std::vector<rikfad_shape> &shapes, int limit, int few, bool more_needed)
{
    int max_blocks = 304, asked = 0;
    int asked_width = -1, answered = 0;
    Plan p;
    const std::string err = build_resident_plan(
        shapes.data(), (int)shapes.size(), 2, max_blocks, p, false, [&](const Plan &plan) {
            ++asked;
            asked_width = plan.band_width;
            answered = 152 * (plan.band_width > limit ? few : 2);
            return answered;
        });
    if (few == 0 && more_needed)
        return err.empty() ? fail("a plan that cannot run", p.band_width, limit) : 0;
    if (!err.empty()) {
        std::printf("FAIL %s\n", err.c_str());
        return 1;
    }
    if (p.band_width != 0 && (p.band_width != asked_width || p.nblocks > answered || max_blocks > answered))
        return fail("a plan whose launch was not found to fit", p.band_width, answered);
    if ((asked > 1) != more_needed)
        return fail("plans asked about", asked, more_needed);
    return 0;
}

static int check_plan(const std::vector<rikfad_shape> &shapes, int grad_bytes, int max_blocks, bool full, int &bands)
{
    Plan p;
    std::string err = build_plan(shapes.data(), (int)shapes.size(), grad_bytes, max_blocks, p, full);
    if (err.empty())
        err = build_tiles(p);
    if (!err.empty()) {
        std::printf("FAIL %s\n", err.c_str());
        return 1;
    }
    if (p.nblocks > max_blocks)
        return fail("blocks", p.nblocks, max_blocks);
    // Pieces, block by block: every panel and vector is walked from its first row
    // (element) to its last.
    std::vector<int64_t> panel_at(p.panels.size(), 0), vector_at(shapes.size(), 0);
    std::vector<int> slots(p.panels.size(), 0), slot_owner(p.slot_off.size(), -1);
    int widest = 0;
    for (int b = 0; b < p.nblocks; ++b) {
        const int q1 = p.block_piece[b + 1];
        for (int q = p.block_piece[b]; q < q1; ++q) {
            const PieceDev &pc = p.pieces[q];
            const TensorDev &td = p.tensors[pc.tensor];
            if (pc.begin < 0 || pc.begin >= pc.end || pc.end > td.rows)
                return fail("piece range", pc.begin, pc.end);
            if (pc.kind == kElements) {
                if (vector_at[pc.tensor] != pc.begin)
                    return fail("elements skipped or repeated", pc.begin, vector_at[pc.tensor]);
                vector_at[pc.tensor] = pc.end;
                continue;
            }
            if (pc.panel < td.panel0 || pc.panel >= td.panel0 + td.npanels)
                return fail("piece panel", pc.panel, td.panel0);
            if (panel_at[pc.panel] != pc.begin)
                return fail("rows skipped or repeated", pc.begin, panel_at[pc.panel]);
            panel_at[pc.panel] = pc.end;
            const PanelDev &pd = p.panels[pc.panel];
            if (slot_owner[pc.slot] != -1 || p.slot_off[pc.slot] != pc.colpart_off)
                return fail("slot", pc.slot, pc.colpart_off);
            slot_owner[pc.slot] = pc.panel;
            if (pc.slot != pd.slot_begin + slots[pc.panel] * pd.slot_step ||
                pc.colpart_off != p.slot_off[pd.slot_begin] + (int64_t)slots[pc.panel] * pd.slot_stride)
                return fail("partials of a panel not evenly spaced", pc.slot, pd.slot_begin);
            ++slots[pc.panel];
            if (pc.band == 0) {
                if (q == p.block_piece[b])
                    return fail("a band that leaves its block", q, b);
                const PieceDev &before = p.pieces[q - 1];
                if (before.kind != kMatrixRows || before.panel != pc.panel - 1 || before.begin != pc.begin ||
                    before.end != pc.end || before.tensor != pc.tensor ||
                    pc.colpart_off != before.colpart_off + p.panels[before.panel].width)
                    return fail("a band's piece without its predecessor", q, pc.panel);
            } else if (pc.band > 1) {
                ++bands;
                if (!td.vec || full || q + pc.band > q1 || pc.panel + pc.band != td.panel0 + td.npanels)
                    return fail("a band not of a matrix's last panels", q, pc.band);
                for (int k = 1; k < pc.band; ++k)
                    if (p.pieces[q + k].band != 0)
                        return fail("a band's pieces", q + k, p.pieces[q + k].band);
                if (pd.slot_step != pc.band || pd.slot_stride != td.cols - pd.col0 || pd.slot_stride > kBandMax)
                    return fail("a band's columns", pd.slot_stride, pc.band);
                widest = std::max(widest, (int)pd.slot_stride);
            }
        }
    }
    if (widest != p.band_width)
        return fail("widest band", widest, p.band_width);
    std::vector<std::pair<int64_t, int64_t>> parts;
    for (size_t s = 0; s < p.slot_off.size(); ++s) {
        if (slot_owner[s] < 0)
            return fail("a slot without a piece", (long long)s, 0);
        parts.push_back({p.slot_off[s], p.slot_off[s] + p.panels[slot_owner[s]].width});
    }
    std::sort(parts.begin(), parts.end());
    for (size_t s = 0; s < parts.size(); ++s)
        if (parts[s].first < (s ? parts[s - 1].second : 0) || parts[s].second > p.colpart_floats)
            return fail("partials overlap", parts[s].first, parts[s].second);
    // Tiles: tile i of a tensor is panel i % npanels of row group i / npanels.
    std::vector<std::vector<int64_t>> tiles(shapes.size());
    for (const TileGroupDev &g : p.tile_groups)
        for (int64_t i = g.first; i < g.first + kTileGroup; ++i)
            tiles[g.tensor].push_back(i);
    for (size_t t = 0; t < shapes.size(); ++t) {
        const TensorDev &td = p.tensors[t];
        for (size_t i = 0; i < tiles[t].size(); ++i)
            if (tiles[t][i] != (int64_t)i)
                return fail("tiles skipped or repeated", (long long)t, tiles[t][i]);
        const int64_t np = std::max(td.npanels, 1);
        if (td.rows > 0 && ((int64_t)tiles[t].size() / np * td.tile_rows < td.rows || td.tile_rows < 1))
            return fail("rows without a tile", (long long)t, td.tile_rows);
        if (td.rows > 0 && td.cols == 0 ? vector_at[t] != td.rows : false)
            return fail("elements without a piece", (long long)t, vector_at[t]);
        for (int k = 0; k < td.npanels; ++k) {
            const PanelDev &pd = p.panels[td.panel0 + k];
            if (panel_at[td.panel0 + k] != td.rows || slots[td.panel0 + k] != pd.nslots)
                return fail("rows without a piece", panel_at[td.panel0 + k], td.rows);
            const int64_t next = k + 1 < td.npanels ? p.panels[td.panel0 + k + 1].col0 : td.cols;
            if (pd.col0 + (int64_t)pd.width != next || pd.width > kPanelMax || (k == 0 && pd.col0 != 0))
                return fail("panel columns", pd.col0, pd.width);
        }
    }
    return 0;
}

int main()
{
    // Plans: the widths that bands are made for, alone and in lists, and random lists.
    int bands = 0;
    std::vector<std::vector<rikfad_shape>> lists = {
        {{5000, 1800}, {2500, 1048}, {2000, 1928}, {1500, 2600}, {300, 768}, {77, 40}, {1000, 0}},
        {{40000, 1032}}, {{16000, 2056}, {0, 16}, {5, 0}}, {{9, 1800}}, {{4096, 9000}, {3, 7}}, {}};
    for (int w = 513; w <= 640; ++w)        // a last panel that splits off a tail, and those around it
        lists.push_back({{20000, w}, {20000, 1024 + w}});
    std::mt19937 rng(7);
    auto upto = [&](int n) { return (int)(rng() % (unsigned)n); };
    for (int i = 0; i < 1500; ++i) {
        std::vector<rikfad_shape> l;
        for (int t = 1 + upto(5); t > 0; --t) {
            const int cols = upto(6) == 0 ? 0 : upto(3) ? 8 * (1 + upto(640)) : 1 + upto(5000);
            l.push_back({upto(12) == 0 ? 0 : 1 + upto(upto(2) ? 300 : 9000), cols});
        }
        lists.push_back(l);
    }
    for (const auto &l : lists)
        for (const int grad_bytes : {2, 4})
            for (const int blocks : {304, 152, 7})
                for (const bool full : {false, true})
                    if (check_plan(l, grad_bytes, blocks, full, bands)) {
                        std::printf("%zu tensors, %d blocks; first %lld x %lld\n", l.size(), blocks,
                                    l.empty() ? 0LL : (long long)l[0].rows, l.empty() ? 0LL : (long long)l[0].cols);
                        return 1;
                    }
    if (bands < 10000)
        return fail("too few bands among the plans", bands, 10000);
    // At 304 blocks the widest band is 1800 columns, at 152 it is 1928: a launch
    // sized for the first plan is too small for the second.
    const std::vector<rikfad_shape> two = {{3200, 1800}, {3200, 1928}};
    Plan a, b;
    if (!build_plan(two.data(), 2, 2, 304, a).empty() || !build_plan(two.data(), 2, 2, 152, b).empty())
        return fail("build_plan", 0, 0);
    if (!(b.band_width > a.band_width && a.band_width > 0))
        return fail("the list no longer has wider bands for fewer blocks", a.band_width, b.band_width);
    if (check_resident(two, 4096, 1, false) || check_resident(two, 1500, 1, true) || check_resident(two, 1900, 1, false) ||
        check_resident(two, 1500, 0, true) || check_resident({{300, 768}, {40, 0}}, 0, 0, false))
        return 1;
    std::printf("OK\n");
    return 0;
}
