// Host check of the static plan's bands (panels walked together): the plan
// that a handle keeps is one whose launch was found to fit.  Compiled with g++
// against the planner source by tests/test_planner_bands.py; prints "OK" or the
// first violation.
#include <cstdio>
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

int main()
{
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
