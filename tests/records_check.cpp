// Host check of the recorded steps of a quadratic run (rikfad_records.hpp):
// the step loop of rikfad_quadratic.cu, with the steps left out, over every
// list of up to four entries from a set with values out of range on both
// sides, 32-bit wrap-arounds among them, in any order.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "rikfad_records.hpp"

using namespace rikfad;

// The recorded entries of steps k0 .. k0 + steps as (entry, step) pairs, or
// false if the loop has not reached its last step after more turns than any list
// can need.
static bool run(const std::vector<int64_t> &rec, int64_t k0, int steps, std::vector<std::pair<int64_t, int>> &got)
{
    const int64_t n = (int64_t)rec.size();
    int64_t ri = n > 0 ? first_record_at_or_after(rec.data(), n, k0) : 0;
    int next = record_in_launch(rec.data(), n, ri, k0, 0, steps);
    int turns = 0;
    for (int s = 0;;) {
        if (++turns > steps + n + 4)
            return false;
        const int stop = next >= 0 ? next : steps;
        for (; s < stop; ++s)
            if (s >= steps)
                return false;
        while (s == next) {
            got.push_back({ri, s});
            ++ri;
            next = record_in_launch(rec.data(), n, ri, k0, s, steps);
        }
        if (s == steps)
            return true;
    }
}

int main()
{
    const int64_t k0 = 128;
    const int steps = 6;
    const std::vector<int64_t> values = {-((int64_t)1 << 32) + k0 + 4, -5,      k0 - 1, k0,
                                         k0 + 2, k0 + 3, k0 + 5, k0 + steps, k0 + steps + 1,
                                         ((int64_t)1 << 32) + k0 + 5};
    const int nv = (int)values.size();
    int64_t lists = 0;
    for (int len = 0; len <= 4; ++len) {
        int total = 1;
        for (int i = 0; i < len; ++i)
            total *= nv;
        for (int code = 0; code < total; ++code, ++lists) {
            std::vector<int64_t> rec;
            bool ascending = true;
            for (int i = 0, c = code; i < len; ++i, c /= nv) {
                rec.push_back(values[c % nv]);
                ascending &= i == 0 || rec[i] >= rec[i - 1];
            }
            std::vector<std::pair<int64_t, int>> got;
            bool ok = run(rec, k0, steps, got);
            size_t want = 0;        // ascending: every entry in range, in order
            for (size_t i = 0; i < got.size(); ++i)
                ok &= rec[got[i].first] == k0 + got[i].second && (i == 0 || got[i].first > got[i - 1].first);
            for (int64_t r : rec)
                want += r >= k0 && r <= k0 + steps;
            ok &= !ascending || got.size() == want;
            if (!ok) {
                std::printf("list of %d entries (code %d) does not end, or records a wrong step\n", len, code);
                return 1;
            }
        }
    }
    std::printf("%lld lists OK\n", (long long)lists);
    return 0;
}
