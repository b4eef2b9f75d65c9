// Host check of the gram tables (compiled and run by test_gram_lists.py): a
// bucket holds little more than the patterns that share its gram, also for
// alphabets of fewer than four letters.
#include <algorithm>
#include <cstdio>
#include <random>

#include "pm_internal.h"

using namespace pm;

int main()
{
    std::mt19937 rng(9);
    int bad = 0;
    for (const char *letters : {"AC", "AG", "ACG", "ACGT"})
        for (int lo : {6, 8, 10, 12})
            for (int d : {100, 1000, 3000}) {
                const size_t nl = letters[2] ? letters[3] ? 4 : 3 : 2;
                std::vector<uint8_t> P;
                std::vector<int64_t> off{0};
                for (int r = 0; r < d; ++r) {
                    const int len = lo + int(rng() % 13u);
                    for (int j = 0; j < len; ++j) P.push_back(uint8_t(letters[rng() % nl]));
                    off.push_back(int64_t(P.size()));
                }
                GramTables t;
                if (build_gram(P.data(), off.data(), d, 0, PM_ALGO_WMV, 2, t) || !t.ok) return 2;
                // entries of a gram, by the characters they have of it
                double mean = 0.0, of = 1.0;
                for (int j = 0; j < t.q && j < lo; ++j) of *= double(nl);
                mean = double(d) * t.s / of;
                uint32_t longest = 0;
                for (size_t b = 0; 2 * b + 2 < t.dir.size(); ++b)
                    longest = std::max(longest, (t.dir[2 * b + 2] & 0xFFFFFFu) - (t.dir[2 * b] & 0xFFFFFFu));
                if (longest > 12.0 + 3.0 * mean) {
                    std::printf("%s, %d patterns from %d letters: s %d q %d, longest %u, mean %.1f\n", letters, d, lo,
                                t.s, t.q, longest, mean);
                    ++bad;
                }
            }
    return bad ? 1 : 0;
}
