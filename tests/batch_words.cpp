// Host check of the batch planner (compiled and run by test_batch_words.py):
// whatever plan pm_tune gives a set after its batch was prepared, the layouts
// of that batch need the words its workspace was sized for.
#include <cstdio>
#include <cstring>
#include <random>

#include "pm_internal.h"

using namespace pm;

int main()
{
    std::mt19937 rng(5);
    const int sizes[][2] = {{10000, 32}, {300, 12}, {9000, 16}};   // patterns, length
    const int64_t texts[] = {8192, 3 << 20, 200000};
    pm_set sets[3];
    BatchInst inst[3];
    for (int k = 0; k < 3; ++k) {
        const int64_t d = sizes[k][0], m = sizes[k][1];
        std::vector<uint8_t> P(size_t(d * m));
        for (auto &c : P) c = "ACGT"[rng() & 3u];
        sets[k].algo = PM_ALGO_AC;
        if (build_ac(P.data(), d, int32_t(m), sets[k].ac) ||
            build_gram(P.data(), nullptr, d, int32_t(m), PM_ALGO_AC, 0, sets[k].gram) || !sets[k].gram.ok)
            return 2;
        sets[k].dac.dg = &sets[k].dgram;   // the scans of a set just compiled take its grams
        inst[k] = BatchInst{&sets[k], 0, texts[k], 0, 0, texts[k], k, batch_takes_grams(&sets[k])};
        if (!inst[k].gram) return 3;
    }
    int bad = 0, gram_items = 0;
    for (int warps : {8, 12, 16})
        for (int policy : {0, 1})
            for (bool list : {true, false}) {
                BatchShape sh;             // a device of 152 SMs with 227 KB a block
                sh.warps = warps;
                sh.policy = policy;
                sh.region_bytes = 230400 - warps * 8192;
                sh.gram_smem = 230400;
                sh.sm_count = 152;
                std::vector<BatchDesc> items;
                int64_t spill[2], words[2], bound = 0;
                for (int tuned : {0, 1}) {   // 1: the tuner took every set off the grams
                    for (pm_set &s : sets) s.dac.dg = tuned ? nullptr : &s.dgram;
                    words[tuned] = batch_items(inst, 3, sh, list, items, &spill[tuned]);
                    gram_items += batch_gram_items(items);
                }
                for (const BatchInst &I : inst) bound += batch_words_bound(I, sh, list);
                if (words[0] != words[1] || spill[0] != spill[1] || words[0] + spill[0] > bound) {
                    std::printf("warps %d policy %d list %d: %lld + %lld words, tuned %lld + %lld, bound %lld\n", warps,
                                policy, int(list), (long long)words[0], (long long)spill[0], (long long)words[1],
                                (long long)spill[1], (long long)bound);
                    ++bad;
                }
            }
    return bad || gram_items == 0 ? 1 : 0;
}
