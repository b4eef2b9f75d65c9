// gram.cpp -- host-side tables of the sampled-gram scan (scan_gram.cu) and a
// host walk of them.
//
// Every pattern of the set is at least m characters long (m the shortest
// length). Take a stride s and a gram length q with q <= m - s + 1. Of the s
// consecutive text positions i .. i + s - 1 after a start i exactly one, t, is
// a multiple of s, and the q characters at t are the characters k .. k + q - 1
// of any pattern that occurs at i, k = t - i < s. So it is enough to look at
// the grams at multiples of s: each pattern enters a table under its first s
// grams (offset k = 0 .. s - 1), a text gram not in the table rules out s
// starts at once, and a gram that is in it names the candidates (pattern, k),
// which are compared with the text byte by byte. This is the block idea of
// Wu-Manber's SHIFT and HASH tables (Section 3.2, Algorithms 4 and 5) with a
// fixed shift s, so that no position depends on the one before it.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <string_view>
#include <unordered_map>

#include "pm_internal.h"

namespace pm {

namespace {

inline uint32_t code2(uint32_t b) { return (b >> 1) & 3u; }

// odd multipliers of the gram hash (any odd numbers with mixed bits do)
constexpr uint32_t kMul[4] = {0x9E3779B1u, 0x5DB3D743u, 0xA54FF53Bu, 0x510E527Fu};

// the gram's hash, and the filter bit it sets: the word by the hash's top
// bits, the bit by the low bits of the gram's codes (or of a byte gram's hash)
uint32_t gram_hash(const GramTables &t, const uint8_t *g, uint32_t *bit)
{
    uint32_t h = 0;
    if (t.qw == 0) {
        for (int j = 0; j < t.q; ++j) h |= code2(g[j]) << (2 * j);
        const uint32_t x = h * t.K[0];
        *bit = (x >> (37 - t.fb)) << 5 | (h & 31u);
        return x;
    }
    for (int w = 0; w < t.qw; ++w) {
        const uint32_t x = uint32_t(g[4 * w]) | uint32_t(g[4 * w + 1]) << 8 | uint32_t(g[4 * w + 2]) << 16 |
                           uint32_t(g[4 * w + 3]) << 24;
        h += x * t.K[w];
    }
    *bit = (h >> (37 - t.fb)) << 5 | (h & 31u);
    return h;
}

// the 2-bit codes of up to 16 of len characters, first one lowest
uint32_t codes(const uint8_t *p, int64_t len)
{
    uint32_t x = 0;
    for (int j = 0; j < 16 && j < len; ++j) x |= code2(p[j]) << (2 * j);
    return x;
}

// What a set and its gram plan are like, per position of random text.
struct GramShape {
    int64_t d;
    int letters, hi;
    bool packed;
    double matches;     // matches
    double hits;        // entries of one gram
    double pass;        // grams that pass the filter, per probe
    double states;      // the set's trie
};

// When the method's own scan is taken all the same. Times are of one pass over
// 64 MiB, list mode, unless they say otherwise.
struct GramLimits {
    double cost;        // planned instructions per lane and 16 characters (sampled grams)
    double dense_pass;  // part of all texts' m-grams in a dense set
    uint32_t longest;   // entries of one gram
};

GramLimits gram_limits(int32_t algo, int32_t B, const GramShape &g)
{
    // Cost. The transition-table walk of a one-length Aho-Corasick set takes, in
    // units of about 4.6 us per GiB: tables of fewer than about 2,000 patterns in
    // shared memory 0.8 ms per GiB, larger ones past it 3 ms, general alphabets
    // 4.4 ms; a PFAC walk 11 ms and more. Wu-Manber compares every candidate of a
    // window in turn and is never faster (1.2 to 70 times slower).
    //
    // Dense sets that hold most m-grams. 8 MiB: 3,000 5-mers (95 % of all) 336 us
    // and 319 by the automaton (PFAC 338 and 294), 300 4-mers (69 %) 199 and 204
    // (199 and 189); 3,000 6-mers (52 %) 128 and 181 (127 and 185).
    //
    // A gram with hundreds of entries means repetitive patterns (runs of one
    // letter): in a text with such repeats every occurrence costs them all, and
    // work grows as text times d. The automata do not care. 16 MiB with 2 % of
    // runs of A, 4,000 32-mers of which f begin with 24 A (576, 2,304 and 36,000
    // entries at f = 64, 256 and 4,000): grams 0.18, 0.72 and 16 ms; automaton
    // 0.09, one or mixed lengths 0.10, PFAC 0.37. The limits are about where the
    // two meet at 2 %. Wu-Manber depends on its blocks: the exact tables (four
    // letters or fewer, up to 32 characters) take 0.28, 0.33 and 2.0 ms with B = 2
    // and 0.10, 0.10 and 0.22 with B = 4; byte-hash tables over 20 letters 0.29,
    // 0.45 and 4.2 with B = 2, 0.04 with B = 4. Where a block names more than 64
    // patterns (d / letters^B) every window compares them, and grams win at any
    // length: 4,000 patterns of 32 to 47 letters over ACGT 0.18, 0.74 and 17 ms,
    // without 8.1, 13 and 101.
    // Lists a few times longer than those of random text are no sign of
    // repetition. (At most 2^18: a tile's keys are added up in 32 bits, at most
    // 2^14 starts with all patterns of one gram each.)
    constexpr uint32_t most = (1u << 18) - 1u;
    auto longest = [&](uint32_t n) { return uint32_t(std::min(std::max(double(n), 4.0 * g.hits), double(most))); };
    constexpr double any = 1e30;
    switch (algo) {
    case PM_ALGO_AC: return {g.packed ? (g.d < 2000 ? 170.0 : 650.0) : 900.0, 0.6, longest(256)};
    case PM_ALGO_PFAC: return {2400.0, 0.6, longest(1024)};
    case PM_ALGO_ACV: return {any, 1.0, longest(256)};
    default: break;
    }
    const bool exact = g.packed && g.hi <= 32;
    if (!exact && double(g.d) > 64.0 * std::pow(double(g.letters), double(B))) return {any, 1.0, most};
    return {any, 1.0, longest(B < 3 ? 1024 : exact ? 256 : 64)};
}

// Mixed lengths: the automaton against grams, in list mode and for counts, by
// estimates in us per 64 MiB of random text. Both were fitted to some 100 sets
// (30 to 100,000 patterns from 3 to 65 characters, 2, 4 and 20 letters): grams
// cost by windows that pass, entries compared and keys, the automaton by
// matches, far more in list mode, and by whether its table is small. Counts with
// grams and without: 3,000 patterns of 3 to 65 letters over ACGT 11,600 us and
// 3,800, 8,000 of 5 to 8 3,740 and 3,050, 8,000 of 6 to 9 1,370 and 3,080, 8,000
// of 8 to 16 95 and 340; list mode 12,800 and 7,700, 4,440 and 11,050, 1,530 and
// 6,130, 102 and 406.
void acv_modes(const GramShape &g, int s, bool &list, bool &counts)
{
    const double M = g.matches, grams = 40.0 + 1000.0 * g.pass / s + 300.0 * g.hits / s;
    const double base = g.packed ? 75.0 : 150.0;
    const bool small = g.states < 8192.0;
    counts = grams <= (small ? base + 900.0 * M : 250.0 + 3400.0 * std::sqrt(M));
    list = grams + 500.0 * M <=
           (small ? base + M * (1500.0 + 3000.0 * M) : 250.0 + 8000.0 * std::sqrt(M) + 1000.0 * M * M);
}

}  // namespace

int build_gram(const uint8_t *P, const int64_t *off, int64_t d, int32_t m, int32_t algo, int32_t B, GramTables &t)
{
    t = GramTables();
    try {
        const bool var = off != nullptr;
        auto first = [&](int64_t r) { return var ? off[r] : r * int64_t(m); };
        auto len_of = [&](int64_t r) { return int(var ? off[r + 1] - off[r] : m); };
        // (the other compilers refuse bad offsets and sizes: no plan here)
        if (d > (int64_t(1) << 23) || (var && off[0] != 0) || (!var && m > 255)) return PM_OK;
        for (int64_t r = 0; var && r < d; ++r)
            if (off[r + 1] <= off[r] || off[r + 1] - off[r] > 255) return PM_OK;
        bool present[256] = {};
        int lo = 1 << 30, hi = 0;
        int64_t with_len[256] = {};
        for (int64_t r = 0; r < d; ++r) {
            const int L = len_of(r);
            ++with_len[L];
            lo = std::min(lo, L);
            hi = std::max(hi, L);
            const uint8_t *p = P + first(r);
            for (int j = 0; j < L; ++j) present[p[j]] = true;
        }
        int letters = 0;
        bool packed = true, seen[4] = {};
        for (uint32_t b = 0; b < 256; ++b) {
            if (!present[b]) continue;
            ++letters;
            if (seen[code2(b)]) packed = false;
            seen[code2(b)] = true;
        }

        // Plan: the stride and gram that cost least per 16 text bytes, in
        // instructions per lane: each probe, each gram that passes the filter
        // (by chance in the hashed filter, or because so many grams of the
        // alphabet are in the table), and each entry compared (G / space is
        // the mean number of entries under a gram of random text; without
        // that term a set of 8,000 8-mers would take 1-character grams). With 40
        // and 60 in place of 60 and 130, 2,000 12-mers over 20 letters took
        // 4-character grams (58 us per 64 MiB against 46 with 8) and 1,000
        // patterns of 8-16 characters every second position (155 us per 128
        // MiB against 129). The dense form's cost is fitted to 1,000 and 8,000
        // 8-mers; its base keeps 100 8-mers sampled, which is faster on short texts
        // and slower on long ones (14.4 us per MiB against 16.2, 64 MiB 36.9 against
        // 38.9, 256 MiB 121 against 113).
        //
        // 2-bit grams may be longer than the shortest rest m - s + 1: a gram of
        // which the pattern has only the first L characters enters with all 4^(q
        // - L) endings. Up to 10 characters the filter is exact, so this turns
        // away most windows of the longer patterns in a mixed set: 8,000 of 8 to
        // 16 characters with 8-character grams took 567 us per 256 MiB, 1,000
        // 121 us per 128 MiB.
        double best = 1e30, best_hits = 0.0, best_pass = 0.0;
        for (int s = 16; s >= 1; s >>= 1) {
            const int shortest = lo - s + 1;
            for (int form = 0; form < (packed ? 3 : 1); ++form) {
                int q = form == 0 ? std::min(16, shortest) : form == 1 ? 9 : 10;
                if (!packed) q &= ~3;
                if (q < (packed ? 3 : 4) || shortest < 1 || (form > 0 && q <= shortest)) continue;
                // (buckets of exact 10-character grams go by their last six: 64 of
                // 4,096 with two letters. 1,000 patterns of 10 to 20 of them as a
                // mixed set, 4 MiB: 640 us, hashed or 9-character grams 120)
                if (form == 2 && letters < 4) continue;
                // entries, and how many of them a gram of random text has
                double G = 0.0, hits = 0.0;
                for (int L = lo; L <= hi; ++L)
                    for (int k = 0; k < s && with_len[L]; ++k) {
                        const int have = std::min(q, L - k);
                        G += double(with_len[L]) * std::pow(4.0, double(q - have));
                        hits += double(with_len[L]) / std::pow(double(std::max(letters, 2)), double(have));
                    }
                if (G > (form == 0 ? 8.0e6 : 1.0e5)) continue;
                const bool direct = packed && 2 * q <= 20 && (form > 0 || 2 * q <= 18);
                const bool dense = form == 0 && direct && s == 1 && !var && q == hi && d < 32768;
                int fb = direct ? 2 * q : 12;
                if (!direct)
                    while (fb < 20 && double(1u << fb) < 32.0 * G) ++fb;
                const double natural = 1.0 - std::exp(-hits);
                const double chance = direct ? 0.0 : 1.0 - std::exp(-G / double(1u << fb));
                const double pass = 1.0 - (1.0 - natural) * (1.0 - chance);
                const double probes = 16.0 / s;
                double cost = dense ? 125.0 + probes * 74.0 * pass
                                    : 24.0 + probes * ((packed ? 9.0 : 8.0 + q / 4) + 60.0 * pass + 130.0 * hits);
                if (form == 2) cost += 10.0;  // 128 KiB of filter to load
                if (cost < best) {
                    best = cost;
                    t.s = s;
                    t.q = q;
                    t.qw = packed ? 0 : q / 4;
                    t.fb = fb;
                    t.direct = direct;
                    t.rank = direct && 2 * q <= 18;
                    t.dense = dense;
                    best_hits = hits;
                    best_pass = dense ? natural : pass;
                }
            }
        }
        // too short for any gram, too many patterns, or so many candidates that
        // the method's own scan is faster
        GramShape shape{d, letters, hi, packed, 0.0, best_hits, best_pass, 1.0};
        for (int L = hi, longer = 0; L >= 1; --L) {
            const double grams = std::pow(double(std::max(letters, 2)), double(L));
            longer += int(with_len[L]);
            shape.matches += double(with_len[L]) / grams;
            shape.states += std::min(grams, double(longer));
        }
        const GramLimits lim = gram_limits(algo, B, shape);
        if (t.s == 0 || (t.dense ? best_pass > lim.dense_pass : best > lim.cost)) {
            t = GramTables();
            return PM_OK;
        }
        t.var = var;
        t.cost = best;
        t.d = d;
        t.m_min = lo;
        t.m_max = hi;
        for (int w = 0; w < 4; ++w) t.K[w] = kMul[w];
        if (packed) t.K[0] = (t.direct ? 1u : kMul[0]) << (32 - 2 * t.q);

        // distinct patterns of a one-length set (groups of equal patterns, as
        // in the other tables); every pattern of its own in a mixed one
        std::vector<int64_t> rep;
        if (!var) {
            std::unordered_map<std::string_view, uint32_t> index;
            index.reserve(size_t(d) * 2);
            std::vector<uint32_t> cls(static_cast<size_t>(d)), mult;
            for (int64_t r = 0; r < d; ++r) {
                const std::string_view key(reinterpret_cast<const char *>(P + r * int64_t(m)), size_t(m));
                const auto it = index.emplace(key, uint32_t(rep.size()));
                if (it.second) {
                    rep.push_back(r);
                    mult.push_back(0);
                }
                cls[size_t(r)] = it.first->second;
                ++mult[it.first->second];
            }
            t.code.resize(rep.size());
            std::vector<uint32_t> fill(rep.size(), 0);
            t.grp_off.push_back(0);
            for (size_t c = 0; c < rep.size(); ++c) {
                t.code[c] = uint32_t(rep[c]);
                if (mult[c] < 2) continue;
                t.code[c] = 0x80000000u | uint32_t(t.grp_off.size() - 1);
                fill[c] = t.grp_off.back();
                t.grp_off.push_back(t.grp_off.back() + mult[c]);
            }
            t.grp_ids.resize(t.grp_off.back());
            // tiles add up their keys in 32 bits: at most 2^14 positions each
            t.max_keys = *std::max_element(mult.begin(), mult.end());
            if (t.max_keys >= 1u << 18) {
                t = GramTables();
                return PM_OK;
            }
            for (int64_t r = 0; r < d; ++r) {
                const uint32_t c = cls[size_t(r)];
                if (mult[c] >= 2) t.grp_ids[fill[c]++] = uint32_t(r);
            }
        } else {
            rep.resize(size_t(d));
            t.code.resize(size_t(d));
            for (int64_t r = 0; r < d; ++r) {
                rep[size_t(r)] = r;
                t.code[size_t(r)] = uint32_t(r);
            }
        }
        const size_t nc = rep.size();
        t.pw = (hi + 15) / 16 * 4;   // whole 16-byte blocks
        t.pats.assign(nc * size_t(t.pw), 0u);
        for (size_t c = 0; c < nc; ++c)
            std::memcpy(reinterpret_cast<uint8_t *>(t.pats.data() + c * size_t(t.pw)), P + first(rep[c]),
                        size_t(len_of(rep[c])));

        // entries, bucket-major; inside a bucket by (k descending, pattern
        // ascending), so that the starts t - k come out in ascending order
        // and equal starts in ascending pattern id
        struct Gram {
            uint32_t h, ck;   // hash; distinct pattern (d <= 2^23) | offset << 24
        };
        std::vector<Gram> grams;
        grams.reserve(nc * size_t(t.s));
        t.filter.assign(size_t(1) << (t.fb - 5), 0u);
        for (int k = t.s - 1; k >= 0; --k)
            for (size_t c = 0; c < nc; ++c) {
                const uint8_t *p = P + first(rep[c]) + k;
                const int have = len_of(rep[c]) - k;
                if (have >= t.q) {
                    uint32_t b;
                    const uint32_t x = gram_hash(t, p, &b);
                    t.filter[b >> 5] |= 1u << (b & 31u);
                    grams.push_back({x, uint32_t(c) | uint32_t(k) << 24});
                    continue;
                }
                const uint32_t head = codes(p, have);   // direct grams: every ending
                for (uint32_t e = 0; e < 1u << (2 * (t.q - have)); ++e) {
                    const uint32_t b = head | e << (2 * have);
                    t.filter[b >> 5] |= 1u << (b & 31u);
                    grams.push_back({b * t.K[0], uint32_t(c) | uint32_t(k) << 24});
                }
            }
        const size_t G = grams.size();
        uint32_t run[4];   // (K is odd: different grams have different hashes)
        for (uint32_t c = 0; c < 4; ++c) run[c] = (0x55555555u >> (32 - 2 * t.q)) * c * t.K[0];
        for (const Gram &x : grams)
            t.runs = t.runs || (packed && (x.h == run[0] || x.h == run[1] || x.h == run[2] || x.h == run[3]));
        auto bucket = [&](uint32_t x) -> uint32_t {
            if (!t.rank) return x >> (32 - t.db);
            const uint32_t b = x >> (32 - t.fb);
            return t.rank_base[b >> 5] + uint32_t(__builtin_popcount(t.filter[b >> 5] & ((1u << (b & 31)) - 1u)));
        };
        size_t nb;
        if (t.rank) {
            t.rank_base.resize(t.filter.size());
            uint32_t run = 0;
            for (size_t w = 0; w < t.filter.size(); ++w) {
                t.rank_base[w] = run;
                run += uint32_t(__builtin_popcount(t.filter[w]));
            }
            nb = run;
        } else {
            // (a pattern's endings are the top bits of direct grams and at most
            // as many as there are buckets: they fall into different ones)
            t.db = 12;
            while (t.db < 24 && (size_t(1) << t.db) < G) ++t.db;
            nb = size_t(1) << t.db;
        }
        std::vector<uint32_t> at(nb + 1, 0u);
        for (const Gram &x : grams) ++at[bucket(x.h) + 1];
        for (size_t b = 0; b < nb; ++b) at[b + 1] += at[b];
        uint32_t longest = 0;
        for (size_t b = 0; b < nb; ++b) longest = std::max(longest, at[b + 1] - at[b]);
        if (longest > lim.longest) {
            if (algo != PM_ALGO_WM && algo != PM_ALGO_WMV) {
                t = GramTables();
                return PM_OK;
            }
            t.list = t.counts = false;
        }
        t.dir.assign(2 * (nb + 1), 0u);
        for (size_t b = 0; b <= nb; ++b) {
            const uint32_t cnt = b < nb ? at[b + 1] - at[b] : 0u;
            t.dir[2 * b] = at[b] | std::min(cnt, 255u) << 24;
        }
        t.ent.resize(G);
        for (const Gram &x : grams) {
            const uint32_t b = bucket(x.h), e = at[b]++, c = x.ck & 0xFFFFFFu, k = x.ck >> 24;
            const int len = len_of(rep[c]);
            GramEntry &en = t.ent[e];
            en.h = t.qw == 0 ? codes(P + first(rep[c]) + k, len - int(k)) : x.h;
            en.idx = c;
            en.k_len = k | uint32_t(len) << 8;
            en.code = t.code[c];
            const uint32_t i = e - (t.dir[2 * b] & 0xFFFFFFu);
            for (uint32_t u = i; u < 4 && !t.rank; ++u) {
                t.dir[2 * b + 1] &= ~(0xFFu << (8 * u));
                t.dir[2 * b + 1] |= ((x.h >> (24 - t.db)) & 0xFFu) << (8 * u);
            }
        }
        for (uint32_t c = 0; packed && c < 4; ++c) {
            uint32_t b = 0;
            while (b < 256 && !(present[b] && code2(b) == c)) ++b;
            // an absent letter: a byte with another code never equals the text's
            t.lut |= (b < 256 ? b : (c ^ 1u) << 1) << (8 * c);
        }
        if (t.dense) {
            t.id_off.push_back(0);
            for (const GramEntry &e : t.ent) {
                const uint32_t gi = e.code & 0x7FFFFFFFu;
                if (e.code & 0x80000000u)
                    t.ids.insert(t.ids.end(), t.grp_ids.begin() + t.grp_off[gi], t.grp_ids.begin() + t.grp_off[gi + 1]);
                else t.ids.push_back(uint16_t(e.code));
                t.id_off.push_back(uint16_t(t.ids.size()));
            }
        }
        if (algo == PM_ALGO_ACV) acv_modes(shape, t.s, t.list, t.counts);
        t.ok = true;
        return PM_OK;
    } catch (const std::bad_alloc &) {
        t = GramTables();
        return PM_ENOMEM;
    }
}

void host_walk_gram(const GramTables &t, const uint8_t *T, int64_t n, std::vector<uint64_t> &occ,
                    std::vector<int64_t> &counts)
{
    occ.clear();
    counts.assign(size_t(t.d), 0);
    uint8_t g[16];
    for (int64_t p = 0; p < n; p += t.s) {
        for (int j = 0; j < 16; ++j) g[j] = p + j < n ? T[p + j] : uint8_t(0);
        uint32_t b;
        const uint32_t x = gram_hash(t, g, &b);
        if (!((t.filter[b >> 5] >> (b & 31)) & 1u)) continue;
        uint32_t bk;
        if (t.rank)
            bk = t.rank_base[b >> 5] + uint32_t(__builtin_popcount(t.filter[b >> 5] & ((1u << (b & 31)) - 1u)));
        else bk = x >> (32 - t.db);
        const uint32_t first = t.dir[2 * bk] & 0xFFFFFFu;
        uint32_t cnt = t.dir[2 * bk] >> 24;
        if (!t.rank && cnt <= 4) {
            bool any = false;
            for (int u = 0; u < 4; ++u)
                any = any || ((t.dir[2 * bk + 1] >> (8 * u)) & 0xFFu) == ((x >> (24 - t.db)) & 0xFFu);
            if (!any) continue;
        }
        if (cnt == 255) cnt = (t.dir[2 * bk + 2] & 0xFFFFFFu) - first;
        for (uint32_t e = first; e < first + cnt; ++e) {
            const GramEntry &en = t.ent[e];
            const int64_t start = p - int64_t(en.k_len & 255u), len = int64_t(en.k_len >> 8);
            if (start < 0 || start + len > n) continue;
            if (t.qw != 0 ? en.h != x : en.h != codes(T + p, start + len - p)) continue;
            if (std::memcmp(T + start, t.pats.data() + size_t(en.idx) * size_t(t.pw), size_t(len)) != 0) continue;
            auto put = [&](uint32_t r) {
                occ.push_back((uint64_t(start) << 32) | r);
                ++counts[r];
            };
            if (en.code & 0x80000000u) {
                const uint32_t gi = en.code & 0x7FFFFFFFu;
                for (uint32_t j = t.grp_off[gi]; j < t.grp_off[gi + 1]; ++j) put(t.grp_ids[j]);
            } else {
                put(en.code);
            }
        }
    }
}

}  // namespace pm
