// gram_device.cuh -- device building blocks of the sampled-gram scans (plain
// and batched): text loads, 2-bit packing, pattern comparison, and the shape
// of a warp's work.
#pragma once

#include "scan_common.cuh"

namespace pm {
namespace gramdev {

using dev::kFull;

constexpr int kRow = 512;        // text bytes per warp row

// Four bytes in place of those at o, past a text's end: mixed bits (the last
// steps of MurmurHash3), which pass the filter as seldom as other text. Zeros
// are the codes of A, and with a gram of A only in the set one warp looked at
// every position of the last tile's rest: 48 MiB and 100 bytes against 600
// 16-mers, counts, 28.5 us, with A^16 among them 147, now 28.
__device__ __forceinline__ uint32_t past_end(long long o)
{
    uint32_t x = uint32_t(o) * 0x85EBCA6Bu;
    x = (x ^ x >> 13) * 0xC2B2AE35u;
    return x ^ x >> 16;
}

// bytes [off, off + 16) of the text, past_end from n on (a match is compared
// with the text itself and ends inside it). ENDS: a branch of its own for what
// lies past the end, which saves a short scan up to 0.5 us (200 10-mers, 900 KB:
// 12.8 us, 12.4 with it); the batched walks have no registers for it.
template <bool ENDS = true>
__device__ __forceinline__ uint4 load16(const uint8_t *text, long long n, bool aligned, long long off)
{
    if (aligned && off + 16 <= n) return __ldg(reinterpret_cast<const uint4 *>(text + off));
    if (ENDS && off >= n)
        return make_uint4(past_end(off), past_end(off + 4), past_end(off + 8), past_end(off + 12));
    uint4 v;
    if (off + 20 <= n) {
        // unaligned text: five aligned words (the last one ends inside the text)
        const uint8_t *p = text + off;
        const uint32_t sh = uint32_t(reinterpret_cast<uintptr_t>(p) & 3u) * 8u;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(p - (sh >> 3));
        if (off >= 3) {
            const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2), w3 = __ldg(w + 3), w4 = __ldg(w + 4);
            v.x = __funnelshift_r(w0, w1, sh);
            v.y = __funnelshift_r(w1, w2, sh);
            v.z = __funnelshift_r(w2, w3, sh);
            v.w = __funnelshift_r(w3, w4, sh);
            return v;
        }
    }
    uint32_t b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = past_end(off + 4 * j);
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if (off + j < n) {
            const uint32_t sh = 8u * (j & 3);
            b[j >> 2] = (b[j >> 2] & ~(0xFFu << sh)) | uint32_t(text[off + j]) << sh;
        }
    return make_uint4(b[0], b[1], b[2], b[3]);
}

// the 2-bit codes (byte >> 1) & 3 of 16 bytes, first character lowest: the
// multiply gathers a word's four codes in its top byte
__device__ __forceinline__ uint32_t pack16(const uint4 &v)
{
    constexpr uint32_t M = 0x06060606u, G = 0x00820820u;
    const uint32_t p0 = (v.x & M) * G, p1 = (v.y & M) * G, p2 = (v.z & M) * G, p3 = (v.w & M) * G;
    return __byte_perm(__byte_perm(p0, p1, 0x0073), __byte_perm(p2, p3, 0x0073), 0x5410);
}

// Bytes outside the alphabet have some letter's code (N that of G), so a long
// run of them passes wherever the set has a gram of that letter only, and is
// turned away by the comparison with the text, 32 positions at a time. The
// scans of such sets (RUNS) read a row once more when all its grams pass, and
// only those that start with a letter stay. 64 MiB with 9 % of runs of 10,000 N
// against 1,000 16-mers, G^16 among them: 290 us, now 88 (the automaton 75).
// Other sets do without: the test costs 1 % of a scan bound by instruction issue.
//
// Of the probes at every S-th of the 16 bytes at off, the first one lowest,
// those at a letter (not inlined: the scans have no registers to spare for it).
template <int S>
__device__ __noinline__ uint32_t letter_probes(const uint8_t *text, long long n, long long off, uint32_t lut)
{
    uint32_t m = 0;
    for (int k = 0; k < 16 / S; ++k) {
        const uint32_t b = off + S * k < n ? text[off + S * k] : 0u;
        if (((lut >> (8u * ((b >> 1) & 3u))) & 0xFFu) == b) m |= 1u << k;
    }
    return m;
}

// Text bytes that must follow a window's start, inside the text, for the word
// path of same_bytes: its 16-byte blocks and the word after them.
__device__ __forceinline__ int compare_span(int len) { return ((len + 15) & ~15) + 4; }

// pattern bytes (a row of zero-padded 16-byte blocks) against the text at p;
// `room`: compare_span(len) bytes from p on, and the three before it, are the
// text's. A block's loads are independent: one at a time, a 62-byte pattern
// took 16 dependent trips to L2 (158 KB of text with 5,000 matches of such
// patterns: 607 us on one CTA).
__device__ __forceinline__ bool same_bytes(const uint8_t *p, int len, const uint32_t *pat, bool room)
{
    if (room) {
        const uint32_t lead = uint32_t(reinterpret_cast<uintptr_t>(p) & 3u), sh = lead * 8u;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(p - lead);
        const uint4 *row = reinterpret_cast<const uint4 *>(pat);
#pragma unroll 2
        for (int left = len; left > 0; left -= 16, w += 4, ++row) {
            const uint4 q = __ldg(row);
            const uint32_t t0 = __ldg(w), t1 = __ldg(w + 1), t2 = __ldg(w + 2);
            uint32_t x = __funnelshift_r(t0, t1, sh) ^ q.x, y = __funnelshift_r(t1, t2, sh) ^ q.y;
            if (left < 8) {
                if (left < 4) x &= (1u << (8 * left)) - 1u;
                y &= left <= 4 ? 0u : (1u << (8 * (left - 4))) - 1u;
            }
            if (left > 8) {
                const uint32_t t3 = __ldg(w + 3), t4 = __ldg(w + 4);
                uint32_t z = __funnelshift_r(t2, t3, sh) ^ q.z, v = __funnelshift_r(t3, t4, sh) ^ q.w;
                if (left < 16) {
                    if (left < 12) z &= (1u << (8 * (left - 8))) - 1u;
                    v &= left <= 12 ? 0u : (1u << (8 * (left - 12))) - 1u;
                }
                x |= z | v;
            }
            if (x | y) return false;
        }
        return true;
    }
    for (int j = 0; j < len; ++j)
        if (p[j] != uint8_t(__ldg(pat + (j >> 2)) >> (8 * (j & 3)))) return false;
    return true;
}

// One batch of 32 passing grams: lane l has the entries e0 .. e0 + cnt - 1 for
// the gram at offset pos of the tile (cnt 0: none); win: the codes of the 16
// characters there, or (RAW) the byte gram's hash. Each lane first compares its
// entries' codes (16 of the pattern's characters, or the hash) with win, which
// leaves few to compare byte by byte. When a gram still has several, the (gram,
// entry) pairs are dealt out to the lanes in order, 32 at a time, so that one
// long list does not hold up the warp. emit(ok, entry, pos) is called by the
// whole warp; the pairs that match have ok set, and ascend by lane and call in
// output order.
struct GramTile {
    const uint4 *ent;
    const uint32_t *pats;
    int pw;
    const uint8_t *text;             // the tile's first byte
    int low, rem;                    // starts from low on, ends up to rem, are inside the text
};

// The entries of bucket bk (see GramTables::dir): first, and how many; 0 when
// none of at most four has the hash bits `fp`. One 8-byte read settles a gram
// that passed the filter by chance; a bucket's end and its entries were two
// reads more (100,000 32-mers, where four grams in five pass: 190 us per 256
// MiB).
template <bool RANK>
__device__ __forceinline__ uint32_t bucket_entries(const uint2 *dir, uint32_t bk, uint32_t fp, uint32_t &cnt)
{
    const uint2 d = __ldg(dir + bk);
    const uint32_t first = d.x & 0xFFFFFFu;
    cnt = d.x >> 24;
    if (!RANK && cnt <= 4u) {
        const uint32_t z = d.y ^ (fp & 0xFFu) * 0x01010101u;
        if (((z - 0x01010101u) & ~z & 0x80808080u) == 0u) cnt = 0u;
    }
    if (cnt == 255u) cnt = (__ldg(dir + bk + 1).x & 0xFFFFFFu) - first;
    return first;
}

template <bool RAW>
__device__ __forceinline__ bool same_code(const uint4 &en, uint32_t win)
{
    if (RAW) return en.x == win;
    const uint32_t nc = (en.z >> 8) - (en.z & 255u);   // characters from the gram on
    return ((en.x ^ win) & (nc >= 16u ? kFull : ~(kFull << (2u * nc)))) == 0u;
}

template <bool RAW, class Emit>
__device__ __forceinline__ void verify_batch(const GramTile &g, uint32_t e0, uint32_t cnt, uint32_t win, int pos,
                                             Emit &&emit)
{
    const int lane = threadIdx.x & 31;
    uint32_t nm = 0, first = 0;
    if (__any_sync(kFull, cnt > 8u)) {
        // a long list (a run of one letter in many patterns): straight to the
        // pairs, all lanes on it. With one lane on it, 64 MiB of text with 2 %
        // of runs of A against 8,000 32-mers took 3.0 ms.
        nm = cnt;
        first = e0;
    } else {
        for (uint32_t k = 0; k < cnt; ++k) {
            if (!same_code<RAW>(__ldg(g.ent + e0 + k), win)) continue;
            if (nm++ == 0) first = e0 + k;
        }
    }
    if (!__any_sync(kFull, nm != 0u)) return;
    auto one = [&](bool in, uint32_t e, uint32_t w, int p) {
        uint4 en = make_uint4(0u, 0u, 0u, 0u);
        bool ok = false;
        if (in) {
            en = __ldg(g.ent + e);
            const int start = p - int(en.z & 255u), len = int(en.z >> 8);
            ok = same_code<RAW>(en, w) && start >= g.low && start + len <= g.rem;
            if (ok)
                ok = same_bytes(g.text + start, len, g.pats + (size_t)en.y * g.pw,
                                start >= g.low + 3 && start + compare_span(len) <= g.rem);
        }
        if (__any_sync(kFull, ok)) emit(ok, en, p);
    };
    if (!__any_sync(kFull, nm > 1u)) {
        one(nm != 0u, first, win, pos);
        return;
    }
    if (nm == 0u) cnt = 0u;
    const uint32_t inc = dev::warp_incl_scan(cnt, lane), total = __shfl_sync(kFull, inc, 31);
    const uint32_t shift = e0 - (inc - cnt);   // pair x of this lane's gram is entry shift + x
    for (uint32_t x0 = 0; x0 < total; x0 += 32) {
        const uint32_t x = x0 + lane;
        int o = 0;                             // the first lane whose pairs reach past x
#pragma unroll
        for (int s = 16; s > 0; s >>= 1)
            if (__shfl_sync(kFull, inc, o + s - 1) <= x) o += s;
        const uint32_t e = x + __shfl_sync(kFull, shift, o), w = __shfl_sync(kFull, win, o);
        const int p = __shfl_sync(kFull, pos, o);
        one(x < total, e, w, p);
    }
}

}  // namespace gramdev
}  // namespace pm
