// gram_device.cuh -- device building blocks of the sampled-gram scan: text loads, 2-bit packing, pattern comparison, and the shape
// of a warp's work.
#pragma once

#include "scan_common.cuh"

namespace pm {
namespace gramdev {

using dev::kFull;

constexpr int kRow = 512;        // text bytes per warp row

// bytes [off, off + 16) of the text, zeros from n on
__device__ __forceinline__ uint4 load16(const uint8_t *text, long long n, bool aligned, long long off)
{
    if (aligned && off + 16 <= n) return __ldg(reinterpret_cast<const uint4 *>(text + off));
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
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
    uint32_t b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if (off + j < n) b[j >> 2] |= uint32_t(text[off + j]) << (8 * (j & 3));
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

// pattern bytes against the text at p; `room`: whole words around them lie
// inside the text
__device__ __forceinline__ bool same_bytes(const uint8_t *p, int len, const uint32_t *pat, bool room)
{
    if (room) {
        const uint32_t lead = uint32_t(reinterpret_cast<uintptr_t>(p) & 3u), sh = lead * 8u;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(p - lead);
        uint32_t cur = __ldg(w);
        for (int left = len; left > 0; left -= 4) {
            const uint32_t nxt = __ldg(++w);
            uint32_t x = __funnelshift_r(cur, nxt, sh) ^ __ldg(pat++);
            if (left < 4) x &= (1u << (8 * left)) - 1u;
            if (x) return false;
            cur = nxt;
        }
        return true;
    }
    for (int j = 0; j < len; ++j)
        if (p[j] != uint8_t(__ldg(pat + (j >> 2)) >> (8 * (j & 3)))) return false;
    return true;
}

}  // namespace gramdev
}  // namespace pm
