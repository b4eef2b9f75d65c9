// scan_gram.cu -- sampled-gram scan on sm_103a: one table lookup per s text
// positions (the tables are described in gram.cpp).
//
// A warp takes rows of 512 text bytes, 16 per lane, two rows per load batch
// with the next batch in flight. The lane's 16 characters become one 32-bit
// word of 2-bit codes (one multiply-add per 4 bytes); with the next lane's
// word that gives the gram at any offset by one funnel shift, and its hash by
// one multiply. A filter bit in shared memory drops almost every gram. No
// lookup depends on another one, so a lane has 16 / s of them in flight: the
// walk of the transition table, by contrast, is one dependent shared-memory
// access per character.
//
// Grams that pass are packed into the warp's queue in text order and taken 32
// at a time: bucket, entries, byte comparison with the text (which also
// settles bytes outside the alphabet). The matches of a tile go to its slot
// in text order, and the expand kernel of the other scans writes the keys.
//
// Bound: instruction issue (62-76 % of the issue slots, 53 % of DRAM at stride 8
// and 16, 10-38 % below; about 90 warp instructions per row at stride 16, 102 at
// 8, 153 at 4). Filters of 192 KiB passed fewer grams and were slower (20,000
// 32-mers 96 us against 75): candidates live on what L1 the filter leaves.
// 256 MiB of EST-shaped text, list mode, this scan against the one it replaces:
// 20,000 32-mers 73 us (s = 16) against 1.64 ms (hybrid transition table),
// 100,000 32-mers 129 us against 2.46 ms, 8,000 16-mers compiled as Wu-Manber 98
// us (s = 4) against 2.10 ms, 8,000 patterns of 8-16 characters 347 us (s = 1)
// against 1.41 ms; counts of 1,000 16-mers 62 us (s = 8) against 183.
#include <algorithm>
#include <type_traits>

#include "gram_device.cuh"

namespace pm {
namespace {

using dev::kFull;
using namespace gramdev;

constexpr int kMaxWarps = 32;

// rows per load batch: enough bytes in flight, at most 16 grams a lane
__host__ __device__ constexpr int rows_of(int s) { return s >= 8 ? 4 : s >= 2 ? 2 : 1; }
// the shortest tile, whole batches and at least kWarpTile bytes
__host__ __device__ constexpr int min_tile(int s) { return s >= 8 ? 4096 : 3072; }

struct GramArgs {
    const uint8_t *text;
    long long n;
    int aligned;
    uint32_t K[4];
    uint32_t lut;                 // the letter of code c in byte c
    int fshift, wshift, bshift;   // 32 - fb, 32 - (fb - 5), 32 - db
    int fwords;                   // filter words
    const uint32_t *filter_g;
    const uint32_t *rank_g;
    const uint2 *dir;
    const uint4 *ent;
    const uint32_t *pats;
    int pw;
    const uint32_t *code;
    const uint32_t *grp_off, *grp_ids;
    int ncodes;
    int tile;                     // text bytes per tile (a multiple of kRow * rows_of(S))
    long long ntiles;
    int list, hist_smem;
    int slot_kind;                // 0: (off << 16) | code16, 1: (off << 32) | code, 2: (off << 20) | r
    long long slot_stride;        // entries per tile
    void *slots;
    uint32_t *tile_ent, *tile_out;
    unsigned long long *seg_sum;
    long long seg_tiles;
    long long *counts;
    long long *n_occ;
};

__host__ __device__ constexpr int qcap(int s) { return 32 + rows_of(s) * kRow / s; }

// S: stride; QW: 0 2-bit grams, else words of a byte gram; RANK: buckets by
// rank in the filter, else by hash. The queue holds each passing gram's offset
// and the codes of the 16 characters from it on (a byte gram's hash). RUNS: see
// letter_probes.
template <int S, int QW, bool RANK, bool RUNS>
__global__ void __launch_bounds__(kMaxWarps * 32, 1) gram_scan_kernel(const GramArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NP = 16 / S;       // probes per lane and row
    constexpr int R = rows_of(S);
    constexpr int QCAP = qcap(S);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;

    uint32_t *s_filter = reinterpret_cast<uint32_t *>(smem);
    uint32_t *s_rank = s_filter + ((a.fwords + 3) & ~3);
    uint32_t *s_hist = s_rank + (RANK ? (a.fwords + 3) & ~3 : 0);
    uint32_t *q32 = s_hist + (a.hist_smem ? (a.ncodes + 3) & ~3 : 0) + warp * (QCAP + QCAP / 2);
    uint16_t *q16 = reinterpret_cast<uint16_t *>(q32 + QCAP);

    {   // the tables are padded to 16 bytes
        uint4 *f4 = reinterpret_cast<uint4 *>(s_filter), *r4 = reinterpret_cast<uint4 *>(s_rank);
        for (int i = threadIdx.x; i < (a.fwords + 3) / 4; i += blockDim.x) {
            f4[i] = __ldg(reinterpret_cast<const uint4 *>(a.filter_g) + i);
            if (RANK) r4[i] = __ldg(reinterpret_cast<const uint4 *>(a.rank_g) + i);
        }
    }
    if (a.hist_smem)
        for (int i = threadIdx.x; i < a.ncodes; i += blockDim.x) s_hist[i] = 0u;
    dev::grid_trigger();
    __syncthreads();
    dev::grid_wait();   // the zeroed counts and sums

    const uint32_t ntiles = uint32_t(a.ntiles);
    const uint32_t G = gridDim.x * (blockDim.x >> 5);
    const int ngroups = a.tile / (kRow * R);
    uint32_t st = blockIdx.x * (blockDim.x >> 5) + warp;
    unsigned long long my_total = 0;
    const uint32_t K0 = a.K[0];

    uint4 v[R + 1];                  // a batch's rows, and the 16 bytes after them (lane 0)
    auto load = [&](uint32_t t, int g) {
        const long long base = (long long)t * a.tile + g * (kRow * R);
        if (a.aligned && base + kRow * R + 16 <= a.n) {
            const uint4 *p = reinterpret_cast<const uint4 *>(a.text + base) + lane;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = __ldg(p + 32 * r);
            if (lane == 0) v[R] = __ldg(p + 32 * R);
        } else {
#pragma unroll
            for (int r = 0; r <= R; ++r)
                if (r < R || lane == 0) v[r] = load16(a.text, a.n, a.aligned, base + lane * 16 + r * kRow);
        }
    };
    if (st < ntiles) load(st, 0);
    int g = 0;
    uint32_t ent = 0, outs = 0;      // the tile's entries (uniform) and this lane's keys
    uint32_t qn = 0;                 // queue length (uniform)

    while (st < ntiles) {
        const bool last = g + 1 == ngroups;
        const uint32_t stn = last ? st + G : st;
        const int gn = last ? 0 : g + 1;

        // ---- the batch's grams: hash, and the word that names the bit ----
        uint32_t lo[R], hi[R];           // 2-bit grams: 16 characters and the 16 after them
        uint32_t H[QW == 0 ? 1 : R * NP];
        if (QW == 0) {
            uint32_t c[R + 1];
#pragma unroll
            for (int r = 0; r <= R; ++r) c[r] = pack16(v[r]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                lo[r] = c[r];
                hi[r] = __shfl_sync(kFull, lane == 0 ? c[r + 1] : c[r], (lane + 1) & 31);
            }
        } else {
            constexpr int NX = (16 - S + 4 * QW - 1) / 4 - 3;  // words of the next lane a gram may reach
#pragma unroll
            for (int r = 0; r < R; ++r) {
                uint32_t x[8];
                x[0] = v[r].x; x[1] = v[r].y; x[2] = v[r].z; x[3] = v[r].w;
                if (NX > 0) x[4] = __shfl_sync(kFull, lane == 0 ? v[r + 1].x : v[r].x, (lane + 1) & 31);
                if (NX > 1) x[5] = __shfl_sync(kFull, lane == 0 ? v[r + 1].y : v[r].y, (lane + 1) & 31);
                if (NX > 2) x[6] = __shfl_sync(kFull, lane == 0 ? v[r + 1].z : v[r].z, (lane + 1) & 31);
                if (NX > 3) x[7] = __shfl_sync(kFull, lane == 0 ? v[r + 1].w : v[r].w, (lane + 1) & 31);
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    uint32_t h = 0u;
#pragma unroll
                    for (int j = 0; j < QW; ++j) {
                        const int o = S * k + 4 * j;
                        const uint32_t y = (o & 3) == 0 ? x[o >> 2]
                                                        : __funnelshift_r(x[o >> 2], x[(o >> 2) + 1], 8 * (o & 3));
                        h += y * a.K[j];
                    }
                    H[QW == 0 ? 0 : r * NP + k] = h;
                }
            }
        }
        // the rows are in registers as grams: the next batch's loads
        if (stn < ntiles) load(stn, gn);

        // ---- a filter bit per probe, the first one lowest ----
        uint32_t mask[R], any = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const uint32_t win = QW == 0 ? (k == 0 ? lo[r] : __funnelshift_r(lo[r], hi[r], 2 * S * k))
                                             : H[QW == 0 ? 0 : r * NP + k];
                const uint32_t h = QW == 0 ? win * K0 : win;
                const uint32_t w = s_filter[h >> a.wshift];
                m = __funnelshift_r(m, __funnelshift_r(w, 0u, win), 1);  // bit `win mod 32` of w, appended
            }
            mask[r] = m >> (32 - NP);
            any |= mask[r];
        }
        // ---- passing grams -> queue, row by row, lane by lane (text order) ----
        if (__any_sync(kFull, any != 0u)) {
            // Each lane's place: with one gram a row from ballots, else from one
            // scan of all rows' counts. A row's count stays below the next field
            // (32 lanes x NP; four rows only up to two grams each).
            constexpr int F = R == 4 ? 8 : 16;
            uint32_t ex = 0, tot = 0;
            auto places = [&]() {
                uint32_t cnt = 0;
#pragma unroll
                for (int r = 0; r < R; ++r) cnt |= uint32_t(__popc(mask[r])) << (F * r);
                const uint32_t inc = dev::warp_incl_scan(cnt, lane);
                ex = inc - cnt;
                tot = __shfl_sync(kFull, inc, 31);
            };
            if (NP > 1) places();
            if (RUNS && (NP > 1 ? (tot & ((1u << F) - 1u)) == 32u * NP : __all_sync(kFull, mask[0]))) {
                const long long base = (long long)st * a.tile + g * (kRow * R) + lane * 16;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    mask[r] &= letter_probes<S>(a.text, a.n, base + r * kRow, a.lut);
                if (NP > 1) places();
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                uint32_t m = mask[r], at = qn;
                if (NP == 1) {
                    const uint32_t bal = __ballot_sync(kFull, m);
                    at += __popc(bal & lt);
                    qn += __popc(bal);
                } else {
                    constexpr uint32_t M = (1u << F) - 1u;
                    at += (ex >> (F * r)) & M;
                    qn += (tot >> (F * r)) & M;
                }
                const uint32_t off0 = uint32_t(g * R + r) * kRow + uint32_t(lane) * 16u;
                if (QW == 0 && NP > 1) {
                    while (m) {
                        const uint32_t k = uint32_t(__ffs(int(m))) - 1u;
                        m &= m - 1u;
                        q32[at] = __funnelshift_r(lo[r], hi[r], 2 * S * k);
                        q16[at++] = uint16_t(off0 + S * k);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < NP; ++k)
                        if ((m >> k) & 1u) {
                            q32[at] = QW == 0 ? lo[r] : H[QW == 0 ? 0 : r * NP + k];
                            q16[at++] = uint16_t(off0 + S * k);
                        }
                }
            }
            __syncwarp();
        }
        // ---- full batches of 32 (at the tile's end the rest too) ----
        if (qn >= 32u || (last && qn > 0u)) {
            const long long tile0 = (long long)st * a.tile;
            // starts relative to the tile, inside the text
            const GramTile view{a.ent, a.pats, a.pw, a.text + tile0, tile0 == 0 ? 0 : -S,
                                int(min(a.n - tile0, 1LL << 30))};
            int done = 0;
            do {
                const int i = done + lane;
                uint32_t e0 = 0, cnt = 0, win = 0, off = 0;
                if (i < int(qn)) {
                    win = q32[i];
                    off = q16[i];
                    const uint32_t h = QW == 0 ? win * K0 : win;
                    uint32_t bk;
                    if (RANK) {
                        const uint32_t b = h >> a.fshift;
                        bk = s_rank[b >> 5] + __popc(s_filter[b >> 5] & ~(kFull << (b & 31u)));
                    } else {
                        bk = h >> a.bshift;
                    }
                    e0 = bucket_entries<RANK>(a.dir, bk, h >> (a.bshift - 8), cnt);
                }
                done += 32;
                verify_batch<QW != 0>(view, e0, cnt, win, int(off), [&](bool ok, const uint4 &en, int pos) {
                    const uint32_t bal = __ballot_sync(kFull, ok);
                    if (ok) {
                        uint32_t mult = 1u;
                        if (a.hist_smem) atomicAdd(&s_hist[en.y], 1u);
                        if (en.w & 0x80000000u) {
                            const uint32_t gi = en.w & 0x7FFFFFFFu;
                            const uint32_t j0 = __ldg(a.grp_off + gi), j1 = __ldg(a.grp_off + gi + 1);
                            mult = j1 - j0;
                            if (!a.hist_smem)
                                for (uint32_t j = j0; j < j1; ++j)
                                    atomicAdd(reinterpret_cast<unsigned long long *>(a.counts) + __ldg(a.grp_ids + j),
                                              1ull);
                        } else if (!a.hist_smem) {
                            atomicAdd(reinterpret_cast<unsigned long long *>(a.counts) + en.w, 1ull);
                        }
                        outs += mult;
                        if (a.list) {
                            // start in the tile, shifted by S - 1 so that it is never negative
                            const uint32_t o = uint32_t(pos + (S - 1)) - (en.z & 255u), code = en.w;
                            const long long p = (long long)st * a.slot_stride + (ent + __popc(bal & lt));
                            if (a.slot_kind == 0)
                                static_cast<uint32_t *>(a.slots)[p] =
                                    (o << 16) | ((code >> 16) & 0x8000u) | (code & 0x7FFFu);
                            else if (a.slot_kind == 1)
                                static_cast<unsigned long long *>(a.slots)[p] = ((unsigned long long)o << 32) | code;
                            else
                                static_cast<uint32_t *>(a.slots)[p] = (o << 20) | code;
                        }
                    }
                    ent += __popc(bal);
                });
            } while (int(qn) - done >= 32 || (last && int(qn) - done > 0));
            // the rest (fewer than 32) moves to the front
            const int left = max(int(qn) - done, 0);
            uint32_t h = 0, o = 0;
            if (lane < left) {
                h = q32[done + lane];
                o = q16[done + lane];
            }
            __syncwarp();
            if (lane < left) {
                q32[lane] = h;
                q16[lane] = uint16_t(o);
            }
            __syncwarp();
            qn = uint32_t(left);
        }
        if (last) {
            if (a.list) {
                uint32_t o_tot = outs;
                if (ent != 0u) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) o_tot += __shfl_xor_sync(kFull, o_tot, o);
                }
                if (lane == 0) {
                    a.tile_ent[st] = ent;
                    a.tile_out[st] = o_tot;
                    if (o_tot) atomicAdd(&a.seg_sum[st / uint32_t(a.seg_tiles)], (unsigned long long)o_tot);
                }
            } else {
                my_total += outs;
            }
            ent = 0;
            outs = 0;
        }
        st = stn;
        g = gn;
    }

    if (!a.list) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) my_total += __shfl_down_sync(kFull, my_total, o);
        if (lane == 0 && my_total) atomicAdd(reinterpret_cast<unsigned long long *>(a.n_occ), my_total);
    }
    if (!a.hist_smem) return;
    __syncthreads();
    for (int c = threadIdx.x; c < a.ncodes; c += blockDim.x) {
        const uint32_t x = s_hist[c];
        if (!x) continue;
        const uint32_t code = __ldg(a.code + c);
        if (code & 0x80000000u) {
            const uint32_t gi = code & 0x7FFFFFFFu;
            for (uint32_t j = a.grp_off[gi]; j < a.grp_off[gi + 1]; ++j)
                atomicAdd(reinterpret_cast<unsigned long long *>(a.counts) + a.grp_ids[j], (unsigned long long)x);
        } else {
            atomicAdd(reinterpret_cast<unsigned long long *>(a.counts) + code, (unsigned long long)x);
        }
    }
}

// ---------------------------------------------------------------------------
// Dense form: one-length sets whose m-gram is looked up at every position (s =
// 1, q = m <= 9), where a gram in the table is a match unless a byte outside
// the alphabet hides in it. There are no buckets and no pattern bytes: the
// gram's rank in the filter is the distinct pattern's number, and the window
// is compared with the gram spelled out in letters.
//
// What bounds it is instruction issue, then the shared-memory pipe (32 random
// words cost about 3.5 wavefronts), so PAIR takes two positions per lookup: a
// word of the pair table, picked by the characters 2 .. m of an (m + 1)-gram,
// holds for each pair of first characters whether the two m-grams in it are in
// the set. 64 KB at m = 8; longer grams test the filter's bits. 1 GiB of
// EST-shaped text, 8,000 8-mers (one position in nine matches), list mode: 1.12
// ms, with the transition table 1.38, with sampled grams 2.29; 128 MiB, 1,000
// 8-mers (PFAC): 80 us, sampled 185. 256 MiB of the first: 73 % of the issue
// slots and 78 % of the shared-memory and L1 pipe in use.
// ---------------------------------------------------------------------------
struct DenseArgs {
    GramArgs a;
    int pwords;                   // pair table words, 4^(m - 1)
    uint32_t pmask;               // (pwords - 1) * 4
    uint32_t gmask;               // 4^m - 1
    int m;
    const uint16_t *id_off, *ids; // each distinct pattern's ids
};

constexpr int kDenseQueue = 32 + 2 * kRow;   // queue entries: two rows, and a rest of fewer than 32

// MW: words of a window (m <= 4 MW)
template <bool PAIR, int MW>
__global__ void __launch_bounds__(kMaxWarps * 32, 1) gram_dense_kernel(const DenseArgs da)
{
    const GramArgs &a = da.a;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;

    uint32_t *s_pair = reinterpret_cast<uint32_t *>(smem);
    uint2 *s_mr = reinterpret_cast<uint2 *>(s_pair + (PAIR ? da.pwords : 0));   // filter word, rank
    uint32_t *s_hist = reinterpret_cast<uint32_t *>(s_mr + a.fwords);
    uint32_t *s_exp = s_hist + a.ncodes;                                        // four characters spelled out
    uint16_t *q16 = reinterpret_cast<uint16_t *>(s_exp + 256) + warp * kDenseQueue;
    uint8_t *s_ext = reinterpret_cast<uint8_t *>(q16 + (nwarps - warp) * kDenseQueue);  // min(keys - 1, 3)

    for (int i = threadIdx.x; i < a.fwords; i += blockDim.x)
        s_mr[i] = make_uint2(__ldg(a.filter_g + i), __ldg(a.rank_g + i));
    for (int i = threadIdx.x; i < a.ncodes; i += blockDim.x) {
        s_hist[i] = 0u;
        s_ext[i] = uint8_t(min(int(__ldg(da.id_off + i + 1)) - int(__ldg(da.id_off + i)) - 1, 3));
    }
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        uint32_t x = 0;
        for (int j = 0; j < 4; ++j) x |= ((a.lut >> (8 * ((i >> (2 * j)) & 3))) & 0xFFu) << (8 * j);
        s_exp[i] = x;
    }
    __syncthreads();
    if (PAIR) {
        // Word w, bits 2p and 2p + 1: the (m + 1)-gram x = 16 w + p starts with
        // the m-gram x mod 4^m and ends with x / 4, so the word interleaves 16
        // filter bits with 4 others, each of them four times.
        for (int i = threadIdx.x; i < da.pwords; i += blockDim.x) {
            const uint32_t b = (uint32_t(i) << 4) & da.gmask;
            uint32_t f = (s_mr[b >> 5].x >> (b & 16u)) & 0xFFFFu;
            f = (f | f << 8) & 0x00FF00FFu;
            f = (f | f << 4) & 0x0F0F0F0Fu;
            f = (f | f << 2) & 0x33333333u;
            f = (f | f << 1) & 0x55555555u;
            const uint32_t e = uint32_t(i) << 2, n = s_mr[e >> 5].x >> (e & 31u);
            s_pair[i] = f | ((n & 1u) | (n & 2u) << 7 | (n & 4u) << 14 | (n & 8u) << 21) * 0xAAu;
        }
        __syncthreads();
    }
    // no grid_trigger: expand CTAs that start while scan CTAs still run crowd on
    // the SMs that finish first (1.24 ms per GiB in place of 1.13)
    dev::grid_wait();   // the zeroed counts and sums

    // A warp takes a run of consecutive tiles, so that a row's characters
    // after the last lane are the next row's, packed once.
    const int m = da.m;
    const uint32_t gmask = da.gmask, pmask = da.pmask;
    const uint32_t tail = (m & 3) ? (1u << (8 * (m & 3))) - 1u : 0xFFFFFFFFu;  // bytes of the last word compared
    const uint32_t W = gridDim.x * nwarps, w = blockIdx.x * nwarps + warp;
    const uint32_t ntiles = uint32_t(a.ntiles), each = ntiles / W, extra = ntiles % W;
    uint32_t st = w * each + min(w, extra);
    const uint32_t st_end = st + each + (w < extra ? 1u : 0u);
    const uint32_t nrows = uint32_t(a.tile) / kRow;          // even
    const uint32_t nfull = a.aligned ? uint32_t(a.n / kRow) : 0u;   // rows wholly inside an aligned text
    unsigned long long my_total = 0;

    auto load = [&](uint32_t row) -> uint4 {
        if (row < nfull) return __ldg(reinterpret_cast<const uint4 *>(a.text + (long long)row * kRow) + lane);
        return load16(a.text, a.n, a.aligned, (long long)row * kRow + lane * 16);
    };
    // a bit per position whose m-gram is in the set: position k at bit 31 - k
    auto probe = [&](uint32_t lo, uint32_t hi) -> uint32_t {
        uint32_t mask = 0;
        if (PAIR) {
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const uint32_t at = __funnelshift_r(lo, hi, 2 * k + 2) & pmask;
                const uint32_t e = *reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(s_pair) + at);
                const uint32_t win = k == 0 ? lo : __funnelshift_r(lo, hi, 2 * k);
                mask = __funnelshift_r(mask, __funnelshift_r(e, 0u, win << 1), 2);  // bits 2 (win mod 16) and + 1
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const uint32_t win = k == 0 ? lo : __funnelshift_r(lo, hi, 2 * k);
                const uint32_t e = s_mr[(win & gmask) >> 5].x;
                mask = __funnelshift_r(mask, __funnelshift_r(e, 0u, win), 1);
            }
        }
        return __brev(mask & 0xFFFF0000u) << 16;
    };

    uint32_t c0 = 0;
    uint4 v1, v2;
    uint32_t row = st * nrows;
    if (st < st_end) {
        c0 = pack16(load(row));
        v1 = load(row + 1);
        v2 = load(row + 2);
    }
    uint32_t r = 0, ent = 0, outs = 0;
    int qn = 0;
    while (st < st_end) {
        const uint32_t c1 = pack16(v1), c2 = pack16(v2);
        const bool last = r + 2 == nrows;
        if (!last || st + 1 < st_end) {
            v1 = load(row + 3);
            v2 = load(row + 4);
        }
        const uint32_t h0 = __shfl_sync(kFull, lane == 0 ? c1 : c0, (lane + 1) & 31);
        const uint32_t h1 = __shfl_sync(kFull, lane == 0 ? c2 : c1, (lane + 1) & 31);
        uint32_t m0 = probe(c0, h0), m1 = probe(c1, h1);
        c0 = c2;

        // ---- hits -> queue (offsets in the tile), lane by lane: both rows'
        // counts in one scan ----
        {
            uint32_t cnt = __popc(m0) | __popc(m1) << 16;
            uint32_t inc = dev::warp_incl_scan(cnt, lane), tot = __shfl_sync(kFull, inc, 31);
            if ((tot & 0xFFFFu) == uint32_t(kRow)) {   // (see letter_probes)
                const long long base = (long long)row * kRow + lane * 16;
                m0 &= __brev(letter_probes<1>(a.text, a.n, base, a.lut));
                m1 &= __brev(letter_probes<1>(a.text, a.n, base + kRow, a.lut));
                cnt = __popc(m0) | __popc(m1) << 16;
                inc = dev::warp_incl_scan(cnt, lane);
                tot = __shfl_sync(kFull, inc, 31);
            }
            uint32_t at = uint32_t(qn) + ((inc - cnt) & 0xFFFFu);
            uint32_t off = r * kRow + uint32_t(lane) * 16u;
            while (m0) {
                const uint32_t k = __clz(int(m0));
                m0 &= 0x7FFFFFFFu >> k;
                q16[at++] = uint16_t(off + k);
            }
            at = uint32_t(qn) + (tot & 0xFFFFu) + ((inc - cnt) >> 16);
            off += kRow;
            while (m1) {
                const uint32_t k = __clz(int(m1));
                m1 &= 0x7FFFFFFFu >> k;
                q16[at++] = uint16_t(off + k);
            }
            qn += int(tot & 0xFFFFu) + int(tot >> 16);
            __syncwarp();
        }
        // ---- full batches of 32 (at the tile's end the rest too) ----
        if (qn >= 32 || (last && qn > 0)) {
            const long long tile0 = (long long)st * a.tile;
            const uint8_t *tp = a.text + tile0;
            uint32_t *dst = static_cast<uint32_t *>(a.slots) + (long long)st * a.slot_stride;
            // offsets whose words (up to three after the first) lie inside an aligned text
            const int safe = a.aligned ? int(min(a.n - tile0, 1LL << 30)) - 16 : -1;
            const int fits = int(min(a.n - tile0, 1LL << 30)) - m;
            int done = 0;
            do {
                const bool in = done + lane < qn;
                const int off = in ? int(q16[done + lane]) : 0;
                done += 32;
                bool ok = in;
                uint32_t gram;
                if (off <= safe) {
                    const uint32_t *wp = reinterpret_cast<const uint32_t *>(tp) + (off >> 2);
                    const uint32_t sh = uint32_t(off) * 8u;   // the funnel shift takes it modulo 32
                    uint32_t y[3], p[3];
                    uint32_t cur = __ldg(wp);
#pragma unroll
                    for (int j = 0; j < MW; ++j) {
                        const uint32_t nxt = __ldg(wp + j + 1);
                        y[j] = __funnelshift_r(cur, nxt, sh);
                        p[j] = (y[j] & 0x06060606u) * 0x00820820u;   // four codes in the top byte (pack16)
                        y[j] ^= s_exp[p[j] >> 24];
                        cur = nxt;
                    }
                    y[MW - 1] &= tail;
                    gram = MW == 1 ? p[0] >> 24 : __byte_perm(p[0], p[1], 0x0073) & 0xFFFFu;
                    if (MW == 3) gram |= (p[2] >> 24) << 16;
                    ok = ok && (MW == 1 ? y[0] : MW == 2 ? y[0] | y[1] : y[0] | y[1] | y[2]) == 0u;
                } else {
                    gram = 0u;
                    ok = ok && off <= fits;
                    for (int j = 0; ok && j < m; ++j) {
                        const uint32_t b = tp[off + j], c = (b >> 1) & 3u;
                        ok = b == ((a.lut >> (8 * c)) & 0xFFu);
                        gram |= c << (2 * j);
                    }
                }
                gram &= gmask;
                const uint2 mr = s_mr[gram >> 5];
                const uint32_t c = mr.y + __popc(mr.x & ~(kFull << (gram & 31u)));
                const uint32_t bal = __ballot_sync(kFull, ok);
                if (ok) {
                    const uint32_t ext = s_ext[c];
                    atomicAdd(&s_hist[c], 1u);
                    outs += ext + 1u;
                    if (ext == 3u) outs += uint32_t(__ldg(da.id_off + c + 1) - __ldg(da.id_off + c)) - 4u;
                    if (a.list) dst[ent + __popc(bal & lt)] = uint32_t(off) << 18 | ext << 16 | c;
                }
                ent += __popc(bal);
            } while (qn - done >= 32 || (last && qn > done));
            const int left = max(qn - done, 0);
            const uint32_t q = lane < left ? q16[done + lane] : 0u;
            __syncwarp();
            if (lane < left) q16[lane] = uint16_t(q);
            __syncwarp();
            qn = left;
        }
        row += 2;
        r += 2;
        if (last) {
            if (a.list) {
                uint32_t o_tot = outs;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) o_tot += __shfl_xor_sync(kFull, o_tot, o);
                if (lane == 0) {
                    a.tile_ent[st] = ent;
                    a.tile_out[st] = o_tot;
                    if (o_tot) atomicAdd(&a.seg_sum[st / uint32_t(a.seg_tiles)], (unsigned long long)o_tot);
                }
            } else {
                my_total += outs;
            }
            ent = 0;
            outs = 0;
            r = 0;
            ++st;
        }
    }

    if (!a.list) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) my_total += __shfl_down_sync(kFull, my_total, o);
        if (lane == 0 && my_total) atomicAdd(reinterpret_cast<unsigned long long *>(a.n_occ), my_total);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < a.ncodes; c += blockDim.x) {
        const uint32_t x = s_hist[c];
        if (!x) continue;
        const uint32_t j1 = __ldg(da.id_off + c + 1);
        for (uint32_t j = __ldg(da.id_off + c); j < j1; ++j)
            atomicAdd(reinterpret_cast<unsigned long long *>(a.counts) + __ldg(da.ids + j), (unsigned long long)x);
    }
}

// ---------------------------------------------------------------------------
// Keys of the dense form. An entry is (start in the tile << 18) | (min(keys -
// 1, 3) << 16) | distinct pattern; id_off / ids list each distinct pattern's
// ids. CTA b owns segment b's tiles, a warp takes a tile in rows of 32 entries,
// eight rows loaded together and the next eight in flight. A key's place in a
// row comes from two ballots of the entries' key counts, so the tables are read
// for the ids only; the row is issue-bound, and looking the counts up (as the
// expand kernel of the other scans does) took twice the instructions.
// ---------------------------------------------------------------------------
constexpr int kDenseExpandThreads = 512;

template <bool SM>
__global__ void __launch_bounds__(kDenseExpandThreads)
dense_expand_kernel(const uint32_t *slots, const uint32_t *tile_ent, const uint32_t *tile_out,
                    const unsigned long long *seg_sum, long long seg_tiles, long long ntiles, uint32_t tile,
                    const uint16_t *__restrict__ id_off, const uint16_t *__restrict__ ids, int nc, int d,
                    unsigned long long *__restrict__ occ, long long occ_cap, long long *n_occ,
                    const unsigned long long *occ_base, unsigned long long pos_base)
{
    constexpr int T = kDenseExpandThreads, NW = T / 32, R = 8;
    extern __shared__ __align__(16) unsigned char esm[];
    unsigned long long *s_off = reinterpret_cast<unsigned long long *>(esm);
    uint32_t *s_ent = reinterpret_cast<uint32_t *>(s_off + seg_tiles);
    uint16_t *s_io = reinterpret_cast<uint16_t *>(s_ent + seg_tiles), *s_id = s_io + nc + 1;
    __shared__ unsigned long long s_red[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const long long t0 = (long long)blockIdx.x * seg_tiles;
    const int nt = int(max(0LL, min(seg_tiles, ntiles - t0)));
    if (nt == 0) return;
    if (SM) {
        for (int i = tid; i <= nc; i += T) s_io[i] = __ldg(id_off + i);
        for (int i = tid; i < d; i += T) s_id[i] = __ldg(ids + i);
    }
    dev::grid_wait();   // the scan's tiles and slots
    const unsigned long long run = dev::segment_offsets<T>(tile_ent, tile_out, seg_sum, blockIdx.x, t0, nt, occ_base,
                                                           tile, s_off, s_ent, s_red);
    if (tid == T - 1 && t0 + nt == ntiles) *n_occ = (long long)run;
    __syncthreads();
    auto first_of = [&](uint32_t c) -> uint32_t { return SM ? s_io[c] : __ldg(id_off + c); };
    auto id_at = [&](uint32_t j) -> uint32_t { return SM ? s_id[j] : __ldg(ids + j); };

    const unsigned long long cap = (unsigned long long)occ_cap;
    uint32_t x[R], y[R];
    auto load = [&](uint32_t (&z)[R], int q, uint32_t g) {
        const uint32_t ent = s_ent[q];
        const uint32_t *src = slots + (t0 + q) * tile + g + lane;
#pragma unroll
        for (int u = 0; u < R; ++u) z[u] = g + u * 32 + lane < ent ? __ldcs(src + u * 32) : 0u;
    };
    int q = warp;
    while (q < nt && s_ent[q] == 0) q += NW;
    uint32_t g = 0, pos = 0, room = 0;
    unsigned long long *out = occ;
    if (q < nt) load(x, q, 0);
    while (q < nt) {
        const uint32_t ent = s_ent[q];
        if (g == 0) {  // 32-bit key offsets from the tile's base, clipped to the capacity left after it
            const unsigned long long b = s_off[q];
            out = occ + b;
            room = b < cap ? uint32_t(min(cap - b, 0xFFFFFFFFull)) : 0u;
            pos = 0;
        }
        int qn = q;
        uint32_t gn = g + R * 32;
        if (gn >= ent) {
            gn = 0;
            do qn += NW;
            while (qn < nt && s_ent[qn] == 0);
        }
        if (qn < nt) load(y, qn, gn);
        const uint32_t tile0 = uint32_t(pos_base) + uint32_t(t0 + q) * tile;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const uint32_t row = g + u * 32;
            if (row >= ent) break;
            const uint32_t cnt = min(ent - row, 32u);
            const bool valid = uint32_t(lane) < cnt;
            const uint32_t v = x[u], c = v & 0xFFFFu;
            const uint32_t hi = tile0 + (v >> 18);
            const uint32_t e0 = __ballot_sync(kFull, v & 0x10000u), e1 = __ballot_sync(kFull, v & 0x20000u);
            const uint32_t j = first_of(c);
            if ((e0 & e1) == 0u) {
                const uint32_t o = pos + lane + __popc(e0 & lt) + 2u * __popc(e1 & lt);
                if (valid && o < room) out[o] = (unsigned long long)hi << 32 | id_at(j);
                if ((v & 0x30000u) && o + 1u < room) out[o + 1u] = (unsigned long long)hi << 32 | id_at(j + 1u);
                if ((v & 0x20000u) && o + 2u < room) out[o + 2u] = (unsigned long long)hi << 32 | id_at(j + 2u);
                pos += cnt + __popc(e0) + 2u * __popc(e1);
            } else {  // four or more equal patterns
                const uint32_t n = valid ? first_of(c + 1u) - j : 0u;
                const uint32_t inc = dev::warp_incl_scan(n, lane);
                const uint32_t o = pos + inc - n;
                for (uint32_t k = 0; k < n; ++k)
                    if (o + k < room) out[o + k] = (unsigned long long)hi << 32 | id_at(j + k);
                pos += __shfl_sync(kFull, inc, 31);
            }
        }
#pragma unroll
        for (int u = 0; u < R; ++u) x[u] = y[u];
        q = qn;
        g = gn;
    }
}

// shared memory of the dense form (mirrors the kernel's carve-up)
long long dense_smem(const GramTables &t, bool pair, int warps)
{
    const long long nc = (long long)t.code.size();
    return 4 * ((pair ? 1LL << (2 * (t.q - 1)) : 0) + 2 * (long long)t.filter.size() + nc + 256) +
           2 * (long long)warps * kDenseQueue + nc;
}

// Zeroes what a scan adds to: one launch in place of three memsets, which cost
// about 1.5 us each, and the scan kernel loads its tables meanwhile.
struct ZeroArgs {
    unsigned long long *p[3];
    long long n[3];               // 8-byte words
};

__global__ void __launch_bounds__(256) gram_zero_kernel(const ZeroArgs z, int64_t *n_occ)
{
    dev::grid_trigger();
    if (n_occ && blockIdx.x == 0 && threadIdx.x == 0) *n_occ = 0;
    for (int k = 0; k < 3; ++k)
        for (long long i = blockIdx.x * 256LL + threadIdx.x; i < z.n[k]; i += gridDim.x * 256LL) z.p[k][i] = 0ull;
}

typedef void (*DenseKernel)(const DenseArgs);

DenseKernel dense_kernel_of(const GramTables &t, bool pair)
{
    if (t.q <= 4) return pair ? gram_dense_kernel<true, 1> : gram_dense_kernel<false, 1>;
    if (t.q <= 8) return pair ? gram_dense_kernel<true, 2> : gram_dense_kernel<false, 2>;
    return gram_dense_kernel<false, 3>;
}

int dense_expand(const GramTables &t, const DevGram &dv, const GramArgs &a, const GramWs &ws, const DeviceProps &dp,
                 uint64_t *d_occ, int64_t occ_cap, int64_t *d_n_occ, const unsigned long long *occ_base,
                 unsigned long long pos_base, cudaStream_t st)
{
    const int nc = int(t.code.size());
    const long long base = a.seg_tiles * 12, tab = 2 * ((long long)nc + 1 + t.d);
    const long long per_cta = std::min<long long>((long long)dp.smem_per_sm / 2 - 2048, dp.smem_optin - 1024);
    const bool sm = base + tab <= per_cta;
    const long long smem = base + (sm ? tab : 0);
    const auto fn = sm ? dense_expand_kernel<true> : dense_expand_kernel<false>;
    const int rc = kernel_smem_attr(reinterpret_cast<const void *>(fn), smem);
    if (rc) return rc;
    const cudaError_t e = dev::launch_dependent(
        fn, dim3(unsigned((a.ntiles + a.seg_tiles - 1) / a.seg_tiles)), dim3(kDenseExpandThreads), size_t(smem), st,
        static_cast<const uint32_t *>(ws.slots), ws.tile_ent, ws.tile_out, ws.seg_sum, a.seg_tiles, a.ntiles,
        uint32_t(a.tile), dv.id_off, dv.ids, nc, int(t.d), reinterpret_cast<unsigned long long *>(d_occ),
        (long long)(d_occ ? occ_cap : 0), reinterpret_cast<long long *>(d_n_occ), occ_base, pos_base);
    if (e != cudaSuccess) { set_cuda_error(int(e)); return PM_ECUDA; }
    return PM_OK;
}

typedef void (*GramKernel)(const GramArgs);

inline long long up4w(long long x) { return (x + 3) & ~3LL; }

template <int QW, bool RANK, bool RUNS>
GramKernel by_stride(int s)
{
    switch (s) {
    case 1: return gram_scan_kernel<1, QW, RANK, RUNS>;
    case 2: return gram_scan_kernel<2, QW, RANK, RUNS>;
    case 4: return gram_scan_kernel<4, QW, RANK, RUNS>;
    case 8: return gram_scan_kernel<8, QW, RANK, RUNS>;
    default: return gram_scan_kernel<16, QW, RANK, RUNS>;
    }
}

GramKernel kernel_of(const GramTables &t)
{
    switch (t.qw) {
    case 0:
        if (t.runs) return t.rank ? by_stride<0, true, true>(t.s) : by_stride<0, false, true>(t.s);
        return t.rank ? by_stride<0, true, false>(t.s) : by_stride<0, false, false>(t.s);
    case 1: return by_stride<1, false, false>(t.s);
    case 2: return by_stride<2, false, false>(t.s);
    case 3: return by_stride<3, false, false>(t.s);
    default: return by_stride<4, false, false>(t.s);
    }
}

long long table_words(const GramTables &t)
{
    return up4w((long long)t.filter.size()) * (t.rank ? 2 : 1);
}

long long queue_words(const GramTables &t) { return qcap(t.s) + qcap(t.s) / 2; }

}  // namespace

int gram_plan(const GramTables &t, const DeviceProps &dp, DevGram &dev)
{
    dev.use = false;
    if (!t.ok) return PM_OK;
    const long long budget = (long long)dp.smem_optin - 1024;
    const long long nc = (long long)t.code.size();
    if (t.dense) {
        for (int w : {32, 28, 24, 20, 16})
            for (bool pair : {true, false}) {
                if ((pair && t.q > 8) || dense_smem(t, pair, w) > budget) continue;
                dev.warps = w;
                dev.hist_smem = 1;
                dev.pair = pair ? 1 : 0;
                dev.use = true;
                return PM_OK;
            }
        return PM_OK;
    }
    // counters in shared memory if they fit beside 24 warps' queues
    for (int hist : {1, 0})
        for (int w : {32, 24, 16}) {
            const long long need = 4 * (table_words(t) + (hist ? up4w(nc) : 0) + w * queue_words(t));
            if (need > budget || (hist && w < 24)) continue;
            dev.warps = w;
            dev.hist_smem = hist;
            dev.use = true;
            return PM_OK;
        }
    return PM_OK;
}

int gram_slot_bytes(const GramTables &t)
{
    if (t.var) return t.d <= (1 << 20) ? 4 : 8;
    return t.d < 32768 ? 4 : 8;
}

int gram_launch(const GramTables &t, const DevGram &dv, const uint8_t *d_text, int64_t n, bool list,
                int64_t *d_counts, uint64_t *d_occ, int64_t occ_cap, int64_t *d_n_occ, const GramWs &ws,
                const unsigned long long *occ_base, unsigned long long pos_base, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    DeviceProps dp;
    int rc = device_props(dp);
    if (rc) return rc;
    GramArgs a;
    a.text = d_text;
    a.n = n;
    a.aligned = (reinterpret_cast<uintptr_t>(d_text) & 15) == 0;
    for (int j = 0; j < 4; ++j) a.K[j] = t.K[j];
    a.lut = t.lut;
    a.fshift = 32 - t.fb;
    a.wshift = 37 - t.fb;
    a.bshift = 32 - t.db;
    a.fwords = int(t.filter.size());
    a.filter_g = dv.filter;
    a.rank_g = dv.rank_base;
    a.dir = reinterpret_cast<const uint2 *>(dv.dir);
    a.ent = static_cast<const uint4 *>(dv.ent);
    a.pats = dv.pats;
    a.pw = t.pw;
    a.code = dv.code;
    a.grp_off = dv.grp_off;
    a.grp_ids = dv.grp_ids;
    a.ncodes = int(t.code.size());
    a.list = list ? 1 : 0;
    a.hist_smem = dv.hist_smem;
    a.counts = reinterpret_cast<long long *>(d_counts);
    a.n_occ = reinterpret_cast<long long *>(d_n_occ);
    // Tiles: long ones waste fewer lanes on a tile's last batch (about as much as
    // 500 more bytes), short ones spread a short text over the SMs, and their
    // number has to fill whole rounds of all warps: 128 MiB in 8 KiB tiles took
    // four rounds for 3.4 rounds' work (1,000 8-mers as PFAC: 84 us). The
    // workspace holds one count per kWarpTile bytes, so a tile is longer than
    // that; the slots of a mixed set of 2^15 patterns or more have 12 bits for
    // the start, a dense slot 14.
    int warps = dv.warps;
    const long long lanes = (long long)dp.sm_count * warps;
    const int step = t.dense ? 2 * kRow : rows_of(t.s) * kRow;
    const int most = t.var && t.d >= 32768 ? 4096 : t.dense ? 8192 : 16384;
    static_assert(min_tile(1) >= kWarpTile && min_tile(8) >= kWarpTile, "one count per kWarpTile bytes");
    int tile = min_tile(t.s);
    double best = 0.0;
    for (int x = tile; x <= most; x += step) {
        const long long tiles = (n + x - 1) / x, rounds = (tiles + lanes - 1) / lanes;
        const double score = double(n) / (double(rounds) * double(lanes) * (x + 500));
        if (score > best) {
            best = score;
            tile = x;
        }
    }
    a.tile = tile;
    a.ntiles = (n + tile - 1) / tile;
    const int per_pos = t.var ? ws.per_pos : 1;
    const int se = gram_slot_bytes(t);
    a.slot_kind = se == 8 ? 1 : t.var && t.d >= 32768 ? 2 : 0;
    a.slot_stride = (long long)tile * per_pos;
    a.slots = ws.slots;
    a.tile_ent = ws.tile_ent;
    a.tile_out = ws.tile_out;
    a.seg_sum = ws.seg_sum;
    a.seg_tiles = (a.ntiles + ws.segs - 1) / ws.segs;

    // a short text: fewer warps per CTA, spread over every SM (at least 8,
    // which load the tables)
    const long long spread = (a.ntiles + dp.sm_count - 1) / dp.sm_count;
    if (spread < warps) warps = int(spread < 8 ? 8 : spread);
    long long grid = dp.sm_count;
    const long long want = (a.ntiles + warps - 1) / warps;
    if (want < grid) grid = want;
    const dim3 gd{unsigned(grid)}, bd{unsigned(warps * 32)};
    cudaError_t e = cudaSuccess;
    if (t.dense) {
        DenseArgs da;
        da.a = a;
        // a short text does not repay the pair table (1,000 8-mers, 4 MiB: 18.9 us
        // without it, 23.3 with; 8 MiB 22.5 with)
        const bool pair = dv.pair && n >= (int64_t(8) << 20);
        da.pwords = 1 << (2 * (t.q - 1));
        da.pmask = uint32_t(da.pwords - 1) * 4u;
        da.gmask = (1u << (2 * t.q)) - 1u;
        da.m = t.q;
        da.id_off = dv.id_off;
        da.ids = dv.ids;
        const long long smem = dense_smem(t, pair, warps);
        const DenseKernel fn = dense_kernel_of(t, pair);
        rc = kernel_smem_attr(reinterpret_cast<const void *>(fn), smem);
        if (rc) return rc;
        e = dev::launch_dependent(fn, gd, bd, size_t(smem), st, da);
    } else {
        const GramKernel fn = kernel_of(t);
        const long long smem =
            4 * (table_words(t) + (dv.hist_smem ? up4w(a.ncodes) : 0) + (long long)warps * queue_words(t));
        rc = kernel_smem_attr(reinterpret_cast<const void *>(fn), smem);
        if (rc) return rc;
        e = dev::launch_dependent(fn, gd, bd, size_t(smem), st, a);
    }
    if (e != cudaSuccess) { set_cuda_error(int(e)); cudaGetLastError(); return PM_ECUDA; }
    if (!list) return PM_OK;
    if (t.dense) return dense_expand(t, dv, a, ws, dp, d_occ, occ_cap, d_n_occ, occ_base, pos_base, st);
    ExpandTiles tl;
    tl.tile = tile;
    tl.slot_stride = a.slot_stride;
    tl.ntiles = a.ntiles;
    tl.seg_tiles = a.seg_tiles;
    tl.slot_kind = a.slot_kind;
    tl.slots = ws.slots;
    tl.tile_ent = ws.tile_ent;
    tl.tile_out = ws.tile_out;
    tl.seg_sum = ws.seg_sum;
    return expand_tiles_launch(tl, dv.grp_off, dv.grp_ids, (int64_t)t.grp_off.size(), (int64_t)t.grp_ids.size(),
                               d_occ, occ_cap, d_n_occ, occ_base, pos_base - (unsigned long long)(t.s - 1), stream);
}

int gram_launch_ws(const GramTables &t, const DevGram &dv, const uint8_t *d_text, int64_t n, bool list,
                   int64_t *d_counts, uint64_t *d_occ, int64_t occ_cap, int64_t *d_n_occ, void *d_ws,
                   int64_t nterms, int slot_bytes, int per_pos, bool first, const unsigned long long *occ_base,
                   unsigned long long pos_base, void *stream)
{
    ListParts L;
    list_workspace_parts(d_ws, warp_tiles(n), nterms, slot_bytes, L);
    GramWs ws;
    ws.tile_ent = L.tile_ent;
    ws.tile_out = L.tile_out;
    ws.seg_sum = L.seg_sum;
    ws.slots = L.slots;
    ws.segs = L.segs;
    ws.per_pos = per_pos;
    ZeroArgs z{};
    if (list) {
        z.p[0] = L.seg_sum;
        z.n[0] = (static_cast<char *>(d_ws) + L.zeroed_bytes - reinterpret_cast<char *>(L.seg_sum)) / 8;
    }
    if (first) {
        z.p[1] = reinterpret_cast<unsigned long long *>(d_counts);
        z.n[1] = t.d;
        z.p[2] = static_cast<unsigned long long *>(d_ws);
        z.n[2] = kWsHeader / 8;
    }
    const long long words = std::max<long long>(z.n[0] + z.n[1] + z.n[2], 1);
    gram_zero_kernel<<<unsigned(std::min<long long>((words + 255) / 256, 1024)), 256, 0,
                       static_cast<cudaStream_t>(stream)>>>(z, first ? d_n_occ : nullptr);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_cuda_error(int(e)); return PM_ECUDA; }
    return gram_launch(t, dv, d_text, n, list, d_counts, d_occ, occ_cap, d_n_occ, ws, occ_base, pos_base, stream);
}

}  // namespace pm
