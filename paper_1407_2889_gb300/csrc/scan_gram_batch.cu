// scan_gram_batch.cu -- sampled-gram scans (gram.cpp, scan_gram.cu) of many
// independent instances in one persistent launch: the batched form for sets
// that take the gram scan, beside the transition-table kernel of
// scan_batch.cu, whose queue, splitting of large instances and workspace it
// shares.
//
// A CTA loads the instance's filter (and its counters, when they fit) into
// shared memory; its warps take tiles of the item in rounds. A warp keeps the
// tile's matches (start, code) until a prefix over the warps' totals gives
// their place, then writes the keys. A tile with more matches than its buffer
// holds is scanned once more, writing as it goes: the planner sizes tiles so
// that this is rare.
//
// Against walking the transition tables this removes the per-character
// lookups, many of which read table rows past the shared-memory prefix from L2
// or DRAM: 1,024 instances (0.58 GB of text, 10 to 10,000 patterns each) took
// 2.87 ms, and take 0.43. What is left is latency: warps wait at the round's
// barrier and for the entries and patterns of candidates, which nothing has
// brought into L2 (issue slots 29 % in use).
#include <algorithm>
#include <cmath>

#include "gram_device.cuh"
#include "scan_gram_batch.cuh"

namespace pm {
namespace {

using dev::kFull;
using namespace gramdev;

// Most walks spill at 24 warps (80 registers; 8 to 220 bytes by ptxas, stride 16
// most), more at 32 (64 registers): 570 us for the batch above against 502.
constexpr int kWarps = 24;
constexpr int kHits = 192;           // matches a warp keeps per tile
constexpr int kMaxTile = 32768;      // a match's offset has 16 bits

// rows per load batch, and a warp's queue
__host__ __device__ constexpr int brows(int s) { return s >= 8 ? 2 : 1; }
__host__ __device__ constexpr int bqueue(int s) { return 32 + brows(s) * kRow / s; }
// bytes: queue (hash, offset), matches (code, offset)
__host__ __device__ constexpr int bwarp_bytes(int s) { return (bqueue(s) + kHits) * 6; }

template <int S, bool RANK>
__device__ __noinline__ void run_gram(const BatchArgs &a, const BatchDesc &D, unsigned char *smem,
                                      unsigned long long *s_tot)
{
    constexpr int NP = 16 / S, R = brows(S), Q = bqueue(S);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint8_t *text = a.text + D.text_off;
    const long long n = D.n;
    const bool aligned = (reinterpret_cast<uintptr_t>(text) & 15) == 0;

    uint32_t *q32 = reinterpret_cast<uint32_t *>(smem) + warp * (Q + kHits);
    uint32_t *h32 = q32 + Q;
    uint16_t *q16 = reinterpret_cast<uint16_t *>(smem + kWarps * (Q + kHits) * 4) + warp * (Q + kHits);
    uint16_t *h16 = q16 + Q;
    uint32_t *s_filter = reinterpret_cast<uint32_t *>(smem + rr16(kWarps * bwarp_bytes(S)));
    uint32_t *s_rank = s_filter + D.g_fwords;
    uint32_t *s_hist = D.hist_off >= 0 ? s_filter + D.hist_off / 4 : nullptr;
    unsigned long long *g_hist = a.ccount + D.ccount_off;
    // a short item probes the filter where it is: loading it takes longer
    const uint32_t *filter = D.g_direct ? D.g_filter : s_filter;
    const uint32_t *rank = D.g_direct ? D.g_rank_base : s_rank;
    if (!D.g_direct) {
        const uint4 *src = reinterpret_cast<const uint4 *>(D.g_filter);
        uint4 *dst = reinterpret_cast<uint4 *>(s_filter);
        const int nv = D.g_fwords / 4;
#pragma unroll 4
        for (int i = threadIdx.x; i < nv; i += kWarps * 32) dst[i] = __ldg(src + i);
        if (RANK) {
            const uint4 *rs = reinterpret_cast<const uint4 *>(D.g_rank_base);
            uint4 *rd = reinterpret_cast<uint4 *>(s_rank);
#pragma unroll 4
            for (int i = threadIdx.x; i < nv; i += kWarps * 32) rd[i] = __ldg(rs + i);
        }
    }
    if (s_hist)
        for (int i = threadIdx.x; i < D.nterms; i += blockDim.x) s_hist[i] = 0u;
    __syncthreads();

    const uint32_t K0 = D.g_k;
    const uint4 *entries = static_cast<const uint4 *>(D.g_ent);
    unsigned long long *odst = a.occ + D.occ_off;
    unsigned long long ocap = (unsigned long long)D.occ_cap;

    auto keys_of = [&](uint32_t code, uint32_t &j0) -> uint32_t {
        j0 = 0u;
        if (!(code & 0x80000000u)) return 1u;
        const uint32_t g = code & 0x7FFFFFFFu;
        j0 = __ldg(D.g_grp_off + g);
        return __ldg(D.g_grp_off + g + 1) - j0;
    };
    auto put = [&](unsigned long long at, uint32_t pos, uint32_t code, uint32_t j0, uint32_t keys) {
        for (uint32_t k = 0; k < keys; ++k) {
            const uint32_t r = (code & 0x80000000u) ? __ldg(D.g_grp_ids + j0 + k) : code;
            if (at + k < ocap) odst[at + k] = (unsigned long long)pos << 32 | r;
        }
    };
    // One scan of the tile at byte `lo` of the item (probes below `hi`).
    // direct false: matches to the warp's buffer (the first kHits), counted if
    // `count`; true: keys written from output offset `base` on. Returns the
    // warp's keys; ent: its matches.
    auto scan_tile = [&](long long lo, long long hi, bool count, bool direct, unsigned long long base,
                         uint32_t &ent) -> uint32_t {
        const uint8_t *tp = text + lo;
        const int rem = int(min(n - lo, 1LL << 30));
        const GramTile view{entries, D.g_pats, D.g_pw, tp, lo == 0 ? 0 : -S, rem};
        const int rows = int((hi - lo + kRow - 1) / kRow);
        uint32_t qn = 0, keys = 0;
        ent = 0;
        uint4 v[R + 1];
        auto load = [&](int off) {
            if (aligned && off + R * kRow + 16 <= rem) {
                const uint4 *p = reinterpret_cast<const uint4 *>(tp + off) + lane;
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = __ldg(p + 32 * r);
                if (lane == 0) v[R] = __ldg(p + 32 * R);
            } else {
#pragma unroll
                for (int r = 0; r <= R; ++r)
                    if (r < R || lane == 0) v[r] = load16<false>(text, n, aligned, lo + off + r * kRow + lane * 16);
            }
        };
        v[R] = make_uint4(0u, 0u, 0u, 0u);
        load(0);
        for (int r0 = 0; r0 < rows; r0 += R) {
            const int off = r0 * kRow;
            uint32_t c[R + 1];
#pragma unroll
            for (int r = 0; r <= R; ++r) c[r] = pack16(v[r]);
            uint32_t cl[R], ch[R], mask[R], any = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                cl[r] = c[r];
                ch[r] = __shfl_sync(kFull, lane == 0 ? c[r + 1] : c[r], (lane + 1) & 31);
                uint32_t m = 0;
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const uint32_t win = k == 0 ? cl[r] : __funnelshift_r(cl[r], ch[r], 2 * S * k);
                    const uint32_t w = filter[(win * K0) >> D.g_wshift];
                    m = __funnelshift_r(m, __funnelshift_r(w, 0u, win), 1);
                }
                mask[r] = r0 + r < rows ? m >> (32 - NP) : 0u;
                any |= mask[r];
            }
            if (r0 + R < rows) load(off + R * kRow);   // the next batch, while this one is looked at
            if (__any_sync(kFull, any != 0u)) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    uint32_t m = mask[r];
                    const uint32_t cnt = __popc(m), inc = dev::warp_incl_scan(cnt, lane);
                    uint32_t at = qn + inc - cnt;
                    qn += __shfl_sync(kFull, inc, 31);
                    const uint32_t o = uint32_t(off + r * kRow) + uint32_t(lane) * 16u;
                    while (m) {
                        const uint32_t k = uint32_t(__ffs(int(m))) - 1u;
                        m &= m - 1u;
                        q32[at] = __funnelshift_r(cl[r], ch[r], 2 * S * k);
                        q16[at++] = uint16_t(o + S * k);
                    }
                }
                __syncwarp();
            }
            const bool last = r0 + R >= rows;
            int done = 0;
            while (int(qn) - done >= 32 || (last && int(qn) > done)) {
                uint32_t win = 0, e0 = 0, cnt = 0;
                int pos = 0;
                if (done + lane < int(qn)) {
                    win = q32[done + lane];
                    pos = int(q16[done + lane]);
                    const uint32_t h = win * K0;
                    uint32_t bk;
                    if (RANK) {
                        const uint32_t b = h >> D.g_fshift;
                        bk = rank[b >> 5] + __popc(filter[b >> 5] & ~(kFull << (b & 31u)));
                    } else {
                        bk = h >> D.g_bshift;
                    }
                    e0 = bucket_entries<RANK>(reinterpret_cast<const uint2 *>(D.g_dir), bk, h >> (D.g_bshift - 8), cnt);
                }
                done += 32;
                verify_batch<false>(view, e0, cnt, win, pos, [&](bool ok, const uint4 &en, int p) {
                    const uint32_t bal = __ballot_sync(kFull, ok);
                    uint32_t j0 = 0, kk = 0;
                    if (ok) {
                        if (count) {
                            if (s_hist) atomicAdd(&s_hist[en.y], 1u);
                            else atomicAdd(&g_hist[en.y], 1ull);
                        }
                        kk = keys_of(en.w, j0);
                    }
                    const uint32_t start = uint32_t(p + (S - 1)) - (en.z & 255u);   // shifted, never negative
                    if (!direct) {
                        const uint32_t i = ent + __popc(bal & lt);
                        if (ok && i < uint32_t(kHits)) {
                            h32[i] = en.w;
                            h16[i] = uint16_t(start);
                        }
                    } else {
                        const uint32_t ik = dev::warp_incl_scan(kk, lane);
                        put(base + ik - kk, uint32_t(lo) + start - uint32_t(S - 1), en.w, j0, kk);
                        base += __shfl_sync(kFull, ik, 31);
                    }
                    ent += __popc(bal);
                    keys += kk;
                });
            }
            if (done) {
                const int left = max(int(qn) - done, 0);
                uint32_t h = 0, o = 0;
                __syncwarp();
                if (lane < left) {
                    h = q32[done + lane];
                    o = q16[done + lane];
                }
                __syncwarp();
                if (lane < left) {
                    q32[lane] = h;
                    q16[lane] = uint16_t(o);
                }
                qn = uint32_t(left);
                __syncwarp();
            }
        }
        return __reduce_add_sync(kFull, keys);
    };

    const long long t_lo = D.t_lo * kWarpTile, t_hi = min(D.t_hi * (long long)kWarpTile, n);
    auto pass = [&](bool count, bool write, unsigned long long base0) -> unsigned long long {
        const long long rounds = t_hi > t_lo ? (t_hi - t_lo + (long long)D.tile * kWarps - 1) / ((long long)D.tile * kWarps) : 0;
        unsigned long long running = base0, mine = 0;
        for (long long rd = 0; rd < rounds; ++rd) {
            const long long lo = t_lo + (rd * kWarps + warp) * D.tile, hi = min(lo + D.tile, t_hi);
            uint32_t ent = 0;
            const uint32_t keys = lo < hi ? scan_tile(lo, hi, count, false, 0ull, ent) : 0u;
            if (!write) {   // totals only: no round needs another warp's
                mine += keys;
                continue;
            }
            if (lane == 0) s_tot[warp] = keys;
            __syncthreads();
            const uint32_t tot = lane < kWarps ? uint32_t(s_tot[lane]) : 0u;
            const uint32_t inc = dev::warp_incl_scan(tot, lane);
            const uint32_t before = __shfl_sync(kFull, inc - tot, warp);
            const unsigned long long base = running + before;
            running += __shfl_sync(kFull, inc, 31);
            if (keys > 0) {
                if (ent <= uint32_t(kHits)) {
                    unsigned long long at = base;
                    for (uint32_t i = 0; i < ent; i += 32) {
                        const bool in = i + lane < ent;
                        const uint32_t code = in ? h32[i + lane] : 0u, start = in ? h16[i + lane] : 0u;
                        uint32_t j0 = 0;
                        const uint32_t kk = in ? keys_of(code, j0) : 0u, ik = dev::warp_incl_scan(kk, lane);
                        put(at + ik - kk, uint32_t(lo) + start - uint32_t(S - 1), code, j0, kk);
                        at += __shfl_sync(kFull, ik, 31);
                    }
                } else {
                    uint32_t again;
                    (void)scan_tile(lo, hi, false, true, base, again);
                }
            }
            __syncthreads();   // s_tot is rewritten next round
        }
        if (!write) {
            if (lane == 0) s_tot[warp] = mine;
            __syncthreads();
            for (int w = 0; w < kWarps; ++w) running += s_tot[w];
            __syncthreads();
        }
        return running - base0;
    };
    long long *cnt_out = a.counts + D.count_off;
    auto write_counts = [&](bool from_device) {
        for (int c = threadIdx.x; c < D.nterms; c += blockDim.x) {
            const long long v = from_device ? (long long)dev::ld_acquire(&g_hist[c]) : (long long)s_hist[c];
            const uint32_t code = __ldg(D.g_code + c);
            uint32_t j0;
            const uint32_t k = keys_of(code, j0);
            for (uint32_t j = 0; j < k; ++j) cnt_out[(code & 0x80000000u) ? __ldg(D.g_grp_ids + j0 + j) : code] = v;
        }
    };
    run_item(a, D, s_hist, g_hist, odst, ocap, pass, write_counts);
}

__global__ void __launch_bounds__(kWarps * 32, 1) gram_batch_kernel(const BatchArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_next;
    __shared__ unsigned long long s_tot[kWarps];
    __shared__ BatchDesc D;   // the item at hand
    while (true) {
        if (threadIdx.x == 0) {
            const unsigned long long j = atomicAdd(&a.ws->queue2, 1ull);
            s_next = j < (unsigned long long)a.k ? int(j) : -1;
        }
        __syncthreads();
        const int j = s_next;
        if (j < 0) break;
        static_assert(sizeof(BatchDesc) % 8 == 0, "copied in 8-byte words");
        if (threadIdx.x < sizeof(BatchDesc) / 8)
            reinterpret_cast<unsigned long long *>(&D)[threadIdx.x] =
                reinterpret_cast<const unsigned long long *>(a.desc + j)[threadIdx.x];
        __syncthreads();
        if (D.g_rank) {
            switch (D.g_s) {
            case 1: run_gram<1, true>(a, D, smem, s_tot); break;
            case 2: run_gram<2, true>(a, D, smem, s_tot); break;
            case 4: run_gram<4, true>(a, D, smem, s_tot); break;
            case 8: run_gram<8, true>(a, D, smem, s_tot); break;
            default: run_gram<16, true>(a, D, smem, s_tot);
            }
        } else {
            switch (D.g_s) {
            case 1: run_gram<1, false>(a, D, smem, s_tot); break;
            case 2: run_gram<2, false>(a, D, smem, s_tot); break;
            case 4: run_gram<4, false>(a, D, smem, s_tot); break;
            case 8: run_gram<8, false>(a, D, smem, s_tot); break;
            default: run_gram<16, false>(a, D, smem, s_tot);
            }
        }
    }
}

long long smem_budget()
{
    DeviceProps dp;
    return device_props(dp) ? 0 : gram_batch_smem(dp);
}

}  // namespace

long long gram_batch_smem(const DeviceProps &dp)
{
    return ((long long)dp.smem_optin - 2048) & ~15LL;   // static shared memory and slack
}

bool gram_batch_layout(const GramTables &t, long long smem, int &hist_off, int &tile)
{
    if (!t.ok || t.var || t.qw != 0) return false;
    if (t.max_keys > 4096u) return false;   // a round's keys are added up in 32 bits
    const long long room = smem - rr16((long long)kWarps * bwarp_bytes(t.s));
    const long long nc = (long long)t.code.size();
    const long long tab = (long long)t.filter.size() * 4 * (t.rank ? 2 : 1);
    if (tab > room || t.filter.size() % 4 != 0) return false;
    hist_off = tab + nc * 4 <= room ? int(tab) : -1;
    // tiles of at most kHits / 2 = 96 expected matches
    const double density = double(nc) / std::pow(4.0, double(std::min(t.m_min, 16)));
    const int step = kRow;
    tile = step;
    while (tile + step <= kMaxTile && density * (tile + step) <= kHits / 2) tile += step;
    return true;
}

void gram_batch_fill(const GramTables &t, const DevGram &dv, int tile, BatchDesc &D)
{
    D.gram = 1;
    D.tile = tile;
    D.g_s = t.s;
    D.g_rank = t.rank ? 1 : 0;
    D.g_fwords = int(t.filter.size());
    D.g_direct = 0;
    D.g_pw = t.pw;
    D.g_k = t.K[0];
    D.g_fshift = uint32_t(32 - t.fb);
    D.g_wshift = uint32_t(37 - t.fb);
    D.g_bshift = uint32_t(32 - t.db);
    D.g_filter = dv.filter;
    D.g_rank_base = dv.rank_base;
    D.g_dir = dv.dir;
    D.g_ent = dv.ent;
    D.g_pats = dv.pats;
    D.g_code = dv.code;
    D.g_grp_off = dv.grp_off;
    D.g_grp_ids = dv.grp_ids;
    D.nterms = int(t.code.size());
}

int gram_batch_tile(BatchDesc &D, int most)
{
    // 128 KiB of filter load in about 4 us; as many probes from L2 as a text of
    // a quarter of that makes take less
    D.g_direct = (D.t_hi - D.t_lo) * kWarpTile <= (long long)D.g_fwords ? 1 : 0;
    // as few rounds as the matches allow, and every warp an equal share
    const long long bytes = std::min(D.t_hi * kWarpTile, D.n) - D.t_lo * kWarpTile;
    const int step = kRow;
    const long long rounds = std::max<long long>(1, (bytes + (long long)most * kWarps - 1) / ((long long)most * kWarps));
    const long long each = (bytes + rounds * kWarps - 1) / (rounds * kWarps);
    return int(std::min<long long>(most, std::max<long long>(1, (each + step - 1) / step) * step));
}

int gram_batch_attr() { return kernel_smem_attr(reinterpret_cast<const void *>(gram_batch_kernel), smem_budget()); }

int gram_batch_enqueue(const BatchArgs &a, int grid, void *stream)
{
    gram_batch_kernel<<<dim3(unsigned(grid)), dim3(kWarps * 32), size_t(smem_budget()),
                        static_cast<cudaStream_t>(stream)>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_cuda_error(int(e)); return PM_ECUDA; }
    return PM_OK;
}

}  // namespace pm
