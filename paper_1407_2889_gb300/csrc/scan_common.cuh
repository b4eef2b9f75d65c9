// scan_common.cuh -- device helpers shared by the Aho-Corasick and Wu-Manber
// scan kernels: inline PTX for mbarriers and 1-D TMA bulk copies
// (cp.async.bulk), acquire/release global accesses, a bounded spin, warp
// scans and the per-pattern counters.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "pm_internal.h"

namespace pm {
namespace dev {

constexpr uint32_t kFull = 0xFFFFFFFFu;
// ~1-4 s at GB300 clocks: a wait that long means something is wrong
constexpr long long kSpinLimit = 4000000000LL;

// status word codes in the workspace header
constexpr uint32_t kErrTimeoutTma = 1;
constexpr uint32_t kErrTimeoutWait = 2;       // reserved: a bounded wait on another CTA gave up
constexpr uint32_t kErrInternal = 3;        // a consistency check failed

struct WsHeader {           // lives at the start of the workspace
    uint32_t status;        // 0 = ok, else kErr*
    uint32_t done_ctas;     // CTAs that finished (the last one finalises counts)
    uint32_t done_expand;   // expand CTAs that finished (late ids: the last one finalises counts)
    uint32_t pad0;
    unsigned long long queue;  // batched scan: next instance to take
    unsigned long long queue2; // batched gram scan: next item to take
    unsigned long long pad1[28];
};
static_assert(sizeof(WsHeader) <= kWsHeader, "workspace header too large");

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of `bar` to complete; false if the limit ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > kSpinLimit) return false;
    }
    return true;
}

// 1-D bulk copy global -> this CTA's shared memory, completing on `bar`.
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, uint32_t bytes,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Look-back statuses carry their own "published" flag bits and every reader
// spins until those bits are set, so no other data is ordered behind them:
// relaxed (volatile) accesses suffice and avoid a memory barrier per tile.
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void set_status(WsHeader *h, uint32_t code)
{
    atomicCAS(&h->status, 0u, code);
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

__device__ __forceinline__ void count_pattern(uint32_t r, uint32_t *s_hist, long long *g_counts)
{
    if (s_hist) atomicAdd(&s_hist[r], 1u);
    else atomicAdd(reinterpret_cast<unsigned long long *>(g_counts) + r, 1ull);
}

// Output offsets of a segment of nt warp tiles (from tile t0 on), by the whole
// CTA of THREADS threads: s_off[q] gets the number of keys before tile t0 + q
// (those of the segments before this one, number seg, and *base included),
// s_ent[q] its entries (at most max_ent). Returns, on the last thread, the
// keys up to the segment's end. s_red: THREADS / 32 words.
template <int THREADS>
__device__ __forceinline__ unsigned long long
segment_offsets(const uint32_t *tile_ent, const uint32_t *tile_out, const unsigned long long *seg_sum, long long seg,
                long long t0, long long nt, const unsigned long long *base, uint32_t max_ent,
                unsigned long long *s_off, uint32_t *s_ent, unsigned long long *s_red)
{
    constexpr int NW = THREADS / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // base of the segment: sum of the earlier segments
    unsigned long long part = 0;
    for (long long q = tid; q < seg; q += THREADS) part += seg_sum[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
    if (lane == 0) s_red[warp] = part;
    __syncthreads();
    // a chunk of a longer scan writes after the keys of the chunks before it
    unsigned long long seg_base = base ? *base : 0ull;
#pragma unroll
    for (int w = 0; w < NW; ++w) seg_base += s_red[w];
    __syncthreads();
    // per-tile offsets: each thread scans a run of consecutive tiles
    const long long per = (nt + THREADS - 1) / THREADS;
    const long long r0 = min(nt, (long long)tid * per), r1 = min(nt, r0 + per);
    unsigned long long mine = 0;
    for (long long q = r0; q < r1; ++q) {
        const uint32_t o = tile_out[t0 + q];
        s_ent[q] = min(tile_ent[t0 + q], max_ent);
        s_off[q] = o;  // the tile's own total, replaced by its offset below
        mine += o;
    }
    unsigned long long inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_red[warp] = inc;
    __syncthreads();
    unsigned long long run = seg_base + inc - mine;
    for (int w = 0; w < warp; ++w) run += s_red[w];
    for (long long q = r0; q < r1; ++q) {
        const unsigned long long o = s_off[q];
        s_off[q] = run;
        run += o;
    }
    return run;
}

// Kernels of one scan follow one another in a stream and each starts with work
// that does not need the one before (table loads): launched as programmatic
// dependents they do that work while the other still runs. Every such kernel
// calls grid_wait() before it reads or writes what earlier kernels touch, and
// the kernels before it let it start early with grid_trigger(). What an earlier
// kernel of the chain writes is written during this kernel's lifetime, so it is
// read with ordinary loads: its pointers are not const __restrict__ and not
// read by __ldg, which may use the non-coherent path.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_dependent(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

}  // namespace dev
}  // namespace pm
