// batch_device.cuh -- what the batched kernels share: their arguments, and how
// a queue item (a whole instance, or a part of one split over several CTAs)
// turns its pass over the text into counts, keys and a total.
#pragma once

#include "scan_common.cuh"

namespace pm {

struct BatchArgs {
    const BatchDesc *desc;
    int k;
    const uint8_t *text;
    long long *counts;
    unsigned long long *occ;
    long long *n_occ;
    dev::WsHeader *ws;
    unsigned long long *ccount;
    unsigned long long *spill;     // key staging of split instances' parts
    int list;
    int region_bytes;              // per-CTA shared memory for table, ids and counters
};

__host__ __device__ constexpr long long rr16(long long x) { return (x + 15) & ~15LL; }

// All threads of the CTA call it. pass(count, write, base) scans the item:
// `count` bumps the counters (s_hist, or g_hist in device memory when s_hist is
// NULL), `write` writes the keys to odst (at most ocap of them) from offset
// base on; it returns the item's keys. write_counts(from_device) writes the
// instance's counts from g_hist or s_hist.
template <class Pass, class Counts>
__device__ __forceinline__ void run_item(const BatchArgs &a, const BatchDesc &D, uint32_t *s_hist, unsigned long long *g_hist,
                         unsigned long long *&odst, unsigned long long &ocap, Pass &&pass, Counts &&write_counts)
{
    if (D.nparts <= 1) {
        const unsigned long long total = pass(true, a.list != 0, 0ull);
        if (threadIdx.x == 0) a.n_occ[D.out_slot] = (long long)total;
        write_counts(s_hist == nullptr);
        __syncthreads();
        return;
    }

    // ---- a part of a split instance ----------------------------------------
    __shared__ unsigned long long s_base;
    __shared__ int s_last;
    unsigned long long *pstat = a.ccount + D.pstat_off;  // (1 << 63) | part total
    const bool staged = a.list && D.spill_cap > 0;
    if (staged) {
        odst = a.spill + D.spill_off;
        ocap = (unsigned long long)D.spill_cap;
    }
    const unsigned long long total = pass(true, staged, 0ull);
    if (threadIdx.x == 0) dev::st_relaxed(&pstat[D.part], (1ull << 63) | total);
    if (threadIdx.x < 32) {
        // the parts before this one were taken earlier by running CTAs, and
        // publish their totals without waiting for anything; a lane waits for
        // every 32nd of them (one thread after another took 0.7 us a part)
        unsigned long long base = 0;
        if (a.list) {
            const long long t0c = clock64();
            for (int q = threadIdx.x; q < D.part; q += 32) {
                unsigned long long v = dev::ld_relaxed(&pstat[q]);
                while (!(v >> 63)) {
                    if (clock64() - t0c > dev::kSpinLimit) {
                        dev::set_status(a.ws, dev::kErrTimeoutWait);
                        break;
                    }
                    __nanosleep(128);
                    v = dev::ld_relaxed(&pstat[q]);
                }
                base += v & ~(1ull << 63);
            }
            __syncwarp();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(dev::kFull, base, o);
        }
        if (threadIdx.x == 0) s_base = base;
    }
    __syncthreads();
    if (a.list) {
        odst = a.occ + D.occ_off;
        ocap = (unsigned long long)D.occ_cap;
        const unsigned long long b0 = s_base;
        if (staged && total <= (unsigned long long)D.spill_cap) {
            // this CTA's own stores, ordered by the barrier above
            const unsigned long long *sp = a.spill + D.spill_off;
            const unsigned long long nkeep = b0 < ocap ? min(total, ocap - b0) : 0ull;
            for (unsigned long long i = threadIdx.x; i < nkeep; i += blockDim.x) odst[b0 + i] = sp[i];
        } else if (b0 < ocap) {
            (void)pass(false, true, b0);
        }
    }
    // counters into the instance's device counters; the last part writes
    // the instance's counts and its total
    if (s_hist)
        for (int c = threadIdx.x; c < D.nterms; c += blockDim.x)
            if (s_hist[c]) atomicAdd(&g_hist[c], (unsigned long long)s_hist[c]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int *done = reinterpret_cast<unsigned int *>(a.ccount + D.done_off);
        s_last = atomicAdd(done, 1u) == unsigned(D.nparts - 1);
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        write_counts(true);
        if (threadIdx.x == 0) {
            unsigned long long all = 0;
            for (int q = 0; q < D.nparts; ++q) all += dev::ld_acquire(&pstat[q]) & ~(1ull << 63);
            a.n_occ[D.out_slot] = (long long)all;
        }
    }
    __syncthreads();
}

}  // namespace pm
