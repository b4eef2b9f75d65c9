// scan_gram_batch.cuh -- the gram items of the batched scan (scan_gram_batch.cu)
// as the batch planner and launcher see them.
#pragma once

#include "batch_device.cuh"

namespace pm {

long long gram_batch_smem(const DeviceProps &dp);  // per-CTA shared memory of the kernel
// Do the set's gram tables fit it? hist_off: byte offset of its
// counters behind the filter, -1 when they stay in device memory; tile: text
// bytes a warp takes at a time.
bool gram_batch_layout(const GramTables &t, long long smem, int &hist_off, int &tile);
void gram_batch_fill(const GramTables &t, const DevGram &dv, int tile, BatchDesc &D);
// the tile length of an item whose range is set, at most `most`; also decides
// whether the item's filter is probed in device memory
int gram_batch_tile(BatchDesc &D, int most);
int gram_batch_attr();  // raises the kernel's shared memory limit (before any capture)
int gram_batch_enqueue(const BatchArgs &a, int grid, void *stream);

}  // namespace pm
