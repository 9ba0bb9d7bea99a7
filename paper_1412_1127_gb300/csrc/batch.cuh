// batch.cuh -- internal entry of the batched-region path for other parts of
// the library (the served request loop).
#pragma once

#include "common.cuh"

namespace accr {
// Plans and launches `nregions` regions (the accr_batch_reduce device path)
// on `stream`; variables go to the device addresses in the descriptors.
// tile_bytes > 0 cuts long regions into tiles of that size instead of the
// process-wide tiling (accr_batch_tiling); the split of a region still
// depends only on its own type and length.
int batch_launch_regions(const accr_region *regions, int64_t nregions, accr_stream_t stream, int64_t tile_bytes = 0);

// Bytes up to which one warp folds a region (accr_batch_tiling), below 64 GiB.
int64_t batch_small_bytes();
// Bytes of a longer region's tiles, below 64 GiB.
int64_t batch_tile_bytes();

// A stream's staging for one call's plan: pinned memory to write it into and the
// device memory it is uploaded to.  Held (the stream's plans are made one at a
// time) from begin() to end() or destruction.
struct StreamBufs;
struct PlanStage {
    char *host = nullptr, *dev = nullptr;
    unsigned *counters = nullptr;  // reserve()'s words: zero, and left zero by the kernel
    int begin(accr_stream_t stream, size_t bytes);
    // More device memory (before upload(); `dev` may change), and counter words.
    int reserve(size_t bytes, size_t words, cudaStream_t s);
    int upload(size_t bytes, cudaStream_t s);
    void end();
    PlanStage() = default;
    PlanStage(const PlanStage &) = delete;
    PlanStage &operator=(const PlanStage &) = delete;
    ~PlanStage() { end(); }

private:
    StreamBufs *bufs = nullptr;
    int slot = 0;
};
}  // namespace accr
