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

// The same for the listed segments values[off[s] .. off[s + 1]), s = idx[0 .. n),
// whose offsets the caller has checked; `cl`: lowered clauses, whose outputs are
// the starts of the variables' arrays.
struct ClauseDev;
int batch_launch_segments(const void *values, const int64_t *off, const int32_t *idx, int64_t n, int in_type,
                          const ClauseDev *cl, int nc, accr_stream_t stream);

// Bytes up to which one warp folds a region (accr_batch_tiling), below 64 GiB.
int64_t batch_small_bytes();

// A stream's staging for one call's plan: pinned memory to write it into and the
// device memory it is uploaded to.  Held (the stream's plans are made one at a
// time) from begin() to end() or destruction.
struct StreamBufs;
struct PlanStage {
    char *host = nullptr, *dev = nullptr;
    int begin(accr_stream_t stream, size_t bytes);
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
