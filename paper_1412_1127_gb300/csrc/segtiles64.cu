// segtiles64.cu -- the kernels of segtiles.cu for elements of 8 bytes.
#include <string.h>

#include "segments.cuh"

namespace accr {

int segments_launch_tiled64(SegArgs &a, int in_type, cudaStream_t s) {
    return in_type == ACCR_I64 ? row_launch<int64_t>(a, SegLaunch<true>{}, s) : row_launch<double>(a, SegLaunch<true>{}, s);
}

}  // namespace accr
