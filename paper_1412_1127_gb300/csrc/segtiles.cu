// segtiles.cu -- segmented reductions with long segments (accr_segmented_reduce): the
// kernel whose CTAs fold those segments' tiles before its warps take the others, for
// elements of 4 bytes (those of 8: segtiles64.cu, compiled beside it).
//
// A sum with a max or min has fixed codes here too: 1,060 segments of up to 31,853 floats
// take 51 us with the generic fold of two clauses, 22 so (43 as a batch).
#include <string.h>

#include "segments.cuh"

namespace accr {

int segments_launch_tiled(SegArgs &a, int in_type, cudaStream_t s) {
    switch (in_type) {
    case ACCR_I32: return row_launch<int32_t>(a, SegLaunch<true>{}, s);
    case ACCR_F32: return row_launch<float>(a, SegLaunch<true>{}, s);
    default: return segments_launch_tiled64(a, in_type, s);
    }
}

}  // namespace accr
