// segtiles.cu -- segmented reductions with long segments (accr_segmented_reduce): the
// kernel whose CTAs fold those segments' tiles before its warps take the others.
//
// Generic codes only: a call with tiles streams most of its bytes in them, and the
// generic kernels give the others the bits the fixed-code ones give.
#include <string.h>

#include "segments.cuh"

namespace accr {

template <typename T>
static int tiled(SegArgs &a, cudaStream_t s) {
    switch (a.nc) {
    case 1: return SegLaunch<true>{}.run<T, 1, -1, -1>(a, s);
    case 2: return SegLaunch<true>{}.run<T, 2, -1, -1>(a, s);
    case 3: return SegLaunch<true>{}.run<T, 3, -1, -1>(a, s);
    default: return SegLaunch<true>{}.run<T, 4, -1, -1>(a, s);
    }
}

int segments_launch_tiled(SegArgs &a, int in_type, cudaStream_t s) {
    switch (in_type) {
    case ACCR_I32: return tiled<int32_t>(a, s);
    case ACCR_I64: return tiled<int64_t>(a, s);
    case ACCR_F32: return tiled<float>(a, s);
    default: return tiled<double>(a, s);
    }
}

}  // namespace accr
