// segments.cu -- consecutive segments of one array, one variable per segment
// (accr_segmented_reduce): every segment has the same element type and clauses,
// so the device needs nothing per segment but its offsets.
//
// A batch's plan holds a descriptor (112 bytes) and a queue entry per region;
// for 100,000 segments of about 150 floats the host spent 0.5 ms writing and
// uploading 11.6 MB of them, and the kernel 0.14 ms at a warp per segment, for
// 60 MB of elements (9 us).  Here the host checks the offsets and uploads them
// (four bytes each while the array has fewer than 2^32 elements), and one launch
// folds, by the segment's own length alone:
//
//   * segments of at most GROUP_BYTES (4 KiB): a warp takes SEG_PER_WARP
//     neighbouring segments and folds them a length class at a time, in groups of
//     2, 8 or 32 lanes (at most eight vectors a lane, all in flight);
//   * longer ones up to the batch's warp-region limit (64 KiB by default): a warp
//     each, from a list the host makes, longest class first;
//   * longer ones still are cut into tiles (accr_batch_tiling's size) that CTAs fold
//     ahead of the others, from a queue of their own.  (As a second, batched launch
//     behind this one a few hundred of them took longer than a batch of all segments:
//     1,236 segments of up to 47,765 doubles 66 us, 50 as a batch, 40 so.)
//
// 100,000 segments of 1 to 1,024 floats, sum and max: 518 -> 51 us a call.
#include <string.h>

#include <algorithm>
#include <vector>

#include "batch.cuh"
#include "segments.cuh"

namespace accr {

// Segments past the short ones, a class per power of two of their bytes, the longest
// first, in index order in each: `mid` (a warp each) and `tiled`.
struct LongSegments {
    std::vector<int32_t> mid[4], tiled[6];
    void clear() {
        for (auto &v : mid) v.clear();
        for (auto &v : tiled) v.clear();
    }
};

// Checks the offsets and writes them to dst, relative to off[0] (which is not
// negative); returns the first segment that ends before it starts, or -1.  Whole
// blocks are checked by their smallest and largest length; a block that starts or has a
// length beyond any array, where a length may overflow, by its offsets; and only a
// block with a longer segment is looked through one by one.
template <typename O>
static int64_t copy_offsets(const int64_t *off, int64_t nseg, O *dst, int64_t max_short, int64_t max_mid, LongSegments &L) {
    constexpr int64_t BLK = 512, FAR = (int64_t)1 << 52;  // FAR + BLK * FAR still fits
    const int64_t base = off[0];
    for (int64_t b = 0; b < nseg; b += BLK) {
        const int64_t e = std::min(nseg, b + BLK);
        int64_t lo = INT64_MAX, hi = 0;
        for (int64_t s = b; s < e; ++s) {
            const int64_t n = (int64_t)((uint64_t)off[s + 1] - (uint64_t)off[s]);
            lo = n < lo ? n : lo;
            hi = n > hi ? n : hi;
            dst[s] = (O)((uint64_t)off[s] - (uint64_t)base);
        }
        if (lo < 0 || hi > FAR || off[b] > FAR) {
            for (int64_t s = b; s < e; ++s)
                if (off[s + 1] < off[s]) return s;
        }
        if (hi <= max_short) continue;
        for (int64_t s = b; s < e; ++s) {
            const int64_t n = off[s + 1] - off[s];
            if (n <= max_short) continue;
            if (n > max_mid) {
                int c = 5;
                while (c > 0 && n > max_mid << (6 - c)) --c;
                L.tiled[c].push_back((int32_t)s);
            } else L.mid[n > 8 * max_short ? 0 : n > 4 * max_short ? 1 : n > 2 * max_short ? 2 : 3].push_back((int32_t)s);
        }
    }
    dst[nseg] = (O)((uint64_t)off[nseg] - (uint64_t)base);
    return -1;
}

}  // namespace accr

using namespace accr;

extern "C" ACCR_API int accr_segmented_reduce(const void *values, const int64_t *offsets, int64_t nseg,
                                              int32_t in_type, const accr_clause *clauses, int32_t nclauses,
                                              uint32_t flags, accr_stream_t stream) {
    ACCR_TRACE("accr_segmented_reduce");
    clear_error();
    if (flags & ~(ACCR_SYNC | ACCR_COMPENSATED))
        return set_error(ACCR_EINVAL, "accr_segmented_reduce: unsupported flags 0x%x", flags);
    if (nseg < 0 || (nseg > 0 && !offsets)) return set_error(ACCR_EINVAL, "segmented: bad offsets");
    if (nseg > INT32_MAX / 2) return set_error(ACCR_EINVAL, "segmented: too many segments");
    SegArgs a;
    memset(&a, 0, sizeof a);
    int rc = lower_clauses(in_type, clauses, nclauses, flags & ACCR_COMPENSATED, a.cl);
    if (rc != ACCR_OK) return rc;
    if (nseg == 0) return ACCR_OK;
    const int64_t eb = type_bytes(in_type);
    if (offsets[0] < 0) return set_error(ACCR_EINVAL, "segmented: offsets not non-decreasing at 0");
    if (((uintptr_t)values & (uintptr_t)(eb - 1)) != 0)
        return set_error(ACCR_EINVAL, "region 0: in is not aligned to its element size");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t total = (int64_t)((uint64_t)offsets[nseg] - (uint64_t)offsets[0]);
    // (a total below zero, or above what the narrow form holds, takes the wide one;
    // the check below finds decreasing offsets either way)
    const bool wide = total < 0 || total > (int64_t)UINT32_MAX;
    // staging: the offsets, then the lists (4 bytes a warp's segment, 8 a tiled one and 4)
    const size_t obytes = (size_t)(nseg + 1) * (wide ? 8 : 4), list_off = (obytes + 255) & ~(size_t)255;
    static thread_local LongSegments L;
    L.clear();
    const int64_t max_short = GROUP_BYTES / eb, max_mid = std::max(GROUP_BYTES, batch_small_bytes()) / eb;
    PlanStage st;
    rc = st.begin(stream, list_off + 8 * (size_t)nseg + 4);
    if (rc != ACCR_OK) return rc;
    const int64_t bad = wide ? copy_offsets(offsets, nseg, (int64_t *)st.host, max_short, max_mid, L)
                             : copy_offsets(offsets, nseg, (uint32_t *)st.host, max_short, max_mid, L);
    if (bad >= 0) return set_error(ACCR_EINVAL, "segmented: offsets not non-decreasing at %lld", (long long)bad);
    if (total > 0 && !values) return set_error(ACCR_EINVAL, "segmented: values is NULL");
    Scratch *scr = scratch_for(stream, 0);
    if (!scr) return ACCR_ENOMEM;
    int32_t *list = (int32_t *)(st.host + list_off);
    for (const auto &v : L.mid) {
        if (!v.empty()) memcpy(list + a.nmid, v.data(), sizeof(int32_t) * v.size());
        a.nmid += (int)v.size();
    }
    int32_t *tiled = list + a.nmid;
    for (const auto &v : L.tiled) {
        if (!v.empty()) memcpy(tiled + a.ntiled, v.data(), sizeof(int32_t) * v.size());
        a.ntiled += (int)v.size();
    }
    a.tile_elems = batch_tile_bytes() / eb;
    int64_t ntiles = 0;
    if (a.ntiled) {
        int32_t *tile0 = tiled + a.ntiled;
        for (int i = 0; i < a.ntiled; ++i) {
            tile0[i] = (int32_t)ntiles;
            ntiles += (offsets[tiled[i] + 1] - offsets[tiled[i]] + a.tile_elems - 1) / a.tile_elems;
            if (ntiles > INT32_MAX) return set_error(ACCR_EINVAL, "batch: more than 2^31 tiles");
        }
        tile0[a.ntiled] = (int32_t)ntiles;
    }
    const size_t words = (size_t)a.nmid + (a.ntiled ? 2 * (size_t)a.ntiled + 1 : 0);
    const size_t bytes = words ? list_off + 4 * words : obytes, part_off = (bytes + 255) & ~(size_t)255;
    if (ntiles > a.ntiled) {  // some segment has several tiles
        rc = st.reserve(part_off + sizeof(Partial) * (size_t)nclauses * (size_t)ntiles, (size_t)a.ntiled, s);
        if (rc != ACCR_OK) return rc;
    }
    rc = st.upload(bytes, s);
    if (rc != ACCR_OK) return rc;
    log_msg(2, "accr_segmented_reduce: %lld segments type=%d clauses=%d, %d by a warp, %d tiled (%lld tiles)", (long long)nseg,
            in_type, nclauses, a.nmid, a.ntiled, (long long)ntiles);
    a.values = (const char *)values + offsets[0] * eb;
    a.off = st.dev;
    a.mid = (const int32_t *)(st.dev + list_off);
    a.tiled = a.mid + a.nmid;
    a.tile0 = a.tiled + a.ntiled;
    a.ntiles = (int)ntiles;
    a.partials = (Partial *)(st.dev + part_off);
    a.tiles_done = st.counters;
    a.nseg = nseg;
    a.wide_off = wide;
    a.nc = nclauses;
    a.queue = scr->counters + 24;  // words 24-26
    rc = a.ntiled ? segments_launch_tiled(a, in_type, s) : row_dispatch(a, in_type, SegLaunch<false>{}, s);
    if (rc != ACCR_OK) return rc;
    if (flags & ACCR_SYNC) return cuda_check(cudaStreamSynchronize(s), "batch: sync");
    return ACCR_OK;
}
