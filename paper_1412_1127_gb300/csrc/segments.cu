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
//   * longer ones still are cut into tiles by the batched-region path.
//
// 100,000 segments of 1 to 1,024 floats, sum and max: 518 -> 51 us a call.
#include <string.h>

#include <algorithm>
#include <vector>

#include "batch.cuh"
#include "common.cuh"
#include "fold.cuh"
#include "group.cuh"
#include "overlap.cuh"
#include "rows.cuh"

namespace accr {

constexpr int SB = 256;           // threads per CTA
constexpr int SEG_PER_WARP = 16;  // short segments a warp takes at a time

struct SegArgs {
    const void *values;            // the element offset 0 counts from
    const void *off;               // nseg + 1 offsets, 32 or 64 bits
    const int32_t *mid;            // segments a warp folds alone
    int64_t nseg;
    int nmid, wide_off, nc;
    ClauseDev cl[ACCR_MAX_CLAUSES];
    uint64_t neutral[ACCR_MAX_CLAUSES];
    unsigned *queue;               // [2] next item, CTAs done; zero on entry and exit
};

__device__ __forceinline__ int64_t seg_offset(const SegArgs &p, int64_t i) {
    return p.wide_off ? ((const int64_t *)p.off)[i] : (int64_t)((const uint32_t *)p.off)[i];
}

template <typename T, int NC, int W0, int W1>
__global__ void __launch_bounds__(SB) segment_kernel(const __grid_constant__ SegArgs p) {
    constexpr bool E64 = sizeof(T) == 8;
    constexpr int EPV = 16 / (int)sizeof(T);
    grid_wait();
    const int lane = threadIdx.x & 31;
    int w[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) w[c] = (c == 0 && W0 >= 0) ? W0 : (c == 1 && W1 >= 0) ? W1 : p.cl[c].wcode;
    Acc A[NC];
    auto store = [&](int64_t s, bool empty) {
#pragma unroll
        for (int c = 0; c < NC; ++c) store_var(p.cl[c], s, finish(p.cl[c], E64, empty, to_final(w[c], A[c])));
    };
    // items: the listed segments, then groups of short ones; the next item is
    // fetched while this one is folded
    const int64_t items = p.nmid + (p.nseg + SEG_PER_WARP - 1) / SEG_PER_WARP;
    unsigned q = 0;
    if (lane == 0) q = atomicAdd(&p.queue[0], 1u);
    int64_t it = __shfl_sync(0xffffffffu, q, 0);
    while (it < items) {
        if (lane == 0) q = atomicAdd(&p.queue[0], 1u);
        if (it < p.nmid) {
            const int64_t s = p.mid[it];
            const int64_t lo = seg_offset(p, s), hi = seg_offset(p, s + 1);
            fold_stretch<T, NC, (W0 >= 0)>((const T *)p.values + lo, hi - lo, p.cl, w, lane, A);
            if (lane == 0) store(s, false);
        } else {
            const int64_t s0 = (it - p.nmid) * SEG_PER_WARP;
            // lane i < SEG_PER_WARP: segment s0 + i
            const bool have = lane < SEG_PER_WARP && s0 + lane < p.nseg;
            const int64_t lo = have ? seg_offset(p, s0 + lane) : 0, hi = have ? seg_offset(p, s0 + lane + 1) : 0;
            const int64_t bytes = (hi - lo) * (int64_t)sizeof(T);
            const int len = bytes <= GROUP_BYTES ? (int)(hi - lo) : 0;
            const int nv = (len + EPV - 1) / EPV;
            // lanes a segment takes: by its length alone
            const int cls = !have || bytes > GROUP_BYTES ? -1 : nv <= 2 * GROUP_GV ? 0 : nv <= 8 * GROUP_GV ? 1 : 2;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int L = k == 0 ? 2 : k == 1 ? 8 : 32;
                unsigned todo = __ballot_sync(0xffffffffu, cls == k);
                while (todo) {
                    // group g takes the g-th segment of the class that is left
                    int src = -1;
                    unsigned m = todo;
                    const int g = lane / L;
                    for (int j = 0; j < 32 / L && m; ++j) {
                        const int b = __ffs(m) - 1;
                        m &= m - 1;
                        if (j == g) src = b;
                    }
                    todo = m;
                    const int from = src < 0 ? 0 : src;
                    const int64_t slo = __shfl_sync(0xffffffffu, lo, from);
                    const int slen = __shfl_sync(0xffffffffu, len, from);
                    const bool live = src >= 0;
                    const int rounds = __reduce_max_sync(0xffffffffu, live ? (slen / EPV + L - 1) / L : 0);
                    group_fold<T, NC, W0, W1, GROUP_GV>((const T *)p.values + slo, slen, live, lane & (L - 1), L, rounds, p.cl,
                                              p.neutral, w, A);
                    if (live && (lane & (L - 1)) == 0) store(s0 + src, slen == 0);
                }
            }
        }
        it = __shfl_sync(0xffffffffu, q, 0);
    }
    grid_release();  // a warp of the CTA found the queue empty
    // the last CTA returns the queue to zero for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&p.queue[1], 1u) == gridDim.x - 1) {
            p.queue[0] = 0u;
            p.queue[1] = 0u;
        }
    }
}

// ---- host side ---------------------------------------------------------------------

struct SegLaunch {
    template <typename T, int NC, int W0, int W1>
    int run(SegArgs &a, cudaStream_t s) const {
        static std::atomic<int> cached[64];
        int rc = launch_guard("segment_kernel");
        if (rc != ACCR_OK) return rc;
        for (int c = 0; c < NC; ++c) a.neutral[c] = neutral_element<T>(a.cl[c].wcode);
        const int maxg = resident_ctas(segment_kernel<T, NC, W0, W1>, SB, cached);
        const int64_t items = a.nmid + (a.nseg + SEG_PER_WARP - 1) / SEG_PER_WARP;
        const int grid = clamp_grid((items + SB / 32 - 1) / (SB / 32), maxg);
        launch_overlapped(segment_kernel<T, NC, W0, W1>, dim3((unsigned)grid), SB, 0, s, a);
        return launched("segment_kernel");
    }
};

// Segments past the short ones, in index order: `mid` (a warp each, a class per
// power of two of their bytes) and `tiled`.
struct LongSegments {
    std::vector<int32_t> mid[4], tiled;
    void clear() {
        for (auto &v : mid) v.clear();
        tiled.clear();
    }
};

// Checks the offsets and writes them to dst, relative to off[0] (which is not
// negative); returns the first segment that ends before it starts, or -1.  Whole
// blocks are checked by their smallest and largest length and by their offsets'
// signs (without a negative offset no length overflows); only a block with a
// longer segment is looked through one by one.
template <typename O>
static int64_t copy_offsets(const int64_t *off, int64_t nseg, O *dst, int64_t max_short, int64_t max_mid, LongSegments &L) {
    constexpr int64_t BLK = 512;
    const int64_t base = off[0];
    for (int64_t b = 0; b < nseg; b += BLK) {
        const int64_t e = std::min(nseg, b + BLK);
        int64_t lo = INT64_MAX, hi = 0, signs = 0;
        for (int64_t s = b; s < e; ++s) {
            const int64_t n = (int64_t)((uint64_t)off[s + 1] - (uint64_t)off[s]);
            lo = n < lo ? n : lo;
            hi = n > hi ? n : hi;
            signs |= off[s + 1];
            dst[s] = (O)((uint64_t)off[s] - (uint64_t)base);
        }
        if (lo < 0 || signs < 0) {
            for (int64_t s = b; s < e; ++s)
                if (off[s + 1] < off[s]) return s;
        }
        if (hi <= max_short) continue;
        for (int64_t s = b; s < e; ++s) {
            const int64_t n = off[s + 1] - off[s];
            if (n <= max_short) continue;
            if (n > max_mid) L.tiled.push_back((int32_t)s);
            else L.mid[n > 8 * max_short ? 0 : n > 4 * max_short ? 1 : n > 2 * max_short ? 2 : 3].push_back((int32_t)s);
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
    const size_t obytes = (size_t)(nseg + 1) * (wide ? 8 : 4), mid_off = (obytes + 255) & ~(size_t)255;
    const size_t most = mid_off + sizeof(int32_t) * (size_t)nseg;
    static thread_local LongSegments L;
    L.clear();
    const int64_t max_short = GROUP_BYTES / eb, max_mid = std::max(GROUP_BYTES, batch_small_bytes()) / eb;
    PlanStage st;
    rc = st.begin(stream, most);
    if (rc != ACCR_OK) return rc;
    const int64_t bad = wide ? copy_offsets(offsets, nseg, (int64_t *)st.host, max_short, max_mid, L)
                             : copy_offsets(offsets, nseg, (uint32_t *)st.host, max_short, max_mid, L);
    if (bad >= 0) return set_error(ACCR_EINVAL, "segmented: offsets not non-decreasing at %lld", (long long)bad);
    if (total > 0 && !values) return set_error(ACCR_EINVAL, "segmented: values is NULL");
    Scratch *scr = scratch_for(stream, 0);
    if (!scr) return ACCR_ENOMEM;
    int32_t *mid = (int32_t *)(st.host + mid_off);
    for (const auto &v : L.mid) {
        if (!v.empty()) memcpy(mid + a.nmid, v.data(), sizeof(int32_t) * v.size());
        a.nmid += (int)v.size();
    }
    rc = st.upload(a.nmid ? mid_off + sizeof(int32_t) * (size_t)a.nmid : obytes, s);
    if (rc != ACCR_OK) return rc;
    log_msg(2, "accr_segmented_reduce: %lld segments type=%d clauses=%d, %d by a warp, %zu tiled", (long long)nseg, in_type,
            nclauses, a.nmid, L.tiled.size());
    a.values = (const char *)values + offsets[0] * eb;
    a.off = st.dev;
    a.mid = (const int32_t *)(st.dev + mid_off);
    a.nseg = nseg;
    a.wide_off = wide;
    a.nc = nclauses;
    a.queue = scr->counters + 24;  // words 24-25
    ClauseDev cl[ACCR_MAX_CLAUSES];  // the caller's order, for the tiled ones
    memcpy(cl, a.cl, sizeof cl);
    rc = row_dispatch(a, in_type, SegLaunch{}, s);
    if (rc == ACCR_OK && !L.tiled.empty()) {
        st.end();
        rc = batch_launch_segments(values, offsets, L.tiled.data(), (int64_t)L.tiled.size(), in_type, cl, nclauses, stream);
    }
    if (rc != ACCR_OK) return rc;
    if (flags & ACCR_SYNC) return cuda_check(cudaStreamSynchronize(s), "batch: sync");
    return ACCR_OK;
}
