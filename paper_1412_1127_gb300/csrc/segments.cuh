// segments.cuh -- the kernel of accr_segmented_reduce (see segments.cu), in two forms:
// without tiles, and with the long segments' tiles at the head of its queue.
#pragma once

#include "common.cuh"
#include "debug.cuh"
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
    const int32_t *tiled, *tile0;  // long segments, and the first tile of each (ntiled + 1 entries)
    int ntiled, ntiles;
    int64_t tile_elems;
    Partial *partials;             // [ntiles][nc]: tiles of segments of several
    unsigned *tiles_done;          // [ntiled] zero on entry and exit
    ClauseDev cl[ACCR_MAX_CLAUSES];
    uint64_t neutral[ACCR_MAX_CLAUSES];
    unsigned *queue;               // [3] next item, CTAs done, next tile; zero on entry and exit
};

__device__ __forceinline__ int64_t seg_offset(const SegArgs &p, int64_t i) {
    return p.wide_off ? ((const int64_t *)p.off)[i] : (int64_t)((const uint32_t *)p.off)[i];
}

// Tile `q` of the long segments, folded by the whole CTA; the last tile of a segment of
// several to finish merges their partials in tile order.
template <typename T, int NC, bool FIXED>
__device__ __forceinline__ void segment_tile(const SegArgs &p, int q, const int (&w)[NC], Acc (*sh)[SB / 32], int *s_last) {
    constexpr bool E64 = sizeof(T) == 8;
    int i = q;  // its place in the list: every segment one tile, or by search
    if (p.ntiles != p.ntiled) {
        int lo = 0, hi = p.ntiled;
        while (hi - lo > 1) {
            const int m = (lo + hi) / 2;
            if (p.tile0[m] <= q) lo = m;
            else hi = m;
        }
        i = lo;
    }
    const int64_t s = p.tiled[i], base = seg_offset(p, s), n = seg_offset(p, s + 1) - base;
    const int t0 = p.tile0[i], nt = p.tile0[i + 1] - t0;
    // the same for the whole CTA
    if (!ACCR_DCHECK(i < p.ntiled && q >= t0 && q - t0 < nt && s >= 0 && s < p.nseg, DS_SEGMENT_TILE)) return;
    const int64_t lo = (int64_t)(q - t0) * p.tile_elems, len = n - lo < p.tile_elems ? n - lo : p.tile_elems;
    Acc A[NC];
    uint64_t id[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        id[c] = p.cl[c].ident;
        A[c].a = id[c];
        A[c].c = 0.f;
    }
    stream_fold<T, NC, RU2, SB, true>((const T *)p.values + base + lo, len, (int)threadIdx.x, w, A, ld_stream);
    cta_merge<NC, SB, FIXED>(w, id, E64, A, sh);
    if (nt == 1) {
        if (threadIdx.x == 0) {
#pragma unroll
            for (int c = 0; c < NC; ++c) store_var(p.cl[c], s, finish(p.cl[c], E64, false, to_final(w[c], A[c])));
        }
        return;
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            Partial x;
            x.a = A[c].a;
            x.c = A[c].c;
            x.pad = 0;
            if (ACCR_DCHECK(q >= 0 && q < p.ntiles, DS_SEGMENT_TILE)) p.partials[(int64_t)q * NC + c] = x;
        }
        __threadfence();
        *s_last = atomicAdd(&p.tiles_done[i], 1u) == (unsigned)(nt - 1);
    }
    __syncthreads();
    const int last = *s_last;
    __syncthreads();
    if (!last) return;
    __threadfence();
    int fw[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        fw[c] = final_code(w[c]);
        id[c] = final_ident(p.cl[c]);
        A[c].a = id[c];
        A[c].c = 0.f;
        for (int j = (int)threadIdx.x; j < nt; j += SB) {
            const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(&p.partials[(int64_t)(t0 + j) * NC + c]));
            Acc Q;
            Q.a = ((uint64_t)v.y << 32) | v.x;
            Q.c = __uint_as_float(v.z);
            merge(fw[c], E64, A[c], to_final(w[c], Q));
        }
    }
    cta_merge<NC, SB, FIXED>(fw, id, E64, A, sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) store_var(p.cl[c], s, finish(p.cl[c], E64, false, A[c]));
        p.tiles_done[i] = 0u;
    }
}

template <typename T, int NC, int W0, int W1, bool TILES>
__global__ void __launch_bounds__(SB, TILES ? 2 : 0) segment_kernel(const __grid_constant__ SegArgs p) {
    constexpr bool E64 = sizeof(T) == 8;
    constexpr int EPV = 16 / (int)sizeof(T);
    grid_wait();
    const int lane = threadIdx.x & 31;
    int w[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) w[c] = (c == 0 && W0 >= 0) ? W0 : (c == 1 && W1 >= 0) ? W1 : p.cl[c].wcode;
    Acc A[NC];
    auto store = [&](int64_t s, bool empty) {
        if (!ACCR_DCHECK(s >= 0 && s < p.nseg, DS_SEGMENT_VAR)) return;
#pragma unroll
        for (int c = 0; c < NC; ++c) store_var(p.cl[c], s, finish(p.cl[c], E64, empty, to_final(w[c], A[c])));
    };
    if constexpr (TILES) {  // CTAs take the tiles first; the next one is fetched while this one is folded
        __shared__ Acc sh[NC][SB / 32];
        __shared__ int s_last, s_q;
        if (threadIdx.x == 0) s_q = (int)atomicAdd(&p.queue[2], 1u);
        __syncthreads();
        int q = s_q;
        __syncthreads();
        while (q < p.ntiles) {
            if (threadIdx.x == 0) s_q = (int)atomicAdd(&p.queue[2], 1u);
            segment_tile<T, NC, (W0 >= 0)>(p, q, w, sh, &s_last);
            __syncthreads();
            q = s_q;
            __syncthreads();
        }
    }
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
            p.queue[2] = 0u;
        }
    }
}

// ---- host side ---------------------------------------------------------------------

template <bool TILES>
struct SegLaunch {
    template <typename T, int NC, int W0, int W1>
    int run(SegArgs &a, cudaStream_t s) const {
        static std::atomic<int> cached[64];
        int rc = launch_guard("segment_kernel");
        if (rc != ACCR_OK) return rc;
        for (int c = 0; c < NC; ++c) a.neutral[c] = neutral_element<T>(a.cl[c].wcode);
        const int maxg = resident_ctas(segment_kernel<T, NC, W0, W1, TILES>, SB, cached);
        const int64_t items = a.nmid + (a.nseg + SEG_PER_WARP - 1) / SEG_PER_WARP;
        const int64_t want = (items + SB / 32 - 1) / (SB / 32);
        const int grid = clamp_grid(want < a.ntiles ? a.ntiles : want, maxg);
        launch_overlapped(segment_kernel<T, NC, W0, W1, TILES>, dim3((unsigned)grid), SB, 0, s, a);
        return launched("segment_kernel");
    }
};

int segments_launch_tiled(SegArgs &a, int in_type, cudaStream_t s);    // segtiles.cu
int segments_launch_tiled64(SegArgs &a, int in_type, cudaStream_t s);  // segtiles64.cu

}  // namespace accr
