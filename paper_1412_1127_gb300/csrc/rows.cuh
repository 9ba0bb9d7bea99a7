// rows.cuh -- what the forms of the row nest (and of segments) share: the
// kernels' arguments, a warp's fold of a stretch, launch sizes, and the choice
// of a kernel with fixed clause codes.
#pragma once

#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "fold.cuh"
#include "overlap.cuh"

namespace accr {

struct RowArgs {
    const void *A;
    int64_t rows, cols, ld;
    int nc;
    ClauseDev cl[ACCR_MAX_CLAUSES];
    uint64_t neutral[ACCR_MAX_CLAUSES];  // group form: an element that leaves the clause's fold as it is
    int64_t release_row;  // from this row on a warp (or CTA) lets the next kernel be set up
    int lanes;            // group form: lanes per row
    int64_t chunk;        // split form: elements per chunk; segment form: per segment
    int64_t cpr;          // split form: chunks per row; segment form: segments per row
    Partial *partials;    // split form: [rows][nc][cpr]
    unsigned *counters;   // split form: [rows], zero on entry, zero again on exit (zeroed_words_for)
};

// 16-byte vectors per lane per iteration: picked by the autotuner ("vectors"
// in tuning.json), passed in by the build.
#ifndef ACCR_ROW_RU
#define ACCR_ROW_RU 8
#endif
constexpr int RU2 = ACCR_ROW_RU;

// One stretch of `len` elements (below 64 GiB, as stream_fold takes), folded by one
// warp and merged across its lanes.
template <typename T, int NC, bool FIXED>
__device__ __forceinline__ void fold_stretch(const T *row, int64_t len, const ClauseDev *cl, const int (&w)[NC], int lane,
                                             Acc (&A)[NC]) {
    constexpr bool E64 = sizeof(T) == 8;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        A[c].a = cl[c].ident;
        A[c].c = 0.f;
    }
    stream_fold<T, NC, RU2, 32, true>(row, len, lane, w, A, ld_stream);
#pragma unroll
    for (int c = 0; c < NC; ++c) warp_merge<FIXED>(w[c], E64, A[c]);
}

// CTAs of `threads` threads of a kernel that are resident at once, per device
// (computed once; a racing first computation stores the same value twice).
template <typename K>
static int resident_ctas(K kernel, int threads, std::atomic<int> *cached) {
    const DeviceInfo &d = device_info();
    std::atomic<int> &slot = cached[d.id & 63];
    int g = slot.load(std::memory_order_relaxed);
    if (!g) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
        if (per_sm < 1) per_sm = 1;
        g = per_sm * d.sms;
        slot.store(g, std::memory_order_relaxed);
    }
    return g;
}

static int clamp_grid(int64_t want, int64_t most) { return (int)(want < 1 ? 1 : want < most ? want : most); }

// A sum together with a max or a min (the two-clause form of a region that
// reports a total and an extreme) gets a kernel with both codes fixed: the
// generic two-clause fold needs 64 registers a thread, the fixed one 32-40,
// which leaves room for more rows in flight per SM.
template <typename T, int W0, int W1, typename A, typename L>
static bool pair_launch(A &a, const L &launch, cudaStream_t s, int &rc) {
    if (a.cl[0].wcode != W0 || a.cl[1].wcode != W1) return false;
    rc = launch.template run<T, 2, W0, W1>(a, s);
    return true;
}

template <typename T, typename A, typename L>
static bool row_launch_pair(A &a, const L &launch, cudaStream_t s, int &rc) {
    auto is_sum = [](int w) { return w == W_ADD32 || w == W_ADD64 || w == W_ADDF || w == W_ADDF_COMP; };
    if (!is_sum(a.cl[0].wcode) && is_sum(a.cl[1].wcode)) {  // each clause carries its own output
        const ClauseDev t = a.cl[0];
        a.cl[0] = a.cl[1];
        a.cl[1] = t;
    }
    if constexpr (std::is_same<T, float>::value) {
        return pair_launch<T, W_ADDF, W_MAXF>(a, launch, s, rc) || pair_launch<T, W_ADDF, W_MINF>(a, launch, s, rc) ||
               pair_launch<T, W_ADDF_COMP, W_MAXF>(a, launch, s, rc) || pair_launch<T, W_ADDF_COMP, W_MINF>(a, launch, s, rc);
    } else if constexpr (std::is_same<T, double>::value) {
        return pair_launch<T, W_ADDF, W_MAXF>(a, launch, s, rc) || pair_launch<T, W_ADDF, W_MINF>(a, launch, s, rc);
    } else if constexpr (std::is_same<T, int32_t>::value) {
        return pair_launch<T, W_ADD32, W_MAXI>(a, launch, s, rc) || pair_launch<T, W_ADD32, W_MINI>(a, launch, s, rc) ||
               pair_launch<T, W_ADD64, W_MAXI>(a, launch, s, rc) || pair_launch<T, W_ADD64, W_MINI>(a, launch, s, rc);
    } else {
        return pair_launch<T, W_ADD64, W_MAXI>(a, launch, s, rc) || pair_launch<T, W_ADD64, W_MINI>(a, launch, s, rc);
    }
}

template <typename T, typename A, typename L>
static int row_launch(A &a, const L &launch, cudaStream_t s) {
    int rc = ACCR_OK;
    if (a.nc == 2 && row_launch_pair<T>(a, launch, s, rc)) return rc;
    switch (a.nc) {
    case 1: return launch.template run<T, 1, -1, -1>(a, s);
    case 2: return launch.template run<T, 2, -1, -1>(a, s);
    case 3: return launch.template run<T, 3, -1, -1>(a, s);
    default: return launch.template run<T, 4, -1, -1>(a, s);
    }
}

// The kernel of `launch` for an element type and the clauses of `a` (its `cl` and
// `nc`).
template <typename A, typename L>
static int row_dispatch(A &a, int in_type, const L &launch, cudaStream_t s) {
    switch (in_type) {
    case ACCR_I32: return row_launch<int32_t>(a, launch, s);
    case ACCR_I64: return row_launch<int64_t>(a, launch, s);
    case ACCR_F32: return row_launch<float>(a, launch, s);
    default: return row_launch<double>(a, launch, s);
    }
}

}  // namespace accr
