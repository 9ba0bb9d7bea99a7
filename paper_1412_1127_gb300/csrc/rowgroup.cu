// rowgroup.cu -- the row nest's short rows (at most GROUP_BYTES): a group of
// 1 to 32 neighbouring lanes folds a row.
//
// What bounds a short row is instructions, not bytes: a warp per row pays its
// address arithmetic, head, tail and five-step butterfly for every row (362
// warp instructions for 61 floats and two clauses).  Here a warp folds
// 32 / lanes rows at once and shares them, the butterfly has log2(lanes)
// steps, and every load of a row is in flight before any is folded.  The lane
// count follows the row's length alone, so a row's result does not depend on
// the matrix around it.
#include <string.h>

#include "common.cuh"
#include "debug.cuh"
#include "fold.cuh"
#include "group.cuh"
#include "overlap.cuh"
#include "rows.cuh"

namespace accr {

constexpr int WB = 256;  // threads per CTA

// Rows of at most GROUP_BYTES: p.lanes neighbouring lanes fold a row, so a
// warp takes 32 / p.lanes rows.
// GV: vectors a lane has at most.  400,000 rows of 61 floats (four a lane) take
// 26.7 us with eight and 20.8 us with four: half the predicates, 48 registers
// instead of 80.
template <typename T, int NC, int W0, int W1, int GV>
__global__ void __launch_bounds__(WB) rowgroup_kernel(const __grid_constant__ RowArgs p) {
    constexpr bool E64 = sizeof(T) == 8;
    constexpr int EPV = 16 / (int)sizeof(T);
    grid_wait();
    const int lane = threadIdx.x & 31, L = p.lanes;
    const int l = lane & (L - 1);
    const int rpw = 32 / L;  // rows per warp
    const int cols = (int)p.cols;
    const int rounds = (cols / EPV + L - 1) / L;  // at most GV
    int w[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) w[c] = (c == 0 && W0 >= 0) ? W0 : (c == 1 && W1 >= 0) ? W1 : p.cl[c].wcode;
    const int64_t step = (int64_t)gridDim.x * (WB / 32) * rpw;
    const int64_t first = ((int64_t)blockIdx.x * (WB / 32) + (threadIdx.x >> 5)) * rpw;
    // (released inside the loop, 400,000 rows of 61 took 22.1 us instead of 19.7; a longer
    // call's end releases)
    if (p.release_row <= 0) grid_release();
    for (int64_t rb = first; rb < p.rows; rb += step) {  // uniform across the warp
        const int64_t r = rb + lane / L;
        const bool live = r < p.rows;
        Acc A[NC];
        // rows past GROUP_BYTES / 2 (the launch picks GV so) have a vector in every lane
        group_fold<T, NC, W0, W1, GV, (GV > GROUP_GV / 2)>((const T *)p.A + (live ? r : rb) * p.ld, cols, live, l, L, rounds,
                                                           p.cl, p.neutral, w, A);
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (live && l == 0 && ACCR_DCHECK(r < p.rows, DS_ROW_VAR))
                store_var(p.cl[c], r, finish(p.cl[c], E64, cols == 0, to_final(w[c], A[c])));
    }
}

// ---- host side ---------------------------------------------------------------------

struct GroupLaunch {
    template <typename T, int NC, int W0, int W1, int GV>
    static void go(RowArgs &a, cudaStream_t s) {
        static std::atomic<int> cached[64];
        const int maxg = resident_ctas(rowgroup_kernel<T, NC, W0, W1, GV>, WB, cached);
        const int64_t per_cta = (int64_t)(WB / 32) * (32 / a.lanes);
        const int grid = clamp_grid((a.rows + per_cta - 1) / per_cta, maxg);
        launch_overlapped(rowgroup_kernel<T, NC, W0, W1, GV>, dim3((unsigned)grid), WB, 0, s, a);
    }
    template <typename T, int NC, int W0, int W1>
    int run(RowArgs &a, cudaStream_t s) const {
        int rc = launch_guard("rowgroup_kernel");
        if (rc != ACCR_OK) return rc;
        for (int c = 0; c < NC; ++c) a.neutral[c] = neutral_element<T>(a.cl[c].wcode);
        // longer rows than 2 KiB have more than four vectors a lane
        if (a.cols * (int64_t)sizeof(T) <= GROUP_BYTES / 2) go<T, NC, W0, W1, GROUP_GV / 2>(a, s);
        else go<T, NC, W0, W1, GROUP_GV>(a, s);
        return launched("rowgroup_kernel");
    }
};

int rowgroup_launch(RowArgs &a, int in_type, cudaStream_t s) {
    return row_dispatch(a, in_type, GroupLaunch{}, s);
}

}  // namespace accr
