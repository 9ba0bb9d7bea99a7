// rowreduce.cu -- the nest `for i (gang) { for j (vector) var_i (op)= A[i][j] }`:
// one reduction variable per row of a row-major matrix (the two-level loop
// shape of Listing 1a with an inner reduction; IPMACC Sec. 1.3, Stage 3.4).
//
// Mapping: gang -> CTA, worker -> warp, vector -> lane.  Lanes stream a stretch
// of a row in 16-byte vectors and merge through shuffles; a stretch whose start
// is not 16-byte aligned (ld not a multiple of the vector) folds its head and
// tail element by element.  Four forms, chosen by the row's length alone, so
// a row's result never depends on how many rows the matrix has:
//
//   * rows of at most GROUP_BYTES: a group of 1 to 32 neighbouring lanes
//     per row, about four vectors a lane, so a warp folds up to 32 rows at
//     once and every load of a row is in flight before any is folded.
//   * rows of at most WARP_ROW_BYTES: a warp per row, RU2 vectors in flight a
//     lane; lane 0 writes the row's variable, no cross-warp merge at all.
//   * rows shorter than SPLIT_ROW_BYTES: SEG_BYTES segments, each folded by a
//     warp, merged by one butterfly over the segments' partials (lane s holds
//     segment s).  With enough rows to fill the chip a warp takes its row's
//     segments in turn; with fewer, a CTA per row takes them at once.  Both
//     do the same operations in the same order.
//   * longer rows: the stretch is one of the row's SPLIT_CHUNK_BYTES chunks
//     (a few long rows then spread over every SM instead of a few warps).
//     The launch has one 1024-thread CTA per SM (256-thread CTAs, as many as
//     fit, where the fold needs more registers), and CTA b
//     takes the contiguous run [total b / G, total (b + 1) / G) of the
//     rows x cpr chunks, so every SM streams the same number of chunks to
//     within one; its 32 warps take the run's chunks in turn, so the warps
//     left with a last chunk are many and keep the SM's loads in flight.
//     Lane 0 stores each chunk's partial in the chunk's own slot; the CTA
//     then counts its chunks into each row it touched, and the CTA whose
//     count completes a row merges the row's partials in chunk order (thread
//     t takes chunks t, t + 1024 (or 256), ..., loads in flight, then the CTA's
//     shuffle and shared-memory tree) and writes the variable.  The partial
//     slots and the merge order depend on the row length and the clauses
//     only, not on which warp folded which chunk.
#include <string.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "debug.cuh"
#include "fold.cuh"
#include "group.cuh"
#include "overlap.cuh"
#include "rows.cuh"

namespace accr {


enum RowForm { ROW_SEG = 0, ROW_SPLIT = 1, ROW_SEG_CTA = 2 };

constexpr int WB = 256;  // threads per CTA of the group and warp-per-row forms
// Threads per CTA.  Split form: 1024 (one CTA per SM) where the fold fits 64
// registers (4-byte elements, one or two clauses), else 256 (as many CTAs per
// SM as the registers allow).  One-row CTAs of the segment form: at most 1024
// or 512, one warp per segment (the launch has no more warps than segments).
template <typename T, int NC, int FORM>
constexpr int row_threads() {
    return FORM == ROW_SPLIT     ? ((sizeof(T) == 4 && NC <= 2) ? 1024 : 256)
           : FORM == ROW_SEG_CTA ? ((sizeof(T) == 4 && NC <= 2) ? 1024 : 512)
                                 : WB;
}
constexpr int64_t WARP_ROW_BYTES = 16 * 1024;
constexpr int64_t SEG_BYTES = 8 * 1024;
constexpr int64_t SPLIT_ROW_BYTES = 256 * 1024;
constexpr int64_t SPLIT_CHUNK_BYTES = 32 * 1024;
static_assert(SPLIT_ROW_BYTES / SEG_BYTES <= 32, "a row's segments fit one warp's lanes");
// Segment form: below this many rows per SM a CTA takes each row (a warp per
// row keeps 4 KiB in flight; 24 warps an SM are past what HBM needs).
constexpr int64_t SEG_WARP_ROWS_PER_SM = 24;

__device__ __forceinline__ Partial ld_row_partial(const Partial *p) {
    uint4 v = __ldcg(reinterpret_cast<const uint4 *>(p));
    Partial q;
    q.a = ((uint64_t)v.y << 32) | v.x;
    q.c = __uint_as_float(v.z);
    q.pad = 0;
    return q;
}

// W0 / W1 >= 0 fix the working codes of clauses 0 / 1 at compile time (the
// fold's operator switch then disappears from the row loop); -1 reads them
// from the arguments.  FORM: see the top of the file.
template <typename T, int NC, int W0 = -1, int W1 = -1, int FORM = ROW_SEG>
__global__ void __launch_bounds__(row_threads<T, NC, FORM>()) rowreduce_kernel(const __grid_constant__ RowArgs p) {
    constexpr bool E64 = sizeof(T) == 8, FIXED = W0 >= 0;
    constexpr int NTH = row_threads<T, NC, FORM>(), NW = NTH / 32;
    grid_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * NW + warp;
    const int64_t cols = p.cols;
    int w[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) w[c] = (c == 0 && W0 >= 0) ? W0 : (c == 1 && W1 >= 0) ? W1 : p.cl[c].wcode;
    Acc A[NC];

    if (FORM == ROW_SEG || FORM == ROW_SEG_CTA) {
        // The partial of segment s goes to lane s (identity past the last), in
        // the code of the final merge, and one butterfly merges the lanes.
        const int nseg = (int)p.cpr;
        __shared__ Acc seg[NC][FORM == ROW_SEG_CTA ? 32 : 1];
        Acc P[NC];
        int fw[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) fw[c] = final_code(w[c]);
        const int64_t step = FORM == ROW_SEG ? (int64_t)gridDim.x * NW : (int64_t)gridDim.x;
        for (int64_t r = FORM == ROW_SEG ? gw : (int64_t)blockIdx.x; r < p.rows; r += step) {
            if (r >= p.release_row) grid_release();
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                P[c].a = final_ident(p.cl[c]);
                P[c].c = 0.f;
            }
            const int s0 = FORM == ROW_SEG ? 0 : warp, ds = FORM == ROW_SEG ? 1 : (int)(blockDim.x >> 5);
            for (int s = s0; s < nseg; s += ds) {
                const int64_t lo = s * p.chunk;
                const int64_t len = (cols - lo) < p.chunk ? (cols - lo) : p.chunk;
                if (!ACCR_DCHECK(lo + len <= cols && s < 32, DS_ROW_CHUNK)) continue;
                fold_stretch<T, NC, FIXED>((const T *)p.A + r * p.ld + lo, len, p.cl, w, lane, A);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (FORM == ROW_SEG) {
                        const Acc F = to_final(w[c], A[c]);
                        if (lane == s) P[c] = F;
                    } else if (lane == 0) {
                        seg[c][s] = to_final(w[c], A[c]);
                    }
                }
            }
            if (FORM == ROW_SEG_CTA) {
                __syncthreads();
                if (warp == 0 && lane < nseg) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) P[c] = seg[c][lane];
                }
                __syncthreads();  // the next row's partials may follow
                if (warp != 0) continue;
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (nseg > 1) warp_merge<FIXED>(fw[c], E64, P[c]);
                if (lane == 0 && ACCR_DCHECK(r < p.rows, DS_ROW_VAR))
                    store_var(p.cl[c], r, finish(p.cl[c], E64, cols == 0, P[c]));
            }
        }
        return;
    }
    // this CTA's run of the rows x cpr chunks, its warps taking them in turn
    __shared__ Acc sh[NC][NW];
    const int64_t total = p.rows * p.cpr;
    const int64_t c0 = total * (int64_t)blockIdx.x / gridDim.x, c1 = total * ((int64_t)blockIdx.x + 1) / gridDim.x;
    for (int64_t k = c0 + warp; k < c1; k += NW) {
        if ((c1 - k) * gridDim.x <= RELEASE_BYTES / SPLIT_CHUNK_BYTES) grid_release();
        const int64_t r = k / p.cpr, j = k - r * p.cpr, lo = j * p.chunk;
        const int64_t len = (cols - lo) < p.chunk ? (cols - lo) : p.chunk;
        if (!ACCR_DCHECK(r < p.rows && lo + len <= cols, DS_ROW_CHUNK)) continue;
        fold_stretch<T, NC, FIXED>((const T *)p.A + r * p.ld + lo, len, p.cl, w, lane, A);
        if (lane == 0) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                Partial q;
                q.a = A[c].a;
                q.c = A[c].c;
                q.pad = 0;
                if (ACCR_DCHECK((r * NC + c) * p.cpr + j < p.rows * NC * p.cpr, DS_ROW_PARTIAL))
                    p.partials[(r * NC + c) * p.cpr + j] = q;
            }
        }
    }
    // the CTA counts its chunks into each row it touched, thread t into row
    // r0 + t (an acquire-release add: it releases the CTA's partials, which
    // the barrier before it ordered, and the add that completes a row
    // acquires every other CTA's); the CTA then merges each row it completed
    // in chunk order (thread t takes chunks t, t + NTH, ..., loads in flight,
    // then the CTA tree)
    __shared__ int64_t s_rows[NTH];
    __shared__ int s_nd;
    __syncthreads();
    if (c0 >= c1) return;  // uniform across the CTA
    const int64_t r0 = c0 / p.cpr, r1 = (c1 - 1) / p.cpr;
    for (int64_t rb = r0; rb <= r1; rb += NTH) {
        if (threadIdx.x == 0) s_nd = 0;
        __syncthreads();
        const int64_t r = rb + threadIdx.x;
        if (r <= r1 && ACCR_DCHECK(r < p.rows, DS_ROW_COUNTER)) {
            const int64_t a = (r * p.cpr > c0 ? r * p.cpr : c0), b = ((r + 1) * p.cpr < c1 ? (r + 1) * p.cpr : c1);
            unsigned old;
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;"
                         : "=r"(old)
                         : "l"(&p.counters[r]), "r"((unsigned)(b - a))
                         : "memory");
            if (old + (unsigned)(b - a) == (unsigned)p.cpr) s_rows[atomicAdd(&s_nd, 1)] = r;
        }
        __syncthreads();
        const int nd = s_nd;
        for (int iq = 0; iq < nd; ++iq) {
            const int64_t rr = s_rows[iq];
            int fw[NC];
            uint64_t fid[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                fw[c] = final_code(w[c]);
                fid[c] = final_ident(p.cl[c]);
                A[c].a = fid[c];
                A[c].c = 0.f;
            }
            constexpr int U = NC == 1 ? 4 : NC == 2 ? 2 : 1;  // loads in flight per clause and thread
            for (int64_t b0 = threadIdx.x; b0 < p.cpr; b0 += (int64_t)NTH * U) {
                Partial q[NC][U];
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (b0 + u * NTH < p.cpr)
                            q[c][u] = ld_row_partial(&p.partials[(rr * NC + c) * p.cpr] + b0 + u * NTH);
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (b0 + u * NTH < p.cpr) {
                            Acc Q;
                            Q.a = q[c][u].a;
                            Q.c = q[c][u].c;
                            merge(fw[c], E64, A[c], to_final(w[c], Q));
                        }
                    }
            }
            cta_merge<NC, NTH, FIXED>(fw, fid, E64, A, sh);
            if (threadIdx.x == 0) {
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (ACCR_DCHECK(rr < p.rows, DS_ROW_VAR))
                        store_var(p.cl[c], rr, finish(p.cl[c], E64, cols == 0, A[c]));
                p.counters[rr] = 0u;
            }
            __syncthreads();
        }
    }
}

// ---- host side ---------------------------------------------------------------------

template <typename T, int NC, int W0, int W1, int FORM>
static void row_form(const RowArgs &a, cudaStream_t s) {
    static std::atomic<int> cached[64];
    constexpr int NTH = row_threads<T, NC, FORM>();
    auto kernel = rowreduce_kernel<T, NC, W0, W1, FORM>;
    if (FORM == ROW_SEG_CTA) {  // a CTA per row, a warp per segment
        const int nt = a.cpr * 32 < NTH ? (int)a.cpr * 32 : NTH;
        launch_overlapped(kernel, dim3((unsigned)a.rows), nt, 0, s, a);
        return;
    }
    const int maxg = resident_ctas(kernel, NTH, cached);
    // chunks of long rows: at most one CTA per chunk, each taking a contiguous
    // run; else a warp per row, rows past the resident grid in later rounds
    const int64_t want = FORM == ROW_SPLIT ? a.rows * a.cpr : (a.rows + NTH / 32 - 1) / (NTH / 32);
    launch_overlapped(kernel, dim3((unsigned)clamp_grid(want, maxg)), NTH, 0, s, a);
}

template <typename T, int NC, int W0, int W1>
static int row_launch_t(RowArgs &a, int form, cudaStream_t s) {
    int rc = launch_guard("rowreduce_kernel");
    if (rc != ACCR_OK) return rc;
    if (form == ROW_SPLIT) row_form<T, NC, W0, W1, ROW_SPLIT>(a, s);
    else if (form == ROW_SEG) row_form<T, NC, W0, W1, ROW_SEG>(a, s);
    else row_form<T, NC, W0, W1, ROW_SEG_CTA>(a, s);
    return launched("rowreduce_kernel");
}

struct RowLaunch {
    int form;
    template <typename T, int NC, int W0, int W1>
    int run(RowArgs &a, cudaStream_t s) const {
        return row_launch_t<T, NC, W0, W1>(a, form, s);
    }
};

int rowgroup_launch(RowArgs &a, int in_type, cudaStream_t s);  // rowgroup.cu

}  // namespace accr

using namespace accr;

extern "C" ACCR_API int accr_rowreduce(const void *A, int64_t rows, int64_t cols, int64_t ld, int32_t in_type,
                              const accr_clause *clauses, int32_t nclauses, uint32_t flags,
                              accr_stream_t stream) {
    ACCR_TRACE("accr_rowreduce");
    clear_error();
    if (flags & ~(ACCR_COMPENSATED | ACCR_SYNC))
        return set_error(ACCR_EINVAL, "accr_rowreduce: unsupported flags 0x%x", flags);
    if (rows < 0 || cols < 0) return set_error(ACCR_EINVAL, "accr_rowreduce: negative size");
    if (ld < cols) return set_error(ACCR_EINVAL, "accr_rowreduce: ld = %lld < cols = %lld", (long long)ld, (long long)cols);
    ClauseDev cl[ACCR_MAX_CLAUSES];
    int rc = lower_clauses(in_type, clauses, nclauses, flags, cl);
    if (rc != ACCR_OK) return rc;
    if (rows == 0) return ACCR_OK;
    if (cols > 0 && !A) return set_error(ACCR_EINVAL, "accr_rowreduce: A is NULL");
    if (((uintptr_t)A % (uintptr_t)type_bytes(in_type)) != 0)
        return set_error(ACCR_EINVAL, "accr_rowreduce: A is not aligned to its element size");
    cudaStream_t s = (cudaStream_t)stream;
    RowArgs a;
    memset(&a, 0, sizeof a);
    const int64_t eb = type_bytes(in_type), row_bytes = cols * eb;
    int form = ROW_SEG;
    if (row_bytes <= GROUP_BYTES) {
        // about four vectors a lane: fewer leave lanes idle and pay more
        // shuffles a row, more lengthen each lane's chain
        a.lanes = 1;
        while (a.lanes < 32 && a.lanes * 4 * 16 < row_bytes) a.lanes *= 2;
    } else if (row_bytes >= SPLIT_ROW_BYTES) {
        // chunked form: partials [rows][nclauses][cpr] and one counter per row
        form = ROW_SPLIT;
        a.chunk = SPLIT_CHUNK_BYTES / eb;
        a.cpr = (cols + a.chunk - 1) / a.chunk;
        const size_t pbytes = (size_t)rows * (size_t)nclauses * (size_t)a.cpr * sizeof(Partial);
        Scratch *scr = scratch_for(stream, pbytes);
        if (!scr) return ACCR_ENOMEM;
        a.partials = (Partial *)scr->buf;
        a.counters = zeroed_words_for(stream, (size_t)rows);  // every row completes, so each returns to zero
        if (!a.counters) return ACCR_ENOMEM;
    } else if (row_bytes > WARP_ROW_BYTES) {
        form = rows < SEG_WARP_ROWS_PER_SM * device_info().sms ? ROW_SEG_CTA : ROW_SEG;
        a.chunk = SEG_BYTES / eb;
        a.cpr = (cols + a.chunk - 1) / a.chunk;
    } else {
        a.chunk = cols;  // one stretch, no merge of segments
        a.cpr = 1;
    }
    static const char *const names[] = {"warp per row", "split rows", "CTA per row"};
    log_msg(2, "accr_rowreduce: %lld x %lld (ld %lld) type=%d clauses=%d form=%s", (long long)rows, (long long)cols,
            (long long)ld, in_type, nclauses, a.lanes > 0 ? "lane group per row" : names[form]);
    a.A = A;
    a.rows = rows;
    a.cols = cols;
    a.ld = ld;
    a.nc = nclauses;
    a.release_row = rows - RELEASE_BYTES / (row_bytes > 0 ? row_bytes : 1);
    for (int c = 0; c < nclauses; ++c) a.cl[c] = cl[c];
    rc = a.lanes > 0 ? rowgroup_launch(a, in_type, s) : row_dispatch(a, in_type, RowLaunch{form}, s);
    if (rc != ACCR_OK) return rc;
    if (flags & ACCR_SYNC) return cuda_check(cudaStreamSynchronize(s), "accr_rowreduce: sync");
    return ACCR_OK;
}
