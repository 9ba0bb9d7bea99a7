// patterns.cu -- three region patterns from the paper's application study
// (IPMACC Sec. 4.2), on the same single-pass reduction machinery:
//
//  * Nearest Neighbor: distances to a query point and the k smallest -- a
//    reduction whose operator keeps a sorted list of k (distance, index)
//    pairs.  The scan keeps each thread's nearest point; the last CTA to finish
//    takes a bound from those and looks again at the few threads' points that
//    can be among the k nearest.
//
//  * SRAD: a reduction region whose result feeds a data-parallel region.  The
//    paper's OpenACC code merges the block partials on the CPU and launches
//    the next region; here one cooperative launch does both: every CTA passes a
//    bounded grid barrier, merges the partials and runs the elementwise pass,
//    with what its threads read last still in registers and the rest, as far as
//    it fits, in L2.  Unfused and two-level host forms are kept for comparison.
//
//  * BFS: a level-synchronous loop that stops when no cell changed.  The
//    OpenACC version reduces a global boolean with ||; the CUDA version
//    initialises the flag and lets threads write only `true`.  Both forms run
//    here with the host driving the levels, and a third keeps every level in
//    one cooperative launch: on bitmaps, in tiles whose halo lets a CTA run
//    several levels between two bounded grid barriers.
//
// Every cross-CTA wait spins a bounded number of times; on expiry it records
// a code in a status word and the host reports ACCR_ETIMEDOUT.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "common.cuh"
#include "debug.cuh"
#include "fold.cuh"
#include "overlap.cuh"

namespace accr {

constexpr uint32_t kSpinLimit = 20000000u;  // ~seconds of __nanosleep(64) polls

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid barrier for a cooperative launch that also ORs one CTA-uniform flag:
// generation counting, bounded spin.  `ctas` CTAs take part.  bar[0] counts
// arrivals (low 20 bits) and raised flags (bits 20 and up); bar[1] holds
// (generation << 1) | OR of the flags, published by the last CTA to arrive, so
// the flag comes back with the release instead of through a word of its own.
// Returns 0 if the wait ran out, else 1 + the OR of the flags.
//
// Whether bar[1] shows generation `gen` or one after it.  CTAs that take part in
// the following barrier keep the word from moving on before they have seen it; one
// that does not (it only set up) may look late and find a later generation, which
// must end its wait too (the flag it then reads is not its barrier's: it has no use
// for it).
__host__ __device__ __forceinline__ bool generation_reached(unsigned word, unsigned gen) {
    return (((word >> 1) - gen) & 0x7fffffffu) < 0x40000000u;
}
__device__ __forceinline__ int grid_barrier_or(unsigned *bar, unsigned &gen, bool flag, unsigned ctas) {
    __shared__ int s_res;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned my = (gen + 1) & 0x7fffffffu;
        __threadfence();
        const unsigned old = atomicAdd(&bar[0], 1u + (flag ? (1u << 20) : 0u));
        int res = 0;
        if ((old & 0xfffffu) == ctas - 1) {
            const unsigned any = ((old >> 20) != 0u || flag) ? 1u : 0u;
            bar[0] = 0u;
            st_release(&bar[1], (my << 1) | any);
            res = 1 + (int)any;
        } else {
            uint32_t i = 0;
            unsigned v = ld_acquire(&bar[1]);
            while (!generation_reached(v, my) && ++i <= kSpinLimit) {
                if (i > 256) __nanosleep(64);
                v = ld_acquire(&bar[1]);
            }
            if (generation_reached(v, my)) res = 1 + (int)(v & 1u);
        }
        s_res = res;
    }
    gen = (gen + 1) & 0x7fffffffu;
    __syncthreads();
    return s_res;
}

// ============================================================================
// Nearest Neighbor: k smallest squared distances
// ============================================================================
//
// One plain launch, no CTA waits for another.  The scan keeps one thing per
// thread, its nearest point, so it runs at the rate of its loads: lists of k per
// warp cost it an insertion path, a merge of the lists per CTA and a k-round
// tournament at the end (10 million points, k = 10: 42 us against the 11.8 us
// their bytes take).  The k nearest are then found by the last CTA to finish:
//
//   * the k-th nearest of its 16 warps' shares of the warps' nearest points is a
//     bound that at least k points reach;
//   * a thread that holds one of the k nearest points has a nearest point within
//     the bound, so only such threads' points are looked at again -- a few dozen
//     threads of the 150,000, some hundred points each -- and the points within
//     the bound become candidates;
//   * the candidates are ranked by (distance, index).  If there are ever more
//     than the array holds, the k best of them stay and the k-th is the new bound.
//
// The shares' bound is loose where the points' order keeps the near ones in a few
// of them (a raster 1,024 wide holds a range of columns in each).  Where many warps
// are within it, the k-th nearest of all warps' points takes its place, and where many
// threads are left, the k-th nearest of theirs: k rounds of a minimum over the CTA each.
// 1024 x 1024 raster points, k = 10: 24 us (445 with the shares alone, 8.6 shuffled),
// 9766 x 1024 32 (600, 16.5).
//
// Distances are never negative, so their bits order as unsigned integers, with
// a NaN above infinity: NK_NONE, one above infinity, is "no point yet", and a
// point whose distance is NaN never enters.  Ten million points, k = 10: 42 -> 22.8 us,
// of which the bytes take 11.8 and the last CTA about 6.

constexpr int NK_THREADS = 512;               // two CTAs per SM
constexpr int NK_WARPS = NK_THREADS / 32;
constexpr int NK_U = 8;                       // 16-byte vectors (two points each) a thread and round
constexpr uint32_t NK_NONE = 0x7f800001u;
constexpr int NK_BATCH = 64;                  // warps whose threads are looked at together
constexpr int NK_CAND = 1536;                 // candidates held: one pass adds at most 64 a warp
constexpr int NK_LOOSE = 2 * NK_BATCH;        // more warps than this within the bound: it is tightened
constexpr int NK_PASSES = 8;                  // and so it is before more passes than this
constexpr int NK_MAX_WARPS = 5120;            // warps of the scan (the grid is bounded accordingly: 320 CTAs)

struct __align__(16) PairSlot {
    int64_t i;
    uint32_t d;
    uint32_t pad;
};

// (distance bits, index) order
__device__ __forceinline__ bool pless(uint32_t da, int64_t ia, uint32_t db, int64_t ib) {
    return da < db || (da == db && ia < ib);
}

// Two points.
__device__ __forceinline__ float4 ld_pts(const float4 *p) {
    const uint4 v = ld_stream(reinterpret_cast<const uint4 *>(p));
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

__device__ __forceinline__ uint32_t sqdist(float x, float y, float qx, float qy) {
    const float dx = __fsub_rn(x, qx), dy = __fsub_rn(y, qy);
    return __float_as_uint(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)));  // no fused multiply-add
}

// The smallest (distance, index) pair of a warp, in every lane.
__device__ __forceinline__ void warp_min_pair(uint32_t &d, int64_t &i) {
    const uint32_t m = __reduce_min_sync(0xffffffffu, d);
    uint64_t j = d == m ? (uint64_t)i : ~0ull >> 1;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const uint64_t o = __shfl_xor_sync(0xffffffffu, (unsigned long long)j, s);
        j = o < j ? o : j;
    }
    d = m;
    i = (int64_t)j;
}

struct NearestArgs {
    const float *pts;
    int64_t n;
    float qx, qy;
    int k;
    int64_t *idx_out;
    float *d_out;
    uint32_t *tmin;     // [threads] each thread's smallest distance
    PairSlot *wmin;     // [warps] each warp's nearest point
    unsigned *counter;  // zero on entry and exit
    int threads;        // of the scan: slots of tmin, 32 for each of wmin
};

struct NearestShared {
    uint16_t warps[NK_MAX_WARPS];
    uint32_t units[NK_BATCH * 32], ud[NK_BATCH * 32];  // threads to look at, their smallest distances
    int64_t ci[NK_CAND];
    uint32_t cd[NK_CAND];
    int64_t gi[NK_WARPS];
    uint32_t gd[NK_WARPS];
    int nwarps, nunits, ncand;
    int64_t bi;   // the bound
    uint32_t bd;
};

__device__ __forceinline__ void nk_offer(NearestShared &s, bool ok, uint32_t d, int64_t i, uint32_t bd, int64_t bi) {
    if (ok && d < NK_NONE && !pless(bd, bi, d, i)) {
        const int at = atomicAdd(&s.ncand, 1);
        if (ACCR_DCHECK(at < NK_CAND, DS_NEAREST_SLOT)) {
            s.cd[at] = d;
            s.ci[at] = i;
        }
    }
}

// Rank of candidate c among the first n (distinct points: no two are equal).
__device__ __forceinline__ int nk_rank(const NearestShared &s, int c, int n) {
    const uint32_t d = s.cd[c];
    const int64_t i = s.ci[c];
    int r = 0;
    for (int o = 0; o < n; ++o) r += pless(s.cd[o], s.ci[o], d, i) ? 1 : 0;
    return r;
}

// The k-th smallest of the CTA's (distance, index) pairs, N a thread, all different
// (NK_NONE: none; there are at least k): k rounds, each the smallest pair past the last.
template <int N>
__device__ __forceinline__ void nk_kth(NearestShared &s, const uint32_t (&dv)[N], const int64_t (&iv)[N], int k, uint32_t &kd,
                                       int64_t &ki) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    kd = 0u, ki = -1;
    for (int r = 0; r < k; ++r) {
        uint32_t d = NK_NONE;
        int64_t i = INT64_MAX;
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (pless(kd, ki, dv[j], iv[j]) && pless(dv[j], iv[j], d, i)) d = dv[j], i = iv[j];
        warp_min_pair(d, i);
        if (lane == 0) s.gd[warp] = d, s.gi[warp] = i;
        __syncthreads();
        kd = s.gd[lane % NK_WARPS], ki = s.gi[lane % NK_WARPS];
        warp_min_pair(kd, ki);
        __syncthreads();
    }
}

// A warp's nearest point, as the scan stored it.
__device__ __forceinline__ void nk_warp_min(const NearestArgs &p, int w, uint32_t &d, int64_t &i) {
    const int W = (int)gridDim.x * NK_WARPS;
    const uint4 r = w < W ? __ldcg(reinterpret_cast<const uint4 *>(p.wmin + w)) : make_uint4(~0u, ~0u >> 1, NK_NONE, 0u);
    d = r.z;
    i = (int64_t)(((uint64_t)r.y << 32) | r.x);
}

// The two tightenings, out of line: few calls need them, and their code in the
// select's own cost every call 0.3 us.
__device__ __noinline__ void nk_tighten_warps(const NearestArgs &p, NearestShared &s) {
    constexpr int NW = NK_MAX_WARPS / NK_THREADS;
    const int t = threadIdx.x;
    uint32_t wd[NW], d;
    int64_t wi[NW], i;
#pragma unroll
    for (int j = 0; j < NW; ++j) nk_warp_min(p, t + j * NK_THREADS, wd[j], wi[j]);
    nk_kth(s, wd, wi, p.k, d, i);
    if (t == 0) s.nwarps = 0, s.bd = d, s.bi = i;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NW; ++j)
        if (wd[j] < NK_NONE && !pless(d, i, wd[j], wi[j])) s.warps[atomicAdd(&s.nwarps, 1)] = (uint16_t)(t + j * NK_THREADS);
    __syncthreads();
}

__device__ __noinline__ void nk_tighten_units(const NearestArgs &p, NearestShared &s) {
    constexpr int N = NK_BATCH * 32 / NK_THREADS;
    const int t = threadIdx.x, nu = s.nunits;
    uint32_t ud[N], un[N], d;
    int64_t at[N], i;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const int c = t + j * NK_THREADS;
        un[j] = c < nu ? s.units[c] : 0u;
        ud[j] = c < nu ? s.ud[c] : NK_NONE;
        at[j] = c < nu ? (int64_t)c : INT64_MAX;
    }
    nk_kth(s, ud, at, p.k, d, i);
    if (t == 0) {
        s.nunits = 0;
        if (d < s.bd) s.bd = d, s.bi = INT64_MAX;  // k points within d
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (ud[j] < NK_NONE && ud[j] <= s.bd) s.units[atomicAdd(&s.nunits, 1)] = un[j];
    __syncthreads();
}

// The last CTA: the k nearest of all points, from the threads' nearest ones.
__device__ __noinline__ void nearest_select(const NearestArgs &p, NearestShared &s) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t head = (((uintptr_t)p.pts & 15) != 0 && p.n > 0) ? 1 : 0;
    const float4 *v4 = (const float4 *)(p.pts + 2 * head);
    const int64_t npairs = (p.n - head) / 2, last = head + 2 * npairs;
    const int64_t rstep = (int64_t)gridDim.x * NK_THREADS * NK_U;
    // the bound: the k-th of the warps' shares (scan warp w belongs to warp w % 16
    // here); all of a thread's loads in flight, and kept
    constexpr int NW = NK_MAX_WARPS / NK_THREADS;
    uint32_t wd[NW];
    int64_t wi[NW];
    uint32_t d = NK_NONE;
    int64_t i = INT64_MAX;
#pragma unroll
    for (int j = 0; j < NW; ++j) nk_warp_min(p, warp + NK_WARPS * lane + j * NK_THREADS, wd[j], wi[j]);
#pragma unroll
    for (int j = 0; j < NW; ++j)
        if (pless(wd[j], wi[j], d, i)) d = wd[j], i = wi[j];
    warp_min_pair(d, i);
    if (lane == 0) s.gd[warp] = d, s.gi[warp] = i;
    if (t == 0) s.nwarps = 0, s.ncand = 0, s.bd = NK_NONE, s.bi = INT64_MAX;
    __syncthreads();
    if (t < NK_WARPS) {  // k <= 16 shares; fewer with a point: no bound
        const uint32_t gd = s.gd[t];
        const int64_t gi = s.gi[t];
        int r = 0;
#pragma unroll
        for (int o = 0; o < NK_WARPS; ++o) r += (pless(s.gd[o], s.gi[o], gd, gi)) ? 1 : 0;
        if (gd < NK_NONE && r == p.k - 1) s.bd = gd, s.bi = gi;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NW; ++j)
        if (wd[j] < NK_NONE && !pless(s.bd, s.bi, wd[j], wi[j]))
            s.warps[atomicAdd(&s.nwarps, 1)] = (uint16_t)(warp + NK_WARPS * lane + j * NK_THREADS);
    __syncthreads();
    if (s.nwarps > NK_LOOSE) nk_tighten_warps(p, s);  // the same for all threads; so many warps with a point are at least k
    const int nwarps = s.nwarps;
    const int64_t rounds = npairs > 0 ? (npairs + rstep - 1) / rstep : 1;
    const int64_t nvec = rounds * NK_U, chunks = (nvec + 31) / 32;  // a thread's vectors, 32 to a pass of a warp
    for (int b0 = 0; b0 < nwarps; b0 += NK_BATCH) {
        if (t == 0) s.nunits = 0;
        __syncthreads();
        for (int b = b0 + warp; b < nwarps && b < b0 + NK_BATCH; b += NK_WARPS) {
            const uint32_t u = (uint32_t)s.warps[b] * 32u + lane;
            const uint32_t du = __ldcg(p.tmin + u);
            if (du < NK_NONE && du <= s.bd) {
                const int at = atomicAdd(&s.nunits, 1);
                if (ACCR_DCHECK(at < NK_BATCH * 32, DS_NEAREST_SLOT)) s.units[at] = u, s.ud[at] = du;
            }
        }
        __syncthreads();
        if (s.nunits > p.k && s.nunits * chunks > NK_PASSES * NK_WARPS) nk_tighten_units(p, s);
        const int64_t tasks = s.nunits * chunks;
        for (int64_t t0 = 0; t0 < tasks; t0 += NK_WARPS) {
            const int n = s.ncand;
            __syncthreads();                       // every thread has the same count
            if (n > NK_CAND - NK_WARPS * 68) {     // no room for a pass
                for (int c = t; c < n; c += NK_THREADS) {
                    const int r = nk_rank(s, c, n);
                    if (r < p.k) s.gd[r] = s.cd[c], s.gi[r] = s.ci[c];
                }
                __syncthreads();
                if (t < p.k) s.cd[t] = s.gd[t], s.ci[t] = s.gi[t];
                if (t == 0) s.ncand = p.k, s.bd = s.gd[p.k - 1], s.bi = s.gi[p.k - 1];
                __syncthreads();
            }
            const uint32_t bd = s.bd;
            const int64_t bi = s.bi, task = t0 + warp;
            if (task < tasks) {
                const uint32_t u = s.units[task / chunks];
                const int64_t j = (task % chunks) * 32 + lane;  // vector of the thread
                const int64_t v = (int64_t)(u / NK_THREADS) * (NK_THREADS * NK_U) + (u % NK_THREADS) +
                                  (j % NK_U) * NK_THREADS + (j / NK_U) * rstep;
                const bool ok = j < nvec && v < npairs;
                const float4 q = ok ? ld_pts(v4 + v) : make_float4(0.f, 0.f, 0.f, 0.f);
                nk_offer(s, ok, sqdist(q.x, q.y, p.qx, p.qy), head + 2 * v, bd, bi);
                nk_offer(s, ok, sqdist(q.z, q.w, p.qx, p.qy), head + 2 * v + 1, bd, bi);
                if (j == 0 && u == 0 && head) nk_offer(s, true, sqdist(p.pts[0], p.pts[1], p.qx, p.qy), 0, bd, bi);
                if (j == 0 && u == 1 && last < p.n)
                    nk_offer(s, true, sqdist(p.pts[2 * last], p.pts[2 * last + 1], p.qx, p.qy), last, bd, bi);
            }
            __syncthreads();
        }
    }
    const int n = s.ncand;
    for (int c = t; c < n; c += NK_THREADS) {
        const int r = nk_rank(s, c, n);
        if (r < p.k && ACCR_DCHECK(p.k <= 16, DS_NEAREST_OUT)) {
            p.idx_out[r] = s.ci[c];
            p.d_out[r] = __uint_as_float(s.cd[c]);
        }
    }
    if (t >= n && t < p.k) {  // fewer points than k
        p.idx_out[t] = -1;
        p.d_out[t] = INFINITY;
    }
}

__global__ void __launch_bounds__(NK_THREADS, 2) nearest_kernel(const __grid_constant__ NearestArgs p) {
    __shared__ NearestShared s;
    __shared__ int am_last;
    grid_wait();
    const int t = threadIdx.x, lane = t & 31;
    // points are float2; the vector part starts at a 16-byte boundary
    const int64_t head = (((uintptr_t)p.pts & 15) != 0 && p.n > 0) ? 1 : 0;
    const float4 *v4 = (const float4 *)(p.pts + 2 * head);
    const int64_t npairs = (p.n - head) / 2, last = head + 2 * npairs;
    uint32_t bd = NK_NONE;
    int64_t bi = INT64_MAX;
    if (blockIdx.x == 0 && t == 0 && head) {  // the unaligned first point
        const uint32_t d = sqdist(p.pts[0], p.pts[1], p.qx, p.qy);
        if (d < bd) bd = d, bi = 0;
    }
    // A round's smallest distance first (one compare with the thread's); only a
    // round that beats it looks for its first point with that distance.
    int64_t v = (int64_t)blockIdx.x * (NK_THREADS * NK_U) + t;
    const int64_t step = (int64_t)gridDim.x * (NK_THREADS * NK_U);
    constexpr int H = NK_U / 2;
    auto half = [&](const float4 (&q)[H], int64_t v0) {
        uint32_t m = NK_NONE;
#pragma unroll
        for (int u = 0; u < H; ++u)
            m = min(m, min(sqdist(q[u].x, q[u].y, p.qx, p.qy), sqdist(q[u].z, q[u].w, p.qx, p.qy)));
        if (m < bd) {
            bd = m;
            int j = 0;
#pragma unroll
            for (int u = H - 1; u >= 0; --u) {
                if (sqdist(q[u].z, q[u].w, p.qx, p.qy) == m) j = 2 * u + 1;
                if (sqdist(q[u].x, q[u].y, p.qx, p.qy) == m) j = 2 * u;
            }
            bi = head + 2 * (v0 + (j >> 1) * NK_THREADS) + (j & 1);
        }
    };
    if (v + (NK_U - 1) * NK_THREADS < npairs) {  // full rounds, in halves: one is folded while the other loads
        float4 a[H], b[H];
#pragma unroll
        for (int u = 0; u < H; ++u) a[u] = ld_pts(v4 + v + u * NK_THREADS);
#pragma unroll
        for (int u = 0; u < H; ++u) b[u] = ld_pts(v4 + v + (H + u) * NK_THREADS);
        for (v += step; v + (NK_U - 1) * NK_THREADS < npairs; v += step) {
            half(a, v - step);
#pragma unroll
            for (int u = 0; u < H; ++u) a[u] = ld_pts(v4 + v + u * NK_THREADS);
            half(b, v - step + H * NK_THREADS);
#pragma unroll
            for (int u = 0; u < H; ++u) b[u] = ld_pts(v4 + v + (H + u) * NK_THREADS);
        }
        half(a, v - step);
        half(b, v - step + H * NK_THREADS);
    }
    if (v < npairs) {  // the last, partial round: loads in flight together
        float4 q[NK_U];
#pragma unroll
        for (int u = 0; u < NK_U; ++u)
            if (v + u * NK_THREADS < npairs) q[u] = ld_pts(v4 + v + u * NK_THREADS);
#pragma unroll
        for (int u = 0; u < NK_U; ++u) {
            if (v + u * NK_THREADS < npairs) {
                const uint32_t d0 = sqdist(q[u].x, q[u].y, p.qx, p.qy), d1 = sqdist(q[u].z, q[u].w, p.qx, p.qy);
                const int64_t i = head + 2 * (v + u * NK_THREADS);
                if (d0 < bd) bd = d0, bi = i;
                if (d1 < bd) bd = d1, bi = i + 1;
            }
        }
    }
    if (blockIdx.x == 0 && t == 1 && last < p.n) {  // the odd last point
        const uint32_t d = sqdist(p.pts[2 * last], p.pts[2 * last + 1], p.qx, p.qy);
        if (d < bd) bd = d, bi = last;
    }
    grid_release();  // the points are read: minima, and the last CTA's select, are left
    const int gt = (int)blockIdx.x * NK_THREADS + t;
    if (ACCR_DCHECK(gt < p.threads, DS_NEAREST_SLOT)) p.tmin[gt] = bd;
    warp_min_pair(bd, bi);
    if (lane == 0) {
        PairSlot w;
        w.i = bi;
        w.d = bd;
        w.pad = 0;
        if (ACCR_DCHECK(gt < p.threads, DS_NEAREST_SLOT)) p.wmin[gt >> 5] = w;
    }
    __syncthreads();
    if (t == 0) {
        __threadfence();
        am_last = atomicAdd(p.counter, 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    nearest_select(p, s);
    if (t == 0) *p.counter = 0u;
}

static int nearest_launch(const float *pts, int64_t n, float qx, float qy, int k, int64_t *idx, float *d,
                          cudaStream_t s) {
    static int per_sm = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, nearest_kernel, NK_THREADS, 0);
        if (per_sm < 1) per_sm = 1;
    });
    const DeviceInfo &di = device_info();
    const int64_t want = (n / 2 + NK_THREADS * NK_U - 1) / (NK_THREADS * NK_U);  // one round a thread
    const int64_t resident = std::min<int64_t>((int64_t)per_sm * di.sms, NK_MAX_WARPS / NK_WARPS);
    const int grid = (int)std::min<int64_t>(std::max<int64_t>(want, 1), resident);
    NearestArgs a;
    a.pts = pts;
    a.n = n;
    a.qx = qx;
    a.qy = qy;
    a.k = k;
    a.idx_out = idx;
    a.d_out = d;
    const size_t tbytes = sizeof(uint32_t) * (size_t)grid * NK_THREADS;
    Scratch *scr = scratch_for((accr_stream_t)s, tbytes + sizeof(PairSlot) * (size_t)grid * NK_WARPS);
    if (!scr) return ACCR_ENOMEM;
    a.tmin = (uint32_t *)scr->buf;
    a.wmin = (PairSlot *)((char *)scr->buf + tbytes);
    a.counter = scr->counters + 1;
    a.threads = grid * NK_THREADS;
    int rc = launch_guard("nearest_kernel");
    if (rc != ACCR_OK) return rc;
    launch_overlapped(nearest_kernel, dim3((unsigned)grid), NK_THREADS, 0, s, a);
    return launched("nearest_kernel");
}

// ============================================================================
// SRAD pattern: statistics of an array, then the standardised array
// ============================================================================

constexpr int SD_THREADS = 512;

struct __align__(16) StatPartial {
    float s1, c1, s2, c2;  // compensated sum of x and of x^2
};

struct StdShared {
    double mean, var;
    float mean_f, rstd_f;
};

__device__ __forceinline__ void stat_merge(float &s1, float &c1, float &s2, float &c2, float t1, float e1, float t2,
                                           float e2) {
    two_sum_merge(s1, c1, t1, e1);
    two_sum_merge(s2, c2, t2, e2);
}

// CTA merge of the four running values (NT threads); thread 0 ends with the totals.
template <int NT>
__device__ __forceinline__ void stat_cta(float &s1, float &c1, float &s2, float &c2, StatPartial *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        const float t1 = __shfl_xor_sync(0xffffffffu, s1, m), e1 = __shfl_xor_sync(0xffffffffu, c1, m);
        const float t2 = __shfl_xor_sync(0xffffffffu, s2, m), e2 = __shfl_xor_sync(0xffffffffu, c2, m);
        if (threadIdx.x & m) {  // lane-order independent: every lane gets the same bits
            float a1 = t1, b1 = e1, a2 = t2, b2 = e2;
            stat_merge(a1, b1, a2, b2, s1, c1, s2, c2);
            s1 = a1, c1 = b1, s2 = a2, c2 = b2;
        } else {
            stat_merge(s1, c1, s2, c2, t1, e1, t2, e2);
        }
    }
    if (lane == 0) sh[warp] = StatPartial{s1, c1, s2, c2};
    __syncthreads();
    if (warp == 0) {
        StatPartial p = lane < NT / 32 ? sh[lane] : StatPartial{-0.f, 0.f, -0.f, 0.f};
        s1 = p.s1, c1 = p.c1, s2 = p.s2, c2 = p.c2;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) {
            const float t1 = __shfl_xor_sync(0xffffffffu, s1, m), e1 = __shfl_xor_sync(0xffffffffu, c1, m);
            const float t2 = __shfl_xor_sync(0xffffffffu, s2, m), e2 = __shfl_xor_sync(0xffffffffu, c2, m);
            if (threadIdx.x & m) {
                float a1 = t1, b1 = e1, a2 = t2, b2 = e2;
                stat_merge(a1, b1, a2, b2, s1, c1, s2, c2);
                s1 = a1, c1 = b1, s2 = a2, c2 = b2;
            } else {
                stat_merge(s1, c1, s2, c2, t1, e1, t2, e2);
            }
        }
    }
    __syncthreads();
}

struct StdArgs {
    const float *x;
    float *y;
    int64_t n;
    double *stats;          // device [mean, var] for the caller
    StatPartial *partials;  // [grid]
    unsigned *counter;      // pass-1 arrivals of the unfused form (zero on entry and exit)
    StdShared *shared;      // unfused: statistics for the elementwise launch
    unsigned *bar;          // fused: grid barrier
    unsigned *err;          // fused: `gen` of a call whose barrier wait ran out
    unsigned gen;
};

// x^2 added exactly: p = fl(x*x) through the compensated sum, and the product's
// rounding error e = x*x - p (exact by fused multiply-add) into the compensation.
__device__ __forceinline__ void add_square(float &s, float &c, float x) {
    const float p = __fmul_rn(x, x);
    const float e = __fmaf_rn(x, x, -p);
    add_compensated(s, c, p);
    c = __fadd_rn(c, e);
}

// Merges all CTA partials in double, in a fixed order; thread 0 returns the
// statistics (NT threads call it).
template <int NT>
__device__ __forceinline__ StdShared merge_stats(const StatPartial *part, int G, int64_t n) {
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < G; i += NT) {
        const uint4 raw = __ldcg(reinterpret_cast<const uint4 *>(part + i));
        a += (double)__uint_as_float(raw.x) + (double)__uint_as_float(raw.y);
        b += (double)__uint_as_float(raw.z) + (double)__uint_as_float(raw.w);
    }
    __shared__ double sa[NT / 32], sb[NT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = min(NT / 32, (G + 31) / 32);  // warps that hold partials
    if (warp < nw) {
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, m);
            b += __shfl_xor_sync(0xffffffffu, b, m);
        }
        if (lane == 0) {
            sa[warp] = a;
            sb[warp] = b;
        }
    }
    __syncthreads();
    StdShared r = {0.0, 0.0, 0.f, 0.f};
    if (threadIdx.x == 0 && n > 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < nw; ++w) {
            ta += sa[w];
            tb += sb[w];
        }
        r.mean = ta / (double)n;
        r.var = tb / (double)n - r.mean * r.mean;
        r.mean_f = (float)r.mean;
        r.rstd_f = r.var > 0.0 ? (float)rsqrt(r.var) : 0.0f;
    }
    return r;
}

// SU vectors in flight per thread; a group's loads all come before its
// stores (each element is read and written by the same thread, so the order
// is right even when y aliases x).  The separate elementwise launch keeps four.
template <int SU>
__device__ __forceinline__ void map_pass(const float *x, float *y, int64_t n, float mean_f, float rstd_f) {
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    const bool al = (((uintptr_t)x | (uintptr_t)y) & 15) == 0;
    if (al) {
        const int64_t nv = n / 4;
        const float4 *x4 = (const float4 *)x;
        float4 *y4 = (float4 *)y;
        int64_t v = gtid;
        for (; v + (SU - 1) * nth < nv; v += SU * nth) {
            float4 a[SU];
#pragma unroll
            for (int u = 0; u < SU; ++u) a[u] = x4[v + u * nth];
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                a[u].x = __fmul_rn(__fsub_rn(a[u].x, mean_f), rstd_f);
                a[u].y = __fmul_rn(__fsub_rn(a[u].y, mean_f), rstd_f);
                a[u].z = __fmul_rn(__fsub_rn(a[u].z, mean_f), rstd_f);
                a[u].w = __fmul_rn(__fsub_rn(a[u].w, mean_f), rstd_f);
                y4[v + u * nth] = a[u];
            }
        }
        for (; v < nv; v += nth) {
            float4 a = x4[v];
            a.x = __fmul_rn(__fsub_rn(a.x, mean_f), rstd_f);
            a.y = __fmul_rn(__fsub_rn(a.y, mean_f), rstd_f);
            a.z = __fmul_rn(__fsub_rn(a.z, mean_f), rstd_f);
            a.w = __fmul_rn(__fsub_rn(a.w, mean_f), rstd_f);
            y4[v] = a;
        }
        for (int64_t i = 4 * nv + gtid; i < n; i += nth) y[i] = __fmul_rn(__fsub_rn(x[i], mean_f), rstd_f);
    } else {
        for (int64_t i = gtid; i < n; i += nth) y[i] = __fmul_rn(__fsub_rn(x[i], mean_f), rstd_f);
    }
}

__global__ void __launch_bounds__(SD_THREADS) standardize_kernel(const __grid_constant__ StdArgs p) {
    __shared__ StatPartial sh[SD_THREADS / 32];
    __shared__ int am_last;
    float s1 = -0.f, c1 = 0.f, s2 = -0.f, c2 = 0.f;
    const int64_t gtid = (int64_t)blockIdx.x * SD_THREADS + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * SD_THREADS;
    const bool al = ((uintptr_t)p.x & 15) == 0;
    if (al) {
        const int64_t nv = p.n / 4;
        const float4 *x4 = (const float4 *)p.x;
        for (int64_t v = gtid; v < nv; v += nth) {
            const float4 a = __ldg(x4 + v);
            add_compensated(s1, c1, a.x);
            add_square(s2, c2, a.x);
            add_compensated(s1, c1, a.y);
            add_square(s2, c2, a.y);
            add_compensated(s1, c1, a.z);
            add_square(s2, c2, a.z);
            add_compensated(s1, c1, a.w);
            add_square(s2, c2, a.w);
        }
        for (int64_t i = 4 * nv + gtid; i < p.n; i += nth) {
            const float a = p.x[i];
            add_compensated(s1, c1, a);
            add_square(s2, c2, a);
        }
    } else {
        for (int64_t i = gtid; i < p.n; i += nth) {
            const float a = p.x[i];
            add_compensated(s1, c1, a);
            add_square(s2, c2, a);
        }
    }
    stat_cta<SD_THREADS>(s1, c1, s2, c2, sh);
    const int G = gridDim.x;
    if (threadIdx.x == 0) {
        p.partials[blockIdx.x] = StatPartial{s1, c1, s2, c2};
        __threadfence();
        am_last = atomicAdd(p.counter, 1u) == (unsigned)G - 1u;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    const StdShared st = merge_stats<SD_THREADS>(p.partials, G, p.n);
    if (threadIdx.x == 0) {
        *p.shared = st;
        p.stats[0] = st.mean;
        p.stats[1] = st.var;
        *p.counter = 0u;
    }
}

// ---- the fused form ----
//
// One cooperative launch, one CTA per SM, each over a contiguous slice.  Both
// passes need the array; between them lie the CTA's merge, a grid barrier and
// the merge of the partials, which every CTA does for itself (publishing them
// from the last CTA cost one more round trip through L2).  The last SF_KEEP
// vectors a thread reads stay in registers (20 MB over 152 SMs: an array up to
// 5 million floats is read once), and the second pass takes the rest of the
// slice from its end backwards, so that what the first pass read last is still
// in L2.  2^22 floats: 24.6 -> 16.1 us; what bounds it now is the chain of load, CTA
// merge, barrier, merge and store, a few microseconds each.
constexpr int SF_THREADS = 1024;
constexpr int SF_KEEP = 8;  // 32 of the 64 registers a thread of such a CTA has
constexpr int SF_SU = 4;    // vectors in flight in the streamed part

// Four consecutive elements of an array that may be unaligned.
template <bool AL>
__device__ __forceinline__ float4 ld_quad(const float *x, int64_t q) {
    if (AL) return *(reinterpret_cast<const float4 *>(x) + q);
    return make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
}
template <bool AL>
__device__ __forceinline__ void st_quad(float *y, int64_t q, const float4 &v) {
    if (AL) {
        *(reinterpret_cast<float4 *>(y) + q) = v;
    } else {
        y[4 * q] = v.x;
        y[4 * q + 1] = v.y;
        y[4 * q + 2] = v.z;
        y[4 * q + 3] = v.w;
    }
}

template <bool AL>
__global__ void __launch_bounds__(SF_THREADS, 1) standardize_fused_kernel(const __grid_constant__ StdArgs p) {
    __shared__ StatPartial sh[SF_THREADS / 32];
    __shared__ float s_mean, s_rstd;
    grid_wait();  // (one CTA is launched overlapped)
    const int t = threadIdx.x, G = gridDim.x;
    unsigned gen = (*(volatile unsigned *)&p.bar[1]) >> 1;
    const int64_t nq = p.n / 4, per = (nq + G - 1) / G;
    const int64_t q0 = min(nq, per * (int64_t)blockIdx.x), q1 = min(nq, q0 + per);
    const int64_t k0 = max(q0, q1 - (int64_t)SF_KEEP * SF_THREADS);  // the kept part: [k0, q1)
    float s1 = -0.f, c1 = 0.f, s2 = -0.f, c2 = 0.f;
    auto add = [&](float a) {
        add_compensated(s1, c1, a);
        add_square(s2, c2, a);
    };
    auto add4 = [&](const float4 &v) { add(v.x), add(v.y), add(v.z), add(v.w); };
    int64_t q = q0 + t;
    for (; q + (SF_SU - 1) * SF_THREADS < k0; q += SF_SU * SF_THREADS) {
        float4 v[SF_SU];
#pragma unroll
        for (int u = 0; u < SF_SU; ++u) v[u] = ld_quad<AL>(p.x, q + u * SF_THREADS);
#pragma unroll
        for (int u = 0; u < SF_SU; ++u) add4(v[u]);
    }
    for (; q < k0; q += SF_THREADS) add4(ld_quad<AL>(p.x, q));
    float4 keep[SF_KEEP];
    const int nk = (int)(q1 - k0);
#pragma unroll
    for (int u = 0; u < SF_KEEP; ++u)
        if (u * SF_THREADS + t < nk) keep[u] = ld_quad<AL>(p.x, k0 + u * SF_THREADS + t);
    const int64_t rest = 4 * nq + t;  // up to three elements past the last vector, in CTA 0
    const bool has_rest = blockIdx.x == 0 && rest < p.n;
    const float xr = has_rest ? p.x[rest] : 0.f;
#pragma unroll
    for (int u = 0; u < SF_KEEP; ++u)
        if (u * SF_THREADS + t < nk) add4(keep[u]);
    if (has_rest) add(xr);
    stat_cta<SF_THREADS>(s1, c1, s2, c2, sh);
    if (t == 0) p.partials[blockIdx.x] = StatPartial{s1, c1, s2, c2};
    if (G == 1) {
        __syncthreads();
    } else if (!grid_barrier_or(p.bar, gen, false, (unsigned)G)) {
        if (t == 0) atomicExch(p.err, p.gen);
        return;
    }
    grid_release();
    const StdShared st = merge_stats<SF_THREADS>(p.partials, G, p.n);
    if (t == 0) {
        s_mean = st.mean_f;
        s_rstd = st.rstd_f;
        if (blockIdx.x == 0) {
            p.stats[0] = st.mean;
            p.stats[1] = st.var;
        }
    }
    __syncthreads();
    const float m = s_mean, rs = s_rstd;
    auto map1 = [&](float a) { return __fmul_rn(__fsub_rn(a, m), rs); };
    auto map4 = [&](const float4 &v) { return make_float4(map1(v.x), map1(v.y), map1(v.z), map1(v.w)); };
    // a thread writes only elements it read, so y may alias x
#pragma unroll
    for (int u = 0; u < SF_KEEP; ++u)
        if (u * SF_THREADS + t < nk) st_quad<AL>(p.y, k0 + u * SF_THREADS + t, map4(keep[u]));
    if (has_rest) p.y[rest] = map1(xr);
    q = k0 - SF_THREADS + t;  // backwards through [q0, k0)
    for (; q - (SF_SU - 1) * SF_THREADS >= q0; q -= SF_SU * SF_THREADS) {
        float4 v[SF_SU];
#pragma unroll
        for (int u = 0; u < SF_SU; ++u) v[u] = ld_quad<AL>(p.x, q - u * SF_THREADS);
#pragma unroll
        for (int u = 0; u < SF_SU; ++u) st_quad<AL>(p.y, q - u * SF_THREADS, map4(v[u]));
    }
    for (; q >= q0; q -= SF_THREADS) st_quad<AL>(p.y, q, map4(ld_quad<AL>(p.x, q)));
}

__global__ void map_kernel(const float *x, float *y, int64_t n, const StdShared *st, float mean_f, float rstd_f,
                           int from_device) {
    if (from_device) {
        mean_f = st->mean_f;
        rstd_f = st->rstd_f;
    }
    map_pass<4>(x, y, n, mean_f, rstd_f);
}

// ============================================================================
// BFS pattern: level-synchronous search on a grid with a convergence flag
// ============================================================================

constexpr int BF_THREADS = 256;
constexpr int BFP_THREADS = 1024;  // the persistent form: one CTA per SM

__global__ void bfs_init_kernel(int32_t *dist, int64_t total, int64_t src, const uint8_t *open) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += (int64_t)gridDim.x * blockDim.x)
        dist[c] = (c == src && open[c]) ? 0 : -1;
}

// One level, pull form: an unvisited open cell with a neighbour at level L
// joins level L + 1.  Returns whether this thread changed any cell.
// One level of the pull formulation over the thread's cells, CU cells at a
// time with every load of a group issued before any is tested: the level is
// bound by L2 latency, not bandwidth, at the sizes of the BFS workloads.
__device__ __forceinline__ bool bfs_level(const uint8_t *open, int32_t *dist, int64_t rows,
                                          int64_t cols, int32_t L) {
    constexpr int CU = 4;
    const int64_t total = rows * cols;  // < 2^31 (checked on the host): 32-bit cell arithmetic
    const uint32_t ucols = (uint32_t)cols, urows = (uint32_t)rows;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    bool changed = false;
    for (int64_t c0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c0 < total; c0 += CU * nth) {
        int32_t d[CU];
        bool need[CU];
#pragma unroll
        for (int j = 0; j < CU; ++j) {
            const int64_t c = c0 + j * nth;
            d[j] = c < total ? __ldcg(dist + c) : 0;
            need[j] = c < total && open[c] != 0;
        }
        int32_t nb[CU][4];
#pragma unroll
        for (int j = 0; j < CU; ++j) {  // an unvisited open cell reads its four neighbours
            const uint32_t c = (uint32_t)(c0 + j * nth);
            const bool go = need[j] && d[j] == -1;
            const uint32_t r = c / ucols, q = c - r * ucols;
            nb[j][0] = go && r > 0 ? __ldcg(dist + c - ucols) : -2;
            nb[j][1] = go && r + 1 < urows ? __ldcg(dist + c + ucols) : -2;
            nb[j][2] = go && q > 0 ? __ldcg(dist + c - 1) : -2;
            nb[j][3] = go && q + 1 < ucols ? __ldcg(dist + c + 1) : -2;
        }
#pragma unroll
        for (int j = 0; j < CU; ++j) {
            if (nb[j][0] == L || nb[j][1] == L || nb[j][2] == L || nb[j][3] == L) {
                dist[c0 + j * nth] = L + 1;
                changed = true;
            }
        }
    }
    return changed;
}

// mode 0: `||` reduction of the flag (warp vote, CTA vote, last-CTA merge)
// mode 1: guarded write (the flag was cleared; threads only write 1)
// The host launches BFS_GROUP levels between two read-backs of their flags (a
// read-back per level cost 19 of its 24 us); `before` is the flag of the level
// before in the group: once a level changed nothing, the ones after it return.
constexpr int BFS_GROUP = 8;

__global__ void __launch_bounds__(BF_THREADS) bfs_level_kernel(const uint8_t *open, int32_t *dist,
                                                               int64_t rows, int64_t cols, int32_t L, int mode,
                                                               unsigned *more, const unsigned *before,
                                                               unsigned *partial, unsigned *counter) {
    grid_wait();
    if (before && *(const volatile unsigned *)before == 0u) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *more = 0u;
        return;
    }
    const bool changed = bfs_level(open, dist, rows, cols, L);
    grid_release();
    if (mode == 1) {
        if (changed) *more = 1u;
        return;
    }
    const int any = __syncthreads_or(changed ? 1 : 0);
    __shared__ int am_last;
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = (unsigned)any;
        __threadfence();
        am_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    int v = 0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += BF_THREADS) v |= (int)__ldcg(partial + b);
    v = __syncthreads_or(v);
    if (threadIdx.x == 0) {
        *more = (unsigned)(v != 0);
        *counter = 0u;
    }
}

// All levels in one cooperative launch: per level, the || of the changed
// flags goes to a per-level slot, a bounded grid barrier separates levels.
// One CTA of BFP_THREADS per SM (fewer arrivals per grid barrier) and one
// barrier per level, which also carries the level's `||` flag: every CTA
// learns whether any cell changed from the barrier's release itself.
__global__ void __launch_bounds__(BFP_THREADS, 1) bfs_persistent_kernel(const uint8_t *open, int32_t *dist,
                                                                       int64_t rows, int64_t cols,
                                                                       int64_t max_levels, unsigned *bar,
                                                                       int64_t *levels_out, int *err) {
    unsigned gen = (*(volatile unsigned *)&bar[1]) >> 1;
    int64_t L = 0;
    for (; L < max_levels; ++L) {
        const bool changed = bfs_level(open, dist, rows, cols, (int32_t)L);
        const int any = __syncthreads_or(changed ? 1 : 0);
        const int r = grid_barrier_or(bar, gen, any != 0, gridDim.x);
        if (r == 0) {
            if (threadIdx.x == 0) atomicExch(err, 7);
            return;
        }
        if (r == 1) break;  // no cell changed at this level
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *levels_out = L + 1;  // the level that found nothing new
}


// All levels in one cooperative launch, on bitmaps.  A level of the cell-wise
// form costs a sweep of every cell through L2 and a grid barrier (4.8 us at
// 1024 x 1024); the levels here run in shared memory and registers, several
// between barriers.
//
//   * A cell is a bit of two bitmaps, 32 cells of a row to a word: still free
//     (open and unvisited) and frontier (joined at the current level).  A level
//     is new = (frontier shifted by one cell each way) & free.
//   * A CTA takes a tile of BT_ROWS rows by 32 words: lane = word, thread = four
//     rows of it in registers, rows past a warp's own through shared memory, so
//     a level costs about 60 instructions a warp and one CTA barrier.
//   * A tile carries a halo of `depth` cells on each side that is not the
//     grid's own edge.  A cell's state after d levels depends on cells at most
//     d away, so `depth` levels run on the tile's own copy and leave its
//     interior exact; then the interior goes back to the bitmaps (two copies,
//     read and written in turn), one grid barrier carries the `||` of "a
//     frontier is left", and the tiles load again.  (Within those levels the halo's
//     far rows stop mattering one by one, and their warps only keep the barrier.)
//
// With one tile the loop runs to the end without grid barriers.  1024 x 1024
// cells, 62 % open, about 1,260 levels: 6.2 ms in the cell-wise form, 0.60 ms here
// (0.31 us a level, and 4 us a step of 28 levels for loading, storing and the
// barrier; what is left is the chain of a level's instructions and its CTA barrier).
constexpr int BT_R = 4;                     // rows per thread
constexpr int BT_THREADS = 512;             // 16 warps: 64 rows a tile
constexpr int BT_ROWS = BT_R * (BT_THREADS / 32);
constexpr int BT_MAX_DEPTH = 30;            // at most 31 (five bit planes), and the 32 columns of halo a tile has
                                            // on each side where a row needs several tiles
constexpr int64_t BT_MAX_CELLS = (int64_t)1 << 28;  // larger grids: the cell-wise form (bitmaps are kept as scratch)

struct BfsTiles {
    const uint8_t *open;
    int32_t *dist;
    int rows, cols, wpr;        // wpr: words per row
    int64_t src;                // -1: none
    uint32_t *free_[2], *front[2];
    int tiles_r, tiles_c, int_rows, int_words, depth;  // depth 0: one tile, until nothing changes
    unsigned tile_ctas;         // CTAs with tiles (the others only set up)
    unsigned *bar;
    int *best;                  // largest distance so far, and CTAs done; zero on entry and exit
    unsigned *done;
    int64_t *result;            // pinned: {levels, status}
};

__global__ void __launch_bounds__(BT_THREADS, 1) bfs_tile_kernel(const __grid_constant__ BfsTiles p) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = BT_THREADS / 32;
    __shared__ uint32_t edge[2][NW][2][32];
    __shared__ uint32_t planes[5][BT_ROWS / 2][32];
    unsigned gen = (*(volatile unsigned *)&p.bar[1]) >> 1;

    // set-up: the bitmaps and dist = -1, one word (32 cells) per warp step
    constexpr int SUN = 4;
    const int nwords = p.rows * p.wpr;  // below 2^26: BT_MAX_CELLS cells and at least one cell a word
    for (int i0 = (blockIdx.x * NW + warp) * SUN; i0 < nwords; i0 += gridDim.x * NW * SUN) {
        uint8_t o[SUN];
        int64_t c[SUN];
        bool in[SUN];
#pragma unroll
        for (int j = 0; j < SUN; ++j) {
            const int i = i0 + j, r = i / p.wpr, q = (i - r * p.wpr) * 32 + lane;
            in[j] = i < nwords && q < p.cols;
            c[j] = (int64_t)r * p.cols + q;
            o[j] = in[j] ? __ldg(p.open + c[j]) : (uint8_t)0;
        }
#pragma unroll
        for (int j = 0; j < SUN; ++j) {
            const bool is_src = in[j] && c[j] == p.src && o[j] != 0;
            const unsigned fr = __ballot_sync(0xffffffffu, is_src);
            const unsigned av = __ballot_sync(0xffffffffu, o[j] != 0 && !is_src);
            if (in[j]) p.dist[c[j]] = is_src ? 0 : -1;
            if (lane == 0 && i0 + j < nwords) {
                p.free_[0][i0 + j] = av;
                p.front[0][i0 + j] = fr;
            }
        }
    }
    const bool started = p.src >= 0 && __ldg(p.open + (p.src >= 0 ? p.src : 0)) != 0;
    int ok = grid_barrier_or(p.bar, gen, false, gridDim.x);
    if (ok && blockIdx.x >= p.tile_ctas) return;

    int reached = 0;  // largest distance this thread gave
    int L = 0;
    const int ntiles = p.tiles_r * p.tiles_c;
    for (int k = 0; ok && started; ++k) {
        const uint32_t *fin = p.free_[k & 1], *rin = p.front[k & 1];
        uint32_t *fout = p.free_[(k & 1) ^ 1], *rout = p.front[(k & 1) ^ 1];
        bool left = false;
        for (int tile = blockIdx.x; tile < ntiles; tile += p.tile_ctas) {
            const int tr = tile / p.tiles_c, tc = tile - tr * p.tiles_c;
            const int r0 = tr * p.int_rows, r1 = min(p.rows, r0 + p.int_rows);
            const int top = p.tiles_r > 1 ? r0 - p.depth : 0;
            const int word = p.tiles_c > 1 ? tc * p.int_words - 1 + lane : lane;
            const bool col_in = word >= 0 && word < p.wpr;
            const bool mine = col_in && (p.tiles_c == 1 || (lane >= 1 && lane <= p.int_words));
            uint32_t a[BT_R], f[BT_R];
            bool own[BT_R];
#pragma unroll
            for (int j = 0; j < BT_R; ++j) {
                const int r = top + warp * BT_R + j;
                const bool in = col_in && r >= 0 && r < p.rows;
                own[j] = mine && r >= r0 && r < r1;
                a[j] = in ? __ldcg(fin + (int64_t)r * p.wpr + word) : 0u;
                f[j] = in ? __ldcg(rin + (int64_t)r * p.wpr + word) : 0u;
            }
            const int wr0 = top + warp * BT_R;                   // this warp's first row
            const bool owns = wr0 < r1 && wr0 + BT_R > r0;       // the same for the warp
            bool more = true;
            int base = L;
            do {
                // up to `run` levels; the level each cell joined at (1 .. 30) is kept
                // in five bit planes and its distance stored at the end: stores
                // inside the loop held up the whole CTA at every level's barrier
                uint32_t pl[5][BT_R];
#pragma unroll
                for (int i = 0; i < 5; ++i)
#pragma unroll
                    for (int j = 0; j < BT_R; ++j) pl[i][j] = 0u;
                const int run = p.depth == 0 ? 30 : p.depth;  // even: the next run starts on the other edge words
                for (int d = 1; d <= run; ++d) {
                    edge[d & 1][warp][0][lane] = f[0];
                    edge[d & 1][warp][1][lane] = f[BT_R - 1];
                    uint32_t any = f[0];
#pragma unroll
                    for (int j = 1; j < BT_R; ++j) any |= f[j];
                    if ((d & 3) != 1) {
                        __syncthreads();
                    } else if (!__syncthreads_or((int)any)) {  // no frontier in the tile: the same for the whole CTA
                        more = false;
                        break;
                    }
                    uint32_t above = warp > 0 ? edge[d & 1][warp - 1][1][lane] : 0u;
                    const uint32_t below = warp + 1 < NW ? edge[d & 1][warp + 1][0][lane] : 0u;
                    // Rows further than the levels left from the interior can no longer
                    // reach it, and rows with nothing near them do not change.
                    if (wr0 >= r1 + (run - d) || wr0 + BT_R <= r0 - (run - d)) continue;
                    if (!__any_sync(0xffffffffu, (any | above | below) != 0u)) continue;
#pragma unroll
                    for (int j = 0; j < BT_R; ++j) {
                        uint32_t lw = __shfl_up_sync(0xffffffffu, f[j], 1), rw = __shfl_down_sync(0xffffffffu, f[j], 1);
                        if (lane == 0) lw = 0u;
                        if (lane == 31) rw = 0u;
                        const uint32_t next = j + 1 < BT_R ? f[j + 1] : below;
                        const uint32_t n = (__funnelshift_l(lw, f[j], 1) | __funnelshift_r(f[j], rw, 1) | above | next) & a[j];
                        above = f[j];
                        f[j] = n;
                        a[j] &= ~n;
                    }
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        if (owns && ((d >> i) & 1)) {
#pragma unroll
                            for (int j = 0; j < BT_R; ++j) pl[i][j] |= f[j];
                        }
                    }
                }
                // the interior's planes to shared memory, half a tile of rows at a
                // time, and from there by every warp, a word (32 cells, one a lane) a
                // step: the interior's own warps are few
                const int irows = r1 - r0;
                for (int h = 0; h < irows; h += BT_ROWS / 2) {
#pragma unroll
                    for (int j = 0; j < BT_R; ++j) {
                        const int i = top + warp * BT_R + j - r0 - h;
                        if (i >= 0 && i < BT_ROWS / 2) {
#pragma unroll
                            for (int q = 0; q < 5; ++q) planes[q][i][lane] = own[j] ? pl[q][j] : 0u;
                        }
                    }
                    __syncthreads();
                    const int n = min(BT_ROWS / 2, irows - h) * 32;
                    for (int e = warp; e < n; e += NW) {
                        const int i = e >> 5, c = e & 31;  // c: the lane that holds the word
                        uint32_t q[5], m = 0u;
#pragma unroll
                        for (int z = 0; z < 5; ++z) {
                            q[z] = planes[z][i][c];
                            m |= q[z];
                        }
                        if ((m >> lane) & 1u) {
                            int d = 0;
#pragma unroll
                            for (int z = 0; z < 5; ++z) d |= (int)((q[z] >> lane) & 1u) << z;
                            const int w = p.tiles_c > 1 ? tc * p.int_words - 1 + c : c;
                            p.dist[(int64_t)(r0 + h + i) * p.cols + w * 32 + lane] = base + d;
                            reached = max(reached, base + d);
                        }
                    }
                    __syncthreads();
                }
                base += run;
            } while (p.depth == 0 && more);
#pragma unroll
            for (int j = 0; j < BT_R; ++j) {
                if (own[j]) {
                    const int64_t i = (int64_t)(top + warp * BT_R + j) * p.wpr + word;
                    fout[i] = a[j];
                    rout[i] = f[j];
                    left |= f[j] != 0u;
                }
            }
            __syncthreads();  // the next tile's first level writes the same edge words
        }
        if (p.depth == 0) break;
        ok = grid_barrier_or(p.bar, gen, __syncthreads_or(left ? 1 : 0) != 0, p.tile_ctas);
        if (ok == 1) break;  // no frontier is left anywhere
        L += p.depth;
    }
    // largest distance, then the host's words by the last CTA
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) reached = max(reached, __shfl_xor_sync(0xffffffffu, reached, s));
    __shared__ int far_[NW];
    if (lane == 0) far_[warp] = reached;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < NW; ++w) reached = max(reached, far_[w]);
        if (!ok) {
            p.result[1] = 7;  // a barrier wait ran out; the host resets the words below
        } else {
            if (reached) atomicMax(p.best, reached);
            __threadfence();
            if (atomicAdd(p.done, 1u) == p.tile_ctas - 1) {
                __threadfence();
                p.result[0] = started ? (int64_t)*(volatile int *)p.best + 1 : 0;
                *p.best = 0;
                *p.done = 0u;
            }
        }
    }
}

// ---- host side ---------------------------------------------------------------------

// The grid's tiles.  They are sized so that there is about one per SM (its interior
// then small and its halo, and so the levels between two barriers, large); the
// interior is at most 32 rows and at least 4.
static void bfs_shape(BfsTiles &a, int64_t rows, int64_t cols) {
    const DeviceInfo &di = device_info();
    a.rows = (int)rows;
    a.cols = (int)cols;
    a.wpr = (int)((cols + 31) / 32);
    a.int_words = a.wpr <= 32 ? 32 : 30;
    a.tiles_c = a.wpr <= 32 ? 1 : (a.wpr + 29) / 30;
    if (rows <= BT_ROWS) {
        a.int_rows = (int)rows;
        a.depth = a.tiles_c == 1 ? 0 : BT_MAX_DEPTH;
    } else {
        const int64_t per_sm = (rows * a.tiles_c + di.sms - 1) / di.sms;
        a.int_rows = (int)std::min<int64_t>(std::max<int64_t>(per_sm, 4), 32);
        a.depth = std::min((BT_ROWS - a.int_rows) / 2, BT_MAX_DEPTH);
    }
    a.tiles_r = (int)((rows + a.int_rows - 1) / a.int_rows);
}

// Whether the tiles are the faster form.  A step of `depth` levels takes about 5.4 us
// for each tile an SM has to go through, however few of a tile's 32 words a row fills;
// a level of the cell-wise form 2.25 us a million cells, and 4 us at least.  Tall grids of
// fewer than about 30 columns are the ones to lose by tiles, us a level, tiles / cells:
// 100,000 x 1 7.4 / 3.3, 100,000 x 8 7.4 / 4.7, 1,000,000 x 1 70 / 4.7, 1,000,000 x 8 70 / 19;
// but 1,000,000 x 40 70 / 91, 16,384 x 4,096 6.7 / 150.
static bool bfs_tiles_pay(const BfsTiles &a, int64_t cells, int sms) {
    if (a.depth == 0) return true;
    const int64_t rounds = ((int64_t)a.tiles_r * a.tiles_c + sms - 1) / sms;
    return rounds * 5400 / a.depth <= std::max<int64_t>(4000, cells * 9 / 4000);  // ns a level
}

// One of the four bitmaps.
static size_t bfs_bitmap_each(const BfsTiles &a) { return ((size_t)a.rows * (size_t)a.wpr * 4 + 255) & ~(size_t)255; }
static size_t bfs_bitmap_bytes(const BfsTiles &a) { return 4 * bfs_bitmap_each(a); }

static int bfs_tiled(BfsTiles &a, const uint8_t *open, int64_t src, int32_t *dist, int64_t *levels, cudaStream_t s) {
    const DeviceInfo &di = device_info();
    const int64_t rows = a.rows, cols = a.cols;
    a.open = open;
    a.dist = dist;
    a.src = (src >= 0 && src < rows * cols) ? src : -1;
    const int64_t ntiles = (int64_t)a.tiles_r * a.tiles_c, nwords = rows * a.wpr;
    a.tile_ctas = (unsigned)std::min<int64_t>(ntiles, di.sms);
    // set-up takes 64 words a CTA and step
    const int64_t setup = (nwords + 63) / 64;
    const int grid = (int)std::min<int64_t>(std::max<int64_t>(setup, a.tile_ctas), di.sms);
    const size_t wbytes = bfs_bitmap_each(a);
    Scratch *scr = scratch_for((accr_stream_t)s, bfs_bitmap_bytes(a));
    if (!scr) return ACCR_ENOMEM;
    int64_t *res = (int64_t *)host_staging_for((accr_stream_t)s, 64);
    if (!res) return ACCR_ENOMEM;
    for (int i = 0; i < 2; ++i) {
        a.free_[i] = (uint32_t *)((char *)scr->buf + (size_t)(2 * i) * wbytes);
        a.front[i] = (uint32_t *)((char *)scr->buf + (size_t)(2 * i + 1) * wbytes);
    }
    a.bar = scr->counters + 12;            // arrivals, generation
    a.best = (int *)(scr->counters + 15);
    a.done = scr->counters + 16;
    a.result = res;
    res[0] = -1;
    res[1] = 0;
    int rc = launch_guard("bfs_tile_kernel");
    if (rc != ACCR_OK) return rc;
    void *args[] = {(void *)&a};
    rc = cuda_check(cudaLaunchCooperativeKernel((const void *)bfs_tile_kernel, grid, BT_THREADS, args, 0, s),
                    "accr_grid_bfs: cooperative launch");
    if (rc != ACCR_OK) return rc;
    if ((rc = launched("bfs_tile_kernel")) != ACCR_OK) return rc;
    rc = cuda_check(cudaStreamSynchronize(s), "accr_grid_bfs: sync");
    if (rc != ACCR_OK) return rc;
    if (*(volatile int64_t *)&res[1] != 0 || *(volatile int64_t *)&res[0] < 0) {
        cudaMemsetAsync(a.bar, 0, sizeof(unsigned), s);
        cudaMemsetAsync(a.best, 0, 2 * sizeof(unsigned), s);
        return set_error(ACCR_ETIMEDOUT, "accr_grid_bfs: grid barrier wait ran out");
    }
    *levels = res[0];
    return ACCR_OK;
}

}  // namespace accr

using namespace accr;

// ---- Nearest Neighbor ------------------------------------------------------------

extern "C" ACCR_API int accr_nearest_k(const float *pts, int64_t n, float qx, float qy, int32_t k,
                                       int64_t *idx_out, float *d2_out, uint32_t flags, accr_stream_t stream) {
    ACCR_TRACE("accr_nearest_k");
    clear_error();
    if (n < 0 || k < 1 || k > 16) return set_error(ACCR_EINVAL, "accr_nearest_k: need n >= 0 and 1 <= k <= 16");
    if (flags & ~ACCR_SYNC) return set_error(ACCR_EINVAL, "accr_nearest_k: unsupported flags 0x%x", flags);
    if ((n > 0 && !pts) || !idx_out || !d2_out) return set_error(ACCR_EINVAL, "accr_nearest_k: NULL pointer");
    if (((uintptr_t)pts & 7) || ((uintptr_t)idx_out & 7) || ((uintptr_t)d2_out & 3))
        return set_error(ACCR_EINVAL, "accr_nearest_k: misaligned pointer (points need 8 bytes)");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = nearest_launch(pts, n, qx, qy, k, idx_out, d2_out, s);
    if (rc != ACCR_OK) return rc;
    if (flags & ACCR_SYNC) return cuda_check(cudaStreamSynchronize(s), "accr_nearest_k: sync");
    return ACCR_OK;
}

// ---- SRAD pattern -------------------------------------------------------------------

struct StdState {
    std::mutex mu;
    unsigned gen = 0;
};
static StdState g_std;

extern "C" ACCR_API int accr_standardize(const float *x, int64_t n, float *y, double *stats, uint32_t flags,
                                         accr_stream_t stream) {
    ACCR_TRACE("accr_standardize");
    clear_error();
    if (n < 0 || (n > 0 && (!x || !y)) || !stats) return set_error(ACCR_EINVAL, "accr_standardize: bad arguments");
    if (((uintptr_t)x & 3) || ((uintptr_t)y & 3) || ((uintptr_t)stats & 7))
        return set_error(ACCR_EINVAL, "accr_standardize: misaligned pointer");
    if (flags & ~(ACCR_SYNC | ACCR_UNFUSED | ACCR_TWO_LEVEL_HOST))
        return set_error(ACCR_EINVAL, "accr_standardize: unsupported flags 0x%x", flags);
    cudaStream_t s = (cudaStream_t)stream;
    const DeviceInfo &di = device_info();
    static int per_sm = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, standardize_kernel, SD_THREADS, 0);
        if (per_sm < 1) per_sm = 1;
    });
    const bool fused = !(flags & (ACCR_UNFUSED | ACCR_TWO_LEVEL_HOST));
    // fused: one CTA per SM, fewer where a thread would have less than a vector
    const int64_t want = fused ? (n / 4 + SF_THREADS - 1) / SF_THREADS : (n / 4 + SD_THREADS * 4 - 1) / (SD_THREADS * 4);
    const int grid = (int)std::min<int64_t>(std::max<int64_t>(want, 1), (int64_t)(fused ? 1 : per_sm) * di.sms);
    // scratch: [counters][shared stats][partials]
    Scratch *scr = scratch_for(stream, sizeof(StatPartial) * (size_t)grid + 256);
    if (!scr) return ACCR_ENOMEM;
    StdArgs a;
    memset(&a, 0, sizeof a);
    a.x = x;
    a.y = y;
    a.n = n;
    a.stats = stats;
    a.partials = (StatPartial *)((char *)scr->buf + 256);
    a.counter = scr->counters + 2;
    a.shared = (StdShared *)scr->buf;
    a.bar = scr->counters + 20;
    a.err = scr->counters + 4;
    {
        std::lock_guard<std::mutex> lk(g_std.mu);
        a.gen = ++g_std.gen;
        if (a.gen == 0) a.gen = ++g_std.gen;
    }
    int rc = launch_guard("standardize_kernel");
    if (rc != ACCR_OK) return rc;
    if (flags & ACCR_TWO_LEVEL_HOST) {
        // the paper's form: CTA partials to the host, merged there, then the
        // elementwise region with the statistics as launch arguments
        standardize_kernel<<<grid, SD_THREADS, 0, s>>>(a);
        if ((rc = launched("standardize_kernel")) != ACCR_OK) return rc;
        StatPartial *h = (StatPartial *)host_staging_for(stream, sizeof(StatPartial) * (size_t)grid);
        if (!h) return ACCR_ENOMEM;
        rc = cuda_check(cudaMemcpyAsync(h, a.partials, sizeof(StatPartial) * (size_t)grid, cudaMemcpyDeviceToHost, s),
                        "accr_standardize: partials");
        if (rc == ACCR_OK) rc = cuda_check(cudaStreamSynchronize(s), "accr_standardize: sync");
        if (rc != ACCR_OK) return rc;
        double ta = 0.0, tb = 0.0;
        for (int i = 0; i < grid; ++i) {
            ta += (double)h[i].s1 + (double)h[i].c1;
            tb += (double)h[i].s2 + (double)h[i].c2;
        }
        const double mean = n > 0 ? ta / (double)n : 0.0, var = n > 0 ? tb / (double)n - mean * mean : 0.0;
        const float mean_f = (float)mean, rstd_f = var > 0.0 ? (float)(1.0 / sqrt(var)) : 0.0f;
        map_kernel<<<di.sms * 4, 512, 0, s>>>(x, y, n, nullptr, mean_f, rstd_f, 0);
        if ((rc = launched("map_kernel")) != ACCR_OK) return rc;
        const double st[2] = {mean, var};
        rc = cuda_check(cudaMemcpyAsync(stats, st, sizeof st, cudaMemcpyHostToDevice, s), "accr_standardize: stats");
        if (rc == ACCR_OK) rc = cuda_check(cudaStreamSynchronize(s), "accr_standardize: sync");
        return rc;
    }
    if (flags & ACCR_UNFUSED) {
        // two launches, the statistics stay on the device
        standardize_kernel<<<grid, SD_THREADS, 0, s>>>(a);
        if ((rc = launched("standardize_kernel")) != ACCR_OK) return rc;
        map_kernel<<<di.sms * 4, 512, 0, s>>>(x, y, n, a.shared, 0.f, 0.f, 1);
        if ((rc = launched("map_kernel")) != ACCR_OK) return rc;
    } else {
        // one cooperative launch: co-residency of every CTA is guaranteed, so
        // the wait at the grid barrier cannot starve a CTA that has to arrive
        const bool al = (((uintptr_t)x | (uintptr_t)y) & 15) == 0;
        auto fused_kernel = al ? standardize_fused_kernel<true> : standardize_fused_kernel<false>;
        if (grid == 1) {  // one CTA waits for nobody: an ordinary launch
            launch_overlapped(fused_kernel, dim3(1), SF_THREADS, 0, s, a);
        } else {
            void *args[] = {&a};
            rc = cuda_check(cudaLaunchCooperativeKernel((void *)fused_kernel, dim3((unsigned)grid), dim3(SF_THREADS), args, 0, s),
                            "accr_standardize: cooperative launch");
            if (rc != ACCR_OK) return rc;
        }
        if ((rc = launched("standardize_kernel (fused)")) != ACCR_OK) return rc;
    }
    if (flags & ACCR_SYNC) {
        // the status word holds the number of the last call whose wait ran out
        unsigned h = 0;
        rc = cuda_check(cudaMemcpyAsync(&h, a.err, sizeof h, cudaMemcpyDeviceToHost, s), "accr_standardize: status");
        if (rc == ACCR_OK) rc = cuda_check(cudaStreamSynchronize(s), "accr_standardize: sync");
        if (rc == ACCR_OK && h == a.gen) {
            cudaMemsetAsync(a.bar, 0, sizeof(unsigned), s);
            return set_error(ACCR_ETIMEDOUT, "accr_standardize: grid wait ran out");
        }
    }
    return rc;
}

// ---- BFS pattern -------------------------------------------------------------------

extern "C" ACCR_API int accr_grid_bfs(const uint8_t *open, int64_t rows, int64_t cols, int64_t src, int32_t *dist,
                                      int32_t mode, int64_t *levels, accr_stream_t stream) {
    ACCR_TRACE("accr_grid_bfs");
    clear_error();
    if (rows < 0 || cols < 0 || (rows * cols > 0 && (!open || !dist)) || !levels)
        return set_error(ACCR_EINVAL, "accr_grid_bfs: bad arguments");
    if (rows * cols >= ((int64_t)1 << 31)) return set_error(ACCR_EINVAL, "accr_grid_bfs: grid too large");
    if (mode < ACCR_BFS_REDUCE || mode > ACCR_BFS_PERSISTENT) return set_error(ACCR_EINVAL, "accr_grid_bfs: bad mode");
    *levels = 0;
    const int64_t total = rows * cols;
    if (total == 0) return ACCR_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const DeviceInfo &di = device_info();
    if (mode == ACCR_BFS_PERSISTENT && total <= BT_MAX_CELLS && (int64_t)rows * ((cols + 31) / 32) <= BT_MAX_CELLS / 8) {
        BfsTiles a;
        memset(&a, 0, sizeof a);
        bfs_shape(a, rows, cols);
        if (bfs_tiles_pay(a, total, di.sms)) {
            const int rc = bfs_tiled(a, open, src, dist, levels, s);
            // no room for large bitmaps: cell by cell, which keeps next to nothing
            if (rc != ACCR_ENOMEM || bfs_bitmap_bytes(a) <= ((size_t)1 << 20)) return rc;
            clear_error();
        }
    }
    int rc;
    if ((rc = launch_guard("bfs_init_kernel")) != ACCR_OK) return rc;
    bfs_init_kernel<<<di.sms * 4, 256, 0, s>>>(dist, total, (src >= 0 && src < total) ? src : -1, open);
    if ((rc = launched("bfs_init_kernel")) != ACCR_OK) return rc;
    if (src < 0 || src >= total) return cuda_check(cudaStreamSynchronize(s), "accr_grid_bfs: sync");
    {  // a closed source cell reaches nothing: zero levels
        uint8_t o = 0;
        rc = cuda_check(cudaMemcpyAsync(&o, open + src, 1, cudaMemcpyDeviceToHost, s), "accr_grid_bfs: source");
        if (rc == ACCR_OK) rc = cuda_check(cudaStreamSynchronize(s), "accr_grid_bfs: sync");
        if (rc != ACCR_OK) return rc;
        if (!o) return ACCR_OK;
    }
    static int per_sm = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bfs_level_kernel, BF_THREADS, 0);
        if (per_sm < 1) per_sm = 1;
    });
    const int64_t want = (total + BF_THREADS - 1) / BF_THREADS;
    const int grid = (int)std::min<int64_t>(want, (int64_t)per_sm * di.sms);
    Scratch *scr = scratch_for(stream, sizeof(unsigned) * (size_t)grid + 512);
    if (!scr) return ACCR_ENOMEM;
    unsigned *more = scr->counters + 32;     // BFS_GROUP words
    unsigned *counter = scr->counters + 9;
    unsigned *bar = scr->counters + 12;      // arrivals, generation
    int *err = (int *)(scr->counters + 14);
    int64_t *lv = (int64_t *)((char *)scr->buf);
    unsigned *partial = (unsigned *)((char *)scr->buf + 64);
    unsigned *hmore = (unsigned *)host_staging_for(stream, 64);
    if (!hmore) return ACCR_ENOMEM;
    if (mode == ACCR_BFS_PERSISTENT) {
        rc = cuda_check(cudaMemsetAsync(err, 0, sizeof(int), s), "accr_grid_bfs: clear status");
        if (rc == ACCR_OK) rc = cuda_check(cudaMemsetAsync(bar, 0, sizeof(unsigned), s), "accr_grid_bfs: barrier");
        if (rc != ACCR_OK) return rc;
        int64_t maxl = total + 1;
        void *args[] = {(void *)&open, (void *)&dist, (void *)&rows, (void *)&cols, (void *)&maxl,
                        (void *)&bar, (void *)&lv, (void *)&err};
        if ((rc = launch_guard("bfs_persistent_kernel")) != ACCR_OK) return rc;
        const int pgrid = (int)std::min<int64_t>((total + BFP_THREADS - 1) / BFP_THREADS, (int64_t)di.sms);
        rc = cuda_check(cudaLaunchCooperativeKernel((const void *)bfs_persistent_kernel, pgrid, BFP_THREADS, args, 0, s),
                        "accr_grid_bfs: cooperative launch");
        if (rc != ACCR_OK) return rc;
        if ((rc = launched("bfs_persistent_kernel")) != ACCR_OK) return rc;
        int64_t hl[2] = {0, 0};
        rc = cuda_check(cudaMemcpyAsync(hl, lv, sizeof(int64_t), cudaMemcpyDeviceToHost, s), "accr_grid_bfs: levels");
        int herr = 0;
        if (rc == ACCR_OK)
            rc = cuda_check(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s), "accr_grid_bfs: status");
        if (rc == ACCR_OK) rc = cuda_check(cudaStreamSynchronize(s), "accr_grid_bfs: sync");
        if (rc != ACCR_OK) return rc;
        if (herr) return set_error(ACCR_ETIMEDOUT, "accr_grid_bfs: grid barrier wait ran out");
        *levels = hl[0];
        return ACCR_OK;
    }
    // host-driven levels: one launch per level, the flags of a group read back together
    // (guarded writes need cleared flags; each level clearing the next one's instead of a
    // memset a group took the same 23.4 us a level at 1024 x 1024, 4.2 at 145 x 190)
    for (int64_t L0 = 0; L0 <= total; L0 += BFS_GROUP) {
        if (mode == ACCR_BFS_GUARDED) {
            rc = cuda_check(cudaMemsetAsync(more, 0, BFS_GROUP * sizeof(unsigned), s), "accr_grid_bfs: clear flags");
            if (rc != ACCR_OK) return rc;
        }
        for (int i = 0; i < BFS_GROUP; ++i) {
            if ((rc = launch_guard("bfs_level_kernel")) != ACCR_OK) return rc;
            launch_overlapped(bfs_level_kernel, dim3((unsigned)grid), BF_THREADS, 0, s, open, dist, rows, cols,
                              (int32_t)(L0 + i), mode == ACCR_BFS_GUARDED ? 1 : 0, more + i, i > 0 ? more + i - 1 : nullptr,
                              partial, counter);
            if ((rc = launched("bfs_level_kernel")) != ACCR_OK) return rc;
        }
        rc = cuda_check(cudaMemcpyAsync(hmore, more, BFS_GROUP * sizeof(unsigned), cudaMemcpyDeviceToHost, s),
                        "accr_grid_bfs: flags");
        if (rc == ACCR_OK) rc = cuda_check(cudaStreamSynchronize(s), "accr_grid_bfs: sync");
        if (rc != ACCR_OK) return rc;
        for (int i = 0; i < BFS_GROUP; ++i) {
            if (!hmore[i]) {
                *levels = L0 + i + 1;
                return ACCR_OK;
            }
        }
    }
    *levels = total + 1;
    return ACCR_OK;
}
