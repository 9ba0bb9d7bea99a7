// group.cuh -- a short stretch of elements (at most GROUP_BYTES) folded by a group
// of 1 to 32 neighbouring lanes: short rows and short segments.
#pragma once

#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "fold.cuh"
#include "overlap.cuh"

namespace accr {

constexpr int GROUP_GV = 8;                          // vectors per lane at most
constexpr int64_t GROUP_BYTES = GROUP_GV * 32 * 16;  // 4 KiB

// A running fold of one clause of a fixed code in registers: whole vectors and
// single elements in, an accumulator out.  The primary form keeps the
// accumulator itself; the float sums and extremes keep their own chains between
// vectors, which saves the accumulator's packing and the chains' merge per vector.
// (The generic kernels fold float sums and double ones the same way, so that a sum has
// the same bits alone and beside any other clause.)
template <typename T, int W>
struct GroupFold {
    Acc A;
    __device__ __forceinline__ void init(uint64_t ident) { A.a = ident, A.c = 0.f; }
    __device__ __forceinline__ void vec(const uint4 &v) { fold_vec<T, 1>(W, A, &v); }
    __device__ __forceinline__ void one(T x) { fold_one<T>(W, A, x); }
    __device__ __forceinline__ Acc get() const { return A; }
};
template <>
struct GroupFold<float, W_ADDF> {
    float p0, p1, p2, p3;
    __device__ __forceinline__ void init(uint64_t) { p0 = p1 = p2 = p3 = -0.f; }
    __device__ __forceinline__ void vec(const uint4 &v) {
        p0 = __fadd_rn(p0, __uint_as_float(v.x));
        p1 = __fadd_rn(p1, __uint_as_float(v.y));
        p2 = __fadd_rn(p2, __uint_as_float(v.z));
        p3 = __fadd_rn(p3, __uint_as_float(v.w));
    }
    __device__ __forceinline__ void one(float x) { p0 = __fadd_rn(p0, x); }
    __device__ __forceinline__ Acc get() const {
        Acc A;
        A.a = f2u(__fadd_rn(__fadd_rn(p0, p1), __fadd_rn(p2, p3)));
        A.c = 0.f;
        return A;
    }
};
template <bool MAX>
struct GroupExtreme {
    float m;
    __device__ __forceinline__ void init(uint64_t) { m = MAX ? -INFINITY : INFINITY; }
    __device__ __forceinline__ void vec(const uint4 &v) {
        if (MAX) m = fmax3(fmax3(m, __uint_as_float(v.x), __uint_as_float(v.y)), __uint_as_float(v.z), __uint_as_float(v.w));
        else m = fmin3(fmin3(m, __uint_as_float(v.x), __uint_as_float(v.y)), __uint_as_float(v.z), __uint_as_float(v.w));
    }
    __device__ __forceinline__ void one(float x) { m = MAX ? fmax2(m, x) : fmin2(m, x); }
    __device__ __forceinline__ Acc get() const {
        Acc A;
        A.a = (uint32_t)fkey32(f2u(m));
        A.c = 0.f;
        return A;
    }
};
template <>
struct GroupFold<float, W_MAXF> : GroupExtreme<true> {};
template <>
struct GroupFold<float, W_MINF> : GroupExtreme<false> {};

// Folds the loaded vectors of one lane, the missing ones filled with the clause's
// neutral element, so that an operator switch runs once for all of them: GV, or half
// where no lane has more (`rounds`).  Double sums round once a chunk of at least four
// vectors (chunk_sum_f64), fewer go one by one.
template <typename T, int NV, int GV>
__device__ __forceinline__ void fold_filled(int w, Acc &A, const uint4 (&b)[GV], const bool (&ok)[GV], uint64_t neutral) {
    const uint32_t lo = (uint32_t)neutral, hi = sizeof(T) == 8 ? (uint32_t)(neutral >> 32) : lo;
    uint4 f[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) f[u] = ok[u] ? b[u] : make_uint4(lo, hi, lo, hi);
    fold_vec<T, NV>(w, A, f);
}
template <typename T, int GV>
__device__ __forceinline__ void fold_lane(int w, Acc &A, const uint4 (&b)[GV], const bool (&ok)[GV], int rounds,
                                          uint64_t neutral) {
    if (rounds > GV / 2) {
        fold_filled<T, GV, GV>(w, A, b, ok, neutral);
    } else if (std::is_same<T, double>::value && GV / 2 < 4 && w == W_ADDF) {
#pragma unroll
        for (int u = 0; u < GV / 2; ++u)
            if (ok[u]) fold_vec<T, 1>(W_ADDF, A, &b[u]);
    } else if (rounds > 0) {
        fold_filled<T, GV / 2, GV>(w, A, b, ok, neutral);
    }
}

// One stretch of `len` elements at `in`, folded by a group of L lanes (this lane is
// number l of it) into A and merged across the group.  `rounds`: no lane of the
// warp has more than this many vectors (at most GV).  Lanes that are not live
// take part in the merge only.  Every load is in flight before any is folded.
// EVERY: each lane has a vector of the stretch, live or not (rows past 2 KiB): its
// loads are unconditional, a missing vector's reads the lane's first one again.  Eight
// conditional ones became branches, each waiting for its own load (100,000 rows of
// 1,000 floats, sum and max: 92.4 us, 62.5 without the conditions; sum alone 92.9, 66.0);
// four are predicated.
template <typename T, int NC, int W0, int W1, int GV, bool EVERY = false>
__device__ __forceinline__ void group_fold(const T *in, int len, bool live, int l, int L, int rounds,
                                           const ClauseDev *cl, const uint64_t *neutral, const int (&w)[NC],
                                           Acc (&A)[NC]) {
    constexpr bool E64 = sizeof(T) == 8, PAIR = W0 >= 0;
    constexpr int EPV = 16 / (int)sizeof(T);
    const int mis = (int)(((16 - ((uintptr_t)in & 15)) & 15) / sizeof(T));
    const int end = live ? len : 0;
    const int vec0 = mis < len ? mis : len, head = live ? vec0 : 0;
    const uint4 *vr = (const uint4 *)(in + vec0) + l;
    const int nvec = (end - head) / EPV;
    const int tail0 = head + nvec * EPV;
    uint4 b[GV];
    bool ok[GV];
    T h = T(), t = T();  // this lane's first head and tail element
#pragma unroll
    for (int u = 0; u < GV; ++u) {
        ok[u] = u < rounds && u * L + l < nvec;
        if (EVERY) b[u] = ld_stream(vr + (ok[u] ? u * L : 0));
        else if (ok[u]) b[u] = vr[u * L];
    }
    if (l < head) h = in[l];
    if (tail0 + l < end) t = in[tail0 + l];
    // this lane's head and tail elements, in one order for every kernel
    auto ends = [&](auto &&one) {
        if (l < head) one(h);
        if (tail0 + l < end) one(t);
        if (L < EPV) {  // fewer lanes than a head or tail may have elements
            for (int j = L + l; j < head; j += L) one(in[j]);
            for (int j = tail0 + L + l; j < end; j += L) one(in[j]);
        }
    };
    if constexpr (PAIR) {
        constexpr bool CHUNK = E64 && W0 == W_ADDF;
        GroupFold<T, W0> F0;
        GroupFold<T, W1> F1;
        F0.init(cl[0].ident);
        F1.init(cl[1].ident);
        if constexpr (CHUNK) fold_lane<T, GV>(W0, F0.A, b, ok, rounds, neutral[0]);
#pragma unroll
        for (int u = 0; u < GV; ++u) {
            if (ok[u]) {
                if constexpr (!CHUNK) F0.vec(b[u]);
                F1.vec(b[u]);
            }
        }
        ends([&](T x) { F0.one(x), F1.one(x); });
        A[0] = F0.get();
        A[1] = F1.get();
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if constexpr (std::is_same<T, float>::value) {
                if (w[c] == W_ADDF) {
                    GroupFold<float, W_ADDF> F;
                    F.init(cl[c].ident);
#pragma unroll
                    for (int u = 0; u < GV; ++u)
                        if (ok[u]) F.vec(b[u]);
                    ends([&](T x) { F.one(x); });
                    A[c] = F.get();
                    continue;
                }
            }
            A[c].a = cl[c].ident;
            A[c].c = 0.f;
            fold_lane<T, GV>(w[c], A[c], b, ok, rounds, neutral[c]);
            ends([&](T x) { fold_one<T>(w[c], A[c], x); });
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) group_merge<PAIR>(w[c], E64, A[c], L);
}

}  // namespace accr
