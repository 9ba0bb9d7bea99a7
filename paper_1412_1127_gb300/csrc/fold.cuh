// fold.cuh -- device side of the reduction clause (IPMACC Stage 3.4 item iii,
// Stage 3.7): what one thread folds per element, how two partial results
// merge, and how the merged result meets the variable's prior value.
//
// A clause (op, element type, variable type) is lowered on the host to a
// "working code": the per-element operation in the narrowest exact width.
// Integer max/min/&/|/^/&&/|| work in the element's width and are widened at
// the end (sign extension commutes with them); + and * work in the variable's
// width.  Floating-point max/min order -0 below +0 and are exact: floats fold on the
// hardware's max/min, doubles as order-preserving integer keys, and both merge as
// keys.  Float + may be compensated (each addition's error kept by TwoSum, per thread
// and when merging; double for the cross-gang merge).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "accr.h"

namespace accr {

enum WCode : int {
    W_ADD32 = 0,  // integer + modulo 2^32
    W_ADD64,      // integer + modulo 2^64 (int32 elements sign-extended)
    W_MUL32,      // integer * modulo 2^32
    W_MUL64,      // integer * modulo 2^64
    W_MAXI,       // signed max in the element's width
    W_MINI,       // signed min in the element's width
    W_AND,        // bitwise, element width
    W_OR,
    W_XOR,
    W_LAND,       // 0/1 flag: all elements nonzero
    W_LOR,        // 0/1 flag: some element nonzero
    W_ADDF,       // float + in the element's type
    W_ADDF_COMP,  // float + compensated: (s, c) pairs
    W_ADDF_WIDE,  // float elements summed in double
    W_MULF,       // float * in the element's type
    W_MULF_WIDE,  // float elements multiplied in double
    W_MAXF,       // max over order-preserving keys, element width
    W_MINF,       // min over order-preserving keys, element width
    W_COUNT
};

// Per-clause description passed to kernels by value.
struct ClauseDev {
    int wcode;       // WCode
    int op;          // accr_op
    int acc_type;    // accr_type of the variable
    int pad;
    uint64_t init;   // variable's prior value (bits in acc_type); identity if none
    uint64_t ident;  // identity of the working code (bits of the working slot)
    void *out;       // device pointer of the variable (array for row/segment forms)
};

// A private accumulator: a 64-bit slot (integer bits, float bits, double bits
// or a key) plus the compensation term of compensated float sums.
struct Acc {
    uint64_t a;
    float c;
};

// Partial results in global memory: 16 bytes each.
struct __align__(16) Partial {
    uint64_t a;
    float c;
    uint32_t pad;
};

// ---- bit helpers -------------------------------------------------------------
__host__ __device__ __forceinline__ uint32_t f2u(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    uint32_t u;
    memcpy(&u, &f, 4);
    return u;
#endif
}
__host__ __device__ __forceinline__ float u2f(uint32_t u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}
__host__ __device__ __forceinline__ uint64_t d2u(double d) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t u;
    memcpy(&u, &d, 8);
    return u;
#endif
}
__host__ __device__ __forceinline__ double u2d(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    memcpy(&d, &u, 8);
    return d;
#endif
}

// Round-to-nearest arithmetic usable on both sides (the host path merges the
// block partials of the two-level form).  No multiply-add contraction.
__host__ __device__ __forceinline__ float hd_fadd(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    volatile float r = a + b;
    return r;
#endif
}
__host__ __device__ __forceinline__ float hd_fsub(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fsub_rn(a, b);
#else
    volatile float r = a - b;
    return r;
#endif
}
__host__ __device__ __forceinline__ float hd_fmul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    volatile float r = a * b;
    return r;
#endif
}
__host__ __device__ __forceinline__ double hd_dadd(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dadd_rn(a, b);
#else
    volatile double r = a + b;
    return r;
#endif
}
__host__ __device__ __forceinline__ double hd_dmul(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dmul_rn(a, b);
#else
    volatile double r = a * b;
    return r;
#endif
}

// Order-preserving keys: signed integer compare of keys equals the numeric
// order of the floats, with -0 < +0 (NaN excluded).  The map is an involution.
__host__ __device__ __forceinline__ int32_t fkey32(uint32_t b) {
    const int32_t s = (int32_t)b;
    return s ^ (int32_t)((uint32_t)(s >> 31) >> 1);  // negative: flip all but the sign bit
}
__host__ __device__ __forceinline__ int64_t fkey64(uint64_t b) {
    const int64_t s = (int64_t)b;
    return s ^ (int64_t)((uint64_t)(s >> 63) >> 1);
}

template <typename T>
__device__ __forceinline__ T from_bits32(uint32_t u) {
    if constexpr (std::is_same<T, float>::value) return __uint_as_float(u);
    else return (T)(int32_t)u;
}
template <typename T>
__device__ __forceinline__ T from_bits64(uint64_t u) {
    if constexpr (std::is_same<T, double>::value) return __longlong_as_double((long long)u);
    else return (T)(int64_t)u;
}

// Element k of a 16-byte vector (k a compile-time constant after unrolling).
__device__ __forceinline__ uint32_t word32(const uint4 &v, int k) {
    return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w;
}
__device__ __forceinline__ uint64_t word64(const uint4 &v, int k) {
    return k == 0 ? (((uint64_t)v.y << 32) | v.x) : (((uint64_t)v.w << 32) | v.z);
}

template <typename T, int NV, typename F>
__device__ __forceinline__ void for_each_elem(const uint4 *v, F &&f) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int k = 0; k < 4; ++k) f(from_bits32<T>(word32(v[i], k)));
        } else {
#pragma unroll
            for (int k = 0; k < 2; ++k) f(from_bits64<T>(word64(v[i], k)));
        }
    }
}

// Larger / smaller of two or three floats by the hardware's max/min, whose
// order puts -0 below +0 (the order of the keys above).
__device__ __forceinline__ float fmax2(float a, float b) {
    float r;
    asm("max.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float fmin2(float a, float b) {
    float r;
    asm("min.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Compensated step: (s, c) += x.  The rounding error of s + x comes from
// Knuth's TwoSum: the same exact error as Neumaier's ordered form, in six
// additions for the FMA pipe instead of three plus a compare and two selects
// for the half-rate ALU pipe, which is what bounded compensated sums.
__device__ __forceinline__ void add_compensated(float &s, float &c, float x) {
    const float t = __fadd_rn(s, x);
    const float xp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, xp)), __fsub_rn(x, xp));
    c = __fadd_rn(c, e);
    s = t;
}

// TwoSum merge of two compensated pairs.
__host__ __device__ __forceinline__ void two_sum_merge(float &s, float &c, float s2, float c2) {
    float t = hd_fadd(s, s2);
    float bp = hd_fsub(t, s);
    float e = hd_fadd(hd_fsub(s, hd_fsub(t, bp)), hd_fsub(s2, bp));
    s = t;
    c = hd_fadd(hd_fadd(c, c2), e);
}

// Sum of the 2*NV doubles of a chunk.  GB300's FP64 pipe retires about two
// adds per SM per clock, too few for a double sum at HBM rate, so chunks of
// 8 or more values are summed in integer block floating point: each
// significand (with its implicit bit) is aligned to the chunk's largest
// exponent with 6 guard bits, the aligned magnitudes are added in an int64
// with their signs, and the total is converted and scaled by an exact power
// of two -- two FP64-pipe operations per chunk instead of one per value.
// Bits shifted out are truncated: at most 2^-6 of the largest value's ulp per
// element (under 0.25 ulp for a chunk of 16).  Zeros and subnormals shift out
// whole: chunks whose largest exponent is within 60 of the subnormal range, chunks
// with an infinity or a NaN (which have no such significand), and short chunks are
// added as doubles.  (5 of 16 values on the FP64 pipe meanwhile was faster, 2^27
// doubles 0.158 ms against 0.160, but rounds a chunk five times instead of once:
// about 5 % more error.)
// 16 values at most: 16 aligned magnitudes below 2^59 stay below 2^63.
template <int NV>
__device__ __forceinline__ double chunk_sum_f64(const uint4 *v) {
    constexpr int E = 2 * NV;
    static_assert(E <= 16, "the int64 sum holds 16 magnitudes");
    uint32_t hi[E], lo[E], emax = 0;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        lo[j] = (j & 1) ? v[j >> 1].z : v[j >> 1].x;
        hi[j] = (j & 1) ? v[j >> 1].w : v[j >> 1].y;
        emax = max(emax, hi[j] & 0x7ff00000u);
    }
    // one unsigned compare for both ends: tiny values, whose scale below would leave
    // the normal range (the difference wraps), and the exponent of infinity and NaN
    if (E < 8 || emax - (61u << 20) >= (0x7ffu - 61u) << 20) {
        double t = u2d(word64(v[0], 0));
#pragma unroll
        for (int j = 1; j < E; ++j) t = __dadd_rn(t, u2d(word64(v[j >> 1], j & 1)));
        return t;
    }
    // a negative magnitude is added as its complement, and the ones still
    // missing for two's complement are counted
    uint64_t S = 0;
    int32_t negs = 0;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const uint64_t m = ((uint64_t)((hi[j] & 0x000fffffu) | 0x00100000u) << 32) | lo[j];
        const uint32_t sh = (emax - (hi[j] & 0x7ff00000u)) >> 20;
        uint64_t mag;
        asm("shr.u64 %0, %1, %2;" : "=l"(mag) : "l"(m << 6), "r"(sh));  // 64 and more: 0
        const int32_t s = (int32_t)hi[j] >> 31;
        S += mag ^ (uint64_t)(int64_t)s;
        negs -= s;
    }
    S += (uint64_t)(int64_t)negs;
    // S counts units of 2^(emax - 1075 - 6); that power of two is normal here
    const double scale = u2d((uint64_t)((emax >> 20) - 1081 + 1023) << 52);
    return __dmul_rn(__ll2double_rn((long long)S), scale);
}

// a += the sum of the 4*NV floats of a chunk, in double.  Converting and adding
// each float costs two operations of the FP64 pipe (about two a clock per SM,
// which bounded a float array summed into a double at 0.72 TB/s), so the chunk
// is summed by extraction (Rump, Ogita and Oishi's error-free split against a
// power-of-two anchor): with 2^E <= max |x| < 2^(E+1), adding and subtracting
// 1.5 * 2^(E+2) splits x exactly into a multiple of 2^(E-21) and a remainder,
// whose own split against 2^-23 of that anchor leaves a multiple of 2^(E-44)
// and a second remainder.  The multiples are added as integers (the anchored
// values' bits, modulo 2^32), the second remainders as floats (an error below
// 2^(E-63)), and the total, in units of 2^(E-54), meets the double accumulator
// in one fused multiply-add: two FP64-pipe operations a chunk, and at most
// 2^(E-54) lost before the accumulator's own rounding.  A chunk whose largest
// magnitude is not finite, or outside 2^-70 .. 2^120 (zero included), is added
// as doubles.
template <int NV>
__device__ __forceinline__ double add_chunk_wide(double a, const uint4 *v) {
    constexpr int E = 4 * NV;
    if constexpr (NV < 2) {
#pragma unroll
        for (int j = 0; j < E; ++j) a = __dadd_rn(a, (double)__uint_as_float(word32(v[j >> 2], j & 3)));
        return a;
    } else {
        uint32_t mb = 0;  // largest magnitude, as bits: a NaN's exceed infinity's
#pragma unroll
        for (int j = 0; j < E; ++j) mb = max(mb, word32(v[j >> 2], j & 3) & 0x7fffffffu);
        const int e = (int)(mb >> 23) - 127;
        if (e < -70 || e > 120) {
#pragma unroll
            for (int j = 0; j < E; ++j) {
                double d;  // volatile: the conversions (FP64 pipe) stay inside this branch
                asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(__uint_as_float(word32(v[j >> 2], j & 3))));
                a = __dadd_rn(a, d);
            }
            return a;
        }
        const uint32_t b1 = ((uint32_t)(e + 2 + 127) << 23) | 0x400000u;   // 1.5 * 2^(e + 2)
        const uint32_t b2 = ((uint32_t)(e - 21 + 127) << 23) | 0x400000u;  // 1.5 * 2^(e - 21)
        const float s1 = __uint_as_float(b1), s2 = __uint_as_float(b2);
        uint32_t i1 = 0, i2 = 0;
        float r0 = 0.f, r1 = 0.f;
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const float x = __uint_as_float(word32(v[j >> 2], j & 3));
            const float t = __fadd_rn(x, s1);
            i1 += __float_as_uint(t);
            const float r = __fsub_rn(x, __fsub_rn(t, s1));
            const float u = __fadd_rn(r, s2);
            i2 += __float_as_uint(u);
            const float q = __fsub_rn(r, __fsub_rn(u, s2));
            if (j & 1) r1 = __fadd_rn(r1, q);
            else r0 = __fadd_rn(r0, q);
        }
        const int32_t n1 = (int32_t)(i1 - (uint32_t)E * b1), n2 = (int32_t)(i2 - (uint32_t)E * b2);
        // units of 2^(e - 54): |n1| < 2^28 of 2^33 each, |n2| < 2^28 of 2^10 each
        const float rs = __fmul_rn(__fadd_rn(r0, r1), __uint_as_float((uint32_t)(54 - e + 127) << 23));
        const long long S = ((long long)n1 << 33) + ((long long)n2 << 10) + (long long)__float2int_rn(rs);
        return __fma_rn(__ll2double_rn(S), u2d((uint64_t)(uint32_t)(e - 54 + 1023) << 52), a);
    }
}

// ---- per-element folding -------------------------------------------------------
// Fold NV 16-byte vectors of T into A under working code w (warp-uniform).
template <typename T, int NV>
__device__ __forceinline__ void fold_vec(int w, Acc &A, const uint4 *v) {
    static_assert(NV <= 8 || NV % 8 == 0, "double sums take eight vectors at a time");
    if constexpr (std::is_integral<T>::value) {
        using UT = typename std::make_unsigned<T>::type;
        switch (w) {
        case W_ADD32: {
            uint32_t a = (uint32_t)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a += (uint32_t)x; });
            A.a = a;
        } break;
        case W_ADD64: {
            uint64_t a = A.a;
            for_each_elem<T, NV>(v, [&](T x) { a += (uint64_t)(int64_t)x; });
            A.a = a;
        } break;
        case W_MUL32: {
            uint32_t a = (uint32_t)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a *= (uint32_t)x; });
            A.a = a;
        } break;
        case W_MUL64: {
            uint64_t a = A.a;
            for_each_elem<T, NV>(v, [&](T x) { a *= (uint64_t)(int64_t)x; });
            A.a = a;
        } break;
        case W_MAXI: {
            T a = (T)(UT)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a = x > a ? x : a; });
            A.a = (uint64_t)(UT)a;
        } break;
        case W_MINI: {
            T a = (T)(UT)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a = x < a ? x : a; });
            A.a = (uint64_t)(UT)a;
        } break;
        case W_AND: {
            UT a = (UT)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a &= (UT)x; });
            A.a = a;
        } break;
        case W_OR: {
            UT a = (UT)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a |= (UT)x; });
            A.a = a;
        } break;
        case W_XOR: {
            UT a = (UT)A.a;
            for_each_elem<T, NV>(v, [&](T x) { a ^= (UT)x; });
            A.a = a;
        } break;
        case W_LAND: {
            uint32_t f = (uint32_t)A.a;
            for_each_elem<T, NV>(v, [&](T x) { f &= (uint32_t)(x != 0); });
            A.a = f;
        } break;
        case W_LOR: {
            uint32_t f = (uint32_t)A.a;
            for_each_elem<T, NV>(v, [&](T x) { f |= (uint32_t)(x != 0); });
            A.a = f;
        } break;
        default: break;
        }
    } else {
        constexpr bool F32 = std::is_same<T, float>::value;
        switch (w) {
        case W_ADDF: {
            if constexpr (F32) {
                // one partial sum per vector slot: dependency chains of NV
                // adds instead of 4 NV, merged pairwise at the end
                float p0 = u2f((uint32_t)A.a), p1 = -0.f, p2 = -0.f, p3 = -0.f;
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    p0 = p0 + __uint_as_float(v[i].x);
                    p1 = p1 + __uint_as_float(v[i].y);
                    p2 = p2 + __uint_as_float(v[i].z);
                    p3 = p3 + __uint_as_float(v[i].w);
                }
                A.a = f2u((p0 + p1) + (p2 + p3));
            } else {
                double a = u2d(A.a);
#pragma unroll
                for (int i = 0; i < NV; i += 8) a = __dadd_rn(a, chunk_sum_f64<(NV < 8 ? NV : 8)>(v + i));
                A.a = d2u(a);
            }
        } break;
        case W_ADDF_COMP: {
            if constexpr (F32) {
                float s = u2f((uint32_t)A.a), c = A.c;
                for_each_elem<T, NV>(v, [&](T x) { add_compensated(s, c, x); });
                A.a = f2u(s);
                A.c = c;
            }
        } break;
        case W_ADDF_WIDE: {
            if constexpr (F32) A.a = d2u(add_chunk_wide<NV>(u2d(A.a), v));
        } break;
        case W_MULF: {
            T a = F32 ? (T)u2f((uint32_t)A.a) : (T)u2d(A.a);
            for_each_elem<T, NV>(v, [&](T x) { a = a * x; });
            if constexpr (F32) A.a = f2u((float)a); else A.a = d2u((double)a);
        } break;
        case W_MULF_WIDE: {
            double a = u2d(A.a);
            for_each_elem<T, NV>(v, [&](T x) { a = __dmul_rn(a, (double)x); });
            A.a = d2u(a);
        } break;
        case W_MAXF: {
            if constexpr (F32) {  // two independent chains on the hardware's max, two elements a step
                float a0 = u2f((uint32_t)fkey32((uint32_t)A.a)), a1 = a0;
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    a0 = fmax3(a0, __uint_as_float(v[i].x), __uint_as_float(v[i].y));
                    a1 = fmax3(a1, __uint_as_float(v[i].z), __uint_as_float(v[i].w));
                }
                A.a = (uint32_t)fkey32(f2u(fmax2(a0, a1)));
            } else {
                int64_t a = (int64_t)A.a;
                for_each_elem<T, NV>(v, [&](T x) {
                    int64_t k = fkey64((uint64_t)__double_as_longlong(x));
                    a = k > a ? k : a;
                });
                A.a = (uint64_t)a;
            }
        } break;
        case W_MINF: {
            if constexpr (F32) {  // two independent chains on the hardware's min, two elements a step
                float a0 = u2f((uint32_t)fkey32((uint32_t)A.a)), a1 = a0;
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    a0 = fmin3(a0, __uint_as_float(v[i].x), __uint_as_float(v[i].y));
                    a1 = fmin3(a1, __uint_as_float(v[i].z), __uint_as_float(v[i].w));
                }
                A.a = (uint32_t)fkey32(f2u(fmin2(a0, a1)));
            } else {
                int64_t a = (int64_t)A.a;
                for_each_elem<T, NV>(v, [&](T x) {
                    int64_t k = fkey64((uint64_t)__double_as_longlong(x));
                    a = k < a ? k : a;
                });
                A.a = (uint64_t)a;
            }
        } break;
        default: break;
        }
    }
}

// The element that leaves a fold under working code w as it is (element bits).
template <typename T>
__host__ __device__ __forceinline__ uint64_t neutral_element(int w) {
    constexpr bool e64 = sizeof(T) == 8;
    switch (w) {
    case W_MUL32:
    case W_MUL64:
    case W_LAND: return 1;
    case W_MAXI: return e64 ? (uint64_t)INT64_MIN : (uint64_t)(uint32_t)INT32_MIN;
    case W_MINI: return e64 ? (uint64_t)INT64_MAX : (uint64_t)(uint32_t)INT32_MAX;
    case W_AND: return ~0ull;
    case W_ADDF:
    case W_ADDF_COMP:
    case W_ADDF_WIDE: return e64 ? 0x8000000000000000ull : 0x80000000ull;  // -0
    case W_MULF:
    case W_MULF_WIDE: return e64 ? 0x3ff0000000000000ull : 0x3f800000ull;  // 1
    case W_MAXF: return e64 ? 0xfff0000000000000ull : 0xff800000ull;       // -inf
    case W_MINF: return e64 ? 0x7ff0000000000000ull : 0x7f800000ull;       // +inf
    default: return 0;  // sums, |, ^, ||
    }
}

template <typename T>
__device__ __forceinline__ uint4 neutral_vector(int w) {
    const uint64_t n = neutral_element<T>(w);
    const uint32_t lo = (uint32_t)n, hi = sizeof(T) == 8 ? (uint32_t)(n >> 32) : lo;
    return make_uint4(lo, hi, lo, hi);
}

// Fold one scalar element (unaligned heads and ragged tails).
template <typename T>
__device__ __forceinline__ void fold_one(int w, Acc &A, T x) {
    if constexpr (std::is_integral<T>::value) {
        using UT = typename std::make_unsigned<T>::type;
        switch (w) {
        case W_ADD32: A.a = (uint32_t)((uint32_t)A.a + (uint32_t)x); break;
        case W_ADD64: A.a = A.a + (uint64_t)(int64_t)x; break;
        case W_MUL32: A.a = (uint32_t)((uint32_t)A.a * (uint32_t)x); break;
        case W_MUL64: A.a = A.a * (uint64_t)(int64_t)x; break;
        case W_MAXI: { T a = (T)(UT)A.a; A.a = (uint64_t)(UT)(x > a ? x : a); } break;
        case W_MINI: { T a = (T)(UT)A.a; A.a = (uint64_t)(UT)(x < a ? x : a); } break;
        case W_AND: A.a = (UT)((UT)A.a & (UT)x); break;
        case W_OR: A.a = (UT)((UT)A.a | (UT)x); break;
        case W_XOR: A.a = (UT)((UT)A.a ^ (UT)x); break;
        case W_LAND: A.a = (uint32_t)A.a & (uint32_t)(x != 0); break;
        case W_LOR: A.a = (uint32_t)A.a | (uint32_t)(x != 0); break;
        default: break;
        }
    } else {
        constexpr bool F32 = std::is_same<T, float>::value;
        switch (w) {
        case W_ADDF:
            if constexpr (F32) A.a = f2u(__fadd_rn(u2f((uint32_t)A.a), (float)x));
            else A.a = d2u(__dadd_rn(u2d(A.a), (double)x));
            break;
        case W_ADDF_COMP:
            if constexpr (F32) {
                float s = u2f((uint32_t)A.a), c = A.c;
                add_compensated(s, c, (float)x);
                A.a = f2u(s);
                A.c = c;
            }
            break;
        case W_ADDF_WIDE: A.a = d2u(__dadd_rn(u2d(A.a), (double)x)); break;
        case W_MULF:
            if constexpr (F32) A.a = f2u(__fmul_rn(u2f((uint32_t)A.a), (float)x));
            else A.a = d2u(__dmul_rn(u2d(A.a), (double)x));
            break;
        case W_MULF_WIDE: A.a = d2u(__dmul_rn(u2d(A.a), (double)x)); break;
        case W_MAXF:
            if constexpr (F32) {
                int32_t a = (int32_t)(uint32_t)A.a, k = fkey32(__float_as_uint((float)x));
                A.a = (uint32_t)(k > a ? k : a);
            } else {
                int64_t a = (int64_t)A.a, k = fkey64((uint64_t)__double_as_longlong((double)x));
                A.a = (uint64_t)(k > a ? k : a);
            }
            break;
        case W_MINF:
            if constexpr (F32) {
                int32_t a = (int32_t)(uint32_t)A.a, k = fkey32(__float_as_uint((float)x));
                A.a = (uint32_t)(k < a ? k : a);
            } else {
                int64_t a = (int64_t)A.a, k = fkey64((uint64_t)__double_as_longlong((double)x));
                A.a = (uint64_t)(k < a ? k : a);
            }
            break;
        default: break;
        }
    }
}

// N vectors a thread at `vin`, `cnt` of which this thread has, loaded together, the others
// read as each clause's neutral element.
template <typename T, int NC, int N, int NT, typename LD>
__device__ __forceinline__ void masked_fold(const uint4 *vin, int cnt, const int (&w)[NC], Acc (&A)[NC], LD &&ld) {
    uint4 b[N];
    const uint4 n0 = neutral_vector<T>(w[0]);
#pragma unroll
    for (int u = 0; u < N; ++u) {
        b[u] = n0;
        if (u < cnt) b[u] = ld(vin + u * NT);
    }
    fold_vec<T, N>(w[0], A[0], b);
#pragma unroll
    for (int c = 1; c < NC; ++c) {
        const uint4 n = neutral_vector<T>(w[c]);
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (u >= cnt) b[u] = n;
        fold_vec<T, N>(w[c], A[c], b);
    }
}

// Folds the `len` elements (below 64 GiB) at `in` by NT threads (a warp or a CTA;
// this is thread t of them), NV 16-byte vectors a thread in flight, into the threads' own
// accumulators A, which the caller has initialised.  Latency is what a short
// stretch pays, so nothing waits on its own: the unaligned head's and the
// ragged tail's elements are loaded before the vectors and folded after them, and
// the last, partial round is loaded like a full one, missing vectors read as the
// clause's neutral element.  (Head, tail and each vector of the last round waited
// for in turn, as they were, cost up to six memory latencies a stretch.)
// HALF: a partial round of at most half a round's vectors folds half as many, and one of
// at most a vector a thread just that: folding missing vectors was most of the work of a
// stretch little longer than its full rounds (50,000 rows of 525 doubles 104 us, 59 so,
// 70 with every vector on its own; of 1,206 int32, sum and max, 46.7, 41.7, 43.5).
template <typename T, int NC, int NV, int NT, bool HALF, typename LD>
__device__ __forceinline__ void stream_fold(const T *in, int64_t len, int t, const int (&w)[NC], Acc (&A)[NC], LD &&ld) {
    constexpr int EPV = 16 / (int)sizeof(T);
    const int mis = (int)(((16 - ((uintptr_t)in & 15)) & 15) / sizeof(T));
    const int head = mis < len ? mis : (int)len;
    const uint32_t nvec = (uint32_t)((len - head) / EPV);
    const int tail = (int)(len - head - (int64_t)nvec * EPV);
    T xh = T(), xt = T();
    if (t < head) xh = in[t];
    if (t < tail) xt = in[len - tail + t];
    const uint4 *vin = (const uint4 *)(in + head) + t;
    const uint32_t last = nvec % (NT * NV);  // the partial round's vectors, and this thread's of them
    const int cnt_last = last > (uint32_t)t ? (int)((last - (uint32_t)t + NT - 1) / NT) : 0;
    for (uint32_t left = nvec; left > 0; vin += NT * NV) {
        const bool full = left >= NT * NV;  // the same for all threads
        if (HALF && left <= NT * NV / 2) {
            if (left <= NT) {
                if (cnt_last > 0) {
                    const uint4 b = ld(vin);
#pragma unroll
                    for (int c = 0; c < NC; ++c) fold_vec<T, 1>(w[c], A[c], &b);
                }
            } else {
                masked_fold<T, NC, NV / 2, NT>(vin, cnt_last, w, A, ld);
            }
            break;
        }
        uint4 b[NV];
        if (full) {
#pragma unroll
            for (int u = 0; u < NV; ++u) b[u] = ld(vin + u * NT);
        } else {
            const uint4 n0 = neutral_vector<T>(w[0]);
#pragma unroll
            for (int u = 0; u < NV; ++u) {
                b[u] = n0;
                if (u < cnt_last) b[u] = ld(vin + u * NT);
            }
        }
        fold_vec<T, NV>(w[0], A[0], b);
#pragma unroll
        for (int c = 1; c < NC; ++c) {
            if (!full) {
                const uint4 n = neutral_vector<T>(w[c]);
#pragma unroll
                for (int u = 0; u < NV; ++u)
                    if (u >= cnt_last) b[u] = n;
            }
            fold_vec<T, NV>(w[c], A[c], b);
        }
        left = full ? left - NT * NV : 0u;
    }
    if (t < head) {
#pragma unroll
        for (int c = 0; c < NC; ++c) fold_one<T>(w[c], A[c], xh);
    }
    if (t < tail) {
#pragma unroll
        for (int c = 0; c < NC; ++c) fold_one<T>(w[c], A[c], xt);
    }
}

// ---- merging two partial results ------------------------------------------------
// `elem64`: the element (and so the working slot) is 64 bits wide.
__host__ __device__ __forceinline__ void merge(int w, bool elem64, Acc &A, const Acc &B) {
    switch (w) {
    case W_ADD32: A.a = (uint32_t)((uint32_t)A.a + (uint32_t)B.a); break;
    case W_ADD64: A.a = A.a + B.a; break;
    case W_MUL32: A.a = (uint32_t)((uint32_t)A.a * (uint32_t)B.a); break;
    case W_MUL64: A.a = A.a * B.a; break;
    case W_MAXI:
        if (elem64) A.a = (int64_t)B.a > (int64_t)A.a ? B.a : A.a;
        else A.a = (int32_t)(uint32_t)B.a > (int32_t)(uint32_t)A.a ? B.a : A.a;
        break;
    case W_MINI:
        if (elem64) A.a = (int64_t)B.a < (int64_t)A.a ? B.a : A.a;
        else A.a = (int32_t)(uint32_t)B.a < (int32_t)(uint32_t)A.a ? B.a : A.a;
        break;
    case W_AND: A.a &= B.a; break;
    case W_OR: A.a |= B.a; break;
    case W_XOR: A.a ^= B.a; break;
    case W_LAND: A.a &= B.a; break;
    case W_LOR: A.a |= B.a; break;
    case W_ADDF:
        if (elem64) A.a = d2u(hd_dadd(u2d(A.a), u2d(B.a)));
        else A.a = f2u(hd_fadd(u2f((uint32_t)A.a), u2f((uint32_t)B.a)));
        break;
    case W_ADDF_COMP: {
        float s = u2f((uint32_t)A.a), c = A.c;
        two_sum_merge(s, c, u2f((uint32_t)B.a), B.c);
        A.a = f2u(s);
        A.c = c;
    } break;
    case W_ADDF_WIDE: A.a = d2u(hd_dadd(u2d(A.a), u2d(B.a))); break;
    case W_MULF:
        if (elem64) A.a = d2u(hd_dmul(u2d(A.a), u2d(B.a)));
        else A.a = f2u(hd_fmul(u2f((uint32_t)A.a), u2f((uint32_t)B.a)));
        break;
    case W_MULF_WIDE: A.a = d2u(hd_dmul(u2d(A.a), u2d(B.a))); break;
    case W_MAXF:
        if (elem64) A.a = (int64_t)B.a > (int64_t)A.a ? B.a : A.a;
        else A.a = (int32_t)(uint32_t)B.a > (int32_t)(uint32_t)A.a ? B.a : A.a;
        break;
    case W_MINF:
        if (elem64) A.a = (int64_t)B.a < (int64_t)A.a ? B.a : A.a;
        else A.a = (int32_t)(uint32_t)B.a < (int32_t)(uint32_t)A.a ? B.a : A.a;
        break;
    default: break;
    }
}

// The other half of a butterfly step.  With the working code fixed at compile
// time (FIXED) a 32-bit working value moves in one shuffle, a 64-bit one in two,
// and only compensated sums carry their second term; a code read at run time
// moves all three words (choosing would cost a branch a step).
template <bool FIXED>
__device__ __forceinline__ Acc shfl_xor_acc(int w, bool elem64, const Acc &A, int m) {
    Acc B;
    if (FIXED) {
        const bool wide = elem64 || w == W_ADD64 || w == W_MUL64 || w == W_ADDF_WIDE || w == W_MULF_WIDE;
        const uint32_t lo = __shfl_xor_sync(0xffffffffu, (uint32_t)A.a, m);
        const uint32_t hi = wide ? __shfl_xor_sync(0xffffffffu, (uint32_t)(A.a >> 32), m) : 0u;
        B.a = ((uint64_t)hi << 32) | lo;
        B.c = w == W_ADDF_COMP ? __shfl_xor_sync(0xffffffffu, A.c, m) : 0.f;
    } else {
        B.a = __shfl_xor_sync(0xffffffffu, (unsigned long long)A.a, m);
        B.c = __shfl_xor_sync(0xffffffffu, A.c, m);
    }
    return B;
}

// Butterfly merge across groups of `lanes` (a power of two) neighbouring lanes
// of a warp: every lane ends with its group's total.
template <bool FIXED>
__device__ __forceinline__ void group_merge(int w, bool elem64, Acc &A, int lanes) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        if (m >= lanes) continue;
        Acc B = shfl_xor_acc<FIXED>(w, elem64, A, m);
        // combine in a lane-independent order so all lanes hold identical bits
        Acc lo = (threadIdx.x & m) ? B : A;
        Acc hi = (threadIdx.x & m) ? A : B;
        merge(w, elem64, lo, hi);
        A = lo;
    }
}

template <bool FIXED = false>
__device__ __forceinline__ void warp_merge(int w, bool elem64, Acc &A) {
    group_merge<FIXED>(w, elem64, A, 32);
}

// Merge one accumulator per clause across a CTA of NT threads (all threads
// call it); thread 0 ends with the totals.  `sh` is NC x NT/32 shared slots.
// FIXED: the codes are compile-time constants of the kernel.
template <int NC, int NT, bool FIXED = false>
__device__ __forceinline__ void cta_merge(const int (&w)[NC], const uint64_t (&ident)[NC], bool e64,
                                          Acc (&A)[NC], Acc (*sh)[NT / 32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        warp_merge<FIXED>(w[c], e64, A[c]);
        if (lane == 0) sh[c][warp] = A[c];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            Acc B;
            if (lane < NT / 32) B = sh[c][lane];
            else { B.a = ident[c]; B.c = 0.f; }
            warp_merge<FIXED>(w[c], e64, B);
            A[c] = B;
        }
    }
    __syncthreads();
}

// The cross-gang merge of compensated sums runs in double: each (s, c) pair
// becomes s + c in double and the doubles are added.
__host__ __device__ __forceinline__ int final_code(int w) { return w == W_ADDF_COMP ? W_ADDF_WIDE : w; }
__host__ __device__ __forceinline__ uint64_t final_ident(const ClauseDev &cl) {
    return cl.wcode == W_ADDF_COMP ? d2u(-0.0) : cl.ident;
}
__host__ __device__ __forceinline__ Acc to_final(int w, const Acc &A) {
    if (w != W_ADDF_COMP) return A;
    Acc B;
    B.a = d2u(hd_dadd((double)u2f((uint32_t)A.a), (double)A.c));
    B.c = 0.f;
    return B;
}

// The merged working value `tot` (in final_code(w)) meets the variable's prior
// value: var = init (op) tot, computed in the variable's type.  n == 0 leaves
// the variable as it was.  Returns the variable's bits.
__host__ __device__ __forceinline__ uint64_t finish(const ClauseDev &cl, bool elem64, bool n_zero,
                                          const Acc &tot) {
    if (n_zero) return cl.init;
    const int w = cl.wcode;
    const bool acc64 = cl.acc_type == ACCR_I64 || cl.acc_type == ACCR_F64;
    if (cl.acc_type == ACCR_I32 || cl.acc_type == ACCR_I64) {
        // the total in the variable's width (int32 working values sign-extend)
        uint64_t t = tot.a;
        if (!elem64 && acc64 && w != W_ADD64 && w != W_MUL64) t = (uint64_t)(int64_t)(int32_t)(uint32_t)t;
        uint64_t i = cl.init, r = 0;
        switch (cl.op) {
        case ACCR_ADD: r = i + t; break;
        case ACCR_MUL: r = i * t; break;
        case ACCR_MAX:
            r = acc64 ? ((int64_t)t > (int64_t)i ? t : i)
                      : ((int32_t)(uint32_t)t > (int32_t)(uint32_t)i ? t : i);
            break;
        case ACCR_MIN:
            r = acc64 ? ((int64_t)t < (int64_t)i ? t : i)
                      : ((int32_t)(uint32_t)t < (int32_t)(uint32_t)i ? t : i);
            break;
        case ACCR_BAND: r = i & t; break;
        case ACCR_BOR: r = i | t; break;
        case ACCR_BXOR: r = i ^ t; break;
        case ACCR_LAND: r = (acc64 ? i != 0 : (uint32_t)i != 0) && t != 0; break;
        case ACCR_LOR: r = (acc64 ? i != 0 : (uint32_t)i != 0) || t != 0; break;
        }
        return acc64 ? r : (uint64_t)(uint32_t)r;
    }
    // floating point
    if (cl.acc_type == ACCR_F32) {
        float i = u2f((uint32_t)cl.init), v;
        switch (w) {
        case W_ADDF: v = hd_fadd(i, u2f((uint32_t)tot.a)); break;
        case W_ADDF_COMP: v = (float)hd_dadd((double)i, u2d(tot.a)); break;
        case W_MULF: v = hd_fmul(i, u2f((uint32_t)tot.a)); break;
        case W_MAXF: {
            int32_t k = (int32_t)(uint32_t)tot.a, ki = fkey32(f2u(i));
            v = u2f((uint32_t)fkey32((uint32_t)(k > ki ? k : ki)));
        } break;
        case W_MINF: {
            int32_t k = (int32_t)(uint32_t)tot.a, ki = fkey32(f2u(i));
            v = u2f((uint32_t)fkey32((uint32_t)(k < ki ? k : ki)));
        } break;
        default: v = i; break;
        }
        return f2u(v);
    }
    double i = u2d(cl.init), v;
    switch (w) {
    case W_ADDF:
    case W_ADDF_WIDE: v = hd_dadd(i, u2d(tot.a)); break;
    case W_MULF:
    case W_MULF_WIDE: v = hd_dmul(i, u2d(tot.a)); break;
    case W_MAXF:
    case W_MINF: {
        // the key is in the element's width; bring the element to double first
        double x = elem64 ? u2d((uint64_t)fkey64(tot.a))
                          : (double)u2f((uint32_t)fkey32((uint32_t)tot.a));
        int64_t k = fkey64(d2u(x)), ki = fkey64(d2u(i));
        int64_t r = (w == W_MAXF) ? (k > ki ? k : ki) : (k < ki ? k : ki);
        v = u2d((uint64_t)fkey64((uint64_t)r));
    } break;
    default: v = i; break;
    }
    return d2u(v);
}

// Stores a variable's bits (4 or 8 bytes by type) at element `idx` of out.
__device__ __forceinline__ void store_var(const ClauseDev &cl, int64_t idx, uint64_t bits) {
    if (cl.acc_type == ACCR_I32 || cl.acc_type == ACCR_F32)
        ((uint32_t *)cl.out)[idx] = (uint32_t)bits;
    else
        ((uint64_t *)cl.out)[idx] = bits;
}

}  // namespace accr
