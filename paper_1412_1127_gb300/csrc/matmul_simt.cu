// matmul_simt.cu -- the Listing-1a nest on FP32 CUDA cores.
//
//   for i (gang, independent) for j (vector, independent)
//     { float sum = 0; for l (serial) sum += a[i*LEN+l] * b[l*LEN+j]; c[i*LEN+j] = sum; }
//
// The paper's own CUDA version (Listing 1b) gives every thread one output and
// reads a and b straight from global memory; Sec. 4.2 (Matrix Mul) notes that
// the tiled CUDA SDK version, which stages tiles in shared memory and shares
// them among a block's threads, is much faster.  This kernel is the tiled
// form: a CTA computes a BM x BN block of c, stages 16-wide k slices of a
// (transposed) and b in double-buffered shared memory, and every thread keeps
// a TR x TC register block (a side of 8 is two runs of 4 half a tile apart, so
// the 16-byte shared-memory reads of a warp hit distinct banks or broadcast),
// with its operand fragments double-buffered in registers.
//
// Every output still sums its l terms in order 0..LEN-1.  Mode SERIAL rounds
// each product and then each sum (no fused multiply-add), which is exactly
// the serial float program, bit for bit; mode FMA fuses them (faster, and
// closer to the exact product).
#include <string.h>

#include "common.cuh"
#include "overlap.cuh"

namespace accr {

constexpr int KT = 16;    // k slice per stage

template <bool SERIAL>
__device__ __forceinline__ float mac(float acc, float x, float y) {
    if constexpr (SERIAL) return __fadd_rn(acc, __fmul_rn(x, y));
    else return __fmaf_rn(x, y, acc);
}

// Row r of a's slice at k sits at column r ^ swz(k): the four k groups that a
// warp's loader stores at once then fall into different banks (they were a
// four-way conflict), and four consecutive rows stay together.  (SERIAL's 128 x 128
// tile has no registers left for it: LEN 4096 4612 us with, 4567 without.)
template <int SWZ>
__device__ __forceinline__ int a_col(int r, int k) {
    return r ^ (((k >> 2) & 3) * SWZ);
}

template <bool SERIAL, bool VEC, int BM, int BN, int TR, int TC>
__global__ void __launch_bounds__(BM * BN / (TR * TC), 512 / (BM * BN / (TR * TC)))
    matmul_simt_kernel(const float *a, const float *b, float *c, int64_t len) {
    constexpr int NTH = BM * BN / (TR * TC);  // threads
    constexpr int QR = TR / 4, QC = TC / 4;   // runs of 4 a side
    constexpr int LA = BM * KT / 4 / NTH, LB = BN * KT / 4 / NTH;  // float4 loads per thread and slice
    constexpr int SWZ = SERIAL && BM == 128 ? 0 : 8;
    static_assert(LA * NTH * 4 == BM * KT && LB * NTH * 4 == BN * KT, "loads split evenly");
    grid_wait();
    __shared__ __align__(16) float As[2][KT][BM];  // a slice, transposed: As[k][a_col(row, k)]
    __shared__ __align__(16) float Bs[2][KT][BN];  // b slice: Bs[k][col]
    const int tid = threadIdx.x;
    const int tx = tid % (BN / TC), ty = tid / (BN / TC);
    const int64_t row0 = (int64_t)blockIdx.y * BM, col0 = (int64_t)blockIdx.x * BN;

    // loaders: a slice: four float4 a row (k (tid & 3) * 4), rows tid / 4 and on by NTH / 4;
    //          b slice: BN / 4 float4 a k row, neighbouring threads along it
    const int a_r = tid >> 2, a_k = (tid & 3) * 4;

    auto load_a = [&](int64_t k0, int h, float4 &v) {
        const int64_t r = row0 + a_r + h * (NTH / 4), k = k0 + a_k;
        if (VEC && r < len && k + 3 < len) {
            v = *reinterpret_cast<const float4 *>(a + r * len + k);
        } else {
            v.x = (r < len && k + 0 < len) ? a[r * len + k + 0] : 0.f;
            v.y = (r < len && k + 1 < len) ? a[r * len + k + 1] : 0.f;
            v.z = (r < len && k + 2 < len) ? a[r * len + k + 2] : 0.f;
            v.w = (r < len && k + 3 < len) ? a[r * len + k + 3] : 0.f;
        }
    };
    auto load_b = [&](int64_t k0, int h, float4 &v) {
        const int i = tid + h * NTH;
        const int64_t k = k0 + i / (BN / 4), cc = col0 + (i % (BN / 4)) * 4;
        if (VEC && k < len && cc + 3 < len) {
            v = *reinterpret_cast<const float4 *>(b + k * len + cc);
        } else {
            v.x = (k < len && cc + 0 < len) ? b[k * len + cc + 0] : 0.f;
            v.y = (k < len && cc + 1 < len) ? b[k * len + cc + 1] : 0.f;
            v.z = (k < len && cc + 2 < len) ? b[k * len + cc + 2] : 0.f;
            v.w = (k < len && cc + 3 < len) ? b[k * len + cc + 3] : 0.f;
        }
    };
    auto store_tiles = [&](int buf, const float4 (&va)[LA], const float4 (&vb)[LB]) {
#pragma unroll
        for (int h = 0; h < LA; ++h) {
            const int r = a_col<SWZ>(a_r + h * (NTH / 4), a_k);
            As[buf][a_k + 0][r] = va[h].x;
            As[buf][a_k + 1][r] = va[h].y;
            As[buf][a_k + 2][r] = va[h].z;
            As[buf][a_k + 3][r] = va[h].w;
        }
#pragma unroll
        for (int h = 0; h < LB; ++h) {
            const int i = tid + h * NTH;
            *reinterpret_cast<float4 *>(&Bs[buf][i / (BN / 4)][(i % (BN / 4)) * 4]) = vb[h];
        }
    };

    float acc[TR][TC];
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < TC; ++j) acc[i][j] = 0.f;

    float4 va[LA], vb[LB];
#pragma unroll
    for (int h = 0; h < LA; ++h) load_a(0, h, va[h]);
#pragma unroll
    for (int h = 0; h < LB; ++h) load_b(0, h, vb[h]);
    store_tiles(0, va, vb);
    __syncthreads();
    const int64_t nk = (len + KT - 1) / KT;
    for (int64_t kt = 0; kt < nk; ++kt) {
        const int cur = (int)(kt & 1);
        const bool more = kt + 1 < nk;
        if (more) {  // fetch the next slice while this one is used
#pragma unroll
            for (int h = 0; h < LA; ++h) load_a((kt + 1) * KT, h, va[h]);
#pragma unroll
            for (int h = 0; h < LB; ++h) load_b((kt + 1) * KT, h, vb[h]);
        }
        // operand fragments double-buffered in registers: k+1 is read from
        // shared memory while the products of k issue
        float4 fa[2][QR], fb[2][QC];
        auto fetch = [&](int k, float4 (&xa)[QR], float4 (&xb)[QC]) {
#pragma unroll
            for (int q = 0; q < QR; ++q)
                xa[q] = *reinterpret_cast<const float4 *>(&As[cur][k][a_col<SWZ>(q * (BM / QR) + ty * 4, k)]);
#pragma unroll
            for (int q = 0; q < QC; ++q) xb[q] = *reinterpret_cast<const float4 *>(&Bs[cur][k][q * (BN / QC) + tx * 4]);
        };
        fetch(0, fa[0], fb[0]);
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const int p = k & 1;
            if (k + 1 < KT) fetch(k + 1, fa[p ^ 1], fb[p ^ 1]);
            float ar[TR], br[TC];
#pragma unroll
            for (int q = 0; q < QR; ++q)
                ar[q * 4 + 0] = fa[p][q].x, ar[q * 4 + 1] = fa[p][q].y, ar[q * 4 + 2] = fa[p][q].z, ar[q * 4 + 3] = fa[p][q].w;
#pragma unroll
            for (int q = 0; q < QC; ++q)
                br[q * 4 + 0] = fb[p][q].x, br[q * 4 + 1] = fb[p][q].y, br[q * 4 + 2] = fb[p][q].z, br[q * 4 + 3] = fb[p][q].w;
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = mac<SERIAL>(acc[i][j], ar[i], br[j]);
        }
        if (more) store_tiles(cur ^ 1, va, vb);
        __syncthreads();
    }
    grid_release();  // the block's store is left (in the loop it cost 17 of 69 us)
    // write the register block
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        const int64_t r = row0 + (i >> 2) * (BM / QR) + ty * 4 + (i & 3);
        if (r >= len) continue;
#pragma unroll
        for (int h = 0; h < QC; ++h) {
            const int64_t cc = col0 + h * (BN / QC) + tx * 4;
            float4 v = make_float4(acc[i][h * 4 + 0], acc[i][h * 4 + 1], acc[i][h * 4 + 2], acc[i][h * 4 + 3]);
            if (VEC && cc + 3 < len) {
                *reinterpret_cast<float4 *>(c + r * len + cc) = v;
            } else {
                if (cc + 0 < len) c[r * len + cc + 0] = v.x;
                if (cc + 1 < len) c[r * len + cc + 1] = v.y;
                if (cc + 2 < len) c[r * len + cc + 2] = v.z;
                if (cc + 3 < len) c[r * len + cc + 3] = v.w;
            }
        }
    }
}


// Packed pairs of floats (sm_100 family f32x2): each half is an ordinary
// round-to-nearest fused multiply-add.  Used only by the packed FP32 probe:
// measured on GB300, a packed instruction moves no more float work per clock
// than two scalar ones (the FMA pipe is the limit either way).
typedef unsigned long long f2;

__device__ __forceinline__ float lo_of(f2 v) { return __uint_as_float((unsigned)(v & 0xffffffffull)); }
__device__ __forceinline__ float hi_of(f2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f2 pack2(float lo, float hi) {
    return ((f2)__float_as_uint(hi) << 32) | (f2)__float_as_uint(lo);
}

// FP32 peak probe: 16 independent FMA chains per thread (latency hidden by
// the chains and by 8 warps per SM sub-partition at 4 CTAs per SM); b and c
// keep every chain bounded (x -> 0.999 x + 0.001 tends to 1).
constexpr int PROBE_THREADS = 256;

__global__ void __launch_bounds__(PROBE_THREADS) fma_probe_kernel(int64_t rounds, float *sink, float b, float c) {
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = (float)(threadIdx.x + i) * 1e-3f;
    for (int64_t r = 0; r < rounds; ++r) {
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = __fmaf_rn(a[i], b, c);
    }
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) s += a[i];
    sink[(int64_t)blockIdx.x * PROBE_THREADS + threadIdx.x] = s * (1.f / 16.f);
}

// The same probe issuing packed pairs: 16 independent f32x2 chains per thread,
// 32 fused multiply-adds per round.  If the packed form moves more float work
// per clock than scalar instructions, this is the FP32 peak.
__global__ void __launch_bounds__(PROBE_THREADS) fma2_probe_kernel(int64_t rounds, float *sink, float b, float c) {
    f2 a[16];
    const f2 bb = pack2(b, b), cc = pack2(c, c);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float lo = (float)(threadIdx.x + i) * 1e-3f, hi = (float)(threadIdx.x + i + 16) * 1e-3f;
        a[i] = pack2(lo, hi);
    }
    for (int64_t r = 0; r < rounds; ++r) {
#pragma unroll
        for (int i = 0; i < 16; ++i) asm volatile("fma.rn.f32x2 %0, %0, %1, %2;" : "+l"(a[i]) : "l"(bb), "l"(cc));
    }
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) s += lo_of(a[i]) + hi_of(a[i]);
    sink[(int64_t)blockIdx.x * PROBE_THREADS + threadIdx.x] = s * (1.f / 32.f);
}

template <bool SERIAL, int BM, int BN, int TR, int TC>
static void simt_launch(const float *a, const float *b, float *c, int64_t len, bool vec, cudaStream_t s) {
    const dim3 grid((unsigned)((len + BN - 1) / BN), (unsigned)((len + BM - 1) / BM));
    constexpr int NTH = BM * BN / (TR * TC);
    launch_overlapped(vec ? matmul_simt_kernel<SERIAL, true, BM, BN, TR, TC> : matmul_simt_kernel<SERIAL, false, BM, BN, TR, TC>,
                      grid, NTH, 0, s, a, b, c, len);
}

int matmul_simt(const float *a, const float *b, float *c, int64_t len, bool serial, cudaStream_t s) {
    if (len == 0) return ACCR_OK;
    const int64_t tiles = (len + 127) / 128;
    if (tiles > 65535) return set_error(ACCR_EINVAL, "accr_matmul_nest: len too large for the SIMT grid");
    // 16-byte vector access needs 16-byte aligned rows
    int rc = launch_guard("matmul_simt_kernel");
    if (rc != ACCR_OK) return rc;
    const bool vec = (len % 4 == 0) && ((uintptr_t)a % 16 == 0) && ((uintptr_t)b % 16 == 0) && ((uintptr_t)c % 16 == 0);
    // The tile by how the matrix fills the chip (every form adds an output's terms
    // in the same order, so they give the same bits).  Measured, us, 128 x 128 /
    // 64 x 64 / 32 x 32 tiles: LEN 512 60 / 25 / 19, 900 117 / 68 / 64, 1024 115 / 72 / 76,
    // 1200 150 / 117 / 139, 1448 181 / 179 / 227, 1536 173 / 177 / 228, 2048 411 / 423 / 533.
    // SERIAL's separate products and sums leave the large tile short of registers:
    // 1024 205 / 101 / 102, 1448 308 / 262 / 285, 2048 676 / 625, 3000 1996 / 1934.
    const int64_t sms = device_info().sms;
    const int64_t t128 = tiles * tiles, t64 = ((len + 63) / 64) * ((len + 63) / 64);
    // Past one 128 x 128 tile an SM its rounds (one tile an SM) cost 3.8 of the small
    // tile's: 3072 1997 / 2070 us, 3500 3371 / 2997, 4096 4555 / 4688.
    const int64_t r128 = (t128 + sms - 1) / sms, r64 = (t64 + sms - 1) / sms;
    const bool small = t64 * 10 < sms * 16;
    if (serial) {
        if (small) simt_launch<true, 32, 32, 4, 4>(a, b, c, len, vec, s);
        else if (r128 < 2 || r128 * 38 >= r64 * 10) simt_launch<true, 64, 64, 8, 4>(a, b, c, len, vec, s);
        else simt_launch<true, 128, 128, 8, 8>(a, b, c, len, vec, s);
    } else {
        if (small) simt_launch<false, 32, 32, 4, 4>(a, b, c, len, vec, s);
        else if (t128 * 10 < sms * 9) simt_launch<false, 64, 64, 8, 4>(a, b, c, len, vec, s);
        else simt_launch<false, 128, 128, 8, 8>(a, b, c, len, vec, s);
    }
    return launched("matmul_simt_kernel");
}

}  // namespace accr

extern "C" ACCR_API int accr_probe_fma(int32_t ctas, int64_t rounds, float *sink, accr_stream_t stream) {
    ACCR_TRACE("accr_probe_fma");
    accr::clear_error();
    if (ctas < 1 || rounds < 1 || !sink) return accr::set_error(ACCR_EINVAL, "accr_probe_fma: bad arguments");
    int rc = accr::launch_guard("fma_probe_kernel");
    if (rc != ACCR_OK) return rc;
    accr::fma_probe_kernel<<<ctas, accr::PROBE_THREADS, 0, (cudaStream_t)stream>>>(rounds, sink, 0.999f, 0.001f);
    return accr::launched("fma_probe_kernel");
}

extern "C" ACCR_API int accr_probe_fma_packed(int32_t ctas, int64_t rounds, float *sink, accr_stream_t stream) {
    ACCR_TRACE("accr_probe_fma_packed");
    accr::clear_error();
    if (ctas < 1 || rounds < 1 || !sink) return accr::set_error(ACCR_EINVAL, "accr_probe_fma_packed: bad arguments");
    int rc = accr::launch_guard("fma2_probe_kernel");
    if (rc != ACCR_OK) return rc;
    accr::fma2_probe_kernel<<<ctas, accr::PROBE_THREADS, 0, (cudaStream_t)stream>>>(rounds, sink, 0.999f, 0.001f);
    return accr::launched("fma2_probe_kernel");
}
