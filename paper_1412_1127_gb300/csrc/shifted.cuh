// shifted.cuh -- vector loads of matrix rows that start anywhere.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace accr {

// NV float4s of consecutive elements x[i ..), i any index, from the 16-byte vectors
// that hold them: a row of a matrix whose length is not a multiple of four starts
// anywhere, and element by element its loads cost the split of LEN 4095 70 us more
// than that of 4096.  Vectors that reach outside x[0, total) go element by element;
// elements there are not needed by the caller and read as zero.
template <int NV>
__device__ __forceinline__ void load_shifted(const float *x, int64_t i, int64_t total, float (&out)[4 * NV]) {
    const int m = (int)(((uintptr_t)(x + i) >> 2) & 3);  // elements before x[i] in its vector
    const int64_t v0 = i - m;
    float w[4 * NV + 4];
#pragma unroll
    for (int j = 0; j <= NV; ++j) {
        const int64_t e = v0 + 4 * j;
        if (e >= 0 && e + 4 <= total) {
            const float4 q = (j < NV || m > 0) ? *reinterpret_cast<const float4 *>(x + e) : make_float4(0.f, 0.f, 0.f, 0.f);
            w[4 * j] = q.x, w[4 * j + 1] = q.y, w[4 * j + 2] = q.z, w[4 * j + 3] = q.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) w[4 * j + k] = (e + k >= 0 && e + k < total) ? x[e + k] : 0.f;
        }
    }
    if (m & 1) {
#pragma unroll
        for (int k = 0; k < 4 * NV + 3; ++k) w[k] = w[k + 1];
    }
    if (m & 2) {
#pragma unroll
        for (int k = 0; k < 4 * NV + 2; ++k) w[k] = w[k + 2];
    }
#pragma unroll
    for (int k = 0; k < 4 * NV; ++k) out[k] = w[k];
}

}  // namespace accr
