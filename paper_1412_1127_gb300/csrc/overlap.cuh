// overlap.cuh -- launches whose set-up overlaps the end of the stream's previous
// kernel (programmatic dependent launch).
//
// Back-to-back kernels of a stream start about 2 us apart however short they are
// (an empty grid measured 4.1 us a call, ordinary launches' times come in steps of
// 2.05 us): draining one grid and setting up the next are serial.  With the next
// grid's CTAs set up while this one runs, a region of no elements takes 2.2 us
// (4.1 before), 2^16 int32 5.2 (8.2), 2^20 6.2 (8.2), 2^24 8.9 (12.3).
// Cooperative launches and kernels behind copies keep the ordinary order.
#pragma once

#include <cuda_runtime.h>
#include <string.h>

namespace accr {

// In a kernel launched with launch_overlapped, ahead of everything but a CTA's set-up
// of its own shared memory: waits until the previous kernel of the stream has finished
// and its writes are visible, then lets the stream's next kernel be set up in turn.
// Nothing of this kernel's inputs, outputs or scratch is touched before, and nothing
// is held that a predecessor could wait for (tensor memory).
__device__ __forceinline__ void grid_dependency() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Inputs are read by ordinary loads, not by the read-only path (ld.global.nc, __ldg,
// const __restrict__ parameters): PTX defines that for memory nothing writes while
// the kernel lives, and this kernel's life begins while its predecessor may still be
// writing.  A streaming 16-byte load (read once: no L1 allocation, 256-byte L2
// fetch), volatile with a memory clobber so that none moves above the wait.  Its rate
// is the read-only path's (2^28 floats, sum + max + min: 158.1 us both ways).
__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

template <typename T>
struct SameType {
    using type = T;
};

// Launches `kernel` so; a failure is left to cudaGetLastError, as with <<<>>>.
template <typename... P>
inline void launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                              const typename SameType<P>::type &...args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *ptrs[] = {(void *)&args...};
    cudaLaunchKernelExC(&cfg, (const void *)kernel, ptrs);
}

}  // namespace accr
