// overlap.cuh -- launches whose set-up overlaps the end of the stream's previous
// kernel (programmatic dependent launch).
//
// Back-to-back kernels of a stream start about 2 us apart however short they are
// (an empty grid measured 4.1 us a call, ordinary launches' times come in steps of
// 2.05 us): draining one grid and setting up the next are serial.  With the next
// grid's CTAs set up while this one runs, a region of no elements takes 2.6 us
// (4.1 before), 2^16 int32 5.2 (8.2), 2^20 6.2 (8.2), 2^24 8.9 (12.3).
// Cooperative launches and kernels behind copies keep the ordinary order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace accr {

// In a kernel launched with launch_overlapped, ahead of everything but a CTA's set-up
// of its own shared memory: waits until the previous kernel of the stream has finished
// and its writes are visible.  Nothing of this kernel's inputs, outputs or scratch is
// touched before, and nothing is held that a predecessor could wait for (tensor
// memory).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the stream's next kernel be set up, once every CTA has come here or is done: near
// the end of a CTA's work, not earlier.  The waiting grid holds threads and registers,
// which kernels of other streams then lack: released at the first statement, a small
// region beside a queue of 2^28 regions took 154-298 us (87 without any of this, 80-87
// so), beside LEN 2048 nests 414 (33, 40-43).  The set-up takes about 2 us; CTAs
// run apart by some rounds, so streaming kernels release with about RELEASE_BYTES left
// in the grid, 15 us at HBM's rate (at the last round alone 2^28 floats took 159.0
// instead of 158.2 us, 400,000 rows of 61 21.4 instead of 19.7).  (No memory clobber:
// the next grid waits for this one's end whatever stands on either side.)
constexpr int64_t RELEASE_BYTES = (int64_t)96 << 20;
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;"); }

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
