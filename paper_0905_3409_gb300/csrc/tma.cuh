// tma.cuh -- Tensor Memory Accelerator (TMA) tile loads and mbarrier waits (inline PTX, sm_90+).
//
// A thread block stages the state planes of its tile (with halo) into shared memory with one
// cp.async.bulk.tensor copy tracked by an mbarrier.  Every wait is bounded: after the
// iteration limit the block records an error code in device memory and gives up, so a
// lost copy can never hang the GPU; the host turns the code into GALS_ERR_TIMEOUT.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace gals {

constexpr int kErrTmaTimeout = 1;
constexpr uint32_t kWaitLimit = 1u << 24;  // try_wait polls before a wait counts as lost

// Programmatic dependent launch: wait until the kernel before this one in the stream has
// finished and its writes are visible (at once if it was not launched as its dependent), and
// let the one after it be placed while this one runs.  Every kernel that is launched as a
// dependent waits before its first read or write of global memory.  The step kernels release
// late (3D: at a thread's last pair of nodes) or at their end: blocks of the next step placed
// at their start took the places unevenly (64 x 60 x 50: 9.6 us per step against 8.0).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of the barrier; false if `limit` polls ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  uint32_t limit = kWaitLimit)
{
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// Wait of a whole block for a staged copy: every thread polls (bounded), then the block
// takes one verdict at a barrier (false: the wait ran out for some thread), so that no
// thread is left behind at a later barrier.  Must be reached by every thread.
__device__ __forceinline__ bool mbar_wait_block(uint64_t *bar, uint32_t parity,
                                                uint32_t limit = kWaitLimit)
{
    const bool ok = mbar_wait_bounded(bar, parity, limit);
    return !__syncthreads_or(!ok);
}

// 3D tiled bulk copy global -> shared, completion counted on `bar` (bytes of the box).
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int c0, int c1,
                                            int c2, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

// 4D variant (x, y, z, plane) for 3D grids.
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int c0, int c1,
                                            int c2, int c3, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(smem_u32(bar))
        : "memory");
}

}  // namespace gals
