// copy_planes.cu -- a state's planes to or from a caller's device arrays in one launch.
//
// A copy call per plane and a separate read of the error word cost a few us each, and a
// strided copy runs far below the memory's rate; here one kernel moves all planes and stores
// the error word in page-locked memory, so that the caller waits once.  Repeated calls, us,
// copy calls against this: three planes read from 64^2 26.5 -> 11.6 (launch and wait), 1024^2
// 40.6 -> 13.2, 4096^2 226 -> 70 (bandwidth, part of it from L2); all planes set at 64^2
// 25.3 -> 14.1, 101^3 76 -> 20, 512^3 2304 -> 1231.  No size was found where the calls are better
// (9^3 to 4099^2, 5 x 917490, 10^6 x 4, aligned arrays and others).
//
// A kernel must not touch memory that a copy call would have refused or staged, so the
// launch is taken only for arrays that the driver says lie whole in one plain device
// allocation of the state's context, are float-aligned, and overlap neither one another
// nor the state; everything else (managed or pinned host memory, another device, pool or
// virtual memory, a wrong pointer) stays with the copy calls.
#include <algorithm>

#include "copy_planes.h"
#include "gals_internal.h"
#include "tma.cuh"

namespace gals {
namespace {

constexpr int kCopyThreads = 256, kCopyWarps = kCopyThreads / 32, kCopyPiece = 512;

struct PlaneSet {
    const float *src[kMaxCopyPlanes];
    float *dst[kMaxCopyPlanes];
};

__device__ __forceinline__ void report(const int *err, int *err_host)
{
    if (err_host && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *err_host = *err;
}

// Rows of different pitch: a warp per piece of kCopyPiece nodes of a row, four loads in flight
// per lane.  With whole rows a state of few, long ones kept a handful of warps busy (three
// planes of 10^6 x 4 nodes: 2882 us in whole rows, 21 in pieces, 75 by copy calls).
__global__ void __launch_bounds__(kCopyThreads)
k_copy_rows(const __grid_constant__ PlaneSet ps, int n0, int64_t rows, int pieces, int64_t spitch, int64_t dpitch,
            const int *err, int *err_host)
{
    pdl_wait();
    const float *src = ps.src[blockIdx.y];
    float *dst = ps.dst[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * kCopyWarps;
    for (int64_t w = (int64_t)blockIdx.x * kCopyWarps + (threadIdx.x >> 5); w < rows * pieces; w += step) {
        const int64_t r = pieces == 1 ? w : w / pieces;
        const int c0 = (int)(w - r * pieces) * kCopyPiece, end = min(n0 - c0, kCopyPiece);
        const float *s = src + r * spitch + c0;
        float *d = dst + r * dpitch + c0;
        for (int c = lane; c < end; c += 128) {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c + 32 * k < end) v[k] = s[c + 32 * k];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c + 32 * k < end) d[c + 32 * k] = v[k];
        }
    }
    report(err, err_host);
}

// Dense planes, 16-byte aligned on both sides.
__global__ void __launch_bounds__(kCopyThreads)
k_copy_dense(const __grid_constant__ PlaneSet ps, int64_t n4, const int *err, int *err_host)
{
    pdl_wait();
    const float4 *src = reinterpret_cast<const float4 *>(ps.src[blockIdx.y]);
    float4 *dst = reinterpret_cast<float4 *>(ps.dst[blockIdx.y]);
    for (int64_t i = (int64_t)blockIdx.x * (4 * kCopyThreads) + threadIdx.x; i < n4;
         i += (int64_t)gridDim.x * (4 * kCopyThreads)) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * kCopyThreads < n4) v[k] = src[i + k * kCopyThreads];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * kCopyThreads < n4) dst[i + k * kCopyThreads] = v[k];
    }
    report(err, err_host);
}

// What the driver says of an address (cuPointerGetAttributes, through the runtime's entry
// points); context 0 if it is no plain device memory or the driver says nothing.
struct Allocation {
    void *context = nullptr;
    int device = -1;
    uintptr_t start = 0;
    size_t size = 0;
};

Allocation allocation_of(const void *p)
{
    typedef CUresult (*GetAttributes)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static GetAttributes fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<GetAttributes>(f);
    }();
    Allocation a;
    if (!fn) return a;
    void *context = nullptr;
    unsigned type = 0, managed = 1;
    int device = -1;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute at[6] = {CU_POINTER_ATTRIBUTE_CONTEXT, CU_POINTER_ATTRIBUTE_MEMORY_TYPE,
                                 CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                 CU_POINTER_ATTRIBUTE_RANGE_SIZE, CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL};
    void *out[6] = {&context, &type, &managed, &start, &size, &device};
    if (fn(6, at, out, (CUdeviceptr)p) != CUDA_SUCCESS || type != CU_MEMORYTYPE_DEVICE || managed) return a;
    a.context = context;
    a.device = device;
    a.start = (uintptr_t)start;
    a.size = size;
    return a;
}

}  // namespace

cudaError_t copy_planes(const PlaneCopy &c, cudaStream_t s, bool *done)
{
    *done = false;
    const int64_t count = c.n0 * c.rows;
    if (c.planes > kMaxCopyPlanes) return cudaSuccess;
    const size_t bytes = sizeof(float) * (size_t)count;
    const Allocation own = allocation_of(c.state);
    int current = -1;
    if (!own.context || cudaGetDevice(&current) != cudaSuccess || current != own.device) return cudaSuccess;
    Allocation a;
    for (int p = 0; p < c.planes; ++p) {
        const uintptr_t u = (uintptr_t)c.user[p];
        if (u % sizeof(float)) return cudaSuccess;
        // the planes of one array share an allocation
        if (!a.context || u < a.start || u - a.start >= a.size) a = allocation_of(c.user[p]);
        if (a.context != own.context || a.start == own.start || u < a.start || a.size < bytes ||
            u - a.start > a.size - bytes)
            return cudaSuccess;
        for (int q = 0; q < p; ++q) {
            const uintptr_t o = (uintptr_t)c.user[q];
            if (u < o + bytes && o < u + bytes) return cudaSuccess;
        }
    }
    PlaneSet ps{};
    bool dense = c.pitch == c.n0;
    for (int p = 0; p < c.planes; ++p) {
        float *mine = c.state + p * c.plane;
        ps.src[p] = c.to_user ? mine : c.user[p];
        ps.dst[p] = c.to_user ? c.user[p] : mine;
        dense = dense && (uintptr_t)c.user[p] % 16 == 0;
    }
    const int pieces = (int)((c.n0 + kCopyPiece - 1) / kCopyPiece);
    const int64_t work = dense ? (count / 4 + 4 * kCopyThreads - 1) / (4 * kCopyThreads)
                               : (c.rows * pieces + kCopyWarps - 1) / kCopyWarps;
    const dim3 grid((unsigned)std::min<int64_t>(work, 4096), (unsigned)c.planes);
    *done = true;
    if (dense) return launch_kernel(k_copy_dense, grid, dim3(kCopyThreads), 0, s, true, ps, count / 4, c.err, c.err_host);
    return launch_kernel(k_copy_rows, grid, dim3(kCopyThreads), 0, s, true, ps, (int)c.n0, c.rows, pieces,
                         c.to_user ? c.pitch : c.n0, c.to_user ? c.n0 : c.pitch, c.err, c.err_host);
}

}  // namespace gals
