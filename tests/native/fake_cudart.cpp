// fake_cudart.cpp -- a stand-in for the CUDA runtime (no GPU): four devices, function
// attributes and the largest cluster per device, launches checked against them.
#include <map>
#include <set>
#include <utility>

#include <cuda_runtime_api.h>

#include "fake_cudart.h"

thread_local int fake_device = 0;
int fake_placeable[4] = {16, 16, 8, 0}, fake_launches = 0, fake_refused = 0, fake_cluster = 0;

namespace {

std::map<std::pair<int, const void *>, int> smem_allowed;  // dynamic bytes beyond the default
std::set<std::pair<int, const void *>> large_clusters;
dim3 push_grid, push_block;
size_t push_smem = 0;

cudaError_t check(const void *f, size_t smem, int cluster)
{
    // 36 KB: what is left of the default 48 KB beside the largest static part (a batch tile's)
    const auto it = smem_allowed.find({fake_device, f});
    bool ok = smem <= 36 * 1024 || (it != smem_allowed.end() && smem <= (size_t)it->second);
    if (cluster > 8 && !large_clusters.count({fake_device, f})) ok = false;
    if (cluster > 1 && cluster > fake_placeable[fake_device]) ok = false;
    (ok ? fake_launches : fake_refused)++;
    return ok ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
char __cudaInitModule(void **) { return 0; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t)
{
    push_grid = g; push_block = b; push_smem = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st)
{
    *g = push_grid; *b = push_block; *s = push_smem;
    *(void **)st = nullptr;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t s, cudaStream_t) { return check((const void *)k, s, 1); }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t s, cudaStream_t) { return check(f, s, 1); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    int cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = (int)c->attrs[i].val.clusterDim.x;
    if (cluster > 1) fake_cluster = cluster;
    return check(f, c->dynamicSmemBytes, cluster);
}
cudaError_t cudaGetLastError() { return fake_refused ? cudaErrorInvalidValue : cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = fake_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_allowed[{fake_device, f}] = v;
    if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && v) large_clusters.insert({fake_device, f});
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c)
{
    const int want = (int)c->attrs[0].val.clusterDim.x;
    *n = want <= fake_placeable[fake_device] && (want <= 8 || large_clusters.count({fake_device, f})) ? 1 : 0;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    *n = 4;
    return cudaSuccess;
}
}
