// step2d.cu -- dispatch of the single-grid 2D step to the kernels of its velocity kind, and the
// 2D reconstruction kernel.
#include <algorithm>

#include "step2d_kinds.h"

namespace gals {

namespace {

// phi_xy = d/dx psi_y at every node (approach A with one-sided ends); used after
// set_state and for the COMPACT layout's read-out.  Blocks of 32 x 8 nodes; the grid's
// y dimension is capped at 65535 and its blocks stride over the rows beyond.
__global__ void __launch_bounds__(256) k_recon2d(float *__restrict__ buf, Geom g)
{
    const int i = blockIdx.x * 32 + threadIdx.x;
    if (i >= g.n0) return;
    for (int j = blockIdx.y * 8 + threadIdx.y; j < g.n1; j += gridDim.y * 8) {
        const float *py = buf + 2 * g.plane + (size_t)j * g.pitch;
        float v = dline(i, g.n0, g.i2h0, [&](int q) { return py[q]; });
        buf[3 * g.plane + (size_t)j * g.pitch + i] = v;
    }
}

}  // namespace

cudaError_t launch_step2d(const StepLaunch &a, cudaStream_t s)
{
    if (a.trace == TR_GIVEN) return step2d_given(a, s);
    switch (a.vp.kind) {
    case VK_CONST: return step2d_kind<VK_CONST>(a, s);
    case VK_ROTATION: return step2d_kind<VK_ROTATION>(a, s);
    case VK_VORTEX2D: return step2d_kind<VK_VORTEX2D>(a, s);
    case VK_PSEUDO1D: return step2d_kind<VK_PSEUDO1D>(a, s);
    case VK_FOURIER2D: return step2d_kind<VK_FOURIER2D>(a, s);
    case VK_WAVES2D: return step2d_kind<VK_WAVES2D>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step2d_run(const RunLaunch &a, cudaStream_t s)
{
    switch (a.vp.kind) {
    case VK_CONST: return run2d_kind<VK_CONST>(a, s);
    case VK_ROTATION: return run2d_kind<VK_ROTATION>(a, s);
    case VK_VORTEX2D: return run2d_kind<VK_VORTEX2D>(a, s);
    case VK_PSEUDO1D: return run2d_kind<VK_PSEUDO1D>(a, s);
    case VK_FOURIER2D: return run2d_kind<VK_FOURIER2D>(a, s);
    case VK_WAVES2D: return run2d_kind<VK_WAVES2D>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

int band_unit(int dim) { return dim == 2 ? tile_rows2d() : 4; }

cudaError_t launch_recon2d(const Geom &g, float *buf, cudaStream_t s)
{
    dim3 block(32, 8);
    dim3 grid((g.n0 + 31) / 32, std::min((g.n1 + 7) / 8, 65535));
    k_recon2d<<<grid, block, 0, s>>>(buf, g);
    return cudaGetLastError();
}

}  // namespace gals
