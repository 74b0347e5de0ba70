// step2d_linear.cu -- the 2D step kernels of the constant, rotation and pseudo-1D fields, and of given feet.
#include "step2d_kernels.cuh"

namespace gals {

template cudaError_t step2d_kind<VK_CONST>(const StepLaunch &, cudaStream_t);
template cudaError_t run2d_kind<VK_CONST>(const RunLaunch &, cudaStream_t);
template cudaError_t step2d_kind<VK_ROTATION>(const StepLaunch &, cudaStream_t);
template cudaError_t run2d_kind<VK_ROTATION>(const RunLaunch &, cudaStream_t);
template cudaError_t step2d_kind<VK_PSEUDO1D>(const StepLaunch &, cudaStream_t);
template cudaError_t run2d_kind<VK_PSEUDO1D>(const RunLaunch &, cudaStream_t);

cudaError_t step2d_given(const StepLaunch &a, cudaStream_t s) { return launch_cr<TR_GIVEN, VK_CONST>(a, s); }

int tile_rows2d() { return TY; }

int run2d_tiles(const Geom &g) { return ((g.n0 + TX - 1) / TX) * ((g.n1 + TY - 1) / TY); }

int run2d_max_cells(int axis) { return axis == 0 ? TX - 2 : TY - 2; }

void tile_box2d(int is_short, int np, uint32_t box[3])
{
    box[0] = TWS;
    box[1] = is_short ? Geo<TYS, HYT, TWS>::TH : GT::TH;
    box[2] = (uint32_t)np;
}

}  // namespace gals
