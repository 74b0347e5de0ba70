// step2d_waves.cu -- the 2D step kernels of the plane-wave stream function.
#include "step2d_kernels.cuh"

namespace gals {

template cudaError_t step2d_kind<VK_WAVES2D>(const StepLaunch &, cudaStream_t);
template cudaError_t run2d_kind<VK_WAVES2D>(const RunLaunch &, cudaStream_t);

}  // namespace gals
