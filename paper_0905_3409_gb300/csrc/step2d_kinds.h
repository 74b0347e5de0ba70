// step2d_kinds.h -- the 2D step launchers of each velocity kind (step2d_*.cu).
#pragma once

#include "gals_internal.h"

namespace gals {

template <int VK> cudaError_t step2d_kind(const StepLaunch &a, cudaStream_t s);
template <int VK> cudaError_t run2d_kind(const RunLaunch &a, cudaStream_t s);
cudaError_t step2d_given(const StepLaunch &a, cudaStream_t s);  // TR_GIVEN: no velocity

}  // namespace gals
