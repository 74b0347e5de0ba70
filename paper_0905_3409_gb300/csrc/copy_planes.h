// copy_planes.h -- one-launch copies between a state's planes and a caller's device arrays.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gals {

constexpr int kMaxCopyPlanes = 8;

struct PlaneCopy {
    float *state;          // first plane of the state; its allocation holds nothing of the caller's
    int64_t plane, pitch;  // floats from plane to plane and from row to row of the state
    int64_t n0, rows;      // extent of a plane; the caller's arrays are dense
    float *const *user;    // one array per plane
    int planes;
    bool to_user;
    const int *err;        // with err_host: *err is stored to *err_host (page-locked) after all
    int *err_host;         // earlier work of the stream
};

// Queue the copy on s if it can be one launch (done: whether it was).
cudaError_t copy_planes(const PlaneCopy &c, cudaStream_t s, bool *done);

}  // namespace gals
