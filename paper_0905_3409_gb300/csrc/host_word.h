// host_word.h -- page-locked words of host memory, which the device stores to and a handle reads.
#pragma once

#include <cuda_runtime.h>

namespace gals {

// A word for the current device's context; give it back with release_host_word when no queued
// work stores to it any more.  Both from any thread.
struct HostWord {
    int *at = nullptr;
    unsigned long long context = 0;
};
cudaError_t acquire_host_word(HostWord *word);
void release_host_word(const HostWord &word);

// Unique id of the driver's current context, never reused within a process; 0 when no context
// is current or the driver does not tell.
unsigned long long current_context_id();

}  // namespace gals
