// Device memory for the length of one call (the training entry points, which have no context to keep it in).
#ifndef APEX_WORKSPACE_HPP
#define APEX_WORKSPACE_HPP

#include <cuda_runtime.h>

#include <cstddef>

namespace apex {

// From the library's own memory pool of the current device.  cudaMalloc and cudaFree, which synchronise, took 0.6 ms of a
// call (T = 8192: confidence-model fit 3.9 -> 3.2 ms, router distillation 8.6 -> 7.9); the pool hands the same memory out
// again in 15 us.  It is given back in front of a call's last synchronisation, where the pool keeps kWorkspaceKept bytes at most and the
// system gets the rest; these go back when a context is created or destroyed and on apex_trim_scratch (workspace_trim).
// What the pool hands out is ordered by the streams it is used on, and it may be used from several threads.  Not while `s` is captured: the
// calls wait.
constexpr size_t kWorkspaceKept = 64u << 20;
cudaError_t workspace_alloc(void** out, size_t bytes, cudaStream_t s);
void workspace_free(void* p, cudaStream_t s);
cudaError_t workspace_trim();  // of the current device

}  // namespace apex

#endif  // APEX_WORKSPACE_HPP
