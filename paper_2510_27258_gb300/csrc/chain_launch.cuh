// Launches of one call that follow one another: each is set up while the one before it drains
// (programmatic dependent launch).  A kernel launched so calls chain_begin() before it touches global
// memory: that returns once every block of the launch before it has finished and its writes are
// visible.  The first launch of a call is an ordinary one.
// Measured, ordinary -> so, us: fp32 forward of 8 heads of 200 x 32 33.5 -> 22.0 (five launches), B2 H16
// n1000 d64 80.5 -> 78.2, the tiled backward B2 H16 n4096 d128 527 -> 506 (nine), 8 heads of 1000 65 -> 52.
// No kernel lets the next one in before its own blocks have ended (griddepcontrol.launch_dependents):
// blocks that come early crowd the SMs that are free first, which took the tiled backward to 593 us.
// The one exception is the forward before a final state, whose next launch needs nothing of it.
#pragma once

#include <cuda_runtime.h>

namespace hla {
namespace {

__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename K, typename... A>
cudaError_t chain_launch(bool follows, K kern, dim3 grid, int threads, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = follows ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace
}  // namespace hla
