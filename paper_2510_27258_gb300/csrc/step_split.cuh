// Parts shared by the decode steps that give a head to a cluster of blocks: the split cluster barrier
// and sums over lanes.
#pragma once

#include <cuda_runtime.h>

namespace hla {
namespace {

template <int W>
__device__ __forceinline__ float group_sum(float x) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o, W);
    return x;
}

// sum_i a[i] b[i] over shared-memory vectors, computed by every warp on its own (no block barrier)
__device__ __forceinline__ float warp_dot(const float *a, const float *b, int n) {
    float s = 0.f;
    for (int i = threadIdx.x & 31; i < n; i += 32) s += a[i] * b[i];
    return group_sum<32>(s);
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// sums of a float4 over the lanes whose lane index agrees modulo w (w a power of two, <= 32)
__device__ __forceinline__ float4 column_sum(float4 x, int w) {
    for (int o = 16; o >= w; o >>= 1) {
        x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
        x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
        x.z += __shfl_xor_sync(0xffffffffu, x.z, o);
        x.w += __shfl_xor_sync(0xffffffffu, x.w, o);
    }
    return x;
}
__device__ __forceinline__ void fma4(float4 &a, float s, const float4 &b) {
    a.x = fmaf(s, b.x, a.x); a.y = fmaf(s, b.y, a.y); a.z = fmaf(s, b.z, a.z); a.w = fmaf(s, b.w, a.w);
}
__device__ __forceinline__ float4 axpy4(const float4 &x, float s, const float4 &y) {
    float4 r = x;
    fma4(r, s, y);
    return r;
}

// a launch of `split` blocks for each of `heads` heads, as clusters unless the blocks need not meet
template <typename K, typename... A>
cudaError_t launch_blocks(K kern, int heads, int split, bool cluster, int threads, cudaStream_t stream, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = split;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(heads * split);
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = cluster && split > 1 ? 1 : 0;  // without: clusters of one block, their barrier is trivial
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace
}  // namespace hla
