// Products of a head's S with C and m, for converting between the paper's tuple (S, C, m, G, h) and
// the (S, D, e) form of the carries: D = S C - G, e = S m - h.
#pragma once

namespace hla {
namespace {

constexpr int kStateRows = 16;      // rows of a block
constexpr int kStateThreads = 256;

// emit(a, b, (S C)_ab) for rows a0 .. a0 + 15 and columns b < dv, and emit(a, dv, (S m)_a).  A thread
// takes four rows of a column at a time, so one load of C serves four multiply-adds (at one each the
// kernel waited on L1: 42 us for 32 heads of 128 x 128, now 30, both from cold caches).  `rows` is 16 x 128 floats of
// shared memory.
template <typename F>
__device__ __forceinline__ void state_products(const float *__restrict__ S, const float *__restrict__ C,
                                               const float *__restrict__ m, int d, int dv, int a0, float *rows, F emit) {
    for (int i = threadIdx.x * 4; i < kStateRows * d; i += kStateThreads * 4)
        *reinterpret_cast<float4 *>(rows + i) = *reinterpret_cast<const float4 *>(S + (long long)a0 * d + i);
    __syncthreads();
    for (int u = threadIdx.x; u < (kStateRows / 4) * dv; u += kStateThreads) {
        const int b = u % dv, r = (u / dv) * 4;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int j = 0; j < d; j += 4) {
            float c[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) c[x] = C[(long long)(j + x) * dv + b];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 s = *reinterpret_cast<const float4 *>(rows + (r + i) * d + j);
                acc[i] = fmaf(s.x, c[0], acc[i]);
                acc[i] = fmaf(s.y, c[1], acc[i]);
                acc[i] = fmaf(s.z, c[2], acc[i]);
                acc[i] = fmaf(s.w, c[3], acc[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) emit(a0 + r + i, b, acc[i]);
    }
    // S m: a warp per row
    for (int r = threadIdx.x >> 5; r < kStateRows; r += kStateThreads / 32) {
        float s = 0.f;
        for (int j = threadIdx.x & 31; j < d; j += 32) s = fmaf(rows[r * d + j], m[j], s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) emit(a0 + r, dv, s);
    }
}

}  // namespace
}  // namespace hla
