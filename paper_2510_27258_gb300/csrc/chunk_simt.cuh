// Block-level fp32 products on the CUDA cores for the chunk-parallel kernels (second-order forward,
// AHLA forward, backward), and the prefix sums over chunks that connect them.
//
// A block of 128 threads works on one chunk of 64 tokens.  Operands sit in shared memory as fp32
// rows of N + 4 floats (N = 32, 64 or 128, the head sizes padded with zeros), masked chunk tiles as
// rows of 68; a carry (d x dv, fp32, in global memory) streams through shared memory 16 rows at a
// time (eight at N = 64).  What bounds a product is the shared-memory bandwidth (128 bytes per clock and SM, so a
// 16-byte load of a warp costs four clocks) against four fp32 warp multiply-adds per clock: a thread
// therefore keeps 8 x 8 outputs (8 x 4 at N = 64, 4 x 4 at N = 32) and every load brings 16 bytes,
// 16 loads per 256 multiply-adds at N = 128.  The eight lanes that share a load phase read either
// one address (the row operand) or 128 contiguous bytes (the column operand), so no load has a bank
// conflict.  Rows of a thread are 4 rg .. 4 rg + 3 and 32 + 4 rg .. + 3: of a lower triangular
// operand the upper right quadrant is then skipped by all warps alike.
// Multiply-adds go two to an instruction (fma.rn.f32x2): with one each, the schedulers issued on 56 to
// 68 % of the cycles and stalled on dispatch while the fp32 pipe was half idle.  In pairs: the backward
// of B2 H16 n4096 d128 2331 -> 2087 us, AHLA B1 H32 n1999 d128 with states 404 -> 338 us, the forward of
// B2 H16 n1000 d64 fp32 97 -> 84 us.
#pragma once

#include <type_traits>

#include "chain_launch.cuh"
#include "hla_internal.h"

namespace hla {
namespace {

// Blocks of a (chunk, head) lie along the grid's first dimension, the chunks of a head side by side: the other two
// end at 65535, which heads may pass (chunk_grid, chunk_of).
constexpr int kC = 64;        // tokens of a chunk
constexpr int kCT = 128;      // threads of a block
constexpr int kLdW = kC + 4;  // row length of a masked chunk tile

template <int N>
struct Tile {
    static constexpr int RM = N == 32 ? 4 : 8, CM = N == 128 ? 8 : 4;  // outputs of a thread
    static constexpr int LD = N + 4;
    // rows of a carry in shared memory at a time: at N = 64 eight, so that four blocks fit an SM
    static constexpr int SL = N == 64 ? 8 : 16;
    int rg, cg;
    __device__ Tile() {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (N == 32) {
            cg = lane & 7;
            rg = warp * 4 + (lane >> 3);
        } else {
            cg = (warp & 1) * 8 + (lane & 7);
            rg = (warp >> 1) * 4 + (lane >> 3);
        }
    }
    __device__ __forceinline__ int row(int i) const { return (i >> 2) * 32 + 4 * rg + (i & 3); }
    __device__ __forceinline__ int col(int j) const { return (j >> 2) * 64 + 4 * cg + (j & 3); }
};

// Two fp32 values in a register pair: fma2 is one instruction for two independent fp32 multiply-adds
// (each rounded as fmaf).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float lo(f32x2 v) { return __uint_as_float(static_cast<unsigned>(v)); }
__device__ __forceinline__ float hi(f32x2 v) { return __uint_as_float(static_cast<unsigned>(v >> 32)); }
__device__ __forceinline__ void fma2(f32x2 &d, f32x2 a, f32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// a thread's outputs, two neighbouring columns in a pair
template <int N>
struct Acc {
    f32x2 p[Tile<N>::RM][Tile<N>::CM / 2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < Tile<N>::RM; ++i)
#pragma unroll
            for (int j = 0; j < Tile<N>::CM / 2; ++j) p[i][j] = 0ull;
    }
    __device__ __forceinline__ float get(int i, int j) const { return j & 1 ? hi(p[i][j >> 1]) : lo(p[i][j >> 1]); }
    // x(r, c) <- f(x(r, c), i, j)
    template <typename F>
    __device__ __forceinline__ void each(F f) {
#pragma unroll
        for (int i = 0; i < Tile<N>::RM; ++i)
#pragma unroll
            for (int j = 0; j < Tile<N>::CM / 2; ++j)
                p[i][j] = pack2(f(lo(p[i][j]), i, 2 * j), f(hi(p[i][j]), i, 2 * j + 1));
    }
};

__device__ __forceinline__ float f4(const float4 &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// 16-byte aligned vector loads of tokens as fp32: 4 fp32 or 8 bf16 elements a load
template <typename T>
struct Vec;
template <>
struct Vec<float> {
    static constexpr int W = 4;
    __device__ static __forceinline__ void load(const float *p, float *o) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
    __device__ static __forceinline__ void store4(float *p, const float *x) {
        *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
    }
};
template <>
struct Vec<__nv_bfloat16> {
    static constexpr int W = 8;
    __device__ static __forceinline__ void load(const __nv_bfloat16 *p, float *o) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // a bf16 is the upper half of the fp32 with the same value
            o[2 * i] = __uint_as_float(w[i] << 16);
            o[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    __device__ static __forceinline__ void store4(__nv_bfloat16 *p, const float *x) {
        __nv_bfloat162 h[2] = {__floats2bfloat162_rn(x[0], x[1]), __floats2bfloat162_rn(x[2], x[3])};
        *reinterpret_cast<uint2 *>(p) = *reinterpret_cast<uint2 *>(h);
    }
};

// token rows [rows][width] (width a multiple of 16) into shared rows of N + 4 floats; zero beyond
// the rows and the width.  Returns 0 if all that this thread loaded is finite, else NaN.
template <int N, typename T>
__device__ __forceinline__ float load_tile(float *dst, const T *__restrict__ src, int rows, int width) {
    constexpr int W = Vec<T>::W, PER = N / W;
    float seen = 0.f;
#pragma unroll 4
    for (int i = threadIdx.x; i < kC * PER; i += kCT) {
        const int r = i / PER, c = (i % PER) * W;
        float x[W];
#pragma unroll
        for (int j = 0; j < W; ++j) x[j] = 0.f;
        if (r < rows && c < width) Vec<T>::load(src + (long long)r * width + c, x);
#pragma unroll
        for (int j = 0; j < W; ++j) seen = fmaf(x[j], 0.f, seen);
#pragma unroll
        for (int j = 0; j < W; j += 4)
            *reinterpret_cast<float4 *>(dst + r * (N + 4) + c + j) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
    }
    return seen;
}
// block barrier; on return true in every thread if any `seen` is not zero (N = 32, whose products do not ask: false)
template <int N>
__device__ __forceinline__ bool sync_unless_finite(float seen) {
    if constexpr (N == 32) {
        __syncthreads();
        return false;
    } else {
        return __syncthreads_or(!(seen == 0.f)) != 0;
    }
}

// acc[I0..][.] += sum_{k0 <= k < k1} A(r, k) B(k, c), A row-major in shared memory, B rows over c.
// I0 = 4: only the second half of the rows (A is zero there for the first half).  kDiag: the terms k <= r alone.
template <int N, int I0, bool kDiag = false>
__device__ __forceinline__ void nn_range(Acc<N> &acc, const Tile<N> &t, const float *A, int lda, const float *B,
                                         int ldb, int k0, int k1) {
    constexpr int RM = Tile<N>::RM, CM = Tile<N>::CM;
    for (int k = k0; k < k1; k += 4) {
        float4 x[RM];
#pragma unroll
        for (int i = I0; i < RM; ++i) x[i] = *reinterpret_cast<const float4 *>(A + t.row(i) * lda + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            f32x2 y[CM / 2];
#pragma unroll
            for (int j = 0; j < CM; j += 4) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(B + (k + kk) * ldb + t.col(j));
                y[j / 2] = v.x; y[j / 2 + 1] = v.y;
            }
#pragma unroll
            for (int i = I0; i < RM; ++i) {
                if (kDiag && k + kk > t.row(i)) continue;
                const f32x2 xx = pack2(f4(x[i], kk), f4(x[i], kk));
#pragma unroll
                for (int j = 0; j < CM / 2; ++j) fma2(acc.p[i][j], xx, y[j]);
            }
        }
    }
}
template <int N>
__device__ __forceinline__ void nn(Acc<N> &acc, const Tile<N> &t, const float *A, int lda, const float *B, int ldb,
                                   int K) {
    nn_range<N, 0>(acc, t, A, lda, B, ldb, 0, K);
}
// The same where B has rows that are not finite: A a lower triangular chunk tile, row r takes the rows k <= r of B
// (kUpper: A(k, r), the rows k >= r) and no other.
template <int N, bool kUpper>
__device__ __forceinline__ void masked_rows(Acc<N> &acc, const Tile<N> &t, const float *A, const float *B) {
    constexpr int RM = Tile<N>::RM, CM = Tile<N>::CM;
#pragma unroll 1
    for (int k = 0; k < kC; ++k)
#pragma unroll
        for (int i = 0; i < RM; ++i) {
            const int r = t.row(i);
            if (kUpper ? k < r : k > r) continue;
            const float x = kUpper ? A[k * kLdW + r] : A[r * kLdW + k];
#pragma unroll
            for (int j = 0; j < CM; j += 2)
                fma2(acc.p[i][j / 2], pack2(x, x), *reinterpret_cast<const f32x2 *>(B + k * (N + 4) + t.col(j)));
        }
}
// A a lower triangular chunk tile; K, at N = 32, the tokens that count.  B may have rows that are not finite, and a
// product over whole quadrants multiplies them by the zeros above the diagonal, which would make NaN of earlier
// tokens' rows.  N = 32: a warp's sixteen rows take the terms of the triangle alone (B8 H16 n1000 d32 fp32 99.8 -> 94.8
// us, as what lies beyond a warp's rows is left out).  N = 64, 128: only where `any` (the same in every thread) says
// that there are such rows; finding out costs one multiply-add per loaded value (B2 H16 n1000 d64 fp32 67.5 us without,
// 67.7 with), the triangle alone took 69.8.
template <int N>
__device__ __forceinline__ void nn_lower(Acc<N> &acc, const Tile<N> &t, const float *A, const float *B, bool any,
                                         int K = kC) {
    if constexpr (N == 32) {
        const int rb = t.row(0) & ~15;  // uniform in a warp
        nn_range<N, 0>(acc, t, A, kLdW, B, N + 4, 0, min(rb, K));
        nn_range<N, 0, true>(acc, t, A, kLdW, B, N + 4, rb, min(rb + 16, K));
    } else {
        if (any) return masked_rows<N, false>(acc, t, A, B);
        nn_range<N, 0>(acc, t, A, kLdW, B, N + 4, 0, 32);
        nn_range<N, 4>(acc, t, A, kLdW, B, N + 4, 32, 64);
    }
}

// acc[I0..I1)[.] += sum_{k0 <= k < k1} A(k, r0 + r) B(k, c): the transposed use of a row-major A.  kDiag: the terms
// k >= r alone.
template <int N, int I0, int I1, bool kDiag = false>
__device__ __forceinline__ void tn_range(Acc<N> &acc, const Tile<N> &t, const float *A, int lda, const float *B,
                                         int k0, int k1) {
    constexpr int CM = Tile<N>::CM;
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        float x[I1];
        f32x2 y[CM / 2];
#pragma unroll
        for (int i = I0; i < I1; i += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(A + k * lda + t.row(i));
            x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
        }
#pragma unroll
        for (int j = 0; j < CM; j += 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(B + k * (N + 4) + t.col(j));
            y[j / 2] = v.x; y[j / 2 + 1] = v.y;
        }
#pragma unroll
        for (int i = I0; i < I1; ++i) {
            if (kDiag && k < t.row(i)) continue;
            const f32x2 xx = pack2(x[i], x[i]);
#pragma unroll
            for (int j = 0; j < CM / 2; ++j) fma2(acc.p[i][j], xx, y[j]);
        }
    }
}
template <int N>
__device__ __forceinline__ void tn(Acc<N> &acc, const Tile<N> &t, const float *A, int lda, const float *B) {
    tn_range<N, 0, Tile<N>::RM>(acc, t, A, lda, B, 0, kC);
}
// A a lower triangular chunk tile (A(k, r) = 0 for k < r); `any` as above
template <int N>
__device__ __forceinline__ void tn_lower(Acc<N> &acc, const Tile<N> &t, const float *A, const float *B, bool any) {
    if constexpr (N == 32) {
        const int rb = t.row(0) & ~15;
        tn_range<N, 0, 4, true>(acc, t, A, kLdW, B, rb, rb + 16);
        tn_range<N, 0, 4>(acc, t, A, kLdW, B, rb + 16, kC);
    } else {
        if (any) return masked_rows<N, true>(acc, t, A, B);
        tn_range<N, 0, 4>(acc, t, A, kLdW, B, 0, 32);
        tn_range<N, 0, 8>(acc, t, A, kLdW, B, 32, 64);
    }
}

// Wt = L . (A B^T + r 1^T): the masked 64 x 64 chunk tile of two row-major operands with rows of
// `ld` floats (K of them used); r (64 floats in shared memory) may be null.  The columns of a thread
// are 16 apart, so that eight lanes read eight rows of B at 4-bank steps.
__device__ __forceinline__ void nt_masked(float *Wt, const float *A, const float *B, int ld, int K, const float *r) {
    const Tile<64> t;
    f32x2 acc[8][4];  // even and odd k apart: both operands of a pair come from one 16-byte load
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        ulonglong2 x[8], y[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const ulonglong2 *>(A + t.row(i) * ld + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = *reinterpret_cast<const ulonglong2 *>(B + (t.cg + 16 * j) * ld + k);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < (i < 4 ? 2 : 4); ++j) {  // rows 0..31 x columns 32..63 are masked
                fma2(acc[i][j], x[i].x, y[j].x);
                fma2(acc[i][j], x[i].y, y[j].y);
            }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int rr = t.row(i), c = t.cg + 16 * j;
            Wt[rr * kLdW + c] = c <= rr ? lo(acc[i][j]) + hi(acc[i][j]) + (r ? r[rr] : 0.f) : 0.f;
        }
}

enum CarryUse { kPlain, kTransposed, kSymmetric };  // B = R, R^T, R + R^T

// acc += A B, A row-major in shared memory (rows of N + 4), B (K x width) a carry in global memory:
// R rows of `ldr` floats.  Slices of SL rows of B pass through `stage` (2 x SL x N floats), the next
// one loaded into registers while this one is multiplied.  K and width are multiples of 16.  Ends
// with every thread past its last read of `stage`.
template <int N, CarryUse U>
__device__ __forceinline__ void nn_carry(Acc<N> &acc, const Tile<N> &t, const float *A, const float *__restrict__ R,
                                         int ldr, int K, int width, float *stage) {
    constexpr int kSlice = Tile<N>::SL, PT = kSlice * N / kCT;  // floats of a slice per thread: 16, 4, 4
    float buf[PT];
    const int tid = threadIdx.x;
    const int tc = tid % N, tk = (tid / N) * PT;  // transposed use: column tc, rows tk .. tk + PT - 1
    auto fetch = [&](int s) {
        if constexpr (U == kPlain) {
#pragma unroll
            for (int i = 0; i < PT / 4; ++i) {
                const int e = tid + i * kCT, k = s * kSlice + e / (N / 4), c = (e % (N / 4)) * 4;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < width) v = *reinterpret_cast<const float4 *>(R + (long long)k * ldr + c);
                buf[4 * i] = v.x; buf[4 * i + 1] = v.y; buf[4 * i + 2] = v.z; buf[4 * i + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < PT / 4; ++i) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (tc < width) v = *reinterpret_cast<const float4 *>(R + (long long)tc * ldr + s * kSlice + tk + 4 * i);
                buf[4 * i] = v.x; buf[4 * i + 1] = v.y; buf[4 * i + 2] = v.z; buf[4 * i + 3] = v.w;
            }
            if (U == kSymmetric && tc < width) {
#pragma unroll
                for (int i = 0; i < PT; ++i) buf[i] += R[(long long)(s * kSlice + tk + i) * ldr + tc];
            }
        }
    };
    auto put = [&](float *b) {
        if constexpr (U == kPlain) {
#pragma unroll
            for (int i = 0; i < PT / 4; ++i)
                *reinterpret_cast<float4 *>(b + (tid + i * kCT) * 4) =
                    make_float4(buf[4 * i], buf[4 * i + 1], buf[4 * i + 2], buf[4 * i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < PT; ++i) b[(tk + i) * N + tc] = buf[i];
        }
    };
    const int ns = K / kSlice;
    fetch(0);
    put(stage);
    __syncthreads();
    for (int s = 0; s < ns; ++s) {
        if (s + 1 < ns) fetch(s + 1);
        nn_range<N, 0>(acc, t, A + s * kSlice, N + 4, stage + (s & 1) * kSlice * N, N, 0, kSlice);
        if (s + 1 < ns) put(stage + ((s + 1) & 1) * kSlice * N);
        __syncthreads();
    }
}

// returns 0 if all that this thread stored is finite, else NaN
template <int N>
__device__ __forceinline__ float acc_to_smem(const Acc<N> &acc, const Tile<N> &t, float *dst) {
    float seen = 0.f;
#pragma unroll
    for (int i = 0; i < Tile<N>::RM; ++i)
#pragma unroll
        for (int j = 0; j < Tile<N>::CM; j += 4) {
            const float4 v = make_float4(acc.get(i, j), acc.get(i, j + 1), acc.get(i, j + 2), acc.get(i, j + 3));
            seen = fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, fmaf(v.w, 0.f, seen))));
            *reinterpret_cast<float4 *>(dst + t.row(i) * (N + 4) + t.col(j)) = v;
        }
    return seen;
}

// rows r0 + r < rows, columns < width of the outputs to global memory, rows of `width` elements
template <int N, typename T>
__device__ __forceinline__ void acc_to_global(const Acc<N> &acc, const Tile<N> &t, T *dst, int rows, int width,
                                              int r0 = 0) {
#pragma unroll
    for (int i = 0; i < Tile<N>::RM; ++i) {
        const int r = r0 + t.row(i);
        if (r < rows)
#pragma unroll
            for (int j = 0; j < Tile<N>::CM; j += 4)
                if (t.col(j) < width) {
                    const float x[4] = {acc.get(i, j), acc.get(i, j + 1), acc.get(i, j + 2), acc.get(i, j + 3)};
                    Vec<T>::store4(dst + (long long)r * width + t.col(j), x);
                }
    }
}

// rec (M x width) = A^T B over the chunk's tokens: A, B row-major in shared memory, M real columns of A
template <int N>
__device__ __forceinline__ void atb_to_global(const Tile<N> &t, float *rec, const float *A, const float *B, int M,
                                              int width) {
    for (int r0 = 0; r0 < M; r0 += kC) {
        Acc<N> acc;
        acc.zero();
        if (r0 + 4 * t.rg < M) tn<N>(acc, t, A + r0, N + 4, B);  // rows beyond M would read beyond a row of A
        acc_to_global<N, float>(acc, t, rec, M, width, r0);
    }
}

// out[c] = sum_r w_r A(r, c) over the chunk's rows, c < width (w null: 1)
template <int N>
__device__ __forceinline__ void col_sums(float *out, const float *A, const float *w, int width) {
    for (int c = threadIdx.x; c < width; c += kCT) {
        float s = 0.f;
#pragma unroll 8
        for (int r = 0; r < kC; ++r) s = fmaf(w ? w[r] : 1.f, A[r * (N + 4) + c], s);
        out[c] = s;
    }
}

// x_r = sum_c A(r, c) v_c, c < width (v null: 1; kLower: c <= r), for the row r = threadIdx.x / 2 of a 64-row
// operand with rows of ld floats; both threads of a row return the sum
template <bool kLower = false>
__device__ __forceinline__ float row_dot(const float *A, int ld, const float *v, int width) {
    const int r = threadIdx.x >> 1, h = threadIdx.x & 1;
    float s = 0.f;
    for (int c = 4 * h; c < width; c += 8) {
        const float4 x = *reinterpret_cast<const float4 *>(A + r * ld + c);
        float4 y = v ? *reinterpret_cast<const float4 *>(v + c) : make_float4(1.f, 1.f, 1.f, 1.f);
        if (kLower) {  // the v of later tokens may not be finite
            if (c > r) y.x = 0.f;
            if (c + 1 > r) y.y = 0.f;
            if (c + 2 > r) y.z = 0.f;
            if (c + 3 > r) y.w = 0.f;
        }
        s = fmaf(x.x, y.x, s);
        s = fmaf(x.y, y.y, s);
        s = fmaf(x.z, y.z, s);
        s = fmaf(x.w, y.w, s);
    }
    return s + __shfl_xor_sync(0xffffffffu, s, 1);
}

template <int N>
constexpr int stage_floats() { return 2 * Tile<N>::SL * N; }
template <int N>
constexpr int tile_floats() { return kC * (N + 4); }
// blocks an SM that the chunk kernels are compiled for: as many as their shared memory admits at N = 64 and
// 128; one block more at N = 64 takes 512 blocks (B2 H16 n1000) from two rounds to one, 46 -> 41 us
template <int N>
constexpr int blocks_per_sm() { return N == 128 ? 2 : 4; }

inline dim3 chunk_grid(int nch, int BH, int z = 1) { return dim3((unsigned)nch * (unsigned)BH, 1, z); }
__device__ __forceinline__ void chunk_of(int nch, int &c, int &hd) {
    hd = blockIdx.x / (unsigned)nch;
    c = blockIdx.x % (unsigned)nch;
}

// ---------------------------------------------------------------------------
// per-chunk records and their prefix sums.  Records of a head: nch of them, then one that holds the
// initial value on entry (if there is one) and the total on exit.
// ---------------------------------------------------------------------------
struct Records {
    float *base;
    int len;  // floats of a record, a multiple of 4
    int nch;
    __device__ __forceinline__ float *at(int hd, int c) const { return base + ((long long)hd * (nch + 1) + c) * len; }
};

struct ScanJob {
    Records r;
    const float *init;  // initial value of head hd at init + hd * init_stride, or null: zero
    long long init_stride;
    float *total;       // total of head hd to total + hd * total_stride, or null
    long long total_stride;
    int reverse;        // suffix sums: record c becomes the sum of the records after it
};
struct ScanJobs {
    ScanJob j[2];
};

// exclusive prefix (suffix) sums in place, one float4 a thread; sixteen records' loads in flight, as memory
// latency over the chunks in turn is what bounds it (eight in flight: B4 H8 n2000 d128 fp32 491 us, sixteen 479)
__global__ void __launch_bounds__(64) chunk_scan_kernel(const __grid_constant__ ScanJobs jobs) {
    chain_begin();
    const ScanJob &J = jobs.j[blockIdx.z];
    const int e = (blockIdx.y * 64 + threadIdx.x) * 4, hd = blockIdx.x, nch = J.r.nch;
    if (e >= J.r.len) return;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (J.init) acc = *reinterpret_cast<const float4 *>(J.init + hd * J.init_stride + e);
    const long long step = J.reverse ? -(long long)J.r.len : (long long)J.r.len;
    float *p = J.r.at(hd, J.reverse ? nch - 1 : 0) + e;
    constexpr int U = 16;
    for (int c = 0; c < nch; c += U) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (c + u < nch) v[u] = *reinterpret_cast<const float4 *>(p + u * step);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (c + u < nch) {
                *reinterpret_cast<float4 *>(p + u * step) = acc;
                acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w;
            }
        p += U * step;
    }
    if (J.total) *reinterpret_cast<float4 *>(J.total + hd * J.total_stride + e) = acc;
}

inline cudaError_t launch_scan(const ScanJobs &jobs, int njobs, int BH, cudaStream_t s, bool follows = true) {
    int len = 0;
    for (int i = 0; i < njobs; ++i) len = jobs.j[i].r.len > len ? jobs.j[i].r.len : len;
    return chain_launch(follows, chunk_scan_kernel, dim3(BH, (len / 4 + 63) / 64, njobs), 64, 0, s, jobs);
}

// per chunk, the sums over its tokens A^T B (d x width) and, after it in the record, A^T 1 (d) where
// `sums` is set; blockIdx.z selects the job
template <typename T>
struct SumJob {
    const T *A, *B;
    Records r;
    int d, width, sums;
};
template <typename T>
struct SumJobs {
    SumJob<T> j[2];
};
template <int N, typename T>
__global__ void __launch_bounds__(kCT) chunk_sums_kernel(const __grid_constant__ SumJobs<T> jobs, int n) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    const SumJob<T> &J = jobs.j[blockIdx.z];
    int c, hd;
    chunk_of(J.r.nch, c, hd);
    const int t0 = c * kC, len = min(kC, n - t0);
    float *As = sm, *Bs = sm + tile_floats<N>();
    load_tile<N>(As, J.A + ((long long)hd * n + t0) * J.d, len, J.d);
    if (J.B != J.A) load_tile<N>(Bs, J.B + ((long long)hd * n + t0) * J.width, len, J.width);
    else Bs = As;
    __syncthreads();
    const Tile<N> t;
    float *rec = J.r.at(hd, c);
    atb_to_global<N>(t, rec, As, Bs, J.d, J.width);
    if (J.sums) col_sums<N>(rec + J.d * J.width, As, nullptr, J.d);
}
template <int N, typename T>
cudaError_t launch_sums(bool follows, const SumJobs<T> &jobs, int njobs, int BH, int n, cudaStream_t s) {
    const int smem = 2 * tile_floats<N>() * (int)sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(chunk_sums_kernel<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e) return e;
    return chain_launch(follows, chunk_sums_kernel<N, T>, chunk_grid((n + kC - 1) / kC, BH, njobs), kCT, smem, s, jobs, n);
}

// ---------------------------------------------------------------------------
// outputs from what the chunk itself gives and the carry [M | u] before it: num = num_loc + Q M_p,
// den = den_loc + Q u_p
// ---------------------------------------------------------------------------
struct OutParams {
    Records carry;
    const float *num, *den;  // [BH][n][dv], [BH][n]
    int n, d, dv, normalized;
    float eps;
    int has_in;  // the first chunk has a carry
};
template <int N, typename T>
__global__ void __launch_bounds__(kCT)
    chunk_out_kernel(const T *__restrict__ q, T *__restrict__ out, const __grid_constant__ OutParams P) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    float *b0 = sm, *stage = b0 + tile_floats<N>(), *dens = stage + stage_floats<N>();
    int c, hd;
    chunk_of(P.carry.nch, c, hd);
    const int d = P.d, dv = P.dv, t0 = c * kC, len = min(kC, P.n - t0);
    const long long tok = (long long)hd * P.n + t0;
    const bool carry = c > 0 || P.has_in;
    const float *Mp = P.carry.at(hd, c);
    const Tile<N> t;
    Acc<N> acc;
    acc.zero();
    float den = 0.f;
    if (carry) {
        load_tile<N>(b0, q + tok * d, len, d);
        __syncthreads();
        if (P.normalized) den = row_dot(b0, N + 4, Mp + d * dv, d);
        nn_carry<N, kPlain>(acc, t, b0, Mp, dv, d, dv, stage);
    }
    if (P.normalized) {
        const int r = threadIdx.x >> 1;
        if ((threadIdx.x & 1) == 0) dens[r] = (r < len ? P.den[tok + r] : 0.f) + den + P.eps;
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < Tile<N>::RM; ++i) {
        const int r = t.row(i);
        if (r >= len) continue;
#pragma unroll
        for (int j = 0; j < Tile<N>::CM; j += 4) {
            if (t.col(j) >= dv) continue;
            const float4 x = *reinterpret_cast<const float4 *>(P.num + (tok + r) * dv + t.col(j));
            float y[4] = {acc.get(i, j) + x.x, acc.get(i, j + 1) + x.y, acc.get(i, j + 2) + x.z, acc.get(i, j + 3) + x.w};
            if (P.normalized) {
                const float den_r = dens[r];
#pragma unroll
                for (int u = 0; u < 4; ++u) y[u] /= den_r;
            }
            Vec<T>::store4(out + (tok + r) * dv + t.col(j), y);
        }
    }
}

template <int N, typename T>
cudaError_t launch_out(const T *q, T *out, const OutParams &P, int BH, cudaStream_t s) {
    const int smem = (tile_floats<N>() + stage_floats<N>() + kC) * (int)sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(chunk_out_kernel<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e) return e;
    return chain_launch(true, chunk_out_kernel<N, T>, chunk_grid((P.n + kC - 1) / kC, BH), kCT, smem, s, q, out, P);
}

// the padded head size that serves d and dv
template <typename F>
cudaError_t with_padded_size(int d, int dv, F f) {
    const int m = d > dv ? d : dv;
    if (m <= 32) return f(std::integral_constant<int, 32>());
    if (m <= 64) return f(std::integral_constant<int, 64>());
    return f(std::integral_constant<int, 128>());
}

}  // namespace
}  // namespace hla
