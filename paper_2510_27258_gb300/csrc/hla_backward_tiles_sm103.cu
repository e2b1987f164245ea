// Gradients of masked second-order HLA on the tensor cores for bf16 tokens, d and dv in {64, 128},
// plain or normalised output (hla2_backward; the plain output at d = dv = 64 has its own kernel in
// hla_backward_sm103.cu).  The algebra is that of hla_backward.cu, in tiles of 128 tokens:
//   W = L . (Q K^T), X = W K + Q S_p, T = L . (Q X^T), num = T V + Q D_p, den = T 1 + Q e_p,
//   P = L . (G' V^T + u 1^T), Y = P^T Q + V Gam_s + 1 h_s^T, dV = T^T G' + X Gam_s^T,
//   B = L . (Y K^T), dQ = P X + G' D_p^T + u e_p^T + Y S_p + B K, dK = K Lam_s + W^T Y + B^T Q,
// and every carry a plain sum of what the tiles add (S: K^T K, D: X^T V, Gam^T: Q^T G',
// Lam: Q^T Y + Y^T Q, e: X^T 1, h: Q^T u).
//
// Structure.  With 14 operand tiles of 32 KB (hi and lo parts) a persistent sweep like the d = 64
// kernel's does not fit an SM at head size 128.  So each step is a launch of its own with a block per
// (tile, head), the sums between them run element by element over the tiles of a head, and nothing waits
// on another block.  A block has three 32 KB operand slots, 256 TMEM columns (a masked tile
// and a result) and 256 threads, so two blocks share an SM: one's copies and products run under the
// other's epilogue, which is why no block pipelines within itself (thread 0 issues, everyone waits).
//
// Precision: as in the d = 64 kernel, every intermediate is a bf16 pair hi + lo (2^-17 together), a product of
// two pairs takes hi hi + hi lo + lo hi, accumulation is fp32, the sums between tiles are fp32.
// Masked tiles are formed in TMEM, packed over themselves as hi/lo and read there as the A
// operand; a transposed use is formed as its own product with the mask turned over.
//
// Layouts.  Operand images: 128 x 128 bf16, the 128-byte-swizzled shared-memory image, hi (32 KB) then
// lo, moved by 1-D bulk copies.  Records (fp32 128 x 128, a tile's addition to a carry, or num):
// float4 (r, c..c+3) at index ((r / 32 * 16 + c / 8) * 2 + c / 4 % 2) * 32 + r % 32, so that a warp's
// access is 512 contiguous bytes.  Head size 64 runs zero-padded (TMA fill).
//
// Measured: B2 H16 n4096 d128 normalised 0.486 ms, against 2.04 ms for the CUDA-core kernels (and 37 ms
// for the kernels those replaced); ncu, us: 19 for K^T K, 73 X, 62 G', 64 Y, 165 the gradients, 19 to 24 for
// each of the four sums.  What bounds it is its own traffic: those launches read 1691 MB and write 445 MB, 0.31 ms
// at the measured copy rate, and the gradients run at 80 % of it (they load 26 operands of 32 KB a tile, 17 of them
// distinct).  About 60 products of 128^3 a tile are 0.15 ms at the measured bf16 peak.
//
// Accuracy, against 64-bit results, of the bf16 gradients over B1 H4 n100 to B1 H4 n16384 and B8 H16 n512: 1.66e-3 of
// the norm, as with the fp32 kernels to 2e-5 of that figure (the results' own rounding); the worst row of 65536, where
// the terms of a gradient cancel to a thousandth, 7.4e-3 of its norm instead of 2.6e-3.
#include <algorithm>
#include <cstdlib>

#include "chain_launch.cuh"
#include "hla_internal.h"
#include "sm103_prims.cuh"

namespace hla {
namespace {

using namespace sm103;

constexpr int kTile = 128, kF = 128;
constexpr int kThreads = 256;
constexpr uint32_t kImage = kTileBytes;      // hi or lo
constexpr uint32_t kPair = 2 * kTileBytes;   // hi and lo
constexpr int kRec = kF * kF;                // floats of a record
constexpr unsigned long long kWaitNs = 2000000000ull;

struct Misc {
    uint64_t bar[3];  // copies; products (two commits may be outstanding)
    uint32_t tmem_base;
    int abort_flag;
    float us[kTile], vec[kF], red[kThreads];
    int stains, first[kF], last[kF];  // of each column, the first and last row that drop() took a value from
};
constexpr uint32_t kSmemBytes = 3 * kTileBytes + sizeof(Misc);
enum { bLd = 0, bMma = 1, bMma2 = 2 };

struct Maps {
    CUtensorMap q, k, v, g, dq, dk, dv;
};
struct TParams {
    float *rec, *rec1;                                  // records: the running step's; plain: Gam's, normalised: num
    uint8_t *iS, *iD, *iGam, *iLam, *iX, *iY, *iG;      // image pairs per (head, tile)
    float *e, *h;                                       // [BH][M][128]
    float *den;                                         // [BH][n]: T 1, then u
    int n, M, d, dv, normalized;
    float eps;
    WsHeader *err;
};

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 ::"l"(reinterpret_cast<uint64_t>(dst)), "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}

// ------------------------------- products (thread 0) -------------------------------
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t kLboK = 1u << 16, kLboMN = (kBlockBytes >> 4) << 16;
__device__ __forceinline__ uint64_t dsc(uint32_t lo) { return (static_cast<uint64_t>(kDescHi) << 32) | lo; }
enum Major { K = 0, MN = 1 };

// D (+)= A B, 128 x 128 x 128, operands in shared-memory slots a and b (address >> 4)
template <Major A, Major B>
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t b, bool acc) {
    constexpr uint32_t id = idesc_bf16(128, 128, A, B);
    a += A ? kLboMN : kLboK;
    b += B ? kLboMN : kLboK;
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
        const uint32_t ka = A ? kk * 128u : (kk >> 2) * (kBlockBytes >> 4) + (kk & 3) * 2u;
        const uint32_t kb = B ? kk * 128u : (kk >> 2) * (kBlockBytes >> 4) + (kk & 3) * 2u;
        umma_bf16(d, dsc(a + ka), dsc(b + kb), id, kk > 0 || acc ? 1u : 0u);
    }
}
// the same with A a packed masked tile in TMEM (hi at a, lo at a + 16), B a token tile (K along its rows)
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint32_t b, bool acc) {
    constexpr uint32_t id = idesc_bf16(128, 128, 0, 1);
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
        umma_bf16_ts(d, a + 32u * (kk >> 1) + 8u * (kk & 1), dsc(b + kLboMN + kk * 128u), id, kk > 0 || acc ? 1u : 0u);
}

__device__ __forceinline__ void split2(float x0, float x1, uint32_t &h, uint32_t &l) {
    h = pack_bf16x2(x0, x1);
    l = pack_bf16x2(x0 - __uint_as_float(h << 16), x1 - __uint_as_float(h & 0xFFFF0000u));
}
__device__ __forceinline__ void unpack2(uint32_t v, float &x0, float &x1) {
    x0 = __uint_as_float(v << 16);
    x1 = __uint_as_float(v & 0xFFFF0000u);
}
__device__ __forceinline__ int rec_index(int r, int c) {  // float4 index of (r, c .. c + 3)
    return (((r >> 5) * 16 + (c >> 3)) * 2 + ((c >> 2) & 1)) * 32 + (r & 31);
}

// takes the values that are not finite out of a slot and notes the first and last row of each column's
__device__ __noinline__ void drop_values(uint8_t *slot, Misc *ms) {
    for (int i = threadIdx.x; i < (int)(kTileBytes / 2); i += kThreads) {
        __nv_bfloat16 *p = reinterpret_cast<__nv_bfloat16 *>(slot) + i;
        const float x = __bfloat162float(*p);
        if (x - x == 0.f) continue;
        const int row = i / 64 % kTile;  // element i of a slot: the inverse of tile_off()
        const int col = i / (int)(kBlockBytes / 2) * 64 + ((i / 8 % 8) ^ (row & 7)) * 8 + i % 8;
        atomicMin(&ms->first[col], row);
        atomicMax(&ms->last[col], row);
        *p = __float2bfloat16_rn(0.f);
    }
    if (threadIdx.x == 0) ms->stains = 1;
}

// 64 columns of row r of a region from column c0 (at t): NaN where `how` (Ctx::Stain) says
__device__ __noinline__ void stain_region(uint32_t t, int r, int c0, int how, const Misc *ms) {
    for (int i = 0; i < 64; i += 32) {
        uint32_t a[32];
        __syncwarp();
        tmem_ld32(t + i, a);
        tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            const int f = ms->first[c0 + i + u], l = ms->last[c0 + i + u];
            if (how == 1 ? r >= f : how == 2 ? r <= l : l >= 0) a[u] = 0x7fffffffu;
        }
        tmem_st32(t + i, a);
        tmem_st_wait();
    }
}

// ------------------------------- a block's state -------------------------------
struct Ctx {
    uint8_t *sm;
    Misc *ms;
    const TParams &p;
    int tid, lane, r, half, tile, head, len;
    size_t at;  // head * M + tile
    bool before, after;
    uint32_t tb, s4, lane_base, ld_par = 0, m_par = 0, m2_par = 0;

    __device__ Ctx(uint8_t *smem, const TParams &p_) : sm(smem), ms(reinterpret_cast<Misc *>(smem + 3 * kTileBytes)), p(p_) {
        tid = threadIdx.x;
        lane = tid & 31;
        const int warp = tid >> 5;
        r = 32 * (warp & 3) + lane;  // TMEM lane of this thread
        half = warp >> 2;            // its columns: 64 half .. + 63
        lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        tile = blockIdx.x % (unsigned)p.M;  // the grid's other dimensions end at 65535, which heads may pass
        head = blockIdx.x / (unsigned)p.M;
        at = (size_t)head * p.M + tile;
        len = min(kTile, p.n - tile * kTile);
        before = tile > 0;
        after = tile + 1 < p.M;
        s4 = smem_u32(smem) >> 4;
        if (tid == 0) {
            for (int b = 0; b < 3; ++b) mbar_init(&ms->bar[b], 1);
            ms->stains = 0;
            ms->abort_flag = (smem_u32(smem) & 1023u) != 0;  // the swizzled layout needs 1 KiB alignment
            if (ms->abort_flag) fail(0);
            fence_mbar_init();
        }
        if (tid < kF) {
            ms->first[tid] = kTile;
            ms->last[tid] = -1;
        }
        __syncwarp();
        if (warp == 0) {
            tmem_alloc(&ms->tmem_base, 256);
            tmem_relinquish();
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        tb = ms->tmem_base;
        chain_begin();  // nothing before this reads or writes global memory but a failed alignment check
    }
    __device__ void fail(unsigned where) {
        if (atomicCAS(&p.err->error, 0u, (unsigned)kDevTimeout) == 0u) {
            p.err->where = 600 + where;
            p.err->detail = (unsigned)at;
        }
        ms->abort_flag = 1;
    }
    __device__ bool aborted() const { return ms->abort_flag != 0; }
    __device__ uint8_t *slot(int s) { return sm + s * kTileBytes; }
    __device__ uint32_t sl(int s) const { return s4 + (uint32_t)s * (kTileBytes >> 4); }
    __device__ uint32_t RA() const { return tb; }        // the masked tile
    __device__ uint32_t RB() const { return tb + 128; }  // the result

    // thread 0: announce `n` tiles, then copy each
    __device__ void expect(int n) { mbar_arrive_expect_tx(&ms->bar[bLd], (uint32_t)n * kTileBytes); }
    __device__ void load_tokens(int s, const CUtensorMap *m) {
        tma_load_3d(slot(s), m, &ms->bar[bLd], 0, tile * kTile, head);
        tma_load_3d(slot(s) + kBlockBytes, m, &ms->bar[bLd], 64, tile * kTile, head);
    }
    __device__ void load_image(int s, const uint8_t *base, int lo) {
        bulk_load(slot(s), base + at * kPair + lo * kImage, kImage, &ms->bar[bLd]);
    }
    __device__ bool wait(int b, uint32_t &par) {
        if (!ms->abort_flag && !mbar_wait(&ms->bar[b], par, kWaitNs)) fail(1 + b);
        par ^= 1u;
        __syncthreads();
        tc_fence_after();
        return !ms->abort_flag;
    }
    __device__ bool wait_ld() { return wait(bLd, ld_par); }
    __device__ bool wait_mma() { return wait(bMma, m_par); }
    __device__ bool wait_mma2() { return wait(bMma2, m2_par); }
    __device__ void commit() { umma_commit(&ms->bar[bMma]); }
    __device__ void commit2() { umma_commit(&ms->bar[bMma2]); }
    // what the threads wrote to shared memory and TMEM is seen by the products issued after this
    __device__ void publish() {
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }

    // A masked tile's zeros times a token that is not finite would make NaN of rows that do not depend on the
    // token.  So before a product of a masked tile and the rows of a slot, every value of the slot that is not finite
    // is taken out and noted, and the result is NaN where the triangle holds a noted value (stain()).
    // nonfinite(): whether the slot has any, the same in every thread (a barrier; a hi slot answers for its lo).
    __device__ bool nonfinite(int s) {
        __nv_bfloat162 seen = __floats2bfloat162_rn(0.f, 0.f);
        const __nv_bfloat162 zero = seen;
#pragma unroll
        for (int i = 0; i < (int)(kTileBytes / 16) / kThreads; ++i) {
            const uint4 v = reinterpret_cast<const uint4 *>(slot(s))[tid + i * kThreads];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) seen = __hfma2(*reinterpret_cast<const __nv_bfloat162 *>(&w[u]), zero, seen);
        }
        return __syncthreads_or(!(__low2float(seen) == 0.f && __high2float(seen) == 0.f)) != 0;
    }
    __device__ void drop(int s) {
        drop_values(slot(s), ms);
        publish();
    }
    enum Stain { kNone, kLower, kUpperT, kColumn };  // rows from the first noted one, up to the last, all
    // a result region, where values were dropped: NaN in its place in TMEM
    __device__ void stain(Stain how, uint32_t region) {
        if (how != kNone && ms->stains) stain_region(region + lane_base + 64 * half, r, 64 * half, how, ms);
    }

    // The masked tile of region RA (kUpper: column >= row, else column <= row), with us[column] or
    // us[row] added inside the mask where `add`, packed over itself: hi in the first 16 of each 32
    // columns, lo in the other 16.  Returns the sum of this thread's masked values.
    template <bool kUpper>
    __device__ float mask_pack(bool add) {
        float sum = 0.f;
        __syncwarp();  // thread 0 may come from issuing
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c0 = 64 * half + 32 * i, qd = r >> 5, cq = c0 >> 5;  // blocks of 32 x 32, warp-uniform
            const uint32_t t = tb + lane_base + c0;
            uint32_t hp[16], lp[16];
            if (kUpper ? cq < qd : cq > qd) {
#pragma unroll
                for (int u = 0; u < 16; ++u) hp[u] = lp[u] = 0u;
            } else {
                uint32_t a[32];
                tmem_ld32(t, a);
                tmem_ld_wait();
                const float ur = add && !kUpper ? ms->us[r] : 0.f;
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const int c = c0 + 2 * u;
                    float x0 = __uint_as_float(a[2 * u]) + ur, x1 = __uint_as_float(a[2 * u + 1]) + ur;
                    if (kUpper && add) {
                        x0 += ms->us[c];
                        x1 += ms->us[c + 1];
                    }
                    if (cq == qd) {
                        if (kUpper ? c < r : c > r) x0 = 0.f;
                        if (kUpper ? c + 1 < r : c + 1 > r) x1 = 0.f;
                    }
                    sum += x0 + x1;
                    split2(x0, x1, hp[u], lp[u]);
                }
            }
            tmem_st16(t, hp);
            tmem_st16(t + 16, lp);
        }
        tmem_st_wait();
        return sum;
    }

    // 32 columns of this thread's row of a region, column c0 .. c0 + 31
    __device__ void read32(uint32_t region, int c0, float (&x)[32]) {
        uint32_t a[32];
        __syncwarp();  // thread 0 may come from issuing
        tmem_ld32(region + lane_base + c0, a);
        tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < 32; ++u) x[u] = __uint_as_float(a[u]);
    }
    // hi and lo of 32 values into row r of two slots
    __device__ void split_store(int hi, int lo, int c0, const float (&x)[32]) {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) split2(x[8 * g + 2 * u], x[8 * g + 2 * u + 1], h[u], l[u]);
            const uint32_t off = tile_off(r, c0 + 8 * g);
            *reinterpret_cast<uint4 *>(slot(hi) + off) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4 *>(slot(lo) + off) = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
    // a region -> hi, lo slots, `vec` added to every row where `add`
    __device__ void region_to_slots(uint32_t region, int hi, int lo, bool add, Stain how) {
        stain(how, region);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c0 = 64 * half + 32 * i;
            float x[32];
            read32(region, c0, x);
            if (add) {
#pragma unroll
                for (int u = 0; u < 32; ++u) x[u] += ms->vec[c0 + u];
            }
            split_store(hi, lo, c0, x);
        }
    }
    __device__ void region_to_record(uint32_t region, float *rec, Stain how = kNone) {
        stain(how, region);
        float4 *o = reinterpret_cast<float4 *>(rec + at * kRec);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c0 = 64 * half + 32 * i;
            float x[32];
            read32(region, c0, x);
#pragma unroll
            for (int u = 0; u < 32; u += 4) o[rec_index(r, c0 + u)] = make_float4(x[u], x[u + 1], x[u + 2], x[u + 3]);
        }
    }
    // thread 0, after publish(): a hi/lo pair of slots to its images
    __device__ void store_images(uint8_t *base, int hi, int lo) {
        bulk_store(base + at * kPair, slot(hi), kImage);
        bulk_store(base + at * kPair + kImage, slot(lo), kImage);
        tma_store_commit();
    }
    // sum over the tile's rows of w_t (x_t,f), f = tid % 128, x the bf16 of slot a plus (b >= 0) of slot b, w
    // in shared memory or null: 1; on return the first 128 threads hold their column's sum
    __device__ float column_sums(int a, int b, const float *w) {
        const int f = tid & 127, r0 = (tid >> 7) * 64;
        float s = 0.f;
#pragma unroll 8
        for (int t = r0; t < r0 + 64; ++t) {
            const uint32_t off = tile_off(t, f & ~7) + (f & 7) * 2;
            float x = __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(slot(a) + off));
            if (b >= 0) x += __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(slot(b) + off));
            s = fmaf(w ? w[t] : 1.f, x, s);
        }
        ms->red[tid] = s;
        __syncthreads();
        s = tid < 128 ? ms->red[tid] + ms->red[tid + 128] : 0.f;
        __syncthreads();
        return s;
    }
    // the sum of a value over the two threads of a row
    __device__ float row_total(float x) {
        ms->red[half * 128 + r] = x;
        __syncthreads();
        x = ms->red[r] + ms->red[128 + r];
        __syncthreads();
        return x;
    }
    // a region (plus row_add[r] vec[c] where `add`) as bf16 through slot s to the tile's rows of an output
    __device__ void region_to_output(uint32_t region, int s, const CUtensorMap *m, int width, bool add, Stain how) {
        stain(how, region);
        const float ur = add ? ms->us[r] : 0.f;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c0 = 64 * half + 32 * i;
            float x[32];
            read32(region, c0, x);
            if (add) {
#pragma unroll
                for (int u = 0; u < 32; ++u) x[u] = fmaf(ur, ms->vec[c0 + u], x[u]);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g)
                *reinterpret_cast<uint4 *>(slot(s) + tile_off(r, c0 + 8 * g)) =
                    make_uint4(pack_bf16x2(x[8 * g], x[8 * g + 1]), pack_bf16x2(x[8 * g + 2], x[8 * g + 3]),
                               pack_bf16x2(x[8 * g + 4], x[8 * g + 5]), pack_bf16x2(x[8 * g + 6], x[8 * g + 7]));
        }
        publish();
        if (tid == 0) {
            tma_store_3d(m, slot(s), 0, tile * kTile, head);  // rows beyond n are clipped
            if (width > 64) tma_store_3d(m, slot(s) + kBlockBytes, 64, tile * kTile, head);
            tma_store_commit();
        }
    }
    // every block ends here: bulk stores complete, products and copies finished, TMEM freed
    __device__ void finish() {
        if (tid == 0) {
            tma_store_wait_all();
            if (ms->abort_flag) {  // whatever is in flight ends (bounded) before the memory is given up
                commit2();
                mbar_wait(&ms->bar[bMma2], m2_par, kWaitNs);
                mbar_wait(&ms->bar[bLd], ld_par, kWaitNs);
            }
        }
        tc_fence_before();
        __syncthreads();
        __syncwarp();
        if (tid < 32) {
            tc_fence_after();
            tmem_dealloc(tb, 256);
        }
    }
};

// ---------------------------------------------------------------------------
// additions of a tile to S (K^T K) and, plain output, to Gam^T (Q^T G): blockIdx.z
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads, 2) bt_sums_kernel(const __grid_constant__ Maps m, const __grid_constant__ TParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    Ctx c(smem, p);
    const bool gam = blockIdx.z == 1;
    if (!c.aborted() && (gam ? c.before : c.after)) {  // S before the first tile, Gam after the last are zero
        if (c.tid == 0) {
            c.expect(gam ? 2 : 1);
            c.load_tokens(0, gam ? &m.q : &m.k);
            if (gam) c.load_tokens(1, &m.g);
        }
        if (c.wait_ld()) {
            if (c.tid == 0) {
                mma<MN, MN>(c.RB(), c.sl(0), c.sl(gam ? 1 : 0), false);
                c.commit();
            }
            if (c.wait_mma()) c.region_to_record(c.RB(), gam ? p.rec1 : p.rec);
        }
    }
    c.finish();
}

// ---------------------------------------------------------------------------
// X; additions to D and e; normalised: T V and T 1
// ---------------------------------------------------------------------------
__device__ void x_steps(Ctx &c, const Maps &m) {
    const TParams &p = c.p;
    const bool norm = p.normalized;
    if (c.tid == 0) {
        c.expect(c.before ? 3 : 2);
        c.load_tokens(0, &m.q);
        c.load_tokens(1, &m.k);
        if (c.before) c.load_image(2, p.iS, 0);
    }
    if (!c.wait_ld()) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(0), c.sl(1), false);                    // Q K^T
        if (c.before) mma<K, K>(c.RB(), c.sl(0), c.sl(2), false);      // Q S_p (symmetric)
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.before && c.tid == 0) {
        c.expect(1);
        c.load_image(2, p.iS, 1);
    }
    if (c.nonfinite(1)) c.drop(1);
    c.mask_pack<false>(false);  // W
    c.publish();
    if (c.before && !c.wait_ld()) return;
    if (c.tid == 0) {
        if (c.before) mma<K, K>(c.RB(), c.sl(0), c.sl(2), true);
        mma_ts(c.RB(), c.RA(), c.sl(1), c.before);  // W K
        mma_ts(c.RB(), c.RA() + 16, c.sl(1), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    c.region_to_slots(c.RB(), 1, 2, false, Ctx::kLower);  // X over K and S
    c.publish();
    if (c.tid == 0) c.store_images(p.iX, 1, 2);
    if (norm) {
        if (c.tid == 0) {
            mma<K, K>(c.RA(), c.sl(0), c.sl(1), false);  // Q X^T
            mma<K, K>(c.RA(), c.sl(0), c.sl(2), true);
            c.commit();
        }
        if (!c.wait_mma()) return;
    } else if (!c.after) {
        return;
    }
    if (c.tid == 0) {
        c.expect(1);
        c.load_tokens(0, &m.v);
    }
    if (norm) {
        const float den = c.row_total(c.mask_pack<false>(false));  // T, T 1
        if (c.half == 0 && c.r < c.len) p.den[(size_t)c.head * p.n + c.tile * kTile + c.r] = den;
        const float e = c.column_sums(1, 2, nullptr);
        if (c.tid < kF) p.e[c.at * kF + c.tid] = e;
        c.publish();
    }
    if (!c.wait_ld()) return;
    if (norm && c.nonfinite(0)) c.drop(0);
    if (c.tid == 0) {
        if (norm) {
            mma_ts(c.RB(), c.RA(), c.sl(0), false);  // T V
            mma_ts(c.RB(), c.RA() + 16, c.sl(0), true);
            c.commit();
        }
        if (c.after) {  // X^T V over T, whose products are issued before it
            mma<MN, MN>(c.RA(), c.sl(1), c.sl(0), false);
            mma<MN, MN>(c.RA(), c.sl(2), c.sl(0), true);
            c.commit2();
        }
    }
    if (norm) {
        if (!c.wait_mma()) return;
        c.region_to_record(c.RB(), p.rec1, Ctx::kLower);
    }
    if (c.after) {
        if (!c.wait_mma2()) return;
        c.region_to_record(c.RA(), p.rec, Ctx::kColumn);
    }
}
__global__ void __launch_bounds__(kThreads, 2) bt_x_kernel(const __grid_constant__ Maps m, const __grid_constant__ TParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    Ctx c(smem, p);
    if (!c.aborted()) x_steps(c, m);
    c.finish();
}

// ---------------------------------------------------------------------------
// normalised: num and den of the whole prefix, G' and u, additions to Gam^T and h
// ---------------------------------------------------------------------------
__device__ void upstream_steps(Ctx &c, const Maps &m) {
    const TParams &p = c.p;
    const size_t tok = (size_t)c.head * p.n + c.tile * kTile;
    if (c.tid == 0) {
        c.expect(c.before ? 3 : 2);
        c.load_tokens(0, &m.q);
        if (c.before) {
            c.load_image(1, p.iD, 0);
            c.load_image(2, p.iD, 1);
        } else {
            c.load_tokens(1, &m.g);
        }
    }
    if (c.before && c.tid < kF) c.ms->vec[c.tid] = p.e[c.at * kF + c.tid];
    if (!c.wait_ld()) return;
    float den = 0.f;
    if (c.before) {
        if (c.tid == 0) {
            mma<K, MN>(c.RB(), c.sl(0), c.sl(1), false);  // Q D_p
            mma<K, MN>(c.RB(), c.sl(0), c.sl(2), true);
            c.commit();
        }
#pragma unroll
        for (int g = 0; g < 8; ++g) {  // q . e_p, half a row a thread
            const int c0 = 64 * c.half + 8 * g;
            const uint4 v = *reinterpret_cast<const uint4 *>(c.slot(0) + tile_off(c.r, c0));
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float x0, x1;
                unpack2(w[u], x0, x1);
                den = fmaf(x0, c.ms->vec[c0 + 2 * u], den);
                den = fmaf(x1, c.ms->vec[c0 + 2 * u + 1], den);
            }
        }
        den = c.row_total(den);
        if (!c.wait_mma()) return;
        if (c.tid == 0) {
            c.expect(1);
            c.load_tokens(1, &m.g);
        }
        if (!c.wait_ld()) return;
    }
    const bool ok = c.r < c.len;
    const float inv = ok ? 1.f / (p.den[tok + c.r] + den + p.eps) : 0.f;
    const float4 *num = reinterpret_cast<const float4 *>(p.rec1 + c.at * kRec);
    float go = 0.f;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int c0 = 64 * c.half + 32 * i;
        float x[32], y[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) x[u] = 0.f;
        if (c.before) c.read32(c.RB(), c0, x);
#pragma unroll
        for (int u = 0; u < 32; u += 4) {
            const float4 v = num[rec_index(c.r, c0 + u)];
            x[u] += v.x; x[u + 1] += v.y; x[u + 2] += v.z; x[u + 3] += v.w;
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint4 v = *reinterpret_cast<const uint4 *>(c.slot(1) + tile_off(c.r, c0 + 8 * g));
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float g0, g1;
                unpack2(w[u], g0, g1);
                y[8 * g + 2 * u] = g0 * inv;
                y[8 * g + 2 * u + 1] = g1 * inv;
            }
        }
#pragma unroll
        for (int u = 0; u < 32; ++u) go = fmaf(y[u], x[u], go);
        c.split_store(1, 2, c0, y);  // over the same entries of G
    }
    const float u = -c.row_total(go) * inv;
    if (c.half == 0) {
        c.ms->us[c.r] = u;
        if (ok) p.den[tok + c.r] = u;
    }
    c.publish();
    if (c.tid == 0) {
        c.store_images(p.iG, 1, 2);
        if (c.before) {
            mma<MN, MN>(c.RA(), c.sl(0), c.sl(1), false);  // Q^T G'
            mma<MN, MN>(c.RA(), c.sl(0), c.sl(2), true);
            c.commit();
        }
    }
    if (!c.before) return;
    const float h = c.column_sums(0, -1, c.ms->us);
    if (c.tid < kF) p.h[c.at * kF + c.tid] = h;
    if (c.wait_mma()) c.region_to_record(c.RA(), p.rec);
}
__global__ void __launch_bounds__(kThreads, 2) bt_upstream_kernel(const __grid_constant__ Maps m, const __grid_constant__ TParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    Ctx c(smem, p);
    if (!c.aborted()) upstream_steps(c, m);
    c.finish();
}

// G' (hi and lo images; the plain output's gradient tokens have no lo) into slots; counted by g_tiles()
__device__ __forceinline__ int g_tiles(const Ctx &c) { return c.p.normalized ? 2 : 1; }
__device__ __forceinline__ void load_g(Ctx &c, const Maps &m, int hi, int lo) {
    if (c.p.normalized) {
        c.load_image(hi, c.p.iG, 0);
        c.load_image(lo, c.p.iG, 1);
    } else {
        c.load_tokens(hi, &m.g);
    }
}
__device__ __forceinline__ void load_u(Ctx &c) {
    if (c.p.normalized && c.tid < kTile)
        c.ms->us[c.tid] = c.tid < c.len ? c.p.den[(size_t)c.head * c.p.n + c.tile * kTile + c.tid] : 0.f;
}

// ---------------------------------------------------------------------------
// Y and the additions Q^T Y + Y^T Q to Lam
// ---------------------------------------------------------------------------
__device__ void y_steps(Ctx &c, const Maps &m) {
    const TParams &p = c.p;
    const bool norm = p.normalized;
    if (c.tid == 0) {
        c.expect(1 + g_tiles(c));
        c.load_tokens(0, &m.v);
        load_g(c, m, 1, 2);
    }
    load_u(c);
    if (norm && c.after && c.tid < kF) c.ms->vec[c.tid] = p.h[c.at * kF + c.tid];
    if (!c.wait_ld()) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(0), c.sl(1), false);  // P^T = V G'^T
        if (norm) mma<K, K>(c.RA(), c.sl(0), c.sl(2), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.tid == 0) {
        c.expect(c.after ? 2 : 1);
        if (c.after) {
            c.load_image(1, p.iGam, 0);
            c.load_image(2, p.iGam, 1);
        } else {
            c.load_tokens(1, &m.q);
        }
    }
    c.mask_pack<true>(norm);
    c.publish();
    if (!c.wait_ld()) return;
    if (c.after) {
        if (c.tid == 0) {
            mma<K, K>(c.RB(), c.sl(0), c.sl(1), false);  // V Gam_s: the image holds Gam^T (d rows, dv columns)
            mma<K, K>(c.RB(), c.sl(0), c.sl(2), true);
            c.commit();
        }
        if (!c.wait_mma()) return;
        if (c.tid == 0) {
            c.expect(1);
            c.load_tokens(1, &m.q);
        }
        if (!c.wait_ld()) return;
    }
    if (c.nonfinite(1)) c.drop(1);
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(1), c.after);  // P^T Q
        mma_ts(c.RB(), c.RA() + 16, c.sl(1), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    c.region_to_slots(c.RB(), 0, 2, norm && c.after, Ctx::kUpperT);  // Y over V and Gam; + h_s (rows beyond n meet zero rows of Q)
    c.publish();
    if (c.tid == 0) {
        c.store_images(p.iY, 0, 2);
        if (c.before) {
            mma<MN, MN>(c.RA(), c.sl(1), c.sl(0), false);
            mma<MN, MN>(c.RA(), c.sl(1), c.sl(2), true);
            mma<MN, MN>(c.RA(), c.sl(0), c.sl(1), true);
            mma<MN, MN>(c.RA(), c.sl(2), c.sl(1), true);
            c.commit();
        }
    }
    if (c.before && c.wait_mma()) c.region_to_record(c.RA(), p.rec);
}
__global__ void __launch_bounds__(kThreads, 2) bt_y_kernel(const __grid_constant__ Maps m, const __grid_constant__ TParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    Ctx c(smem, p);
    if (!c.aborted()) y_steps(c, m);
    c.finish();
}

// ---------------------------------------------------------------------------
// gradients: blockIdx.z 0 dQ, 1 dK, 2 dV
// ---------------------------------------------------------------------------
// thread 0: copy one image into a slot once the products issued so far have read it; everyone waits
__device__ __forceinline__ bool swap_in(Ctx &c, int s, const uint8_t *img, int lo) {
    if (c.tid == 0) c.commit();
    if (!c.wait_mma()) return false;
    if (c.tid == 0) {
        c.expect(1);
        c.load_image(s, img, lo);
    }
    return c.wait_ld();
}

__device__ void dq_steps(Ctx &c, const Maps &m) {
    const TParams &p = c.p;
    const bool norm = p.normalized;
    if (c.tid == 0) {
        c.expect(1 + g_tiles(c));
        c.load_tokens(0, &m.v);
        load_g(c, m, 1, 2);
    }
    load_u(c);
    if (norm && c.before && c.tid < kF) c.ms->vec[c.tid] = p.e[c.at * kF + c.tid];
    if (!c.wait_ld()) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(1), c.sl(0), false);  // P = G' V^T
        if (norm) mma<K, K>(c.RA(), c.sl(2), c.sl(0), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.before && c.tid == 0) {
        c.expect(1);
        c.load_image(0, p.iD, 0);
    }
    c.mask_pack<false>(norm);
    c.publish();
    if (c.before) {
        if (!c.wait_ld()) return;
        if (c.tid == 0) {
            mma<K, K>(c.RB(), c.sl(1), c.sl(0), false);  // G' D_p^T
            if (norm) mma<K, K>(c.RB(), c.sl(2), c.sl(0), true);
        }
        if (!swap_in(c, 0, p.iD, 1)) return;
        if (c.tid == 0) {
            mma<K, K>(c.RB(), c.sl(1), c.sl(0), true);
            c.commit();
        }
        if (!c.wait_mma()) return;
    }
    if (c.tid == 0) {
        c.expect(2);
        c.load_image(0, p.iX, 0);
        c.load_image(1, p.iX, 1);
    }
    if (!c.wait_ld()) return;
    if (c.nonfinite(0)) {
        c.drop(0);
        c.drop(1);
    }
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(0), c.before);  // P X
        mma_ts(c.RB(), c.RA() + 16, c.sl(0), true);
        mma_ts(c.RB(), c.RA(), c.sl(1), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.tid == 0) {
        c.expect(3);
        c.load_tokens(0, &m.k);
        c.load_image(1, p.iY, 0);
        c.load_image(2, p.iY, 1);
    }
    if (!c.wait_ld()) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(1), c.sl(0), false);  // B = Y K^T
        mma<K, K>(c.RA(), c.sl(2), c.sl(0), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.nonfinite(0)) c.drop(0);
    c.mask_pack<false>(false);
    c.publish();
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(0), true);  // B K
        mma_ts(c.RB(), c.RA() + 16, c.sl(0), true);
    }
    if (c.before) {
        if (!swap_in(c, 0, p.iS, 0)) return;
        if (c.tid == 0) {
            mma<K, K>(c.RB(), c.sl(1), c.sl(0), true);  // Y S_p
            mma<K, K>(c.RB(), c.sl(2), c.sl(0), true);
        }
        if (!swap_in(c, 0, p.iS, 1)) return;
        if (c.tid == 0) mma<K, K>(c.RB(), c.sl(1), c.sl(0), true);
    }
    if (c.tid == 0) c.commit();
    if (c.wait_mma()) c.region_to_output(c.RB(), 0, &m.dq, p.d, norm && c.before, Ctx::kLower);  // + u e_p^T
}

__device__ void dk_steps(Ctx &c, const Maps &m) {
    const TParams &p = c.p;
    if (c.tid == 0) {
        c.expect(3);
        c.load_tokens(0, &m.k);
        c.load_tokens(1, &m.q);
        c.load_image(2, p.iY, 0);
    }
    if (!c.wait_ld()) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(0), c.sl(1), false);  // W^T = K Q^T
        c.commit();
    }
    if (!c.wait_mma()) return;
    const bool bad_y = c.nonfinite(2);
    if (bad_y) c.drop(2);
    c.mask_pack<true>(false);
    c.publish();
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(2), false);  // W^T Y
        mma_ts(c.RB(), c.RA() + 16, c.sl(2), true);
    }
    if (!swap_in(c, 2, p.iY, 1)) return;
    if (bad_y) c.drop(2);
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(2), true);
        mma<K, K>(c.RA(), c.sl(0), c.sl(2), false);  // B^T = K Y^T over W^T, read by the products before it
    }
    if (!swap_in(c, 2, p.iY, 0)) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(0), c.sl(2), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.after && c.tid == 0) {
        c.expect(1);
        c.load_image(2, p.iLam, 0);
    }
    if (c.nonfinite(1)) c.drop(1);
    c.mask_pack<true>(false);
    c.publish();
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(1), true);  // B^T Q
        mma_ts(c.RB(), c.RA() + 16, c.sl(1), true);
    }
    if (c.after) {
        if (!c.wait_ld()) return;
        if (c.tid == 0) mma<K, K>(c.RB(), c.sl(0), c.sl(2), true);  // K Lam_s (symmetric)
        if (!swap_in(c, 2, p.iLam, 1)) return;
        if (c.tid == 0) mma<K, K>(c.RB(), c.sl(0), c.sl(2), true);
    }
    if (c.tid == 0) c.commit();
    if (c.wait_mma()) c.region_to_output(c.RB(), 0, &m.dk, p.d, false, Ctx::kUpperT);
}

__device__ void dv_steps(Ctx &c, const Maps &m) {
    const TParams &p = c.p;
    if (c.tid == 0) {
        c.expect(3);
        c.load_image(0, p.iX, 0);
        c.load_image(1, p.iX, 1);
        c.load_tokens(2, &m.q);
    }
    if (!c.wait_ld()) return;
    if (c.tid == 0) {
        mma<K, K>(c.RA(), c.sl(0), c.sl(2), false);  // T^T = X Q^T
        mma<K, K>(c.RA(), c.sl(1), c.sl(2), true);
        c.commit();
    }
    if (!c.wait_mma()) return;
    if (c.after && c.tid == 0) {
        c.expect(1);
        c.load_image(2, p.iGam, 0);
    }
    c.mask_pack<true>(false);
    c.publish();
    if (c.after) {
        if (!c.wait_ld()) return;
        if (c.tid == 0) {
            mma<K, MN>(c.RB(), c.sl(0), c.sl(2), false);  // X Gam_s^T
            mma<K, MN>(c.RB(), c.sl(1), c.sl(2), true);
        }
        if (!swap_in(c, 2, p.iGam, 1)) return;
        if (c.tid == 0) {
            mma<K, MN>(c.RB(), c.sl(0), c.sl(2), true);
            c.commit();
        }
        if (!c.wait_mma()) return;
    }
    if (c.tid == 0) {
        c.expect(g_tiles(c));
        load_g(c, m, 0, 1);
    }
    if (!c.wait_ld()) return;
    if (c.nonfinite(0)) {
        c.drop(0);
        if (p.normalized) c.drop(1);
    }
    if (c.tid == 0) {
        mma_ts(c.RB(), c.RA(), c.sl(0), c.after);  // T^T G'
        mma_ts(c.RB(), c.RA() + 16, c.sl(0), true);
        if (p.normalized) mma_ts(c.RB(), c.RA(), c.sl(1), true);
        c.commit();
    }
    if (c.wait_mma()) c.region_to_output(c.RB(), 2, &m.dv, p.dv, false, Ctx::kUpperT);
}
__global__ void __launch_bounds__(kThreads, 2) bt_grad_kernel(const __grid_constant__ Maps m, const __grid_constant__ TParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    Ctx c(smem, p);
    if (!c.aborted()) {
        if (blockIdx.z == 0) dq_steps(c, m);
        else if (blockIdx.z == 1) dk_steps(c, m);
        else dv_steps(c, m);
    }
    c.finish();
}

// ---------------------------------------------------------------------------
// Sums over the tiles of a head: record c becomes, as a hi/lo image pair, the sum of the records before
// it (reverse: after it).  A thread carries 8 columns of a row, eight tiles' loads in flight; two
// neighbouring lanes fill a 32-byte sector of each image.  Block 16 of a head does the same for a vector of 128
// floats in place.  Bound by HBM: 64 KB read and written per tile (with 16 columns a thread, half the threads and
// four tiles in flight, a sum over 1024 tiles took 27 to 33 us, now 20 to 23).
// ---------------------------------------------------------------------------
struct SumsJob {
    const float *rec;
    uint8_t *img;
    float *vec;  // [BH][M][128] or null
    int reverse;
};
struct SumsJobs {
    SumsJob j[2];
};
__global__ void __launch_bounds__(128) bt_scan_kernel(const __grid_constant__ SumsJobs jobs, int M) {
    chain_begin();
    const SumsJob &J = jobs.j[blockIdx.z];
    const int tid = threadIdx.x, head = blockIdx.x / 17, part = blockIdx.x % 17;
    const size_t h0 = (size_t)head * M;
    if (part == 16) {  // the 17 blocks of a head side by side: with all heads' vectors last or first the call took 489 us
        if (!J.vec) return;
        float acc = 0.f;
        for (int i = 0; i < M; ++i) {
            float *p = J.vec + (h0 + (J.reverse ? M - 1 - i : i)) * kF + tid;
            // the last tile's addition (first tile's, in reverse) was not formed
            const float x = i + 1 < M ? *p : 0.f;
            *p = acc;
            acc += x;
        }
        return;
    }
    const int w = part * 4 + (tid >> 5), lane = tid & 31;
    const int r = (w >> 3) * 16 + (lane >> 1), c0 = (w & 7) * 16 + (lane & 1) * 8;
    const uint32_t off = tile_off(r, c0);
    const int i0 = rec_index(r, c0), i1 = rec_index(r, c0 + 4);
    float acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u] = 0.f;
    constexpr int U = 8;
    for (int i = 0; i < M; i += U) {
        float4 v[U][2];
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (i + k + 1 < M) {
                const size_t at = h0 + (J.reverse ? M - 1 - i - k : i + k);
                const float4 *s = reinterpret_cast<const float4 *>(J.rec + at * kRec);
                v[k][0] = s[i0];
                v[k][1] = s[i1];
            }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            if (i + k >= M) break;
            const size_t at = h0 + (J.reverse ? M - 1 - i - k : i + k);
            if (i + k > 0) {  // the first sum is empty and not read
                uint32_t h[4], l[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) split2(acc[2 * u], acc[2 * u + 1], h[u], l[u]);
                uint8_t *o = J.img + at * kPair + off;
                *reinterpret_cast<uint4 *>(o) = make_uint4(h[0], h[1], h[2], h[3]);
                *reinterpret_cast<uint4 *>(o + kImage) = make_uint4(l[0], l[1], l[2], l[3]);
            }
            if (i + k + 1 < M) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    acc[4 * j] += v[k][j].x;
                    acc[4 * j + 1] += v[k][j].y;
                    acc[4 * j + 2] += v[k][j].z;
                    acc[4 * j + 3] += v[k][j].w;
                }
            }
        }
    }
}

// ------------------------------- host side -------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        cudaDriverEntryPointQueryResult qr;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &qr) == cudaSuccess &&
            qr == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(f);
        return static_cast<EncodeTiledFn>(nullptr);
    }();
    return fn;
}

// [BH][n][inner] bf16 (inner 64 or 128), boxes of 64 columns x 128 tokens, 128-byte swizzle, zero fill out of
// range (the box at column 64 of a 64-wide tensor is all fill)
bool make_map(CUtensorMap *m, const void *base, int BH, int n, int inner) {
    cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)n, (cuuint64_t)BH};
    cuuint64_t strides[2] = {(cuuint64_t)inner * 2, (cuuint64_t)n * inner * 2};
    cuuint32_t box[3] = {64, (cuuint32_t)kTile, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct TLayout {
    size_t rec, rec1, iS, iD, iGam, iLam, iX, iY, iG, e, h, den, tokens[4], total;
};
TLayout make_layout(int BH, int n, int d, int dv) {
    const size_t tiles = (size_t)BH * ((n + kTile - 1) / kTile);
    TLayout L;
    size_t o = kWsHeaderBytes;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = align_up(o + bytes, 256);
        return at;
    };
    L.rec = take(tiles * kRec * 4);
    L.rec1 = take(tiles * kRec * 4);
    L.iS = take(tiles * kPair);
    L.iD = take(tiles * kPair);
    L.iGam = take(tiles * kPair);
    L.iLam = take(tiles * kPair);
    L.iX = take(tiles * kPair);
    L.iY = take(tiles * kPair);
    L.iG = take(tiles * kPair);
    L.e = take(tiles * kF * 4);
    L.h = take(tiles * kF * 4);
    L.den = take((size_t)BH * n * 4);
    for (int i = 0; i < 4; ++i) L.tokens[i] = take((size_t)BH * n * (i < 2 ? d : dv) * 2);  // q, k, v, dout
    L.total = o;
    return L;
}

}  // namespace

static bool tiles_sizes(int d, int dv) { return (d == 128 && (dv == 64 || dv == 128)) || (d == 64 && dv == 128); }

size_t backward2_tiles_workspace_bytes(int BH, int n, int d, int dv) {
    if (BH <= 0 || n <= 0 || !tiles_sizes(d, dv)) return kWsHeaderBytes;
    return make_layout(BH, n, d, dv).total;
}

bool backward2_tiles_applicable(const Bwd2 &p) {
    if (getenv("HLA_DISABLE_FUSED")) return false;
    if (p.dt != HLA_BF16 || !tiles_sizes(p.d, p.dv) || p.n <= 0 || p.BH <= 0) return false;
    if (p.ws_bytes < backward2_tiles_workspace_bytes(p.BH, p.n, p.d, p.dv)) return false;
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
    return major == 10 && minor == 3 && encode_fn() != nullptr;
}

cudaError_t backward2_tiles_launch(const Bwd2 &call, cudaStream_t s) {
    Bwd2 p = call;
    const TLayout L = make_layout(p.BH, p.n, p.d, p.dv);
    cudaError_t e = cudaMemsetAsync(p.ws, 0, kWsHeaderBytes, s);
    if (e) return e;
    // the blocks of the last launch write one gradient of a tile each while others read the tile's tokens: a token
    // array that an output lies over is read from a copy
    const void **tokens[4] = {&p.q, &p.k, &p.v, &p.dout};
    for (int i = 0; i < 4; ++i) {
        const size_t bytes = (size_t)p.BH * p.n * (i < 2 ? p.d : p.dv) * 2;
        if (!backward2_over_tokens(call, *tokens[i], bytes)) continue;
        if ((e = cudaMemcpyAsync(p.ws + L.tokens[i], *tokens[i], bytes, cudaMemcpyDeviceToDevice, s))) return e;
        *tokens[i] = p.ws + L.tokens[i];
    }
    Maps m;
    if (!make_map(&m.q, p.q, p.BH, p.n, p.d) || !make_map(&m.k, p.k, p.BH, p.n, p.d) ||
        !make_map(&m.v, p.v, p.BH, p.n, p.dv) || !make_map(&m.g, p.dout, p.BH, p.n, p.dv) ||
        !make_map(&m.dq, p.dq, p.BH, p.n, p.d) || !make_map(&m.dk, p.dk, p.BH, p.n, p.d) ||
        !make_map(&m.dv, p.dval, p.BH, p.n, p.dv))
        return cudaErrorInvalidValue;
    TParams t{};
    t.rec = reinterpret_cast<float *>(p.ws + L.rec);
    t.rec1 = reinterpret_cast<float *>(p.ws + L.rec1);
    auto img = [&](size_t o) { return reinterpret_cast<uint8_t *>(p.ws + o); };
    t.iS = img(L.iS); t.iD = img(L.iD); t.iGam = img(L.iGam); t.iLam = img(L.iLam);
    t.iX = img(L.iX); t.iY = img(L.iY); t.iG = img(L.iG);
    t.e = reinterpret_cast<float *>(p.ws + L.e);
    t.h = reinterpret_cast<float *>(p.ws + L.h);
    t.den = reinterpret_cast<float *>(p.ws + L.den);
    t.n = p.n; t.M = (p.n + kTile - 1) / kTile; t.d = p.d; t.dv = p.dv; t.normalized = p.normalized; t.eps = p.eps;
    t.err = reinterpret_cast<WsHeader *>(p.ws);
    bool follows = false;  // a launch of this call came before
    auto launch = [&](auto kern, int z) -> cudaError_t {
        cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (err) return err;
        err = chain_launch(follows, kern, dim3((unsigned)t.M * (unsigned)p.BH, 1, z), kThreads, kSmemBytes, s, m, t);
        follows = true;
        return err;
    };
    auto sums = [&](SumsJob a, const SumsJob *b) -> cudaError_t {
        SumsJobs jobs{};
        jobs.j[0] = a;
        if (b) jobs.j[1] = *b;
        return chain_launch(true, bt_scan_kernel, dim3(17u * (unsigned)p.BH, 1, b ? 2 : 1), 128, 0, s, jobs, t.M);
    };
    const bool many = t.M > 1, norm = p.normalized;
    if (many) {
        if ((e = launch(bt_sums_kernel, norm ? 1 : 2))) return e;
        const SumsJob gam{t.rec1, t.iGam, nullptr, 1};
        if ((e = sums({t.rec, t.iS, nullptr, 0}, norm ? nullptr : &gam))) return e;
    }
    if ((e = launch(bt_x_kernel, 1))) return e;
    if (many && (e = sums({t.rec, t.iD, norm ? t.e : nullptr, 0}, nullptr))) return e;
    if (norm) {
        if ((e = launch(bt_upstream_kernel, 1))) return e;
        if (many && (e = sums({t.rec, t.iGam, t.h, 1}, nullptr))) return e;
    }
    if ((e = launch(bt_y_kernel, 1))) return e;
    if (many && (e = sums({t.rec, t.iLam, nullptr, 1}, nullptr))) return e;
    return launch(bt_grad_kernel, 3);
}

}  // namespace hla
