// Streaming decode step of second-order HLA (online updates after Theorem 1,
// outputs of Theorem 1 / Eq. hla-row), one block per SM working through heads.
//
// The step is a read-modify-write of the fp32 state tuple (S, C, m, G, h):
//   masked:  G' = G + k (k^T C),  h' = h + k (k^T m)       (previous C, m)
//   S' = S + k k^T,  C' = C + q v^T,  m' = m + q
//   u' = S' q = S q + k (k.q)                               (S symmetric)
//   num = u'^T C' - q^T G' = u'^T C + (u'.q) v^T - q^T G - (q.k)(k^T C)
//   den = u'.m' - q.h'     = u'.(m + q) - q.h - (q.k)(k.m)
// so one pass over S (giving u'), one pass over C (the column sums k^T C and
// u'^T C), then one pass over G that reads q^T G from the old values and writes
// G' = G + k (k^T C) at once.  The unmasked form skips G and h (and leaves them
// untouched).
//
// Memory access: every matrix is read once into shared memory by a 1-D bulk copy
// (one instruction per matrix, completing on an mbarrier), issued a pass or more
// ahead of its use, and written once with 16-byte stores; consecutive threads on
// consecutive columns.
#include "hla_internal.h"
#include "sm103_prims.cuh"
#include "step_split.cuh"

namespace hla {
namespace {

constexpr int kStepThreads = 512;
constexpr int kMaxUnits = 128 * 128 / 4 / kStepThreads;  // float4 units per thread for a 128 x 128 matrix

__device__ __forceinline__ float group_sum_rt(float x, int w) {
    switch (w) {
        case 4: return group_sum<4>(x);
        case 8: return group_sum<8>(x);
        case 16: return group_sum<16>(x);
        default: return group_sum<32>(x);
    }
}

// Sums over the 32 lanes of a warp of eight values v[0..7] at once (9 shuffles instead of 40): on
// return, lane l holds the sum of v[l >> 2] (each step keeps half of the values a lane still holds)
__device__ __forceinline__ float warp_sum8(float (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = (lane & 16) != 0;
        const float send = up ? v[i] : v[i + 4], keep = up ? v[i + 4] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool up = (lane & 8) != 0;
        const float send = up ? v[i] : v[i + 2], keep = up ? v[i + 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    {
        const bool up = (lane & 4) != 0;
        const float send = up ? v[0] : v[1], keep = up ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    float x = v[0];
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x;
}

// 1-D bulk copy global -> shared (16-byte aligned, a multiple of 16 bytes), completing on `bar`
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(sm103::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes),
                   "r"(sm103::smem_u32(bar))
                 : "memory");
}
constexpr unsigned long long kCopyWaitNs = 2000000000ull;
__device__ __forceinline__ void store4(float4 *p, float4 v) { *p = v; }

// One block per SM, heads hd = blockIdx.x, + gridDim.x, ...  The state of a head is staged in shared
// memory in three buffers, one per pass (S; C with m; G with h), each refilled with the next head's
// part as soon as its pass has read it, so that while one pass works the copies of the next two
// parts (and of the next head's tokens) are in flight.  Thread 0 issues each refill as one bulk copy
// on the buffer's mbarrier (phase = the block's head count); every thread waits on it, bounded: a
// copy that never lands ends the block.  Updated values go to global memory straight from registers.
//
// kSDE: the state is (S, D, e) with D = S C - G and e = S m - h (masked operator only; rows of the
// per-head record: S d*d | D d*dv | e d).  A token then updates
//   S' = S + k k^T,  u' = S' q,  D' = D + u' v^T,  e' = e + u'
// and num = q^T D' = q^T D + (q.u') v^T, den = q.e' = q.e + q.u': one pass over S and one over D.
template <typename T, bool kSDE>
__global__ void __launch_bounds__(kStepThreads, 1)
step2_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, T *__restrict__ out,
             float *__restrict__ state, int BH, int d, int dv, int masked, int normalized, float eps) {
    extern __shared__ float4 dyn[];
    __shared__ float qs[128], ks[128], vs[128], us[128];
    __shared__ float part[kStepThreads][12];
    __shared__ float kC[128], uC[128], qG[128];
    __shared__ uint64_t bar[3];  // S and tokens; (C, m) or (D, e); (G, h)

    const int tid = threadIdx.x;
    if (kSDE) masked = 0;  // staging as for (S, C, m): no third buffer
    const long long st_len = kSDE ? (long long)d * d + (long long)d * dv + d : (long long)d * d + 2LL * d * dv + 2LL * d;
    const int nS = (d * d) >> 2, nCm = (d * dv + d) >> 2;  // float4 units of S and of (C, m) / (G, h)
    const int nt_q = d * (int)sizeof(T) / 16, nt_v = dv * (int)sizeof(T) / 16;  // 16-byte token chunks
    float4 *bS = dyn, *bC = bS + nS, *bG = bC + nCm;
    float4 *bT = bG + (masked ? nCm : 0);  // raw tokens q | k | v
    const T *tq = reinterpret_cast<const T *>(bT), *tk = tq + d, *tv = tk + d;

    // thread 0 issues the copies: after a block barrier that ends the generic reads of the buffer
    auto load_S = [&](int hd) {  // S and the head's tokens
        if (tid == 0) {
            sm103::fence_async_smem();
            sm103::mbar_arrive_expect_tx(&bar[0], (uint32_t)(16 * (nS + 2 * nt_q + nt_v)));
            bulk_copy(bS, state + hd * st_len, 16u * nS, &bar[0]);
            bulk_copy(bT, q + (long long)hd * d, 16u * nt_q, &bar[0]);
            bulk_copy(bT + nt_q, k + (long long)hd * d, 16u * nt_q, &bar[0]);
            bulk_copy(bT + 2 * nt_q, v + (long long)hd * dv, 16u * nt_v, &bar[0]);
        }
    };
    auto load_part = [&](float4 *dst, int hd, long long off, int b) {  // (C, m), (D, e) or (G, h)
        if (tid == 0) {
            sm103::fence_async_smem();
            sm103::mbar_arrive_expect_tx(&bar[b], 16u * nCm);
            bulk_copy(dst, state + hd * st_len + off, 16u * nCm, &bar[b]);
        }
    };
    const long long offC = (long long)d * d, offG = offC + (long long)d * dv + d;

    int hd = blockIdx.x;
    if (hd >= BH) return;
    if (tid == 0) {
        for (int b = 0; b < 3; ++b) sm103::mbar_init(&bar[b], 1);
        sm103::fence_mbar_init();
    }
    __syncthreads();
    load_S(hd);
    load_part(bC, hd, offC, 1);
    if (masked) load_part(bG, hd, offG, 2);
    for (uint32_t par = 0; hd < BH; hd += gridDim.x, par ^= 1u) {
        const int nx = hd + gridDim.x;  // this block's next head (none: empty copy groups)
        float *S = state + hd * st_len;
        float *Cm = S + offC;
        float *m = Cm + (long long)d * dv;
        float *G = S + offG;
        float *h = G + (long long)d * dv;

        // ---- tokens, k.q ----
        if (!sm103::mbar_wait(&bar[0], par, kCopyWaitNs)) return;  // S and tokens of this head
        if (tid < d) {
            qs[tid] = to_f32(tq[tid]);
            ks[tid] = to_f32(tk[tid]);
        }
        if (tid < dv) vs[tid] = to_f32(tv[tid]);
        __syncthreads();
        const float kq = warp_dot(ks, qs, d);

        // ---- pass over S: u = S q, S' = S + k k^T ----
        if (d == 128 && kMaxUnits == 8) {
            // a warp covers one row per unit (rows warp + 16 i): the eight row sums in one reduction
            float4 *Sg = reinterpret_cast<float4 *>(S);
            const int c4 = (tid & 31) * 4;
            const float q0 = qs[c4], q1 = qs[c4 + 1], q2 = qs[c4 + 2], q3 = qs[c4 + 3];
            const float k0 = ks[c4], k1 = ks[c4 + 1], k2 = ks[c4 + 2], k3 = ks[c4 + 3];
            float pu[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int f = tid + i * kStepThreads;
                const float4 sv = bS[f];
                pu[i] = sv.x * q0 + sv.y * q1 + sv.z * q2 + sv.w * q3;
                const float kr = ks[f >> 5];
                store4(Sg + f, make_float4(sv.x + kr * k0, sv.y + kr * k1, sv.z + kr * k2, sv.w + kr * k3));
            }
            const float su = warp_sum8(pu);
            if ((tid & 3) == 0) {
                const int row = (tid >> 5) + 16 * ((tid & 31) >> 2);
                us[row] = su + ks[row] * kq;  // u' = S q + k (k.q)
            }
        } else {
            const int w = d >> 2;  // float4 units per row of S
            float4 *Sg = reinterpret_cast<float4 *>(S);
#pragma unroll
            for (int i = 0; i < kMaxUnits; ++i) {
                const int f = tid + i * kStepThreads;
                if (i * kStepThreads < nS) {  // uniform per iteration: shuffles stay convergent
                    float part_u = 0.f;
                    if (f < nS) {
                        const int row = f / w, c4 = (f % w) * 4;
                        const float4 sv = bS[f];
                        part_u = sv.x * qs[c4] + sv.y * qs[c4 + 1] + sv.z * qs[c4 + 2] + sv.w * qs[c4 + 3];
                        const float kr = ks[row];
                        store4(Sg + f, make_float4(sv.x + kr * ks[c4], sv.y + kr * ks[c4 + 1],
                                                      sv.z + kr * ks[c4 + 2], sv.w + kr * ks[c4 + 3]));
                    }
                    part_u = group_sum_rt(part_u, w);
                    if (f < nS && (f % w) == 0) {
                        const int row = f / w;
                        us[row] = part_u + ks[row] * kq;  // u' = S q + k (k.q)
                    }
                }
            }
        }
        __syncthreads();  // S buffer read, u' complete
        if (nx < BH) load_S(nx);

        if constexpr (kSDE) {
            // ---- pass over D: column sums q^T D (old D); D' = D + u' v^T; e' = e + u' ----
            if (!sm103::mbar_wait(&bar[1], par, kCopyWaitNs)) return;  // (D, e) of this head
            const float *ev = reinterpret_cast<const float *>(bC + ((d * dv) >> 2));
            float *eg = Cm + (long long)d * dv;
            if (tid < d) eg[tid] = ev[tid] + us[tid];
            const float qe = warp_dot(qs, ev, d), uq = warp_dot(us, qs, d);
            const int wv = dv >> 2, nD = (d * dv) >> 2, c4 = (tid % wv) * 4;
            {
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                float4 *Dg = reinterpret_cast<float4 *>(Cm);
                const float v0 = vs[c4], v1 = vs[c4 + 1], v2 = vs[c4 + 2], v3 = vs[c4 + 3];
#pragma unroll
                for (int i = 0; i < kMaxUnits; ++i) {
                    const int f = tid + i * kStepThreads;
                    if (f < nD) {
                        const int row = f / wv;
                        const float4 c = bC[f];
                        const float qr = qs[row], ur = us[row];
                        acc.x += qr * c.x; acc.y += qr * c.y; acc.z += qr * c.z; acc.w += qr * c.w;
                        store4(Dg + f, make_float4(c.x + ur * v0, c.y + ur * v1, c.z + ur * v2, c.w + ur * v3));
                    }
                }
                part[tid][0] = acc.x; part[tid][1] = acc.y; part[tid][2] = acc.z; part[tid][3] = acc.w;
            }
            __syncthreads();  // (D, e) buffer read
            if (nx < BH) load_part(bC, nx, offC, 1);
            if (tid < dv) {
                const int grp = tid >> 2, comp = tid & 3;
                float a = 0.f;
                for (int g = grp; g < kStepThreads; g += wv) a += part[g][comp];
                const float num = a + uq * vs[tid];
                from_f32(&out[(long long)hd * dv + tid], normalized ? num / (qe + uq + eps) : num);
            }
            __syncthreads();  // qs, ks, vs, us, part read before the next head rewrites them
            continue;
        }

        // ---- pass over C: column sums k^T C, u'^T C; C' = C + q v^T; m' = m + q ----
        if (!sm103::mbar_wait(&bar[1], par, kCopyWaitNs)) return;  // (C, m) of this head
        const float *mv = reinterpret_cast<const float *>(bC + ((d * dv) >> 2));
        if (tid < d) m[tid] = mv[tid] + qs[tid];
        const float uq = warp_dot(us, qs, d), km = warp_dot(ks, mv, d);
        const float um = warp_dot(us, mv, d) + uq;  // u'.(m + q)
        const int wv = dv >> 2;
        const int nC = (d * dv) >> 2;
        const int c4 = (tid % wv) * 4;  // fixed column group of this thread
        {
            float4 acc_kC = make_float4(0.f, 0.f, 0.f, 0.f), acc_uC = acc_kC;
            float4 *Cg = reinterpret_cast<float4 *>(Cm);
            const float v0 = vs[c4], v1 = vs[c4 + 1], v2 = vs[c4 + 2], v3 = vs[c4 + 3];
#pragma unroll
            for (int i = 0; i < kMaxUnits; ++i) {
                const int f = tid + i * kStepThreads;
                if (f < nC) {
                    const int row = f / wv;
                    const float4 c = bC[f];
                    const float kr = ks[row], ur = us[row], qr = qs[row];
                    acc_kC.x += kr * c.x; acc_kC.y += kr * c.y; acc_kC.z += kr * c.z; acc_kC.w += kr * c.w;
                    acc_uC.x += ur * c.x; acc_uC.y += ur * c.y; acc_uC.z += ur * c.z; acc_uC.w += ur * c.w;
                    store4(Cg + f, make_float4(c.x + qr * v0, c.y + qr * v1, c.z + qr * v2, c.w + qr * v3));
                }
            }
            part[tid][0] = acc_kC.x; part[tid][1] = acc_kC.y; part[tid][2] = acc_kC.z; part[tid][3] = acc_kC.w;
            part[tid][4] = acc_uC.x; part[tid][5] = acc_uC.y; part[tid][6] = acc_uC.z; part[tid][7] = acc_uC.w;
        }
        __syncthreads();  // (C, m) buffer read
        if (nx < BH) load_part(bC, nx, offC, 1);
        if (tid < dv) {
            const int grp = tid >> 2, comp = tid & 3;
            float a = 0.f, b = 0.f;
            for (int g = grp; g < kStepThreads; g += wv) { a += part[g][comp]; b += part[g][4 + comp]; }
            kC[tid] = a; uC[tid] = b;
        }
        __syncthreads();

        // ---- pass over G: column sums q^T G (old G); G' = G + k (k^T C); h' = h + k (k.m) ----
        float qh = 0.f;
        if (masked) {
            if (!sm103::mbar_wait(&bar[2], par, kCopyWaitNs)) return;  // (G, h) of this head
            const float *hv = reinterpret_cast<const float *>(bG + nC);
            if (tid < d) h[tid] = hv[tid] + ks[tid] * km;
            qh = warp_dot(qs, hv, d);
            float4 acc_qG = make_float4(0.f, 0.f, 0.f, 0.f);
            float4 *Gg = reinterpret_cast<float4 *>(G);
            const float a0 = kC[c4], a1 = kC[c4 + 1], a2 = kC[c4 + 2], a3 = kC[c4 + 3];
#pragma unroll
            for (int i = 0; i < kMaxUnits; ++i) {
                const int f = tid + i * kStepThreads;
                if (f < nC) {
                    const int row = f / wv;
                    const float kr = ks[row], qr = qs[row];
                    const float4 g = bG[f];
                    acc_qG.x += qr * g.x; acc_qG.y += qr * g.y; acc_qG.z += qr * g.z; acc_qG.w += qr * g.w;
                    store4(Gg + f, make_float4(g.x + kr * a0, g.y + kr * a1, g.z + kr * a2, g.w + kr * a3));
                }
            }
            part[tid][8] = acc_qG.x; part[tid][9] = acc_qG.y; part[tid][10] = acc_qG.z; part[tid][11] = acc_qG.w;
            __syncthreads();  // part written, the (G, h) buffer read
            if (nx < BH) load_part(bG, nx, offG, 2);
            if (tid < dv) {
                const int grp = tid >> 2, comp = tid & 3;
                float c = 0.f;
                for (int g = grp; g < kStepThreads; g += wv) c += part[g][8 + comp];
                qG[tid] = c;
            }
            __syncthreads();
        }

        // ---- output ----
        if (tid < dv) {
            float num = uC[tid] + uq * vs[tid];
            float den = um;
            if (masked) {
                num -= qG[tid] + kq * kC[tid];
                den -= qh + kq * km;
            }
            from_f32(&out[(long long)hd * dv + tid], normalized ? num / (den + eps) : num);
        }
        __syncthreads();  // qs, ks, vs, us, kC, uC, qG read before the next head rewrites them
    }
}

// ---------------------------------------------------------------------------
// The step with every load issued at once, straight to registers: for head sizes up to 64 (one block of
// 256 threads a head, several on an SM), and for few heads of 128 (a cluster of `split` blocks of 512
// threads a head, block r with columns [r dv / split, ...) of C and G, or D, and the rows of S that it
// writes).  The staged kernel above brings a head through one SM part by part; with small
// heads it waits on each part in turn, with few heads most SMs are idle.  Each block forms u' = S' q from
// all of S (a cluster's redundant reads come from L2 and cost less than an exchange between blocks), so
// the blocks of a cluster meet only once, in a split barrier between their last read of S, m and h and
// the first write to them.  Column sums go by shuffles, then over the warps in shared memory.
// Measured, us a step (staged -> this), bf16 tokens: tuple 64 x 64, 16 heads 6.6 -> 4.8, 256 heads
// 12.1 -> 5.9, 2048 heads 74.9 -> 43.7; (S, D, e) 64 x 64, 16 heads 4.6 -> 4.1, 2048 heads 44.9 -> 28.9;
// tuple 128 x 128, 8 heads 7.7 -> 6.3, 32 heads 7.9 -> 6.7.  It is bound by the latency of a load,
// three barriers and the shuffles between them; with many heads by its registers (two or three blocks
// an SM; one more spilled and was slower).  Sums over a slice take an entry that is exactly zero for the rows
// beyond it, and the output is written after the cluster's barrier: 0 to 4 % less time for up to 256 heads, 2048
// heads of 64 x 64 on the tuple 47.7 -> 49.7 (8 bytes spilled).
// NS, NC: float4 units that a thread takes of S and of a column slice.
// ---------------------------------------------------------------------------
template <typename T, bool kSDE, int TH, int NS, int NC>
__global__ void __launch_bounds__(TH, TH == 256 ? (kSDE ? 3 : 2) : 1)
step2_split_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, T *__restrict__ out,
                   float *state, int split, int d, int dv, int masked, int normalized, float eps) {
    // entry d is zero: it stands for the rows beyond a slice (an infinite entry would make NaN of their zeros)
    __shared__ __align__(16) float qs[132], ks[132], vs[128], us[132];
    // per warp: sums of a column slice (at most 64 columns), for k^T C and u'^T C (or q^T D), and q^T G
    __shared__ __align__(16) float part[3][TH / 32][64];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int hd = blockIdx.x / split, rank = blockIdx.x % split, cw = dv / split, col0 = rank * cw;
    const long long offC = (long long)d * d, lenC = (long long)d * dv + d;
    float *S = state + hd * (offC + lenC * (kSDE ? 1 : 2)), *C = S + offC, *m = C + (long long)d * dv;
    float *G = C + lenC, *h = G + (long long)d * dv;
    const int nS = (d * d) >> 2, wS = d >> 2;     // float4 units of S, of one of its rows
    const int wC = cw >> 2, nC = d * wC;          // of a row of the slice, of the slice
    const int c4 = (tid % wC) * 4, r0 = tid / wC, rstep = TH / wC;

    // every load of the step
    float4 sv[NS], cv[NC], gv[NC];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const int f = tid + i * TH;
        sv[i] = f < nS ? reinterpret_cast<const float4 *>(S)[f] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const int row = r0 + i * rstep;
        const bool ok = tid + i * TH < nC;
        cv[i] = gv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok) cv[i] = *reinterpret_cast<const float4 *>(C + (long long)row * dv + col0 + c4);
        if (!kSDE && masked && ok) gv[i] = *reinterpret_cast<const float4 *>(G + (long long)row * dv + col0 + c4);
    }
    // m and h (or e): four values a lane, in every warp
    float mv[4], hv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = lane + 32 * i;
        mv[i] = a < d ? m[a] : 0.f;
        hv[i] = !kSDE && masked && a < d ? h[a] : 0.f;
    }
    if (tid < d) {
        qs[tid] = to_f32(q[(long long)hd * d + tid]);
        ks[tid] = to_f32(k[(long long)hd * d + tid]);
    }
    if (tid < dv) vs[tid] = to_f32(v[(long long)hd * dv + tid]);
    if (tid == 0) qs[d] = ks[d] = us[d] = 0.f;
    __syncthreads();
    const float kq = warp_dot(ks, qs, d);
    float km = 0.f, qm = 0.f, qh = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = lane + 32 * i;
        if (a < d) {
            km = fmaf(ks[a], mv[i], km);
            qm = fmaf(qs[a], mv[i], qm);
            qh = fmaf(qs[a], hv[i], qh);
        }
    }
    km = group_sum<32>(km);
    qm = group_sum<32>(qm);
    qh = group_sum<32>(qh);

    // u' = S q + k (k.q)
    if constexpr (NS == 8) {  // d = 128: a warp covers one row per unit
        const int c = lane * 4;
        float pu[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            pu[i] = sv[i].x * qs[c] + sv[i].y * qs[c + 1] + sv[i].z * qs[c + 2] + sv[i].w * qs[c + 3];
        const float su = warp_sum8(pu);
        if ((lane & 3) == 0) {
            const int row = wid + TH / 32 * (lane >> 2);
            us[row] = su + ks[row] * kq;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const int f = tid + i * TH, row = f / wS, c = (f % wS) * 4;
            float pu = 0.f;
            if (f < nS) pu = sv[i].x * qs[c] + sv[i].y * qs[c + 1] + sv[i].z * qs[c + 2] + sv[i].w * qs[c + 3];
            pu = group_sum_rt(pu, wS);
            if (f < nS && f % wS == 0) us[row] = pu + ks[row] * kq;
        }
    }
    // sums that need no u': k^T C, q^T G; or q^T D
    float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const int row = min(r0 + i * rstep, d);
        fma4(a0, kSDE ? qs[row] : ks[row], cv[i]);
        if (!kSDE) fma4(a1, qs[row], gv[i]);
    }
    a0 = column_sum(a0, wC);
    if (!kSDE) a1 = column_sum(a1, wC);
    if (lane < wC) {
        *reinterpret_cast<float4 *>(&part[0][wid][c4]) = a0;
        if (!kSDE) *reinterpret_cast<float4 *>(&part[2][wid][c4]) = a1;
    }
    cluster_arrive();  // this block has read S, m, h and the tokens
    __syncthreads();   // us, part
    const float uq = warp_dot(us, qs, d);
    const float4 v4 = *reinterpret_cast<const float4 *>(vs + col0 + c4);
    float4 kC = make_float4(0.f, 0.f, 0.f, 0.f);
    float um = 0.f;
    if (!kSDE) {
        for (int w = 0; w < TH / 32; ++w) fma4(kC, 1.f, *reinterpret_cast<const float4 *>(&part[0][w][c4]));
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (lane + 32 * i < d) um = fmaf(us[lane + 32 * i], mv[i], um);
        um = group_sum<32>(um) + uq;  // u'.(m + q)
        a0 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < NC; ++i) fma4(a0, us[min(r0 + i * rstep, d)], cv[i]);
        a0 = column_sum(a0, wC);
        if (lane < wC) *reinterpret_cast<float4 *>(&part[1][wid][c4]) = a0;
    }
    // the updated slices
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const int row = r0 + i * rstep;
        if (tid + i * TH >= nC) continue;
        *reinterpret_cast<float4 *>(C + (long long)row * dv + col0 + c4) = axpy4(cv[i], kSDE ? us[row] : qs[row], v4);
        if (!kSDE && masked)
            *reinterpret_cast<float4 *>(G + (long long)row * dv + col0 + c4) = axpy4(gv[i], ks[row], kC);
    }
    __syncthreads();  // part[1]
    float result = 0.f;
    if (tid < cw) {
        float x0 = 0.f, x1 = 0.f, x2 = 0.f;
        for (int w = 0; w < TH / 32; ++w) {
            x0 += part[0][w][tid];
            if (!kSDE) {
                x1 += part[1][w][tid];
                x2 += part[2][w][tid];
            }
        }
        float num, den;
        if (kSDE) {
            num = x0 + uq * vs[col0 + tid];
            den = qm + uq;
        } else {
            num = x1 + uq * vs[col0 + tid];
            den = um;
            if (masked) {
                num -= x2 + kq * x0;
                den -= qh + kq * km;
            }
        }
        result = normalized ? num / (den + eps) : num;
    }
    cluster_wait();  // every block of the head has read S, m, h and the tokens, over which `out` may lie
    if (tid < cw) from_f32(&out[(long long)hd * dv + col0 + tid], result);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const int f = tid + i * TH, row = f / wS, c = (f % wS) * 4;
        if (f < nS && row * split / d == rank)
            reinterpret_cast<float4 *>(S)[f] = axpy4(sv[i], ks[row], *reinterpret_cast<const float4 *>(ks + c));
    }
    if (rank == 0 && wid == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int a = lane + 32 * i;
            if (a >= d) continue;
            m[a] = mv[i] + (kSDE ? us[a] : qs[a]);
            if (!kSDE && masked) h[a] = hv[i] + ks[a] * km;
        }
    }
}

// Blocks per head of the kernel above, 0 where the staged kernel serves.  Head sizes up to 64: one,
// for any number of heads (two or four were as fast for few heads and slower for many).  With a size of
// 128, clusters while each fits the chip at once, one block an SM and a cluster within one GPC: 8 heads in
// eights, 32 in fours (16 in eights and 38 in fours take two rounds, 11.5 and 12.1 us); in twos the
// staged kernel is as fast (8.0 against 7.9 us at 40 heads); the unmasked tuple, which has no third pass to wait
// for, stays with the staged kernel at d = 128 unless dv is 16 (16 heads of 128 x 128 6.0 against 6.3 us).  A block's
// slice has 8 to 64 columns.
int step2_split(int BH, int d, int dv, bool unmasked) {
    int s = 1;
    if (unmasked && d == 128 && dv >= 32) return 0;
    if (d == 128 || dv == 128) s = BH <= 8 ? 8 : BH <= 32 ? 4 : 0;
    if (s == 0) return 0;
    while (s > 1 && dv / s < 8) s /= 2;
    while (dv / s > 64) s *= 2;
    return s;
}

template <typename T, bool kSDE>
cudaError_t step2_split_launch(const void *q, const void *k, const void *v, void *out, float *state, int BH, int split,
                               int d, int dv, int masked, int normalized, float eps, cudaStream_t stream) {
    auto go = [&](auto kern, int threads) {
        return launch_blocks(kern, BH, split, true, threads, stream, static_cast<const T *>(q), static_cast<const T *>(k),
                            static_cast<const T *>(v), static_cast<T *>(out), state, split, d, dv, masked, normalized,
                            eps);
    };
    const int units = d * (dv / split) / 4;  // of a slice: of 8 to 64 columns, 8 to 32 at d = 128
    if (d == 128) {
        if (units <= 512) return go(step2_split_kernel<T, kSDE, 512, 8, 1>, 512);
        if (units <= 1024) return go(step2_split_kernel<T, kSDE, 512, 8, 2>, 512);
        return cudaErrorInvalidValue;
    }
    if (units <= 256) return go(step2_split_kernel<T, kSDE, 256, 4, 1>, 256);
    if (units <= 512) return go(step2_split_kernel<T, kSDE, 256, 4, 2>, 256);
    if (units <= 1024) return go(step2_split_kernel<T, kSDE, 256, 4, 4>, 256);
    return cudaErrorInvalidValue;
}

// dynamic shared memory of step2_kernel: S, (C, m), (G, h) if masked, tokens
size_t step2_smem(int d, int dv, int masked, size_t tsize) {
    const size_t nS = (size_t)d * d / 4, nCm = ((size_t)d * dv + d) / 4;
    return 16 * (nS + nCm * (masked ? 2 : 1)) + tsize * (2 * (size_t)d + dv);
}

template <bool kSDE>
cudaError_t step2_launch_t(const void *q, const void *k, const void *v, void *out, hla_dtype dt, int BH, int d,
                           int dv, int masked, int normalized, float eps, float *state, cudaStream_t stream) {
    if (BH == 0) return cudaSuccess;
    if (const int split = step2_split(BH, d, dv, !kSDE && !masked))
        return dt == HLA_BF16 ? step2_split_launch<__nv_bfloat16, kSDE>(q, k, v, out, state, BH, split, d, dv, masked,
                                                                        normalized, eps, stream)
                              : step2_split_launch<float, kSDE>(q, k, v, out, state, BH, split, d, dv, masked, normalized,
                                                                eps, stream);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int grid = BH < sms ? BH : sms;
    if (kSDE) masked = 0;  // shared-memory staging of (S, D, e) is that of (S, C, m)
    if (dt == HLA_BF16) {
        auto kern = step2_kernel<__nv_bfloat16, kSDE>;
        const size_t sm = step2_smem(d, dv, masked, sizeof(__nv_bfloat16));
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
        kern<<<grid, kStepThreads, sm, stream>>>(static_cast<const __nv_bfloat16 *>(q),
                                                static_cast<const __nv_bfloat16 *>(k),
                                                static_cast<const __nv_bfloat16 *>(v),
                                                static_cast<__nv_bfloat16 *>(out), state, BH, d, dv, masked,
                                                normalized, eps);
    } else {
        auto kern = step2_kernel<float, kSDE>;
        const size_t sm = step2_smem(d, dv, masked, sizeof(float));
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
        kern<<<grid, kStepThreads, sm, stream>>>(static_cast<const float *>(q), static_cast<const float *>(k),
                                                static_cast<const float *>(v), static_cast<float *>(out), state,
                                                BH, d, dv, masked, normalized, eps);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t step2_launch(const void *q, const void *k, const void *v, void *out, hla_dtype dt, int BH, int d, int dv,
                         int masked, int normalized, float eps, float *state, cudaStream_t stream) {
    return step2_launch_t<false>(q, k, v, out, dt, BH, d, dv, masked, normalized, eps, state, stream);
}

cudaError_t step2_sde_launch(const void *q, const void *k, const void *v, void *out, hla_dtype dt, int BH, int d,
                             int dv, int normalized, float eps, float *state, cudaStream_t stream) {
    return step2_launch_t<true>(q, k, v, out, dt, BH, d, dv, 1, normalized, eps, state, stream);
}

namespace {

// (S, C, m, G, h) -> (S, D = S C - G, e = S m - h) per head, one block per head, the tuple staged in
// shared memory (dst must not overlap src: blocks of other heads may still be reading it).
__global__ void __launch_bounds__(256) state_to_sde_kernel(const float *src, float *dst, int d, int dv) {
    extern __shared__ float st[];
    const int hd = blockIdx.x, tid = threadIdx.x;
    const long long len = (long long)d * d + 2LL * d * dv + 2LL * d;
    const float4 *s4 = reinterpret_cast<const float4 *>(src + hd * len);
    float4 *st4 = reinterpret_cast<float4 *>(st);
    for (int i = tid; i < (int)(len >> 2); i += blockDim.x) st4[i] = s4[i];
    __syncthreads();
    const float *S = st, *C = S + d * d, *m = C + d * dv, *G = m + d, *h = G + d * dv;
    float *o = dst + hd * ((long long)d * d + (long long)d * dv + d);
    for (int i = tid; i < d * d; i += blockDim.x) o[i] = S[i];
    for (int i = tid; i < d * dv + d; i += blockDim.x) {
        const bool is_e = i >= d * dv;
        const int a = is_e ? i - d * dv : i / dv, b = is_e ? 0 : i % dv;
        float acc = 0.f;
        for (int j = 0; j < d; ++j) acc += S[a * d + j] * (is_e ? m[j] : C[j * dv + b]);
        o[d * d + i] = acc - (is_e ? h[a] : G[i]);
    }
}

}  // namespace

cudaError_t state_to_sde_launch(const float *src, float *dst, int BH, int d, int dv, cudaStream_t stream) {
    if (BH == 0) return cudaSuccess;
    const size_t smem = sizeof(float) * ((size_t)d * d + 2 * (size_t)d * dv + 2 * (size_t)d);
    cudaError_t e = cudaFuncSetAttribute(state_to_sde_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    state_to_sde_kernel<<<BH, 256, smem, stream>>>(src, dst, d, dv);
    return cudaGetLastError();
}

}  // namespace hla
