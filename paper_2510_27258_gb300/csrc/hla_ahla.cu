// Asymmetric second-order HLA (AHLA): chunk-parallel forward and decode step on
// the CUDA cores in fp32 (Sec. "Asymmetric Higher-order Linear Attention").
//
// AHLA is causal linear attention applied twice: with A = L . (Q K^T) (L lower
// triangular incl. the diagonal), r_t = q_t^T P_t = (A V)_t and
// o_t = q_t^T E_t = (A R)_t (Theorem AHLA: P_t = sum_{j<=t} k_j v_j^T,
// E_t = sum_{i<=t} k_i r_i^T; denominators with v -> 1).  Per 64-token chunk, rows
// are its tokens and "p" the prefix before it:
//   R = A V + Q P_p,   s = A 1 + Q m_p,   O = A R + Q E_p,   den = A s + Q n_p.
// Every carry is a plain prefix sum: P += K^T V, m += K^T 1 and, once R is formed
// with the chunk's own P_p, E += K^T R, n += K^T s (the cross term R^KQ_B P_A of
// Eq. AHLA-semidirect is in R).  Launches: K^T V of every chunk; its prefix sums;
// A, R, A R and E's increments; E's prefix sums; outputs.  The states' [P | m] and
// [E | n] start and end the sums as they lie.
//
// The scan that multiplied each chunk's R^KQ with P held 4.5 of 6.1 ms at
// B1 H32 n1999 d128 bf16 with states; as prefix sums the call takes 322 us.
#include <algorithm>

#include "chunk_simt.cuh"
#include "sm103_prims.cuh"
#include "step_split.cuh"

namespace hla {
namespace {

inline long long up16(long long x) { return (x + 15) / 16 * 16; }

struct ALayout {
    int nch, len;  // chunks of a head; floats of a record [P | m] or [E | n]
    // floats from the scratch start: P records, E records, A R (fp32 [BH][n][dv]), A s ([BH][n])
    long long oP, oE, oNum, oDen, total;
};

ALayout make_layout(int BH, int n, int d, int dv) {
    ALayout L;
    L.nch = (n + kC - 1) / kC;
    L.len = d * dv + d;
    const long long recs = (long long)BH * (L.nch + 1);
    long long o = 0;
    L.oP = o; o += recs * L.len;
    L.oE = o; o += recs * L.len;
    L.oNum = o; o += up16((long long)BH * n * dv);
    L.oDen = o; o += up16((long long)BH * n);
    L.total = o;
    return L;
}

struct AParams {
    Records P, E;
    float *num, *den;
    int n, d, dv, normalized;
    float eps;
    int has_in;  // a state comes in: the first chunk has a carry
    int direct;  // one chunk from a zero state: this launch writes the outputs
    int need_E;  // E's increments of the last chunk are wanted too (final state)
};

// per chunk: A, [R | s], A [R | s] and the increments K^T [R | s] of [E | n].  Two token buffers serve in
// turn as Q, K, V and R, as in the second-order kernel.
template <int N, typename T>
__global__ void __launch_bounds__(kCT, blocks_per_sm<N>())
    ahla_chunk_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, T *__restrict__ out,
                      const __grid_constant__ AParams A) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    float *ss = stage + stage_floats<N>(), *dens = ss + kC;
    int c, hd;
    chunk_of(A.P.nch, c, hd);
    const int d = A.d, dv = A.dv, t0 = c * kC, len = min(kC, A.n - t0);
    const long long tok = (long long)hd * A.n + t0;
    const bool carry = c > 0 || A.has_in;
    const float *Pp = A.P.at(hd, c);
    load_tile<N>(b0, q + tok * d, len, d);
    load_tile<N>(b1, k + tok * d, len, d);
    __syncthreads();
    const Tile<N> t;
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);
    Acc<N> acc;
    acc.zero();
    float s = 0.f;
    if (carry) {
        s = row_dot(b0, N + 4, Pp + d * dv, d);
        nn_carry<N, kPlain>(acc, t, b0, Pp, dv, d, dv, stage);
    } else {
        __syncthreads();
    }
    s += row_dot(Wt, kLdW, nullptr, kC);
    if ((threadIdx.x & 1) == 0) ss[threadIdx.x >> 1] = s;
    const bool any_v = sync_unless_finite<N>(load_tile<N>(b0, v + tok * dv, len, dv));
    nn_lower<N>(acc, t, Wt, b0, any_v);
    const float den = row_dot<true>(Wt, kLdW, ss, kC);
    __syncthreads();
    const float seen_r = acc_to_smem<N>(acc, t, b0);  // R
    const int r = threadIdx.x >> 1;
    if ((threadIdx.x & 1) == 0) {
        if (A.direct) dens[r] = den + A.eps;
        else if (r < len) A.den[tok + r] = den;
    }
    const bool any_r = sync_unless_finite<N>(seen_r);
    acc.zero();
    nn_lower<N>(acc, t, Wt, b0, any_r);  // A R
    if (A.direct) {
        if (A.normalized) acc.each([&](float x, int i, int) { return x / dens[t.row(i)]; });
        acc_to_global<N, T>(acc, t, out + tok * dv, len, dv);
    } else {
        acc_to_global<N, float>(acc, t, A.num + tok * dv, len, dv);
    }
    if (c + 1 == A.E.nch && !A.need_E) return;
    float *rec = A.E.at(hd, c);
    atb_to_global<N>(t, rec, b1, b0, d, dv);
    col_sums<N>(rec + d * dv, b1, ss, d);
}

template <int N, typename T>
cudaError_t forward_n(const Fwd2 &p, cudaStream_t s) {
    const ALayout L = make_layout(p.BH, p.n, p.d, p.dv);
    float *ws = reinterpret_cast<float *>(p.ws + kWsHeaderBytes);
    const T *q = static_cast<const T *>(p.q), *k = static_cast<const T *>(p.k), *v = static_cast<const T *>(p.v);
    T *out = static_cast<T *>(p.out);
    const int d = p.d, dv = p.dv, nch = L.nch;
    const long long st_len = 2LL * L.len;
    cudaError_t e;
    AParams A{};
    A.P = {ws + L.oP, L.len, nch};
    A.E = {ws + L.oE, L.len, nch};
    A.num = ws + L.oNum; A.den = ws + L.oDen;
    A.n = p.n; A.d = d; A.dv = dv; A.normalized = p.normalized; A.eps = p.eps;
    A.has_in = p.state_in != nullptr;
    A.need_E = p.state_out != nullptr;
    A.direct = nch == 1 && !p.state_in;
    const bool sums = nch > 1 || p.state_in || p.state_out;
    // state_in and state_out may be the same memory: each value is read by the thread that replaces it
    if (sums) {
        if (nch > 0) {
            SumJobs<T> jobs{};
            jobs.j[0] = {k, v, A.P, d, dv, 1};
            if ((e = launch_sums<N, T>(false, jobs, 1, p.BH, p.n, s))) return e;
        }
        ScanJobs scans{};
        scans.j[0] = {A.P, p.state_in, st_len, p.state_out, st_len, 0};
        if ((e = launch_scan(scans, 1, p.BH, s, nch > 0))) return e;
    }
    if (nch > 0) {
        const int smem = (2 * tile_floats<N>() + kC * kLdW + stage_floats<N>() + 2 * kC) * (int)sizeof(float);
        if ((e = cudaFuncSetAttribute(ahla_chunk_kernel<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)))
            return e;
        if ((e = chain_launch(sums, ahla_chunk_kernel<N, T>, chunk_grid(nch, p.BH), kCT, smem, s, q, k, v, out, A))) return e;
    }
    if (!sums) return cudaSuccess;
    ScanJobs scans{};
    scans.j[0] = {A.E, p.state_in ? p.state_in + L.len : nullptr, st_len,
                  p.state_out ? p.state_out + L.len : nullptr, st_len, 0};
    if ((e = launch_scan(scans, 1, p.BH, s))) return e;
    if (nch == 0 || A.direct) return cudaSuccess;
    const OutParams O{A.E, A.num, A.den, p.n, d, dv, p.normalized, p.eps, A.has_in};
    return launch_out<N, T>(q, out, O, p.BH, s);
}

// ---------------------------------------------------------------------------
// decode step: P' = P + k v^T, m' = m + k, r = q^T P', s = q . m',
// E' = E + k r^T, n' = n + s k, o = q^T E', den = q . n'.  P and E are read and
// written once with 16-byte accesses, consecutive threads on consecutive column
// groups; every thread keeps one column group of the column sums q^T P' (then
// q^T E'), combined across row groups in shared memory.
// ---------------------------------------------------------------------------
// One 512-thread block per SM works through heads (hd = blockIdx.x, + gridDim.x,
// ...), each head's [P | m] and [E | n] staged in shared memory by one 1-D bulk copy each, issued
// a pass or more before use: while the P pass of a head runs, its [E | n] is in flight, and each
// buffer takes the next head's part as soon as its pass has read it.  Updated values go to global
// memory straight from registers.  Every thread waits on the buffer's mbarrier (phase = the block's
// head count), bounded: a copy that never lands ends the block.
constexpr int kStepPThreads = 512;
constexpr unsigned long long kCopyWaitNs = 2000000000ull;

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(sm103::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes),
                   "r"(sm103::smem_u32(bar))
                 : "memory");
}

template <typename T>
__global__ void __launch_bounds__(kStepPThreads, 1)
ahla_step_staged_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, T *__restrict__ out,
                        float *__restrict__ state, int BH, int d, int dv, int normalized, float eps) {
    extern __shared__ float4 dyn[];
    __shared__ float qs[128], ks[128], vs[128], rs[128], part[kStepPThreads][4], red[kStepPThreads / 32];
    __shared__ float s_sc;
    __shared__ uint64_t bar[2];  // [P | m] and tokens; [E | n]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const long long st = 2LL * d * dv + 2 * d;
    const int nP = (d * dv + d) >> 2;  // float4 units of [P | m], of [E | n]
    const int nt_q = d * (int)sizeof(T) / 16, nt_v = dv * (int)sizeof(T) / 16;
    float4 *bP = dyn, *bE = bP + nP, *bT = bE + nP;
    const T *tq = reinterpret_cast<const T *>(bT), *tk = tq + d, *tv = tk + d;
    // thread 0 issues the copies, after a block barrier that ends the generic reads of the buffer
    auto load_P = [&](int hd) {
        if (tid == 0) {
            sm103::fence_async_smem();
            sm103::mbar_arrive_expect_tx(&bar[0], (uint32_t)(16 * (nP + 2 * nt_q + nt_v)));
            bulk_copy(bP, state + hd * st, 16u * nP, &bar[0]);
            bulk_copy(bT, q + (long long)hd * d, 16u * nt_q, &bar[0]);
            bulk_copy(bT + nt_q, k + (long long)hd * d, 16u * nt_q, &bar[0]);
            bulk_copy(bT + 2 * nt_q, v + (long long)hd * dv, 16u * nt_v, &bar[0]);
        }
    };
    auto load_E = [&](int hd) {
        if (tid == 0) {
            sm103::fence_async_smem();
            sm103::mbar_arrive_expect_tx(&bar[1], 16u * nP);
            bulk_copy(bE, state + hd * st + (long long)d * dv + d, 16u * nP, &bar[1]);
        }
    };
    // block sum of one value per thread (all threads call it; ends with a block barrier)
    auto block_sum = [&](float x) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[wid] = x;
        __syncthreads();
        float t = 0.f;
        for (int w = 0; w < kStepPThreads / 32; ++w) t += red[w];
        __syncthreads();
        return t;
    };
    int hd = blockIdx.x;
    if (hd >= BH) return;
    if (tid == 0) {
        sm103::mbar_init(&bar[0], 1);
        sm103::mbar_init(&bar[1], 1);
        sm103::fence_mbar_init();
    }
    __syncthreads();
    load_P(hd);
    load_E(hd);
    const int wv = dv >> 2, n4 = (d * dv) >> 2, c4 = (tid % wv) * 4;  // kStepPThreads is a multiple of wv
    for (uint32_t par = 0; hd < BH; hd += gridDim.x, par ^= 1u) {
        const int nx = hd + gridDim.x;  // this block's next head
        float *P = state + hd * st, *m = P + (long long)d * dv, *E = m + d, *nn = E + (long long)d * dv;
        if (!sm103::mbar_wait(&bar[0], par, kCopyWaitNs)) return;  // [P | m] and tokens of this head
        if (tid < d) {
            qs[tid] = to_f32(tq[tid]);
            ks[tid] = to_f32(tk[tid]);
        }
        if (tid < dv) vs[tid] = to_f32(tv[tid]);
        __syncthreads();
        // ---- [P | m]: P' = P + k v^T, m' = m + k, r = q^T P', s = q . m' ----
        {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            float4 *P4 = reinterpret_cast<float4 *>(P);
            const float v0 = vs[c4], v1 = vs[c4 + 1], v2 = vs[c4 + 2], v3 = vs[c4 + 3];
            for (int f = tid; f < n4; f += kStepPThreads) {
                const int row = f / wv;
                float4 pv = bP[f];
                const float kr = ks[row], qr = qs[row];
                pv.x += kr * v0; pv.y += kr * v1; pv.z += kr * v2; pv.w += kr * v3;
                P4[f] = pv;
                acc.x += qr * pv.x; acc.y += qr * pv.y; acc.z += qr * pv.z; acc.w += qr * pv.w;
            }
            part[tid][0] = acc.x; part[tid][1] = acc.y; part[tid][2] = acc.z; part[tid][3] = acc.w;
            float sm = 0.f;
            if (tid < d) {
                const float mv = reinterpret_cast<const float *>(bP + n4)[tid] + ks[tid];
                m[tid] = mv;
                sm = qs[tid] * mv;
            }
            const float s_tot = block_sum(sm);  // s = q . m' (also: part written, the [P | m] buffer read)
            if (nx < BH) load_P(nx);
            if (tid < dv) {
                const int grp = tid >> 2, comp = tid & 3;
                float a = 0.f;
                for (int g = grp; g < kStepPThreads; g += wv) a += part[g][comp];
                rs[tid] = a;  // r = q^T P'
            }
            if (tid == 0) s_sc = s_tot;
            __syncthreads();
        }
        // ---- [E | n]: E' = E + k r^T, n' = n + s k, o = q^T E', den = q . n' ----
        if (!sm103::mbar_wait(&bar[1], par, kCopyWaitNs)) return;  // [E | n] of this head
        {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            float4 *E4 = reinterpret_cast<float4 *>(E);
            const float r0 = rs[c4], r1 = rs[c4 + 1], r2 = rs[c4 + 2], r3 = rs[c4 + 3];
            for (int f = tid; f < n4; f += kStepPThreads) {
                const int row = f / wv;
                float4 e = bE[f];
                const float kr = ks[row], qr = qs[row];
                e.x += kr * r0; e.y += kr * r1; e.z += kr * r2; e.w += kr * r3;
                E4[f] = e;
                acc.x += qr * e.x; acc.y += qr * e.y; acc.z += qr * e.z; acc.w += qr * e.w;
            }
            part[tid][0] = acc.x; part[tid][1] = acc.y; part[tid][2] = acc.z; part[tid][3] = acc.w;
            float sn = 0.f;
            if (tid < d) {
                const float nv = reinterpret_cast<const float *>(bE + n4)[tid] + s_sc * ks[tid];
                nn[tid] = nv;
                sn = qs[tid] * nv;
            }
            const float den = block_sum(sn);  // den = q . n' (also: part written, the [E | n] buffer read)
            if (nx < BH) load_E(nx);
            if (tid < dv) {
                const int grp = tid >> 2, comp = tid & 3;
                float a = 0.f;
                for (int g = grp; g < kStepPThreads; g += wv) a += part[g][comp];
                from_f32(&out[(long long)hd * dv + tid], normalized ? a / (den + eps) : a);
            }
            __syncthreads();  // qs, ks, vs, rs, part, s_sc read before the next head rewrites them
        }
    }
}

// The step with every load issued at once, straight to registers, by `split` blocks per head, block r
// with columns [r dv / split, ...) of P and E.  From the old values, r = q^T P + (q.k) v and
// o = q^T E + (q.k) r, column by column, so one pass does the step: both column sums, then both updated
// slices.  Only m, n and the tokens are shared.  The plain output needs m and n in block 0 alone; for the
// normalised output, and where `out` lies over the tokens, the blocks of a head form a cluster and meet in a
// split barrier between their last read of these and the first write.  Measured, us a step (staged -> this), bf16 tokens: 64 x 64, 16 heads 3.7 -> 2.8,
// 256 heads 6.1 -> 4.0, 2048 heads 35.6 -> 23.4 (140 MB read and written: 5.9 TB/s); 128 x 128, 32
// heads 5.7 -> 3.3, 2048 heads as fast (90.3 us a step over 541 MB of states).  Bound by the latency of
// one load and two barriers for few heads, by HBM for many.
constexpr int kSplitThreads = 256, kSplitWarps = kSplitThreads / 32;
template <typename T, int NC>
__global__ void __launch_bounds__(kSplitThreads)
ahla_step_split_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, T *__restrict__ out,
                       float *state, int split, int d, int dv, int normalized, float eps) {
    // qs[d] is zero: it stands for the rows beyond a slice (an infinite entry would make NaN of their zeros)
    __shared__ __align__(16) float qs[132], ks[128], vs[128];
    __shared__ __align__(16) float part[2][kSplitWarps][64];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int hd = blockIdx.x / split, rank = blockIdx.x % split, cw = dv / split, col0 = rank * cw;
    const long long len = (long long)d * dv + d;
    float *P = state + hd * 2 * len, *m = P + (long long)d * dv, *E = P + len, *nn = E + (long long)d * dv;
    const int wC = cw >> 2, nC = d * wC, c4 = (tid % wC) * 4, r0 = tid / wC, rstep = kSplitThreads / wC;
    float4 pv[NC], ev[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const long long at = (long long)(r0 + i * rstep) * dv + col0 + c4;
        pv[i] = ev[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tid + i * kSplitThreads < nC) {
            pv[i] = *reinterpret_cast<const float4 *>(P + at);
            ev[i] = *reinterpret_cast<const float4 *>(E + at);
        }
    }
    const bool sums = normalized || rank == 0;  // m and n: four values a lane, in every warp
    float mv[4], nv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = lane + 32 * i;
        mv[i] = sums && a < d ? m[a] : 0.f;
        nv[i] = sums && a < d ? nn[a] : 0.f;
    }
    if (tid < d) {
        qs[tid] = to_f32(q[(long long)hd * d + tid]);
        ks[tid] = to_f32(k[(long long)hd * d + tid]);
    }
    if (tid < dv) vs[tid] = to_f32(v[(long long)hd * dv + tid]);
    if (tid == 0) qs[d] = 0.f;
    __syncthreads();
    const float qk = warp_dot(qs, ks, d);
    float qm = 0.f, qn = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = lane + 32 * i;
        if (a < d) {
            qm = fmaf(qs[a], mv[i], qm);
            qn = fmaf(qs[a], nv[i], qn);
        }
    }
    const float s = group_sum<32>(qm) + qk;        // q . m'
    const float den = group_sum<32>(qn) + s * qk;  // q . n'
    float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const float qr = qs[min(r0 + i * rstep, d)];
        fma4(a0, qr, pv[i]);
        fma4(a1, qr, ev[i]);
    }
    a0 = column_sum(a0, wC);
    a1 = column_sum(a1, wC);
    if (lane < wC) {
        *reinterpret_cast<float4 *>(&part[0][wid][c4]) = a0;
        *reinterpret_cast<float4 *>(&part[1][wid][c4]) = a1;
    }
    cluster_arrive();  // this block has read m, n and the tokens
    __syncthreads();
    const float4 v4 = *reinterpret_cast<const float4 *>(vs + col0 + c4);
    float4 r4 = make_float4(qk * v4.x, qk * v4.y, qk * v4.z, qk * v4.w);
#pragma unroll
    for (int w = 0; w < kSplitWarps; ++w) fma4(r4, 1.f, *reinterpret_cast<const float4 *>(&part[0][w][c4]));
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const int row = r0 + i * rstep;
        const long long at = (long long)row * dv + col0 + c4;
        if (tid + i * kSplitThreads < nC) {
            *reinterpret_cast<float4 *>(P + at) = axpy4(pv[i], ks[row], v4);
            *reinterpret_cast<float4 *>(E + at) = axpy4(ev[i], ks[row], r4);
        }
    }
    float4 o = make_float4(qk * r4.x, qk * r4.y, qk * r4.z, qk * r4.w);
    if (tid < wC) {
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) fma4(o, 1.f, *reinterpret_cast<const float4 *>(&part[1][w][c4]));
    }
    cluster_wait();  // every block of the head has read m, n and the tokens
    if (tid < wC) {
        const float x[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            from_f32(&out[(long long)hd * dv + col0 + c4 + j], normalized ? x[j] / (den + eps) : x[j]);
    }
    if (rank == 0 && wid == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int a = lane + 32 * i;
            if (a >= d) continue;
            m[a] = mv[i] + ks[a];
            nn[a] = nv[i] + s * ks[a];
        }
    }
}

// Blocks per head of the kernel above, 0 where the staged kernel serves: the line lies where the staged kernel,
// whose copies of the next head run during this one, is as fast (measured at 24 to 5000 heads, us, staged / this).
// Head sizes up to 64: two for few heads (16 heads 3.1 -> 2.8 us), one from 128 heads (3.2 against 3.3).
// With a size of 128, four up to 64 heads (64 of 128 x 128 5.6 / 4.2); of small d, normalised, two (64 of 16 x 128
// 3.47 / 3.63 by four, 3.38 by two).  More heads, plain (clusters cost more to launch: the normalised output takes
// them up to 64 heads), two: with the other size up to 32 always (5000 of 32 x 128 73 / 66); with 64 up to 1250 heads
// (1250 29.3 / 24.8, 1500 33.9 / 36.8, 5000 108 / 121); 128 x 128 while two blocks a head are one round or so (175
// 10.0 / 9.4, 200 10.0 / 10.3, 600 18.9 / 21.2, 1500 65.8 / 66.2) and from 2000 (2000 85.6 / 85.4, 5000 210 / 202).
// A block's slice has 8 to 64 columns.
int ahla_step_split(int BH, int d, int dv, int normalized) {
    int s;
    if (d != 128 && dv != 128) s = BH <= 64 ? 2 : 1;
    else if (BH <= 64) s = normalized && d <= 32 ? 2 : 4;
    else if (normalized) s = 0;
    else if (d * dv <= 32 * 128) s = 2;
    else if (d * dv <= 64 * 128) s = BH <= 1250 ? 2 : 0;
    else s = BH <= 180 || BH >= 2000 ? 2 : 0;
    if (s == 0) return 0;
    while (s > 1 && dv / s < 8) s /= 2;
    while (dv / s > 64) s *= 2;
    return s;
}

template <typename T>
cudaError_t ahla_step_split_launch(const void *q, const void *k, const void *v, void *out, float *state, int BH,
                                   int split, int d, int dv, int normalized, float eps, cudaStream_t s) {
    const size_t nq = sizeof(T) * (size_t)BH * d, nv = sizeof(T) * (size_t)BH * dv;
    const bool over = memory_meets(out, nv, q, nq) || memory_meets(out, nv, k, nq) || memory_meets(out, nv, v, nv);
    auto go = [&](auto kern) {
        return launch_blocks(kern, BH, split, normalized || over, kSplitThreads, s, static_cast<const T *>(q), static_cast<const T *>(k),
                            static_cast<const T *>(v), static_cast<T *>(out), state, split, d, dv, normalized, eps);
    };
    const int nc = (d * (dv / split) / 4 + kSplitThreads - 1) / kSplitThreads;
    if (nc <= 1) return go(ahla_step_split_kernel<T, 1>);
    if (nc <= 2) return go(ahla_step_split_kernel<T, 2>);
    if (nc <= 4) return go(ahla_step_split_kernel<T, 4>);
    return go(ahla_step_split_kernel<T, 8>);
}

}  // namespace

size_t ahla_workspace_bytes_internal(int BH, int n, int d, int dv, int) {
    if (n == 0) return kWsHeaderBytes;  // the states are copied, no record is used
    return kWsHeaderBytes + sizeof(float) * (size_t)make_layout(BH, n, d, dv).total;
}

cudaError_t ahla_forward_launch(const Fwd2 &p, cudaStream_t stream) {
    if (ahla_tc_applicable(p)) return ahla_tc_forward(p, stream);
    return with_padded_size(p.d, p.dv, [&](auto size) {
        constexpr int N = decltype(size)::value;
        return p.dt == HLA_BF16 ? forward_n<N, __nv_bfloat16>(p, stream) : forward_n<N, float>(p, stream);
    });
}

cudaError_t ahla_step_launch(const void *q, const void *k, const void *v, void *out, hla_dtype dt, int BH, int d,
                             int dv, int normalized, float eps, float *state, cudaStream_t stream) {
    if (BH == 0) return cudaSuccess;
    // the staged kernel copies whole 16-byte units (token rows, [P | m], [E | n], the head stride):
    // the entry point checks the 16-byte alignment of q, k, v and the state, and d, dv in
    // {16, 32, 64, 128} make every row a multiple of 16 bytes
    const size_t tsz = dt == HLA_BF16 ? 2 : 4;
    if ((d * tsz) % 16 != 0 || (dv * tsz) % 16 != 0 || d % 4 != 0 || dv % 4 != 0 || d > 128 || dv > 128)
        return cudaErrorInvalidValue;
    if (const int split = ahla_step_split(BH, d, dv, normalized))
        return dt == HLA_BF16
                   ? ahla_step_split_launch<__nv_bfloat16>(q, k, v, out, state, BH, split, d, dv, normalized, eps, stream)
                   : ahla_step_split_launch<float>(q, k, v, out, state, BH, split, d, dv, normalized, eps, stream);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = BH < sms ? BH : sms;
    const size_t smem = 2 * 16 * (size_t)((d * dv + d) / 4) + tsz * (2 * (size_t)d + dv);
    cudaError_t e;
    if (dt == HLA_BF16) {
        if ((e = cudaFuncSetAttribute(ahla_step_staged_kernel<__nv_bfloat16>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
            return e;
        ahla_step_staged_kernel<__nv_bfloat16><<<grid, kStepPThreads, smem, stream>>>(
            static_cast<const __nv_bfloat16 *>(q), static_cast<const __nv_bfloat16 *>(k),
            static_cast<const __nv_bfloat16 *>(v), static_cast<__nv_bfloat16 *>(out), state, BH, d, dv, normalized, eps);
    } else {
        if ((e = cudaFuncSetAttribute(ahla_step_staged_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem)))
            return e;
        ahla_step_staged_kernel<float><<<grid, kStepPThreads, smem, stream>>>(
            static_cast<const float *>(q), static_cast<const float *>(k), static_cast<const float *>(v),
            static_cast<float *>(out), state, BH, d, dv, normalized, eps);
    }
    return cudaGetLastError();
}

}  // namespace hla
