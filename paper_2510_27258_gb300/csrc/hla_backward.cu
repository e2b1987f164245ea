// Gradients of masked second-order HLA: a reverse chunk scan with the forward
// states checkpointed at chunk boundaries (Sec. "Chunk-parallel training via
// associative scans": the adjoint of the semidirect product applied by a
// reverse scan), in fp32 on the CUDA cores.
//
// With x_j = S_j q_j, T_tj = q_t . x_j and L = sum_t g_t . o_t, the forward is
// o_t = sum_{j<=t} T_tj v_j (proof of Theorem 1), so with P_tj = g_t . v_j:
//   dv_j = sum_{t>=j} T_tj g_t,   y_j = sum_{t>=j} P_tj q_t,
//   dq_t = sum_{j<=t} P_tj x_j + S_t y_t,
//   dk_i = sum_{j>=i} [ (q_j . k_i) y_j + (y_j . k_i) q_j ].
// The ratio-normalised output o = num / (den + eps) is the same computation
// with values [v | 1] (den is the extra column) and upstream gradient
// [g' | u] = [g / (den + eps) | -(g . o) / (den + eps)]; the plain output has
// g' = g, u = 0 and skips the extra column.
//
// Per 64-token chunk (rows = its tokens; p = sum before the chunk, s = sum after):
//   forward:  W = L . (Q K^T),  X = W K + Q S_p,  T = L . (Q X^T),
//             num = T V + Q D_p,  den = T 1 + Q e_p,
//   backward: P = L . (G' V^T + u 1^T),  Y = P^T Q + V Gam_s + 1 h_s^T,
//             dV = T^T G' + X Gam_s^T,   B = L . (Y K^T),
//             dQ = P X + G' D_p^T + u e_p^T + Y S_p + B K,
//             dK = K (Lam_s + Lam_s^T) + W^T Y + B^T Q.
// Every carry is a plain sum over the chunks: before the chunk S += K^T K,
// D += X^T V, e += X^T 1; after it Gam^T += Q^T G', h += Q^T u, Lam += Q^T Y.
// X is formed with the chunk's own S_p and Y with its own Gam_s, which is where
// the cross terms of the semidirect product and of its adjoint go, so no carry
// is multiplied along the sequence.  Launches (normalised; the plain output
// has Gam's increments in the first and needs no third pair):
//   K^T K | sums of S | X, D, e, num, den | sums of D, e | G', u, Gam, h |
//   sums of Gam, h from the end | Y, Lam | sums of Lam from the end | dQ, dK, dV.
//
// At B2 H16 n4096 d128 normalised the two scans that multiplied carries took 24
// of 36.6 ms; as elementwise sums, with the register-tiled products of
// chunk_simt.cuh, the call takes 2.0 ms.
#include <algorithm>

#include "chunk_simt.cuh"

namespace hla {
namespace {

inline long long up16(long long x) { return (x + 15) / 16 * 16; }

struct BLayout {
    int nch;
    // floats from the scratch start: S | D, e | Gam^T, h | Lam records; X, Y ([BH][n][d]); num, then G'
    // ([BH][n][dv]); den, then u ([BH][n])
    long long oS, oD, oG, oL, oX, oY, oNum, oDen, total;
};

BLayout make_layout(int BH, int n, int d, int dv) {
    BLayout L;
    L.nch = (n + kC - 1) / kC;
    const long long recs = (long long)BH * (L.nch + 1), tok = (long long)BH * n;
    long long o = 0;
    L.oS = o; o += recs * d * d;
    L.oD = o; o += recs * (d * dv + d);
    L.oG = o; o += recs * (d * dv + d);
    L.oL = o; o += recs * d * d;
    L.oX = o; o += up16(tok * d);
    L.oY = o; o += up16(tok * d);
    L.oNum = o; o += up16(tok * dv);
    L.oDen = o; o += up16(tok);
    L.total = o;
    return L;
}

template <typename T>
struct BParams {
    const T *q, *k, *v, *g;
    T *dq, *dk, *dv_out;
    Records S, D, Gam, Lam;
    float *X, *Y, *num, *den;  // num, den become G', u
    WsHeader *err;
    int n, d, dv, normalized;
    float eps;
};

// the chunk of this block
template <typename T>
struct Chunk {
    int c, hd, len;
    long long tok;
    bool before, after;  // chunks before / after it
    __device__ Chunk(const BParams<T> &P) {
        chunk_of(P.S.nch, c, hd);
        len = min(kC, P.n - c * kC);
        tok = (long long)hd * P.n + c * kC;
        before = c > 0;
        after = c + 1 < P.S.nch;
    }
};

// G' rows of a chunk (the output gradient itself for the plain output) and u
template <int N, typename T>
__device__ __forceinline__ float load_upstream(float *dst, float *us, const BParams<T> &P, const Chunk<T> &ch) {
    if (!P.normalized) return load_tile<N>(dst, P.g + ch.tok * P.dv, ch.len, P.dv);
    if (us && threadIdx.x < kC) us[threadIdx.x] = threadIdx.x < ch.len ? P.den[ch.tok + threadIdx.x] : 0.f;
    return load_tile<N>(dst, P.num + ch.tok * P.dv, ch.len, P.dv);
}

// ---------------------------------------------------------------------------
// X, the increments X^T V, X^T 1 of D and e; normalised: T V and T 1
// ---------------------------------------------------------------------------
template <int N, typename T>
__global__ void __launch_bounds__(kCT, blocks_per_sm<N>()) bwd_x_kernel(const __grid_constant__ BParams<T> P) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    // no wait of this call can fail: hla_poll_error finds no error (a memset of its own took 2 us)
    if (blockIdx.x == 0 && threadIdx.x == 0) *P.err = WsHeader{};
    const Chunk<T> ch(P);
    const int d = P.d, dv = P.dv;
    load_tile<N>(b0, P.q + ch.tok * d, ch.len, d);
    const bool any_k = sync_unless_finite<N>(load_tile<N>(b1, P.k + ch.tok * d, ch.len, d));
    const Tile<N> t;
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);
    Acc<N> acc;
    acc.zero();
    if (ch.before) nn_carry<N, kPlain>(acc, t, b0, P.S.at(ch.hd, ch.c), d, d, d, stage);
    else __syncthreads();
    nn_lower<N>(acc, t, Wt, b1, any_k);
    acc_to_global<N, float>(acc, t, P.X + ch.tok * d, ch.len, d);
    __syncthreads();
    acc_to_smem<N>(acc, t, b1);  // X
    __syncthreads();
    if (P.normalized) {
        nt_masked(Wt, b0, b1, N + 4, d, nullptr);  // T
        __syncthreads();
    }
    const bool any_v = sync_unless_finite<N>(load_tile<N>(b0, P.v + ch.tok * dv, ch.len, dv));
    if (P.normalized) {
        const float den = row_dot(Wt, kLdW, nullptr, kC);
        const int r = threadIdx.x >> 1;
        if ((threadIdx.x & 1) == 0 && r < ch.len) P.den[ch.tok + r] = den;
        acc.zero();
        nn_lower<N>(acc, t, Wt, b0, any_v);
        acc_to_global<N, float>(acc, t, P.num + ch.tok * dv, ch.len, dv);
    }
    if (!ch.after) return;
    float *rec = P.D.at(ch.hd, ch.c);
    atb_to_global<N>(t, rec, b1, b0, d, dv);
    col_sums<N>(rec + d * dv, b1, nullptr, d);
}

// ---------------------------------------------------------------------------
// normalised: num and den of the whole prefix, G' and u in their place, and the increments Q^T G',
// Q^T u of Gam^T and h
// ---------------------------------------------------------------------------
template <int N, typename T>
__global__ void __launch_bounds__(kCT, blocks_per_sm<N>()) bwd_upstream_kernel(const __grid_constant__ BParams<T> P) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *stage = b1 + tile_floats<N>(), *us = stage + stage_floats<N>();
    const Chunk<T> ch(P);
    const int d = P.d, dv = P.dv;
    load_tile<N>(b0, P.q + ch.tok * d, ch.len, d);
    __syncthreads();
    const Tile<N> t;
    Acc<N> acc;
    acc.zero();
    float den = 0.f;
    if (ch.before) {
        const float *Dp = P.D.at(ch.hd, ch.c);
        den = row_dot(b0, N + 4, Dp + d * dv, d);
        nn_carry<N, kPlain>(acc, t, b0, Dp, dv, d, dv, stage);
    }
    acc_to_smem<N>(acc, t, b1);  // Q D_p
    __syncthreads();
    // two threads a row, each with every other group of four columns
    const int r = threadIdx.x >> 1, h = threadIdx.x & 1;
    const bool ok = r < ch.len;
    const float inv = ok ? 1.f / (P.den[ch.tok + r] + den + P.eps) : 0.f;
    float *num = P.num + (ch.tok + r) * dv, *row = b1 + r * (N + 4);
    const T *g = P.g + (ch.tok + r) * dv;
    float go = 0.f;
    for (int c = 4 * h; c < N; c += 8) {
        float gp[4] = {0.f, 0.f, 0.f, 0.f};
        if (ok && c < dv) {
            const float4 x = *reinterpret_cast<const float4 *>(num + c), y = *reinterpret_cast<const float4 *>(row + c);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                gp[u] = to_f32(g[c + u]) * inv;
                go = fmaf(gp[u], f4(x, u) + f4(y, u), go);  // g . o
            }
            *reinterpret_cast<float4 *>(num + c) = make_float4(gp[0], gp[1], gp[2], gp[3]);
        }
        *reinterpret_cast<float4 *>(row + c) = make_float4(gp[0], gp[1], gp[2], gp[3]);
    }
    go += __shfl_xor_sync(0xffffffffu, go, 1);
    if (h == 0) {
        us[r] = -go * inv;
        if (ok) P.den[ch.tok + r] = -go * inv;
    }
    __syncthreads();
    if (!ch.before) return;
    float *rec = P.Gam.at(ch.hd, ch.c);
    atb_to_global<N>(t, rec, b0, b1, d, dv);
    col_sums<N>(rec + d * dv, b0, us, d);
}

// ---------------------------------------------------------------------------
// Y and the increments Q^T Y of Lam
// ---------------------------------------------------------------------------
template <int N, typename T>
__global__ void __launch_bounds__(kCT, blocks_per_sm<N>()) bwd_y_kernel(const __grid_constant__ BParams<T> P) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    float *us = stage + stage_floats<N>();
    const Chunk<T> ch(P);
    const int d = P.d, dv = P.dv;
    load_upstream<N>(b0, us, P, ch);
    load_tile<N>(b1, P.v + ch.tok * dv, ch.len, dv);
    __syncthreads();
    const Tile<N> t;
    nt_masked(Wt, b0, b1, N + 4, dv, P.normalized ? us : nullptr);  // P
    Acc<N> acc;
    acc.zero();
    if (ch.after) {
        const float *Gs = P.Gam.at(ch.hd, ch.c);
        nn_carry<N, kTransposed>(acc, t, b1, Gs, dv, dv, d, stage);  // V Gam_s
        if (P.normalized)
            acc.each([&](float x, int, int j) { return x + (t.col(j) < d ? Gs[d * dv + t.col(j)] : 0.f); });
    } else {
        __syncthreads();
    }
    const bool any_q = sync_unless_finite<N>(load_tile<N>(b1, P.q + ch.tok * d, ch.len, d));
    tn_lower<N>(acc, t, Wt, b1, any_q);  // P^T Q
    acc_to_global<N, float>(acc, t, P.Y + ch.tok * d, ch.len, d);
    if (!ch.before) return;
    acc_to_smem<N>(acc, t, b0);  // Y; its rows beyond the sequence meet zero rows of Q
    __syncthreads();
    atb_to_global<N>(t, P.Lam.at(ch.hd, ch.c), b1, b0, d, d);
}

// ---------------------------------------------------------------------------
// the gradients
// ---------------------------------------------------------------------------
// dQ
template <int N, typename T>
__device__ __forceinline__ void grad_q(Acc<N> &acc, const Tile<N> &t, float *sm, const BParams<T> &P, const Chunk<T> &ch) {
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    float *us = stage + stage_floats<N>();
    const int d = P.d, dv = P.dv;
    load_upstream<N>(b0, us, P, ch);
    load_tile<N>(b1, P.v + ch.tok * dv, ch.len, dv);
    __syncthreads();
    nt_masked(Wt, b0, b1, N + 4, dv, P.normalized ? us : nullptr);  // P
    if (ch.before) {
        const float *Dp = P.D.at(ch.hd, ch.c);
        nn_carry<N, kTransposed>(acc, t, b0, Dp, dv, dv, d, stage);  // G' D_p^T
        if (P.normalized)
            acc.each([&](float x, int i, int j) {
                return t.col(j) < d ? fmaf(us[t.row(i)], Dp[d * dv + t.col(j)], x) : x;
            });
    } else {
        __syncthreads();
    }
    const bool any_x = sync_unless_finite<N>(load_tile<N>(b1, P.X + ch.tok * d, ch.len, d));
    nn_lower<N>(acc, t, Wt, b1, any_x);  // P X
    __syncthreads();
    load_tile<N>(b0, P.Y + ch.tok * d, ch.len, d);
    const bool any_k = sync_unless_finite<N>(load_tile<N>(b1, P.k + ch.tok * d, ch.len, d));
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);  // B
    if (ch.before) nn_carry<N, kPlain>(acc, t, b0, P.S.at(ch.hd, ch.c), d, d, d, stage);  // Y S_p
    else __syncthreads();
    nn_lower<N>(acc, t, Wt, b1, any_k);  // B K
}

// dK
template <int N, typename T>
__device__ __forceinline__ void grad_k(Acc<N> &acc, const Tile<N> &t, float *sm, const BParams<T> &P, const Chunk<T> &ch) {
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    const int d = P.d;
    load_tile<N>(b0, P.Y + ch.tok * d, ch.len, d);
    load_tile<N>(b1, P.k + ch.tok * d, ch.len, d);
    __syncthreads();
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);  // B
    if (ch.after) nn_carry<N, kSymmetric>(acc, t, b1, P.Lam.at(ch.hd, ch.c), d, d, d, stage);
    else __syncthreads();
    const bool any_q = sync_unless_finite<N>(load_tile<N>(b0, P.q + ch.tok * d, ch.len, d));
    tn_lower<N>(acc, t, Wt, b0, any_q);  // B^T Q
    __syncthreads();
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);  // W
    __syncthreads();
    const bool any_y = sync_unless_finite<N>(load_tile<N>(b1, P.Y + ch.tok * d, ch.len, d));
    tn_lower<N>(acc, t, Wt, b1, any_y);  // W^T Y
}

// dV
template <int N, typename T>
__device__ __forceinline__ void grad_v(Acc<N> &acc, const Tile<N> &t, float *sm, const BParams<T> &P, const Chunk<T> &ch) {
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    const int d = P.d, dv = P.dv;
    load_tile<N>(b0, P.q + ch.tok * d, ch.len, d);
    load_tile<N>(b1, P.X + ch.tok * d, ch.len, d);
    __syncthreads();
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);  // T
    if (ch.after) nn_carry<N, kPlain>(acc, t, b1, P.Gam.at(ch.hd, ch.c), dv, d, dv, stage);  // X Gam_s^T
    else __syncthreads();
    const bool any_g = sync_unless_finite<N>(load_upstream<N>(b0, static_cast<float *>(nullptr), P, ch));
    tn_lower<N>(acc, t, Wt, b0, any_g);  // T^T G'
}

// blockIdx.z 0 dQ, 1 dK, 2 dV; kOver, where an output lies over the tokens: one block forms all three of a chunk,
// whose tokens no other block reads any more, before it writes any
template <int N, typename T, bool kOver>
__global__ void __launch_bounds__(kCT, blocks_per_sm<N>()) bwd_grad_kernel(const __grid_constant__ BParams<T> P) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    const Chunk<T> ch(P);
    const int d = P.d, dv = P.dv;
    const Tile<N> t;
    Acc<N> acc;
    acc.zero();
    if constexpr (kOver) {
        Acc<N> acc_k, acc_v;
        acc_k.zero();
        acc_v.zero();
        grad_q<N>(acc, t, sm, P, ch);
        __syncthreads();
        grad_k<N>(acc_k, t, sm, P, ch);
        __syncthreads();
        grad_v<N>(acc_v, t, sm, P, ch);
        __syncthreads();
        acc_to_global<N, T>(acc, t, P.dq + ch.tok * d, ch.len, d);
        acc_to_global<N, T>(acc_k, t, P.dk + ch.tok * d, ch.len, d);
        acc_to_global<N, T>(acc_v, t, P.dv_out + ch.tok * dv, ch.len, dv);
    } else if (blockIdx.z == 0) {
        grad_q<N>(acc, t, sm, P, ch);
        acc_to_global<N, T>(acc, t, P.dq + ch.tok * d, ch.len, d);
    } else if (blockIdx.z == 1) {
        grad_k<N>(acc, t, sm, P, ch);
        acc_to_global<N, T>(acc, t, P.dk + ch.tok * d, ch.len, d);
    } else {
        grad_v<N>(acc, t, sm, P, ch);
        acc_to_global<N, T>(acc, t, P.dv_out + ch.tok * dv, ch.len, dv);
    }
}

template <int N, typename T>
cudaError_t backward_n(const Bwd2 &p, cudaStream_t s) {
    const BLayout L = make_layout(p.BH, p.n, p.d, p.dv);
    float *ws = reinterpret_cast<float *>(p.ws + kWsHeaderBytes);
    const int d = p.d, dv = p.dv, nch = L.nch;
    if (nch == 0) return cudaSuccess;
    BParams<T> P{};
    P.q = static_cast<const T *>(p.q); P.k = static_cast<const T *>(p.k); P.v = static_cast<const T *>(p.v);
    P.g = static_cast<const T *>(p.dout);
    P.dq = static_cast<T *>(p.dq); P.dk = static_cast<T *>(p.dk); P.dv_out = static_cast<T *>(p.dval);
    P.S = {ws + L.oS, d * d, nch};
    P.D = {ws + L.oD, d * dv + d, nch};
    P.Gam = {ws + L.oG, d * dv + (p.normalized ? d : 0), nch};
    P.Lam = {ws + L.oL, d * d, nch};
    P.X = ws + L.oX; P.Y = ws + L.oY; P.num = ws + L.oNum; P.den = ws + L.oDen;
    P.err = reinterpret_cast<WsHeader *>(p.ws);
    P.n = p.n; P.d = d; P.dv = dv; P.normalized = p.normalized; P.eps = p.eps;
    const dim3 grid = chunk_grid(nch, p.BH);
    const int smem = (2 * tile_floats<N>() + kC * kLdW + stage_floats<N>() + kC) * (int)sizeof(float);
    cudaError_t e;
    bool follows = false;  // a launch of this call came before
    auto launch = [&](auto kern, dim3 gr) -> cudaError_t {
        cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (err) return err;
        err = chain_launch(follows, kern, gr, kCT, smem, s, P);
        follows = true;
        return err;
    };
    const bool many = nch > 1;
    const ScanJob none{};
    auto scan = [&](const Records &a, int rev_a, const Records *b) -> cudaError_t {
        ScanJobs jobs{};
        jobs.j[0] = none; jobs.j[0].r = a; jobs.j[0].reverse = rev_a;
        if (b) { jobs.j[1].r = *b; jobs.j[1].reverse = 1; }
        return launch_scan(jobs, b ? 2 : 1, p.BH, s);
    };
    if (many) {
        SumJobs<T> jobs{};
        jobs.j[0] = {P.k, P.k, P.S, d, d, 0};
        jobs.j[1] = {P.q, P.g, P.Gam, d, dv, 0};  // Gam^T of the plain output
        if ((e = launch_sums<N, T>(false, jobs, p.normalized ? 1 : 2, p.BH, p.n, s))) return e;
        follows = true;
        if ((e = scan(P.S, 0, p.normalized ? nullptr : &P.Gam))) return e;
    }
    if ((e = launch(bwd_x_kernel<N, T>, grid))) return e;
    if (many && (e = scan(P.D, 0, nullptr))) return e;
    if (p.normalized) {
        if ((e = launch(bwd_upstream_kernel<N, T>, grid))) return e;
        if (many && (e = scan(P.Gam, 1, nullptr))) return e;
    }
    if ((e = launch(bwd_y_kernel<N, T>, grid))) return e;
    if (many && (e = scan(P.Lam, 1, nullptr))) return e;
    const size_t nd = sizeof(T) * (size_t)p.BH * p.n * d, nv = sizeof(T) * (size_t)p.BH * p.n * dv;
    if (backward2_over_tokens(p, p.q, nd) || backward2_over_tokens(p, p.k, nd) || backward2_over_tokens(p, p.v, nv) ||
        backward2_over_tokens(p, p.dout, nv))
        return launch(bwd_grad_kernel<N, T, true>, grid);
    return launch(bwd_grad_kernel<N, T, false>, chunk_grid(nch, p.BH, 3));
}

}  // namespace

size_t backward2_workspace_bytes(int BH, int n, int d, int dv, int) {
    if (n == 0) return kWsHeaderBytes;
    const size_t simt = kWsHeaderBytes + sizeof(float) * (size_t)make_layout(BH, n, d, dv).total;
    const size_t tc = backward2_tc_workspace_bytes(BH, n), tiles = backward2_tiles_workspace_bytes(BH, n, d, dv);
    return std::max(simt, std::max(tc, tiles));
}

bool backward2_over_tokens(const Bwd2 &p, const void *tokens, size_t bytes) {
    const size_t row = p.dt == HLA_BF16 ? 2 : 4, tok = (size_t)p.BH * p.n;
    return memory_meets(tokens, bytes, p.dq, tok * p.d * row) || memory_meets(tokens, bytes, p.dk, tok * p.d * row) ||
           memory_meets(tokens, bytes, p.dval, tok * p.dv * row);
}

cudaError_t backward2_launch(const Bwd2 &p, cudaStream_t stream) {
    if (backward2_tc_applicable(p)) return backward2_tc_launch(p, stream);
    if (backward2_tiles_applicable(p)) return backward2_tiles_launch(p, stream);
    return with_padded_size(p.d, p.dv, [&](auto size) {
        constexpr int N = decltype(size)::value;
        return p.dt == HLA_BF16 ? backward_n<N, __nv_bfloat16>(p, stream) : backward_n<N, float>(p, stream);
    });
}

}  // namespace hla
