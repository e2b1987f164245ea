// Generic second-order HLA forward: fp32 CUDA-core kernels for every supported
// shape (d, dv in {16,32,64,128}, any length, masked/unmasked, normalised or
// not, fp32 or bf16 tokens, optional states).
//
// Formulation (per head; rows are tokens of one 64-token chunk, "p" = prefix
// before the chunk).  With x_t = S_t q_t (S symmetric), masked second order is a
// causal linear attention with query q and key x (proof of Theorem 1: num_t =
// q_t^T sum_{j<=t} S_j q_j v_j^T), and the unmasked form is o_t = x_t^T C_t:
//   W = L . (Q K^T)  (L lower triangular incl. diagonal),   X = W K + Q S_p
//   masked:   T = L . (Q X^T),  num = T V + Q D_p,  den = T 1 + Q e_p
//   unmasked: T = L . (X Q^T),  num = T V + X C_p,  den = T 1 + X m_p
// Every carry is a plain prefix sum of what the chunks add: S += K^T K,
// C += Q^T V, m += Q^T 1, and, once X is formed with the chunk's own S_p,
// D += X^T V, e += X^T 1 (D = S C - G, e = S m - h).  So no carry is multiplied
// along the sequence: the cross term S_A C_B of Eq. semidirect is in X, and
// everything but the sums runs over all chunks at once.  Launches (masked):
// K^T K of every chunk; its prefix sums; X, D's increments and T V; D's prefix
// sums; outputs.  One chunk without states is the third launch alone; one chunk of small heads
// with states, and a few tokens without, are one block a head (g2_one_kernel).
//
// The chain of products S_p C_c over the chunks that the sums replace took 20 %
// of a call and ran on a few blocks, the chunk kernels had one multiply-add per
// shared-memory load: B2 H16 n1000 d64 fp32 1975 us, now 71 us.
#include <algorithm>

#include "chunk_simt.cuh"
#include "state_products.cuh"

namespace hla {
namespace {

inline long long up16(long long x) { return (x + 15) / 16 * 16; }

struct GLayout {
    int BH, n, d, dv, nch, lenS, lenC, lenD;
    // floats from the scratch start: S | C, m | D, e records, T V (fp32 [BH][n][dv]), T 1 ([BH][n]), a copy of
    // state_in (used when state_out overlaps it)
    long long oS, oC, oD, oNum, oDen, oStage, total;
};

long long state_floats(int d, int dv) { return (long long)d * d + 2LL * d * dv + 2LL * d; }

GLayout make_layout(int BH, int n, int d, int dv) {
    GLayout L;
    L.BH = BH; L.n = n; L.d = d; L.dv = dv;
    L.nch = (n + kC - 1) / kC;
    L.lenS = d * d;
    L.lenC = L.lenD = d * dv + d;
    const long long recs = (long long)BH * (L.nch + 1);
    long long o = 0;
    L.oS = o; o += recs * L.lenS;
    L.oC = o; o += recs * L.lenC;
    L.oD = o; o += recs * L.lenD;
    L.oNum = o; o += up16((long long)BH * n * dv);
    L.oDen = o; o += up16((long long)BH * n);
    L.oStage = o; o += up16((long long)BH * state_floats(d, dv));
    L.total = o;
    return L;
}

struct GParams {
    Records S, C, D;
    float *num, *den;
    int n, d, dv, masked, normalized;
    float eps;
    int has_in;   // the records' initial values are set
    int direct;   // one chunk from a zero state: this launch writes the outputs
    int need_D;   // D's increments of the last chunk are wanted too (final state)
};

// D_0 = S_0 C_0 - G_0, e_0 = S_0 m_0 - h_0 of a head's state_in into D's initial record; block (head, 16 rows)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kStateThreads) g2_init_kernel(const float *__restrict__ st, Records D, int d, int dv) {
    __shared__ __align__(16) float rows[kStateRows * 128];
    chain_begin();
    const float *S = st + blockIdx.x * ((long long)d * d + 2LL * d * dv + 2LL * d), *C = S + d * d, *m = C + d * dv;
    const float *G = m + d, *h = G + d * dv;
    float *out = D.at(blockIdx.x, D.nch);
    state_products(S, C, m, d, dv, blockIdx.y * kStateRows, rows, [&](int a, int b, float x) {
        if (b < dv) out[a * dv + b] = x - G[a * dv + b];
        else out[d * dv + a] = x - h[a];
    });
}

// state_out's G = S C - D, h = S m - e (zeros for the unmasked operator) from its S, C, m and D's
// total; block (head, 16 rows)
__global__ void __launch_bounds__(kStateThreads) g2_final_kernel(float *__restrict__ st, Records D, int d, int dv,
                                                                 int masked) {
    __shared__ __align__(16) float rows[kStateRows * 128];
    chain_begin();
    float *S = st + blockIdx.x * ((long long)d * d + 2LL * d * dv + 2LL * d), *C = S + d * d, *m = C + d * dv;
    float *G = m + d, *h = G + d * dv;
    const float *tot = D.at(blockIdx.x, D.nch);
    if (!masked) {
        const int a0 = blockIdx.y * kStateRows;
        for (int i = threadIdx.x; i < kStateRows * dv; i += kStateThreads) G[a0 * dv + i] = 0.f;
        if (threadIdx.x < kStateRows) h[a0 + threadIdx.x] = 0.f;
        return;
    }
    state_products(S, C, m, d, dv, blockIdx.y * kStateRows, rows, [&](int a, int b, float x) {
        if (b < dv) G[a * dv + b] = x - tot[a * dv + b];
        else h[a] = x - tot[d * dv + a];
    });
}

// ---------------------------------------------------------------------------
// per chunk: X, T, T V and, masked, the increments X^T V, X^T 1 of D and e.  Two token buffers serve
// in turn as Q, K, X and V: 94 KB of shared memory at N = 128, so two blocks fit an SM.
// ---------------------------------------------------------------------------
template <int N, typename T>
__global__ void __launch_bounds__(kCT, blocks_per_sm<N>())
    g2_chunk_kernel(const T *__restrict__ q, const T *__restrict__ k, const T *__restrict__ v, T *__restrict__ out,
                    const __grid_constant__ GParams P) {
    extern __shared__ __align__(16) float sm[];
    chain_begin();
    float *b0 = sm, *b1 = b0 + tile_floats<N>(), *Wt = b1 + tile_floats<N>(), *stage = Wt + kC * kLdW;
    float *dens = stage + stage_floats<N>();
    int c, hd;
    chunk_of(P.S.nch, c, hd);
    const int d = P.d, dv = P.dv, t0 = c * kC, len = min(kC, P.n - t0);
    const long long tok = (long long)hd * P.n + t0;
    const bool carry = c > 0 || P.has_in;
    load_tile<N>(b0, q + tok * d, len, d);
    const bool any_k = sync_unless_finite<N>(load_tile<N>(b1, k + tok * d, len, d));
    const Tile<N> t;
    nt_masked(Wt, b0, b1, N + 4, d, nullptr);
    Acc<N> acc;
    acc.zero();
    if (carry) nn_carry<N, kPlain>(acc, t, b0, P.S.at(hd, c), d, d, d, stage);
    else __syncthreads();
    nn_lower<N>(acc, t, Wt, b1, any_k);
    __syncthreads();
    acc_to_smem<N>(acc, t, b1);  // X
    __syncthreads();
    if (P.masked) nt_masked(Wt, b0, b1, N + 4, d, nullptr);
    else nt_masked(Wt, b1, b0, N + 4, d, nullptr);
    __syncthreads();
    const float seen_v = load_tile<N>(b0, v + tok * dv, len, dv);
    float den = row_dot(Wt, kLdW, nullptr, kC);
    acc.zero();
    if (!P.masked && carry) {
        const float *Cp = P.C.at(hd, c);
        den += row_dot(b1, N + 4, Cp + d * dv, d);
        nn_carry<N, kPlain>(acc, t, b1, Cp, dv, d, dv, stage);
    }
    const int r = threadIdx.x >> 1;
    const bool direct = P.direct || !P.masked;
    if ((threadIdx.x & 1) == 0) {
        if (direct) dens[r] = P.normalized ? den + P.eps : 1.f;
        else if (r < len) P.den[tok + r] = den;
    }
    nn_lower<N>(acc, t, Wt, b0, sync_unless_finite<N>(seen_v));  // T V
    if (direct) {
        if (P.normalized) acc.each([&](float x, int i, int) { return x / dens[t.row(i)]; });
        acc_to_global<N, T>(acc, t, out + tok * dv, len, dv);
    } else {
        acc_to_global<N, float>(acc, t, P.num + tok * dv, len, dv);
    }
    if (!P.masked || (c + 1 == P.D.nch && !P.need_D)) return;
    float *rec = P.D.at(hd, c);
    atb_to_global<N>(t, rec, b1, b0, d, dv);
    col_sums<N>(rec + d * dv, b1, nullptr, d);
}

// ---------------------------------------------------------------------------
// one chunk of head sizes up to 32: all of a head in one block, products over the chunk's own tokens
// ---------------------------------------------------------------------------
constexpr int kOneN = 32, kOneLd = kOneN + 4, kOneMat = kOneN * kOneLd;
constexpr int kOneFloats = 4 * tile_floats<kOneN>() + kC * kLdW + 3 * kOneMat + 2 * kOneN + kC;

// Where that kernel serves.  With a state in or out the launches below are three to seven for a few
// microseconds of work; without one they are one, whose products run over 64 tokens however few there are.
// Measured, fp32, us, launches below -> this (-> the kernels before those): 16 x 16, 8 heads of 1 token, states in
// and out 26.8 -> 12.4 (18.6), 512 heads of 16 40.7 -> 22.9 (26.7), 8 of 64 28.7 -> 16.5 (57); 32 x 32, 512
// heads of 64 63.7 -> 41.2 (417); without states 2000 heads of 1 x 16 43.2 -> 26.8 (36.0), of 64 the same.
bool one_block(int n, int d, int dv, bool states) {
    return n > 0 && n <= (states ? kC : 16) && d <= kOneN && dv <= kOneN;
}

// a rows x width matrix in global memory (null: zeros) into kOneN rows of kOneLd floats, zero beyond
__device__ __forceinline__ void load_matrix(float *dst, const float *src, int rows, int width) {
    constexpr int U = kOneN * kOneN / kCT;
    float x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int r = (threadIdx.x + u * kCT) / kOneN, c = threadIdx.x % kOneN;
        x[u] = src && r < rows && c < width ? src[r * width + c] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) dst[(threadIdx.x + u * kCT) / kOneN * kOneLd + threadIdx.x % kOneN] = x[u];
}
// emit(a, b, (S C)_ab)
template <typename F>
__device__ __forceinline__ void state_product(const Tile<kOneN> &t, const float *S, const float *C, int d, int dv, F emit) {
    if (4 * t.rg >= d) return;  // rows beyond d lie beyond S
    Acc<kOneN> acc;
    acc.zero();
    nn_range<kOneN, 0>(acc, t, S, kOneLd, C, kOneLd, 0, d);
#pragma unroll
    for (int i = 0; i < Tile<kOneN>::RM; ++i)
#pragma unroll
        for (int j = 0; j < Tile<kOneN>::CM; ++j)
            if (t.col(j) < dv) emit(t.row(i), t.col(j), acc.get(i, j));
}
// M += A^T B over K tokens (a multiple of 4; d real columns of A)
__device__ __forceinline__ void add_products(const Tile<kOneN> &t, float *M, const float *A, const float *B, int d, int K) {
    if (4 * t.rg >= d) return;  // rows beyond d would read beyond a row of A
    Acc<kOneN> acc;
    acc.zero();
    tn_range<kOneN, 0, Tile<kOneN>::RM>(acc, t, A, kOneLd, B, 0, K);
#pragma unroll
    for (int i = 0; i < Tile<kOneN>::RM; ++i)
#pragma unroll
        for (int j = 0; j < Tile<kOneN>::CM; ++j) M[t.row(i) * kOneLd + t.col(j)] += acc.get(i, j);
}

template <typename T>
__global__ void __launch_bounds__(kCT) g2_one_kernel(const T *__restrict__ q, const T *__restrict__ k,
                                                     const T *__restrict__ v, T *__restrict__ out, const float *in,
                                                     float *to, int n, int d, int dv, int masked, int normalized, float eps) {
    extern __shared__ __align__(16) float sm[];
    constexpr int N = kOneN;
    float *bq = sm, *bk = bq + tile_floats<N>(), *bv = bk + tile_floats<N>(), *bx = bv + tile_floats<N>();
    float *Wt = bx + tile_floats<N>(), *S = Wt + kC * kLdW, *C = S + kOneMat, *D = C + kOneMat;
    float *m = D + kOneMat, *e = m + N, *dens = e + N;
    const int tid = threadIdx.x, kn = (n + 3) & ~3;  // tokens, up to a multiple of 4: the rows beyond n are zero
    const long long hd = blockIdx.x, tok = hd * n, len = (long long)d * d + 2LL * d * dv + 2LL * d;
    const float *st = in ? in + hd * len : nullptr;
    const int oC = d * d, om = oC + d * dv, oG = om + d, oh = oG + d * dv;
    load_tile<N>(bq, q + tok * d, n, d);
    load_tile<N>(bk, k + tok * d, n, d);
    load_tile<N>(bv, v + tok * dv, n, dv);
    if (st || to) {
        load_matrix(S, st, d, d);
        load_matrix(C, st ? st + oC : nullptr, d, dv);
        load_matrix(D, masked && st ? st + oG : nullptr, d, dv);  // G
        if (tid < N) {
            m[tid] = st && tid < d ? st[om + tid] : 0.f;
            e[tid] = masked && st && tid < d ? st[oh + tid] : 0.f;  // h
        }
    }
    __syncthreads();
    const Tile<N> t;
    const int r = tid >> 1;
    if (masked && st) {  // D = S C - G, e = S m - h
        state_product(t, S, C, d, dv, [&](int a, int b, float x) { D[a * kOneLd + b] = x - D[a * kOneLd + b]; });
        const float x = row_dot(S, kOneLd, m, d);  // rows beyond d read C, unused
        if ((tid & 1) == 0 && r < d) e[r] = x - e[r];
    }
    nt_masked(Wt, bq, bk, kOneLd, d, nullptr);
    __syncthreads();
    Acc<N> acc;
    acc.zero();
    if (st) nn_range<N, 0>(acc, t, bq, kOneLd, S, kOneLd, 0, d);
    nn_lower<N>(acc, t, Wt, bk, false, kn);
    acc_to_smem<N>(acc, t, bx);  // X = W K + Q S
    __syncthreads();
    if (masked) nt_masked(Wt, bq, bx, kOneLd, d, nullptr);
    else nt_masked(Wt, bx, bq, kOneLd, d, nullptr);
    __syncthreads();
    const float *left = masked ? bq : bx;  // T V + Q D, or T V + X C
    float den = row_dot(Wt, kLdW, nullptr, kC);
    if (st) den += row_dot(left, kOneLd, masked ? e : m, d);
    if ((tid & 1) == 0) dens[r] = normalized ? den + eps : 1.f;
    acc.zero();
    if (st) nn_range<N, 0>(acc, t, left, kOneLd, masked ? D : C, kOneLd, 0, d);
    nn_lower<N>(acc, t, Wt, bv, false, kn);
    __syncthreads();
    if (normalized) acc.each([&](float x, int i, int) { return x / dens[t.row(i)]; });
    acc_to_global<N, T>(acc, t, out + tok * dv, n, dv);
    if (!to) return;
    // the state after the chunk
    add_products(t, S, bk, bk, d, kn);
    add_products(t, C, bq, bv, d, kn);
    if (masked) add_products(t, D, bx, bv, d, kn);
    if (tid < 2 * N) {  // m += Q^T 1, e += X^T 1
        const int c = tid % N;
        const float *A = tid < N ? bq : bx;
        float x = 0.f;
        for (int i = 0; i < n; ++i) x += A[i * kOneLd + c];
        (tid < N ? m : e)[c] += x;
    }
    __syncthreads();
    float *o = to + hd * len;
    for (int i = tid; i < d * d; i += kCT) o[i] = S[i / d * kOneLd + i % d];
    for (int i = tid; i < d * dv; i += kCT) o[oC + i] = C[i / dv * kOneLd + i % dv];
    if (tid < d) o[om + tid] = m[tid];
    if (masked) {
        state_product(t, S, C, d, dv, [&](int a, int b, float x) { o[oG + a * dv + b] = x - D[a * kOneLd + b]; });
        const float x = row_dot(S, kOneLd, m, d);
        if ((tid & 1) == 0 && r < d) o[oh + r] = x - e[r];
    } else {
        for (int i = tid; i < d * dv; i += kCT) o[oG + i] = 0.f;
        if (tid < d) o[oh + tid] = 0.f;
    }
}

template <typename T>
cudaError_t forward_one(const Fwd2 &p, cudaStream_t s) {
    const int smem = kOneFloats * (int)sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(g2_one_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e) return e;
    g2_one_kernel<T><<<p.BH, kCT, smem, s>>>(static_cast<const T *>(p.q), static_cast<const T *>(p.k),
                                            static_cast<const T *>(p.v), static_cast<T *>(p.out), p.state_in, p.state_out,
                                            p.n, p.d, p.dv, p.masked, p.normalized, p.eps);
    return cudaGetLastError();
}

template <int N, typename T>
cudaError_t forward_n(const Fwd2 &p, const GLayout &L, float *ws, cudaStream_t s) {
    const T *q = static_cast<const T *>(p.q), *k = static_cast<const T *>(p.k), *v = static_cast<const T *>(p.v);
    T *out = static_cast<T *>(p.out);
    const long long st_len = state_floats(L.d, L.dv);
    const int d = L.d, dv = L.dv, nch = L.nch;
    cudaError_t e;
    GParams P{};
    P.S = {ws + L.oS, L.lenS, nch};
    P.C = {ws + L.oC, L.lenC, nch};
    P.D = {ws + L.oD, L.lenD, nch};
    P.num = ws + L.oNum; P.den = ws + L.oDen;
    P.n = L.n; P.d = d; P.dv = dv; P.masked = p.masked; P.normalized = p.normalized; P.eps = p.eps;
    P.has_in = p.state_in != nullptr;
    P.need_D = p.state_out != nullptr;
    P.direct = nch == 1 && !p.state_in;
    bool follows = false;  // a launch of this call came before
    // D's initial value; the states' S and [C | m] start S's and C's sums as they lie
    if (p.state_in && p.masked) {
        if ((e = chain_launch(false, g2_init_kernel, dim3(L.BH, d / kStateRows), kStateThreads, 0, s, p.state_in, P.D, d, dv)))
            return e;
        follows = true;
    }
    const bool sums = nch > 1 || p.state_in || p.state_out, sums_C = !p.masked || p.state_out;
    if (sums) {
        if (nch > 0) {
            SumJobs<T> jobs{};
            jobs.j[0] = {k, k, P.S, d, d, 0};
            jobs.j[1] = {q, v, P.C, d, dv, 1};
            if ((e = launch_sums<N, T>(follows, jobs, sums_C ? 2 : 1, L.BH, L.n, s))) return e;
            follows = true;
        }
        ScanJobs scans{};
        scans.j[0] = {P.S, p.state_in, st_len, p.state_out, st_len, 0};
        scans.j[1] = {P.C, p.state_in ? p.state_in + d * d : nullptr, st_len,
                      p.state_out ? p.state_out + d * d : nullptr, st_len, 0};
        if ((e = launch_scan(scans, sums_C ? 2 : 1, L.BH, s, follows))) return e;
        follows = true;
    }
    const dim3 grid = chunk_grid(nch, L.BH);
    if (nch > 0) {
        const int smem = (2 * tile_floats<N>() + kC * kLdW + stage_floats<N>() + kC) * (int)sizeof(float);
        if ((e = cudaFuncSetAttribute(g2_chunk_kernel<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)))
            return e;
        if ((e = chain_launch(follows, g2_chunk_kernel<N, T>, grid, kCT, smem, s, q, k, v, out, P))) return e;
    }
    if (p.masked && sums) {
        float *total = ws + L.oD + (long long)nch * L.lenD;
        const long long head = (long long)(nch + 1) * L.lenD;
        ScanJobs scans{};
        scans.j[0] = {P.D, p.state_in ? total : nullptr, head, total, head, 0};
        if ((e = launch_scan(scans, 1, L.BH, s))) return e;
        if (nch > 0 && !P.direct) {
            const OutParams O{P.D, P.num, P.den, L.n, d, dv, p.normalized, p.eps, P.has_in};
            if ((e = launch_out<N, T>(q, out, O, L.BH, s))) return e;
        }
    }
    if (p.state_out) {
        if ((e = chain_launch(true, g2_final_kernel, dim3(L.BH, d / kStateRows), kStateThreads, 0, s, p.state_out, P.D, d, dv,
                              p.masked)))
            return e;
    }
    return cudaSuccess;
}

}  // namespace

size_t generic2_workspace_bytes(int BH, int n, int d, int dv, int) {
    return kWsHeaderBytes + sizeof(float) * (size_t)make_layout(BH, n, d, dv).total;
}

int generic2_launches(int n, int d, int dv, int masked, int has_state_in, int has_state_out) {
    if (one_block(n, d, dv, has_state_in || has_state_out)) return 1;
    const int nch = (n + kC - 1) / kC;
    const bool sums = nch > 1 || has_state_in || has_state_out;
    int l = (has_state_in && masked ? 1 : 0) + (has_state_out ? 1 : 0);
    if (sums) l += (nch > 0 ? 1 : 0) + 1;                             // chunk sums, their prefix sums
    if (nch > 0) l += 1;                                              // the chunks
    if (masked && sums) l += 1 + (nch > 1 || (nch > 0 && has_state_in) ? 1 : 0);  // D's prefix sums, outputs
    return l;
}

cudaError_t generic2_forward(const Fwd2 &p, cudaStream_t stream) {
    const GLayout L = make_layout(p.BH, p.n, p.d, p.dv);
    float *scratch = reinterpret_cast<float *>(p.ws + kWsHeaderBytes);
    Fwd2 pp = p;
    if (p.state_in && p.state_out && p.state_in != p.state_out) {
        // threads of one head read state_in while others write state_out: where the two are the same
        // memory each value is read by the thread that overwrites it, or by an earlier launch; where
        // they overlap in another way a private copy is read
        const size_t bytes = sizeof(float) * (size_t)p.BH * (size_t)state_floats(p.d, p.dv);
        const char *a = reinterpret_cast<const char *>(p.state_in), *b = reinterpret_cast<const char *>(p.state_out);
        if (a < b + bytes && b < a + bytes) {
            float *copy = scratch + L.oStage;
            cudaError_t e = cudaMemcpyAsync(copy, p.state_in, bytes, cudaMemcpyDeviceToDevice, stream);
            if (e != cudaSuccess) return e;
            pp.state_in = copy;
        }
    }
    if (one_block(p.n, p.d, p.dv, p.state_in || p.state_out))
        return p.dt == HLA_BF16 ? forward_one<__nv_bfloat16>(pp, stream) : forward_one<float>(pp, stream);
    return with_padded_size(p.d, p.dv, [&](auto size) {
        constexpr int N = decltype(size)::value;
        return p.dt == HLA_BF16 ? forward_n<N, __nv_bfloat16>(pp, L, scratch, stream)
                                : forward_n<N, float>(pp, L, scratch, stream);
    });
}

}  // namespace hla
