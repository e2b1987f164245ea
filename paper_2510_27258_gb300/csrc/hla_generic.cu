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
// sums; outputs.  One chunk without states is the third launch alone.
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
    const bool any_k = sync_unless_finite(load_tile<N>(b1, k + tok * d, len, d));
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
    nn_lower<N>(acc, t, Wt, b0, sync_unless_finite(seen_v));  // T V
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

int generic2_launches(int n, int masked, int has_state_in, int has_state_out) {
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
    return with_padded_size(p.d, p.dv, [&](auto size) {
        constexpr int N = decltype(size)::value;
        return p.dt == HLA_BF16 ? forward_n<N, __nv_bfloat16>(pp, L, scratch, stream)
                                : forward_n<N, float>(pp, L, scratch, stream);
    });
}

}  // namespace hla
