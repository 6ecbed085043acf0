// Per-token coefficient kernels (fp32; the Gram-Schmidt part in fp64):
//   coef_full  norm statistics -> router scores, TopK routing, pre-maps
//              (Eq. fused_normalized_projection, Eq. router, Eq. router_topk, Eq. param_pre)
//   coef_act   active RMS -> post-map, Sinkhorn residual map + row clamp
//              (Eq. param_post, Eq. param_res, App. A)
//   bwd_coef   reverse of coef_act, of the Gram-Schmidt coefficients (Eq. gs) and of the
//              write-back contraction (Eq. sparse_write_delta)
//   full_coef  reverse of coef_full (norm corrections, pre-map sigmoid, router through the
//              selected routed scores only)
//   colsum_out the alpha / b gradients from the column sums that bwd_coef's and full_coef's blocks leave
//
// A block takes a few consecutive tokens.  What it reads of the projections (every partial slot of a
// split reduction: no separate pass sums them) is read with neighbouring threads on neighbouring
// columns and kept in shared memory; the maps are computed with one thread per entry, the Sinkhorn
// iterations with one lane per matrix row.  These kernels are bound by latency, not by bytes: with one
// thread per token, which walked its row of slots alone, and the sums over slots and over tokens in
// passes of their own, a training step of one N = 16, k = 4, C = 256 MLP sublayer of 512 tokens spent
// 0.28 ms in them (bwd_coef 0.10, column sums 0.09, coef_act 0.034) and now 0.09 ms (bwd_coef 0.022);
// at 16384 tokens and C = 2048 bwd_coef went from 0.12 to 0.056 ms.
#include <algorithm>

#include "xhc_internal.cuh"

namespace xhc {

namespace {

// ---------------------------------------------------------------------------------------------
// number of partial slots of 128-row tile m: the persistent CTAs of the stream-K plan that cover it

template <class U>
__device__ __forceinline__ U cta_of(U W, U P, U x) {
    U c = x * P / W;
    while (c > 0 && W * c / P > x) --c;
    while (W * (c + 1) / P <= x) ++c;
    return c;
}
template <class U>
__device__ __forceinline__ int tile_slots(U W, U P, U KB, U m) {
    return (int)(cta_of<U>(W, P, (m + 1) * KB - 1) - cta_of<U>(W, P, m * KB)) + 1;
}
__device__ __forceinline__ int slot_count(const SlotPlan& s, int m) {
    if (s.n > 0) return s.n;
    // 32-bit division where the products fit
    if ((unsigned long long)s.W * (unsigned)(s.P + 1) < (1ull << 32))
        return tile_slots<uint32_t>((uint32_t)s.W, (uint32_t)s.P, (uint32_t)s.KB, (uint32_t)m);
    return tile_slots<unsigned long long>((unsigned long long)s.W, (unsigned long long)s.P,
                                          (unsigned long long)s.KB, (unsigned long long)m);
}

// sum over `cnt` slots of p, `stride` apart, starting at slot q0 in steps of dq, added in slot order with
// U loads in flight
template <int U>
__device__ __forceinline__ float slot_sum(const float* p, long long stride, int cnt, int q0, int dq) {
    float s = 0.f;
    int q = q0;
    for (; q + (U - 1) * dq < cnt; q += U * dq) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = p[(q + u * dq) * stride];
#pragma unroll
        for (int u = 0; u < U; ++u) s += v[u];
    }
#pragma unroll 4
    for (; q < cnt; q += dq) s += p[q * stride];
    return s;
}

// Two arrays of slot sums into shared memory: dst[0, n0) = sums of p0 + e, dst[n0, n0 + n1) = sums of
// p1 + e * step1.  The slots of a stream-K plan are added in slot order; those of an even split, of which
// there are many on few tokens, by groups of threads that take interleaved slots (scr: one float per thread),
// a number of groups that follows from n alone while a block takes one token (below 128 tokens it does).  So a
// token of a call of fewer than 128 has the same bits whatever the others are; from 128 on the plan, and with it
// where the sums are cut, depends on the number of tokens.
// Few elements with many ordered slots pass through shared memory (stage: SS_STAGE floats), so that
// the whole block loads them: 82 sums over 172 slots took 27 us with a thread each.  Ends with a
// block barrier.
constexpr int SS_STAGE = 4096;
__device__ __forceinline__ void slot_sums(bool ordered, const float* p0, long long stride0, int cnt0,
                                          int n0, const float* p1, long long stride1, int cnt1, int n1,
                                          int step1, float* dst, float* scr, float* stage) {
    const int n = n0 + n1, nt = blockDim.x, tid = threadIdx.x;
    const int ng = ordered ? 1 : nt / n;
    if (ng > 1) {
        const int g = tid / n, e = tid - g * n;
        if (g < ng)
            scr[tid] = (e < n0) ? slot_sum<8>(p0 + e, stride0, cnt0, g, ng)
                                : slot_sum<8>(p1 + (long long)(e - n0) * step1, stride1, cnt1, g, ng);
        __syncthreads();
        if (tid < n) {
            float s = 0.f;
            for (int q = 0; q < ng; ++q) s += scr[q * n + tid];
            dst[tid] = s;
        }
    } else if (2 * n <= nt && cnt0 > 16) {
        const int nl = nt / n, sc = SS_STAGE / n;    // slots loaded at a time, slots a chunk
        const int g = tid / n, e = tid - g * n;
        const int cnt = e < n0 ? cnt0 : cnt1;
        const float* p = e < n0 ? p0 + e : p1 + (long long)(e - n0) * step1;
        const long long stride = e < n0 ? stride0 : stride1;
        float s = 0.f;
        for (int q0 = 0; q0 < max(cnt0, cnt1); q0 += sc) {
            const int m = min(sc, cnt - q0);
            if (g < nl) {
#pragma unroll 8
                for (int q = g; q < m; q += nl) stage[q * n + e] = p[(q0 + q) * stride];
            }
            __syncthreads();
            if (tid < n) {
#pragma unroll 8
                for (int q = 0; q < m; ++q) s += stage[q * n + tid];
            }
            __syncthreads();
        }
        if (tid < n) dst[tid] = s;
    } else {
        for (int e = tid; e < n; e += nt)
            dst[e] = (e < n0) ? slot_sum<16>(p0 + e, stride0, cnt0, 0, 1)
                              : slot_sum<16>(p1 + (long long)(e - n0) * step1, stride1, cnt1, 0, 1);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// Sinkhorn of Eq. mhc_sinkhorn on a k x k block (k <= KM), with the App. A row clamp.  KM neighbouring
// lanes hold one matrix, lane a its row a; columns are normalised as rows of the transposed matrix
// (log2 KM exchanges between the lanes: one division a lane and half-step, sums in index order).
// exp(M - rowmax): the first row normalisation removes any per-row scale, so this equals exp(M).

template <int KM>
__device__ __forceinline__ void sk_init(const float (&M)[KM], int a, int k, float (&A)[KM]) {
    float mx = -INFINITY;
#pragma unroll
    for (int b = 0; b < KM; ++b)
        if (b < k) mx = fmaxf(mx, M[b]);
#pragma unroll
    for (int b = 0; b < KM; ++b) A[b] = (a < k && b < k) ? expf(M[b] - mx) : 0.f;
}

// the lanes' KM x KM matrix transposed
template <int KM>
__device__ __forceinline__ void transpose(float (&A)[KM], int a) {
#pragma unroll
    for (int o = 1; o < KM; o <<= 1) {
        const bool up = (a & o) != 0;
#pragma unroll
        for (int b = 0; b < KM; ++b) {
            if (b & o) continue;
            const float lo = A[b], hi = A[b | o];
            const float got = __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
            A[b] = up ? got : lo;
            A[b | o] = up ? hi : got;
        }
    }
}

// normalisation of the lane's row (or column, of the transposed matrix); returns the factor, 0 outside
// the matrix
template <int KM>
__device__ __forceinline__ float sk_half(float (&A)[KM], int a, int k) {
    float s = 0.f;
#pragma unroll
    for (int b = 0; b < KM; ++b) s += A[b];
    const float r = (a < k) ? 1.0f / s : 0.f;
#pragma unroll
    for (int b = 0; b < KM; ++b) A[b] *= r;
    return r;
}

template <int KM>
__device__ __forceinline__ void sk_iter(float (&A)[KM], int a, int k) {
    sk_half<KM>(A, a, k);
    transpose<KM>(A, a);
    sk_half<KM>(A, a, k);
    transpose<KM>(A, a);
}

template <int KM>
__device__ __forceinline__ float row_total(const float (&A)[KM]) {
    float s = 0.f;
#pragma unroll
    for (int b = 0; b < KM; ++b) s += A[b];
    return s;
}

// ---------------------------------------------------------------------------------------------
// coef_full: a block of TB tokens (inside one 128-token tile of the projection)

constexpr int CF_NT = 512;

__global__ void __launch_bounds__(CF_NT) k_coef_full(Dims d, int T, int TB, const float* part,
                                                     const float* pstats, SlotPlan sp,
                                                     const float* wsum, int nws,
                                                     const float* alpha_pre,
                                                     const float* b_pre, float* __restrict__ zfull,
                                                     float* __restrict__ stats, float* __restrict__ wsum_out,
                                                     float* __restrict__ hpre, int* __restrict__ I,
                                                     float* __restrict__ p) {
    pdl_entry();
    extern __shared__ float sm[];   // [TB][n] projections, [TB][2] statistics
    __shared__ float scr[CF_NT], scw[8 * MAXN], ws[MAXN], stage[SS_STAGE];
    const int tid = threadIdx.x, lane = tid & 31, N = d.N, n = d.nfull;
    const long long t0 = (long long)blockIdx.x * TB;
    const int ntok = (int)min((long long)TB, T - t0);
    // column sums of W_r from the partials: eight threads a column, then their sum
    if (d.hr && tid < 8 * N) scw[tid] = slot_sum<8>(wsum + tid % N, N, nws, tid / N, 8);
    const int nsl = slot_count(sp, (int)(t0 >> 7));
    float* zs = sm;
    float* st = sm + ntok * n;
    slot_sums(sp.n == 0, part + t0 * n, (long long)T * n, nsl, ntok * n, pstats + t0 * 2, (long long)T * 2, nsl,
              ntok * 2, 1, zs, scr, stage);
    if (d.hr && tid < N) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) s += scw[q * N + tid];
        ws[tid] = s;
        if (blockIdx.x == 0) wsum_out[tid] = s;
    }
    const float inv_nc = 1.0f / (float)(N * d.C);
    for (int e = tid; e < ntok * 2; e += CF_NT) {
        // mean and mean square, rounded here: what follows is not to be contracted with the product
        const float v = __fmul_rn(st[e], inv_nc);
        st[e] = v;
        stats[t0 * 2 + e] = v;
    }
    __syncthreads();
    const int roff = d.hr ? N : 0, GN = d.G * N;
    for (int e = tid; e < ntok * n; e += CF_NT) {
        const int tt = e / n, o = e - tt * n;
        const float z = zs[e];
        zfull[t0 * n + e] = z;
        if (o >= roff) {
            const int qo = o - roff, slot = qo / N;
            const float rstd = 1.0f / sqrtf(st[tt * 2 + 1] + d.eps);
            hpre[(t0 + tt) * GN + qo] = sigm(alpha_pre[slot] * (z * rstd) + b_pre[qo]);
        }
    }
    __syncthreads();
    // Eq. router_topk, a warp per token with a lane per stream: fixed streams 0..m-1 (p = 1), then TopK
    // over i >= m by router logit (sigmoid and softmax are both monotone in the logit), descending,
    // ties to the lower stream index.
    for (int tt = tid >> 5; tt < ntok; tt += CF_NT / 32) {
        const long long tk = (t0 + tt) * d.k;
        if (lane < d.m) {
            I[tk + lane] = lane;
            p[tk + lane] = 1.0f;
        }
        if (!d.hr) continue;
        const float mu = st[tt * 2], nu = st[tt * 2 + 1];
        const float lstd = 1.0f / sqrtf(nu - mu * mu + d.eps);
        const float z = (lane < N) ? (zs[tt * n + lane] - mu * ws[lane]) * lstd : -INFINITY;
        float zmax = z, den = 0.f;
        if (d.softmax) {
            // softmax router: s_i = exp(z_i) / sum over all N logits (the fixed streams' included)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
            den = warp_sum(lane < N ? expf(z - zmax) : 0.f);
        }
        bool open = lane >= d.m && lane < N;
        for (int j = d.m; j < d.k; ++j) {
            // the first open stream wins over a NaN logit of a later one, and with a NaN of its own
            const unsigned om = __ballot_sync(0xffffffffu, open);
            float key = z;
            if (z != z) key = (lane == __ffs(om) - 1) ? INFINITY : -INFINITY;
            int best = open ? lane : 64;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ko = __shfl_xor_sync(0xffffffffu, key, o);
                const int bo = __shfl_xor_sync(0xffffffffu, best, o);
                if (bo < 64 && (best >= 64 || ko > key || (ko == key && bo < best))) {
                    key = ko;
                    best = bo;
                }
            }
            if (lane == best) {
                open = false;
                I[tk + j] = lane;
                p[tk + j] = d.softmax ? expf(z - zmax) / den : sigm(z);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// coef_act

template <int KM>
__global__ void __launch_bounds__(CF_NT) k_coef_act(Dims d, int slot, int T, int TB, const float* part,
                                                    const float* pstats, int ssplits, SlotPlan sp,
                                                    const float* alpha_post,
                                                    const float* b_post,
                                                    const float* alpha_res,
                                                    const float* b_res, float* __restrict__ zact,
                                                    float* __restrict__ rs, float* __restrict__ hpost,
                                                    float* __restrict__ hres) {
    pdl_entry();
    extern __shared__ float sm[];   // [TB][n] projections, [TB] sums of squares
    __shared__ float scr[CF_NT], stage[SS_STAGE];
    const int tid = threadIdx.x, k = d.k, kK = d.k * d.K[slot], n = d.nact[slot];
    const long long t0 = (long long)blockIdx.x * TB;
    const int ntok = (int)min((long long)TB, T - t0);
    const int nsl = slot_count(sp, (int)(t0 >> 7));
    float* zs = sm;
    float* st = sm + ntok * n;
    slot_sums(sp.n == 0, part + t0 * n, (long long)T * n, nsl, ntok * n, pstats + t0 * 2 + 1, (long long)T * 2,
              ssplits, ntok, 2, zs, scr, stage);
    if (tid < ntok) {
        const float r = 1.0f / sqrtf(st[tid] / (float)(k * d.C) + d.eps);
        st[tid] = r;
        rs[t0 + tid] = r;
    }
    __syncthreads();
    const float ap = alpha_post[slot];
    for (int e = tid; e < ntok * n; e += CF_NT) {
        const int tt = e / n, o = e - tt * n;
        const float z = zs[e];
        zact[t0 * n + e] = z;
        if (o < kK) {
            hpost[(t0 + tt) * kK + o] = 2.0f * sigm(ap * (z * st[tt]) + b_post[o]);
        }
    }
    if (slot != d.G - 1 || (tid & ~31) >= TB * KM) return;
    // whole warps run the iterations (lanes past the last token repeat it)
    const int tq = tid / KM, a = tid - tq * KM;
    const int tt = min(tq, ntok - 1);
    const float ar = alpha_res[0], r = st[tt];
    float M[KM], H[KM];
#pragma unroll
    for (int b = 0; b < KM; ++b)
        M[b] = (a < k && b < k) ? ar * (zs[tt * n + kK + a * k + b] * r) + b_res[a * k + b] : 0.f;
    sk_init<KM>(M, a, k, H);
    for (int it = 0; it < d.iters; ++it) sk_iter<KM>(H, a, k);
    const float s = row_total<KM>(H);
    if (tq < ntok && a < k) {
        float* dst = hres + (t0 + tt) * k * k + a * k;
#pragma unroll
        for (int b = 0; b < KM; ++b)
            if (b < k) dst[b] = (s > 1.f) ? H[b] / s : H[b];
    }
}

// tokens per block: enough blocks for the GPU at few tokens, whole warps of matrix rows at many; a
// power of two up to 32, so that a block lies in one 128-token tile
int coef_tokens(int T) {
    int tb = 1;
    while (tb < 32 && T / (2 * tb) >= 2 * device_sms()) tb *= 2;
    return tb;
}

}  // namespace

cudaError_t launch_coef_full(const Dims& d, int T, const float* part, const float* pstats,
                             const SlotPlan& sp, const float* wsum, int nws, const float* alpha_pre,
                             const float* b_pre, float* zfull, float* stats, float* wsum_out, float* hpre,
                             int* I, float* p, cudaStream_t st) {
    const int TB = coef_tokens(T);
    const size_t sm = (size_t)TB * (d.nfull + 2) * 4;
    XHC_LAUNCH(st, (T + TB - 1) / TB, CF_NT, sm, (k_coef_full), d, T, TB, part, pstats, sp, wsum, nws, alpha_pre, b_pre, zfull, stats, wsum_out, hpre, I, p);
    return cudaGetLastError();
}

cudaError_t launch_coef_act(const Dims& d, int slot, int T, const float* part,
                            const float* pstats, int ssplits, const SlotPlan& sp, const float* alpha_post,
                            const float* b_post, const float* alpha_res, const float* b_res,
                            float* zact, float* rs, float* hpost, float* hres, cudaStream_t st) {
    const int TB = coef_tokens(T);
    const size_t sm = (size_t)TB * (d.nact[slot] + 1) * 4;
    const unsigned grid = (unsigned)((T + TB - 1) / TB);
    if (d.k <= 4) {
        XHC_LAUNCH(st, grid, CF_NT, sm, (k_coef_act<4>), d, slot, T, TB, part, pstats, ssplits, sp, alpha_post, b_post, alpha_res, b_res, zact, rs, hpost, hres);
    } else {
        XHC_LAUNCH(st, grid, CF_NT, sm, (k_coef_act<8>), d, slot, T, TB, part, pstats, ssplits, sp, alpha_post, b_post, alpha_res, b_res, zact, rs, hpost, hres);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// bwd_coef: per token, from the reductions
//   P[j][a] = <dXn_j, u_a>   Q[j][i] = <dXn_j, x_act_i> (last slot)   Gm[a][b] = <u_a, u_b> (GS)
// produce E[j][a] = p_j sum_q Hpost[j][q] B[q][a], D = dG + dG^T, H_res, the scaled projection
// gradient dZs = dz * r, the RMS coefficient cx, dp and the alpha / b contributions (summed over the
// block's tokens).
//
// A block takes TB tokens: its first warp the post-map and Gram-Schmidt reverse of token `lane`, its
// other warps (last slot) the Sinkhorn reverse with one lane per matrix row.  The matrix entering every
// iteration is kept in shared memory, so the reverse sweep rebuilds one half-step an iteration.

namespace {

template <int KM>
__device__ void sinkhorn_bwd(const float (&M)[KM], int a, int k, int iters, float* ck, int stride,
                             const float (&dH)[KM], float (&H)[KM], float (&dM)[KM]) {
    float A[KM], A0[KM], dA[KM];
    sk_init<KM>(M, a, k, A);
#pragma unroll
    for (int b = 0; b < KM; ++b) A0[b] = A[b];
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int b = 0; b < KM; ++b) ck[(it * KM + b) * stride] = A[b];
        sk_iter<KM>(A, a, k);
    }
    // clamp
    const float s = row_total<KM>(A);
    if (s > 1.f) {
        float dot = 0.f;
#pragma unroll
        for (int b = 0; b < KM; ++b) {
            H[b] = A[b] / s;
            dot += dH[b] * H[b];
        }
#pragma unroll
        for (int b = 0; b < KM; ++b) dA[b] = (dH[b] - dot) / s;
    } else {
#pragma unroll
        for (int b = 0; b < KM; ++b) {
            H[b] = A[b];
            dA[b] = dH[b];
        }
    }
    for (int it = iters - 1; it >= 0; --it) {
        // R: after the row step; A: its transpose after the column step; dA follows
        float R[KM];
#pragma unroll
        for (int b = 0; b < KM; ++b) R[b] = ck[(it * KM + b) * stride];
        const float rr = sk_half<KM>(R, a, k);
#pragma unroll
        for (int b = 0; b < KM; ++b) A[b] = R[b];
        transpose<KM>(A, a);
        const float rc = sk_half<KM>(A, a, k);
        transpose<KM>(dA, a);
        float dot = 0.f;
#pragma unroll
        for (int b = 0; b < KM; ++b) dot += dA[b] * A[b];
#pragma unroll
        for (int b = 0; b < KM; ++b) dA[b] = (dA[b] - dot) * rc;
        transpose<KM>(dA, a);
        dot = 0.f;
#pragma unroll
        for (int b = 0; b < KM; ++b) dot += dA[b] * R[b];
#pragma unroll
        for (int b = 0; b < KM; ++b) dA[b] = (dA[b] - dot) * rr;
    }
#pragma unroll
    for (int b = 0; b < KM; ++b) dM[b] = (a < k && b < k) ? dA[b] * A0[b] : 0.f;
}

// shared memory of one token, in floats: reductions, E, D, H_res, scaled gradients, column terms and
// the two parts of sum_o dz_o zact_o
template <int KM>
struct BwdTok {
    static constexpr int R = 0;                       // [KM*4] P, [KM*KM] Q
    static constexpr int E = R + KM * 4 + KM * KM;    // [KM*4]
    static constexpr int D = E + KM * 4;              // [16]
    static constexpr int H = D + 16;                  // [KM*KM]
    static constexpr int DZ = H + KM * KM;            // [KM*4 + KM*KM]
    static constexpr int TG = DZ + KM * 4 + KM * KM;  // [KM*4 + 1 + KM*KM + 1]
    static constexpr int S = TG + KM * 4 + KM * KM + 2;
    static constexpr int ROW = (S + KM + 1) | 1;      // odd: a lane per token hits different banks
};

template <int KM, bool SIX>
__global__ void __launch_bounds__(160) k_bwd_coef(Dims d, int slot, int T, int TB, const float* red,
                                                  int nslice, const float* zact,
                                                  const float* rs, const float* p,
                                                  const float* hpost, const double* gram,
                                                  const float* alpha_post,
                                                  const float* alpha_res,
                                                  const float* b_res, float* __restrict__ tokmat,
                                                  float* __restrict__ dzs, float* dp,
                                                  float* __restrict__ colp, DzPack pack, WRows wrows, int nblk) {
    pdl_entry();
    if ((int)blockIdx.x >= nblk) {
        pack_wrows_of<SIX>(wrows, (int)blockIdx.x - nblk);
        return;
    }
    using L = BwdTok<KM>;
    extern __shared__ float sm[];   // [TB][ROW], then the Sinkhorn iterates
    const int tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;
    const int k = d.k, K = d.K[slot], kK = k * K, n = d.nact[slot];
    const bool last = (slot == d.G - 1);
    const bool gs = (K > 1) && d.gs;
    const long long t0 = (long long)blockIdx.x * TB;
    const int ntok = (int)min((long long)TB, T - t0);
    // reduction slots per token (see wb_bred): P at j*4 + a, Q at KM*4 + j*KM + i
    {
        const int nv = last ? KM * 4 + KM * KM : KM * 4;
        for (int e = tid; e < ntok * nv; e += nt) {
            const int tt = e / nv, q = e - tt * nv;
            bool used;
            if (q < KM * 4) used = (q >> 2) < k && (q & 3) < K;
            else used = (q - KM * 4) / KM < k && (q - KM * 4) % KM < k;
            float s = 0.f;
            if (used) s = slot_sum<8>(red + (t0 + tt) * nslice * NRED + q, NRED, nslice, 0, 1);
            sm[tt * L::ROW + L::R + q] = s;
        }
    }
    __syncthreads();
    const float ar = last ? alpha_res[0] : 0.f;
    if (tid < 32) {
        if (lane < ntok) {
            const long long t = t0 + lane;
            float* row = sm + lane * L::ROW;
            const float r = rs[t], ap = alpha_post[slot];
            const float* za = zact + t * n;
            float B[MAXCOMP][MAXCOMP];
            double Gm[NGRAM];
            GramSchmidt G;
            if (gs) {
#pragma unroll
                for (int q = 0; q < NGRAM; ++q) Gm[q] = 0.0;
#pragma unroll
                for (int a = 0; a < MAXCOMP; ++a)
#pragma unroll
                    for (int b = 0; b <= a; ++b)
                        if (a < K) Gm[a * (a + 1) / 2 + b] = gram[t * NGRAM + a * (a + 1) / 2 + b];
                G.forward(Gm, (double)d.eps_gs);
                G.coef(B);
            } else {
#pragma unroll
                for (int q = 0; q < MAXCOMP; ++q)
#pragma unroll
                    for (int a = 0; a < MAXCOMP; ++a) B[q][a] = (q == a) ? 1.f : 0.f;
            }
            double d10 = 0.0, d20 = 0.0, d21 = 0.0, d30 = 0.0, d31 = 0.0, d32 = 0.0;
            float dap = 0.f, sdz = 0.f;
#pragma unroll
            for (int j = 0; j < KM; ++j) {
                if (j >= k) continue;
                const float pj = p[t * k + j];
                float h[MAXCOMP], P[MAXCOMP], dpj = 0.f;
#pragma unroll
                for (int q = 0; q < MAXCOMP; ++q) {
                    h[q] = (q < K) ? hpost[(t * k + j) * K + q] : 0.f;
                    P[q] = row[L::R + j * 4 + q];
                }
#pragma unroll
                for (int a = 0; a < MAXCOMP; ++a) {
                    float e = 0.f;
#pragma unroll
                    for (int q = a; q < MAXCOMP; ++q) e += h[q] * B[q][a];
                    row[L::E + j * 4 + a] = pj * e;
                }
#pragma unroll
                for (int q = 0; q < MAXCOMP; ++q) {
                    if (q >= K) continue;
                    float pb = 0.f;
#pragma unroll
                    for (int a = 0; a <= q; ++a) pb += P[a] * B[q][a];
                    dpj += h[q] * pb;
                    // H = 2 sigma(y): dy = dH * H * (1 - H / 2)
                    const float dy = pj * pb * h[q] * (1.0f - 0.5f * h[q]);
                    const int o = j * K + q;
                    const float z = za[o], dzo = ap * dy;
                    dap += dy * (z * r);
                    sdz += dzo * z;
                    row[L::TG + o] = dy;
                    row[L::DZ + o] = dzo * r;
                }
                if (gs) {
                    // dB[q][a] = sum_j p_j H_post[j][q] P[j][a], below the diagonal
                    const double p0 = (double)P[0], p1 = (double)P[1], p2 = (double)P[2];
                    const double h1 = (double)(pj * h[1]), h2 = (double)(pj * h[2]), h3 = (double)(pj * h[3]);
                    d10 = fma(h1, p0, d10);
                    d20 = fma(h2, p0, d20);
                    d21 = fma(h2, p1, d21);
                    d30 = fma(h3, p0, d30);
                    d31 = fma(h3, p1, d31);
                    d32 = fma(h3, p2, d32);
                }
                // slots run from the last to the first: the last one stores, the others add
                dp[t * k + j] = last ? dpj : dp[t * k + j] + dpj;
            }
            row[L::TG + kK] = dap;
            row[L::S + KM] = sdz;
            double D[NGRAM];
#pragma unroll
            for (int q = 0; q < NGRAM; ++q) D[q] = 0.0;
            if (gs) G.reverse(Gm, d10, d20, d21, d30, d31, d32, D);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    row[L::D + a * 4 + b] = (float)D[a >= b ? a * (a + 1) / 2 + b : b * (b + 1) / 2 + a];
        }
    } else if (last) {
        const int tq = (tid - 32) / KM, a = (tid - 32) - tq * KM;
        const int tt = min(tq, ntok - 1);
        const long long t = t0 + tt;
        float* row = sm + tt * L::ROW;
        const float r = rs[t];
        float M[KM], z[KM], dH[KM], H[KM], dM[KM];
#pragma unroll
        for (int b = 0; b < KM; ++b) {
            const bool v = (a < k && b < k);
            z[b] = v ? zact[t * n + kK + a * k + b] : 0.f;
            M[b] = v ? ar * (z[b] * r) + b_res[a * k + b] : 0.f;
            dH[b] = v ? row[L::R + KM * 4 + a * KM + b] : 0.f;
        }
        sinkhorn_bwd<KM>(M, a, k, d.iters, sm + TB * L::ROW + (tid - 32), TB * KM, dH, H, dM);
        if (tq < ntok) {
            float sdz = 0.f, dar = 0.f;
#pragma unroll
            for (int b = 0; b < KM; ++b) {
                if (a >= k || b >= k) continue;
                const int o = kK + a * k + b;
                const float dzo = ar * dM[b];
                dar += dM[b] * (z[b] * r);
                sdz += dzo * z[b];
                row[L::TG + kK + 1 + a * k + b] = dM[b];
                row[L::DZ + o] = dzo * r;
                row[L::H + a * KM + b] = H[b];
            }
            row[L::S + a] = sdz;
            // this row's share of d alpha_res: the reductions of the row are read by no one any more
            row[L::R + KM * 4 + a * KM] = dar;
        }
    }
    __syncthreads();
    // per-token matrices and gradients, neighbouring threads on neighbouring words
    for (int e = tid; e < ntok * (KM * 4 + 16); e += nt) {
        const int tt = e / (KM * 4 + 16), q = e - tt * (KM * 4 + 16);
        const float v = sm[tt * L::ROW + L::E + q];
        if (q >= KM * 4) tokmat[(t0 + tt) * TOKMAT + 32 + q - KM * 4] = v;
        else if ((q >> 2) < k) tokmat[(t0 + tt) * TOKMAT + q] = v;
    }
    if (last)
        for (int e = tid; e < ntok * KM * KM; e += nt) {
            const int tt = e / (KM * KM), q = e - tt * KM * KM, a = q / KM, b = q - a * KM;
            if (a < k && b < k) tokmat[(t0 + tt) * TOKMAT + 48 + a * 8 + b] = sm[tt * L::ROW + L::H + q];
        }
    for (int e = tid; e < ntok * n; e += nt) {
        const int tt = e / n, o = e - tt * n;
        dzs[t0 * n + e] = sm[tt * L::ROW + L::DZ + o];
    }
    pack_dz_of<SIX>(pack, sm + L::DZ, L::ROW, n, t0, ntok);
    if (tid < ntok) {
        // active RMS: z_o = r * zraw_o, r = (sum x^2 / kC + eps)^(-1/2)
        const float* row = sm + tid * L::ROW;
        const float r = rs[t0 + tid];
        float sdz = row[L::S + KM];
        if (last)
            for (int a = 0; a < k; ++a) sdz += row[L::S + a];
        tokmat[(t0 + tid) * TOKMAT + 112] = r * r * r / (float)(k * d.C) * sdz;
    }
    // column sums over the block's tokens: [dy (k K) | d alpha_post | dM (k k) | d alpha_res]
    const int ncol = kK + 1 + (last ? k * k + 1 : 0);
    for (int c = tid; c < ncol; c += nt) {
        float s = 0.f;
        if (c <= kK + k * k) {
            for (int tt = 0; tt < ntok; ++tt) s += sm[tt * L::ROW + L::TG + c];
        } else {
            for (int tt = 0; tt < ntok; ++tt)
                for (int a = 0; a < k; ++a) s += sm[tt * L::ROW + L::R + KM * 4 + a * KM];
        }
        colp[(long long)blockIdx.x * ncol + c] = s;
    }
}

template <int KM>
cudaError_t bwd_coef_km(const Dims& d, int slot, int T, const float* red, int nslice, const float* zact,
                        const float* rs, const float* p, const float* hpost, const double* gram,
                        const float* alpha_post, const float* alpha_res, const float* b_res, float* tokmat,
                        float* dz, float* dp, float* colp, int* nblk, const DzPack& pack, const WRows& wrows,
                        cudaStream_t st) {
    // 32 tokens a block (k <= 4) fill the fp64 warp, which is what bounds the kernel at many tokens;
    // a quarter of that at few, for more blocks.  (k > 4: 16 and 4.)  The iterates of a long Sinkhorn
    // run (k > 4: more than 43 iterations; k <= 4: none of the 64 allowed) only fit with the small block.
    const bool last = (slot == d.G - 1);
    auto smem = [&](int tb) {
        return (size_t)tb * BwdTok<KM>::ROW * 4 + (last ? (size_t)d.iters * KM * tb * KM * 4 : 0);
    };
    int TB = 128 / KM;
    if (T < TB * 2 * device_sms() || smem(TB) > 200 * 1024) TB = 32 / KM;
    const size_t sm = smem(TB);
    auto* const kern = wrows.terms == 6 ? &k_bwd_coef<KM, true> : &k_bwd_coef<KM, false>;
    const cudaError_t e = smem_optin((const void*)kern, sm);
    if (e != cudaSuccess) return e;
    *nblk = (T + TB - 1) / TB;
    XHC_LAUNCH(st, *nblk + wrows_blocks(wrows, 32 + TB * KM), 32 + TB * KM, sm, (kern), d, slot, T, TB, red, nslice, zact, rs, p,
               hpost, gram, alpha_post, alpha_res, b_res, tokmat, dz, dp, colp, pack, wrows, *nblk);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_bwd_coef(const Dims& d, int slot, int T, const float* red, int nslice,
                            const float* zact, const float* rs, const float* p,
                            const float* hpost, const double* gram, const float* alpha_post,
                            const float* alpha_res, const float* b_res,
                            float* tokmat, float* dz, float* dp, float* colp, int* nblk, const DzPack& pack,
                            const WRows& wrows, cudaStream_t st) {
    if (d.k <= 4)
        return bwd_coef_km<4>(d, slot, T, red, nslice, zact, rs, p, hpost, gram, alpha_post, alpha_res, b_res,
                              tokmat, dz, dp, colp, nblk, pack, wrows, st);
    return bwd_coef_km<8>(d, slot, T, red, nslice, zact, rs, p, hpost, gram, alpha_post, alpha_res, b_res,
                          tokmat, dz, dp, colp, nblk, pack, wrows, st);
}

// ---------------------------------------------------------------------------------------------
// full_coef: reverse of coef_full.  dz columns follow zfull: [router | pre_0..].  A warp takes a token
// at a time with a lane per column, and keeps the column sums of its tokens in registers:
// [dy (G N) | dy * z * rstd (G N), summed over a slot's N columns: d alpha_pre (G) | mu dZ_r (N): the
// router logit subtracts mu * colsum(W_r), so every row of dW_r also receives -sum_t mu_t dZ_r[t]].
// scal: (d mu / NC, 2 d nu / NC), the per-token scalars of the full-state dX.  Like bwd_coef it also leaves
// dz as the bf16 operands of the tensor-core kernels, and further blocks pack their weight: five launches
// a slot fewer.

namespace {

constexpr int FC_NT = 256;
constexpr int FC_R = 4;   // pre-map columns per lane: G N <= 128

template <bool SIX>
__global__ void __launch_bounds__(FC_NT) k_full_coef(Dims d, int T, int TB, const float* dhpre,
                                                     const float* hpre,
                                                     const float* zfull,
                                                     const float* stats,
                                                     const float* wsum, const int* I,
                                                     const float* dp,
                                                     const float* alpha_pre, float* __restrict__ dz,
                                                     float* __restrict__ scal, float* __restrict__ colp,
                                                     DzPack pack, WRows wrows, int nblk) {
    pdl_entry();
    extern __shared__ float dzs[];   // [TB][n] dz, for the packed operands
    if ((int)blockIdx.x >= nblk) {
        pack_wrows_of<SIX>(wrows, (int)blockIdx.x - nblk);
        return;
    }
    __shared__ float sh[FC_NT / 32][NCOLP];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = d.N, GN = d.G * d.N, n = d.nfull, roff = d.hr ? N : 0;
    const long long t0 = (long long)blockIdx.x * TB;
    const int ntok = (int)min((long long)TB, T - t0);
    const float inv_nc = 1.0f / (float)(N * d.C);
    const float ws = (d.hr && lane < N) ? wsum[lane] : 0.f;
    float al[FC_R], sdy[FC_R], sda[FC_R], srt = 0.f;
#pragma unroll
    for (int q = 0; q < FC_R; ++q) {
        const int e = lane + 32 * q;
        al[q] = (e < GN) ? alpha_pre[e / N] : 0.f;
        sdy[q] = sda[q] = 0.f;
    }
    for (int tt = warp; tt < ntok; tt += FC_NT / 32) {
        const long long t = t0 + tt;
        const float mu = stats[t * 2], nu = stats[t * 2 + 1];
        const float rstd = 1.0f / sqrtf(nu + d.eps);
        const float* zf = zfull + t * n;
        float drstd = 0.f;
#pragma unroll
        for (int q = 0; q < FC_R; ++q) {
            const int e = lane + 32 * q;
            if (e >= GN) continue;
            const float h = hpre[t * GN + e];
            const float dy = dhpre[t * GN + e] * h * (1.0f - h);
            const float z = zf[roff + e];
            const float v = al[q] * dy * rstd;
            dz[t * n + roff + e] = v;
            dzs[tt * n + roff + e] = v;
            drstd += al[q] * dy * z;
            sdy[q] += dy;
            sda[q] += dy * (z * rstd);
        }
        drstd = warp_sum(drstd);
        float dmu = 0.f;
        float dnu = -0.5f * drstd * rstd * rstd * rstd;
        if (d.hr) {
            const float lstd = 1.0f / sqrtf(nu - mu * mu + d.eps);
            const float zc = (lane < N) ? zf[lane] - mu * ws : 0.f;
            // the routed stream of lane j, and its routing-weight gradient
            const bool rj = lane >= d.m && lane < d.k;
            const int Ij = rj ? I[t * d.k + lane] : -1;
            const float dj = rj ? dp[t * d.k + lane] : 0.f;
            float g = 0.f;
            bool sel = false;
            for (int j = d.m; j < d.k; ++j) {
                const int ij = __shfl_sync(0xffffffffu, Ij, j);
                const float gj = __shfl_sync(0xffffffffu, dj, j);
                if (ij == lane) {
                    g = gj;
                    sel = true;
                }
            }
            float dzr = 0.f;
            if (!d.softmax) {
                // sigmoid scores: only the selected routed streams' logits receive a gradient
                if (sel) {
                    const float s = sigm(zc * lstd);
                    dzr = g * s * (1.0f - s);
                }
            } else {
                // softmax scores s = softmax(z): dz_l = s_l (g_l - sum_j dp_j s_{I_j}), g_l = dp_j
                // where l = I_j is a selected routed stream, 0 elsewhere; every logit receives one
                const float zl = (lane < N) ? zc * lstd : -INFINITY;
                float zmax = zl;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
                const float ex = (lane < N) ? expf(zl - zmax) : 0.f;
                const float s = ex / warp_sum(ex);
                dzr = s * (g - warp_sum(g * s));
            }
            if (lane < N) {
                dz[t * n + lane] = dzr * lstd;
                dzs[tt * n + lane] = dzr * lstd;
            }
            srt += mu * dzr * lstd;
            dmu = -warp_sum(dzr * lstd * ws);
            const float dlstd = warp_sum(dzr * zc);
            const float l3 = lstd * lstd * lstd;
            dnu += -0.5f * dlstd * l3;
            dmu += dlstd * mu * l3;
        }
        if (lane == 0) {
            scal[t * 2] = dmu * inv_nc;
            scal[t * 2 + 1] = 2.0f * dnu * inv_nc;
        }
    }
#pragma unroll
    for (int q = 0; q < FC_R; ++q) {
        const int e = lane + 32 * q;
        if (e < GN) {
            sh[warp][e] = sdy[q];
            sh[warp][GN + e] = sda[q];
        }
    }
    if (d.hr && lane < N) sh[warp][2 * GN + lane] = srt;
    __syncthreads();
    pack_dz_of<SIX>(pack, dzs, n, n, t0, ntok);
    for (int c = tid; c < 2 * GN + roff; c += FC_NT) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < FC_NT / 32; ++w) s += sh[w][c];
        sh[0][c] = s;   // column c is this thread's alone
    }
    __syncthreads();
    const int ncol = GN + d.G + roff;
    for (int c = tid; c < ncol; c += FC_NT) {
        float s;
        if (c < GN) {
            s = sh[0][c];
        } else if (c < GN + d.G) {
            s = 0.f;
            for (int i = 0; i < N; ++i) s += sh[0][GN + (c - GN) * N + i];
        } else {
            s = sh[0][GN - d.G + c];
        }
        colp[(long long)blockIdx.x * ncol + c] = s;
    }
}

}  // namespace

cudaError_t launch_full_coef(const Dims& d, int T, const float* dhpre, const float* hpre,
                             const float* zfull, const float* stats, const float* wsum,
                             const int* I, const float* dp, const float* alpha_pre, float* dz,
                             float* scal, float* colp, int* nblk, const DzPack& pack, const WRows& wrows,
                             cudaStream_t st) {
    // 8 tokens a block (a token per warp) at few tokens, 32 at many
    const int TB = (T >= 32 * 2 * device_sms()) ? 32 : 8;
    *nblk = (T + TB - 1) / TB;
    auto* const kern = wrows.terms == 6 ? &k_full_coef<true> : &k_full_coef<false>;
    XHC_LAUNCH(st, *nblk + wrows_blocks(wrows, FC_NT), FC_NT, (size_t)TB * d.nfull * 4, (kern), d, T, TB, dhpre, hpre, zfull,
               stats, wsum, I, dp, alpha_pre, dz, scal, colp, pack, wrows, *nblk);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// colsum_out: the block partials' column sums into their targets; a block per output

namespace {

__global__ void __launch_bounds__(128) k_colsum_out(const float* colp, int nblk, int ncol, ColOut out) {
    pdl_entry();
    __shared__ float sh[4];
    int o = blockIdx.x;
    // the target of output o, selected with static indices
    float* ptr = nullptr;
    int off = 0, set = 0;
    bool found = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (!found) {
            if (o < out.n[q]) {
                ptr = out.ptr[q] + o;
                off = out.off[q] + o;
                set = out.set[q];
                found = true;
            } else {
                o -= out.n[q];
            }
        }
    }
    float s = warp_sum(slot_sum<8>(colp + off, ncol, nblk, threadIdx.x, 128));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        const float v = (sh[0] + sh[1]) + (sh[2] + sh[3]);
        *ptr = set ? v : *ptr + v;
    }
}

}  // namespace

cudaError_t launch_colsum_out(const float* colp, int nblk, int ncol, const ColOut& out, cudaStream_t st) {
    int n = 0;
    for (int q = 0; q < 4; ++q) n += out.n[q];
    XHC_LAUNCH(st, n, 128, 0, (k_colsum_out), colp, nblk, ncol, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// wgrad_reduce: G[e][o] += sum over the slots of wpart[slot][e][o].  A block column takes one 128-row
// tile of the plan, so the number of slots is found once per block.

namespace {

__global__ void __launch_bounds__(256) k_wgrad_reduce(const float* wpart, SlotPlan sp, int E, int n,
                                                      WSegsOut G, const float* sub) {
    pdl_entry();
    const int e0 = blockIdx.y * 128, ne = min(128, E - e0) * n;
    const int nsl = slot_count(sp, blockIdx.y);
    for (int idx = blockIdx.x * 256 + threadIdx.x; idx < ne; idx += gridDim.x * 256) {
        float s = slot_sum<4>(wpart + (long long)e0 * n + idx, (long long)E * n, nsl, 0, 1);
        const int e = e0 + idx / n, o = idx % n;
        // the segment of column o, selected with static indices (no local copy of the parameter)
        float* p = G.ptr[0];
        int width = G.width[0], off = G.off[0];
        if (sub != nullptr && o < G.off[1]) s -= sub[o];
#pragma unroll
        for (int q = 1; q < MAXSEG; ++q)
            if (q < G.n && o >= G.off[q]) {
                p = G.ptr[q];
                width = G.width[q];
                off = G.off[q];
            }
        p[(long long)e * width + (o - off)] += s;
    }
}

}  // namespace

cudaError_t launch_wgrad_reduce(const float* wpart, const SlotPlan& sp, int E, int n, const WSegsOut& G,
                                const float* sub, cudaStream_t st) {
    // a few elements a thread where there are many tiles (the slot count costs a division)
    const int tiles = (E + 127) / 128, per = (128 * n + 255) / 256;
    const dim3 grid((unsigned)std::max(1, tiles >= 256 ? per / 8 : per), (unsigned)tiles);
    XHC_LAUNCH(st, grid, 256, 0, (k_wgrad_reduce), wpart, sp, E, n, G, sub);
    return cudaGetLastError();
}

}  // namespace xhc
