// Launchers of the forward write-back kernels (wb_gram, wb_coef, wb_fwd).
#include "k_wb.cuh"

namespace xhc {
namespace {

// ---------------------------------------------------------------------------------------------
// wb_coef: with Gram-Schmidt, the slice partials of the Gram matrix are summed in fp64, kept in `gram`
// for the backward and turned into the coefficients B of Eq. gs (orthogonalised component q = sum_a
// B[q][a] u_a), so that the write-back of active slot j is sum_a E[j][a] u_a with E[j][a] = p_j sum_q
// H_post[j][q] B[q][a]; without it B is the identity.  E goes to the per-token matrix buffer (rows
// j < k, four entries each).  Slots without a conv (K = 1, E[j][0] = p_j H_post[j]) form it in wb_fwd8
// instead, a launch less: T = 8192, N = 4, one slot: 6 us of 762; T = 1536, four slots: 3.4 of 293.
// A block takes TB <= 32 tokens: a thread per (token, Gram entry) for the sums, a lane per token for the
// coefficients, a thread per (token, entry of E).

constexpr int WC_NT = 128;

__global__ void __launch_bounds__(WC_NT) k_wb_coef(Dims d, int slot, int T, int TB, const float* red,
                                                   int nslice, const float* p,
                                                   const float* hpost,
                                                   double* __restrict__ gram, float* __restrict__ emat) {
    pdl_entry();
    __shared__ double Gs[32][NGRAM + 1];
    __shared__ float Bs[32][MAXCOMP * MAXCOMP + 1];
    const int tid = threadIdx.x, k = d.k, K = d.K[slot];
    const bool gs = (K > 1) && d.gs;
    const long long t0 = (long long)blockIdx.x * TB;
    const int ntok = (int)min((long long)TB, T - t0);
    if (gs) {
        const int nq = K * (K + 1) / 2;
        for (int e = tid; e < ntok * NGRAM; e += WC_NT) {
            const int tt = e / NGRAM, q = e - tt * NGRAM;
            const float* rp = red + (t0 + tt) * nslice * NRED + q;
            double s = 0.0;
            if (q < nq) {
#pragma unroll 8
                for (int sl = 0; sl < nslice; ++sl) s += (double)rp[sl * NRED];
                gram[t0 * NGRAM + e] = s;
            }
            Gs[tt][q] = s;
        }
        __syncthreads();
    }
    if (tid < ntok) {
        float B[MAXCOMP][MAXCOMP];
        if (gs) {
            double Gm[NGRAM];
#pragma unroll
            for (int q = 0; q < NGRAM; ++q) Gm[q] = Gs[tid][q];
            GramSchmidt G;
            G.forward(Gm, (double)d.eps_gs);
            G.coef(B);
        }
#pragma unroll
        for (int q = 0; q < MAXCOMP; ++q)
#pragma unroll
            for (int a = 0; a < MAXCOMP; ++a) Bs[tid][q * MAXCOMP + a] = gs ? B[q][a] : (q == a ? 1.f : 0.f);
    }
    __syncthreads();
    for (int e = tid; e < ntok * k * 4; e += WC_NT) {
        const int tt = e / (k * 4), q4 = e - tt * k * 4, j = q4 >> 2, a = q4 & 3;
        const long long tj = (t0 + tt) * k + j;
        float v = 0.f;
        for (int q = a; q < K; ++q) v += hpost[tj * K + q] * Bs[tt][q * MAXCOMP + a];
        emat[(t0 + tt) * TOKMAT + q4] = p[tj] * v;
    }
}

template <int KW, int KS>
cudaError_t gram_kw(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw, int nslice,
                    float* red, cudaStream_t st) {
    const int TB = pick_run(d, T, true, nslice, 4, 12, 64);
    const size_t sm = (size_t)TB * (WT / 32) * 16 * sizeof(float);
    cudaError_t e = smem_optin((const void*)k_wb_gram<KW, KS>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid(nslice, (unsigned)n_runs(d, T, TB, true));
    XHC_LAUNCH(st, grid, WT, sm, (k_wb_gram<KW, KS>), d, slot, T, TB, out, cw, nslice, red);
    return cudaGetLastError();
}

template <int KM, int KW, int KS>
cudaError_t fwd_kw(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw, const float* emat,
                   int nslice, const uint16_t* xact, const int* I, const float* hres,
                   uint16_t* xact_next, uint16_t* X, cudaStream_t st) {
    // 128 measured faster than 96 with the block ring
    const int TB = pick_run(d, T, true, nslice, KM == 4 ? 4 : 3, 12, 128);
    const size_t sm = sizeof(FRing<KM>) + (size_t)TB * (KM * 4 + KM * KM + KM) * 4;
    cudaError_t e = smem_optin((const void*)k_wb_fwd<KM, KW, KS>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid(nslice, (unsigned)n_runs(d, T, TB, KW > 0));
    XHC_LAUNCH(st, grid, WT, sm, (k_wb_fwd<KM, KW, KS>), d, slot, T, TB, out, cw, emat, xact, I, hres, xact_next, X);
    return cudaGetLastError();
}

template <int KM>
cudaError_t fwd8_kw(const Dims& d, int slot, int T, const uint16_t* out, const float* p, const float* hpost,
                    const uint16_t* xact, const int* I, const float* hres, uint16_t* xact_next,
                    uint16_t* X, cudaStream_t st) {
    const int TB = pick_run(d, T, false, (d.C + W8 - 1) / W8, KM == 4 ? 6 : 3, 4, 32);
    const size_t sm = (size_t)TB * (KM + KM * KM + KM) * 4;
    dim3 grid((d.C + W8 - 1) / W8, (T + TB - 1) / TB);
    XHC_LAUNCH(st, grid, WT, sm, (k_wb_fwd8<KM>), d, slot, T, TB, out, p, hpost, xact, I, hres, xact_next, X);
    return cudaGetLastError();
}

}  // namespace

int wb_nslice(int C) { return (C + WSL - 1) / WSL; }
int wb_conv_runs(const Dims& d, int64_t T) {
    return (int)n_runs(d, T, bapp_run(d, T), true);
}

// the two-pair Gram kernel: the (4, 8, 12) taps and C a multiple of WSL2
static bool gram2_ok(const Dims& d) { return paper_kaps(d) && d.C % WSL2 == 0; }

// partial-sum slices per token of the Gram kernel (read back by wb_coef)
int wb_gram_slices(const Dims& d) { return gram2_ok(d) ? d.C / WSL2 : wb_nslice(d.C); }

cudaError_t launch_wb_gram(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                           int nslice, float* red, cudaStream_t st) {
    if (gram2_ok(d)) {
        const int TB = pick_run(d, T, true, d.C / WSL2, 2, 12, 64);
        const size_t sm = (size_t)TB * (WT / 32) * 16 * sizeof(float);
        dim3 grid(d.C / WSL2, (unsigned)n_runs(d, T, TB, true));
        XHC_LAUNCH(st, grid, WT, sm, (k_wb_gram2), d, slot, T, TB, out, cw, nslice, red);
        return cudaGetLastError();
    }
    XHC_KW_DISPATCH(d, d.C % WSL == 0, (gram_kw<KWC, KSC>(d, slot, T, out, cw, nslice, red, st)));
}

cudaError_t launch_wb_coef(const Dims& d, int slot, int T, const float* red, int nslice, const float* p,
                           const float* hpost, double* gram, float* emat, cudaStream_t st) {
    // full fp64 warps at many tokens, more blocks at few
    const int TB = (T >= 32 * device_sms()) ? 32 : 8;
    XHC_LAUNCH(st, (T + TB - 1) / TB, WC_NT, 0, (k_wb_coef), d, slot, T, TB, red, nslice, p, hpost, gram, emat);
    return cudaGetLastError();
}

cudaError_t launch_wb_fwd(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                          const float* emat, const float* p, const float* hpost, int nslice,
                          const uint16_t* xact, const int* I, const float* hres, uint16_t* xact_next, uint16_t* X,
                          cudaStream_t st) {
    const bool conv = d.K[slot] > 1;
    if (d.k <= 4) {
        if (!conv) return fwd8_kw<4>(d, slot, T, out, p, hpost, xact, I, hres, xact_next, X, st);
        XHC_KW_DISPATCH(d, wb_fast(d), (fwd_kw<4, KWC, KSC>(d, slot, T, out, cw, emat, nslice, xact, I, hres, xact_next, X, st)));
    }
    if (!conv) return fwd8_kw<8>(d, slot, T, out, p, hpost, xact, I, hres, xact_next, X, st);
    XHC_KW_DISPATCH(d, false, (fwd_kw<8, KWC, KSC>(d, slot, T, out, cw, emat, nslice, xact, I, hres, xact_next, X, st)));
}

}  // namespace xhc
