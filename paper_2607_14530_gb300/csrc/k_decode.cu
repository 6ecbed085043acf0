// Decode: the write-back of a slot for one new token per sequence.
//
// In decoding, token t of the call is the next token of its own sequence b = t, at position
// pos[t] of that sequence.  The causal conv of Eq. aug (Sec. 3.3.4: g_j[s] = sum_{i < kappa_j}
// w_j[i] out[s - i], zero before the sequence start) needs the R = max(kappa) - 1 previous `out`
// rows of the sequence, which no longer exist as a contiguous [T][C] buffer: they are kept in a
// per-sequence ring [B][R][C] bf16 (row (s mod R) holds out[s]).
//
// One kernel does a slot's write-back (Eq. gs, Eq. sparse_write_delta, Eq. sparse_write): a cluster of
// up to 8 CTAs takes DT tokens, its CTAs the channel slices.  Each CTA forms the conv components of
// its channels once and keeps them in shared memory; the CTAs exchange their Gram partials through
// distributed shared memory, CTA (token mod cluster size) turns a token's Gram matrix into the
// coefficients E and hands them back, and every CTA applies them to its channels, stores the token's
// `out` in its ring row, and on the group's last slot the cluster advances pos.  Bound by latency: the
// loads of a token's 12 conv rows and 24 taps are issued together, and of the three launches before
// (Gram reduction, coefficients, write-back with the conv over again) one is left.
#include <algorithm>
#include <utility>

#include <cooperative_groups.h>

#include "xhc_internal.cuh"

namespace xhc {
namespace {

namespace cg = cooperative_groups;

constexpr int DSL = 256;     // channels of a slice: 128 threads, a channel pair each
constexpr int DMAXC = 8;     // CTAs of a cluster
constexpr int DMAXT = 8;     // tokens of a cluster

__device__ __forceinline__ float2 ldp(const uint16_t* p) {
    const uint32_t u = *reinterpret_cast<const uint32_t*>(p);
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

// the conv components of channels (c, c + 1): g_j = sum_i w_j[i] out[pos - i], i ascending.  KW: most
// taps of a component; PAPER: the (4, 8, 12) taps, their loops folded.  pos: the position, at most KW
// of it; r0: its ring row.
template <int KW, bool PAPER>
__device__ __forceinline__ void dec_conv(const Dims& d, const ConvPtrs& cw, const uint16_t* rt, int c,
                                         float2 o, int pos, int r0, float2 (&g)[3]) {
    const int C = d.C, R = d.kapmax - 1;
    float2 v[KW];
    v[0] = o;
#pragma unroll
    for (int i = 1; i < KW; ++i) {
        int r = r0 - i;                              // row of position pos - i (i <= R)
        if (r < 0) r += R;
        v[i] = (i < d.kapmax && i <= pos) ? ldp(rt + (long long)r * C) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        g[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < KW; ++i) {
            if (PAPER ? i >= 4 * (j + 1) : (j >= d.nconv || i >= d.kap[j])) break;
            float2 w = make_float2(0.f, 0.f);        // no term before the sequence start
            if (i <= pos) w = make_float2(cw.w[j][(size_t)i * C + c], cw.w[j][(size_t)i * C + c + 1]);
            g[j].x = fmaf(w.x, v[i].x, g[j].x);
            g[j].y = fmaf(w.y, v[i].y, g[j].y);
        }
    }
}

// shared memory of a CTA (dynamic), DT tokens and q slices of its own, ns slices in all
struct DecSmem {
    int u, wred, gpart, gs, bs, e, h, bytes;
    __host__ __device__ DecSmem(int DT, int q, int ns, int k, bool conv) {
        int o = 0;
        gs = o; o += DT * 12 * 8;                            // f64 [DT][12]: Gram matrices (this rank's tokens)
        u = o; o += conv ? DT * q * 3 * 128 * 8 : 0;         // float2 [DT][q][3][128]: conv components
        wred = o; o += conv ? DT * q * 4 * 10 * 4 : 0;       // f32 [DT][q][4 warps][10]
        gpart = o; o += conv ? DT * ns * 10 * 4 : 0;         // f32 [DT][ns][10]: Gram partials (this rank's tokens)
        bs = o; o += DT * 16 * 4;                            // f32 [DT][4][4]: coefficients B
        e = o; o += DT * k * 4 * 4;                          // f32 [DT][k][4]: E
        h = o; o += DT * k * k * 4;                          // f32 [DT][k][k]: H_res (last slot)
        bytes = o;
    }
};

// warp reduce-scatter of 16 values: every lane returns the total of value lane >> 1
__device__ __forceinline__ float wred16(float (&v)[16], int lane) {
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = (lane & (2 * h)) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const float send = up ? v[q] : v[q + h], keep = up ? v[q + h] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// KM: most active slots; KW, PAPER: see dec_conv; KW = 0: a slot without conv (no exchange, so the
// CTAs of a token need no cluster)
template <int KM, int KW, bool PAPER>
__global__ void __launch_bounds__(512, 2) k_dec_post(Dims d, int slot, int B, int DT, int q, int ns,
                                                  const uint16_t* out, ConvPtrs cw,
                                                  uint16_t* ring, long long* pos,
                                                  const float* p, const float* hpost,
                                                  double* __restrict__ gram, const uint16_t* xact,
                                                  const int* I, const float* hres,
                                                  uint16_t* __restrict__ xact_next, uint16_t* __restrict__ X) {
    pdl_entry();
    constexpr bool CONV = KW > 0;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long ps[DMAXT];
    __shared__ int rows[DMAXT];
    const int C = d.C, k = d.k, K = d.K[slot], R = d.kapmax - 1;
    const bool last = (slot == d.G - 1);
    const DecSmem L(DT, q, ns, k, CONV);
    double* Gs = reinterpret_cast<double*>(smem + L.gs);
    float2* us = reinterpret_cast<float2*>(smem + L.u);
    float* wr = reinterpret_cast<float*>(smem + L.wred);
    float* gp = reinterpret_cast<float*>(smem + L.gpart);
    float* Bs = reinterpret_cast<float*>(smem + L.bs);
    float* Es = reinterpret_cast<float*>(smem + L.e);
    float* Hs = reinterpret_cast<float*>(smem + L.h);
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int sl = tid >> 7, st = tid & 127;         // slice of this thread in a step, its place there
    const int nsl = nt >> 7;                         // slices at a time
    const int t0 = blockIdx.x * DT, ntok = min(DT, B - t0);
    const int rank = blockIdx.y, nr = gridDim.y;     // CTA of the cluster, and their number
    const int s0 = rank * q, sn = min(q, ns - s0);   // this CTA's slices
    if ((CONV || rank == 0) && tid < ntok) {
        const long long v = pos[t0 + tid];
        ps[tid] = v;
        rows[tid] = R > 0 ? (int)(v % R) : 0;        // ring row of the position
    }
    if (last)
        for (int e = tid; e < ntok * k * k; e += nt) Hs[e] = hres[(long long)t0 * k * k + e];
    __syncthreads();
    if constexpr (CONV) {
        cg::cluster_group cl = cg::this_cluster();
        auto started = cl.barrier_arrive();   // waited for before the first access to another CTA
        // the conv components, and the Gram partials of each slice (lower triangle, the order of the
        // prefill's reduction)
        for (int tt = 0; tt < ntok; ++tt) {
            const long long t = t0 + tt;
            for (int s = sl; s < sn; s += nsl) {
                const int c = (s0 + s) * DSL + 2 * st;
                float2 uu[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if (c < C) {
                    uu[0] = ldp(out + t * C + c);
                    float2 g[3];
                    dec_conv<KW, PAPER>(d, cw, ring + t * R * C + c, c, uu[0], (int)min(ps[tt], (long long)KW), rows[tt], g);
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        uu[1 + j] = g[j];
                        us[((tt * q + s) * 3 + j) * 128 + st] = g[j];
                    }
                }
                if (d.gs) {
                    float v[16];
                    int e = 0;
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b <= a; ++b, ++e) v[e] = fmaf(uu[a].x, uu[b].x, uu[a].y * uu[b].y);
#pragma unroll
                    for (; e < 16; ++e) v[e] = 0.f;
                    const float tot = wred16(v, lane);
                    if ((lane & 1) == 0 && lane < 20) wr[((tt * q + s) * 4 + (st >> 5)) * 10 + (lane >> 1)] = tot;
                }
            }
        }
        __syncthreads();
        cl.barrier_wait(std::move(started));
        if (d.gs) {
            // each slice's partial to the CTA that owns the token
            for (int e = tid; e < ntok * sn * 10; e += nt) {
                const int tt = e / (sn * 10), r = e - tt * sn * 10, s = r / 10, x = r - s * 10;
                const float* w = wr + (tt * q + s) * 40 + x;
                float* dst = cl.map_shared_rank(gp, tt % nr);
                dst[(tt * ns + s0 + s) * 10 + x] = ((w[0] + w[10]) + w[20]) + w[30];
            }
            cl.sync();
            for (int e = tid; e < ntok * NGRAM; e += nt) {
                const int tt = e / NGRAM, x = e - tt * NGRAM;
                if (tt % nr != rank) continue;
                double s = 0.0;
                if (x < K * (K + 1) / 2) {
                    for (int g = 0; g < ns; ++g) s += (double)gp[(tt * ns + g) * 10 + x];
                    gram[(long long)(t0 + tt) * NGRAM + x] = s;
                }
                Gs[tt * 12 + x] = s;
            }
            __syncthreads();
        }
        if (tid < ntok && (tid % nr == rank)) {
            float Bm[MAXCOMP][MAXCOMP];
            if (d.gs) {
                double Gm[NGRAM];
#pragma unroll
                for (int x = 0; x < NGRAM; ++x) Gm[x] = Gs[tid * 12 + x];
                GramSchmidt G;
                G.forward(Gm, (double)d.eps_gs);
                G.coef(Bm);
            }
#pragma unroll
            for (int a = 0; a < MAXCOMP; ++a)
#pragma unroll
                for (int b = 0; b < MAXCOMP; ++b) Bs[tid * 16 + a * 4 + b] = d.gs ? Bm[a][b] : (a == b ? 1.f : 0.f);
        }
        __syncthreads();
        // E[j][a] = p_j sum_b H_post[j][b] B[b][a] to every CTA of the cluster
        for (int e = tid; e < ntok * k * 4 * nr; e += nt) {
            const int to = e / (ntok * k * 4), r = e - to * ntok * k * 4;
            const int tt = r / (k * 4), j = (r >> 2) % k, a = r & 3;
            if (tt % nr != rank) continue;
            const long long tj = (long long)(t0 + tt) * k + j;
            float v = 0.f;
            for (int b = a; b < K; ++b) v += hpost[tj * K + b] * Bs[tt * 16 + b * 4 + a];
            cl.map_shared_rank(Es, to)[r] = p[tj] * v;
        }
        cl.sync();
    } else {
        for (int e = tid; e < ntok * k; e += nt) {
            const long long tj = (long long)t0 * k + e;
            Es[e * 4] = p[tj] * hpost[tj];
        }
        __syncthreads();
    }
    // X_act_new_j = (H_res x_act)_j (last slot) or x_act_j, + sum_a E[j][a] u_a; the last slot scatters
    // into the state rows I_j, the others write the next slot's active state
    for (int tt = 0; tt < ntok; ++tt) {
        const long long t = t0 + tt;
        for (int s = sl; s < sn; s += nsl) {
            const int c = (s0 + s) * DSL + 2 * st;
            if (c >= C) continue;
            float2 x[KM], uu[4];
#pragma unroll
            for (int j = 0; j < KM; ++j) x[j] = (j < k) ? ldp(xact + (t * k + j) * C + c) : make_float2(0.f, 0.f);
            const uint32_t raw = *reinterpret_cast<const uint32_t*>(out + t * C + c);
            uu[0] = make_float2(__uint_as_float(raw << 16), __uint_as_float(raw & 0xffff0000u));
            if constexpr (CONV) {
#pragma unroll
                for (int j = 0; j < 3; ++j) uu[1 + j] = us[((tt * q + s) * 3 + j) * 128 + st];
            }
#pragma unroll
            for (int j = 0; j < KM; ++j) {
                if (j >= k) break;
                float2 v = x[j];
                if (last) {
                    v = make_float2(0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < KM; ++i) {
                        if (i >= k) break;
                        const float h = Hs[(tt * k + j) * k + i];
                        v.x = fmaf(h, x[i].x, v.x);
                        v.y = fmaf(h, x[i].y, v.y);
                    }
                }
                const float* E = Es + (tt * k + j) * 4;
#pragma unroll
                for (int a = 0; a < (CONV ? 4 : 1); ++a) {
                    v.x = fmaf(E[a], uu[a].x, v.x);
                    v.y = fmaf(E[a], uu[a].y, v.y);
                }
                uint16_t* dst = last ? X + (t * d.N + I[t * k + j]) * C + c : xact_next + (t * k + j) * C + c;
                *reinterpret_cast<uint32_t*>(dst) = pack2(v.x, v.y);
            }
            if (CONV && R > 0) *reinterpret_cast<uint32_t*>(ring + (t * R + rows[tt]) * C + c) = raw;
        }
    }
    // the conv's CTAs have all read pos (before their last cluster barrier); without conv only this one does
    if (last && rank == 0 && tid < ntok) pos[t0 + tid] = ps[tid] + 1;
}

template <int KM, int KW, bool PAPER>
cudaError_t dec_post_kw(const Dims& d, int slot, int B, const uint16_t* out, ConvPtrs cw, uint16_t* ring,
                        long long* pos, const float* p, const float* hpost, double* gram, const uint16_t* xact,
                        const int* I, const float* hres, uint16_t* xact_next, uint16_t* X, cudaStream_t st) {
    constexpr bool CONV = KW > 0;
    const int ns = (d.C + DSL - 1) / DSL;
    const int q = (ns + DMAXC - 1) / DMAXC, nr = (ns + q - 1) / q;   // slices a CTA, CTAs a cluster
    const int nt = std::min(q, 4) * 128;
    // as many tokens a cluster as fill the GPU once (1024 threads per SM: more clusters would wait for
    // the 8 free CTA places of a GPC), and their components within 64 KB.  256 tokens of C = 4096: 4
    // tokens a cluster; with 7 and half the threads resident it took 48 us, and three kernels 70.
    const long long cap = (long long)(1024 / nt) * device_sms();
    int DT = std::min(DMAXT, std::max(1, (int)(((long long)B * nr + cap - 1) / cap)));
    while (DT > 1 && CONV && DT * q * 3 * 128 * 8 > 64 * 1024) --DT;
    const DecSmem L(DT, q, ns, d.k, CONV);
    cudaError_t e = smem_optin((const void*)k_dec_post<KM, KW, PAPER>, L.bytes);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((B + DT - 1) / DT), (unsigned)nr);
    cfg.blockDim = dim3((unsigned)nt);
    cfg.dynamicSmemBytes = (size_t)L.bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = CONV ? (unsigned)nr : 1u;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl_on() ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, k_dec_post<KM, KW, PAPER>, d, slot, B, DT, q, ns, out, cw, ring, pos, p, hpost, gram,
                           xact, I, hres, xact_next, X);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int KM>
cudaError_t dec_post_km(const Dims& d, int slot, int B, const uint16_t* out, ConvPtrs cw, uint16_t* ring,
                        long long* pos, const float* p, const float* hpost, double* gram, const uint16_t* xact,
                        const int* I, const float* hres, uint16_t* xact_next, uint16_t* X, cudaStream_t st) {
#define XHC_DEC(KW_, PAPER_) \
    dec_post_kw<KM, KW_, PAPER_>(d, slot, B, out, cw, ring, pos, p, hpost, gram, xact, I, hres, xact_next, X, st)
    if (d.K[slot] <= 1) return XHC_DEC(0, false);
    if (d.nconv == 3 && d.kap[0] == 4 && d.kap[1] == 8 && d.kap[2] == 12) return XHC_DEC(12, true);
    if (d.kapmax <= 8) return XHC_DEC(8, false);
    return XHC_DEC(16, false);
#undef XHC_DEC
}

// ring rows from a prefill: sequence b of S tokens (rows b*S .. b*S + S - 1 of out) leaves its
// last min(S, R) rows in ring rows (s mod R)
__global__ void k_ring_fill(const uint16_t* out, int B, int S, int C, int R,
                            uint16_t* __restrict__ ring) {
    pdl_entry();
    const long long n = (long long)B * R * (C / 8);
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int c8 = (int)(idx % (C / 8));
        const long long r = idx / (C / 8);
        const int lag = (int)(r % R) + 1;           // 1..R: token S - lag
        const int b = (int)(r / R);
        const long long s = (long long)S - lag;
        if (s < 0) continue;
        *reinterpret_cast<uint4*>(ring + ((long long)b * R + (int)(s % R)) * C + c8 * 8) =
            *reinterpret_cast<const uint4*>(out + ((long long)b * S + s) * C + c8 * 8);
    }
}

// halo rows for the next chunk of B sequences of S tokens: halo[b][r] = out of position
// S - R + r of sequence b (zero where that position is before the sequence start)
__global__ void k_halo_fill(const uint16_t* out, int B, int S, int C, int R,
                            uint16_t* __restrict__ halo) {
    pdl_entry();
    const long long n = (long long)B * R * (C / 8);
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int c8 = (int)(idx % (C / 8));
        const long long br = idx / (C / 8);
        const int r = (int)(br % R);
        const long long b = br / R;
        const long long s = (long long)S - R + r;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (s >= 0) v = *reinterpret_cast<const uint4*>(out + (b * S + s) * C + c8 * 8);
        *reinterpret_cast<uint4*>(halo + br * C + c8 * 8) = v;
    }
}

// the gradient of a chunk's halo rows, returned to the chunk that produced them: d_out of
// position S - R + r of sequence b += d_halo[b][r] (in fp32, one bf16 rounding)
__global__ void k_halo_add(uint16_t* d_out, int B, int S, int C, int R,
                           const float* dhalo) {
    pdl_entry();
    const long long n = (long long)B * R * (C / 2);
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int c2 = (int)(idx % (C / 2));
        const long long br = idx / (C / 2);
        const int r = (int)(br % R);
        const long long b = br / R;
        const long long s = (long long)S - R + r;
        if (s < 0) continue;
        uint32_t* p = reinterpret_cast<uint32_t*>(d_out + (b * S + s) * C + c2 * 2);
        const float2 g = *reinterpret_cast<const float2*>(dhalo + br * C + c2 * 2);
        const uint32_t u = *p;
        *p = pack2(__uint_as_float(u << 16) + g.x, __uint_as_float(u & 0xffff0000u) + g.y);
    }
}

}  // namespace

cudaError_t launch_dec_post(const Dims& d, int slot, int B, const uint16_t* out, ConvPtrs cw,
                            uint16_t* ring, long long* pos, const float* p, const float* hpost, double* gram,
                            const uint16_t* xact, const int* I, const float* hres, uint16_t* xact_next,
                            uint16_t* X, cudaStream_t st) {
    if (d.k <= 4)
        return dec_post_km<4>(d, slot, B, out, cw, ring, pos, p, hpost, gram, xact, I, hres, xact_next, X, st);
    return dec_post_km<8>(d, slot, B, out, cw, ring, pos, p, hpost, gram, xact, I, hres, xact_next, X, st);
}

cudaError_t launch_ring_fill(const Dims& d, int B, int S, const uint16_t* out, uint16_t* ring,
                             cudaStream_t st) {
    const int R = d.kapmax - 1;
    if (R <= 0) return cudaSuccess;
    const long long n = (long long)B * R * (d.C / 8);
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    XHC_LAUNCH(st, blocks, 256, 0, (k_ring_fill), out, B, S, d.C, R, ring);
    return cudaGetLastError();
}

cudaError_t launch_halo_fill(const Dims& d, int B, int S, const uint16_t* out, uint16_t* halo,
                             cudaStream_t st) {
    const int R = d.kapmax - 1;
    if (R <= 0) return cudaSuccess;
    const long long n = (long long)B * R * (d.C / 8);
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    XHC_LAUNCH(st, blocks, 256, 0, (k_halo_fill), out, B, S, d.C, R, halo);
    return cudaGetLastError();
}

cudaError_t launch_halo_add(const Dims& d, int B, int S, uint16_t* d_out, const float* dhalo,
                            cudaStream_t st) {
    const int R = d.kapmax - 1;
    if (R <= 0) return cudaSuccess;
    const long long n = (long long)B * R * (d.C / 2);
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    XHC_LAUNCH(st, blocks, 256, 0, (k_halo_add), d_out, B, S, d.C, R, dhalo);
    return cudaGetLastError();
}

}  // namespace xhc
