// Internal declarations of libxhc: dimensions, buffer layout, device helpers, launchers.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/xhc.h"

namespace xhc {

constexpr int MAXN = 32;     // streams
constexpr int MAXK = 8;      // active streams
constexpr int MAXKAP = 16;   // conv kernel size
constexpr int MAXCOMP = 4;   // write-back components (1 + r)
constexpr int MAXSEG = 5;    // weight segments of one projection (router + 4 pre-maps)

// Everything a kernel needs to know about the group's shape (passed by value).
struct Dims {
    int N, k, m, C, G;
    int hr;              // 1 if the group has a router (m < k)
    int nfull;           // columns of the full-state projection: (hr ? N : 0) + G * N
    int S;               // sequence length
    int iters;           // Sinkhorn iterations
    float eps;           // norm epsilon
    float eps_gs;        // Gram-Schmidt epsilon (already resolved)
    int gs;              // Gram-Schmidt on/off
    int nconv;           // conv branches r
    int kap[3];          // kernel sizes
    int kapmax;          // max kernel size
    int kapsum;          // sum of kernel sizes
    int K[4];            // write-back components per slot
    int nact[4];         // active projection width per slot: k*K_t (+ k*k for the last slot)
    int softmax;         // router scores: 0 sigmoid (Eq. router), 1 softmax over the N logits
    int dense;           // 1: dense read of all N streams (Eq. dense_read); 0: active streams only
};

// Column segments of a projection weight: column o of the logical [rows, n] matrix lives in
// segment s with off[s] <= o < off[s+1] at ptr[s][row * width[s] + (o - off[s])].
struct WSegs {
    const float* ptr[MAXSEG];
    int width[MAXSEG];
    int off[MAXSEG + 1];
    int n;  // number of segments
};
struct WSegsOut {
    float* ptr[MAXSEG];
    int width[MAXSEG];
    int off[MAXSEG + 1];
    int n;
};

// Stream-K plan of the tensor-core full-state projection.
struct ProjTcPlan {
    int KB, MT;      // k-blocks per tile, token tiles
    long long W;     // total k-blocks
    int P;           // persistent CTAs
    int nseg;        // partial slots per tile
    int NB;          // B rows (hi + lo + pad)
    int nchunk;      // MMA instructions per k-step
    int kps;         // k-blocks of 64 per stage
    int ctas;        // CTAs per SM
};
ProjTcPlan plan_proj_tc(int T, int K, int nfull, int nsm, bool proj);  // proj: A = X rows (else weight gradient)
int device_sms();

// Partial slots of a split reduction: `n` of them for every row, or (n == 0) those of a stream-K plan,
// whose persistent CTAs cover each 128-row tile with a number of segments of its own.
struct SlotPlan {
    long long W;
    int P, KB, n;
};
inline SlotPlan slots_of(const ProjTcPlan& p) { return SlotPlan{p.W, p.P, p.KB, 0}; }
inline SlotPlan slots_of(int n) { return SlotPlan{0, 0, 0, n}; }

// Byte offsets of the per-group buffers for a given T (all 256-byte aligned).
struct Layout {
    // saved
    size_t xact;            // bf16 [G][T][k][C]: active state entering slot t
    size_t I;               // int32 [T][k]
    size_t p;               // f32 [T][k]
    size_t stats;           // f32 [T][2]: mu, nu of the flattened entry state
    size_t zfull;           // f32 [T][nfull]: raw projections x W
    size_t hpre;            // f32 [T][G][N]
    size_t zact[4];         // f32 [T][nact_t]: raw active projections
    size_t rs[4];           // f32 [T]: active rstd
    size_t hpost[4];        // f32 [T][k*K_t]
    size_t hres;            // f32 [T][k*k]
    size_t wsum;            // f32 [N]: column sums of W_r (left by the forward for the backward)
    size_t gram[4];         // f64 [T][NGRAM]: Gram matrix of the write-back components (lower
                            // triangle), slots with a temporal conv and Gram-Schmidt
    size_t saved_total;
    // workspace
    size_t err;             // int: device error word (first 256 bytes of the workspace)
    size_t wpack;           // bf16 [NB][N*C]: hi / lo rows of the full-state projection weight
    size_t wpacka;          // bf16 [NB][k*C]: hi / lo rows of a slot's active-state projection weight
    size_t part;            // f32 [splits][T][nmax] projection split-K partials
    size_t pstats;          // f32 [splits][T][2]
    size_t astat;           // f32 [stream_warps(C)][T][2]: per-warp partial sums of squares (at 1;
                            // 0 is not written) of the active state being mapped
    size_t wsump;           // f32 [64][N]: partial column sums of W_r
    size_t rsum;            // f32 [N]: sum_t mu_t dZ_r[t] (router mean-term gradient)
    size_t base;            // bf16 [G-1][T][C]: non-active base readouts of slots 1..G-1
    size_t red;             // f32 [T][nslice][NRED]: per-slice reduction partials
    size_t dxact;           // f32 [T][k][C]: active-state gradient
    size_t dinput;          // bf16 [G][T][C]: copies of d_input
    size_t dotp;            // f32 [k][C/32][T]: <x_act_j, d_input> over 32-channel groups
    size_t dp;              // f32 [T][k]: routing-weight gradient accumulated over slots
    size_t dhpre;           // f32 [T][G][N]
    size_t tokmat;          // f32 [T][TOKMAT]: per-token matrices (E, D, H_res, scalars)
    size_t dz;              // f32 [T][max(nfull, nact)]: projection-output gradients
    size_t scal;            // f32 [T][2]: per-token scalars of the full-state dX (d mu / NC, 2 d nu / NC)
    size_t colp;            // f32 [blocks][ncol]: per-block column sums of the alpha / b gradients
    size_t wpart;           // f32 [tsplits][rows * n]: weight-gradient partials
    size_t cpart;           // f32 [ntiles][kapsum][C]: conv weight-gradient partials
    size_t ws_total;
    int splits_full, splits_act, nslice, tsplits, ntiles;
    ProjTcPlan tc;          // full-state projection: rows T, K = N*C
    ProjTcPlan tca;         // active projection: rows T, K = k*C
    ProjTcPlan twf;         // full weight gradient: rows N*C, K = T
    ProjTcPlan twa;         // active weight gradient: rows k*C, K = T
    size_t dzpack;          // bf16 [NB][T]: hi / lo rows of the projection-output gradient
    size_t dz16;            // bf16 [T][ld]: projection-output gradient (full-state dX GEMM)
    size_t w16;             // bf16 [N*C][ld]: full-state projection weight rows
};

constexpr int NGRAM = 10;    // lower triangle of the 4 x 4 component Gram matrix, (a, b) at a (a + 1) / 2 + b
constexpr int NRED = 112;    // per-token reduction slots (>= k*K + k*k + K*K)
constexpr int TOKMAT = 176;  // E[k][4] + D[4][4] + Hres[k][k] + dX_act mix + scalars (k<=8)
constexpr int NCOLP = 320;   // column sums a coefficient kernel's block leaves (full: 2 G N + N)

// Conv taps of one MLP slot (by value into kernels): w[j] is [kappa_j, C].  For a call on a
// later chunk of its sequences (sequence split), halo [B][R][C] bf16 holds the R = max(kappa) - 1
// sublayer outputs preceding each sequence of the call (null: none, zero padding as at a
// sequence start) and dhalo [B][R][C] fp32 receives their gradient (backward apply only).
struct ConvPtrs {
    const float* w[3];
    const uint16_t* halo;
    float* dhalo;
};
struct ConvGradPtrs {
    float* w[3];
};

struct Handle {
    xhc_config cfg;
    Dims d;
};

}  // namespace xhc

// The opaque handle of the C ABI (include/xhc.h), defined once for every translation unit.
struct xhc_handle {
    xhc::Handle h;
};

namespace xhc {

Layout make_layout(const Dims& d, int64_t T);
Dims make_dims(const xhc_config& c);

// ---------------------------------------------------------------------------------------------
// device helpers

__device__ __forceinline__ float bf2f(uint16_t v) {
    return __uint_as_float(((uint32_t)v) << 16);
}
__device__ __forceinline__ uint16_t f2bf(float f) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}
__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
    f[0] = __uint_as_float(u.x << 16); f[1] = __uint_as_float(u.x & 0xffff0000u);
    f[2] = __uint_as_float(u.y << 16); f[3] = __uint_as_float(u.y & 0xffff0000u);
    f[4] = __uint_as_float(u.z << 16); f[5] = __uint_as_float(u.z & 0xffff0000u);
    f[6] = __uint_as_float(u.w << 16); f[7] = __uint_as_float(u.w & 0xffff0000u);
}
// two floats to bf16 (round to nearest even) in one conversion: a in the low half, b in the high
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    uint32_t r;
    memcpy(&r, &h, sizeof(r));
    return r;
}
// 8 bf16 as 4 channel pairs (low half first)
__device__ __forceinline__ void unpack4x2(const uint4& u, float2* f) {
    f[0] = make_float2(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u));
    f[1] = make_float2(__uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
    f[2] = make_float2(__uint_as_float(u.z << 16), __uint_as_float(u.z & 0xffff0000u));
    f[3] = make_float2(__uint_as_float(u.w << 16), __uint_as_float(u.w & 0xffff0000u));
}
__device__ __forceinline__ uint4 pack8(const float* f) {
    return make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7]));
}
__device__ __forceinline__ float sigm(float z) { return 1.0f / (1.0f + expf(-z)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ int seg_of(const WSegs& w, int o) {
    int s = 0;
#pragma unroll
    for (int q = 1; q < MAXSEG; ++q)
        if (q < w.n && o >= w.off[q]) s = q;
    return s;
}
// W[r][o] of the segmented weight (the segment of column o): the segment's fields are selected
// with static indices, so the kernel parameter is not copied to local memory for a dynamic index
__device__ __forceinline__ float seg_elem(const WSegs& w, long long r, int o) {
    const float* p = w.ptr[0];
    int width = w.width[0], off = w.off[0];
#pragma unroll
    for (int q = 1; q < MAXSEG; ++q)
        if (q < w.n && o >= w.off[q]) {
            p = w.ptr[q];
            width = w.width[q];
            off = w.off[q];
        }
    return p[r * width + (o - off)];
}

// ---------------------------------------------------------------------------------------------
// Gram-Schmidt of Eq. gs expressed on the Gram matrix of u = [out, g_1, ..., g_r]:
// v_j = sum_a B[j][a] u_a, B unit lower-triangular.  Denominators <v_i, v_i> + eps.

// Gm is the lower triangle (a, b) at a (a + 1) / 2 + b; rows of absent components (a >= K) are zero,
// which makes their coefficients zero (the denominators are at least eps > 0).  The products
// y_i = Gm B[i] serve the numerators <g_j, v_i> = y_i[j], the norms <v_i, v_i> = <B[i], y_i> and the
// reverse mode, and each denominator is inverted once: about 60 fp64 operations forward and 60 in
// reverse (the literal sums took 150 and 250).  fp64 runs at two FMAs per clock and SM here, so
// these counts are what bounds the per-token kernels at many tokens, and their dependent chain (three
// reciprocals) at few.
struct GramSchmidt {
    double c10, c20, c30, c21, c31, c32;      // c[j][i] = <g_j, v_i> / (<v_i, v_i> + eps)
    double b10, b20, b21, b30, b31, b32;      // B below its unit diagonal
    double iv0, iv1, iv2;                     // 1 / (<v_i, v_i> + eps)
    double y10, y11, y20, y21, y22;           // y_i[a], a <= i

    __device__ __forceinline__ void forward(const double (&g)[NGRAM], double eps) {
        iv0 = 1.0 / (g[0] + eps);
        c10 = g[1] * iv0;
        c20 = g[3] * iv0;
        c30 = g[6] * iv0;
        b10 = -c10;
        y10 = fma(g[0], b10, g[1]);
        y11 = fma(g[1], b10, g[2]);
        iv1 = 1.0 / (fma(b10, y10, y11) + eps);
        c21 = fma(g[3], b10, g[4]) * iv1;
        c31 = fma(g[6], b10, g[7]) * iv1;
        b20 = fma(-c21, b10, -c20);
        b21 = -c21;
        y20 = fma(g[0], b20, fma(g[1], b21, g[3]));
        y21 = fma(g[1], b20, fma(g[2], b21, g[4]));
        y22 = fma(g[3], b20, fma(g[4], b21, g[5]));
        iv2 = 1.0 / (fma(b20, y20, fma(b21, y21, y22)) + eps);
        c32 = fma(g[6], b20, fma(g[7], b21, g[8])) * iv2;
        b30 = fma(-c32, b20, fma(-c31, b10, -c30));
        b31 = fma(-c32, b21, -c31);
        b32 = -c32;
    }

    // B[q][a] as fp32 (zero above the diagonal)
    __device__ __forceinline__ void coef(float (&B)[MAXCOMP][MAXCOMP]) const {
#pragma unroll
        for (int q = 0; q < MAXCOMP; ++q)
#pragma unroll
            for (int a = 0; a < MAXCOMP; ++a) B[q][a] = (q == a) ? 1.f : 0.f;
        B[1][0] = (float)b10;
        B[2][0] = (float)b20;
        B[2][1] = (float)b21;
        B[3][0] = (float)b30;
        B[3][1] = (float)b31;
        B[3][2] = (float)b32;
    }

    // D = dG + dG^T (lower triangle) from dB below the diagonal (d10, d20, d21, d30, d31, d32)
    __device__ __forceinline__ void reverse(const double (&g)[NGRAM], double d10, double d20, double d21,
                                            double d30, double d31, double d32, double (&D)[NGRAM]) const {
        // row 3: B[3] = e_3 - sum_i c[3][i] B[i]
        double dn = -fma(d30, b20, fma(d31, b21, d32)) * iv2;   // d<g_3, v_2>
        double v2 = -dn * c32;                                   // d(<v_2, v_2> + eps)
        d20 = fma(dn, g[6], fma(-c32, d30, d20));
        d21 = fma(dn, g[7], fma(-c32, d31, d21));
        D[6] = dn * b20;
        D[7] = dn * b21;
        D[8] = dn;
        dn = -fma(d30, b10, d31) * iv1;
        double v1 = -dn * c31;
        d10 = fma(dn, g[6], fma(-c31, d30, d10));
        D[6] = fma(dn, b10, D[6]);
        D[7] += dn;
        dn = -d30 * iv0;
        double v0 = -dn * c30;
        D[6] += dn;
        // row 2
        d20 = fma(2.0 * v2, y20, d20);
        d21 = fma(2.0 * v2, y21, d21);
        dn = -fma(d20, b10, d21) * iv1;
        v1 = fma(-dn, c21, v1);
        d10 = fma(dn, g[3], fma(-c21, d20, d10));
        D[3] = dn * b10;
        D[4] = dn;
        dn = -d20 * iv0;
        v0 = fma(-dn, c20, v0);
        D[3] += dn;
        // row 1
        d10 = fma(2.0 * v1, y10, d10);
        dn = -d10 * iv0;
        v0 = fma(-dn, c10, v0);
        // the norms' own terms, v_i B[i] B[i]^T, counted from both triangles
        const double w2 = 2.0 * v2, w1 = 2.0 * v1;
        D[0] = fma(w2 * b20, b20, fma(w1 * b10, b10, 2.0 * v0));
        D[1] = fma(w2 * b20, b21, fma(w1, b10, dn));
        D[2] = fma(w2 * b21, b21, w1);
        D[3] = fma(w2, b20, D[3]);
        D[4] = fma(w2, b21, D[4]);
        D[5] = w2;
        D[9] = 0.0;
    }
};

// ---------------------------------------------------------------------------------------------
// launch accounting and tracing (host side)

void note_launch();  // counts every kernel launch of the library

// Every kernel begins with pdl_entry.  Launched with programmatic stream serialization, its blocks are
// placed while the last blocks of the kernel before run out, and wait there until that kernel's
// writes are visible; launched without, both instructions do nothing.  No kernel touches global memory
// before, so one whose wait has ended follows all that came before it in its stream.
// The buffers it reads may be written while its blocks already wait, so they are not read-only for the life
// of the kernel: they are read with plain loads, never with __ldg, and pointers to const are not
// __restrict__, which would let the compiler take the read-only path or lift a load over the wait.
__device__ __forceinline__ void pdl_entry() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// A 16-byte read that the compiler leaves where it stands, among the other ones and after the wait.
__device__ __forceinline__ uint4 ld_stream(const void* p) {
    uint4 r;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    return r;
}
// Whether the launches of the call that runs on this thread use it.  It takes a microsecond off every
// kernel of a chain, and costs where the waiting blocks take places from kernels that would still use
// them: us a pass without / with, N C T bf16 state of 4 MB 221 / 185, 52 MB 600 / 558, 100 MB 332 / 289,
// 134 MB 827 / 780, but 537 MB 952 / 967 and 1 GB 3255 / 3278.  In a captured graph, whose kernels
// follow one another closely anyway, it gains nothing (174 / 176) or loses (217 / 229, 758 / 768).
struct PdlScope {
    PdlScope() {}
    PdlScope(const PdlScope&) = delete;
    ~PdlScope();
    void set(size_t state_bytes, cudaStream_t st);
};
bool pdl_on();

template <class... KA, class... A>
inline cudaError_t launch_pdl(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*k)(KA...), A... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl_on() ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, KA(a)...);
    note_launch();
    return e;
}
// More dynamic shared memory than a launch has without asking (48 KB with the static part).  The limit of
// a kernel is only ever raised: a call's size depends on its tokens and widths, and a smaller one set from another
// host thread, between this call and its launch, would make the launch fail.
cudaError_t smem_optin(const void* fn, size_t bytes);
// launch of kernel `k` (in parentheses), counted; returns from the launcher on failure
#define XHC_LAUNCH(st, grid, block, smem, k, ...)                                        \
    do {                                                                                  \
        const cudaError_t le_ = launch_pdl(st, dim3(grid), dim3(block), smem, UNPAREN_ k, __VA_ARGS__); \
        if (le_ != cudaSuccess) return le_;                                               \
    } while (0)
#define UNPAREN_(...) __VA_ARGS__
// test hooks (xhc_debug_set): the limit of the bounded device waits, and a one-shot request that
// the next full-state projection time out before it issues any copy
uint64_t debug_wait_ns();
int debug_take_force_timeout();

// ---------------------------------------------------------------------------------------------
// launchers (each returns cudaGetLastError() after enqueueing)

// Partial column sums of W_r [rows][N], formed in the launch of the projection: parts 0, none wanted.
struct ColJob {
    const float* W;
    int N, parts, rchunk;
    float* out;   // [parts][N]
};
ColJob colsum_of(const float* W_r, int rows, int N, float* out);
// fp32 CUDA-core projection into *nslots partial slots at most (on return: the number written)
constexpr int ROWPROJ_SMALL = 128;   // fewer tokens than this: the kernel for few tokens
cudaError_t launch_rowproj(const uint16_t* A, int64_t lda, int K, int T, const WSegs& W, int n,
                           int* nslots, float* part, float* pstats, const ColJob& cj, cudaStream_t st);
// One weight packed for k_proj_tc: rows 0..n-1 of dst [NB][K] the bf16 hi parts of W[e][o], rows
// n..2n-1 the lo parts, the rest zero.
struct PackJob {
    WSegs W;
    int n, NB, K;
    uint16_t* dst;   // null: nothing to pack
};
constexpr int PACK_E = 256;   // rows of the weight per block of pack_rows_of
// A block's share of a pack job, a thread per weight row (its n columns are whole sectors, the stores are
// contiguous over the threads): for the small weights of the active-state projections, which ride
// along with a kernel that does not depend on them.
__device__ __forceinline__ void pack_rows_of(const PackJob& j, int blk) {
    for (int e = blk * PACK_E + threadIdx.x; e < min(j.K, (blk + 1) * PACK_E); e += blockDim.x) {
#pragma unroll 4
        for (int o = 0; o < j.n; ++o) {
            const float w = seg_elem(j.W, e, o);
            const __nv_bfloat16 h = __float2bfloat16_rn(w);
            j.dst[(int64_t)o * j.K + e] = __bfloat16_as_ushort(h);
            j.dst[(int64_t)(j.n + o) * j.K + e] = __bfloat16_as_ushort(__float2bfloat16_rn(w - __bfloat162float(h)));
        }
        for (int r = 2 * j.n; r < j.NB; ++r) j.dst[(int64_t)r * j.K + e] = 0;
    }
}
// How a bf16 product takes two fp32 operands of n columns each:
//   1 term   both rounded once
//   3 terms  two parts each, hi and lo: columns hi | lo | hi of one operand times hi | hi | lo of the other (the
//            products keep 16 bits)
//   6 terms  three parts each, hi | mid | lo with every part padded to whole MMA k-steps of 16 columns; the
//            product's k-steps take the pairs of parts lo hi, mid mid, hi lo, mid hi, hi mid, hi hi, the smallest
//            first (a part has 8 bits, so that what is left out is 2^-24 of the product, as fp32 leaves)
__host__ __device__ inline int split_step(int n) { return (n + 15) / 16 * 16; }
__host__ __device__ inline int split_cols(int n, int terms) { return terms == 6 ? 3 * split_step(n) : terms * n; }
inline int split_ld(int n, int terms) { return (split_cols(n, terms) + 7) / 8 * 8; }   // 16-byte rows
// the parts of a pair of the six terms, at its place in their order
__device__ __forceinline__ int split_pair_a(int pr) { return (0x046 >> (2 * pr)) & 3; }   // 2 1 0 1 0 0
__device__ __forceinline__ int split_pair_b(int pr) { return (0x124 >> (2 * pr)) & 3; }   // 0 1 2 0 1 0
// part q of v (6 terms).  A value that bf16 cannot round to a finite one is its lo part alone, which only one
// product takes: an infinity stays one (inf - inf, and infinity times another part, would be NaN).
__device__ __forceinline__ float split_part(float v, int q) {
    const float hi = __bfloat162float(__float2bfloat16_rn(v));
    if (!(fabsf(hi) <= 3.4e38f)) return q < 2 ? 0.f : __bfloat162float(__float2bfloat16_rz(v));
    if (q == 0) return hi;
    const float mid = __bfloat162float(__float2bfloat16_rn(v - hi));
    return q == 1 ? mid : (v - hi) - mid;
}
inline int pack_blocks(const PackJob& j) { return j.dst ? (j.K + PACK_E - 1) / PACK_E : 0; }
// bf16 operands that the tensor-core backward takes from a slot's (or the full-state) projection-output
// gradient dz [T][n], written by the coefficient kernel that forms it:
//   hilo [NB][Tp]  rows 0..n-1 the hi parts, n..2n-1 the lo parts, the rest zero (k_proj_tc's B operand of
//                  the weight gradient)
//   rows [T][ld]   the A operand of the input gradient, in the columns of `terms`, zero past them
// null pointers: not wanted.
struct DzPack {
    uint16_t *hilo, *rows;
    int NB, Tp, ld, terms;
};
// dz of a block's ntok tokens from t0 on, in shared memory (row stride rs), into the two operands (SIX: terms is
// 6; a kernel of its own, as a branch cost the others 1 % of a small step)
template <bool SIX>
__device__ __forceinline__ void pack_dz_of(const DzPack& p, const float* dz, int rs, int n, long long t0, int ntok) {
    if (p.hilo != nullptr)
        for (int idx = threadIdx.x; idx < p.NB * ntok; idx += blockDim.x) {
            const int r = idx / ntok, tt = idx - r * ntok;
            float v = 0.f;
            if (r < 2 * n) {
                v = dz[tt * rs + (r < n ? r : r - n)];
                if (r >= n) v -= __bfloat162float(__float2bfloat16_rn(v));
            }
            p.hilo[(long long)r * p.Tp + t0 + tt] = f2bf(v);
        }
    if (p.rows == nullptr) return;
    if (SIX) {
        const int np = split_step(n);
        for (int idx = threadIdx.x; idx < ntok * p.ld; idx += blockDim.x) {
            const int tt = idx / p.ld, c = idx - tt * p.ld, part = c / np, o = c - part * np;
            p.rows[(t0 + tt) * p.ld + c] = f2bf(o < n && part < 3 ? split_part(dz[tt * rs + o], part) : 0.f);
        }
        return;
    }
    for (int idx = threadIdx.x; idx < ntok * p.ld; idx += blockDim.x) {
        const int tt = idx / p.ld, c = idx - tt * p.ld;
        float v = 0.f;
        if (c < p.terms * n) {
            const int part = c / n;
            v = dz[tt * rs + c - part * n];
            if (part == 1) v -= __bfloat162float(__float2bfloat16_rn(v));
        }
        p.rows[(t0 + tt) * p.ld + c] = f2bf(v);
    }
}
// the weight side of the input gradient: dst [rows][ld] bf16, a weight row in the columns of `terms`, zero past
// them; packed by further blocks of the same launch
struct WRows {
    WSegs W;
    int n, rows, ld, terms;
    uint16_t* dst;   // null: nothing to pack
    int C;           // > 0: slots of C rows, each padded to dxa_width(C), in the order of dxa_row
};
// The weight row at place r of k_dx_tc's B operand: in every 32 rows, the one at 8 g + 2 q + e is channel 8 q +
// 2 g + e, so that the accumulator's 16x256b fragments give a lane 8 neighbouring channels.
__device__ __forceinline__ int dxa_row(int r) {
    return (r & ~31) | (((r >> 1) & 3) << 3) | (((r >> 3) & 3) << 1) | (r & 1);
}
inline int __host__ __device__ dxa_width(int C) { return (C + 31) / 32 * 32; }
constexpr int WROWS_U = 8;   // elements per thread
template <bool SIX>
__device__ __forceinline__ void pack_wrows_of(const WRows& j, int blk) {
    const int at = blk * (int)blockDim.x * WROWS_U + threadIdx.x, tot = j.rows * j.ld;   // < 2^31
    float v[WROWS_U];
    int part[WROWS_U];
#pragma unroll
    for (int u = 0; u < WROWS_U; ++u) {
        const int idx = at + u * (int)blockDim.x;
        v[u] = 0.f;
        part[u] = 0;
        if (idx < tot) {
            int r = idx / j.ld;
            const int c = idx - r * j.ld;
            const int np = SIX ? split_step(j.n) : j.n;
            bool in = c < (SIX ? 3 : j.terms) * np;
            if (j.C > 0) {
                const int slot = r / dxa_width(j.C), ch = dxa_row(r - slot * dxa_width(j.C));
                in = in && ch < j.C;
                r = slot * j.C + ch;
            }
            if (in) {
                part[u] = c / np;
                const int o = c - part[u] * np;
                if (!SIX || o < j.n) v[u] = seg_elem(j.W, r, o);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < WROWS_U; ++u) {
        const int idx = at + u * (int)blockDim.x;
        if (SIX) v[u] = split_part(v[u], part[u]);
        else if (part[u] == 2) v[u] -= __bfloat162float(__float2bfloat16_rn(v[u]));
        if (idx < tot) j.dst[idx] = f2bf(v[u]);
    }
}
inline int wrows_blocks(const WRows& j, int threads) {
    return j.dst ? (int)(((long long)j.rows * j.ld + threads * WROWS_U - 1) / (threads * WROWS_U)) : 0;
}

// the full-state weight packed, the partial column sums of W_r (null: none) and the slot-0 active weight,
// in one launch
cudaError_t launch_pack_full(const PackJob& full, const float* W_r, int N, float* wsump, const PackJob& act,
                             cudaStream_t st);
// pstats null: no row statistics (the caller has them from the kernel that wrote X)
cudaError_t launch_proj_tc(const uint16_t* X, int T, int K, const uint16_t* Wpack, int nfull,
                           const ProjTcPlan& p, float* part, float* pstats, int* err,
                           cudaStream_t st);
// dzpack: the hi / lo rows of dz (DzPack::hilo, Tp tokens a row)
cudaError_t launch_wgrad_tc(const uint16_t* A, int T, int E, int n, const uint16_t* dzpack, int Tp,
                            const ProjTcPlan& p, float* part, int* err, cudaStream_t st);
// terms of the full-state and of the active-state input gradient's product, 0: not on the tensor cores
int dx_tc_terms(int T, int N, int C, int nfull, int G);
int dxa_tc_terms(int T, int k, int C, int nact);
// dX_act += dZ_act W_act^T (in dxa_tc_terms bf16 terms on the tensor cores) + H_pre[slot][I_j] d_input
//           - cx x_act (the write-back's own term, cx per token in tokmat);
// in the same pass: dotp[j][g][t] = <x_act_j, d_input> over channels 32 g .. 32 g + 31, and the
// copy dcopy[slot][t][:] = d_input[t][:]
// (dzr, wr: the operands in those terms, DzPack / WRows)
cudaError_t launch_dxa_tc(const Dims& d, int slot, int T, int nact,
                          const uint16_t* dzr, const uint16_t* wr, const uint16_t* d_input, const float* hpre,
                          const int* I, const uint16_t* xact, const float* tokmat, float* dxact,
                          float* dotp, uint16_t* dcopy, int* err, cudaStream_t st);
// dH_pre[t][slot][I_j] = sum over the groups g of 32 channels of dotp[j][g][t] (g in order)
cudaError_t launch_dots_act(const Dims& d, int slot, int T, const float* dotp, const int* I, float* dhpre,
                            cudaStream_t st);
// (dz16, w16: the operands in dx_tc_terms terms)
cudaError_t launch_dx_tc(const Dims& d, int T, const uint16_t* dz16,
                         const uint16_t* w16, const uint16_t* X, const uint16_t* dinput, const float* hpre,
                         const int* I, const float* dxact, const float* scal, int scal_ld,
                         uint16_t* dX, int* err, cudaStream_t st);
int wb_nslice(int C);
int wb_gram_slices(const Dims& d);  // partial-sum slices of wb_gram (and wb_coef)
int wb_conv_runs(const Dims& d, int64_t T);
int wb_bred_slices(const Dims& d, int slot);  // partial-sum slices of wb_bred (and bwd_coef)  // runs (conv weight-gradient partials) of wb_bapp
// decode (one token per sequence, conv history in a per-sequence ring of max(kappa) - 1 rows)
cudaError_t launch_dec_post(const Dims& d, int slot, int B, const uint16_t* out, ConvPtrs cw,
                            uint16_t* ring, long long* pos, const float* p, const float* hpost, double* gram,
                            const uint16_t* xact, const int* I, const float* hres, uint16_t* xact_next,
                            uint16_t* X, cudaStream_t st);
cudaError_t launch_ring_fill(const Dims& d, int B, int S, const uint16_t* out, uint16_t* ring,
                             cudaStream_t st);
// model glue: N copies of a hidden vector per token, and the sum of the N streams
cudaError_t launch_stream_bcast(int T, int N, int C, const uint16_t* h, uint16_t* X, cudaStream_t st);
cudaError_t launch_stream_sum(int T, int N, int C, const uint16_t* X, uint16_t* y, cudaStream_t st);
// sequence split: the halo rows a chunk passes to the next, and the return of their gradient
cudaError_t launch_halo_fill(const Dims& d, int B, int S, const uint16_t* out, uint16_t* halo,
                             cudaStream_t st);
cudaError_t launch_halo_add(const Dims& d, int B, int S, uint16_t* d_out, const float* dhalo,
                            cudaStream_t st);
cudaError_t launch_wb_gram(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                           int nslice, float* red, cudaStream_t st);
cudaError_t launch_wb_coef(const Dims& d, int slot, int T, const float* red, int nslice, const float* p,
                           const float* hpost, double* gram, float* emat, cudaStream_t st);
cudaError_t launch_wb_fwd(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                          const float* emat, const float* p, const float* hpost, int nslice,
                          const uint16_t* xact, const int* I, const float* hres, uint16_t* xact_next, uint16_t* X,
                          cudaStream_t st);
// Xr (both): the last slot's x_j rows are also put back into this state; null: not, as it has to be unless
// wb_puts_back
bool wb_puts_back(const Dims& d);
cudaError_t launch_wb_bred(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                           const uint16_t* dX, const int* I, const float* dxact,
                           const uint16_t* xact, int nslice, float* red, uint16_t* Xr, cudaStream_t st);
cudaError_t launch_wb_b8(const Dims& d, int slot, int T, const uint16_t* out, const uint16_t* dX,
                         const int* I, const float* p, const float* hpost, const float* hres,
                         const float* dxact, float* dxact_out, const uint16_t* xact, int nslice,
                         float* red, uint16_t* d_out, uint16_t* Xr, cudaStream_t st);
cudaError_t launch_wb_bapp(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                           const uint16_t* dX, const int* I, const float* dn_in,
                           const float* tokmat, float* dxact_out, uint16_t* d_out, float* cpart,
                           cudaStream_t st);
// G[e][o] += sum of the slots of wpart[slot][e][o], less sub[o] on the first segment's columns (sub
// null: nothing is subtracted)
cudaError_t launch_wgrad_reduce(const float* wpart, const SlotPlan& sp, int E, int n, const WSegsOut& G,
                                const float* sub, cudaStream_t st);
// partial column sums of in [rows][n]: out [colsum_parts(rows)][n], part q over the rows of chunk q
constexpr int COLSUM_PARTS = 64;   // at most
int colsum_parts(int rows);
int colsum_chunk(int rows);        // rows of a chunk
// chunk `part`, by the first 8 n threads of a block (n <= MAXN): eight threads a column over interleaved
// rows (U loads each in flight), then their sum in order.  sh: 8 n floats.  Has block barriers.
__device__ __forceinline__ void colsum_chunk_of(const float* in, int rows, int n, int rchunk, int part,
                                                float* sh, float* __restrict__ out) {
    constexpr int U = 32;
    const int o = threadIdx.x % n, ty = threadIdx.x / n;
    const int r0 = part * rchunk, r1 = min(rows, r0 + rchunk);
    if (ty < 8) {
        float s = 0.f;
        int r = r0 + ty;
        for (; r + 8 * (U - 1) < r1; r += 8 * U) {
            float v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = in[(int64_t)(r + 8 * u) * n + o];
#pragma unroll
            for (int u = 0; u < U; ++u) s += v[u];
        }
#pragma unroll 4
        for (; r < r1; r += 8) s += in[(int64_t)r * n + o];
        sh[threadIdx.x] = s;
    }
    __syncthreads();
    if (ty == 0) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) t += sh[q * n + o];
        out[part * n + o] = t;
    }
}
// wsum: [nws][N] partial column sums of W_r; their sum is left in wsum_out [N]
cudaError_t launch_coef_full(const Dims& d, int T, const float* part, const float* pstats,
                             const SlotPlan& sp, const float* wsum, int nws, const float* alpha_pre,
                             const float* b_pre, float* zfull, float* stats, float* wsum_out, float* hpre,
                             int* I, float* p, cudaStream_t st);
cudaError_t launch_coef_act(const Dims& d, int slot, int T, const float* part,
                            const float* pstats, int ssplits, const SlotPlan& sp, const float* alpha_post,
                            const float* b_post, const float* alpha_res, const float* b_res,
                            float* zact, float* rs, float* hpost, float* hres, cudaStream_t st);
int stream_warps(int C);  // warps per block of the one-block-per-token stream kernels
cudaError_t launch_read(const Dims& d, int T, const uint16_t* X, const float* hpre, const int* I,
                        uint16_t* input0, uint16_t* base, uint16_t* xact0, float* astat, cudaStream_t st);
// pack: the slot's active weight, packed by further blocks of the same launch
cudaError_t launch_input(const Dims& d, int slot, int T, const uint16_t* base, const uint16_t* xact,
                         const float* hpre, const int* I, uint16_t* input, float* astat, const PackJob& pack,
                         cudaStream_t st);
cudaError_t launch_restore(const Dims& d, int T, const uint16_t* xact0, const int* I,
                           uint16_t* X, cudaStream_t st);
cudaError_t launch_bwd_coef(const Dims& d, int slot, int T, const float* red, int nslice,
                            const float* zact, const float* rs, const float* p,
                            const float* hpost, const double* gram, const float* alpha_post,
                            const float* alpha_res, const float* b_res,
                            float* tokmat, float* dz, float* dp, float* colp, int* nblk, const DzPack& pack,
                            const WRows& wrows, cudaStream_t st);
// adds the column sums over the blocks' partials colp [nblk][ncol] to up to four targets: target q
// takes columns off[q] .. off[q] + n[q] - 1
struct ColOut {
    float* ptr[4];
    int off[4], n[4];
    int set[4];   // 1: stored instead of added
};
cudaError_t launch_colsum_out(const float* colp, int nblk, int ncol, const ColOut& out, cudaStream_t st);
cudaError_t launch_gemm_dzw(const Dims& d, int T, const float* dz, int ldz, int n,
                            const WSegs& W, int E, float* dxact, cudaStream_t st);
cudaError_t launch_conv_wgrad_reduce(const Dims& d, int slot, const float* cpart, int ntiles,
                                     ConvGradPtrs gconv, cudaStream_t st);
cudaError_t launch_wgrad(const uint16_t* A, int64_t lda, int E, int T, const float* dz, int ldz,
                         int n, int tsplits, float* wpart, const WSegsOut& G, const float* sub,
                         cudaStream_t st);
cudaError_t launch_dinput_act(const Dims& d, int slot, int T, int add_dx, const uint16_t* d_input,
                              const uint16_t* xact, const float* hpre, const int* I,
                              float* dxact, float* dhpre, uint16_t* dinput_copy,
                              const float* tokmat, cudaStream_t st);
cudaError_t launch_full_dots(const Dims& d, int T, const uint16_t* X, const uint16_t* dinput,
                             const int* I, float* dhpre, cudaStream_t st);
cudaError_t launch_full_coef(const Dims& d, int T, const float* dhpre, const float* hpre,
                             const float* zfull, const float* stats, const float* wsum,
                             const int* I, const float* dp, const float* alpha_pre, float* dz,
                             float* scal, float* colp, int* nblk, const DzPack& pack, const WRows& wrows,
                             cudaStream_t st);
cudaError_t launch_full_dx(const Dims& d, int T, const float* dz, const WSegs& W,
                           const uint16_t* X, const uint16_t* dinput, const float* hpre,
                           const int* I, const float* dxact, const float* scal,
                           uint16_t* dX, cudaStream_t st);

}  // namespace xhc
