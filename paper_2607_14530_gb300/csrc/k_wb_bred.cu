// Launcher of the backward write-back reductions (wb_bred).
#include "k_wb.cuh"

namespace xhc {
namespace {

template <int KM, int KW, int NV, int KS, bool PUT>
cudaError_t bred_kw(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw, const uint16_t* dX,
                    const int* I, const float* dxact, const uint16_t* xact, int nslice, float* red,
                    uint16_t* Xr, cudaStream_t st) {
    constexpr int NVP = NV < 32 ? 16 : NV;
    // 64 measured faster than 48 with the block ring
    int TB = pick_run(d, T, true, nslice, KM == 4 ? 3 : 2, 12, 64);
    while (TB > 4 && (size_t)TB * (WT / 32) * NVP * 4 > 96 * 1024) TB -= 4;
    const size_t sm = sizeof(BRing<KM>) + (size_t)TB * KM * 4 + (size_t)TB * (WT / 32) * NVP * sizeof(float);
    cudaError_t e = smem_optin((const void*)k_wb_bred<KM, KW, NV, KS, PUT>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid(nslice, (unsigned)n_runs(d, T, TB, KW > 0));
    XHC_LAUNCH(st, grid, WT, sm, (k_wb_bred<KM, KW, NV, KS, PUT>), d, slot, T, TB, out, cw, dX, I, dxact, xact, nslice, red, Xr);
    return cudaGetLastError();
}

template <int KM, int NV, bool PUT>
cudaError_t bred2_kw(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw, const uint16_t* dX,
                     const int* I, const float* dxact, const uint16_t* xact, int nslice, float* red,
                     uint16_t* Xr, cudaStream_t st) {
    constexpr int NVP = NV < 32 ? 16 : NV;
    const int TB = pick_run(d, T, true, d.C / WSL2, 2, 12, 64);
    const size_t sm = sizeof(BRing2<KM>) + (size_t)TB * KM * 4 + (size_t)TB * (WT / 32) * NVP * sizeof(float);
    cudaError_t e = smem_optin((const void*)k_wb_bred2<KM, NV, PUT>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid(d.C / WSL2, (unsigned)n_runs(d, T, TB, true));
    XHC_LAUNCH(st, grid, WT, sm, (k_wb_bred2<KM, NV, PUT>), d, slot, T, TB, out, cw, dX, I, dxact, xact, nslice, red, Xr);
    return cudaGetLastError();
}

// the two-pair reductions: the (4, 8, 12) taps, k = 4, C a multiple of WSL2
bool bred2_ok(const Dims& d) { return paper_kaps(d) && d.k == 4 && d.C % WSL2 == 0; }

template <int KM, bool PUT>
cudaError_t b8_kw(const Dims& d, int slot, int T, const uint16_t* out, const uint16_t* dX, const int* I,
                  const float* p, const float* hpost, const float* hres, const float* dxact,
                  float* dxact_out, const uint16_t* xact, int nslice, float* red, uint16_t* d_out,
                  uint16_t* Xr, cudaStream_t st) {
    constexpr int NQ = KM + KM * KM;
    constexpr int NV = NQ <= 32 ? 32 : 96;
    const int TB = pick_run(d, T, false, (d.C + W8 - 1) / W8, KM == 4 ? 3 : 2, 4, 32);
    const size_t sm = (size_t)TB * (2 * KM + KM * KM) * 4 + (size_t)TB * (WT / 32) * NV * 4;
    cudaError_t e = smem_optin((const void*)k_wb_b8<KM, PUT>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid((d.C + W8 - 1) / W8, (T + TB - 1) / TB);
    XHC_LAUNCH(st, grid, WT, sm, (k_wb_b8<KM, PUT>), d, slot, T, TB, out, dX, I, p, hpost, hres, dxact, dxact_out, xact, nslice, red, d_out, Xr);
    return cudaGetLastError();
}

}  // namespace

// The last slot of a group of one reads the entry rows themselves: its kernel puts them back into X.  The
// forms for eight streams leave that to restore: wb_bred's stores cost more than the launch (T = 1000, k =
// 8, C = 1160: 422 -> 428 us a step), wb_b8 spills as it is.  k = 4, against restore before them: T =
// 16384, C = 2048 3205 -> 3146 us a step; T = 8192, N = 4, no conv, 755 -> 740; T = 512, C =
// 256, 182.5 -> 177.5.
bool wb_puts_back(const Dims& d) { return d.G == 1 && d.k <= 4; }

// slices (partial sums per token) of the backward reductions of a slot
int wb_bred_slices(const Dims& d, int slot) {
    if (d.K[slot] == 1) return (d.C + W8 - 1) / W8;
    return bred2_ok(d) ? d.C / WSL2 : wb_nslice(d.C);
}

cudaError_t launch_wb_bred(const Dims& d, int slot, int T, const uint16_t* out, ConvPtrs cw,
                           const uint16_t* dX, const int* I, const float* dxact,
                           const uint16_t* xact, int nslice, float* red, uint16_t* Xr, cudaStream_t st) {
    const bool conv = d.K[slot] > 1;
    const bool last = (slot == d.G - 1);
    // a slot without conv takes the one-pass backward (launch_wb_b8), not this kernel
    if (!conv) return cudaErrorInvalidValue;
    if (bred2_ok(d)) {
        if (last && Xr) return bred2_kw<4, 32, true>(d, slot, T, out, cw, dX, I, dxact, xact, nslice, red, Xr, st);
        if (last) return bred2_kw<4, 32, false>(d, slot, T, out, cw, dX, I, dxact, xact, nslice, red, Xr, st);
        return bred2_kw<4, 16, false>(d, slot, T, out, cw, dX, I, dxact, xact, nslice, red, Xr, st);
    }
#define XHC_BRED(KM_, NV_, FAST_, PUT_)                                                                 \
    do {                                                                                            \
        XHC_KW_DISPATCH(d, FAST_, (bred_kw<KM_, KWC, NV_, KSC, PUT_>(d, slot, T, out, cw, dX, I, dxact, xact, nslice, red, Xr, st))); \
    } while (0)
    if (d.k <= 4) {
        if (last && Xr) XHC_BRED(4, 32, wb_fast(d), true);
        if (last) XHC_BRED(4, 32, wb_fast(d), false);
        XHC_BRED(4, 16, wb_fast(d), false);
    }
    if (last) XHC_BRED(8, 96, false, false);
    XHC_BRED(8, 32, false, false);
#undef XHC_BRED
}

// backward reductions and apply of a slot without conv (K = 1), in one pass over dXn
cudaError_t launch_wb_b8(const Dims& d, int slot, int T, const uint16_t* out, const uint16_t* dX,
                         const int* I, const float* p, const float* hpost, const float* hres,
                         const float* dxact, float* dxact_out, const uint16_t* xact, int nslice,
                         float* red, uint16_t* d_out, uint16_t* Xr, cudaStream_t st) {
    if (d.K[slot] != 1) return cudaErrorInvalidValue;
    if (d.k <= 4 && Xr)
        return b8_kw<4, true>(d, slot, T, out, dX, I, p, hpost, hres, dxact, dxact_out, xact, nslice, red, d_out, Xr, st);
    if (d.k <= 4)
        return b8_kw<4, false>(d, slot, T, out, dX, I, p, hpost, hres, dxact, dxact_out, xact, nslice, red, d_out, Xr, st);
    return b8_kw<8, false>(d, slot, T, out, dX, I, p, hpost, hres, dxact, dxact_out, xact, nslice, red, d_out, Xr, st);
}

}  // namespace xhc
