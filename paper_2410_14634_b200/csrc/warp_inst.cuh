// Launchers of the few-channel kernels (WARP family, its grad_w and its masked convolution); one translation unit per
// channel count instantiates them, so that they build in parallel.
#pragma once

#include <cstdio>

#include "lib_internal.h"
#include "warp_kernels.cuh"
#include "gradw_kernels.cuh"
#include "conv_kernels.cuh"

namespace invconv_internal {

using namespace invconv;

template <int C, int K, bool BWD>
int launch_warp_ck(const WarpPlan& pl, WarpParams prm, bool allow_ring, bool allow_split, bool dependent, cudaStream_t st)
{
    // global-memory mode: streamed through a shared-memory ring unless grad_w rides along in the wavefront
    const bool ring = pl.glb && pl.ring && prm.grad_w == nullptr && allow_ring;
    // channel-split walk (its own row-block geometry) unless grad_w rides along in the wavefront
    bool cs = false;
    if constexpr (C >= 3 && K == 5) cs = pl.cs && prm.grad_w == nullptr && allow_split;
    auto kern = ring ? warp_wavefront_kernel<C, K, BWD, true, true, true>
                     : (pl.glb ? warp_wavefront_kernel<C, K, BWD, true, true>
                               : (pl.nb > 1 ? warp_wavefront_kernel<C, K, BWD, true> : warp_wavefront_kernel<C, K, BWD, false>));
    size_t smem = ring ? pl.smem_ring : pl.smem;
    int nb = pl.nb, ipc = pl.ipc, grid = pl.grid;
    if constexpr (C >= 3 && K == 5) {
        if (cs) {
            kern = pl.nb_cs > 1 ? warp_wavefront_kernel<C, K, BWD, true, false, false, true>
                                : warp_wavefront_kernel<C, K, BWD, false, false, false, true>;
            smem = pl.smem_cs; nb = pl.nb_cs; ipc = pl.ipc_cs; grid = pl.grid_cs;
            prm.nb = nb; prm.ipc = ipc;
        }
    }
    const int rc = set_smem_limit(kern, smem);
    if (rc) return rc;
    // Programmatic dependent launch: the kernel may be scheduled while its predecessor on the stream drains;
    // it touches no global memory before griddepcontrol.wait, which waits for that predecessor to complete.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(nb * ipc * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, prm);
    if (e != cudaSuccess) {
        std::fprintf(stderr, "invconv: warp launch failed: %s\n", cudaGetErrorString(e));
        cudaGetLastError();
        return INVCONV_CUDA_ERROR;
    }
    return check_launch();
}

template <int C, int K>
int launch_gradw_small_ck(const GradWSmallPlan& gs, const GradWSmallParams& prm, bool dependent, cudaStream_t st)
{
    auto kern = gradw_small_kernel<C, K>;
    const int rc = set_smem_limit(kern, gs.smem);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(gs.grid);
    cfg.blockDim = dim3(GradWSmallShape<C, K>::NT);
    cfg.dynamicSmemBytes = gs.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, prm);
    if (e != cudaSuccess) {
        std::fprintf(stderr, "invconv: grad_w launch failed: %s\n", cudaGetErrorString(e));
        cudaGetLastError();
        return INVCONV_CUDA_ERROR;
    }
    return check_launch();
}

template <int C, int K>
int launch_masked_conv_ck(const float* x, const float* w, float* y, Geom g, bool dependent, cudaStream_t st)
{
    // warps per band of rows: one, or one per output channel where the kernel does not fit a lane's registers
    constexpr int wsplit = (C * C * K * K <= 108) ? 1 : C;
    constexpr int maxw = 8 / wsplit;             // eight warps per CTA
    int wpi = (g.H + 7) / 8;                     // about eight rows per warp
    if (wpi > maxw) wpi = maxw;
    if (wpi < 1) wpi = 1;
    int ipc = maxw / wpi;
    if (ipc > g.B) ipc = g.B;
    if (ipc < 1) ipc = 1;
    while (ipc > 1 && masked_conv_smem<C, K>(g.H, g.W, ipc) > kMaxDynSmem) --ipc;
    size_t smem = masked_conv_smem<C, K>(g.H, g.W, ipc);
    const size_t chw = (size_t)g.C * g.H * g.W;
    ConvParams prm;
    prm.x = x; prm.w = w; prm.y = y; prm.B = g.B; prm.H = g.H; prm.W = g.W;
    prm.bulk = ((reinterpret_cast<uintptr_t>(x) & 15) == 0 && chw % 4 == 0) ? 1 : 0;
    int grid = (g.B + ipc - 1) / ipc;
    // few (fewer CTAs than half the SMs) or very large images: one CTA per band of rows instead, about two CTAs per SM
    const bool rows_ok = (reinterpret_cast<uintptr_t>(x) & 15) == 0 && g.W % 4 == 0;
    if (rows_ok && g.H >= 16 && (smem > kMaxDynSmem || 2 * grid <= sm_count())) {
        int bands = (2 * sm_count() + g.B - 1) / g.B;
        if (bands > (g.H + 7) / 8) bands = (g.H + 7) / 8;             // at least eight rows per band
        int bh = (g.H + bands - 1) / bands;
        while (masked_conv_smem<C, K>(bh + K - 1, g.W, 1) > kMaxDynSmem && bh > 1) bh = (bh + 1) / 2;
        bands = (g.H + bh - 1) / bh;
        if (bands > 1 && masked_conv_smem<C, K>(bh + K - 1, g.W, 1) <= kMaxDynSmem) {
            prm.bands = bands; prm.bh = bh; prm.bulk = 1;
            ipc = 1;
            wpi = bh >= 16 ? 4 : (bh >= 8 ? 2 : 1);
            if (wpi > maxw) wpi = maxw;
            smem = masked_conv_smem<C, K>(bh + K - 1, g.W, 1);
            grid = g.B * bands;
        }
    }
    if (smem > kMaxDynSmem) return INVCONV_UNSUPPORTED;
    auto kern = masked_conv_warp_kernel<C, K>;
    const int rc = set_smem_limit(kern, smem);
    if (rc) return rc;
    prm.ipc = ipc; prm.wpi = wpi;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(ipc * wpi * wsplit * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // launch latency overlaps the kernel before
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, prm) != cudaSuccess) {
        cudaGetLastError();
        return INVCONV_CUDA_ERROR;
    }
    return check_launch();
}

}  // namespace invconv_internal

#define INVCONV_WARP_UNIT(C_)                                                                                              \
    namespace invconv_internal {                                                                                           \
    int launch_warp_c##C_(int k, bool bwd, const WarpPlan& pl, const WarpParams& prm, bool ring, bool split, bool dep, cudaStream_t st) \
    {                                                                                                                      \
        switch (k) {                                                                                                       \
        case 2: return bwd ? launch_warp_ck<C_, 2, true>(pl, prm, ring, split, dep, st) : launch_warp_ck<C_, 2, false>(pl, prm, ring, split, dep, st); \
        case 3: return bwd ? launch_warp_ck<C_, 3, true>(pl, prm, ring, split, dep, st) : launch_warp_ck<C_, 3, false>(pl, prm, ring, split, dep, st); \
        case 5: return bwd ? launch_warp_ck<C_, 5, true>(pl, prm, ring, split, dep, st) : launch_warp_ck<C_, 5, false>(pl, prm, ring, split, dep, st); \
        default: return INVCONV_UNSUPPORTED;                                                                               \
        }                                                                                                                  \
    }                                                                                                                      \
    int launch_masked_conv_c##C_(const float* x, const float* w, float* y, Geom g, bool dep, cudaStream_t st)              \
    {                                                                                                                      \
        switch (g.k) {                                                                                                     \
        case 2: return launch_masked_conv_ck<C_, 2>(x, w, y, g, dep, st);                                                  \
        case 3: return launch_masked_conv_ck<C_, 3>(x, w, y, g, dep, st);                                                  \
        case 5: return launch_masked_conv_ck<C_, 5>(x, w, y, g, dep, st);                                                  \
        default: return INVCONV_UNSUPPORTED;                                                                               \
        }                                                                                                                  \
    }                                                                                                                      \
    }
