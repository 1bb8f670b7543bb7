// Weight gradient for the shapes the tensor pipe does not take (Theorem 2 in closed form):
//   grad_w[co][ci][K-1-dh][K-1-dw] = - sum_{n,h,w} grad_y[n,co,h,w] * x[n,ci,h-dh,w-dw]
// any width, any kernel side up to 11, fp32 throughout.
//
// A CTA owns one tile of T input channels, a few tiles of T output channels, all kernel rows, and a share of the (image, row
// band) units.  A unit's channel planes are staged in shared memory by asynchronous copies, zero-padded (columns beyond the
// image, rows above it, K-1 columns to its left), one unit ahead of the arithmetic.  A warp (or WPT of them) owns one task --
// output tile, kernel row dh -- and its lanes walk the band's quads of four pixels with the T*T*K sums in registers: per
// quad T 16-byte loads of grad_y, T times one plus (K-1)/4 rounded up of x, and 4*T*T*K multiply-adds.
// Lanes are summed by transposed shuffles, shares by gradw_reduce_kernel in a fixed order.
// Bound: FMA pipe for T = 4 (192 multiply-adds per 12 loads at k = 3), shared-memory bandwidth below.  Before it, widths that
// are no multiple of four and kernels of 7 to 11 went to one CTA per weight reading global memory (100 to 550 us on
// shapes whose solve takes 15 to 50 us).
#pragma once

#include "common.cuh"
#include "tma.cuh"
#include "gradw_quad_plan.h"

namespace invconv {

struct GradWQuadParams {
    const float* gy;       // [B][C][H][W]
    const float* x;
    float* partials;       // [shares][K*K][C][C]
    int B, C, H, W;
    int RB, nbands, shares;
    int NCO, cotiles;      // output tiles per CTA, groups of them
    int tiles;             // input tiles
    int WPT;               // warps per task
    int gst, xst;          // row strides of the staged planes (floats, multiples of 4); x has LP zero columns on its left
    int gfloats, stage;    // floats of the grad_y part and of a whole stage
    int vec;               // rows are 16-byte aligned multiples of 16 bytes
    int long_rows;         // copied a row per warp, not element by element
    FastDiv div_bands, div_grow, div_gch, div_xch, div_q, div_k;
};

template <int T, int K>
__global__ void __launch_bounds__(384, T * T * K <= 32 ? 2 : 1) gradw_quad_kernel(const __grid_constant__ GradWQuadParams p)
{
    constexpr int LP = (K - 1 + 3) / 4 * 4, NL = 1 + LP / 4;      // zero columns left of the image; 16-byte loads per window
    extern __shared__ __align__(128) float smem[];
    const int C = p.C, H = p.H, W = p.W, HW = H * W, RB = p.RB;
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
    int bid = blockIdx.x;
    const int share = bid % p.shares; bid /= p.shares;
    const int ci0 = (bid % p.tiles) * T, co0 = (bid / p.tiles) * p.NCO * T;
    const int nco = min(p.NCO * T, C - co0), nci = min(T, C - ci0);
    const int task = (tid >> 5) / p.WPT, slice = ((tid >> 5) - task * p.WPT) * 32 + lane;
    const int cot = fast_div(task, p.div_k), dh = task - cot * K;

    float acc[T][T][K];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j)
#pragma unroll
            for (int d = 0; d < K; ++d) acc[i][j][d] = 0.f;
    for (int i = tid; i < 2 * p.stage; i += NT) smem[i] = 0.f;     // padding and channels beyond C stay zero
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();

    const int units = p.B * p.nbands;
    const int xr_rows = RB + K - 1;
    // stages unit u: rows h0 .. h0+RB-1 of grad_y, h0-K+1 .. h0+RB-1 of x; rows outside the image become zeros
    auto stage = [&](int u, float* base) {
        const int n = fast_div(u, p.div_bands), h0 = (u - n * p.nbands) * RB;
        const float* gsrc = p.gy + ((size_t)n * C + co0) * HW;
        const float* xsrc = p.x + ((size_t)n * C + ci0) * HW;
        if (p.long_rows) {
            // long rows of single elements: a row to each warp, its place worked out once (per element that costs 30
            // against 27 us at 163x3x62x62; but with rows of 9 pixels most of a warp idles, 35 against 24 us at 150x24x9x9)
            const int grows = nco * RB, rows = grows + nci * xr_rows;
            for (int q = tid >> 5; q < rows; q += NT >> 5) {
                const bool isg = q < grows;
                const int row = isg ? q : q - grows;
                const int c = isg ? fast_div(row, p.div_gch) : fast_div(row, p.div_xch), r = row - c * (isg ? RB : xr_rows);
                const int h = h0 + r - (isg ? 0 : K - 1);
                const bool in = h >= 0 && h < H;
                const float* src = (isg ? gsrc : xsrc) + (in ? c * HW + h * W : 0);
                float* dst = base + (isg ? row * p.gst : p.gfloats + row * p.xst + LP);
                for (int w = lane; w < W; w += 32) cp_async_f32(dst + w, src + w, in);
            }
            return;
        }
        const int ppr = p.vec ? W >> 2 : W;                        // pieces per row
        const int gi = nco * RB * ppr, xi = nci * xr_rows * ppr;
        for (int e = tid; e < gi + xi; e += NT) {
            const bool isg = e < gi;
            const int f = isg ? e : e - gi;
            const int row = fast_div(f, p.div_q), pc = f - row * ppr;
            const int c = isg ? fast_div(row, p.div_gch) : fast_div(row, p.div_xch), r = row - c * (isg ? RB : xr_rows);
            const int h = h0 + r - (isg ? 0 : K - 1);
            const bool in = h >= 0 && h < H;
            const float* src = (isg ? gsrc : xsrc) + (in ? c * HW + h * W + (p.vec ? pc * 4 : pc) : 0);
            float* dst = base + (isg ? row * p.gst : p.gfloats + row * p.xst + LP) + (p.vec ? pc * 4 : pc);
            if (p.vec) cp_async_f32x4(dst, src, in); else cp_async_f32(dst, src, in);
        }
    };
    int buf = 0;
    if (share < units) stage(share, smem);
    cp_async_commit();
    const int qpr = p.gst >> 2, nq = RB * qpr;
    for (int u = share; u < units; u += p.shares, buf ^= 1) {
        if (u + p.shares < units) stage(u + p.shares, smem + (buf ^ 1) * p.stage);
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();
        const float* gq = smem + buf * p.stage + cot * T * RB * p.gst;
        const float* xq = smem + buf * p.stage + p.gfloats + (K - 1 - dh) * p.xst;     // band row r meets x row r - dh
        for (int q = slice; q < nq; q += p.WPT * 32) {
            const int r = fast_div(q, p.div_grow), w0 = (q - r * qpr) * 4;
            float g[T][4];
#pragma unroll
            for (int i = 0; i < T; ++i) {
                const float4 t = *reinterpret_cast<const float4*>(gq + (i * RB + r) * p.gst + w0);
                g[i][0] = t.x; g[i][1] = t.y; g[i][2] = t.z; g[i][3] = t.w;
            }
#pragma unroll
            for (int j = 0; j < T; ++j) {
                float v[4 * NL];
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    const float4 t = *reinterpret_cast<const float4*>(xq + (j * xr_rows + r) * p.xst + w0 + 4 * l);
                    v[4 * l] = t.x; v[4 * l + 1] = t.y; v[4 * l + 2] = t.z; v[4 * l + 3] = t.w;
                }
#pragma unroll
                for (int d = 0; d < K; ++d)
#pragma unroll
                    for (int px = 0; px < 4; ++px)
#pragma unroll
                        for (int i = 0; i < T; ++i) acc[i][j][d] = fmaf(g[i][px], v[LP + px - d], acc[i][j][d]);
            }
        }
        __syncthreads();       // everyone is done with this stage before it is filled again
    }
    cp_async_wait<0>();

    // lanes, then the warps of a task, in a fixed order
    constexpr int NS = T * T * K;
    float* red = smem;                                 // [warp][NS]
#pragma unroll
    for (int base = 0; base < NS; base += 32) {
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int e = base + i;
            v[i] = e < NS ? acc[e / (T * K) % T][e / K % T][e % K] : 0.f;
        }
        const float tot = transpose_reduce32(v, lane);
        if (base + lane < NS) red[(tid >> 5) * NS + base + lane] = tot;
    }
    __syncthreads();
    float* dst = p.partials + (size_t)share * K * K * C * C;
    const int ntask = (NT >> 5) / p.WPT;
    for (int e = tid; e < ntask * NS; e += NT) {
        const int tk = e / NS, f = e - tk * NS, i = f / (T * K), j = f / K % T, d = f % K;
        float s = 0.f;
        for (int q = 0; q < p.WPT; ++q) s += red[(tk * p.WPT + q) * NS + f];
        const int c = tk / K, row = tk - c * K, co = co0 + c * T + i, ci = ci0 + j;
        if (co < C && ci < C) dst[((size_t)(row * K + d) * C + co) * C + ci] = s;
    }
}

}  // namespace invconv
