// The inverse convolution together with the two layers that follow it in one step of the paper's
// Inverse-Flow model (Section 4, Fig. 3): Actnorm, z = s*x + b per channel, and the 1x1 convolution,
// u = V z per pixel.  Both act on one pixel at a time.  For the few-channel (warp) family they are applied
// inside the wavefront kernel while the image is in shared memory -- u is written beside x in the store
// epilogue, and grad_x = s * (V^T grad_u) is formed in the load prologue of the transposed solve -- so that x
// is not read back from memory; for the other families the step is composed from the layer's kernels and the
// per-pixel kernels below (the image is then still in L2).  The parameter gradients of the neighbours are sums
// over pixels of grad_u x^T and grad_u, reduced in a fixed order.
#include <cuda_runtime.h>

#include <cstdio>

#include "invconv.h"

#include "common.cuh"
#include "lib_internal.h"

using namespace invconv;
using invconv_internal::check_launch;

namespace {

constexpr int kMixPixels = 64;      // pixels per CTA tile of the per-pixel kernels

// out[n][o][p] = sum_c A[o][c] * in[n][c][p] + cb[o]  with
//   forward : A = V diag(s), cb = V b   (u from x)
//   backward: A = diag(s) V^T, cb = 0   (grad_x from grad_u)
// One CTA per (image, tile of 64 pixels); the input tile and A are staged in shared memory.
template <bool BWD>
__global__ void __launch_bounds__(256) flow_mix_kernel(const float* __restrict__ in, const float* __restrict__ V,
                                                       const float* __restrict__ s, const float* __restrict__ b,
                                                       float* __restrict__ out, int C, int HW, int tiles)
{
    extern __shared__ __align__(16) float fsm[];
    float* A = fsm;                         // [C][C + 1]
    float* cb = A + C * (C + 1);            // [C]
    float* tile = cb + C;                   // [C][kMixPixels]
    const int n = blockIdx.x / tiles, t0 = (blockIdx.x - n * tiles) * kMixPixels;
    const int np = min(kMixPixels, HW - t0);
    for (int e = threadIdx.x; e < C * C; e += blockDim.x) {
        const int o = e / C, c = e - o * C;
        A[o * (C + 1) + c] = BWD ? __ldg(s + o) * __ldg(V + c * C + o) : __ldg(V + o * C + c) * __ldg(s + c);
    }
    for (int o = threadIdx.x; o < C; o += blockDim.x) {
        float acc = 0.f;
        if (!BWD) for (int c = 0; c < C; ++c) acc = fmaf(__ldg(V + o * C + c), __ldg(b + c), acc);
        cb[o] = acc;
    }
    const float* src = in + (size_t)n * C * HW + t0;
    for (int e = threadIdx.x; e < C * kMixPixels; e += blockDim.x) {
        const int c = e / kMixPixels, p = e - c * kMixPixels;
        tile[e] = p < np ? __ldg(src + (size_t)c * HW + p) : 0.f;
    }
    __syncthreads();
    float* dst = out + (size_t)n * C * HW + t0;
    for (int e = threadIdx.x; e < C * kMixPixels; e += blockDim.x) {
        const int o = e / kMixPixels, p = e - o * kMixPixels;
        float acc = cb[o];
        for (int c = 0; c < C; ++c) acc = fmaf(A[o * (C + 1) + c], tile[c * kMixPixels + p], acc);
        if (p < np && INVCONV_CHECKED((size_t)n * C * HW + t0 + (size_t)o * HW + p, (size_t)gridDim.x / tiles * C * HW, 401))
            dst[(size_t)o * HW + p] = acc;
    }
}

// Partial sums over a share of the (image, pixel tile) items:
//   G1[o][c] = sum grad_u[n][o][p] * x[n][c][p],   g0[o] = sum grad_u[n][o][p]
// partials[share][C*C + C] (double).  Thread (o, c-lane) walks the pixels of a staged tile.  With few channels there are
// few entries, each one long sum that may cancel almost completely (and nothing larger to be measured against), so a
// thread that owns at most four entries adds the exact fp32 products in double; with many channels the sums
// stay fp32 (up to 68 per thread).
__global__ void __launch_bounds__(256) flow_mix_grad_kernel(const float* __restrict__ gu, const float* __restrict__ x,
                                                            double* __restrict__ partials, int B, int C, int HW, int tiles)
{
    extern __shared__ __align__(16) float fsm[];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float* tg = fsm;                              // [C][kMixPixels + 1]
    float* tx = tg + C * (kMixPixels + 1);        // [C][kMixPixels + 1]
    const int items = B * tiles, NE = C * C + C;
    const int per = (NE + blockDim.x - 1) / blockDim.x;     // entries per thread (at most 65 for C = 128)
    const bool wide_acc = per <= 4;
    float acc[68];
    double dacc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int q = 0; q < 68; ++q) acc[q] = 0.f;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int n = it / tiles, t0 = (it - n * tiles) * kMixPixels;
        const int np = min(kMixPixels, HW - t0);
        const float* sg = gu + (size_t)n * C * HW + t0;
        const float* sx = x + (size_t)n * C * HW + t0;
        __syncthreads();
        for (int e = threadIdx.x; e < C * kMixPixels; e += blockDim.x) {
            const int c = e / kMixPixels, p = e - c * kMixPixels;
            tg[c * (kMixPixels + 1) + p] = p < np ? __ldg(sg + (size_t)c * HW + p) : 0.f;
            tx[c * (kMixPixels + 1) + p] = p < np ? __ldg(sx + (size_t)c * HW + p) : 0.f;
        }
        __syncthreads();
        if (wide_acc) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = threadIdx.x + q * blockDim.x;
                if (q >= per || e >= NE) break;
                double a = dacc[q];
                if (e < C * C) {
                    const int o = e / C, c = e - o * C;
                    const float* pg = tg + o * (kMixPixels + 1);
                    const float* px = tx + c * (kMixPixels + 1);
                    for (int p = 0; p < kMixPixels; ++p) a = fma((double)pg[p], (double)px[p], a);
                } else {
                    const float* pg = tg + (e - C * C) * (kMixPixels + 1);
                    for (int p = 0; p < kMixPixels; ++p) a += (double)pg[p];
                }
                dacc[q] = a;
            }
            continue;
        }
        for (int q = 0; q < per; ++q) {
            const int e = threadIdx.x + q * blockDim.x;
            if (e >= NE) break;
            float a = acc[q];
            if (e < C * C) {
                const int o = e / C, c = e - o * C;
                const float* pg = tg + o * (kMixPixels + 1);
                const float* px = tx + c * (kMixPixels + 1);
                for (int p = 0; p < kMixPixels; ++p) a = fmaf(pg[p], px[p], a);
            } else {
                const float* pg = tg + (e - C * C) * (kMixPixels + 1);
                for (int p = 0; p < kMixPixels; ++p) a += pg[p];
            }
            acc[q] = a;
        }
    }
    for (int q = 0; q < per; ++q) {
        const int e = threadIdx.x + q * blockDim.x;
        if (e < NE) partials[(size_t)blockIdx.x * NE + e] = wide_acc ? dacc[q < 4 ? q : 0] : (double)acc[q];
    }
}

// The same for up to four channels: a thread per pixel keeps all C*C + C sums in double registers (the products of two fp32 are
// exact there), walks the pixels of its share, and the block adds its lanes' sums by shuffles.  The tile kernel above
// left 244 of its 256 threads without an entry (C = 3: 20 us; this one 4 us).
template <int C>
__global__ void __launch_bounds__(256) flow_mix_grad_few_kernel(const float* __restrict__ gu, const float* __restrict__ x,
                                                                double* __restrict__ partials, int B, int HW)
{
    constexpr int NE = C * C + C;
    __shared__ double red[8][NE];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    double acc[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) acc[e] = 0.0;
    const int total = B * HW, stride = gridDim.x * blockDim.x;
#pragma unroll 2
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        const int n = i / HW, px = i - n * HW;
        const float* pg = gu + (size_t)n * C * HW + px;
        const float* pxx = x + (size_t)n * C * HW + px;
        float g[C], v[C];
#pragma unroll
        for (int c = 0; c < C; ++c) { g[c] = __ldg(pg + c * HW); v[c] = __ldg(pxx + c * HW); }
#pragma unroll
        for (int o = 0; o < C; ++o) {
#pragma unroll
            for (int c = 0; c < C; ++c) acc[o * C + c] = fma((double)g[o], (double)v[c], acc[o * C + c]);
            acc[C * C + o] += (double)g[o];
        }
    }
#pragma unroll
    for (int e = 0; e < NE; ++e)
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int e = 0; e < NE; ++e) red[threadIdx.x >> 5][e] = acc[e];
    }
    __syncthreads();
    if (threadIdx.x < NE) {
        double a = 0.0;
        for (int w = 0; w < 8; ++w) a += red[w][threadIdx.x];
        partials[(size_t)blockIdx.x * NE + threadIdx.x] = a;
    }
}

// Sums entry e of the shares: `lanes` adjacent threads (a power of two up to 32) take every lanes-th share, in order and eight loads
// in flight, and are combined in a fixed order.  Every lane of the group returns the total.
__device__ __forceinline__ double sum_shares(const double* __restrict__ partials, int shares, int NE, int e, int lane, int lanes)
{
    double a = 0.0;
    for (int s0 = lane; s0 < shares; s0 += 8 * lanes) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = s0 + q * lanes < shares ? __ldcg(partials + (size_t)(s0 + q * lanes) * NE + e) : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) a += v[q];
    }
    for (int o = 1; o < lanes; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// Many entries: the sums over the shares on many CTAs (eight lanes per entry), in place of the first share.
__global__ void __launch_bounds__(256) flow_mix_grad_sum_kernel(const double* __restrict__ partials, double* __restrict__ G, int shares, int NE)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int e = (blockIdx.x * 256 + threadIdx.x) >> 3;
    const double a = sum_shares(partials, shares, NE, e < NE ? e : NE - 1, threadIdx.x & 7, 8);
    if (e < NE && (threadIdx.x & 7) == 0) G[e] = a;
}

// Sums the shares in order (unless `summed`: partials then holds the sums) and forms the parameter gradients:
//   grad_V[o][c] = s[c] * G1[o][c] + b[c] * g0[o];  grad_s[c] = sum_o V[o][c] * G1[o][c];  grad_b[c] = sum_o V[o][c] * g0[o].
__global__ void __launch_bounds__(1024) flow_mix_grad_final_kernel(const double* __restrict__ partials, int shares, int summed,
                                                                   const float* __restrict__ V, const float* __restrict__ s,
                                                                   const float* __restrict__ b, float* __restrict__ grad_V,
                                                                   float* __restrict__ grad_s, float* __restrict__ grad_b, int C, int lanes)
{
    extern __shared__ __align__(16) double fsmd[];
    double* G = fsmd;                 // [C*C + C]
    const int NE = C * C + C;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (summed || shares == 0) {
        for (int e = threadIdx.x; e < NE; e += blockDim.x) G[e] = shares == 0 ? 0.0 : __ldcg(partials + e);
    } else {
        const int per = blockDim.x / lanes, l = threadIdx.x & (lanes - 1), g = threadIdx.x / lanes;
        for (int e0 = 0; e0 < NE; e0 += per) {
            const int e = e0 + g;
            const double a = sum_shares(partials, shares, NE, e < NE ? e : NE - 1, l, lanes);
            if (e < NE && l == 0) G[e] = a;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < C * C; e += blockDim.x) {
        const int o = e / C, c = e - o * C;
        grad_V[e] = (float)((double)__ldg(s + c) * G[e] + (double)__ldg(b + c) * G[C * C + o]);
    }
    // a warp per channel: the sum over o in a fixed order
    for (int c = threadIdx.x >> 5; c < C; c += blockDim.x >> 5) {
        double gs = 0.0, gb = 0.0;
        for (int o = threadIdx.x & 31; o < C; o += 32) {
            const double v = (double)__ldg(V + o * C + c);
            gs += v * G[o * C + c];
            gb += v * G[C * C + o];
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) { gs += __shfl_xor_sync(0xffffffffu, gs, o); gb += __shfl_xor_sync(0xffffffffu, gb, o); }
        if ((threadIdx.x & 31) == 0) { grad_s[c] = (float)gs; grad_b[c] = (float)gb; }
    }
}

// logdet[0] = H*W * ( -sum_c log|w[c][c][k-1][k-1]| + sum_c log|s[c]| + log|det V| ), in double; the determinant by
// Gaussian elimination with partial pivoting in shared memory (one CTA, C <= 128): warp 0 finds the pivot among the rows
// not used yet (rows stay where they are, `used` marks them), then all threads eliminate.  Reads only the parameters, so it is
// launched dependently behind the solve and runs beside it; it waits for the solve before it ends, which keeps the stream's order.
__global__ void __launch_bounds__(256) flow_logdet_kernel(const float* __restrict__ w, const float* __restrict__ s,
                                                          const float* __restrict__ V, float* __restrict__ logdet,
                                                          int C, int H, int W, int K)
{
    extern __shared__ __align__(16) double dsm[];
    double* M = dsm;                  // [C][C]
    double* pivot = M + C * C;        // [C]
    __shared__ unsigned char used[128];
    __shared__ int piv;
    const int tid = threadIdx.x, lane = tid & 31;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int e = tid; e < C * C; e += blockDim.x) M[e] = (double)__ldg(V + e);
    if (tid < 128) used[tid] = 0;
    __syncthreads();
    for (int j = 0; j < C; ++j) {
        if (tid < 32) {
            double bv = -1.0;
            int best = 0;
            for (int i = lane; i < C; i += 32)
                if (!used[i] && fabs(M[i * C + j]) > bv) { bv = fabs(M[i * C + j]); best = i; }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const int oi = __shfl_xor_sync(0xffffffffu, best, o);
                if (ov > bv || (ov == bv && oi < best)) { bv = ov; best = oi; }
            }
            if (lane == 0) { piv = best; used[best] = 1; pivot[j] = bv; }
        }
        __syncthreads();
        const int pr = piv;
        const double inv = 1.0 / M[pr * C + j];
        const int cols = C - j - 1;
        for (int i = tid >> 5; i < C; i += blockDim.x >> 5) {
            if (used[i]) continue;
            const double f = M[i * C + j] * inv;
            for (int c = lane; c < cols; c += 32) M[i * C + j + 1 + c] -= f * M[pr * C + j + 1 + c];
        }
        __syncthreads();
    }
    if (tid < 32) {
        double a = 0.0;
        for (int c = lane; c < C; c += 32)
            a += log(fabs((double)__ldg(s + c))) - log(fabs((double)__ldg(w + ((size_t)(c * C + c) * K + (K - 1)) * K + (K - 1)))) + log(pivot[c]);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) logdet[0] = (float)((double)(H * W) * a);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launch with programmatic dependence on the kernel before: every kernel launched this way waits for it (griddepcontrol.wait).
template <typename... P, typename... A>
int launch_dependent(void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t st, A... args)
{
    const int rc = invconv_internal::set_smem_limit(kern, smem);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) != cudaSuccess) { cudaGetLastError(); return INVCONV_CUDA_ERROR; }
    return check_launch();
}

struct Scratch {
    void* p = nullptr;
    cudaStream_t st = nullptr;
    int acquire(size_t bytes, cudaStream_t s)
    {
        st = s;
        if (bytes == 0) return INVCONV_OK;
        { const int rc = invconv_internal::scratch_alloc(&p, bytes, st); if (rc) { p = nullptr; return rc; } }
        if (cudaMemsetAsync(p, 0, INVCONV_WS_CONTROL_BYTES, st) != cudaSuccess) { cudaGetLastError(); return INVCONV_CUDA_ERROR; }
        return INVCONV_OK;
    }
    ~Scratch() { if (p) cudaFreeAsync(p, st); }
};

inline size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

template <bool BWD>
int launch_mix(const float* in, const float* V, const float* s, const float* b, float* out, int B, int C, int HW, cudaStream_t st)
{
    const int tiles = (HW + kMixPixels - 1) / kMixPixels;
    const size_t sm = sizeof(float) * ((size_t)C * (C + 1) + C + (size_t)C * kMixPixels);
    auto kern = flow_mix_kernel<BWD>;
    const int rc = invconv_internal::set_smem_limit(kern, sm);
    if (rc) return rc;
    kern<<<B * tiles, 256, sm, st>>>(in, V, s, b, out, C, HW, tiles);
    return check_launch();
}

}  // namespace

namespace invconv_internal {

int flow_bounds_info(int* info)
{
#ifdef INVCONV_DEBUG_BOUNDS
    const int zero[4] = {0, 0, 0, 0};
    if (cudaMemcpyFromSymbol(info, g_bounds_record, 4 * sizeof(int)) != cudaSuccess) { cudaGetLastError(); return INVCONV_CUDA_ERROR; }
    cudaMemcpyToSymbol(g_bounds_record, zero, sizeof(zero));
#else
    info[0] = info[1] = info[2] = info[3] = 0;
#endif
    return INVCONV_OK;
}

}  // namespace invconv_internal

namespace {

// Scratch of a flow-step call: the layer's own workspace (its control words first), the gradient with respect to x where the
// step is composed, and the shares of the parameter gradients.
struct FlowScratch {
    size_t layer, act, part, total;
    int tiles, shares;
};

FlowScratch flow_scratch(int B, int C, int H, int W, int k)
{
    FlowScratch f;
    f.layer = up256(invconv_workspace_bytes(B > 0 ? B : 1, C, H, W, k) + INVCONV_WS_CONTROL_BYTES);
    f.act = up256(sizeof(float) * (size_t)B * C * H * W);
    f.tiles = (H * W + kMixPixels - 1) / kMixPixels;
    f.shares = invconv_internal::sm_count();
    if (f.shares > B * f.tiles) f.shares = B * f.tiles;
    if (f.shares < 1) f.shares = 1;
    f.part = up256(sizeof(double) * ((size_t)C * C + C) * (f.shares + 1));
    f.total = f.layer + f.act + f.part;
    return f;
}

bool bad_shape(int B, int C, int H, int W, int k, int* rc)
{
    *rc = INVCONV_OK;
    if (B < 0 || C < 1 || H < 1 || W < 1 || k < 1) *rc = INVCONV_BAD_ARG;
    else if (k > INVCONV_MAX_K || C > INVCONV_MAX_C || (long long)B * C * H * W >= (1LL << 31)) *rc = INVCONV_UNSUPPORTED;
    return *rc != INVCONV_OK;
}

}  // namespace

extern "C" {

size_t invconv_flow_step_workspace_bytes(int B, int C, int H, int W, int k)
{
    int rc;
    if (bad_shape(B, C, H, W, k, &rc)) return 0;
    return flow_scratch(B, C, H, W, k).total;
}

int invconv_flow_step_forward_ws(const float* y, const float* w, const float* s, const float* b, const float* V,
                                 float* x, float* u, float* logdet, int B, int C, int H, int W, int k,
                                 void* workspace, size_t workspace_bytes, void* stream)
{
    int rc;
    if (bad_shape(B, C, H, W, k, &rc)) return rc;
    if (!w || !s || !b || !V) return INVCONV_BAD_ARG;
    if (B > 0 && (!y || !x || !u || y == x || u == x || u == y)) return INVCONV_BAD_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (B > 0) {
        if (!workspace || workspace_bytes < flow_scratch(B, C, H, W, k).total) return INVCONV_WORKSPACE_TOO_SMALL;
        rc = invconv_internal::warp_step_forward(y, w, s, b, V, x, u, Geom{B, C, H, W, k}, workspace, st);
        if (rc == INVCONV_UNSUPPORTED) {
            rc = invconv_forward_ws(y, w, x, B, C, H, W, k, workspace, workspace_bytes, stream);
            if (rc) return rc;
            rc = launch_mix<false>(x, V, s, b, u, B, C, H * W, st);
        }
        if (rc) return rc;
    }
    if (logdet) {
        return launch_dependent(flow_logdet_kernel, 1, 256, sizeof(double) * ((size_t)C * C + C), st, w, s, V, logdet, C, H, W, k);
    }
    return INVCONV_OK;
}

int invconv_flow_step_forward(const float* y, const float* w, const float* s, const float* b, const float* V,
                              float* x, float* u, float* logdet, int B, int C, int H, int W, int k, void* stream)
{
    Scratch sc;
    const size_t need = B > 0 ? invconv_flow_step_workspace_bytes(B, C, H, W, k) : 0;
    const int ra = sc.acquire(need, reinterpret_cast<cudaStream_t>(stream));
    if (ra) return ra;
    return invconv_flow_step_forward_ws(y, w, s, b, V, x, u, logdet, B, C, H, W, k, sc.p, need, stream);
}

int invconv_flow_step_backward_ws(const float* grad_u, const float* x, const float* w, const float* s, const float* b,
                                  const float* V, float* grad_y, float* grad_w, float* grad_s, float* grad_b, float* grad_V,
                                  int B, int C, int H, int W, int k, void* workspace, size_t workspace_bytes, void* stream)
{
    int rc;
    if (bad_shape(B, C, H, W, k, &rc)) return rc;
    if (!w || !s || !b || !V || !grad_w || !grad_s || !grad_b || !grad_V) return INVCONV_BAD_ARG;
    if (B > 0 && (!grad_u || !x || !grad_y || grad_u == grad_y || x == grad_y)) return INVCONV_BAD_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int HW = H * W;
    const FlowScratch f = flow_scratch(B, C, H, W, k);
    if (!workspace || workspace_bytes < f.total) return INVCONV_WORKSPACE_TOO_SMALL;
    char* base = static_cast<char*>(workspace);
    float* grad_x = reinterpret_cast<float*>(base + f.layer);
    double* partials = reinterpret_cast<double*>(base + f.layer + f.act);
    int shares = f.shares;
    if (B > 0) {
        rc = invconv_internal::warp_step_backward(grad_u, x, w, s, V, grad_y, grad_w, Geom{B, C, H, W, k}, workspace, st);
        if (rc == INVCONV_UNSUPPORTED) {
            rc = launch_mix<true>(grad_u, V, s, b, grad_x, B, C, HW, st);
            if (rc) return rc;
            rc = invconv_backward_ws(grad_x, x, w, grad_y, grad_w, B, C, H, W, k, workspace, f.layer, stream);
        }
        if (rc) return rc;
        if (C <= 4) {
            switch (C) {
            case 1: rc = launch_dependent(flow_mix_grad_few_kernel<1>, shares, 256, 0, st, grad_u, x, partials, B, HW); break;
            case 2: rc = launch_dependent(flow_mix_grad_few_kernel<2>, shares, 256, 0, st, grad_u, x, partials, B, HW); break;
            case 3: rc = launch_dependent(flow_mix_grad_few_kernel<3>, shares, 256, 0, st, grad_u, x, partials, B, HW); break;
            default: rc = launch_dependent(flow_mix_grad_few_kernel<4>, shares, 256, 0, st, grad_u, x, partials, B, HW); break;
            }
        } else {
            rc = launch_dependent(flow_mix_grad_kernel, shares, 256, sizeof(float) * 2 * (size_t)C * (kMixPixels + 1), st, grad_u, x, partials,
                                  B, C, HW, f.tiles);
        }
        if (rc) return rc;
    } else {
        rc = invconv_backward_ws(grad_u, x, w, grad_y, grad_w, 0, C, H, W, k, nullptr, 0, stream);   // zeroes grad_w
        if (rc) return rc;
        shares = 0;
    }
    // few entries: summed by the final kernel itself, as many lanes per entry as its 1024 threads give; many: on CTAs of their own
    const int NE = C * C + C;
    const bool separate = NE > 512 && shares > 0;
    if (separate) {
        double* sums = partials + (size_t)NE * shares;
        rc = launch_dependent(flow_mix_grad_sum_kernel, (NE * 8 + 255) / 256, 256, 0, st, partials, sums, shares, NE);
        if (rc) return rc;
        partials = sums;
    }
    int lanes = 1;
    while (lanes < 32 && NE * lanes * 2 <= 1024) lanes *= 2;
    return launch_dependent(flow_mix_grad_final_kernel, 1, 1024, sizeof(double) * (size_t)NE, st, partials, shares, separate ? 1 : 0, V, s, b,
                            grad_V, grad_s, grad_b, C, lanes);
}

int invconv_flow_step_backward(const float* grad_u, const float* x, const float* w, const float* s, const float* b,
                               const float* V, float* grad_y, float* grad_w, float* grad_s, float* grad_b, float* grad_V,
                               int B, int C, int H, int W, int k, void* stream)
{
    Scratch sc;
    const size_t need = invconv_flow_step_workspace_bytes(B, C, H, W, k);
    const int ra = sc.acquire(need, reinterpret_cast<cudaStream_t>(stream));
    if (ra) return ra;
    return invconv_flow_step_backward_ws(grad_u, x, w, s, b, V, grad_y, grad_w, grad_s, grad_b, grad_V, B, C, H, W, k, sc.p, need, stream);
}

}  // extern "C"
