// LINE wavefront: one thread per (image row, output channel), for few and medium channel counts, any image size.
//
// A CTA walks the anti-diagonals of one image at a time (Section 3: pixels on one anti-diagonal are unordered).  Row r
// is at column s - r in step s.  The substitution runs in SCATTER form: with A_delta = L^-1 W_delta (the kernel in
// the paper's unit-diagonal form) and A_0 = L^-1,
//     u[p] = A_0 rhs[p] - sum_{delta != 0} A_delta u[p - delta],
// a thread (row r, channel a) keeps row a of every A_delta in registers together with 2K-3 pending sums, one for each of
// the next columns of its row.  In a step it reads the newest solved pixel of rows r, r-1, ... r-K+1 (K short vectors of
// C channels from a small exchange buffer in shared memory), finishes its own pixel with the two taps that reach it from
// them -- (0,1) and (1,0), the only ones on the dependent chain --, publishes it, and then adds every other tap of those
// vectors to the pending sums.  Each value is read once and used for K taps; nothing but the newest pixel of each
// row is ever exchanged, so shared memory holds no image and the image size is not limited by it.
//
// Reading and writing global memory is the job of separate I/O warps: a ring of 32 columns per row takes the right-hand
// side in chunks of eight columns, requested three and placed two chunks ahead of the wavefront; the solution overwrites it in
// place and leaves one chunk behind.  Images taller than a CTA's rows are walked in bands from top to bottom; the K-1 rows above
// a band are "halo" rows whose threads publish the values that the band before wrote to global memory.  Images and bands
// follow one another on one virtual column axis with zero columns between them, so a CTA with several images pays the ramp
// of the wavefront once.
//
// The compute warps share one named barrier per step (a barrier, a shared-memory load and a short dependent sum take about
// 80 to 110 cycles; an mbarrier that lets a warp's other multiply-adds overlap the wait was measured 60 to 70 cycles
// slower per step); chunks are handed over between compute and I/O warps through mbarriers.
//
// The transposed solve (Theorem 1) is the same walk on the image rotated by 180 degrees with L^-T W_delta^T.
//
// Bound: for few channels the dependent step (barrier, shared-memory load, 2C multiply-adds, store), for many the FMA
// pipe (C*C*K*K multiply-adds per pixel at 1.2 to 1.5 cycles per warp instruction, measured; packed fma.f32x2 gives the
// same rate in half the issue slots and is used for even channel counts).
#pragma once

#include <cuda_bf16.h>
#include <type_traits>

#include "common.cuh"
#include "tma.cuh"
#include "line_params.h"
#include "line_plan.h"

namespace invconv {

namespace line_detail {

using u64 = unsigned long long;
constexpr int kRing = 32;

// The NB input channels of a slice as NV operands: packed pairs for even NB.
template <int NB, bool PACK = (NB % 2 == 0)>
struct Vec {
    static constexpr int NV = NB;
    using T = float;
    static __device__ __forceinline__ T fma(T a, T b, T c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ float sum(T a) { return a; }
    static __device__ __forceinline__ T zero() { return 0.f; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    template <bool AL16>
    static __device__ __forceinline__ void load(const float* p, T (&v)[NV])
    {
        if constexpr (AL16 && NB >= 3) {
#pragma unroll
            for (int q = 0; q < (NB + 3) / 4; ++q) {
                if (NB - 4 * q == 1) { v[4 * q] = p[4 * q]; continue; }
                const float4 t = *reinterpret_cast<const float4*>(p + 4 * q);
                const float e[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) if (4 * q + j < NB) v[4 * q + j] = e[j];
            }
        } else {
#pragma unroll
            for (int q = 0; q < NB; ++q) v[q] = p[q];
        }
    }
};
template <int NB>
struct Vec<NB, true> {
    static constexpr int NV = NB / 2;
    using T = u64;
    static __device__ __forceinline__ T fma(T a, T b, T c)
    {
        T d;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
        return d;
    }
    static __device__ __forceinline__ float sum(T a)
    {
        float lo, hi;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
        return lo + hi;
    }
    static __device__ __forceinline__ T zero() { return 0ull; }
    static __device__ __forceinline__ T pair(float lo, float hi)
    {
        T d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
        return d;
    }
    static __device__ __forceinline__ T add(T a, T b)
    {
        T d;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
        return d;
    }
    template <bool AL16>
    static __device__ __forceinline__ void load(const float* p, T (&v)[NV])
    {
        if constexpr (AL16) {
#pragma unroll
            for (int q = 0; q < NV / 2; ++q) {
                const ulonglong2 t = reinterpret_cast<const ulonglong2*>(p)[q];
                v[2 * q] = t.x; v[2 * q + 1] = t.y;
            }
            if constexpr (NV % 2 == 1) v[NV - 1] = reinterpret_cast<const T*>(p)[NV - 1];
        } else {
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] = reinterpret_cast<const T*>(p)[q];
        }
    }
};

__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

// The transformed kernel into shared memory: As[(tap*CSB + b)*CA + a], tap = dh*K + dw, CA = C|1, negative for every tap but
// 0, zero for b >= C.  wsm holds w ([C][C][K][K]); li is scratch for L^-1.  The caller has zeroed As and li
// and synchronised after filling wsm.
//   forward : A[a][b] = sum_m Li[a][m] w[m][b][tap'],   backward: sum_m Li[m][a] w[b][m][tap'],   Li = L^-1, tap' flipped
// With mix_in tap 0 also carries the flow step's neighbours: A_0 diag(s) V^T.
// Only the NT compute threads take part (named barrier 1).  A warp forms four columns of L^-1 at a time: lane i holds the
// residuals of row i, a step is one shuffle and one multiply-add on the dependent chain.  The products keep a column of W in
// registers and read rows of L^-1 as 16-byte broadcasts.  The code is kept short on purpose: it runs once, and
// unrolled versions spent longer on instruction fetches than on arithmetic.
template <int K, int CSB>
__device__ void build_kernel(const LineParams& p, float* As, const float* wsm, float* li, int NT)
{
    constexpr int KK = K * K, ctr = KK - 1, LS = (CSB + 3) / 4 * 4;
    const int C = p.C, tid = threadIdx.x, lane = tid & 31, CA = C | 1;
    for (int j0 = (tid >> 5) * 4; j0 < C; j0 += (NT >> 5) * 4) {
        const float d = lane < C ? 1.0f / wsm[(lane * C + lane) * KK + ctr] : 0.f;
        float r[4], y[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) { r[q] = lane == j0 + q ? 1.f : 0.f; y[q] = 0.f; }
        for (int i = j0; i < C; ++i) {
            const float l = lane > i && lane < C ? wsm[(lane * C + i) * KK + ctr] : 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float yi = __shfl_sync(0xffffffffu, r[q] * d, i);
                y[q] = lane == i ? yi : y[q];
                r[q] = fmaf(-l, yi, r[q]);
            }
        }
        // li[a*LS + m] = Li[a][m] (forward) or Li[m][a] (backward)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (lane < C && j0 + q < C) li[p.rot ? (j0 + q) * LS + lane : lane * LS + j0 + q] = y[q];
    }
    bar_sync(1, NT);
    // column (tap, b) per lane of bk_warps warps; the warps beyond them take further shares of the rows a
    const int wq = fast_div(tid >> 5, p.div_bk), part = wq;
    if (part < p.bk_parts) {
        const int a0 = part * p.bk_per, a1 = min(C, a0 + p.bk_per);
        for (int col = tid - part * p.bk_warps * 32; col < C * (KK - 1); col += p.bk_warps * 32) {
            const int tq = fast_div(col, p.div_c), b = col - tq * C, tap = tq + 1;
            const float* src = wsm + (p.rot ? b * C : b) * KK + KK - 1 - tap;
            const int st = p.rot ? KK : C * KK;
            float wv[LS];
#pragma unroll
            for (int m = 0; m < LS; ++m) wv[m] = m < C ? src[m * st] : 0.f;
#pragma unroll 2
            for (int a = a0; a < a1; ++a) {
                float v0 = 0.f, v1 = 0.f;
#pragma unroll
                for (int m = 0; m < LS; m += 4) {
                    const float4 l = *reinterpret_cast<const float4*>(li + a * LS + m);
                    v0 = fmaf(l.x, wv[m], v0); v1 = fmaf(l.y, wv[m + 1], v1);
                    v0 = fmaf(l.z, wv[m + 2], v0); v1 = fmaf(l.w, wv[m + 3], v1);
                }
                As[(tap * CSB + b) * CA + a] = -(v0 + v1);
            }
        }
    }
    for (int e = tid; e < C * C; e += NT) {
        const int b = fast_div(e, p.div_c), a = e - b * C;
        float v = 0.f;
        if (!p.mix_in) v = li[a * LS + b];
        else
            for (int m = 0; m < C; ++m) v = fmaf(li[a * LS + m], __ldg(p.mix_s + m) * __ldg(p.mix_V + b * C + m), v);
        As[b * CA + a] = v;
    }
    bar_sync(1, NT);
}

}  // namespace line_detail

// NB: input channels per slice; S: slices (adjacent lanes) that share an output; PR: adjacent rows per thread.
template <int NB, int K, int S, int PR, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) line_wavefront_kernel(const __grid_constant__ LineParams p)
{
    using namespace line_detail;
    using V = Vec<NB>;
    using T = typename V::T;
    constexpr int NV = V::NV, KK = K * K, KM = K - 1;
    constexpr int NPEND = 2 * K - 3;                   // pending sums: the next columns that solved pixels reach
    constexpr int CSB = S * NB, CS = (CSB + 3) / 4 * 4;          // channels of a pixel in shared memory, padded to 16 bytes
    constexpr int RS = line_row_stride(kRing, CS);
    constexpr bool AL16 = S == 1 || NB % 4 == 0;
    constexpr int UNR = PR * NV * KK <= 64 ? 4 : 2;    // steps per turn of the loop
    extern __shared__ __align__(128) float sm[];
    __shared__ unsigned long long bars[4];             // chunk ready [2], chunk done [2]
    __shared__ int gave_up_flag;
    volatile int* gave_up = &gave_up_flag;
    const int C = p.C, H = p.H, W = p.W, HW = H * W;
    const int HBt = p.HB + p.halo;
    const int exrow = (HBt + KM + PR) * CS;
    float* EX = sm;                                    // [2][HBt + K-1 + PR][CS]: newest pixel of every row, by step
    float* RG = sm + p.off_ring;                       // [HBt][32 columns][CS] (row stride RS)
    float* As = sm + p.off_a;
    unsigned long long* ready_bar = bars;
    unsigned long long* done_bar = bars + 2;
    float* const dummy = sm + p.off_dummy;             // scratch words for lanes without a pixel
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int NT = blockDim.x, nct = p.ncw * 32;
    const int nimg = (p.B - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // images blockIdx.x, + gridDim.x, ...
    const int nseg = nimg * p.nbands;
    const int VC = (nseg - 1) * p.SW + W;              // virtual columns
    const int T_compute = (VC + p.HB - 1 + 7) >> 3;    // intervals of eight steps
    const int T_end = ((VC - 1) >> 3) + 1 + ((p.HB - 1 + 7) >> 3);

    if (tid == 0) {
        mbar_init(ready_bar, p.niow * 32); mbar_init(ready_bar + 1, p.niow * 32);
        mbar_init(done_bar, p.ncw); mbar_init(done_bar + 1, p.ncw);
        gave_up_flag = 0;
        fence_mbar_init();
    }
    for (int i = tid; i < 2 * exrow; i += NT) EX[i] = 0.f;
    if (C < CSB)                                       // channels beyond C meet zero weights but must not be NaN
        for (int i = tid; i < HBt * RS; i += NT) RG[i] = 0.f;
    for (int i = p.off_a + tid; i < p.off_w; i += NT) sm[i] = 0.f;     // As and li
    __syncthreads();
    // everything above touched no global memory; from here on the predecessor kernel's results are needed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---------------------------------------------------------------- I/O
    // A piece is four columns of one (row, channel), half a chunk; a thread owns the same BV pieces of every chunk, so it may
    // place a chunk where it has just stored one.  Row r is floor(r/8) chunks behind row 0 when read, ceil(r/8) when
    // stored.  Loads are unconditional (from a valid address) and kept as raw bits until they are placed, so that all of
    // a thread's requests are in flight at once.
    constexpr int BV = line_pieces(NB, S);
    const bool io_warp = warp >= p.ncw;
    const int io = tid - nct, nio = p.niow * 32;
    const int half4 = 4 * (io & 1), sgn = p.rot ? -1 : 1;
    int ring_off[BV], gofs[BV], row[BV];
    // per piece: column within its segment, segment, and the element of the segment row's first column (-1: no such row) --
    // of the chunk requested next and of the chunk stored next
    int rcol[BV], rseg[BV], rbase[BV], scol[BV], sseg[BV], sbase[BV];
    auto seg_base = [&](int b, int seg) -> int {
        if (seg >= nseg) return -1;
        const int i = p.nbands == 1 ? seg : fast_div(seg, p.div_nb), band = seg - i * p.nbands;
        const int h = band * p.HB + row[b];
        if (h < 0 || h >= H) return -1;
        return ((int)blockIdx.x + i * (int)gridDim.x) * C * HW + gofs[b] + sgn * band * p.HB * W;
    };
    if (io_warp) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const int rc = (io + b * nio) >> 1, rr = fast_div(rc, p.div_c), c = rc - rr * C, r = rr - p.halo;
            const bool ok = rr < HBt;
            row[b] = ok ? r : -1000000;                // never inside the image
            ring_off[b] = ok ? rr * RS + c : 0;
            gofs[b] = ok ? c * HW + (p.rot ? HW - 1 - r * W : r * W) : 0;
            rcol[b] = half4 - (ok ? 8 * (r >> 3) : 0); scol[b] = half4 - (ok ? 8 * ((r + 7) >> 3) : 0);
            rseg[b] = 0; sseg[b] = 0;
            rbase[b] = seg_base(b, 0);
            sbase[b] = r < 0 ? -1 : rbase[b];
        }
    }
    auto advance = [&](int b, int& col, int& seg, int& base) {
        col += 8;
        if (nseg > 1)
            while (col >= p.SW) { col -= p.SW; ++seg; base = seg_base(b, seg); }
    };
    const int safe = (int)blockIdx.x * C * HW;         // an element every load may touch
    // fp32: asynchronous copies straight into the ring (chunk t), zeros outside the image
    auto copy = [&](int t) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const bool have = rbase[b] >= 0 && rcol[b] >= 0;
            const int vc = 8 * (t - (row[b] >> 3)) + half4;
            const float* g = reinterpret_cast<const float*>(row[b] < 0 ? p.out : p.rhs) + (have ? rbase[b] + sgn * rcol[b] : safe);
            float* d = row[b] > -1000 ? RG + ring_off[b] + (vc & (kRing - 1)) * CS : dummy;
            const int ds = row[b] > -1000 ? CS : 0, left = have ? W - rcol[b] : 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) cp_async_f32(d + j * ds, j < left ? g + sgn * j : g, j < left);
            advance(b, rcol[b], rseg[b], rbase[b]);
        }
    };
    // bf16: requested into registers a chunk ahead, widened when placed
    int rnv[BV];                                       // columns inside the image of the pieces requested last
    auto request = [&](unsigned (&v)[4 * BV]) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const int nv = rbase[b] >= 0 && rcol[b] >= 0 ? min(max(W - rcol[b], 0), 4) : 0;
            const int f = rbase[b] + sgn * rcol[b];
            rnv[b] = nv;
            const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(row[b] < 0 ? p.out : p.rhs);
            if (p.vec) {
                const uint2 u = *reinterpret_cast<const uint2*>(src + (nv > 0 ? (p.rot ? f - 3 : f) : safe));
                v[4 * b] = u.x; v[4 * b + 1] = u.y;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) v[4 * b + j] = reinterpret_cast<const unsigned short*>(src)[j < nv ? f + sgn * j : safe];
            }
            advance(b, rcol[b], rseg[b], rbase[b]);
        }
    };
    auto place = [&](const unsigned (&v)[4 * BV], int t) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const int vc = 8 * (t - (row[b] >> 3)) + half4;
            unsigned u[4];
            if (p.vec) { u[3] = v[4 * b + 1] & 0xffff0000u; u[2] = v[4 * b + 1] << 16; u[1] = v[4 * b] & 0xffff0000u; u[0] = v[4 * b] << 16; }
            else {
#pragma unroll
                for (int j = 0; j < 4; ++j) u[j] = v[4 * b + j] << 16;
            }
            float* d = row[b] > -1000 ? RG + ring_off[b] + (vc & (kRing - 1)) * CS : dummy;
            const int ds = row[b] > -1000 ? CS : 0;
            const bool flip = p.vec && p.rot;
#pragma unroll
            for (int j = 0; j < 4; ++j) d[j * ds] = j < rnv[b] ? __uint_as_float(flip ? u[3 - j] : u[j]) : 0.f;
        }
    };
    // u = V (s x + b) of the flow step for one channel of one pixel
    auto mixed = [&](const float* px, int c) -> float {
        float u = 0.f;
        for (int m = 0; m < C; ++m) u = fmaf(__ldg(p.mix_V + c * C + m), fmaf(__ldg(p.mix_s + m), px[m], __ldg(p.mix_b + m)), u);
        return u;
    };
    auto store = [&](int t) {
        float f[BV][4];
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const int vc = 8 * (t - ((row[b] + 7) >> 3)) + half4;
            const float* px = RG + ring_off[b] + (vc & (kRing - 1)) * CS;
#pragma unroll
            for (int j = 0; j < 4; ++j) f[b][j] = px[j * CS];
        }
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const int nv = sbase[b] >= 0 && scol[b] >= 0 ? min(max(W - scol[b], 0), 4) : 0;
            int i = sbase[b] + sgn * scol[b];
            advance(b, scol[b], sseg[b], sbase[b]);
            if (row[b] < 0) sbase[b] = -1;             // halo rows are not stored
            if (nv == 0) continue;
            if (p.vec) {
                float g[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) g[j] = p.rot ? f[b][3 - j] : f[b][j];
                if (p.rot) i -= 3;
                if (p.bf16) {
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(g[0], g[1]), hi = __floats2bfloat162_rn(g[2], g[3]);
                    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + i) =
                        make_uint2(*reinterpret_cast<const unsigned*>(&lo), *reinterpret_cast<const unsigned*>(&hi));
                } else {
                    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + i) = make_float4(g[0], g[1], g[2], g[3]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < nv) {
                        if (p.bf16) reinterpret_cast<__nv_bfloat16*>(p.out)[i + sgn * j] = __float2bfloat16_rn(f[b][j]);
                        else reinterpret_cast<float*>(p.out)[i + sgn * j] = f[b][j];
                    }
            }
            if (p.mix_out != nullptr) {                  // forward only
                const int c = ring_off[b] % RS, vc = 8 * (t - ((row[b] + 7) >> 3)) + half4;
                for (int j = 0; j < nv; ++j) p.mix_out[i + j] = mixed(RG + ring_off[b] - c + ((vc + j) & (kRing - 1)) * CS, c);
            }
        }
    };
    if (!io_warp) {
        {
            float* wsm = sm + p.off_w;
            const int NW = C * C * KK;
            for (int e0 = tid; e0 < NW; e0 += 8 * nct) {
                float t[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) t[q] = e0 + q * nct < NW ? __ldg(p.w + e0 + q * nct) : 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) if (e0 + q * nct < NW) wsm[e0 + q * nct] = t[q];
            }
            bar_sync(1, nct);
            build_kernel<K, CSB>(p, As, wsm, sm + p.off_li, nct);
        }
        const int ti = tid / S, sl = tid - ti * S;
        const int g = fast_div(ti, p.div_c), a = ti - g * C;      // row group, channel
        const bool live = g * PR < HBt;
        const int rr0 = live ? g * PR : 0;
        T W0[NV], Wt[KK][NV];
        {
            const int CA = C | 1;
            const float* src = As + sl * NB * CA + (live ? a : 0);
#pragma unroll
            for (int t = 0; t < KK; ++t)
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    T v;
                    if constexpr (NB % 2 == 0) v = V::pair(src[(t * CSB + 2 * q) * CA], src[(t * CSB + 2 * q + 1) * CA]);
                    else v = src[(t * CSB + q) * CA];
                    if (t == 0) W0[q] = v; else Wt[t][q] = v;
                }
        }
        T acc[PR][NPEND];
#pragma unroll
        for (int i = 0; i < PR; ++i)
#pragma unroll
            for (int j = 0; j < NPEND; ++j) acc[i][j] = V::zero();
        // band of the row's segment, and the columns the row has there: none for rows outside the image and for the halo rows of
        // the first band
        int band[PR];
        unsigned width[PR];
        auto row_width = [&](int i, int bnd) -> unsigned {
            const int r = rr0 + i - p.halo;
            const bool have = live && rr0 + i < HBt && (r < 0 ? bnd > 0 : bnd * p.HB + r < H);
            return have ? (unsigned)W : 0u;
        };
#pragma unroll
        for (int i = 0; i < PR; ++i) { band[i] = 0; width[i] = row_width(i, 0); }
        // rows of this warp: the warp works in an interval while any of them is between K-1 columns before its first and its last
        const int g_lo = fast_div((warp * 32) / S, p.div_c), g_hi = fast_div((warp * 32 + 31) / S, p.div_c);
        const int t_lo = max(0, (g_lo * PR - p.halo - KM) >> 3), t_hi = (VC + min(g_hi * PR + PR - 1, HBt - 1) - p.halo + 7) >> 3;
        // column within the segment of each row's pixel in the warp's first step; negative before its first column
        int col[PR];
#pragma unroll
        for (int i = 0; i < PR; ++i) col[i] = 8 * t_lo - (rr0 + i - p.halo);
        bool pub[PR];                                  // this lane publishes the row's pixel
#pragma unroll
        for (int i = 0; i < PR; ++i) pub[i] = live && sl == 0 && rr0 + i < HBt;
        float* const ex_rd = EX + (rr0 + KM) * CS + sl * NB;
        float* const ex_wr = EX + (rr0 + KM) * CS + a;
        float* const ring0 = RG + rr0 * RS;
        // One step; `odd`: its parity, HALO: the CTA walks bands.  No branches: on the dependent path of a step each cost 15 to
        // 20 cycles (a C = 3, k = 3 step went from 310 to 150 cycles).
        auto step = [&](int s, bool odd, auto halo_tag) {
            constexpr bool HALO = decltype(halo_tag)::value;
            const int rd = odd ? 0 : exrow, wr = exrow - rd;
            // newest pixels of the rows this thread's rows can see (v[m] is row rr0 + PR-1 - m) and the right-hand sides of the
            // next columns; all loads go first, so that the sums off the dependent chain fill its gaps
            T v[PR + KM][NV], rh[PR][NV];
#pragma unroll
            for (int m = 0; m < PR + KM; ++m) V::template load<AL16>(ex_rd + rd + (PR - 1 - m) * CS, v[m]);
#pragma unroll
            for (int i = 0; i < PR; ++i)
                V::template load<AL16>(ring0 + i * RS + ((s - (rr0 + i - p.halo) + 1) & (kRing - 1)) * CS + sl * NB, rh[i]);
#pragma unroll
            for (int i = 0; i < PR; ++i) {
                T c0 = acc[i][0], c1 = V::zero();
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    c0 = V::fma(Wt[1][q], v[PR - 1 - i][q], c0);
                    c1 = V::fma(Wt[K][q], v[PR - i][q], c1);
                }
                float x = V::sum(V::add(c0, c1));
#pragma unroll
                for (int o = 1; o < S; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                // lanes without a pixel store to scratch words
                float* rg = ring0 + i * RS + ((s - (rr0 + i - p.halo)) & (kRing - 1)) * CS + a;
                const bool inside = (unsigned)col[i] < width[i];
                if constexpr (HALO) {                            // halo row: the value the band above left
                    const float h = *rg;
                    x = rr0 + i < p.halo ? h : x;
                }
                x = inside ? x : 0.f;
                *(pub[i] ? ex_wr + wr + i * CS : dummy) = x;
                *(pub[i] && inside && (!HALO || rr0 + i >= p.halo) ? rg : dummy) = x;
            }
            // off the dependent chain: the pending sums of the next columns, two per column (even and odd kernel rows), so that no
            // chain of multiply-adds is longer than its issue
#pragma unroll
            for (int i = 0; i < PR; ++i) {
                T na[NPEND], nb[NPEND];
#pragma unroll
                for (int j = 0; j < NPEND; ++j) { na[j] = j + 1 < NPEND ? acc[i][j + 1 < NPEND ? j + 1 : 0] : V::zero(); nb[j] = V::zero(); }
#pragma unroll
                for (int dh = 0; dh < K; ++dh)
#pragma unroll
                    for (int q = 0; q < NV; ++q)
#pragma unroll
                        for (int dw = 0; dw < K; ++dw)
                            if (dh + dw >= 2) {
                                T& sum = (dh & 1) ? nb[dh + dw - 2] : na[dh + dw - 2];
                                sum = V::fma(Wt[dh * K + dw][q], v[PR - 1 - i + dh][q], sum);
                            }
#pragma unroll
                for (int q = 0; q < NV; ++q) nb[0] = V::fma(W0[q], rh[i][q], nb[0]);
#pragma unroll
                for (int j = 0; j < NPEND; ++j) acc[i][j] = V::add(na[j], nb[j]);
                const bool wrap = ++col[i] == p.SW;
                col[i] = wrap ? 0 : col[i];
                if constexpr (HALO) {
                    if (wrap) {
                        band[i] = band[i] + 1 == p.nbands ? 0 : band[i] + 1;
                        width[i] = row_width(i, band[i]);
                    }
                }
            }
        };
        auto walk = [&](auto halo_tag) {
            for (int t = 0; t < T_compute; ++t) {
                // interval t-1 is finished; chunk t+1 (and all before it) is in the ring
                __syncwarp();
                if (t > 0 && lane == 0) mbar_arrive(done_bar + (t & 1));
                mbar_wait_or_give_up(ready_bar + (t & 1), (t >> 1) & 1, gave_up);
                if (t >= t_lo && t < t_hi) {                     // warp-uniform
                    if (t == 0) {
                        // the first row's first pixel: its right-hand side is otherwise taken one step ahead
#pragma unroll
                        for (int i = 0; i < PR; ++i) {
                            T rh[NV];
                            V::template load<AL16>(ring0 + i * RS + sl * NB, rh);
                            if (rr0 + i == p.halo) {
#pragma unroll
                                for (int q = 0; q < NV; ++q) acc[i][0] = V::fma(W0[q], rh[q], acc[i][0]);
                            }
                        }
                    }
#pragma unroll(UNR)
                    for (int u = 0; u < 8; ++u) {
                        bar_sync(1, nct);                        // every row's pixel of the step before is published
                        step(8 * t + u, (u & 1) != 0, halo_tag);
                    }
                } else {
                    for (int u = 0; u < 8; ++u) bar_sync(1, nct);
                }
            }
        };
        if (p.halo > 0) walk(std::true_type{}); else walk(std::false_type{});
        __syncwarp();
        if (lane == 0) mbar_arrive(done_bar + (T_compute & 1));
    } else {
        // at time t (interval t of the compute warps): store what interval t-1 finished, bring chunk t+2, which interval t+1 waits for
        if (!p.rot && p.logdet_out != nullptr && blockIdx.x == 0 && warp == p.ncw) warp_logdet(p.w, p.logdet_out, C, HW, K, lane);
        if (!p.bf16) {
            copy(0);
            copy(1);
            cp_async_mbar_arrive(ready_bar);
#pragma unroll 1
            for (int t = 0; t <= T_end; ++t) {
                if (t > 0 && t <= T_compute) mbar_wait_or_give_up(done_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (t > 0) store(t - 1);
                if (p.mix_out != nullptr) bar_sync(2, nio);      // the mix reads every channel of a pixel before any is overwritten
                if (t + 1 < T_compute) {
                    copy(t + 2);
                    cp_async_mbar_arrive(ready_bar + ((t + 1) & 1));
                }
            }
        } else {
            unsigned pre[4 * BV];
#pragma unroll 1
            for (int t = -3; t <= T_end; ++t) {
                if (t > 0 && t <= T_compute) mbar_wait_or_give_up(done_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (t > 0) store(t - 1);
                if (t + 1 < T_compute) {
                    if (t >= -2) place(pre, t + 2);
                    if (t >= -1) mbar_arrive(ready_bar + ((t + 1) & 1));
                    request(pre);
                }
            }
        }
    }
    __syncthreads();
    if (tid == 0 && *gave_up) raise_status(INVCONV_TIMEOUT);
}

}  // namespace invconv
