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
// Reading and writing global memory is the job of separate I/O warps: a ring of 64 columns per row and channel takes the
// right-hand side in chunks of eight columns (16-byte asynchronous copies) two chunks ahead of the wavefront; the solution
// overwrites it in place and leaves one chunk behind.  Images taller than a CTA's rows are walked in bands from top to bottom; the K-1 rows above
// a band are "halo" rows whose threads publish the values that the band before wrote to global memory.  Images and bands
// follow one another on one virtual column axis with zero columns between them, so a CTA with several images pays the ramp
// of the wavefront once.
//
// Large images with few of them in a batch are walked by a cluster instead, a band per CTA, all bands at the same time: the band
// below starts as soon as the bottom rows above have reached global memory (a counter in its shared memory tells; 24
// columns and the band's height behind).
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
constexpr int kRing = 64, kChan = kRing + 4;      // columns of a row and channel in the ring, and floats between channels

// The NB input channels of a slice as NV operands: packed pairs for even NB.
template <int NB, bool PACK = (NB % 2 == 0)>
struct Vec {
    static constexpr int NV = NB;
    using T = float;
    static __device__ __forceinline__ T fma(T a, T b, T c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ float sum(T a) { return a; }
    static __device__ __forceinline__ T zero() { return 0.f; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ T pick(const float (&f)[NB], int q) { return f[q]; }
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
    static __device__ __forceinline__ T pick(const float (&f)[NB], int q) { return pair(f[2 * q], f[2 * q + 1]); }
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

// Add to a counter in a cluster peer's shared memory (after a fence by this thread).
__device__ __forceinline__ void red_add_cluster(uint32_t remote, unsigned v)
{
    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(remote), "r"(v) : "memory");
}
// Bounded wait until a counter of this CTA, raised by a cluster peer, reaches `need`; one thread polls, one fence follows (an
// acquiring poll would pay for it every time).
__device__ __forceinline__ void wait_count(unsigned* count, unsigned need, volatile int* gave_up)
{
    const long long t0 = clock64();
    for (;;) {
        unsigned v;
        asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(count)) : "memory");
        if (v >= need || *gave_up) break;
        if (clock64() - t0 > (1ll << 24)) { *gave_up = 1; break; }
    }
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
}

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
    constexpr bool AL16 = S == 1 || NB % 4 == 0;
    constexpr int UNR = 2;    // steps per turn of the loop
    extern __shared__ __align__(128) float sm[];
    __shared__ unsigned long long bars[6];             // chunk ready [2], chunk done [2], chunk read for storing [2]
    __shared__ int gave_up_flag;
    __shared__ unsigned above;                         // cluster: store rounds of the band above, summed over its storing warps
    volatile int* gave_up = &gave_up_flag;
    // cluster: its CTAs are the bands of one image, all walked at the same time
    const int crank = p.cluster > 1 ? (int)(blockIdx.x % (unsigned)p.cluster) : 0;
    const int cid = p.cluster > 1 ? (int)(blockIdx.x / (unsigned)p.cluster) : (int)blockIdx.x;
    const int ncl = p.cluster > 1 ? (int)(gridDim.x / (unsigned)p.cluster) : (int)gridDim.x;
    const int C = p.C, H = p.H, W = p.W, HW = H * W;
    const int HBt = p.HB + p.halo;
    const int exrow = (HBt + KM + PR) * CS;
    float* EX = sm;                                    // [2][HBt + K-1 + PR][CS]: newest pixel of every row, by step
    float* EY = sm + p.off_y;                          // [2][HBt + PR][CS]: right-hand side of the next pixel of every row, by step parity
    float* RG = sm + p.off_ring;                       // [HBt][C][64 columns]
    const int rm = p.rot ? kRing - 1 : 0;              // slot of virtual column vc: (vc ^ rm) & 63, which is memory order either way
    const int yrow = (HBt + PR) * CS, RS = C * kChan;
    float* As = sm + p.off_a;
    unsigned long long* ready_bar = bars;
    unsigned long long* done_bar = bars + 2;
    unsigned long long* read_bar = bars + 4;
    float* const dummy = sm + p.off_dummy;             // scratch words for lanes without a pixel
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int NT = blockDim.x, nct = p.ncw * 32;
    const int nimg = (p.B - cid + ncl - 1) / ncl;      // images cid, cid + ncl, ...
    const int nseg = nimg * p.nbands;
    // virtual columns; in a cluster the first image starts late enough for the halo rows, which run ahead, to pass their first columns
    const int lead = p.cluster > 1 ? (K > 9 ? 16 : 8) : 0;
    const int VC = lead + (nseg - 1) * p.SW + W;
    const int T_compute = (VC + p.HB - 1 + 7) >> 3;    // intervals of eight steps
    const int T_end = ((VC - 1) >> 3) + 1 + ((p.HB - 1 + 7) >> 3);

    if (tid == 0) {
        mbar_init(ready_bar, p.niow * 32); mbar_init(ready_bar + 1, p.niow * 32);
        mbar_init(done_bar, p.ncw); mbar_init(done_bar + 1, p.ncw);
        mbar_init(read_bar, p.niow); mbar_init(read_bar + 1, p.niow);
        gave_up_flag = 0;
        above = 0u;
        fence_mbar_init();
    }
    for (int i = tid; i < 2 * exrow; i += NT) EX[i] = 0.f;
    for (int i = tid; i < 2 * yrow; i += NT) EY[i] = 0.f;          // channels beyond C meet zero weights but must not be NaN
    for (int i = p.off_a + tid; i < p.off_w; i += NT) sm[i] = 0.f;     // As and li
    __syncthreads();
    if (p.cluster > 1) {                               // the counters exist before the band above adds to them
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    // everything above touched no global memory; from here on the predecessor kernel's results are needed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---------------------------------------------------------------- I/O
    // Half of the I/O warps load, half store (together their loop outgrew the instruction cache: 2500 cycles a chunk against 1000
    // and 1300 apart).  A piece is four columns of one (row, channel), half a chunk; a thread owns the same BV pieces of
    // every chunk.  Row r is floor(r/8) chunks behind row 0 when read, ceil(r/8) when stored.
    constexpr int BV = kLinePieces;                    // at most; p.pieces of them are used
    const bool io_warp = warp >= p.ncw, loader = warp < p.ncw + p.niow;
    const int nio = p.niow * 32, io = tid - nct - (loader ? 0 : nio);
    const int half4 = 4 * (io & 1), sgn = p.rot ? -1 : 1;
    int ring_off[BV], gofs[BV], row[BV];
    // per piece, of the chunk moved next: column within its segment, segment, and the element of the segment row's first column
    // (-1: no such row)
    int pcol[BV], pseg[BV], pbase[BV];
    auto behind = [&](int r) { return r >= -8 && r < 0 ? 0 : r >> 3; };      // chunks behind row 0 when read (halo rows: d columns ahead)
    auto seg_base = [&](int b, int seg) -> int {
        if (seg >= nseg) return -1;
        const int i = p.nbands == 1 ? seg : fast_div(seg, p.div_nb), band = seg - i * p.nbands;
        const int h = (band + crank) * p.HB + row[b];
        if (h < 0 || h >= H) return -1;
        return (cid + i * ncl) * C * HW + gofs[b] + sgn * (band + crank) * p.HB * W;
    };
    if (io_warp) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            const int rc = (io + b * nio) >> 1, rr = fast_div(rc, p.div_c), c = rc - rr * C, r = rr - p.halo;
            const bool ok = rr < HBt;
            row[b] = ok ? r : -1000000;                // never inside the image
            ring_off[b] = ok ? rr * RS + c * kChan : 0;
            gofs[b] = ok ? c * HW + (p.rot ? HW - 1 - r * W : r * W) : 0;
            pcol[b] = half4 - lead - (ok ? 8 * (loader ? behind(r) : (r + 7) >> 3) : 0);
            pseg[b] = 0;
            pbase[b] = r < 0 && !loader ? -1 : seg_base(b, 0);
        }
    }
    auto advance = [&](int b, int& col, int& seg, int& base) {
        col += 8;
        if (nseg > 1)
            while (col >= p.SW) { col -= p.SW; ++seg; base = seg_base(b, seg); }
    };
    const int safe = cid * C * HW;         // an element every load may touch
    // fp32: asynchronous copies straight into the ring (chunk t), zeros outside the image
    auto copy = [&](int t) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            if (b >= p.pieces) break;                  // uniform
            const bool have = pbase[b] >= 0 && pcol[b] >= 0;
            const int vc = 8 * (t - behind(row[b])) + half4, left = have ? W - pcol[b] : 0;
            const float* g = reinterpret_cast<const float*>(row[b] < 0 ? p.out : p.rhs) + (left > 0 ? pbase[b] + sgn * pcol[b] : safe);
            float* d = RG + ring_off[b];
            if (row[b] > -1000) {
                if (p.vec) {
                    cp_async_f32x4(d + (((vc ^ rm) & (kRing - 1)) & ~3), left > 0 && p.rot ? g - 3 : g, left > 0);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) cp_async_f32(d + (((vc + j) ^ rm) & (kRing - 1)), j < left ? g + sgn * j : g, j < left);
                }
            }
            advance(b, pcol[b], pseg[b], pbase[b]);
        }
    };
    // bf16: requested into registers a chunk ahead, widened when placed
    int rnv[BV];                                       // columns inside the image of the pieces requested last
    auto request = [&](unsigned (&v)[4 * BV]) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            if (b >= p.pieces) break;
            const int nv = pbase[b] >= 0 && pcol[b] >= 0 ? min(max(W - pcol[b], 0), 4) : 0;
            const int f = pbase[b] + sgn * pcol[b];
            rnv[b] = nv;
            const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(row[b] < 0 ? p.out : p.rhs);
            if (p.vec) {
                const uint2 u = *reinterpret_cast<const uint2*>(src + (nv > 0 ? (p.rot ? f - 3 : f) : safe));
                v[4 * b] = u.x; v[4 * b + 1] = u.y;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) v[4 * b + j] = reinterpret_cast<const unsigned short*>(src)[j < nv ? f + sgn * j : safe];
            }
            advance(b, pcol[b], pseg[b], pbase[b]);
        }
    };
    auto place = [&](const unsigned (&v)[4 * BV], int t) {
#pragma unroll
        for (int b = 0; b < BV; ++b) {
            if (b >= p.pieces) break;
            const int vc = 8 * (t - behind(row[b])) + half4;
            unsigned u[4];
            if (row[b] <= -1000) continue;
            float* d = RG + ring_off[b];
            if (p.vec) {                                 // memory order is slot order
                u[3] = v[4 * b + 1] & 0xffff0000u; u[2] = v[4 * b + 1] << 16; u[1] = v[4 * b] & 0xffff0000u; u[0] = v[4 * b] << 16;
                if (rnv[b] == 0) u[0] = u[1] = u[2] = u[3] = 0u;
                *reinterpret_cast<uint4*>(d + (((vc ^ rm) & (kRing - 1)) & ~3)) = make_uint4(u[0], u[1], u[2], u[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    d[((vc + j) ^ rm) & (kRing - 1)] = j < rnv[b] ? __uint_as_float(v[4 * b + j] << 16) : 0.f;
            }
        }
    };
    auto hand_back = [&](int t) {                      // the finished chunk has been read
        __syncwarp();
        if (lane == 0) mbar_arrive(read_bar + (t & 1));
    };
    auto store = [&](int t) {                          // at time t: what interval t-1 finished
#pragma unroll
        for (int b0 = 0; b0 < BV; b0 += 4) {
        if (b0 >= p.pieces) break;
        float4 f[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int vc = 8 * (t - 1 - ((row[b0 + q] + 7) >> 3)) + half4;
            f[q] = *reinterpret_cast<const float4*>(RG + ring_off[b0 + q] + (((vc ^ rm) & (kRing - 1)) & ~3));      // memory order
        }
        if (b0 + 4 >= p.pieces) hand_back(t);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int b = b0 + q;
            const int nv = pbase[b] >= 0 && pcol[b] >= 0 ? min(max(W - pcol[b], 0), 4) : 0;
            const int i = pbase[b] + sgn * pcol[b];
            advance(b, pcol[b], pseg[b], pbase[b]);
            if (row[b] < 0) pbase[b] = -1;             // halo rows are not stored
            if (nv == 0) continue;
            if (p.vec) {
                const int lo = p.rot ? i - 3 : i;
                if (p.bf16) {
                    const __nv_bfloat162 a = __floats2bfloat162_rn(f[q].x, f[q].y), c = __floats2bfloat162_rn(f[q].z, f[q].w);
                    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + lo) =
                        make_uint2(*reinterpret_cast<const unsigned*>(&a), *reinterpret_cast<const unsigned*>(&c));
                } else {
                    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + lo) = f[q];
                }
            } else {
                const float e[4] = {f[q].x, f[q].y, f[q].z, f[q].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float v = p.rot ? e[3 - j] : e[j];
                    if (j < nv) {
                        if (p.bf16) reinterpret_cast<__nv_bfloat16*>(p.out)[i + sgn * j] = __float2bfloat16_rn(v);
                        else reinterpret_cast<float*>(p.out)[i + sgn * j] = v;
                    }
                }
            }
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
            const bool have = live && rr0 + i < HBt && (r < 0 ? bnd + crank > 0 : (bnd + crank) * p.HB + r < H);
            return have ? (unsigned)W : 0u;
        };
#pragma unroll
        for (int i = 0; i < PR; ++i) { band[i] = 0; width[i] = row_width(i, 0); }
        // rows of this warp: the warp works in an interval while any of them is between K-1 columns before its first and its last
        const int g_lo = fast_div((warp * 32) / S, p.div_c), g_hi = fast_div((warp * 32 + 31) / S, p.div_c);
        const int t_lo = max(0, (g_lo * PR - p.halo - (KM > 2 ? KM : 2)) >> 3), t_hi = (VC + min(g_hi * PR + PR - 1, HBt - 1) - p.halo + 7) >> 3;
        // column within the segment of each row's pixel in the warp's first step; negative before its first column
        int col[PR];
#pragma unroll
        for (int i = 0; i < PR; ++i) col[i] = 8 * t_lo - lead - (rr0 + i - p.halo);
        bool pub[PR];                                  // this lane publishes the row's pixel
#pragma unroll
        for (int i = 0; i < PR; ++i) pub[i] = live && sl == 0 && rr0 + i < HBt;
        float* const ex_rd = EX + (rr0 + KM) * CS + sl * NB;
        float* const ex_wr = EX + (rr0 + KM) * CS + a;
        float* const ring0 = RG + rr0 * RS + a * kChan;
        float* const ey_rd = EY + rr0 * CS + sl * NB;
        float* const ey_wr = EY + rr0 * CS + a;
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
                V::template load<AL16>(ey_rd + (odd ? 0 : yrow) + i * CS, rh[i]);
            float y2[PR];                              // own channel's right-hand side two columns ahead, published for the next step
#pragma unroll
            for (int i = 0; i < PR; ++i) y2[i] = ring0[i * RS + (((s - (rr0 + i - p.halo) + 2) ^ rm) & (kRing - 1))];
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
                float* rg = ring0 + i * RS + (((s - (rr0 + i - p.halo)) ^ rm) & (kRing - 1));
                const bool inside = (unsigned)col[i] < width[i];
                if constexpr (HALO) {                            // halo row: the value the band above left
                    const float h = *rg;
                    x = rr0 + i < p.halo ? h : x;
                }
                x = inside ? x : 0.f;
                *(pub[i] ? ex_wr + wr + i * CS : dummy) = x;
                *(pub[i] ? ey_wr + (odd ? yrow : 0) + i * CS : dummy) = y2[i];
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
                if (t == 0) {
                    // what step -1 would have left: the first row's first right-hand side in its pending sum, every row's next one
                    // in the exchange buffer that step 0 reads
#pragma unroll
                    for (int i = 0; i < PR; ++i) {
                        if (pub[i]) ey_wr[yrow + i * CS] = ring0[i * RS + (((1 - (rr0 + i - p.halo)) ^ rm) & (kRing - 1))];
                        if (live && rr0 + i == p.halo) {
                            float f[NB];
#pragma unroll
                            for (int q = 0; q < NB; ++q) f[q] = sl * NB + q < C ? RG[(rr0 + i) * RS + (sl * NB + q) * kChan + rm] : 0.f;
#pragma unroll
                            for (int q = 0; q < NV; ++q) acc[i][0] = V::fma(W0[q], V::pick(f, q), acc[i][0]);
                        }
                    }
                }
                if (t >= t_lo && t < t_hi) {                     // warp-uniform
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
        // At time t (interval t of the compute warps) the storing warps store what interval t-1 finished, the loading warps bring chunk
        // t+2, which interval t+1 waits for; they hand it over only when the finished chunk has been read, so that neither
        // side falls more than one interval behind.
        if (!loader) {
            if (!p.rot && p.logdet_out != nullptr && blockIdx.x == 0 && warp == p.ncw + p.niow) warp_logdet(p.w, p.logdet_out, C, HW, K, lane);
            // Tells the band below that a round of stores has reached global memory (its halo rows come from there) -- one round later,
            // when the fence no longer has to wait for them.
            auto tell = [&](uint32_t counter) {
                __threadfence();
                __syncwarp();
                if (lane == 0) red_add_cluster(counter, 1u);
            };
            const uint32_t below = crank + 1 < p.cluster ? cluster_map_u32(smem_u32(&above), (uint32_t)(crank + 1)) : 0u;
#pragma unroll 1
            for (int t = 1; t <= T_end; ++t) {
                if (t <= T_compute) mbar_wait_or_give_up(done_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (crank + 1 < p.cluster && t > 1) tell(below);
                store(t);
            }
            if (crank + 1 < p.cluster) tell(below);
        } else if (!p.bf16) {
#pragma unroll 1
            for (int t = -2; t + 1 < T_compute; ++t) {
                if (t > 0) mbar_wait_or_give_up(done_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (crank > 0) {                       // chunk t+2 of the bottom rows above has been stored
                    const unsigned need = (unsigned)(p.niow * min(T_end, t + 3 + ((p.HB - 1 + 7) >> 3)));
                    if (lane == 0) wait_count(&above, need, gave_up);
                    __syncwarp();
                }
                copy(t + 2);
                if (t > 0) mbar_wait_or_give_up(read_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (t >= -1) cp_async_mbar_arrive(ready_bar + ((t + 1) & 1));
            }
        } else {
            unsigned pre[4 * BV];
#pragma unroll 1
            for (int t = -3; t + 1 < T_compute; ++t) {
                if (t > 0) mbar_wait_or_give_up(done_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (t >= -2) place(pre, t + 2);
                if (t > 0) mbar_wait_or_give_up(read_bar + (t & 1), ((t - 1) >> 1) & 1, gave_up);
                if (t >= -1) mbar_arrive(ready_bar + ((t + 1) & 1));
                request(pre);
            }
        }
    }
    __syncthreads();
    if (p.cluster > 1) {                               // no CTA leaves while the band above may still add to its counter
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (tid == 0 && *gave_up) raise_status(INVCONV_TIMEOUT);
}

}  // namespace invconv
