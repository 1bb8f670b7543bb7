// Wide-channel wavefront: one CTA -- or one thread-block cluster -- per image.
//
// With many channels the per-diagonal update is a contraction
//     u[p][a] = sum_b A0[a][b] rhs[p][b] - sum_{delta != 0, b} A_delta[a][b] u[p - delta][b]
// of length C*k^2 for each of (pixels on the diagonal) x C outputs, and the fp32
// FMA pipe is the bound (Section 3.3: k^2 work per diagonal, here times C^2).
// The transformed kernel A (see team_solve_kernel) is the stationary operand: it
// is distributed once over the REGISTERS of the CTA -- thread (slice s, lane l)
// keeps the entries for its share of the contraction range (a few groups of
// four input channels of one tap) and its TA output channels -- and stays
// there for every image the CTA processes.  Solved pixels live in shared
// memory as [pixel][channel], so the four input channels of a group arrive
// as one broadcast 16-byte load feeding 4*TA FMAs.
//
// When C*C*k^2 floats outgrow one SM's register file the output channels are
// split over the CTAs of a cluster: each CTA finishes its C/R channels of the
// diagonal's pixels and stores them into every peer's shared-memory image
// (distributed shared memory), then one cluster barrier closes the step.
// Every CTA therefore always reads only its own shared memory.
//
// The transposed solve (grad_y = M^-T grad_x, Theorem 1) runs the same kernel:
// the image is rotated by 180 degrees while it is loaded and stored, and
// team_solve_kernel supplies L^-T W_delta^T.
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "common.cuh"
#include "tma.cuh"

namespace invconv {
namespace cg = cooperative_groups;

// ---------------------------------------------------------------------------
// Transformed kernel  A[tap][b][a], tap = dh*K + dw,
//   forward : tap 0 -> L^-1[a][b];   tap != 0 -> sum_m L^-1[a][m] w[m][b][K-1-dh][K-1-dw]
//   backward: tap 0 -> L^-1[b][a];   tap != 0 -> sum_m L^-1[m][a] w[b][m][K-1-dh][K-1-dw]
// L = w[:, :, K-1, K-1] restricted to ci <= co.
// One CTA per input channel b (plus CTAs for tap 0) solves  T S = RHS  by substitution,
// T = L (forward, rows ascending) or L^T (backward, rows descending):
//   b <  C : RHS[m][kk] = w[m][b][kk] (forward) / w[b][m][kk] (backward); S[a][kk] -> A[flip(kk)][b][a]
//   b >= C : RHS = 32 columns of the identity;                            S[a][b'] -> A[0][b'][a]
// The columns of RHS are independent, so each warp takes two of them and runs the whole substitution inside
// the warp: lane l holds the residuals of the rows at positions l, l+32, ... (NS of them) of its two columns in
// registers; step j broadcasts y_j = r_j / T_jj from the lane that owns row j by one shuffle and every lane
// subtracts T_ij y_j from its rows, T read column by column from shared memory (stored transposed, Tt[j][i],
// zero on and above the diagonal, so no lane needs a predicate and row j keeps its final residual).  A step is
// one multiply, one shuffle and one multiply-add on the dependent chain and there is no block barrier inside
// the substitution (the earlier blocked scheme with a barrier per eight rows took 1.8 k cycles per eight rows
// at C = 48; this one takes about 35 cycles per row).
// ---------------------------------------------------------------------------
inline int team_solve_ns(int C) { return (C + 31) / 32; }
inline size_t team_solve_smem(int C, int K)
{
    const size_t nc = K * K > 32 ? K * K : 32;
    return sizeof(float) * ((size_t)C * (32 * team_solve_ns(C) + 1) + ((C + 3) & ~3) + (size_t)C * nc + (size_t)C * (nc | 1));
}

// Value v of input channel j (of a chunk's eight) and operand row `row` in the operand form of the tensor-core kernels:
// planes of 16-byte rows, two-term (tf32 hi in planes 0, 1; bf16 remainder; bf16 value) or three-term (bf16 terms w0, w1, w0, w2).
__device__ __forceinline__ void pack_operand(unsigned char* blk, int rows, int row, int j, float v, bool three)
{
    if (three) {
        const __nv_bfloat16 a = __float2bfloat16_rn(v);
        const float r = v - __bfloat162float(a);
        const __nv_bfloat16 b = __float2bfloat16_rn(r);
        *reinterpret_cast<__nv_bfloat16*>(blk + (size_t)row * 16 + j * 2) = a;
        *reinterpret_cast<__nv_bfloat16*>(blk + ((size_t)rows + row) * 16 + j * 2) = b;
        *reinterpret_cast<__nv_bfloat16*>(blk + ((size_t)2 * rows + row) * 16 + j * 2) = a;
        *reinterpret_cast<__nv_bfloat16*>(blk + ((size_t)3 * rows + row) * 16 + j * 2) = __float2bfloat16_rn(r - __bfloat162float(b));
    } else {
        const float hi = tf32_hi(v);
        *reinterpret_cast<float*>(blk + ((size_t)(j >> 2) * rows + row) * 16 + (j & 3) * 4) = hi;
        *reinterpret_cast<__nv_bfloat16*>(blk + ((size_t)2 * rows + row) * 16 + j * 2) = __float2bfloat16_rn(v - hi);
        *reinterpret_cast<__nv_bfloat16*>(blk + ((size_t)3 * rows + row) * 16 + j * 2) = __float2bfloat16_rn(v);
    }
}

template <bool BWD, int NS>
__global__ void __launch_bounds__(512) team_solve_kernel(const float* __restrict__ w, float* __restrict__ A, int C, int K,
                                                         unsigned char* __restrict__ wop, int NCH, unsigned wbytes, int CP_, int three,
                                                         float* __restrict__ logdet_out, int HW)
{
    extern __shared__ __align__(128) float sm[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the wavefront kernel may set itself up meanwhile
    if (logdet_out != nullptr && blockIdx.x == gridDim.x - 1 && threadIdx.x >= 480)
        warp_logdet(w, logdet_out, C, HW, K, threadIdx.x & 31);        // the layer's log-det, by a warp of the lightest CTA
    constexpr int C32 = 32 * NS, CP = C32 + 1;
    const int KK = K * K, ctr = KK - 1;
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = NT >> 5;
    const int b = blockIdx.x;
    // CTAs C .. CP_-1 (operand form only): channels that pad the operand, zeros; CTAs CP_, CP_+1, ...: 32-column chunks of the
    // identity (tap 0)
    const bool ident = b >= CP_;
    const int c0 = ident ? (b - CP_) * 32 : 0;  // first identity column of this CTA
    const int NC = ident ? min(32, C - c0) : KK;   // right-hand-side columns
    const int NCB = KK > 32 ? KK : 32, YS = NCB | 1;
    float* Tt = sm;                           // [C][CP]   Tt[pa*CP + pi] = T[row at position pi][row at position pa], pi > pa
    float* invd = Tt + C * CP;                // [C]       1 / T[p][p], by position
    float* RHS = invd + ((C + 3) & ~3);       // [C][NC]   by row index
    float* Y = RHS + C * NCB;                 // [C][YS]   solved rows, by row index
    if (!ident && b >= C) {
        const int chunk = b >> 3, j = b & 7, rk = chunk / NCH, cl = chunk - rk * NCH, KCP = K * CP_;
        for (int e = tid; e < K * KCP; e += NT) {
            const int dh = e / KCP, row = e - dh * KCP;
            pack_operand(wop + (size_t)rk * wbytes + (size_t)((dh * NCH + cl) * 4) * KCP * 16, KCP, row, j, 0.f, three != 0);
        }
        return;
    }
    auto idx = [&](int pos) { return BWD ? C - 1 - pos : pos; };              // position in solve order -> row index

    // every global load of the CTA is issued before the first shared-memory store that waits for one
    const unsigned mKK = 0xFFFFFFFFu / (unsigned)KK + 1u;                      // e / KK = umulhi(e, mKK) for e < 2^16
    float rv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int e = tid + q * NT;
        rv[q] = 0.f;
        if (!ident && e < C * KK) {
            const int m = KK == 1 ? e : (int)__umulhi((unsigned)e, mKK), kk = e - m * KK;
            rv[q] = BWD ? __ldg(w + (size_t)b * C * KK + e) : __ldg(w + ((size_t)m * C + b) * KK + kk);
        }
    }
    for (int e0 = tid; e0 < C * C32 || e0 == tid; e0 += NT * 8) {            // at least one trip: it also stores rv
        float tv[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * NT, pa = e / C32, pi = e - pa * C32;
            tv[q] = 0.f;
            if (e < C * C32 && pi < C && pi >= pa) {
                const int row = BWD ? idx(pa) : pi, col = BWD ? idx(pi) : pa;   // T[pi][pa] = L[pi][pa] or L^T: L[idx(pa)][idx(pi)]
                tv[q] = __ldg(w + ((size_t)row * C + col) * KK + ctr);
            }
        }
        if (e0 == tid) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (!ident && tid + q * NT < C * KK) RHS[tid + q * NT] = rv[q];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * NT, pa = e / C32, pi = e - pa * C32;
            if (e < C * C32) {
                Tt[pa * CP + pi] = pi == pa ? 0.f : tv[q];
                if (pi == pa) invd[pa] = 1.0f / tv[q];
            }
        }
    }
    if (!ident)
        for (int e = tid + 8 * NT; e < C * KK; e += NT) {                      // kernels beyond 4096 right-hand-side values
            const int m = e / KK, kk = e - m * KK;
            RHS[e] = BWD ? __ldg(w + (size_t)b * C * KK + e) : __ldg(w + ((size_t)m * C + b) * KK + kk);
        }
    __syncthreads();

    for (int cb = 2 * warp; cb < NC; cb += 2 * nwarps) {
        float r[NS][2];
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                const int p = lane + 32 * s, c = cb + col;
                float v = 0.f;
                if (p < C && c < NC) v = ident ? (idx(p) == c0 + c ? 1.f : 0.f) : RHS[idx(p) * NC + c];
                r[s][col] = v;
            }
#pragma unroll
        for (int sj = 0; sj < NS; ++sj) {
            const int jend = min(32, C - 32 * sj);
#pragma unroll 4
            for (int jj = 0; jj < jend; ++jj) {
                const int j = 32 * sj + jj;
                float t[NS];
#pragma unroll
                for (int s = sj; s < NS; ++s) t[s] = Tt[j * CP + lane + 32 * s];
                const float dj = invd[j];
#pragma unroll
                for (int col = 0; col < 2; ++col) {
                    const float yj = __shfl_sync(0xffffffffu, r[sj][col] * dj, jj);
#pragma unroll
                    for (int s = sj; s < NS; ++s) r[s][col] = fmaf(-t[s], yj, r[s][col]);
                }
            }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                const int p = lane + 32 * s, c = cb + col;
                if (p < C && c < NC) Y[idx(p) * YS + c] = r[s][col] * invd[p];
            }
    }
    __syncthreads();

    if (wop == nullptr) {
        for (int col = warp; col < NC; col += nwarps) {
            if (!ident && col == ctr) continue;
            float* dst = ident ? A + (size_t)(c0 + col) * C : A + ((size_t)(KK - 1 - col) * C + b) * C;   // A[tap][b][.]
            for (int a = lane; a < C; a += 32) dst[a] = Y[a * YS + col];
        }
        return;
    }
    // Tensor-core operand form instead (see tensor_kernels.cuh): per CTA rank r = chunk / NCH one block
    //   [dh][chunk % NCH][plane 0,1: tf32 hi | plane 2: bf16 remainder | plane 3: bf16 value][row = dw*C + a][16 bytes],
    // chunk = input channel / 8; the sign is flipped for every tap but tap 0.
    const int KC = K * CP_;
    for (int col = warp; col < NC; col += nwarps) {
        if (!ident && col == ctr) continue;
        const int tap = ident ? 0 : KK - 1 - col, ci = ident ? c0 + col : b;
        const int chunk = ci >> 3, j = ci & 7, rk = chunk / NCH, cl = chunk - rk * NCH;
        const int dh = tap / K, dw = tap - dh * K;
        unsigned char* blk = wop + (size_t)rk * wbytes + (size_t)((dh * NCH + cl) * 4) * KC * 16;
        for (int a = lane; a < CP_; a += 32) {
            const float y = a < C ? Y[a * YS + col] : 0.f;
            pack_operand(blk, KC, dw * CP_ + a, j, ident ? y : -y, three != 0);
        }
    }
}

// Launch on `st` (grid: one CTA per input channel plus the identity chunks); cudaSuccess or the launch's error.
inline cudaError_t team_solve_launch(bool bwd, const float* w, float* A, int C, int K, unsigned char* wop, int NCH,
                                     unsigned wbytes, int padded, bool three, float* logdet_out, int HW, cudaStream_t st)
{
    using Kern = void (*)(const float*, float*, int, int, unsigned char*, int, unsigned, int, int, float*, int);
    Kern kern = nullptr;
    switch (team_solve_ns(C) * 2 + (bwd ? 1 : 0)) {
    case 2: kern = team_solve_kernel<false, 1>; break;
    case 3: kern = team_solve_kernel<true, 1>; break;
    case 4: kern = team_solve_kernel<false, 2>; break;
    case 5: kern = team_solve_kernel<true, 2>; break;
    case 6: kern = team_solve_kernel<false, 3>; break;
    case 7: kern = team_solve_kernel<true, 3>; break;
    case 8: kern = team_solve_kernel<false, 4>; break;
    case 9: kern = team_solve_kernel<true, 4>; break;
    default: return cudaErrorInvalidValue;
    }
    const size_t sm = team_solve_smem(C, K);
    if (sm > 40 * 1024) {      // static shared memory counts towards the 48 KB available without opting in
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    kern<<<padded + (C + 31) / 32, 512, sm, st>>>(w, A, C, K, wop, NCH, wbytes, padded, three ? 1 : 0, logdet_out, HW);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
struct TeamParams {
    const float* rhs;   // y (forward) or grad_x (backward), [B][C][H][W]
    const float* A;     // transformed kernel [K*K][C(b)][C(a)]
    float* out;         // x or grad_y
    int B, C, H, W, K;
    int R;              // CTAs per image (cluster size)
    int CA;             // output channels per CTA (C / R)
    int LG;             // lanes per slice (power of two), LG*TA >= CA
    int NS;             // slices per pixel group (multiple of 32/LG)
    int NPG;            // pixel groups per CTA (pixel-team variant: teams per CTA)
    int KW;             // pixel-team variant: warps per team
    int CS;             // floats per pixel in the shared-memory images: C rounded up to 4, padded to 4 mod 8
                        // so that pixel-major accesses spread over the banks
    int rot;            // 1: walk the image rotated by 180 degrees (transposed solve)
    int vec;            // 1: images are 16-byte aligned and H*W is a multiple of 4
    FastDiv div_w, div_hw, div_q4;   // divisions by W, H*W and H*W/4
    int ncl;            // clusters in the grid
};


__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Fold SPW pixel slots x TA channels across the SPW slices of a warp (slices are LG lanes apart) by halving:
// after log2(SPW) levels the lanes of slice sw hold the warp-wide sums of pixel slot sw in v[0..TA).  This
// takes (SPW-1)*TA shuffles where folding every value separately takes SPW*TA*log2(SPW).
template <int SPW, int TA>
__device__ __forceinline__ void transposed_fold(float (&v)[SPW * TA], int sw, int LG)
{
#pragma unroll
    for (int hs = SPW / 2; hs >= 1; hs >>= 1) {
        const bool hi = (sw & hs) != 0;
#pragma unroll
        for (int q = 0; q < hs * TA; ++q) {
            const float send = hi ? v[q] : v[q + hs * TA];
            const float keep = hi ? v[q + hs * TA] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, hs * LG);
        }
    }
}

// Thread (pixel group pg, slice s, lane l) owns a few groups of four input
// channels of one tap each and TA output channels, split into the groups whose
// tap reads the previous diagonal (taps (0,1) and (1,0): the only ones on the
// dependent chain) and all the others, which read diagonals solved at least two
// steps ago.  Per diagonal it first runs the second kind for its pixels -- this
// overlaps the arrival of the previous diagonal -- then waits for that diagonal,
// runs the first kind, folds the slices that share its warp by shuffles and
// leaves one partial sum per warp in shared memory.  After one block barrier
// every (pixel, channel) of the diagonal is summed over the warps and published:
// a plain store into this CTA's image and an asynchronous store (st.async) into
// the image of every other CTA of the cluster.  Each CTA owns two mbarriers
// (even / odd diagonals): all of its threads arrive after publishing and its
// peers' asynchronous stores are counted in bytes, so one wait covers both.
template <int TA, int NGN, int NGC, int PM, int MAXT>
__global__ void __launch_bounds__(MAXT) team_wavefront_kernel(TeamParams p)
{
    extern __shared__ __align__(128) float smem[];
    __shared__ unsigned long long bars[2];
    __shared__ int gave_up_flag;                   // a bounded wait of this CTA ran out: later waits no longer block
    const int C = p.C, H = p.H, W = p.W, K = p.K, CS = p.CS, R = p.R, CA = p.CA;
    const int HP = H + K - 1, WP = W + K - 1, HW = H * W;
    const int IMG = HP * WP * CS;
    float* U = smem;
    float* RH = smem + IMG;
    float* red = smem + 2 * IMG;
    const int cl = blockIdx.x / R;
    const int r = blockIdx.x - cl * R;              // rank in the cluster (1-D clusters of R consecutive CTAs)
    const int tid = threadIdx.x, NT = blockDim.x;
    const int LG = p.LG, NS = p.NS, per_pg = NS * LG, NPG = p.NPG;
    const int pg = tid / per_pg, tq = tid - pg * per_pg;
    const int s = tq / LG, l = tq - s * LG;
    const int wq = tq >> 5, NWP = per_pg >> 5;
    const int CAp = LG * TA;
    const int CB4 = (C + 3) >> 2;
    const int GN = (K > 1 ? K * K - 2 : 1) * CB4, GC = (K > 1 ? 2 : 0) * CB4;
    const int DS = (WP - 1) * CS;                   // from one pixel of a diagonal to the next (one row down, one column left)
    const bool tfold = (LG == 4 || LG == 8 || LG == 16) && (PM % (32 / LG) == 0);   // transposed fold applies

    // Set-up that needs no global memory runs first, so that under programmatic dependent launch it overlaps
    // the kernel-transform kernel that precedes this one on the stream; griddepcontrol.wait then waits for it.
    if (tid == 0) { gave_up_flag = 0; mbar_init(&bars[0], NT >> 5); mbar_init(&bars[1], NT >> 5); fence_mbar_init(); }   // one arrival per warp
    for (int i = tid; i < 2 * IMG; i += NT) smem[i] = 0.f;     // zero padding (and the channel padding) once
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // this thread's share of the transformed kernel, signs folded in
    float wn[NGN][4][TA], wc[NGC][4][TA];
    int offn[NGN], offc[NGC];
    auto fetch = [&](bool live, int tap, int b4, float (&dst)[4][TA], int& off) {
        const int dh = tap / K, dw = tap - dh * K;
        off = live ? (tap == 0 ? IMG : 0) - (dh * WP + dw) * CS + b4 * 4 : 0;
#pragma unroll
        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
            for (int t = 0; t < TA; ++t) {
                const int b = b4 * 4 + bb, al = l * TA + t;
                float v = 0.f;
                if (live && b < C && al < CA) v = __ldg(p.A + ((size_t)tap * C + b) * C + r * CA + al);
                dst[bb][t] = tap == 0 ? v : -v;
            }
    };
#pragma unroll
    for (int i = 0; i < NGN; ++i) {
        const int g = s + i * NS;
        const int tnc = g / CB4, b4 = g - tnc * CB4;
        const int tap = tnc == 0 ? 0 : (tnc <= K - 2 ? tnc + 1 : tnc + 2);   // skips taps 1 and K
        fetch(g < GN, g < GN ? tap : 0, b4, wn[i], offn[i]);
    }
#pragma unroll
    for (int i = 0; i < NGC; ++i) {
        const int g = s + i * NS;
        const int tcr = g / CB4, b4 = g - tcr * CB4;
        fetch(g < GC, g < GC ? (tcr == 0 ? 1 : K) : 0, b4, wc[i], offc[i]);
    }
    // peers' images and mbarriers (shared::cluster addresses)
    uint32_t peerU[8], peerBar[8];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        const uint32_t rk = (uint32_t)(rr < R ? rr : r);
        peerU[rr] = R > 1 ? cluster_map_u32(smem_u32(U), rk) : 0u;
        peerBar[rr] = R > 1 ? cluster_map_u32(smem_u32(&bars[0]), rk) : 0u;
    }

    __syncthreads();
    if (R > 1) { cluster_arrive_release(); cluster_wait_acquire(); }   // every CTA's barriers exist before anyone sends

    // finalize items of this thread walk (pixel, channel) pairs in steps of NT without divisions
    const int fin_i0 = tid / CA, fin_a0 = tid - fin_i0 * CA;
    const int fin_di = NT / CA, fin_da = NT - fin_di * CA;
    const int CAQ = CA >> 2 > 0 ? CA >> 2 : 1;      // channel quads per pixel (used when CA is a multiple of four)
    const int finq_i0 = tid / CAQ, finq_a0 = tid - finq_i0 * CAQ;
    const int finq_di = NT / CAQ, finq_da = NT - finq_di * CAQ;

    const int ND = H + W - 1;
    const int nq4 = HW >> 2;
    unsigned stepno = 0;                            // diagonals processed so far by this CTA, across images
    volatile int* gave_up = &gave_up_flag;
    for (int n = cl; n < p.B; n += p.ncl) {
        // right-hand side of this image, all channels, rotated for the transposed solve; the loads go out in
        // batches of eight requests per thread so that their latency is paid once per batch
        const float* src = p.rhs + (size_t)n * C * HW;
        if (p.vec) {
            const float4* src4 = reinterpret_cast<const float4*>(src);
            const int nvec = C * nq4;
            for (int v0 = tid; v0 < nvec; v0 += NT * 8) {
                float4 tv[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (v0 + k * NT < nvec) tv[k] = __ldg(src4 + v0 + k * NT);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (v0 + k * NT < nvec) {
                        const int vi = v0 + k * NT;
                        const int c = fast_div(vi, p.div_q4), pp = (vi - c * nq4) << 2;
                        const float vals[4] = {tv[k].x, tv[k].y, tv[k].z, tv[k].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            int h = fast_div(pp + i, p.div_w), w = (pp + i) - h * W;
                            if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                            RH[((h + K - 1) * WP + (w + K - 1)) * CS + c] = vals[i];
                        }
                    }
                }
            }
        } else {
            for (int e0 = tid; e0 < C * HW; e0 += NT * 8) {
                float tv[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (e0 + k * NT < C * HW) tv[k] = __ldg(src + e0 + k * NT);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (e0 + k * NT < C * HW) {
                        const int e = e0 + k * NT;
                        const int c = fast_div(e, p.div_hw), pp = e - c * HW;
                        int h = fast_div(pp, p.div_w), w = pp - h * W;
                        if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                        RH[((h + K - 1) * WP + (w + K - 1)) * CS + c] = tv[k];
                    }
                }
            }
        }
        __syncthreads();

        for (int d = 0; d < ND; ++d, ++stepno) {
            const int hlo = max(0, d - (W - 1));
            const int npix = min(H - 1, d) - hlo + 1;
            // pixel i of the diagonal is (hlo + i, d - hlo - i); this thread's pixels are i = pg, pg + NPG, ...
            const float* ubase = U + ((hlo + K - 1) * WP + (d - hlo) + K - 1) * CS + pg * DS;
            const int qstep = NPG * DS;
            float acc[PM][TA];
#pragma unroll
            for (int q = 0; q < PM; ++q)
#pragma unroll
                for (int t = 0; t < TA; ++t) acc[q][t] = 0.f;
            // taps that read diagonals <= d-2 (and the right-hand side)
#pragma unroll
            for (int q = 0; q < PM; q += 2) {
                const int i0 = pg + NPG * q;
                if (i0 < npix) {
                    const float* u0 = ubase + q * qstep;
                    const float* u1 = (i0 + NPG < npix) ? u0 + qstep : u0;
                    // all loads first, then FMAs ordered so that neighbours in the instruction stream hit
                    // different accumulators (2*TA independent chains)
                    float xa[NGN][4], xb[NGN][4];
#pragma unroll
                    for (int g = 0; g < NGN; ++g) {
                        const float4 x0 = *reinterpret_cast<const float4*>(u0 + offn[g]);
                        const float4 x1 = *reinterpret_cast<const float4*>(u1 + offn[g]);
                        xa[g][0] = x0.x; xa[g][1] = x0.y; xa[g][2] = x0.z; xa[g][3] = x0.w;
                        xb[g][0] = x1.x; xb[g][1] = x1.y; xb[g][2] = x1.z; xb[g][3] = x1.w;
                    }
#pragma unroll
                    for (int g = 0; g < NGN; ++g)
#pragma unroll
                        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
                            for (int t = 0; t < TA; ++t) {
                                acc[q][t] = fmaf(wn[g][bb][t], xa[g][bb], acc[q][t]);
                                acc[q + 1][t] = fmaf(wn[g][bb][t], xb[g][bb], acc[q + 1][t]);
                            }
                }
            }
            // the previous diagonal: published by this CTA's threads and by the peers
            if (d > 0) {
                const unsigned prev = stepno - 1u;
                mbar_wait_or_give_up(&bars[prev & 1u], (prev >> 1) & 1u, gave_up);
            }
            // the two taps that read diagonal d-1
#pragma unroll
            for (int q = 0; q < PM; q += 2) {
                const int i0 = pg + NPG * q;
                if (i0 < npix) {
                    const float* u0 = ubase + q * qstep;
                    const float* u1 = (i0 + NPG < npix) ? u0 + qstep : u0;
                    float xa[NGC][4], xb[NGC][4];
#pragma unroll
                    for (int g = 0; g < NGC; ++g) {
                        const float4 x0 = *reinterpret_cast<const float4*>(u0 + offc[g]);
                        const float4 x1 = *reinterpret_cast<const float4*>(u1 + offc[g]);
                        xa[g][0] = x0.x; xa[g][1] = x0.y; xa[g][2] = x0.z; xa[g][3] = x0.w;
                        xb[g][0] = x1.x; xb[g][1] = x1.y; xb[g][2] = x1.z; xb[g][3] = x1.w;
                    }
#pragma unroll
                    for (int g = 0; g < NGC; ++g)
#pragma unroll
                        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
                            for (int t = 0; t < TA; ++t) {
                                acc[q][t] = fmaf(wc[g][bb][t], xa[g][bb], acc[q][t]);
                                acc[q + 1][t] = fmaf(wc[g][bb][t], xb[g][bb], acc[q + 1][t]);
                            }
                    if (!tfold) {
                        // fold the slices that share this warp, then one partial sum per warp and pixel
                        for (int o = LG; o < 32; o <<= 1) {
#pragma unroll
                            for (int t = 0; t < TA; ++t) {
                                acc[q][t] += __shfl_xor_sync(0xffffffffu, acc[q][t], o);
                                acc[q + 1][t] += __shfl_xor_sync(0xffffffffu, acc[q + 1][t], o);
                            }
                        }
                        if ((tq & 31) < LG) {
                            float* dst = red + ((size_t)i0 * NWP + wq) * CAp + l * TA;
#pragma unroll
                            for (int t = 0; t < TA; ++t) dst[t] = acc[q][t];
                            if (i0 + NPG < npix) {
#pragma unroll
                                for (int t = 0; t < TA; ++t) dst[NPG * NWP * CAp + t] = acc[q + 1][t];
                            }
                        }
                    }
                }
            }
            if (tfold) {
                // all pixel slots at once: slot sw of each round of SPW slots ends up in the lanes of slice sw
                const int sw = (tq & 31) / LG;
                auto fold_rounds = [&](auto spw_tag) {
                    constexpr int SPW = decltype(spw_tag)::value;
                    if constexpr (PM % SPW == 0) {
#pragma unroll
                        for (int rd = 0; rd < PM / SPW; ++rd) {
                            if (pg + NPG * (rd * SPW) < npix) {
                                float v[SPW * TA];
#pragma unroll
                                for (int x = 0; x < SPW; ++x)
#pragma unroll
                                    for (int t = 0; t < TA; ++t) v[x * TA + t] = acc[rd * SPW + x][t];
                                transposed_fold<SPW, TA>(v, sw, LG);
                                const int i = pg + NPG * (rd * SPW + sw);
                                float* dst = red + ((size_t)i * NWP + wq) * CAp + l * TA;
#pragma unroll
                                for (int t = 0; t < TA; ++t) dst[t] = v[t];
                            }
                        }
                    }
                };
                if (LG == 16) fold_rounds(std::integral_constant<int, 2>{});
                else if (LG == 8) fold_rounds(std::integral_constant<int, 4>{});
                else fold_rounds(std::integral_constant<int, 8>{});
            }
            __syncthreads();
            // finish the diagonal: sum the warps' partial sums and publish to every CTA of the cluster
            unsigned long long* mybar = &bars[stepno & 1u];
            if (R > 1 && tid == 0) mbar_expect_tx_only(mybar, (unsigned)((R - 1) * npix * CA * 4));
            const int obase = ((hlo + K - 1) * WP + (d - hlo) + K - 1) * CS + r * CA;
            if ((CA & 3) == 0) {
                // four channels per item: one 16-byte store here and one 16-byte asynchronous store per peer
                for (int i = finq_i0, aq = finq_a0; i < npix; ) {
                    const float* src2 = red + (size_t)i * NWP * CAp + aq * 4;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if constexpr (NGN <= 6) {
                        // all warps' partial sums in flight at once (NWP <= 8); the variants that hold more taps
                        // per thread have no registers to spare for this and measured slower with it
                        float4 tv[8];
#pragma unroll
                        for (int ww = 0; ww < 8; ++ww)
                            tv[ww] = ww < NWP ? *reinterpret_cast<const float4*>(src2 + ww * CAp) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int ww = 0; ww < 8; ++ww) { v.x += tv[ww].x; v.y += tv[ww].y; v.z += tv[ww].z; v.w += tv[ww].w; }
                    } else {
                        for (int ww = 0; ww < NWP; ++ww) {
                            const float4 t4 = *reinterpret_cast<const float4*>(src2 + ww * CAp);
                            v.x += t4.x; v.y += t4.y; v.z += t4.z; v.w += t4.w;
                        }
                    }
                    const int o = obase + i * DS + aq * 4;
                    *reinterpret_cast<float4*>(U + o) = v;
                    if (R > 1) {
#pragma unroll
                        for (int rr = 0; rr < 8; ++rr)
                            if (rr < R && rr != r)
                                st_async_f32x4(peerU[rr] + 4u * (unsigned)o, v, peerBar[rr] + 8u * (stepno & 1u));
                    }
                    i += finq_di; aq += finq_da;
                    if (aq >= CAQ) { aq -= CAQ; ++i; }
                }
            } else {
            for (int i = fin_i0, al = fin_a0; i < npix; ) {
                const float* src2 = red + (size_t)i * NWP * CAp + al;
                float v = 0.f;
                for (int ww = 0; ww < NWP; ++ww) v += src2[ww * CAp];
                const int o = obase + i * DS + al;
                U[o] = v;
                if (R > 1) {
#pragma unroll
                    for (int rr = 0; rr < 8; ++rr)
                        if (rr < R && rr != r)
                            st_async_f32(peerU[rr] + 4u * (unsigned)o, v, peerBar[rr] + 8u * (stepno & 1u));
                }
                i += fin_di; al += fin_da;
                if (al >= CA) { al -= CA; ++i; }
            }
            }
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(mybar);      // the warp's stores are ordered before its one arrival
        }
        {   // the last diagonal
            const unsigned prev = stepno - 1u;
            mbar_wait_or_give_up(&bars[prev & 1u], (prev >> 1) & 1u, gave_up);
        }
        // write back this CTA's channels
        float* dst = p.out + (size_t)n * C * HW + (size_t)r * CA * HW;
        if (p.vec) {
            float4* dst4 = reinterpret_cast<float4*>(dst);
            for (int vi = tid; vi < CA * nq4; vi += NT) {
                const int al = fast_div(vi, p.div_q4), pp = (vi - al * nq4) << 2;
                float vals[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    int h = fast_div(pp + i, p.div_w), w = (pp + i) - h * W;
                    if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                    vals[i] = U[((h + K - 1) * WP + (w + K - 1)) * CS + r * CA + al];
                }
                dst4[vi] = make_float4(vals[0], vals[1], vals[2], vals[3]);
            }
        } else {
            for (int e = tid; e < CA * HW; e += NT) {
                const int al = fast_div(e, p.div_hw), pp = e - al * HW;
                int h = fast_div(pp, p.div_w), w = pp - h * W;
                if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                dst[e] = U[((h + K - 1) * WP + (w + K - 1)) * CS + r * CA + al];
            }
        }
        // nobody publishes the next image's first diagonal into an image that is still being written back
        if (R > 1) { cluster_arrive_release(); cluster_wait_acquire(); } else __syncthreads();
    }
    if (tid == 0 && *gave_up) raise_status(INVCONV_TIMEOUT);
    if (R > 1) { cluster_arrive_release(); cluster_wait_acquire(); }   // no CTA exits while peers may still store into it
}

// ---------------------------------------------------------------------------
// Pixel-team variant: no block barrier inside a diagonal.
//
// A team of KW warps owns a pair of neighbouring pixels of every diagonal (and
// further pairs NTEAM pairs apart if the diagonal is long).  The contraction
// range is split over the KW*NS slices of the team -- over the lanes of a warp
// first -- so each pixel's sums are folded by shuffles inside the warp, joined
// across the team's warps through a few floats of shared memory and a named
// barrier of the team only, and published by the team's first warp (plain
// store + st.async to the peers, as above).  Teams never wait for one another
// inside a step: the only cross-team dependency is the mbarrier of the
// previous diagonal, on which one lane of every team arrives.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void named_barrier_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

template <int TA, int NGN, int NGC, int PJ>
__global__ void __launch_bounds__(256, (NGN <= 3 ? 2 : 1)) team_pixel_kernel(TeamParams p)
{
    extern __shared__ __align__(128) float smem[];
    __shared__ unsigned long long bars[2];
    __shared__ int gave_up_flag;                   // a bounded wait of this CTA ran out: later waits no longer block
    const int C = p.C, H = p.H, W = p.W, K = p.K, CS = p.CS, R = p.R, CA = p.CA;
    const int HP = H + K - 1, WP = W + K - 1, HW = H * W;
    const int IMG = HP * WP * CS;
    float* U = smem;
    float* RH = smem + IMG;
    float* tred = smem + 2 * IMG;                   // [team][kw][2 pixels][CAp]
    const int cl = blockIdx.x / R;
    const int r = blockIdx.x - cl * R;
    const int tid = threadIdx.x, NT = blockDim.x;
    const int LG = p.LG, NS = p.NS, KW = p.KW, NTEAM = p.NPG;
    const int warp = tid >> 5, lane = tid & 31;
    const int team = warp / KW, kw = warp - team * KW;
    const int s = lane / LG, l = lane - s * LG;
    const int gs = kw * NS + s, GSL = KW * NS;      // this thread's slice of the contraction range
    const int CAp = LG * TA;
    const int CB4 = (C + 3) >> 2;
    const int GN = (K > 1 ? K * K - 2 : 1) * CB4, GC = (K > 1 ? 2 : 0) * CB4;
    const int DS = (WP - 1) * CS;

    if (tid == 0) { gave_up_flag = 0; mbar_init(&bars[0], NTEAM); mbar_init(&bars[1], NTEAM); fence_mbar_init(); }   // one arrival per team
    for (int i = tid; i < 2 * IMG; i += NT) smem[i] = 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");          // the kernel transform before us has completed
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    float wn[NGN][4][TA], wc[NGC][4][TA];
    int offn[NGN], offc[NGC];
    auto fetch = [&](bool live, int tap, int b4, float (&dst)[4][TA], int& off) {
        const int dh = tap / K, dw = tap - dh * K;
        off = live ? (tap == 0 ? IMG : 0) - (dh * WP + dw) * CS + b4 * 4 : 0;
#pragma unroll
        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
            for (int t = 0; t < TA; ++t) {
                const int b = b4 * 4 + bb, al = l * TA + t;
                float v = 0.f;
                if (live && b < C && al < CA) v = __ldg(p.A + ((size_t)tap * C + b) * C + r * CA + al);
                dst[bb][t] = tap == 0 ? v : -v;
            }
    };
#pragma unroll
    for (int i = 0; i < NGN; ++i) {
        const int g = gs + i * GSL;
        const int tnc = g / CB4, b4 = g - tnc * CB4;
        const int tap = tnc == 0 ? 0 : (tnc <= K - 2 ? tnc + 1 : tnc + 2);
        fetch(g < GN, g < GN ? tap : 0, b4, wn[i], offn[i]);
    }
#pragma unroll
    for (int i = 0; i < NGC; ++i) {
        const int g = gs + i * GSL;
        const int tcr = g / CB4, b4 = g - tcr * CB4;
        fetch(g < GC, g < GC ? (tcr == 0 ? 1 : K) : 0, b4, wc[i], offc[i]);
    }
    uint32_t peerU[8], peerBar[8];
#pragma unroll
    for (int rr = 0; rr < 8; ++rr) {
        const uint32_t rk = (uint32_t)(rr < R ? rr : r);
        peerU[rr] = R > 1 ? cluster_map_u32(smem_u32(U), rk) : 0u;
        peerBar[rr] = R > 1 ? cluster_map_u32(smem_u32(&bars[0]), rk) : 0u;
    }

    __syncthreads();
    if (R > 1) { cluster_arrive_release(); cluster_wait_acquire(); }

    const int ND = H + W - 1;
    const int nq4 = HW >> 2;
    unsigned stepno = 0;
    volatile int* gave_up = &gave_up_flag;
    for (int n = cl; n < p.B; n += p.ncl) {
        const float* src = p.rhs + (size_t)n * C * HW;
        if (p.vec) {
            const float4* src4 = reinterpret_cast<const float4*>(src);
            const int nvec = C * nq4;
            for (int v0 = tid; v0 < nvec; v0 += NT * 8) {
                float4 tv[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (v0 + k * NT < nvec) tv[k] = __ldg(src4 + v0 + k * NT);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (v0 + k * NT < nvec) {
                        const int vi = v0 + k * NT;
                        const int c = fast_div(vi, p.div_q4), pp = (vi - c * nq4) << 2;
                        const float vals[4] = {tv[k].x, tv[k].y, tv[k].z, tv[k].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            int h = fast_div(pp + i, p.div_w), w = (pp + i) - h * W;
                            if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                            RH[((h + K - 1) * WP + (w + K - 1)) * CS + c] = vals[i];
                        }
                    }
                }
            }
        } else {
            for (int e0 = tid; e0 < C * HW; e0 += NT * 8) {
                float tv[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (e0 + k * NT < C * HW) tv[k] = __ldg(src + e0 + k * NT);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (e0 + k * NT < C * HW) {
                        const int e = e0 + k * NT;
                        const int c = fast_div(e, p.div_hw), pp = e - c * HW;
                        int h = fast_div(pp, p.div_w), w = pp - h * W;
                        if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                        RH[((h + K - 1) * WP + (w + K - 1)) * CS + c] = tv[k];
                    }
                }
            }
        }
        __syncthreads();

        for (int d = 0; d < ND; ++d, ++stepno) {
            const int hlo = max(0, d - (W - 1));
            const int npix = min(H - 1, d) - hlo + 1;
            const int dbase = ((hlo + K - 1) * WP + (d - hlo) + K - 1) * CS;   // pixel 0 of the diagonal
            float acc[PJ][2][TA];
#pragma unroll
            for (int j = 0; j < PJ; ++j)
#pragma unroll
                for (int t = 0; t < TA; ++t) { acc[j][0][t] = 0.f; acc[j][1][t] = 0.f; }
            // taps that read diagonals <= d-2 (and the right-hand side)
#pragma unroll
            for (int j = 0; j < PJ; ++j) {
                const int i0 = 2 * (team + NTEAM * j);
                if (i0 < npix) {
                    const float* u0 = U + dbase + i0 * DS;
                    const float* u1 = (i0 + 1 < npix) ? u0 + DS : u0;
#pragma unroll
                    for (int g = 0; g < NGN; ++g) {
                        const float4 x0 = *reinterpret_cast<const float4*>(u0 + offn[g]);
                        const float4 x1 = *reinterpret_cast<const float4*>(u1 + offn[g]);
                        const float a0[4] = {x0.x, x0.y, x0.z, x0.w}, a1[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
                            for (int t = 0; t < TA; ++t) {
                                acc[j][0][t] = fmaf(wn[g][bb][t], a0[bb], acc[j][0][t]);
                                acc[j][1][t] = fmaf(wn[g][bb][t], a1[bb], acc[j][1][t]);
                            }
                    }
                }
            }
            // the previous diagonal: published by every team of this CTA and by the peers.  A single CTA uses
            // the block barrier (every warp passes it only after its own publish of the previous step)
            if (R == 1) {
                __syncthreads();
            } else if (d > 0) {
                const unsigned prev = stepno - 1u;
                mbar_wait_or_give_up(&bars[prev & 1u], (prev >> 1) & 1u, gave_up);
            }
            unsigned long long* mybar = &bars[stepno & 1u];
            if (R > 1 && tid == 0) mbar_expect_tx_only(mybar, (unsigned)((R - 1) * npix * CA * 4));
#pragma unroll
            for (int j = 0; j < PJ; ++j) {
                const int i0 = 2 * (team + NTEAM * j);
                if (i0 < npix) {
                    const bool two = i0 + 1 < npix;
                    const float* u0 = U + dbase + i0 * DS;
                    const float* u1 = two ? u0 + DS : u0;
#pragma unroll
                    for (int g = 0; g < NGC; ++g) {
                        const float4 x0 = *reinterpret_cast<const float4*>(u0 + offc[g]);
                        const float4 x1 = *reinterpret_cast<const float4*>(u1 + offc[g]);
                        const float a0[4] = {x0.x, x0.y, x0.z, x0.w}, a1[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                        for (int bb = 0; bb < 4; ++bb)
#pragma unroll
                            for (int t = 0; t < TA; ++t) {
                                acc[j][0][t] = fmaf(wc[g][bb][t], a0[bb], acc[j][0][t]);
                                acc[j][1][t] = fmaf(wc[g][bb][t], a1[bb], acc[j][1][t]);
                            }
                    }
                    // fold the slices of this warp
                    for (int o = LG; o < 32; o <<= 1) {
#pragma unroll
                        for (int t = 0; t < TA; ++t) {
                            acc[j][0][t] += __shfl_xor_sync(0xffffffffu, acc[j][0][t], o);
                            acc[j][1][t] += __shfl_xor_sync(0xffffffffu, acc[j][1][t], o);
                        }
                    }
                    if (KW > 1) {
                        float* mine = tred + ((size_t)(team * KW + kw) * 2) * CAp + l * TA;
                        if (kw > 0 && lane < LG) {
#pragma unroll
                            for (int t = 0; t < TA; ++t) { mine[t] = acc[j][0][t]; mine[CAp + t] = acc[j][1][t]; }
                        }
                        named_barrier_sync(1 + team, KW * 32);
                        if (kw == 0 && lane < LG) {
                            for (int ow = 1; ow < KW; ++ow) {
                                const float* oth = tred + ((size_t)(team * KW + ow) * 2) * CAp + l * TA;
#pragma unroll
                                for (int t = 0; t < TA; ++t) { acc[j][0][t] += oth[t]; acc[j][1][t] += oth[CAp + t]; }
                            }
                        }
                        if (PJ > 1) named_barrier_sync(1 + team, KW * 32);   // the next pair reuses the exchange buffer
                    }
                    if (kw == 0 && lane < LG) {
                        const int o0 = dbase + i0 * DS + r * CA + l * TA;
#pragma unroll
                        for (int t = 0; t < TA; ++t) {
                            if (l * TA + t < CA) {
                                U[o0 + t] = acc[j][0][t];
                                if (two) U[o0 + DS + t] = acc[j][1][t];
                                if (R > 1) {
#pragma unroll
                                    for (int rr = 0; rr < 8; ++rr)
                                        if (rr < R && rr != r) {
                                            st_async_f32(peerU[rr] + 4u * (unsigned)(o0 + t), acc[j][0][t], peerBar[rr] + 8u * (stepno & 1u));
                                            if (two)
                                                st_async_f32(peerU[rr] + 4u * (unsigned)(o0 + DS + t), acc[j][1][t], peerBar[rr] + 8u * (stepno & 1u));
                                        }
                                }
                            }
                        }
                    }
                }
            }
            if (R > 1 && kw == 0) {
                __syncwarp();
                if (lane == 0) mbar_arrive(mybar);
            }
        }
        if (R > 1) {
            const unsigned prev = stepno - 1u;
            mbar_wait_or_give_up(&bars[prev & 1u], (prev >> 1) & 1u, gave_up);
        }
        __syncthreads();
        float* dst = p.out + (size_t)n * C * HW + (size_t)r * CA * HW;
        if (p.vec) {
            float4* dst4 = reinterpret_cast<float4*>(dst);
            for (int vi = tid; vi < CA * nq4; vi += NT) {
                const int al = fast_div(vi, p.div_q4), pp = (vi - al * nq4) << 2;
                float vals[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    int h = fast_div(pp + i, p.div_w), w = (pp + i) - h * W;
                    if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                    vals[i] = U[((h + K - 1) * WP + (w + K - 1)) * CS + r * CA + al];
                }
                dst4[vi] = make_float4(vals[0], vals[1], vals[2], vals[3]);
            }
        } else {
            for (int e = tid; e < CA * HW; e += NT) {
                const int al = fast_div(e, p.div_hw), pp = e - al * HW;
                int h = fast_div(pp, p.div_w), w = pp - h * W;
                if (p.rot) { h = H - 1 - h; w = W - 1 - w; }
                dst[e] = U[((h + K - 1) * WP + (w + K - 1)) * CS + r * CA + al];
            }
        }
        if (R > 1) { cluster_arrive_release(); cluster_wait_acquire(); } else __syncthreads();
    }
    if (tid == 0 && *gave_up) raise_status(INVCONV_TIMEOUT);
    if (R > 1) { cluster_arrive_release(); cluster_wait_acquire(); }
}

// ---------------------------------------------------------------------------
// Host-side launch plan.
// ---------------------------------------------------------------------------
struct TeamPlan {
    bool ok = false;
    bool pixel = false;      // pixel-team variant
    int KW = 1, PJ = 1;
    int R = 1, CA = 0, TA = 3, LG = 0, NS = 0, NPG = 1, CS = 0, PM = 0, NGN = 0, NGC = 0;
    int threads = 0, ncl = 0, maxt = 256;
    size_t smem = 0;
};

// Pixel-team variant: smallest estimated time over cluster size and warps per team.
inline TeamPlan plan_team_pixel(int B, int C, int H, int W, int K, size_t max_smem, int sm_count, bool forced = false)
{
    TeamPlan best;
    double best_cost = 1e30;
    const int CB4 = (C + 3) / 4;
    int CS = CB4 * 4;
    if (CS % 8 == 0) CS += 4;
    const int GN = (K > 1 ? K * K - 2 : 1) * CB4, GC = (K > 1 ? 2 : 0) * CB4;
    const int maxdiag = H < W ? H : W;
    const int pairs = (maxdiag + 1) / 2;
    const size_t img = (size_t)(H + K - 1) * (W + K - 1) * CS;
    const int menu[3][2] = {{3, 1}, {6, 2}, {12, 3}};
    // Measured on B200: across a cluster the slice variant is faster (wide48_k3: 108 us vs 181 us), for images
    // that one CTA serves the pixel teams are (cifar_sq: 41 us vs 72 us); so only R = 1 is planned here unless
    // the variant is forced (a measurement control).
    const int rmax = forced ? 8 : 1;
    for (int R = 1; R <= rmax; R *= 2) {
        if (C % R != 0) continue;
        const int CA = C / R;
        if (R > 1 && CA < 3) continue;
        const int TA = (CA % 3 == 0) ? 3 : 4;
        int LG = 1;
        while (LG * TA < CA) LG *= 2;
        if (LG > 32) continue;
        const int NS = 32 / LG;
        for (int KW = 1; KW <= 4; KW *= 2) {
            const int gsl = KW * NS;
            const int ngn = (GN + gsl - 1) / gsl, ngc = GC > 0 ? (GC + gsl - 1) / gsl : 0;
            int mi = -1;
            for (int m = 0; m < 3; ++m)
                if (ngn <= menu[m][0] && ngc <= menu[m][1]) { mi = m; break; }
            if (mi < 0) continue;
            int nteam = 8 / KW;
            if (nteam > pairs) nteam = pairs;
            const int pj = (pairs + nteam - 1) / nteam;
            if (pj > 2) continue;
            const size_t smem = sizeof(float) * (2 * img + (size_t)nteam * KW * 2 * LG * TA);
            if (smem > max_smem) continue;
            int conc = sm_count / R;                      // clusters in flight
            if (smem * 2 + 4096 <= max_smem && menu[mi][0] <= 6) conc *= 2;   // two CTAs fit one SM
            if (conc < 1) conc = 1;
            const int waves = (B + conc - 1) / conc;
            const double cost = (double)waves * pj * (menu[mi][0] + menu[mi][1] + 8 + (KW > 1 ? 4 : 0) + (R > 1 ? 4 : 0));
            if (cost < best_cost) {
                best_cost = cost;
                TeamPlan pl;
                pl.ok = true; pl.pixel = true;
                pl.R = R; pl.CA = CA; pl.TA = TA; pl.LG = LG; pl.NS = NS; pl.CS = CS;
                pl.NGN = menu[mi][0]; pl.NGC = menu[mi][1];
                pl.KW = KW; pl.PJ = pj; pl.NPG = nteam; pl.PM = 0;
                pl.threads = nteam * KW * 32;
                pl.smem = smem;
                int ncl = conc;
                if (ncl > B) ncl = B;
                pl.ncl = ncl;
                best = pl;
            }
        }
    }
    return best;
}

// variant: 0 by shape, 1 channel-slice kernel, 2 pixel-team kernel; forced_r: 0 by shape, else the cluster size
// of the channel-slice kernel (test and measurement controls).
inline TeamPlan plan_team(int B, int C, int H, int W, int K, size_t max_smem, int sm_count, int variant = 0, int forced_r = 0)
{
    TeamPlan best;
    if (C < 1 || K < 1) return best;
    if (variant != 1) {
        const TeamPlan px = plan_team_pixel(B, C, H, W, K, max_smem, sm_count, variant == 2);
        if (px.ok) return px;
    }
    // cluster size: enough CTAs that the kernel's share fits one CTA's registers, then fill the SMs
    int R = 1;
    auto divisible = [&](int rr) { return C % rr == 0 && (C / rr) >= 3; };
    while (R < 8 && (long long)C * C * K * K / R > 30000 && divisible(R * 2)) R *= 2;
    if ((long long)C * C * K * K / R > 30000) return best;
    while (R < 8 && (long long)B * R * 2 <= sm_count && divisible(R * 2)) R *= 2;
    if (forced_r >= 1 && forced_r <= 8 && C % forced_r == 0) R = forced_r;
    const int CA = C / R;
    const int CB4 = (C + 3) / 4;
    int CS = CB4 * 4;
    if (CS % 8 == 0) CS += 4;
    const int GN = (K > 1 ? K * K - 2 : 1) * CB4, GC = (K > 1 ? 2 : 0) * CB4;
    const int maxdiag = H < W ? H : W;
    const size_t img = (size_t)(H + K - 1) * (W + K - 1) * CS;
    const int TA = (CA % 3 == 0) ? 3 : 4;
    int LG = 1;
    while (LG * TA < CA) LG *= 2;
    if (LG > 32) return best;
    const int SPW = 32 / LG;
    const int menu[3][2] = {{3, 1}, {6, 2}, {9, 1}};
    for (int m = 0; m < 3; ++m) {
        const int NGN = menu[m][0], NGC = menu[m][1];
        int NS = (GN + NGN - 1) / NGN;
        if (GC > 0 && (GC + NGC - 1) / NGC > NS) NS = (GC + NGC - 1) / NGC;
        NS = (NS + SPW - 1) / SPW * SPW;
        const int maxt = 256;
        if (NS * LG > maxt) continue;
        TeamPlan pl;
        pl.R = R; pl.CA = CA; pl.TA = TA; pl.LG = LG; pl.NS = NS; pl.CS = CS; pl.NGN = NGN; pl.NGC = NGC;
        pl.maxt = maxt;
        int NPG = maxt / (NS * LG);
        const int want = (maxdiag + 1) / 2;                    // pixels are processed in pairs
        if (NPG > want) NPG = want;
        if (NPG < 1) NPG = 1;
        const int per = (maxdiag + NPG - 1) / NPG;             // pixel slots per group on the longest diagonal
        if (per > 16 || (maxt == 512 && per > 8)) continue;
        pl.PM = per <= 8 ? 8 : 16;
        pl.NPG = NPG;
        pl.threads = NPG * NS * LG;
        const size_t red = (size_t)(NPG * pl.PM + NPG) * (NS * LG / 32) * LG * TA;
        pl.smem = sizeof(float) * (2 * img + red);
        if (pl.smem > max_smem) continue;
        int ncl = sm_count / R;
        if (ncl > B) ncl = B;
        if (ncl < 1) ncl = 1;
        pl.ncl = ncl;
        pl.ok = true;
        best = pl;
        break;
    }
    return best;
}

}  // namespace invconv
