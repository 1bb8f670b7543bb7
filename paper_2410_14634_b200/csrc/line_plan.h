// Launch geometry of the LINE wavefront (host side; the kernel is in line_kernels.cuh).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace invconv {

// Instances: X(K, NB, S, PR, MAXT, CMIN, CMAX) -- NB input channels per slice, S slices, PR rows per thread, most threads
// of a CTA (65536 / MAXT registers each), channel counts served.  A thread holds NB*K*K weights; slices keep that below about
// 160 registers, rows per thread keep C*S*rows/PR threads within the register file.
#define INVCONV_LINE_K2(X) \
    X(2, 1, 1, 1, 768, 1, 1) X(2, 2, 1, 1, 768, 2, 2) X(2, 3, 1, 1, 768, 3, 3) X(2, 4, 1, 1, 768, 4, 4) \
    X(2, 6, 1, 1, 640, 5, 6) X(2, 8, 1, 1, 640, 7, 8) X(2, 12, 1, 1, 512, 9, 12) X(2, 16, 1, 1, 512, 13, 16) \
    X(2, 12, 2, 2, 512, 17, 24) X(2, 16, 2, 2, 384, 25, 32)
#define INVCONV_LINE_K3(X) \
    X(3, 1, 1, 1, 768, 1, 1) X(3, 2, 1, 1, 768, 2, 2) X(3, 3, 1, 1, 640, 3, 3) X(3, 4, 1, 1, 640, 4, 4) \
    X(3, 6, 1, 1, 512, 5, 6) X(3, 8, 1, 1, 512, 7, 8) X(3, 12, 1, 1, 384, 9, 12) X(3, 12, 1, 2, 256, 9, 12) \
    X(3, 8, 2, 2, 384, 13, 16) X(3, 6, 4, 4, 384, 17, 24) X(3, 8, 4, 4, 256, 25, 32)
#define INVCONV_LINE_K5(X) \
    X(5, 1, 1, 1, 640, 1, 1) X(5, 2, 1, 1, 512, 2, 2) X(5, 3, 1, 1, 512, 3, 3) X(5, 4, 1, 1, 384, 4, 4) \
    X(5, 2, 2, 1, 640, 3, 4) X(5, 4, 2, 1, 384, 5, 8) X(5, 3, 4, 2, 512, 9, 12) X(5, 6, 2, 2, 256, 9, 12) X(5, 4, 4, 4, 256, 13, 16)
#define INVCONV_LINE_K7(X) \
    X(7, 1, 1, 1, 512, 1, 1) X(7, 2, 1, 1, 384, 2, 2) X(7, 2, 2, 1, 384, 3, 4)
#define INVCONV_LINE_K9(X) \
    X(9, 1, 1, 1, 512, 1, 1) X(9, 1, 2, 1, 512, 2, 2) X(9, 1, 4, 1, 512, 3, 4)
#define INVCONV_LINE_K11(X) \
    X(11, 1, 1, 1, 384, 1, 1) X(11, 1, 2, 1, 384, 2, 2) X(11, 1, 4, 1, 384, 3, 4)
#define INVCONV_LINE_ALL(X) \
    INVCONV_LINE_K2(X) INVCONV_LINE_K3(X) INVCONV_LINE_K5(X) INVCONV_LINE_K7(X) INVCONV_LINE_K9(X) INVCONV_LINE_K11(X)

struct LinePlan {
    bool ok = false;
    int NB = 0, S = 0, PR = 0;
    int HB = 0, nbands = 0, halo = 0, SW = 0;
    int cluster = 1;        // bands of an image walked at the same time by as many CTAs (nbands is then 1)
    int ncw = 0, niow = 0, grid = 0;                  // compute warps; loading warps, and as many storing ones
    int pieces = 0;
    int bk_warps = 0, bk_parts = 0, bk_per = 0;       // kernel transform: warps per share of the rows, shares, rows per share
    int off_dummy = 0, off_y = 0, off_ring = 0, off_a = 0, off_w = 0, off_li = 0;
    size_t smem = 0;
    double cycles = 0;      // estimated time of the wavefront
};

__host__ __device__ constexpr int line_cs(int NB, int S) { return (S * NB + 3) / 4 * 4; }
constexpr int kLinePieces = 8;      // pieces of four columns that an I/O thread moves per chunk, at most

inline LinePlan plan_line_instance(int B, int C, int H, int W, int K, int NB, int S, int PR, int MAXT, size_t max_smem, int sms, int max_bands = 32, bool clusters = false)
{
    LinePlan best;
    const int CSB = NB * S, CS = line_cs(NB, S);
    auto up = [](int v) { return (v + 31) & ~31; };
    for (int mode = 0; mode < (clusters ? 2 : 1); ++mode)
    for (int nb = 1; nb <= max_bands && nb <= H; nb = nb + (nb < 8 ? 1 : 4)) {
        LinePlan pl;
        pl.NB = NB; pl.S = S; pl.PR = PR;
        pl.HB = (H + nb - 1) / nb;
        pl.nbands = (H + pl.HB - 1) / pl.HB;
        if (pl.nbands != nb) continue;
        const bool cl = mode == 1;                     // the bands of an image in a cluster
        if (cl && nb != 2 && nb != 4 && nb != 8) continue;
        if (cl) { pl.cluster = nb; pl.nbands = 1; }
        pl.halo = nb > 1 ? K - 1 : 0;
        const int HBt = pl.HB + pl.halo;
        pl.ncw = ((HBt + PR - 1) / PR * C * S + 31) / 32;
        // pieces per I/O thread and chunk: few where a step is short, more where the threads are needed for rows
        for (int want = 3; want <= kLinePieces; want += (want < 4 ? 1 : 2)) {
        pl.niow = (HBt * C * 2 + 32 * want - 1) / (32 * want);
        pl.pieces = (HBt * C * 2 + 32 * pl.niow - 1) / (32 * pl.niow);
        const int threads = (pl.ncw + 2 * pl.niow) * 32;
        if (threads > MAXT) continue;
        pl.bk_warps = (C * (K * K - 1) + 31) / 32;
        if (pl.bk_warps > pl.ncw) pl.bk_warps = pl.ncw;
        pl.bk_parts = pl.ncw / pl.bk_warps;
        pl.bk_per = (C + pl.bk_parts - 1) / pl.bk_parts;
        // columns of one (image, band) and the zero gap behind it; a band's halo rows are read after the band above
        // has stored them (see line_kernels.cuh), chunk alignment lets whole 16-byte pieces move
        int sw = W + K - 1;
        sw = (sw + 3) & ~3;
        if (nb > 1 && !cl) {
            const int least = 8 * (7 + (pl.HB - 1 + 7) / 8);
            if (sw < least) sw = least;
            sw = (sw + 7) & ~7;
        }
        pl.SW = sw;
        int off = up(2 * (HBt + K - 1 + PR) * CS);
        pl.off_dummy = off; off += 32;
        pl.off_y = off;     off = up(off + 2 * (HBt + PR) * CS);
        pl.off_ring = off;  off = up(off + (HBt + PR) * C * 68);
        pl.off_a = off;     off = up(off + (C | 1) * K * K * CSB);
        pl.off_li = off;    off = up(off + CS * CS);
        pl.off_w = off;     off = up(off + C * C * K * K);
        pl.smem = sizeof(float) * (size_t)off;
        if (pl.smem > max_smem) continue;
        // time: dependent step plus the multiply-adds of the warps that share a scheduler
        int occ = MAXT / threads;
        const int by_smem = (int)((max_smem + 1024) / (pl.smem + 1024));
        if (occ > by_smem) occ = by_smem;
        if (occ > 4) occ = 4;
        const double fma = (double)PR * NB * K * K;
        for (int o = 1; o <= occ; ++o) {
            const int room = o * sms / pl.cluster;     // images in flight
            if (room < 1) continue;
            const int images = B < room ? B : room, grid = images * pl.cluster;
            const int resident = (grid + sms - 1) / sms, nimg = (B + images - 1) / images;
            const double warps = (double)((pl.ncw * resident + 3) / 4);
            // fitted to timings of all instances; a lone warp on its scheduler issues a multiply-add only every 2.6 cycles
            double step = 160.0 + 1.5 * fma * (warps < 1.75 ? 1.75 : warps) + 35.0 * warps;
            if (nb > 1) step *= 1.15;                  // halo rows
            const double io = (500.0 + (W % 4 == 0 ? 250.0 : 400.0) * pl.pieces) / 8;
            if (io > step) step = io;
            const double t = 7000.0 + ((double)(nimg * pl.nbands - 1) * pl.SW + W + pl.HB + (pl.cluster - 1) * (pl.HB + 56.0)) * step;
            if (!best.ok || t < best.cycles) {
                best = pl;
                best.grid = grid;
                best.cycles = t;
                best.ok = true;
            }
        }
        }
    }
    return best;
}

inline LinePlan plan_line(int B, int C, int H, int W, int K, size_t max_smem, int sms, int max_bands = 32, bool clusters = false)
{
    LinePlan best;
    if (B < 1) return best;
#define X(K_, NB_, S_, PR_, MAXT_, CMIN_, CMAX_)                                                                   \
    if (K == K_ && C >= CMIN_ && C <= CMAX_) {                                                                       \
        const LinePlan pl = plan_line_instance(B, C, H, W, K, NB_, S_, PR_, MAXT_, max_smem, sms, max_bands, clusters);            \
        if (pl.ok && (!best.ok || pl.cycles < best.cycles)) best = pl;                                              \
    }
    INVCONV_LINE_ALL(X)
#undef X
    return best;
}

}  // namespace invconv
