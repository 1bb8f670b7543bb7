// Arguments of the LINE wavefront kernel (line_kernels.cuh).
#pragma once

#include "common.cuh"
#include "tma.cuh"

namespace invconv {

struct LineParams {
    const void* rhs;       // y (forward) or grad_x (backward), [B][C][H][W]
    const float* w;        // [C][C][K][K]
    void* out;             // x or grad_y
    int B, C, H, W;
    int HB, nbands, halo;  // rows per band, bands per image, halo rows (K-1 or 0)
    int cluster;           // CTAs per image, one band each (1: the bands of an image follow one another in one CTA)
    int SW;                // virtual columns per (image, band)
    FastDiv div_sw, div_c, div_nb;
    int rot;               // 1: transposed solve on the rotated image
    int bf16;              // rhs and out are bfloat16
    int vec;               // W is a multiple of four and every image pointer is aligned to four elements: pieces of four columns
    int bk_warps, bk_parts, bk_per;   // kernel transform: warps per share of the rows, shares, rows per share
    FastDiv div_bk;
    int pieces;            // pieces of four columns per I/O thread and chunk
    int ncw, niow;         // compute warps; loading warps, and as many storing ones
    int off_dummy, off_y, off_ring, off_a, off_w, off_li;   // float offsets in shared memory
    // the flow step's per-pixel neighbours (see WarpParams) on the way in: grad_x = s V^T grad_u
    const float* mix_V; const float* mix_s; int mix_in;
    float* logdet_out;
};

}  // namespace invconv
