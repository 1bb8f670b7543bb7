// Launch geometry of the WARP family (host side; see warp_kernels.cuh for the kernel).
#pragma once

#include <stddef.h>

namespace invconv {

struct WarpPlan {
    bool ok = false;
    bool glb = false;      // image too large for shared memory: operands stay in global memory
    bool ring = false;     // ... and a ring of 128 columns per warp fits: streamed through shared memory
    bool cs = false;       // channel-split walk available (lane = (row, output channel)); its own geometry below
    int nb = 0, ipc = 0, grid = 0;
    int nb_cs = 0, ipc_cs = 0, grid_cs = 0;
    size_t smem = 0, smem_ring = 0, smem_cs = 0;
};

}  // namespace invconv
