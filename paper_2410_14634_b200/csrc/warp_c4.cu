#include "warp_inst.cuh"

INVCONV_WARP_UNIT(4)
