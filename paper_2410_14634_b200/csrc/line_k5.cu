#include "line_inst.cuh"

INVCONV_LINE_UNIT(launch_line_k5, INVCONV_LINE_K5)
