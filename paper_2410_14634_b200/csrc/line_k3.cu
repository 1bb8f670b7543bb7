#include "line_inst.cuh"

INVCONV_LINE_UNIT(launch_line_k3, INVCONV_LINE_K3)
