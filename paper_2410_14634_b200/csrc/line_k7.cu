#include "line_inst.cuh"

INVCONV_LINE_UNIT(launch_line_k7, INVCONV_LINE_K7)
INVCONV_LINE_UNIT(launch_line_k9, INVCONV_LINE_K9)
INVCONV_LINE_UNIT(launch_line_k11, INVCONV_LINE_K11)
