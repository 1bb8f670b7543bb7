#include "warp_inst.cuh"

INVCONV_WARP_UNIT(1)

namespace invconv_internal {
int launch_gradw_small_c1(int k, const GradWSmallPlan& gs, const GradWSmallParams& prm, bool dep, cudaStream_t st)
{
    switch (k) {
    case 2: return launch_gradw_small_ck<1, 2>(gs, prm, dep, st);
    case 3: return launch_gradw_small_ck<1, 3>(gs, prm, dep, st);
    case 5: return launch_gradw_small_ck<1, 5>(gs, prm, dep, st);
    default: return INVCONV_UNSUPPORTED;
    }
}
}  // namespace invconv_internal
