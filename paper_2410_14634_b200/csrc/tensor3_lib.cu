// The tensor-core wavefront with three-term products (fp32 accuracy): its own translation unit, for build time.
#include "tensor_inst.cuh"

namespace invconv_internal {

int tensor3_launch(const TensorPlan& pl, const TensorParams& prm, int k, cudaStream_t st)
{
#define X(R_, K_) if (pl.three && pl.R == R_ && k == K_) return launch_tensor_inst<R_, K_, true>(pl, prm, st);
    X(2, 2) X(2, 3) X(2, 5) X(4, 2) X(4, 3) X(4, 5) X(6, 2) X(6, 3) X(6, 5) X(8, 2) X(8, 3) X(8, 5) X(10, 2) X(10, 3) X(12, 2) X(12, 3)
#undef X
    return INVCONV_UNSUPPORTED;
}

}  // namespace invconv_internal
