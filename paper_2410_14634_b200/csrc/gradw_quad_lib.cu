// Launch side of the fp32 correlation kernel (gradw_quad.cuh): its own translation unit, for build time.
#include <cstdio>

#include "lib_internal.h"
#include "gradw_quad.cuh"

using namespace invconv;

namespace invconv_internal {

namespace {
template <int T, int K>
int launch(const GradWQuadPlan& pl, const GradWQuadParams& prm, bool dependent, cudaStream_t st)
{
    auto kern = gradw_quad_kernel<T, K>;
    const int rc = set_smem_limit(kern, pl.smem);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.grid);
    cfg.blockDim = dim3(pl.threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, prm) != cudaSuccess) {
        std::fprintf(stderr, "invconv: grad_w launch failed: %s\n", cudaGetErrorString(cudaGetLastError()));
        return INVCONV_CUDA_ERROR;
    }
    return check_launch();
}
}  // namespace

int gradw_quad_launch(const GradWQuadPlan& pl, const float* gy, const float* x, float* partials, Geom g, bool dependent, cudaStream_t st)
{
    GradWQuadParams prm = {};
    prm.gy = gy; prm.x = x; prm.partials = partials;
    prm.B = g.B; prm.C = g.C; prm.H = g.H; prm.W = g.W;
    prm.RB = pl.RB; prm.nbands = pl.nbands; prm.shares = pl.shares; prm.NCO = pl.NCO; prm.cotiles = pl.cotiles; prm.tiles = pl.tiles;
    prm.WPT = pl.WPT; prm.gst = pl.gst; prm.xst = pl.xst; prm.gfloats = pl.gfloats; prm.stage = pl.stage;
    prm.vec = (((reinterpret_cast<uintptr_t>(gy) | reinterpret_cast<uintptr_t>(x)) & 15) == 0 && g.W % 4 == 0) ? 1 : 0;
    prm.div_bands = make_fast_div((unsigned)pl.nbands);
    prm.div_grow = make_fast_div((unsigned)(pl.gst / 4));
    prm.div_gch = make_fast_div((unsigned)pl.RB);
    prm.div_xch = make_fast_div((unsigned)(pl.RB + g.k - 1));
    prm.long_rows = !prm.vec && g.W >= 24;
    prm.div_q = make_fast_div((unsigned)(prm.vec ? g.W / 4 : g.W));
    prm.div_k = make_fast_div((unsigned)g.k);
#define X(T_, K_) if (pl.T == T_ && g.k == K_) return launch<T_, K_>(pl, prm, dependent, st);
    X(1, 1) X(2, 1) X(3, 1) X(4, 1) X(1, 2) X(2, 2) X(3, 2) X(4, 2) X(1, 3) X(2, 3) X(3, 3) X(4, 3) X(1, 4) X(2, 4) X(3, 4) X(4, 4)
    X(1, 5) X(2, 5) X(3, 5) X(4, 5) X(1, 7) X(2, 7) X(3, 7) X(1, 9) X(2, 9) X(3, 9) X(1, 11) X(2, 11) X(3, 11)
#undef X
    return INVCONV_UNSUPPORTED;
}

}  // namespace invconv_internal
