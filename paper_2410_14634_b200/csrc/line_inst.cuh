// One translation unit per kernel side instantiates the LINE kernels it launches (they build in parallel).
#pragma once

#include <cstdio>

#include "lib_internal.h"
#include "line_kernels.cuh"

namespace invconv_internal {

template <int NB, int K, int S, int PR, int MAXT>
int launch_line_inst(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st)
{
    auto kern = invconv::line_wavefront_kernel<NB, K, S, PR, MAXT>;
    const int rc = set_smem_limit(kern, pl.smem);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.grid);
    cfg.blockDim = dim3((pl.ncw + 2 * pl.niow) * 32);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)pl.cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = pl.cluster > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, kern, prm) != cudaSuccess) {
        std::fprintf(stderr, "invconv: line launch failed: %s\n", cudaGetErrorString(cudaGetLastError()));
        return INVCONV_CUDA_ERROR;
    }
    return check_launch();
}

}  // namespace invconv_internal

#define INVCONV_LINE_CASE(K_, NB_, S_, PR_, MAXT_, CMIN_, CMAX_)                                                          \
    if (pl.NB == NB_ && pl.S == S_ && pl.PR == PR_) return launch_line_inst<NB_, K_, S_, PR_, MAXT_>(pl, prm, dependent, st);

#define INVCONV_LINE_UNIT(name, list)                                                                                     \
    namespace invconv_internal {                                                                                          \
    int name(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st)                 \
    {                                                                                                                     \
        list(INVCONV_LINE_CASE) return INVCONV_UNSUPPORTED;                                                               \
    }                                                                                                                     \
    }
