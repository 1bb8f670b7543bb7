// Launcher of the tensor-core wavefront; the translation units that include it instantiate the kernels they launch.
#pragma once

#include <cstdio>

#include "lib_internal.h"
#include "tensor_kernels.cuh"

namespace invconv_internal {

using namespace invconv;

template <int R, int K, bool T3>
int launch_tensor_inst(const TensorPlan& pl, const TensorParams& prm, cudaStream_t st)
{
    auto kern = tensor_wavefront_kernel<R, K, T3>;
    if (R > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return INVCONV_UNSUPPORTED;
    }
    const int rc = invconv_internal::set_smem_limit(kern, pl.smem);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.ncl * pl.R);
    cfg.blockDim = dim3(kTensorThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    // Programmatic dependent launch: the CTAs set themselves up (barriers, tensor memory, the right-hand side)
    // while the kernel transform still runs; they wait for it (griddepcontrol.wait) before reading its output.
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = pl.R; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, prm);
    if (e != cudaSuccess) {
        std::fprintf(stderr, "invconv: tensor launch failed: %s\n", cudaGetErrorString(e));
        cudaGetLastError();
        return INVCONV_CUDA_ERROR;
    }
    return invconv_internal::check_launch();
}

}  // namespace invconv_internal
