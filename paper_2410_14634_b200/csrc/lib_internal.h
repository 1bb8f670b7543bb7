// Host-side declarations shared by the translation units of the library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdio>

#include "common.cuh"
#include "tensor_plan.h"
#include "line_plan.h"
#include "warp_plan.h"
#include "gradw_quad_plan.h"

namespace invconv {
struct LineParams;
struct WarpParams;
struct TensorParams;
struct GradWSmallPlan;
struct GradWSmallParams;
}  // namespace invconv

namespace invconv_internal {

constexpr size_t kMaxDynSmem = 226 * 1024;   // 227 KiB per CTA minus the kernels' static shared memory

// Every translation unit has its own copy of the device status word (common.cuh); each registers the function that reads and clears
// its copy on the current device, and invconv_get_status asks all of them.
using StatusReader = int (*)(int*);
int register_status_reader(StatusReader reader);
namespace {
int read_clear_status(int* status_out)
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, invconv::g_device_status, sizeof(int)) != cudaSuccess) { cudaGetLastError(); return INVCONV_CUDA_ERROR; }
    if (v != 0) {
        const int zero = 0;
        cudaMemcpyToSymbol(invconv::g_device_status, &zero, sizeof(int));
    }
    *status_out = v;
    return INVCONV_OK;
}
[[maybe_unused]] const int status_reader_registered = register_status_reader(&read_clear_status);
}  // namespace

// Counts the launch and turns cudaGetLastError into a status code.
int check_launch();

// Stream-ordered device scratch from the library's own memory pool; release with cudaFreeAsync on the same stream.
int scratch_alloc(void** out, size_t bytes, cudaStream_t st);

// Multiprocessors of the current device (cached per device).
int sm_count();

template <typename Kern>
inline int set_smem_limit(Kern kern, size_t smem)
{
    // the 48 KB a kernel may use without opting in include its static shared memory (up to a few KB in some kernels)
    if (smem <= 40 * 1024) return INVCONV_OK;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return INVCONV_CUDA_ERROR;
    }
    return INVCONV_OK;
}

// invconv_lib.cu: forward / backward of the layer with Actnorm and the 1x1 convolution applied inside the warp-family
// kernel (see flow_step_lib.cu); INVCONV_UNSUPPORTED where that kernel does not serve the shape.
int warp_step_forward(const float* y, const float* w, const float* s, const float* b, const float* V, float* x, float* u,
                      invconv::Geom g, void* ws, cudaStream_t st);
int warp_step_backward(const float* grad_u, const float* x, const float* w, const float* s, const float* V,
                       float* grad_y, float* grad_w, invconv::Geom g, void* ws, cudaStream_t st);

// tensor_lib.cu: the tcgen05 wavefront (kernel transform into A, operand packing into wop, solve).
int tensor_launch(const invconv::TensorPlan& pl, bool bwd, const float* rhs, const float* w, float* out,
                  invconv::Geom g, float* A, unsigned char* wop, cudaStream_t st, float* logdet_out = nullptr);
// tensor3_lib.cu: the same wavefront with three-term products.
int tensor3_launch(const invconv::TensorPlan& pl, const invconv::TensorParams& prm, int k, cudaStream_t st);
int tensor_bounds_info(int* info);                        // debug-bounds build: first violation and count (both units)
int flow_bounds_info(int* info);
int tensor_selftest_bounds(cudaStream_t st);

// tensor_lib.cu: y = f(x) on the tensor cores; `pack` is device scratch of pl.pack_bytes bytes.
int conv_tensor_launch(const invconv::ConvTensorPlan& pl, const float* x, const float* w, float* y, invconv::Geom g,
                       unsigned char* pack, cudaStream_t st);

// tensor_lib.cu: the tcgen05 correlation kernel of grad_w; partial sums [pl.S][k*k][C][C] go to `partials`.
int gradw_tensor_launch(const invconv::GradWTensorPlan& pl, const float* gy, const float* x, float* partials,
                        invconv::Geom g, cudaStream_t st);

// warp_c*.cu: the few-channel kernels (WARP family, its grad_w, its masked convolution) of one channel count; INVCONV_UNSUPPORTED
// for a kernel side they do not have.
int launch_warp_c1(int k, bool bwd, const invconv::WarpPlan& pl, const invconv::WarpParams& prm, bool ring, bool split, bool dep, cudaStream_t st);
int launch_gradw_small_c1(int k, const invconv::GradWSmallPlan& gs, const invconv::GradWSmallParams& prm, bool dep, cudaStream_t st);
int launch_masked_conv_c1(const float* x, const float* w, float* y, invconv::Geom g, bool dep, cudaStream_t st);
int launch_warp_c2(int k, bool bwd, const invconv::WarpPlan& pl, const invconv::WarpParams& prm, bool ring, bool split, bool dep, cudaStream_t st);
int launch_masked_conv_c2(const float* x, const float* w, float* y, invconv::Geom g, bool dep, cudaStream_t st);
int launch_warp_c3(int k, bool bwd, const invconv::WarpPlan& pl, const invconv::WarpParams& prm, bool ring, bool split, bool dep, cudaStream_t st);
int launch_masked_conv_c3(const float* x, const float* w, float* y, invconv::Geom g, bool dep, cudaStream_t st);
int launch_warp_c4(int k, bool bwd, const invconv::WarpPlan& pl, const invconv::WarpParams& prm, bool ring, bool split, bool dep, cudaStream_t st);
int launch_masked_conv_c4(const float* x, const float* w, float* y, invconv::Geom g, bool dep, cudaStream_t st);

// gradw_quad_lib.cu: the fp32 correlation kernel of grad_w; partial sums [pl.shares][k*k][C][C] go to `partials`.
int gradw_quad_launch(const invconv::GradWQuadPlan& pl, const float* gy, const float* x, float* partials, invconv::Geom g,
                      bool dependent, cudaStream_t st);

// line_k*.cu: the LINE wavefront instances of one kernel side.
int launch_line_k2(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st);
int launch_line_k3(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st);
int launch_line_k5(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st);
int launch_line_k7(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st);
int launch_line_k9(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st);
int launch_line_k11(const invconv::LinePlan& pl, const invconv::LineParams& prm, bool dependent, cudaStream_t st);

}  // namespace invconv_internal
