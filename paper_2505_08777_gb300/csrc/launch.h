// Launchers of the D-templated transform kernels (one translation unit per
// range of D so the instantiations compile in parallel).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace ash {

// Launches a kernel that begins with pdl_begin(): its blocks are scheduled while
// the kernel before it on the stream still runs (programmatic dependent launch),
// which hides the launch latencies of a call made kernel by kernel (forward
// 1024^2 N = 400 79 -> 71 us, calibration sweep 770 -> 701). Not while the
// stream is captured: a graph's own edges are shorter (WGS loop 1700 / 1723 us,
// batch of 16 1926 / 2057 with these edges).
template <typename... K, typename... A>
cudaError_t launch_pdl(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(s, &cap);
  if (e != cudaSuccess) return e;
  c.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, static_cast<K>(args)...);
}

struct LaunchInfo {
  int threads;        // CTA size of the pixel-stationary kernels
  int fwd_ctas_per_sm;
  int adj_ctas_per_sm;
  int gradc_ctas_per_sm;
  int tc_adj_ctas_per_sm;   // 0 if the tensor-core path is not available for this D
  int tc_fwd_ctas_per_sm;
  int tc_grad_ctas_per_sm;   // 0 if the tensor-core moment pass is not available
};

// Each returns cudaErrorInvalidValue when D is outside its range.
#define ASH_DECLARE_RANGE(R)                                                                  \
  cudaError_t prepare_r##R(int D, LaunchInfo* info);                                          \
  cudaError_t launch_forward_r##R(int D, const FwdParams& p, int grid, cudaStream_t s);       \
  cudaError_t launch_adjoint_r##R(int D, const AdjParams& p, int grid, cudaStream_t s);       \
  cudaError_t launch_gradc_r##R(int D, const GradCParams& p, dim3 grid, cudaStream_t s);
ASH_DECLARE_RANGE(0)
ASH_DECLARE_RANGE(1)
ASH_DECLARE_RANGE(2)
ASH_DECLARE_RANGE(3)
#undef ASH_DECLARE_RANGE

// Range r covers D in [4r + 1, 4r + 4].
inline int range_of(int D) { return (D - 1) / 4; }

}  // namespace ash
