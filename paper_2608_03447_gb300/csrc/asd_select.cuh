// The selection as a kernel of its own, launched right behind a row stage: the
// TMA row stage of asd_verify.cu and the fused LM head of asd_lmhead.cu.
//
// One warp per request. It is launched with programmatic dependent launch and
// small enough to fit beside the row stage's CTAs on an SM; griddepcontrol.wait
// returns once the row stage has completed and its writes are visible, so no
// counters and no fences are needed, and the row stage's CTAs leave their SMs
// as soon as they have merged their rows.
#pragma once

#include <cuda_runtime.h>

#include "asd.h"
#include "asd_device.cuh"

namespace asd_detail {

constexpr int kSelectThreads = 128;

template <typename T, bool kStrict>
static __global__ void __launch_bounds__(kSelectThreads) select_kernel(const __grid_constant__ VerifyParams p) {
  pdl_signal_dependents();
  pdl_wait_prerequisites();
  const int lane = threadIdx.x & 31;
  const int warps = kSelectThreads / 32;
  for (int b = blockIdx.x * warps + (threadIdx.x >> 5); b < p.B; b += gridDim.x * warps)
    select_request<T, kStrict>(p, b, lane);
}

template <typename T, bool kStrict>
int launch_select(const VerifyParams& p, bool pdl, cudaStream_t stream) {
  constexpr int kWarps = kSelectThreads / 32;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((p.B + kWarps - 1) / kWarps));
  cfg.blockDim = dim3(kSelectThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  if (pdl) {
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
  }
  if (cudaLaunchKernelEx(&cfg, select_kernel<T, kStrict>, p) != cudaSuccess) return ASD_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? ASD_OK : ASD_ERR_CUDA;
}

}  // namespace asd_detail
