// The selection as kernels of their own, launched right behind a row stage: the
// streaming and the TMA row stage of asd_verify.cu (which is also how a shard's rows
// become partials) and the fused LM head of asd_lmhead.cu.
//
// One warp per request, or with several blocks one CTA. It is launched with
// programmatic dependent launch and small enough to fit beside the row stage's
// CTAs on an SM; griddepcontrol.wait returns once the row stage has completed and
// its writes are visible, so no counters and no fences are needed, and the row
// stage's CTAs leave their SMs as soon as they have merged their rows.
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

// Several blocks of the same requests: one CTA per request, whose warps load as
// many blocks at once; only the walk over a block's mismatches, which needs the
// ledger as the block before left it, goes from warp to warp. One warp for all of
// a request's blocks took 0.85 us per block, most of it waiting for its loads:
// captured, 3 blocks of 23 requests 18.4 -> 16.1 us, 23 of 3 35 -> 26 us, 8 of 8 27
// -> 23 us (and 15.8, 24.5 and 22.2 us since the walk visits mismatches only).
constexpr int kSelectBlocksThreads = 256;

template <typename T>
static __global__ void __launch_bounds__(kSelectBlocksThreads)
    select_blocks_kernel(const __grid_constant__ VerifyParams p) {
  constexpr int kWarps = kSelectBlocksThreads / 32;
  __shared__ float s_spent;
  __shared__ bool s_wrote;
  pdl_signal_dependents();
  pdl_wait_prerequisites();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x;
  const float budget = __ldcg(&p.ledger[b].budget);
  if (threadIdx.x == 0) {
    s_spent = __ldcg(&p.ledger[b].spent);
    s_wrote = false;
  }
  for (int i0 = 0; i0 < p.nblk; i0 += kWarps) {
    const int i = i0 + warp;
    const long long vb = static_cast<long long>(i) * p.B + b;
    BlockInputs in;
    if (i < p.nblk) in = load_block<true>(p, vb, lane);
    for (int w = 0; w < kWarps && i0 + w < p.nblk; ++w) {
      __syncthreads();
      if (w != warp) continue;
      float spent = s_spent;
      bool wrote = s_wrote;
      select_block<T, false>(p, vb, in, budget, spent, wrote, lane);
      __syncwarp();
      if (lane == 0) {
        s_spent = spent;
        s_wrote = wrote;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_wrote) p.ledger[b].spent = s_spent;
}

template <typename T, bool kStrict>
int launch_select(const VerifyParams& p, bool pdl, cudaStream_t stream) {
  const bool blocks = !kStrict && p.nblk > 1 && !p.partials;
  constexpr int kWarps = kSelectThreads / 32;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks ? p.B : (p.B + kWarps - 1) / kWarps));
  cfg.blockDim = dim3(blocks ? kSelectBlocksThreads : kSelectThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  if (pdl) {
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
  }
  auto kernel = blocks ? select_blocks_kernel<T> : select_kernel<T, kStrict>;
  if (cudaLaunchKernelEx(&cfg, kernel, p) != cudaSuccess) return ASD_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? ASD_OK : ASD_ERR_CUDA;
}

}  // namespace asd_detail
