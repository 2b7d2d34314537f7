// libasd: combine step of the vocabulary-sharded verifier.
//
// Each vocabulary shard has reduced every target row to an asd_partial (key
// with the global index, exact top logit, the draft token's logit if the
// shard holds it). Here one warp per request merges row j's S partials in lane
// j -- the largest key wins (larger logit, then lower global index), its
// shard's top value comes with it, the draft logit comes from the shard that
// holds the draft token -- and runs the same selection as asd_verify, so the
// result equals the unsharded verify bit for bit.
#include <cuda_runtime.h>
#include <stdint.h>

#include "asd.h"
#include "asd_device.cuh"
#include "asd_launch.cuh"

namespace {

using namespace asd_detail;

constexpr int kCombineThreads = 256;
// Shards whose partials are in flight at once, beside the ledger and the draft:
// read shard by shard the combine was five L2 round trips in a row.
constexpr int kCombineBatch = 4;

// Through L1, since the three words of a partial share their sectors with the
// neighbouring lanes' (griddepcontrol.wait makes the writes of the kernels ahead
// visible to ordinary loads; not left to the compiler, which may choose the read-only
// path for a pointer that the kernel does not write through). Past L1 each word asked
// for its sector again: 8 shards of 32 requests took 2.58 us where shard by shard it
// had been 2.46, and 16 of 5000 requests of 32 rows 16.4 where it had been 8.0 (now
// 2.37 and 7.2). Four shards of 32 requests: 2.19 shard by shard, 1.88, now 1.76 us.
__device__ __forceinline__ asd_partial load_partial(const asd_partial* at) {
  const unsigned long long* w = reinterpret_cast<const unsigned long long*>(at);
  unsigned long long key, values, flags;
  asm volatile("ld.global.u64 %0, [%1];" : "=l"(key) : "l"(w));
  asm volatile("ld.global.u64 %0, [%1];" : "=l"(values) : "l"(w + 1));
  asm volatile("ld.global.u64 %0, [%1];" : "=l"(flags) : "l"(w + 2));
  asd_partial q;
  q.key = key;
  q.top = __uint_as_float(static_cast<uint32_t>(values));
  q.draft_logit = __uint_as_float(static_cast<uint32_t>(values >> 32));
  q.flags = static_cast<uint32_t>(flags);
  q.reserved = 0u;
  return q;
}

__global__ void __launch_bounds__(kCombineThreads) shard_combine_kernel(const asd_partial* __restrict__ parts,
                                                                        int S, const __grid_constant__ VerifyParams p) {
  const int lane = threadIdx.x & 31;
  const int warps = blockDim.x / 32;
  const int K = p.K, K1 = p.K + 1;
  const long long R = static_cast<long long>(p.B) * K1;
  pdl_signal_dependents();
  pdl_wait_prerequisites();  // the partials are read only once the kernel before this one is done
  for (int b = blockIdx.x * warps + (threadIdx.x >> 5); b < p.B; b += gridDim.x * warps) {
    BlockInputs in;
    in.key = 0ull;
    in.x = -1;
    in.zx = -INFINITY;
    in.top = 0.0f;
    in.top_exact = true;  // every shard sends its top value exactly as stored
    unsigned flags = 0u;
    float budget = 0.0f, spent = 0.0f;
    if (lane == 0) {
      budget = __ldcg(&p.ledger[b].budget);
      spent = __ldcg(&p.ledger[b].spent);
    }
    if (lane < K1) {
      const long long row = static_cast<long long>(b) * K1 + lane;
      if (lane < K) in.x = __ldcg(p.draft + static_cast<long long>(b) * K + lane);
      asd_partial best = load_partial(parts + row);
      float zx = best.draft_logit;
      flags = best.flags;
      for (int s0 = 1; s0 < S; s0 += kCombineBatch) {
        asd_partial q[kCombineBatch];
#pragma unroll
        for (int i = 0; i < kCombineBatch; ++i) {
          q[i].key = 0ull;  // past the last shard: what changes nothing
          q[i].draft_logit = -INFINITY;
          q[i].flags = 0u;
          if (s0 + i < S) q[i] = load_partial(parts + static_cast<long long>(s0 + i) * R + row);
        }
#pragma unroll
        for (int i = 0; i < kCombineBatch; ++i) {
          if (q[i].key > best.key) best = q[i];
          if (q[i].draft_logit != -INFINITY) zx = q[i].draft_logit;  // the shard that holds the draft token
          flags |= q[i].flags;
        }
      }
      in.key = best.key;
      in.top = best.top;
      if (lane < K) in.zx = zx;
    }
    in.flags = __reduce_or_sync(kFull, flags);
    budget = __shfl_sync(kFull, budget, 0);
    spent = __shfl_sync(kFull, spent, 0);
    bool wrote = false;
    select_block<float, false>(p, b, in, budget, spent, wrote, lane);
    if (lane == 0 && wrote) p.ledger[b].spent = spent;
  }
}

}  // namespace

extern "C" int asd_shard_combine(const asd_partial* partials, int S, int B, int K, int V, const int32_t* draft,
                                 asd_ledger* ledger, float gate, int cap, int32_t* accepted_len,
                                 int32_t* committed, int32_t* recovery, int32_t* row_argmax, float* row_regret,
                                 int32_t* status, asd_stream_t stream) {
  int rc = check_shape(B, K, V, ASD_F32);
  if (rc != ASD_OK) return rc;
  if (S < 1) return ASD_ERR_SHAPE;
  if (B == 0) return ASD_OK;
  if (!partials || !ledger || !accepted_len || !committed || !recovery) return ASD_ERR_NULL;
  if (K > 0 && !draft) return ASD_ERR_NULL;
  if (gate != gate || gate < 0.0f || cap < 0) return ASD_ERR_CONTROL;
  VerifyParams p = {};
  p.logits = nullptr;
  p.B = B;
  p.K = K;
  p.V = V;
  p.nblk = 1;
  p.v_total = V;
  p.draft = draft;
  p.ledger = ledger;
  p.gate = gate;
  p.cap = cap;
  p.accepted_len = accepted_len;
  p.committed = committed;
  p.recovery = recovery;
  p.row_argmax = row_argmax;
  p.row_regret = row_regret;
  p.status = status;
  constexpr int kWarps = kCombineThreads / 32;
  const unsigned grid = static_cast<unsigned>((B + kWarps - 1) / kWarps);
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg =
      pdl_config(dim3(grid), dim3(kCombineThreads), reinterpret_cast<cudaStream_t>(stream), &attr);
  if (cudaLaunchKernelEx(&cfg, shard_combine_kernel, partials, S, p) != cudaSuccess) return ASD_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? ASD_OK : ASD_ERR_CUDA;
}
