// libasd: fused LM-head + verify for GB300 (sm_103a).
//
// z = h W^T (h: [T, H] bf16 hidden states of the T = B(K+1) target rows,
// W: [V, H] bf16 LM-head weight) is computed on the 5th-generation tensor cores
// with fp32 accumulation in tensor memory, and reduced in the epilogue to what
// the verifier needs (Sec. 3.3: the top token, the top logit and the draft
// token's logit, with no [T, V] logit buffer); the selection of Alg. 1 then
// runs as in asd_verify. The logits never reach global memory.
//
// Tiling: two CTAs on a pair of SMs (a cluster of 2) share 2-SM MMAs
// (tcgen05 cta_group::2). An MMA's M is 256 vocabulary rows (128 per SM: the
// TMEM lanes), its N is one token tile (the TMEM columns): the T token rows are
// cut into as few tiles of at most 256 columns as hold them, all of the same
// width (T = 576: three of 192, no padding; T = 18: one of 32). With several
// token tiles a pair works through items of two vocabulary tiles (512 rows) by one
// token tile: per 64-deep K step each SM loads 2 x 128 rows of W and half of the
// token rows and issues two MMAs per K slice over the same token slab, so the token
// rows cross from L2 once per two vocabulary tiles; with one token tile an item is
// one vocabulary tile (see launch_lmhead). Items are dealt to the pairs in one
// sequence, token tiles innermost, so the pairs that need a W row run at the
// same time and it comes from HBM about once (see LmDeal for the last round).
// Per CTA: warp 0 issues TMA loads (128B-swizzled 64-wide K slabs) into a ring
// of as many stages as fit, whose completion is counted on the first CTA's
// barrier; warp 1 allocates tensor memory, and in the first CTA one of its
// threads issues the MMAs; the other warps reduce the accumulators. Accumulators
// are slots in a ring of two to four (512 columns / token tile width), each handed
// over by barriers of its own, so that the MMAs of the next item begin when one
// tile has been read and run ahead in it while the other is being read.
// The epilogue reads each 32 x 32 block (vocabulary rows x token columns) of a
// warp as matrix fragments, four rows of eight columns per thread, so a column's
// maximum over a thread's rows is register arithmetic; it goes on to find where
// a maximum sits only in blocks where some column reaches the best logit that
// the token has so far (see reduce_block).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "asd.h"
#include "asd_device.cuh"
#include "asd_lm_deal.h"
#include "asd_select.cuh"

namespace {

using namespace asd_detail;

constexpr int kHalfM = 128;               // vocabulary rows per CTA in one MMA (TMEM lanes)
constexpr int kBK = 64;                   // K per stage: 64 bf16 = one 128-byte swizzle row
constexpr int kUmmaK = 16;                // K per tcgen05.mma (kind::f16)
constexpr int kMaxStages = 12;
constexpr int kSlabA = kHalfM * kBK * 2;  // 16 KB of vocabulary rows per tile
constexpr int kMaxSlots = 4;              // accumulators in tensor memory
// Epilogue warps: a tile's 32-column blocks go in turn to the warps of each TMEM
// lane quarter. A reduction that still has to look for its maxima (a pair's first
// item) takes 1.2 us a block, and nothing hides it behind a pair's last item. With
// one token tile, where that is what a call adds to streaming the weight, there are
// sixteen warps instead of eight: on 38912 rows 73.5 us instead of 77.2 for 256
// tokens, 68.5 instead of 70.8 for 160. With more tiles (or logits to write) the
// tensor cores set the pace, and sixteen gain nothing.
constexpr int kEpiWarpsOneTile = 16;
constexpr int kEpiWarps = 8;
constexpr int lm_threads(int epi_warps) { return (2 + epi_warps) * 32; }  // producer, MMA, epilogue warps
constexpr int kTmemCols = 512;
static_assert(kEpiWarps * 32 >= kMaxTN, "one epilogue thread per token column");

struct LmShared {
  unsigned long long full[kMaxStages];   // first CTA: both CTAs' loads of a stage have landed
  unsigned long long empty[kMaxStages];  // each CTA: the MMAs have read its part of a stage
  unsigned long long acc_full[kMaxSlots];   // each CTA: the slot's accumulator is complete
  unsigned long long acc_empty[kMaxSlots];  // first CTA: both CTAs' epilogues have read it
  unsigned long long drain;
  uint32_t tmem_base;
  int abort;
  int draft[kMaxTN];                  // x of the tile's token rows (-1: no draft / out of range)
  alignas(16) float thr[kMaxTN];      // each token's best logit when the item began: less cannot win
  unsigned long long best[kMaxTN];    // each token's best (value, index) key, as far as this CTA knows
};
// dynamic shared memory: [1 KB alignment slack][stages x B][stages x A][LmShared]
constexpr size_t kLmSmemMax = 232448;
constexpr size_t lm_stage_bytes(int tn, int kw) { return kw * kSlabA + static_cast<size_t>(tn) / 2 * kBK * 2; }
constexpr int lm_stages(int tn, int kw) {
  const size_t fit = (kLmSmemMax - 1024 - sizeof(LmShared)) / lm_stage_bytes(tn, kw);
  const int most = kw == 1 ? kMaxStages : kMaxStages / 2;
  return fit < static_cast<size_t>(most) ? static_cast<int>(fit) : most;
}
constexpr size_t lm_smem_bytes(int tn, int kw) {
  return 1024 + lm_stages(tn, kw) * lm_stage_bytes(tn, kw) + sizeof(LmShared);
}
static_assert(lm_stages(192, 2) == 5 && lm_stages(kMaxTN, 2) == 4, "ring depth at the widths that serve most");

// ---------------------------------------------------------------- tcgen05 / TMA / cluster helpers

// Shared-memory matrix descriptor of a K-major operand tile written by TMA with
// 128-byte swizzling: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);          // start address
  d |= static_cast<uint64_t>(1u) << 16;                         // leading byte offset (unused when swizzled)
  d |= static_cast<uint64_t>((1024u >> 4) & 0x3FFFu) << 32;     // stride byte offset: 8 rows x 128 B
  d |= static_cast<uint64_t>(1u) << 46;                         // descriptor version
  d |= static_cast<uint64_t>(2u) << 61;                         // 128-byte swizzle
  return d;
}

// Instruction descriptor: kind::f16 with bf16 A and B, fp32 D, both K-major,
// M = kPairM (across the pair), N = the token tile's width.
__device__ __forceinline__ uint32_t instr_desc(int tn) {
  return (1u << 4)                                     // D format: f32
         | (1u << 7)                                   // A format: bf16
         | (1u << 10)                                  // B format: bf16
         | (static_cast<uint32_t>(tn >> 3) << 17)      // N / 8
         | (static_cast<uint32_t>(kPairM >> 4) << 24); // M / 16
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The shared::cluster address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// One bounded wait on the phase with the given parity. The thread may sleep
// until the phase completes (at most kSuspendNs per call), so the warps that
// wait -- most of them, most of the time -- take no issue slots from the MMA
// and TMA threads (polling them cost this kernel about 7 %).
constexpr uint32_t kSuspendNs = 1000000;
// Longer than any load takes: what is waited, after a timeout, for loads that no barrier counts.
constexpr unsigned long long kLandNs = 10000000;
__device__ __forceinline__ bool mbar_try_wait_cluster(unsigned long long* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return done != 0;
}
// Whether the phase with the given parity has completed; never sleeps.
__device__ __forceinline__ bool mbar_test_cluster(unsigned long long* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// mbar_wait for barriers that the other CTA of the pair also signals; the
// abort flag and the clock are checked every 16 sleeps.
__device__ inline bool mbar_wait_cluster(unsigned long long* bar, uint32_t parity, volatile int* abort) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (unsigned it = 1;; ++it) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((it & 15u) == 0) {
      if (*abort) return false;
      if (global_ns() - t0 > kWaitLimitNs) return false;
    }
  }
}

// The wait of the two warps that feed the tensor cores: by the whole warp, with
// one answer for all of it, so that the compiler can keep what the loop around
// it counts in uniform registers, which the MMA and TMA instructions take their
// operands from; and with the hardware's own short suspend time, which wakes
// sooner than a long one (609 -> 600 us for 576 tokens).
__device__ inline bool mbar_wait_warp(unsigned long long* bar, uint32_t parity, volatile int* abort) {
  auto completed = [&] {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return __all_sync(kFull, done != 0) != 0;
  };
  if (completed()) return true;
  const unsigned long long t0 = global_ns();
  for (unsigned it = 1;; ++it) {
    if (completed()) return true;
    if ((it & 255u) == 0 && __any_sync(kFull, *abort != 0 || global_ns() - t0 > kWaitLimitNs)) return false;
  }
}
// True in one lane of the warp, the same one every time.
__device__ __forceinline__ bool elect_lane() {
  uint32_t one;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(one));
  return one != 0;
}

// TMA tile load into this CTA's shared memory whose completion is counted on
// an mbarrier of either CTA of the pair (cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster, int x,
                                                 int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void umma_pair_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The mbarrier at this offset in both CTAs of the pair arrives once every
// tcgen05 operation this thread issued so far has completed.
__device__ __forceinline__ void umma_commit_pair(unsigned long long* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(smem_u32(bar)), "h"(static_cast<uint16_t>(0x3)) : "memory");
}
// Same, for this CTA's barrier only.
__device__ __forceinline__ void umma_commit_local(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 32 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// Rows l / 4 and l / 4 + 8 (of 16 TMEM lanes from the one addressed on) of lane
// l's warp, 32 consecutive fp32 columns: r[4g + e] is row l / 4, r[4g + 2 + e]
// row l / 4 + 8, both of column 8g + 2 (l % 4) + e.
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The sticky error word, when the call has a workspace (asd_lmhead_logits has none).
__device__ __forceinline__ void report_timeout(const VerifyParams& p) {
  if (p.error) atomicExch(p.error, static_cast<unsigned>(ASD_ERR_TIMEOUT));
}

// Sets the abort flag of both CTAs of the pair.
__device__ __forceinline__ void abort_pair(LmShared& sh, uint32_t peer) {
  sh.abort = 1;
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_rank(smem_u32(&sh.abort), peer)), "r"(1) : "memory");
}

// Order-preserving bits of a column maximum; NaN is mapped above +inf
// whatever its sign bit, so a NaN anywhere in a row reaches the row's key.
__device__ __forceinline__ uint32_t max_bits(float v) { return v != v ? 0xffc00000u : ordered_bits(v); }

// Meets the threads of the epilogue warps.
template <int kEpi>
__device__ __forceinline__ void epilogue_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kEpi * 32) : "memory");
}

// Argmax of one warp's 32 x 32 block of logits: vocabulary rows v_warp on (TMEM
// lanes lane_base on) by token columns c on of the tile.
//
// What this costs is the time the tensor cores wait for it, so the common case
// is kept short: as fragments, a thread holds rows l/4 + {0, 8, 16, 24} of eight
// columns, three maxima a column with no other lane needed, and one vote tells
// whether any column of the block reaches its token's best logit so far. Once
// the first units are in, that is rare (a block of 32 of the V rows holds the
// best of all rows so far for a token), and only then the lanes exchange maxima
// (seven shuffles leave one column per lane) and look for the lowest row that
// holds them. Turning the block around through shared memory instead, which
// gives every column's index every time, took about 520 cycles a block with
// eight warps at it, and 36 KB that now hold a fifth stage of the ring. Back to
// back under the power cap: 604 -> 597 us for 576 tokens (624 against 658 us
// for a first pass), 2159 -> 2134 us for 2304, 90.8 -> 85.7 us for 160 tokens on
// a 37984-row shard. A NaN passes the vote and reaches the token's key.
__device__ __forceinline__ void reduce_block(LmShared& sh, const VerifyParams& p, uint32_t tmem_block, int c,
                                             int tok0, int T, int v_warp, int lane) {
  uint32_t r[2][16];
  tmem_ld_frag(tmem_block, r[0]);
  tmem_ld_frag(tmem_block + (16u << 16), r[1]);
  const int q = lane >> 2, j = lane & 3;
  float2 thr[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) thr[g] = *reinterpret_cast<const float2*>(&sh.thr[c + 8 * g + 2 * j]);
  const int x = sh.draft[c + lane] - v_warp;  // lane l: the row of column c + l's draft token
  tmem_ld_wait();

  // draft logits: the thread holding row x of column i keeps z_i(x) (rare: at most one row per column)
  unsigned hit = __ballot_sync(kFull, static_cast<unsigned>(x) < 32u);
  while (hit) {
    const int i = __ffs(hit) - 1;
    hit &= hit - 1;
    const int row = __shfl_sync(kFull, x, i);
    if (q == (row & 7) && j == ((i & 7) >> 1)) {
      const int at = 4 * (i >> 3) + 2 * ((row >> 3) & 1) + (i & 1);
      float z = 0.0f;
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (k == at) z = __uint_as_float(row & 16 ? r[1][k] : r[0][k]);
      p.draft_logit[tok0 + c + i] = z;
    }
  }
  if (v_warp + 31 >= p.V) {  // the last, partial tile: rows past V never win
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (v_warp + 16 * h + 8 * ((k >> 1) & 1) + q >= p.V) r[h][k] = __float_as_uint(-INFINITY);
  }

  float m[8];  // column 8 (i / 2) + 2j + i % 2: the maximum of this thread's four rows
  bool reaches = false;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = 4 * (i >> 1) + (i & 1);
    m[i] = fmax_nan(fmax_nan(__uint_as_float(r[0][k]), __uint_as_float(r[0][k + 2])),
                    fmax_nan(__uint_as_float(r[1][k]), __uint_as_float(r[1][k + 2])));
    reaches |= !(m[i] < (i & 1 ? thr[i >> 1].y : thr[i >> 1].x));
  }
  if (!__any_sync(kFull, reaches)) return;

  // One column per lane: of its columns a lane keeps those whose index bit
  // equals its own bit, and hands the others over.
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float m4[4], m2[2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    m4[i] = fmax_nan(b4 ? m[i + 4] : m[i], __shfl_xor_sync(kFull, b4 ? m[i] : m[i + 4], 16));
#pragma unroll
  for (int i = 0; i < 2; ++i)
    m2[i] = fmax_nan(b3 ? m4[i + 2] : m4[i], __shfl_xor_sync(kFull, b3 ? m4[i] : m4[i + 2], 8));
  const float zmax = fmax_nan(b2 ? m2[1] : m2[0], __shfl_xor_sync(kFull, b2 ? m2[0] : m2[1], 4));
  const int mine = c + ((lane >> 3) & 3) * 8 + 2 * j + ((lane >> 2) & 1);
  const uint32_t hi = max_bits(zmax);
  const bool wins = tok0 + mine < T && hi >= static_cast<uint32_t>(sh.best[mine] >> 32);
  if (!__any_sync(kFull, wins)) return;

  // the lowest row that holds each column's maximum; none does for a NaN
  int w[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float z = __shfl_sync(kFull, zmax, (i << 2) | j);
    const int k = 4 * (i >> 1) + (i & 1);
    w[i] = __uint_as_float(r[0][k]) == z       ? q
           : __uint_as_float(r[0][k + 2]) == z ? q + 8
           : __uint_as_float(r[1][k]) == z     ? q + 16
           : __uint_as_float(r[1][k + 2]) == z ? q + 24
                                               : 32;
  }
  int w4[4], w2[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) w4[i] = min(b4 ? w[i + 4] : w[i], __shfl_xor_sync(kFull, b4 ? w[i] : w[i + 4], 16));
#pragma unroll
  for (int i = 0; i < 2; ++i) w2[i] = min(b3 ? w4[i + 2] : w4[i], __shfl_xor_sync(kFull, b3 ? w4[i] : w4[i + 2], 8));
  const int row = min(b2 ? w2[1] : w2[0], __shfl_xor_sync(kFull, b2 ? w2[0] : w2[1], 4)) & 31;
  if (wins)
    atomicMax(&sh.best[mine], (static_cast<unsigned long long>(hi) << 32) |
                                  (0xffffffffu - static_cast<uint32_t>(v_warp + row)));
}

struct LmParams {
  int T, H, V;
  int tn;           // token rows per tile
  int token_tiles;  // ceil(T / tn)
  int stages;       // ring stages
  int slots;        // accumulator slots
  int k_steps;      // ceil(H / kBK)
  int full, entries;  // of the deal
  float* logits_out;  // [T, V] when writing logits instead of verifying
};

// One entry of the deal.
struct LmItem {
  int row0;  // first vocabulary row
  int kw;    // vocabulary tiles
  int m;     // token tile
};
template <int kW>
__device__ __forceinline__ LmItem lm_item(const LmParams& q, int entry) {
  const int half = entry - q.full;
  const int item = half < 0 ? entry : q.full + (half >> 1);
  LmItem it;
  it.m = item % q.token_tiles;
  it.row0 = (item / q.token_tiles) * (kW * kPairM) + (half < 0 ? 0 : (half & 1) * kPairM);
  it.kw = kW == 2 && half < 0 && it.row0 + kPairM < q.V ? 2 : 1;  // no second tile past the vocabulary
  return it;
}

// One CTA pair (cluster of 2) works through entries pair, pair + pairs, ...
// kW: vocabulary tiles per item.
template <bool kWriteLogits, int kEpi, int kW>
__global__ void __launch_bounds__(lm_threads(kEpi), 1)
    lmhead_verify_kernel(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_w,
                         const __grid_constant__ VerifyParams p, const __grid_constant__ LmParams q) {
  extern __shared__ __align__(1024) unsigned char lm_smem_raw[];
  const uint32_t raw = smem_u32(lm_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // 1024-byte aligned for the 128-byte swizzle
  unsigned char* gbase = lm_smem_raw + (base - raw);
  const int stages = q.stages;
  const uint32_t stage_b = static_cast<uint32_t>(q.tn) / 2 * kBK * 2;  // this CTA's half of the token rows
  const uint32_t sB = base;                                            // stages x stage_b
  constexpr uint32_t kStageA = kW * kSlabA;
  const uint32_t sA = base + static_cast<uint32_t>(stages) * stage_b;  // stages x kStageA
  LmShared& sh = *reinterpret_cast<LmShared*>(gbase + static_cast<uint32_t>(stages) * (kStageA + stage_b));

  const int warp = __shfl_sync(kFull, static_cast<int>(threadIdx.x >> 5), 0);  // uniform, to the compiler too
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank() & 1u;
  const uint32_t peer = rank ^ 1u;
  const bool leader = rank == 0;
  const int pair = static_cast<int>(blockIdx.x >> 1), pairs = static_cast<int>(gridDim.x >> 1);
  const int K1 = p.K + 1;

  pdl_signal_dependents();  // the selection's CTAs may take their places beside this kernel's
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    for (int s = 0; s < kMaxSlots; ++s) {
      mbar_init(&sh.acc_full[s], 1);
      mbar_init(&sh.acc_empty[s], 2 * kEpi);  // the epilogue warps of both CTAs
    }
    mbar_init(&sh.drain, 1);
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {  // tensor memory of both SMs, allocated together by one warp of each CTA
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&sh.tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers exist before either signals the other's
  tc_fence_after();
  const uint32_t tmem = __reduce_max_sync(kFull, sh.tmem_base);  // uniform, to the compiler too
  // everything above touches this SM only; the hidden states, drafts, the workspace and the outputs may be the
  // previous kernel's
  pdl_wait_prerequisites();

  int issued = 0, issued_stage = 0;  // producer: loads issued, and the stage the next one goes to
  uint32_t issued_phase = 0;
  // The producer and the MMA warp run their loops as whole warps and let one lane issue: counters, descriptors
  // and coordinates stay in uniform registers. With one thread in the loop each MMA waited for its operands to
  // be moved there: 576 tokens (three tiles of 192 columns) took as long per item as 256 columns do, 645 us a
  // call against 525 us with all else equal.
  if (warp == 0) {
    // ---------------- TMA producer (both CTAs; completion counted on the first CTA's barrier)
    const bool elected = elect_lane();
    if (elected) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_h)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_w)) : "memory");
    }
    const uint32_t full0 = map_rank(smem_u32(&sh.full[0]), 0);
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int e = pair; ok && e < q.entries; e += pairs) {
      const LmItem it = lm_item<kW>(q, e);
      const int tok = it.m * q.tn + static_cast<int>(rank) * (q.tn / 2);
      const int row = it.row0 + static_cast<int>(rank) * kHalfM;
      const uint32_t tx = 2u * (static_cast<uint32_t>(it.kw) * kSlabA + stage_b);  // both CTAs' bytes
      for (int k = 0; k < q.k_steps; ++k) {
        ok = mbar_wait_warp(&sh.empty[s], ph ^ 1u, &sh.abort);
        if (!ok) break;
        if (elected) {
          if (leader) mbar_expect_tx(&sh.full[s], tx);
          const uint32_t bar = full0 + static_cast<uint32_t>(s * sizeof(unsigned long long));
          tma_load_2d_pair(sB + s * stage_b, &map_h, bar, k * kBK, tok);
          // this CTA's 128 rows of each vocabulary tile
          tma_load_2d_pair(sA + s * kStageA, &map_w, bar, k * kBK, row);
          if (it.kw == 2) tma_load_2d_pair(sA + s * kStageA + kSlabA, &map_w, bar, k * kBK, row + kPairM);
        }
        ++issued;
        if (++s == stages) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    if (!ok && elected) {
      abort_pair(sh, peer);
      report_timeout(p);
    }
    issued_stage = s;
    issued_phase = ph;
  } else if (warp == 1) {
    // ---------------- MMA issuer (one warp of the first CTA, for both SMs)
    if (leader) {
      const bool elected = elect_lane();
      const uint32_t idesc = instr_desc(q.tn);
      const uint64_t a_desc = smem_desc_sw128(sA), b_desc = smem_desc_sw128(sB);
      // the MMAs of one K step of vocabulary tile j: stage s into the accumulator at column d
      auto mma_step = [&](int s, int j, uint32_t d, bool first) {
        const uint64_t ad = a_desc + static_cast<uint32_t>((s * static_cast<int>(kStageA) + j * kSlabA) >> 4);
        const uint64_t bd = b_desc + ((static_cast<uint32_t>(s) * stage_b) >> 4);
#pragma unroll
        for (int kk = 0; kk < kBK / kUmmaK; ++kk)  // 16 elements (32 bytes, encoded 2) along K inside the swizzle row
          umma_pair_bf16(d, ad + 2u * kk, bd + 2u * kk, idesc, !first || kk > 0 ? 1u : 0u);
      };
      int s0 = 0, s1 = 0;  // the stages the first and the second tile's next K step read
      uint32_t ph = 0;     // of s0
      int slot = 0;
      uint32_t slot_ph = 1;
      bool ok = true;
      for (int e = pair; ok && e < q.entries; e += pairs) {
        const int kw = lm_item<kW>(q, e).kw;
        const int slot0 = slot;
        const uint32_t d0 = tmem + static_cast<uint32_t>(slot0 * q.tn);
        ok = mbar_wait_warp(&sh.acc_empty[slot0], slot_ph, &sh.abort);
        if (!ok) break;
        if (++slot == q.slots) {
          slot = 0;
          slot_ph ^= 1u;
        }
        const int slot1 = slot;
        const uint32_t ph1 = slot_ph;
        const uint32_t d1 = tmem + static_cast<uint32_t>(slot1 * q.tn);
        if (kw == 2 && ++slot == q.slots) {
          slot = 0;
          slot_ph ^= 1u;
        }
        bool free1 = false;  // the second tile's slot has been read
        int k1 = 0;          // K steps issued for the second tile
        for (int k = 0; k < q.k_steps; ++k) {
          ok = mbar_wait_warp(&sh.full[s0], ph, &sh.abort);
          if (!ok) break;
          tc_fence_after();
          const bool last = k == q.k_steps - 1;
          if (elected) {
            mma_step(s0, 0, d0, k == 0);
            if (last) umma_commit_pair(&sh.acc_full[slot0]);
            if (kw == 1) umma_commit_pair(&sh.empty[s0]);  // frees the stage in both CTAs once these MMAs have read it
          }
          if (kw == 1) {
            if (++s1 == stages) s1 = 0;
          } else {
            // while the second tile's slot is still being read, the first tile runs ahead as far as the ring goes
            if (!free1) {
              if (last || k - k1 + 1 >= stages) {
                ok = mbar_wait_warp(&sh.acc_empty[slot1], ph1, &sh.abort);
                if (!ok) break;
                free1 = true;
              } else {
                free1 = __all_sync(kFull, mbar_test_cluster(&sh.acc_empty[slot1], ph1));
              }
              tc_fence_after();
            }
            for (; free1 && k1 <= k; ++k1) {
              if (elected) {
                mma_step(s1, 1, d1, k1 == 0);
                umma_commit_pair(&sh.empty[s1]);
              }
              if (++s1 == stages) s1 = 0;
            }
          }
          if (++s0 == stages) {
            s0 = 0;
            ph ^= 1u;
          }
        }
        if (ok && kw == 2 && elected) umma_commit_pair(&sh.acc_full[slot1]);
      }
      if (elected) {
        if (!ok) {
          abort_pair(sh, peer);
          report_timeout(p);
        }
        umma_commit_local(&sh.drain);  // arrives once every MMA issued above has finished
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(&sh.drain, 0) && global_ns() - t0 < kWaitLimitNs) {
        }
      }
      __syncwarp();
    }
  } else {
    // ---------------- epilogue: warps 2 on, each on one TMEM lane quarter, whose warps take turns at the 32-column
    // blocks of every accumulator
    constexpr int kTurns = kEpi / 4;
    const int quarter = warp & 3;  // TMEM lanes this warp may read
    const int turn = (warp - 2) >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t acc_empty0 = map_rank(smem_u32(&sh.acc_empty[0]), 0);
    const int et = static_cast<int>(threadIdx.x) - 64;  // this thread among the epilogue's: its token column
    int slot = 0;
    uint32_t slot_ph = 0;
    bool ok = true;
    for (int e = pair; e < q.entries; e += pairs) {
      const LmItem it = lm_item<kW>(q, e);
      const int tok0 = it.m * q.tn;
      // While the item's MMAs run: its draft tokens, and what each token has to beat, over all CTAs so far
      const bool has_token = et < q.tn && tok0 + et < q.T;
      unsigned long long known = 0ull;
      if (!kWriteLogits) {
        if (et < q.tn) {
          int x = -1;
          if (has_token) {
            const int tok = tok0 + et, b = tok / K1, j = tok - b * K1;
            known = __ldcg(&p.row_key[tok]);
            // the row of this weight that holds the draft token (a vocabulary shard starts at global index
            // v_offset), if any
            if (j < p.K) x = __ldcg(p.draft + static_cast<long long>(b) * p.K + j) - p.v_offset;
            if (x < 0 || x >= p.V) x = -1;
          }
          sh.draft[et] = x;
          sh.best[et] = known;
          sh.thr[et] = !has_token ? INFINITY : known ? ordered_value(static_cast<uint32_t>(known >> 32)) : -INFINITY;
        }
        epilogue_sync<kEpi>();
      }
      for (int t = 0; t < it.kw; ++t) {
        // after a wait that gave up the warp goes on without reducing: the other warps meet it at the barriers
        if (ok) {
          ok = __all_sync(kFull, mbar_wait_cluster(&sh.acc_full[slot], slot_ph, &sh.abort));
          if (!ok && lane == 0) {
            abort_pair(sh, peer);
            report_timeout(p);
          }
        }
        if (ok) {
          tc_fence_after();
          const uint32_t acc = tmem + lane_base + static_cast<uint32_t>(slot * q.tn);
          const int v_warp = it.row0 + t * kPairM + static_cast<int>(rank) * kHalfM + quarter * 32;
          if (v_warp < q.V) {  // rows past the vocabulary: nothing to reduce
            for (int c = turn * 32; c < q.tn; c += kTurns * 32) {
              if (kWriteLogits) {
                const int v = v_warp + lane;  // this thread's vocabulary row
                uint32_t r[32];
                tmem_ld32(acc + static_cast<uint32_t>(c), r);
                tmem_ld_wait();
                if (v < q.V) {
                  float* out = q.logits_out + static_cast<long long>(tok0 + c) * q.V + v;
#pragma unroll
                  for (int i = 0; i < 32; ++i)
                    if (tok0 + c + i < q.T) out[static_cast<long long>(i) * q.V] = __uint_as_float(r[i]);
                }
              } else {
                reduce_block(sh, p, acc + static_cast<uint32_t>(c), c, tok0, q.T, v_warp, lane);
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(acc_empty0 + static_cast<uint32_t>(slot * sizeof(unsigned long long)));
        }
        if (++slot == q.slots) {
          slot = 0;
          slot_ph ^= 1u;
        }
      }
      if (!kWriteLogits) {
        epilogue_sync<kEpi>();  // every warp's maxima are in sh.best
        if (has_token) {
          const unsigned long long key = sh.best[et];
          if (key != known) {
            atomicMax(&p.row_key[tok0 + et], key);
            if ((key >> 32) == 0xffc00000ull) atomicOr(&p.flags[(tok0 + et) / K1], ASD_STATUS_NAN_LOGIT);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (sh.abort && leader && warp == 0 && lane == 0) {
    // wait (bounded) for the loads still in flight before the pair exits
    for (int n = issued < stages ? issued : stages; n > 0; --n) {
      if (--issued_stage < 0) {
        issued_stage = stages - 1;
        issued_phase ^= 1u;
      }
      const unsigned long long t0 = global_ns();
      while (!mbar_try_wait_cluster(&sh.full[issued_stage], issued_phase) && global_ns() - t0 < kWaitLimitNs) {
      }
    }
  }
  if (sh.abort && !leader && warp == 0 && lane == 0) {
    // the second CTA may be a load ahead of the first, whose barrier does not wait for that one: give it time to land
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < kLandNs) {
    }
  }
  __syncthreads();
  cluster_sync_all();  // neither CTA frees tensor memory or exits while the other may still use the pair
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------- host side

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &res) ==
            cudaSuccess &&
        res == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  return fn;
}

// 2-D bf16 row-major [rows, cols] tensor, boxes of box_rows x kBK columns,
// 128-byte swizzle; out-of-range rows and columns read as zero.
bool make_map(CUtensorMap* map, const void* ptr, int rows, int cols, int box_rows) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(cols) * 2};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct LmDevice {
  int sms = 0;
  int major = 0, minor = 0;
  // CTA pairs resident at once, per kernel instance (0: not set up yet); the
  // set-up is idempotent, so two threads racing to do it store the same value
  std::atomic<int> pairs[4] = {};
};

int lm_device(LmDevice** out) {
  constexpr int kMaxDevices = 64;
  static LmDevice info[kMaxDevices];
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ASD_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return ASD_ERR_DEVICE;
  std::lock_guard<std::mutex> g(mu);
  if (info[dev].sms == 0) {
    if (cudaDeviceGetAttribute(&info[dev].sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&info[dev].major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&info[dev].minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
      return ASD_ERR_CUDA;
  }
  *out = &info[dev];
  return ASD_OK;
}

cudaLaunchConfig_t pair_config(unsigned grid, int threads, size_t smem, cudaStream_t stream,
                               cudaLaunchAttribute (&attr)[2], bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cfg;
}

LmParams lm_params(int T, int V, int H, int kw, int pairs) {
  const LmDeal d = lm_deal(T, V, kw, pairs);
  LmParams q = {};
  q.T = T;
  q.H = H;
  q.V = V;
  q.tn = d.tn;
  q.token_tiles = d.token_tiles;
  q.full = d.full;
  q.entries = d.entries;
  q.stages = lm_stages(d.tn, kw);
  q.slots = kTmemCols / d.tn < kMaxSlots ? kTmemCols / d.tn : kMaxSlots;
  q.k_steps = 1 + (H - 1) / kBK;
  return q;
}

template <bool kWriteLogits, int kEpi, int kW>
int launch_lmhead_kernel(LmDevice* dev, const void* hidden, const void* weight, int H, int T, const VerifyParams& p,
                         float* logits_out, cudaStream_t stream) {
  if (dev->major != 10) return ASD_ERR_DEVICE;  // tcgen05 needs a Blackwell (sm_10x) device
  auto kernel = lmhead_verify_kernel<kWriteLogits, kEpi, kW>;
  std::atomic<int>& resident = dev->pairs[2 * (kW - 1) + (kWriteLogits ? 1 : 0)];
  cudaLaunchAttribute attr[2];
  int pairs = resident.load(std::memory_order_acquire);
  if (pairs == 0) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kLmSmemMax)) !=
        cudaSuccess)
      return ASD_ERR_CUDA;
    // every token tile width leaves room for one CTA per SM
    cudaLaunchConfig_t probe =
        pair_config(static_cast<unsigned>(dev->sms & ~1), lm_threads(kEpi), kLmSmemMax, stream, attr, false);
    if (cudaOccupancyMaxActiveClusters(&pairs, kernel, &probe) != cudaSuccess || pairs < 1) return ASD_ERR_CUDA;
    resident.store(pairs, std::memory_order_release);
  }
  LmParams q = lm_params(T, p.V, H, kW, pairs);
  q.logits_out = logits_out;
  CUtensorMap map_h, map_w;
  if (!make_map(&map_h, hidden, T, H, q.tn / 2) || !make_map(&map_w, weight, p.V, H, kHalfM)) return ASD_ERR_CUDA;
  const unsigned grid = 2u * static_cast<unsigned>(q.entries < pairs ? q.entries : pairs);
  cudaLaunchConfig_t cfg = pair_config(grid, lm_threads(kEpi), lm_smem_bytes(q.tn, kW), stream, attr, true);
  if (cudaLaunchKernelEx(&cfg, kernel, map_h, map_w, p, q) != cudaSuccess) return ASD_ERR_CUDA;
  if (kWriteLogits) return cudaGetLastError() == cudaSuccess ? ASD_OK : ASD_ERR_CUDA;
  return launch_select<float, false>(p, true, stream);
}

// With one token tile an item is one vocabulary tile and a stage half as long (the
// ring twice as deep): the token rows are read from L2 once more, but the first of
// two tiles is reduced while the second one's weight streams, instead of both at
// the end. On 38912 vocabulary rows 18 tokens take 60.9 us instead of 63.5, 64 61.4
// instead of 63.8, 160 63.4 instead of 66.1, 256 68.5 instead of 71.4 (their logits
// 74.3 instead of 76.5); on four times as many rows 222.5 / 223 / 228 / 245.5 us
// instead of 226.5 / 227 / 229 / 249.5. With several token tiles the tensor cores
// set the pace, and two vocabulary tiles per token slab feed them with less.
template <bool kWriteLogits>
int launch_lmhead(const void* hidden, const void* weight, int H, int T, const VerifyParams& p, float* logits_out,
                  cudaStream_t stream) {
  LmDevice* dev = nullptr;
  const int rc = lm_device(&dev);
  if (rc != ASD_OK) return rc;
  if (T > kMaxTN || (kWriteLogits && lm_logits_in_two_tiles(p.V, dev->sms / 2)))
    return launch_lmhead_kernel<kWriteLogits, kEpiWarps, 2>(dev, hidden, weight, H, T, p, logits_out, stream);
  constexpr int kEpi = kWriteLogits ? kEpiWarps : kEpiWarpsOneTile;
  return launch_lmhead_kernel<kWriteLogits, kEpi, 1>(dev, hidden, weight, H, T, p, logits_out, stream);
}

// Verify or partials of p.B requests, in as many launches as their rows need.
int verify_lmhead(const void* hidden, const void* weight, int H, const VerifyParams& p, cudaStream_t stream) {
  const int K1 = p.K + 1, most = lm_rows_per_launch(p.V) / K1;
  for (long long b = 0; b < p.B; b += most) {
    const long long row = b * K1;
    VerifyParams c = p;
    c.B = static_cast<int>(p.B - b < most ? p.B - b : most);
    c.draft = p.draft + b * p.K;
    c.row_key = p.row_key + row;
    c.draft_logit = p.draft_logit + row;
    c.done = p.done + b;
    c.flags = p.flags + b;
    if (p.partials) {
      c.partials = p.partials + row;
    } else {
      c.ledger = p.ledger + b;
      c.accepted_len = p.accepted_len + b;
      c.committed = p.committed + row;
      c.recovery = p.recovery + b;
      if (p.row_argmax) c.row_argmax = p.row_argmax + row;
      if (p.row_regret) c.row_regret = p.row_regret + b * p.K;
      if (p.row_top) c.row_top = p.row_top + row;
      if (p.status) c.status = p.status + b;
    }
    const int rc = launch_lmhead<false>(static_cast<const char*>(hidden) + 2 * row * H, weight, H, c.B * K1, c, nullptr,
                                        stream);
    if (rc != ASD_OK) return rc;
  }
  return ASD_OK;
}

int check_lm_inputs(const void* hidden, const void* weight, int H) {
  if (!hidden || !weight) return ASD_ERR_NULL;
  if (H < 8 || H % 8 != 0) return ASD_ERR_SHAPE;  // TMA: row pitch a multiple of 16 bytes
  if (reinterpret_cast<uintptr_t>(hidden) % 16 != 0 || reinterpret_cast<uintptr_t>(weight) % 16 != 0)
    return ASD_ERR_ALIGN;
  return ASD_OK;
}

}  // namespace

extern "C" {

int asd_lmhead_workspace_size(int B, int K, int V, int H, size_t* bytes) {
  if (!bytes) return ASD_ERR_NULL;
  int rc = check_shape(B, K, V, ASD_BF16);
  if (rc != ASD_OK) return rc;
  if (H < 8 || H % 8 != 0) return ASD_ERR_SHAPE;
  *bytes = layout_for(B, K).total;
  return ASD_OK;
}

int asd_lmhead_verify(const void* hidden, const void* weight, int H, int B, int K, int V, const int32_t* draft,
                      asd_ledger* ledger, float gate, int cap, int32_t* accepted_len, int32_t* committed,
                      int32_t* recovery, int32_t* row_argmax, float* row_regret, float* row_top, int32_t* status,
                      void* workspace, size_t workspace_bytes, asd_stream_t stream) {
  int rc = check_shape(B, K, V, ASD_BF16);
  if (rc != ASD_OK) return rc;
  if (B == 0) return ASD_OK;
  rc = check_lm_inputs(hidden, weight, H);
  if (rc != ASD_OK) return rc;
  if (!accepted_len || !committed || !recovery || !workspace || !ledger) return ASD_ERR_NULL;
  if (K > 0 && !draft) return ASD_ERR_NULL;
  if (gate != gate || gate < 0.0f || cap < 0) return ASD_ERR_CONTROL;
  const WorkspaceLayout l = layout_for(B, K);
  if (workspace_bytes < l.total) return ASD_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % 16 != 0) return ASD_ERR_ALIGN;
  char* ws = static_cast<char*>(workspace);
  VerifyParams p = {};
  p.logits = nullptr;
  p.B = B;
  p.K = K;
  p.V = V;
  p.total = static_cast<long long>(B) * (K + 1);
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
  p.row_key = reinterpret_cast<unsigned long long*>(ws + l.row_key);
  p.draft_logit = reinterpret_cast<float*>(ws + l.draft_logit);
  p.done = reinterpret_cast<unsigned long long*>(ws + l.done);
  p.flags = reinterpret_cast<unsigned int*>(ws + l.flags);
  p.error = reinterpret_cast<unsigned int*>(ws + l.error);
  p.row_top = row_top;
  p.nblk = 1;
  return verify_lmhead(hidden, weight, H, p, reinterpret_cast<cudaStream_t>(stream));
}

int asd_lmhead_partials(const void* hidden, const void* weight, int H, int B, int K, int Vs, int v_offset,
                        int V, const int32_t* draft, asd_partial* partials, void* workspace,
                        size_t workspace_bytes, asd_stream_t stream) {
  int rc = check_shape(B, K, Vs, ASD_BF16);
  if (rc != ASD_OK) return rc;
  if (v_offset < 0 || V < 1 || static_cast<long long>(v_offset) + Vs > V) return ASD_ERR_SHAPE;
  if (B == 0) return ASD_OK;
  rc = check_lm_inputs(hidden, weight, H);
  if (rc != ASD_OK) return rc;
  if (!partials || !workspace) return ASD_ERR_NULL;
  if (K > 0 && !draft) return ASD_ERR_NULL;
  const WorkspaceLayout l = layout_for(B, K);
  if (workspace_bytes < l.total) return ASD_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % 16 != 0) return ASD_ERR_ALIGN;
  char* ws = static_cast<char*>(workspace);
  VerifyParams p = {};
  p.logits = nullptr;
  p.B = B;
  p.K = K;
  p.V = Vs;
  p.total = static_cast<long long>(B) * (K + 1);
  p.draft = draft;
  p.row_key = reinterpret_cast<unsigned long long*>(ws + l.row_key);
  p.draft_logit = reinterpret_cast<float*>(ws + l.draft_logit);
  p.done = reinterpret_cast<unsigned long long*>(ws + l.done);
  p.flags = reinterpret_cast<unsigned int*>(ws + l.flags);
  p.error = reinterpret_cast<unsigned int*>(ws + l.error);
  p.nblk = 1;
  p.v_offset = v_offset;
  p.v_total = V;
  p.partials = partials;
  return verify_lmhead(hidden, weight, H, p, reinterpret_cast<cudaStream_t>(stream));
}

int asd_lmhead_logits(const void* hidden, const void* weight, int H, int T, int V, float* logits,
                      asd_stream_t stream) {
  if (T < 0 || V < 1) return ASD_ERR_SHAPE;
  if (T == 0) return ASD_OK;
  int rc = check_lm_inputs(hidden, weight, H);
  if (rc != ASD_OK) return rc;
  if (!logits) return ASD_ERR_NULL;
  VerifyParams p = {};
  p.V = V;
  p.K = 0;
  p.nblk = 1;
  const int most = lm_rows_per_launch(V);
  for (long long t = 0; t < T; t += most) {
    rc = launch_lmhead<true>(static_cast<const char*>(hidden) + 2 * t * H, weight, H,
                             static_cast<int>(T - t < most ? T - t : most), p, logits + t * V,
                             reinterpret_cast<cudaStream_t>(stream));
    if (rc != ASD_OK) return rc;
  }
  return ASD_OK;
}

}  // extern "C"
