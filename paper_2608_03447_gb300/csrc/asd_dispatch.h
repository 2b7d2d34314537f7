// Which row-stage kernel of the logit-streaming path a call gets: plain host
// arithmetic on its sizes and on the device's SM count.
#pragma once

#include "asd.h"

namespace asd_detail {

// verify_small_kernel: a CTA's threads, and the 128-bit vectors per lane that one round of loads takes.
constexpr int kSmallThreads = 512;
constexpr int kSmallUnroll = 8;
constexpr long long kSmallCtaBytes = 16LL * kSmallThreads * kSmallUnroll;  // 64 KB: one round of loads
constexpr int kSmallMaxCluster = 8;                                        // the largest portable cluster

// The SMs of the GB300 that the lines below were measured on. Lines that stand
// for how much fills the GPU go with the SM count of the device at hand.
constexpr int kMeasuredSms = 152;

// Which kernel streams the logits.
//   kTma     resident inputs of more than kTmaMinBytes with long rows: a slice is
//            streamed ahead of the kernels before it, which a unit's CTA, that has
//            to wait for them when it ends, cannot (11.7-12.1 against 14.5 us per
//            step of 87.5 MB with 304 KB rows) once the units of one call fill the
//            GPU. Below that the next call's units find room beside them (with
//            64 KB rows 6.0 against 5.1 us at 20.6 MB, 6.2 against 6.7 at 21.8 MB;
//            with 80 KB rows 5.4 against 5.3 at 21.6 MB, 5.6 against 6.5 at 22.3
//            MB) unless the rows are few (20 of 517 KB: 3.0 against 3.5 us).
//            A slice pays for every row it enters, so the more rows there are, the
//            longer they have to be: with 64 KB rows 7.2 against 7.3 us at 27.6 MB
//            (432 rows) but 8.7 against 8.3 at 37.4 MB (585); with 88 KB rows 11.1
//            against 11.3 at 59 MB (657) but 14.3 against 13.8 at 80 MB (882); with
//            112 KB rows 13.4 against 13.8 at 80 MB and 16.2 against 16.5 at 99 MB
//            (864), but 19.2 against 19.1 at 120 MB (1044) and 25.1 against 24.5
//            at 160 MB; with 128 KB rows 23.7 against 24.3 at 160 MB (1215), 30.0
//            against 29.6 at 200 MB. One line for more than kTmaManyRows a slice,
//            at 112 KB: beyond 1000 rows it costs rows of 112 to 128 KB up to 3 %,
//            a line at 128 KB would cost them 2 to 18 % below that.
//   kSmall   a request fits one round of loads of a cluster (508 KB; 60 KB for
//            one CTA) and there are few enough: no hand-off to a selection, one
//            launch. With one CTA each 2.5 against 3.0 us (8 requests of 18 KB),
//            3.1 against 3.8 (152 of 18 KB), 4.9 against 5.0 us (128 of 54 KB);
//            beyond a CTA per SM 5.4 against 4.6 us (256 of 18 KB). A request of few
//            and short rows has a CTA of few warps (small_plan); below a megabyte as
//            many as fit the SMs at once: 3.2 against 3.9 us (1024 of 34 bytes), 3.2
//            against 4.0 (304 of 1.8 KB), but 5.4 against 4.4 us (400 of 1.8 KB, two
//            at a time on an SM) and 6.5 against 4.6 (4096 of 4 bytes). With a
//            cluster 3.6 against 3.7 us (16 of 144 KB), 3.2 both (2 of 320 KB),
//            and with resident inputs 1.5-1.7 against 2.4-2.7 us; half the launches,
//            which is what an eager call waits for (6.5 against 8.7 us). A GPU full
//            of clusters is slower: of two CTAs 2.6 against 2.8 us at 60 of 72 KB
//            but 3.4 against 2.9 at 76 (resident; 3.8 against 3.7 waiting), of four
//            2.8 both at 32 of 130 KB but 3.3 against 2.8 at 36, of eight 3.1 both
//            at 14 of 261 KB but 4.1 against 3.1 at 16, where they are no longer
//            resident at once. The line for all is a CTA per SM, for the launch
//            saved, up to 5 MB of clusters of four and eight (2.8 both at 14 of 360
//            KB, 5.0 MB, 4.4 against 2.8 at 16, 5.8 MB); with resident inputs, which
//            come in captured rounds, no more clusters of eight than fit at once.
//   kStream  everything else. A call that waits for the kernel ahead of it has
//            nothing to overlap and takes 14.8-15.1 us for 87.5 MB where the TMA
//            pipeline took 20.5 us, 91.7 against 100 us for 662 MB, 3.6 against
//            8.2 us for 2.7 MB, 7 against 26 us for 16 MB in 2 KB rows.
// With the selection inside the row stage (a launch option) the streaming kernel's
// CTAs each fence and count their units, the pipeline's a slice: 15.4 against 18.4 us
// at 43 MB, but 24.5 against 23.5 at 86 MB with 200 KB rows, 146 against 102 at 659 MB
// with 304 KB rows; with 64 KB rows 129 against 140 us.
// The launch options can force a kernel (the tests use that to cover every
// kernel); a forced `small` falls back to the default when the shape does not
// qualify.
constexpr long long kTmaMinBytes = 41LL << 19;           // 21.5 MB on kMeasuredSms
constexpr long long kTmaMinBytesFewRows = 1LL << 20;     // up to kTmaFewRows
constexpr long long kTmaFewRows = 64;
constexpr long long kTmaMinRowBytes = 64LL << 10;        // up to kTmaManyRows
constexpr long long kTmaMinRowBytesManyRows = 112LL << 10;
constexpr long long kTmaManyRows = 3;                    // a slice, of which there is one a SM
constexpr long long kFusedTmaMinBytes = 80LL * 1000 * 1000;
constexpr long long kFusedTmaMinRowBytes = 192LL << 10;
constexpr long long kSmallMaxBytes = 1LL << 20;         // below this as many one-CTA requests as fit at once
constexpr int kSmallWarpsPerSm = 22;                    // at 88 registers a thread
constexpr long long kSmallMaxClusterBytes = 5LL << 20;  // of clusters larger than two
constexpr int kSmallMaxLargestClusters = 14;            // resident inputs: at once on kMeasuredSms

enum class Path { kSmall, kStream, kTma };

// CTAs that take one request together: every lane's share in one round of loads
// (0: too large).
inline int small_cluster(long long request_bytes) {
  for (int ctas = 1; ctas <= kSmallMaxCluster; ctas *= 2)
    if (request_bytes <= ctas * kSmallCtaBytes - kSmallCtaBytes / (kSmallThreads / 32)) return ctas;
  return 0;
}

// How verify_small_kernel cuts a request: every row into `units`, cut every `per`
// vectors (a multiple of 32), for the CTAs' warps, one of which fetches the drafts'
// logits instead. A request's only CTA has no more warps than units: sixteen for
// every request let one CTA onto an SM at a time, and 256 requests of 34 bytes took
// 4.6 us instead of 2.7, 1024 of them 14.5 us instead of 3.2.
struct SmallPlan {
  int units;
  int per;
  int warps;  // per CTA
  int line;   // where in its 128-byte line the first vector of the logits lies
};
// nvec: whole vectors of a row, at most.
inline SmallPlan small_plan(int nvec, int K, int ctas) {
  SmallPlan q = {};
  q.warps = kSmallThreads / 32;
  const int warps = ctas * q.warps - 1;
  const int share = warps / (K + 1) > 0 ? warps / (K + 1) : 1;  // units of a row that start at once
  q.per = ((nvec + 7 + share - 1) / share + 31) / 32 * 32;
  if (q.per > 32 * kSmallUnroll) q.per = 32 * kSmallUnroll;
  q.units = nvec <= q.per ? 1 : (nvec + 7 + q.per - 1) / q.per;  // + 7: the first unit may begin inside a line
  if (ctas == 1 && (K + 1) * q.units + 1 < q.warps) q.warps = (K + 1) * q.units + 1;
  return q;
}

inline Path choose_path(int forced, long long bytes, long long request_bytes, int B, int K, bool single_block,
                        bool resident, bool fused, int sms) {
  const int ctas = single_block ? small_cluster(request_bytes) : 0;
  if (forced == ASD_PATH_TMA) return Path::kTma;
  if (forced == ASD_PATH_STREAM) return Path::kStream;
  if (forced == ASD_PATH_SMALL && ctas > 0) return Path::kSmall;
  if (ctas == 1) {
    const int warps = small_plan(static_cast<int>(request_bytes / (K + 1) / 16), K, 1).warps;
    if (B <= (bytes < kSmallMaxBytes ? kSmallWarpsPerSm / warps : 1) * static_cast<long long>(sms)) return Path::kSmall;
  }
  if (ctas > 1 && static_cast<long long>(B) * ctas <= sms && (ctas == 2 || bytes <= kSmallMaxClusterBytes) &&
      !(resident && ctas == kSmallMaxCluster && B > kSmallMaxLargestClusters * sms / kMeasuredSms))
    return Path::kSmall;
  const long long row_bytes = request_bytes / (K + 1), rows = bytes / row_bytes;
  if (resident && bytes >= (rows <= kTmaFewRows ? kTmaMinBytesFewRows : kTmaMinBytes * sms / kMeasuredSms) &&
      row_bytes >= (rows <= kTmaManyRows * sms ? kTmaMinRowBytes : kTmaMinRowBytesManyRows))
    return Path::kTma;
  if (fused && bytes >= kFusedTmaMinBytes && row_bytes >= kFusedTmaMinRowBytes) return Path::kTma;
  return Path::kStream;
}

}  // namespace asd_detail
