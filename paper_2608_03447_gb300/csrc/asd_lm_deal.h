// How the fused LM head cuts token and vocabulary rows into items and deals them
// to the CTA pairs: plain host arithmetic.
#pragma once

namespace asd_detail {

constexpr int kPairM = 256;  // vocabulary rows per CTA pair in one MMA (MMA M)
constexpr int kMaxTN = 256;  // most token rows per tile (MMA N; a multiple of 32)

struct LmDeal {
  int tn;           // token rows per tile
  int token_tiles;  // ceil(T / tn)
  // Items 0 .. full - 1: item i is vocabulary rows (i / token_tiles) * kw * kPairM on by token tile i % token_tiles.
  // When the last round of the deal would leave more than half of the pairs idle, its items are dealt in
  // halves (one vocabulary tile each): entries full + 2 h and full + 2 h + 1 are the tiles of item full + h.
  int full, entries;
};

// Vocabulary units of kw tiles.
inline int lm_units(int V, int kw) { return 1 + (V - 1) / (kw * kPairM); }

// The most token rows of one launch: the kernel counts items in 32 bits, and the
// largest vocabularies and batches have more (V = 2^31 - 1 with 2^17 rows: 2^31).
// A call with more rows takes several launches, of at least 65536 rows each.
#ifndef ASD_LM_MAX_ITEMS
#define ASD_LM_MAX_ITEMS (1 << 30)  // tests of the split lower it
#endif
inline int lm_rows_per_launch(int V) {
  const int tiles = ASD_LM_MAX_ITEMS / lm_units(V, 2);
  return (tiles > 1 ? tiles < (1 << 22) ? tiles : 1 << 22 : 1) * kMaxTN;
}

// How T token rows and V vocabulary rows are cut and dealt to `pairs` CTA pairs.
//
// Token tiles: as few as hold T at up to 256 columns (each tile reads W once
// more from L2, and a wider MMA reads its vocabulary operand from shared memory
// less often per product), all of one width, rounded up to the 32 columns of an
// epilogue block. Against a fixed width of 192: 320 rows took 384 columns and
// take 2 x 160, 18 rows take 32, 2304 rows take 9 tiles instead of 12.
//
// The last round of the deal: `left` items for more pairs. Up to half of the
// pairs' number, half items keep twice as many pairs busy for half the time;
// beyond that, halves would only begin a second round.
//
// Few units: where all items go in one round but leave pairs idle, one tile more
// makes them narrower and is still one round. Taken for tiles of 224 and 256
// columns, of which tensor memory holds two: 477 rows on 12509 vocabulary rows
// 58.9 -> 43.6 us (their logits 55.1 -> 41.9), 600 on 9717 53.7 -> 43.1 (49.6 ->
// 40.6); narrower tiles gain nothing (300 on 12509 41.5 -> 40.4, H = 3000 30.9 -> 32.4).
inline LmDeal lm_deal(int T, int V, int kw, int pairs) {
  const int units = lm_units(V, kw);
  LmDeal d;
  int items = 0;
  const auto cut = [&](int token_tiles) {
    d.token_tiles = token_tiles;
    const int per = 1 + (T - 1) / token_tiles;
    d.tn = (per + 31) / 32 * 32;
    items = units * token_tiles;
  };
  cut(1 + (T - 1) / kMaxTN);
  if (kw == 2 && d.tn > 192 && items + units <= pairs && 2 * items > pairs) cut(d.token_tiles + 1);
  const int left = items % pairs;
  const int halved = kw == 2 && 2 * left <= pairs ? left : 0;
  d.full = items - halved;
  d.entries = items + halved;
  return d;
}

// Logits of one token tile: items of two vocabulary tiles where items of one would
// begin a second round with few of them. On 19500 to 24000 vocabulary rows, H = 3000,
// 109 rows 31.8-37.2 -> 28.9-31.4 us, 250 rows 41.6-48.1 -> 37.9-40.9; a fuller second
// round gains nothing (32000 rows, H = 5120: 57.0 against 58.3), nor does the verify,
// which stores nothing (250 rows, H = 5120: 58.2 against 59.5 us).
inline bool lm_logits_in_two_tiles(int V, int pairs) {
  const int units = lm_units(V, 1);
  return units > pairs && units <= pairs + pairs / 4;
}

}  // namespace asd_detail
