// How the attention takes a sequence apart, as far as the host side plans with it: the sizes at which its forms change,
// and the slabs of query rows in which a layer may leave for host memory.
#pragma once

namespace lv {

constexpr int kFaTileKeys = 128;  // keys of a K/V tile, two steps
#ifndef LV_FA_CHUNK_TILES
#define LV_FA_CHUNK_TILES 512
#endif
constexpr int kFaChunkTiles = LV_FA_CHUNK_TILES;  // 65536 keys: K and V of one head = 16 MiB
// Sequences of at most this many rows take CTAs of one query tile, two to an SM (figures in attention.cu).
#ifndef LV_FA_ONE_TILE_ROWS
#define LV_FA_ONE_TILE_ROWS 4096
#endif
constexpr long long kFaOneTileRows = LV_FA_ONE_TILE_ROWS;

// one counter per launch of an attention core: the key chunks of at most 4 Mi keys, or the slabs of one chunk
constexpr int kAttnCounters = 64;

// Query rows of so many rounds of CTAs, in whole query blocks of every head.
inline long long attention_rounds_rows(int num_sms, int heads, int rounds) { return (long long)rounds * num_sms / heads * 256; }

// Where the slab ends that starts at row0: after one round, so that the first rows are soon there, then two at a time.
// m at once for a sequence that is not to be taken apart: a short one, one of several key chunks, or one on so few SMs
// that a round is no whole query block or the slabs are more than the counters.
inline long long attention_slab_end(long long m, long long row0, int num_sms, int heads) {
  const long long first = attention_rounds_rows(num_sms, heads, 1), others = attention_rounds_rows(num_sms, heads, 2);
  if (m <= kFaOneTileRows || (m + kFaTileKeys - 1) / kFaTileKeys > kFaChunkTiles) return m;
  if (first == 0 || m > first + (kAttnCounters - 1) * others) return m;
  const long long end = row0 + (row0 == 0 ? first : others);
  return end < m ? end : m;
}
// Whether a layer of n tokens is sooner in host memory in slabs: the attention that is left behind the first slab, in proportion
// to (m - first) m, has to hide what is slower about it, in proportion to n (the writers at 45 GB/s, a copy at 55).
// Calls and drains in a row, ms in slabs / by a copy, by (m - first) m / n: 949 (7 frames of 37 x 37, 4,386 rows) 0.61 /
// 0.57, 1066 0.58 / 0.54, 1149 0.68 / 0.67 (on another machine 0.64 / 0.67), 1405 0.46 / 0.44 (0.45 / 0.45), 1457 0.41 /
// 0.42, 1753 0.44 / 0.48, 1538 0.78 / 0.84, 1818 0.29 / 0.34, 10538 (15,932 rows) 2.30 / 2.83.
inline bool attention_slabs_pay(long long m, long long n, int num_sms, int heads) {
  const long long first = attention_slab_end(m, 0, num_sms, heads);
  return first < m && (m - first) * m >= 1400 * n;
}
// The slab's number.
inline int attention_slab_index(long long row0, int num_sms, int heads) {
  if (row0 == 0) return 0;
  return 1 + (int)((row0 - attention_rounds_rows(num_sms, heads, 1)) / attention_rounds_rows(num_sms, heads, 2));
}

}  // namespace lv
