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
// The slab's number.
inline int attention_slab_index(long long row0, int num_sms, int heads) {
  if (row0 == 0) return 0;
  return 1 + (int)((row0 - attention_rounds_rows(num_sms, heads, 1)) / attention_rounds_rows(num_sms, heads, 2));
}

}  // namespace lv
