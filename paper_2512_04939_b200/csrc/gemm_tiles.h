// Which tiles a matrix product takes: host arithmetic on its sizes.
#pragma once

#include <initializer_list>

namespace lv {

constexpr int kGemmBM = 128;  // rows of a CTA

// What a launch costs, in units of what one column of a tile costs per k-block, times k: every wave of pairs pays
// about 150 columns' worth for the 128 rows of A that each CTA loads, a wave of single CTAs 205, whose B is not
// shared; a pair about 111 x 1024 more, once, for its cluster-wide hand-overs.  (us at k = 1024, one wave / every
// further one: a pair at 256 columns 11.3 / 5.3, 192: 9.8 / 4.6, 128: 8.0 / 3.75, 64: 7.6 / 2.8; one CTA at 256
// columns 10.6 / 6.2, of which the formula gives 6.0 so that two waves of either, equal within 2 %, stay with
// single CTAs.)  Where finer rows save one wave of many, pairs are still ahead: 52,050 x 1024 x 1024, 11 waves of
// single CTAs 106 us, 12 of pairs 96; 12,850 x 4096 x 1024, 11 and 12 waves, 95 and 87.
inline long long gemm_cost(long long waves, int bn, long long k, bool pair) {
  return pair ? waves * (150 + bn) * k + 90 * 1024 : waves * (205 + bn) * k - 21 * 1024;
}

// Whether a pair's tile may end in half a chunk of 64 columns (224, 160), whose rows leave the epilogue as 64-byte pieces of their
// own.  They fill a last wave of few better.  Of many waves the last counts less than the formula has it, and at short k
// the epilogue shows.  Measured over 512 to 4096 columns and k (us, with multiples of 64 / with these, the chip warm):
//   k = 512:  5,601 x 2048 13.8 / 15.3, 12,545 x 1536 21.2 / 22.0, 3,553 x 1536 9.8 / 9.9; ahead by 2 % at most
//   k = 1024: up to five waves 3,809 x 4096 27.7 / 26.5, 6,273 x 3072 33.8 / 32.8, 15,073 x 1024 26.9 / 26.1 (9,473 x 1024 20.2 / 20.5;
//             below the power cap the longer ones are the same or 2 % behind); twelve and thirteen 17,153 x 3072 91.7 / 97.3
//   k = 1536: 12,545 x 1536 51.4 / 48.5; thirteen waves 17,153 x 3072 127 / 129
//   k = 4096: five waves 6,273 x 3072 131 / 118, thirteen 34,561 x 1536 344 / 332
inline bool half_chunks_pay(long long k, long long waves) { return k >= 2048 || (k >= 768 && waves <= 5); }

// Columns of a pair's tile, or 0: CTAs of their own, 256 columns.  Narrower tiles win where wider ones
// would leave pairs idle in the only or the last wave, CTAs of their own where 128 rows a block save a wave,
// and below k = 512 (104,100 rows x 128 x 320: 36 us, a pair 50).  Of the multiples of 32 that a pair's tile can have, 224 and
// 160 cut 1024 columns into five and seven (3,360 rows x 1024 x 4096 then make one wave of 70 tiles where they
// made 56: 25.2 -> 23.2 us).  `heads`: a tile holds whole heads of 64 columns, of which the epilogue takes a statistic.
inline int gemm_tile_columns(long long m, long long n, long long k, bool heads, int num_sms) {
  if (k < 512) return 0;
  auto waves = [&](int rows, int bn, int groups) {
    return (((m + rows - 1) / rows) * ((n + bn - 1) / bn) + groups - 1) / groups;
  };
  int best = 0;
  long long best_cost = gemm_cost(waves(kGemmBM, 256, num_sms), 256, k, false);
  for (const int bn : {256, 224, 192, 160, 128, 64}) {  // (a pair's tile has a multiple of 32)
    const long long w = waves(2 * kGemmBM, bn, num_sms / 2), cost = gemm_cost(w, bn, k, true);
    if (bn % 64 != 0 && (heads || !half_chunks_pay(k, w))) continue;
    if (cost < best_cost) {
      best = bn;
      best_cost = cost;
    }
  }
  return best;
}

}  // namespace lv
