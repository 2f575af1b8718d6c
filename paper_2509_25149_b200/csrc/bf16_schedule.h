// Which column tiles of a BF16 launch are 512 wide (host code; the kernel is gemm_bf16.cuh).  Plain C++ without CUDA.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "tile_memo.h"

namespace nvfp4 {

// What the estimate sees of a product.  Products that agree in it get the same tiles, whatever their ragged edges.
struct Bf16Walk {
  int rows, cols, k_blocks;  // tiles of 256 rows and of 256 columns, k-blocks of 64
  int a_rows, b_rows;        // bf16_on_sector() of the operands
};
struct Bf16Wide {
  int n[2];  // column tiles 512 wide of each product of the launch
};

// Of two neighbouring rows of an operand, ld elements apart, those that begin on 32 bytes.  (Judged by ld alone, slices that begin 16
// bytes behind such a boundary kept 256 columns: 4096 x 4096 x 4096 with rows 8256 bytes apart 188.7 us, now 152.4, 8192 x 2048 x
// 1024 48.0, now 41.2.)
inline int bf16_on_sector(uint64_t base, int64_t ld) { return ld % 16 != 0 ? 1 : base % 32 == 0 ? 2 : 0; }

inline Bf16Walk bf16_walk(int64_t M, int64_t N, int64_t K, uint64_t a, int64_t lda, uint64_t b, int64_t ldb) {
  return Bf16Walk{(int)((M + 255) / 256), (int)((N + 255) / 256), (int)((K + 63) / 64), bf16_on_sector(a, lda), bf16_on_sector(b, ldb)};
}

// Estimated SM cycles of a launch of one or two products on `pairs` CTA pairs.
class Bf16Estimate {
 public:
  Bf16Estimate(const Bf16Walk* w, int n, int pairs) : w_(w), n_(n), pairs_(pairs) {
    for (int i = 0; i < n; ++i)
      for (int halves = 1; halves <= 2; ++halves) {
        auto bytes = [](int on_sector) { return 16384.0 * (1.75 - 0.375 * on_sector); };
        const double k_block = std::max(halves * 530.0, (bytes(w[i].a_rows) + halves * bytes(w[i].b_rows)) / 63.0);
        cost_[halves - 1][i] = std::llround(k_block * w[i].k_blocks) + (halves == 2 ? 3000 : 500);
        if (halves == 1) beside_[i] = n > 1 ? std::llround(1.04 * k_block * w[i].k_blocks) + 500 : cost_[0][i];
      }
  }
  // No schedule with these wide tiles (some) ends before this: the work in equal shares.
  int64_t least(const Bf16Wide& wide) const {
    int64_t sum = 0;
    for (int i = 0; i < n_; ++i)
      sum += w_[i].rows * (wide.n[i] * cost_[1][i] + (w_[i].cols - 2 * wide.n[i]) * beside_[i]);
    return sum / pairs_;
  }
  // Until the last pair has stored its last tile: the tiles 512 wide of both products, then those 256 wide, in rounds of the pairs
  // (odd ones in reverse order where there are wide tiles).  A pair has floor(e / pairs) of the first e tiles, and one more where its
  // place in the next round lies below e % pairs, so what the pairs have to do differs at four places of their order at most.
  int64_t until_the_last(const Bf16Wide& wide) const {
    const bool snake = wide.n[0] + wide.n[1] > 0;
    struct Segment {
      int64_t rounds, rest, cost;
      bool back;  // the round that it ends in runs backwards
    } seg[4];
    int64_t t = 0, wide_end = 0;
    int segs = 0;
    for (int k = 0; k < 4; ++k) {
      if ((k & 1) >= n_) continue;
      const Bf16Walk& g = w_[k & 1];
      t += (int64_t)g.rows * (k < 2 ? wide.n[k & 1] : g.cols - 2 * wide.n[k & 1]);
      seg[segs++] = Segment{t / pairs_, t % pairs_, k < 2 ? cost_[1][k & 1] : snake ? beside_[k & 1] : cost_[0][k & 1],
                            snake && (t / pairs_ & 1)};
      if (k < 2) wide_end = t;
    }
    auto time_of = [&](int64_t p) {
      int64_t done = 0, load = 0;
      for (int s = 0; s < segs; ++s) {
        const int64_t tiles = seg[s].rounds + ((seg[s].back ? pairs_ - 1 - p : p) < seg[s].rest ? 1 : 0);
        load += (tiles - done) * seg[s].cost;
        done = tiles;
      }
      const int64_t rnd = done - 1, last = rnd * pairs_ + (snake && (rnd & 1) ? pairs_ - 1 - p : p);
      return load + (done > 0 && last < wide_end ? 3000 : 0);
    };
    int64_t worst = time_of(0);
    for (int s = 0; s < segs; ++s)
      if (seg[s].rest) worst = std::max(worst, time_of(seg[s].back ? pairs_ - seg[s].rest : seg[s].rest));
    return worst;
  }

 private:
  const Bf16Walk* w_;
  int n_, pairs_;
  int64_t cost_[2][2];  // a tile 256 or 512 wide, of product 0 or 1
  int64_t beside_[2];   // a tile 256 wide in a launch that has some of 512, with four stages for it instead of six
};

// Column tiles 512 wide of each product (the other columns in tiles of 256, behind them) whose schedule is estimated shortest;
// {0, 0}: 256-wide tiles everywhere.  A k-block of a tile takes as long as its MMAs (530 SM cycles per 256 columns) or as its
// loads: 63 bytes per clock, and 1.75 times as many for a 128-byte row of a box that does not begin on 32 bytes (narrow tiles, 4096 x
// 4096 x 4096: every row on 32 bytes 101 to 104 us, none 189).  Where the MMAs are longer, what 512 columns gain is fewer
// hand-overs and, with tiles of two sizes, shorter last rounds.  256 wide / chosen: forward of 4088 x 5128 x 5112 208 / 179 us,
// backward 414 / 330, forward of 2048 x 7168 x 2056 68 / 55, backward of 3000 x 3000 x 1000 45.2 / 39.6; rows 128 bytes apart: backward
// of 4096 x 2048 x 1024 38.5 / 27.1.  A hand-over of two accumulators takes 3000 cycles and a pair whose last tile is such a one 3000
// more, its halves leaving one after the other: with half of that forward of 1040 x 3664 x 904 came out at 14.8 / 15.6, 1384 x 3624 x
// 928 at 14.8 / 15.4.  Contractions of fewer than 14 k-blocks keep 256 columns (1112 x 3672 x 552 11.5 / 12.7, 2344 x 1856 x 264 9.2 /
// 10.3).
// A schedule with wide tiles has to be estimated 3 % shorter, and the 256-wide tiles beside them, which have four stages instead of
// six, count 4 % more per k-block where two products (with transposed operands) share the launch.  Fitted to 3306 drawn calls
// (forward, backward, accumulating), each timed with 256-wide tiles, with the chosen and with two other numbers of wide ones: the
// geometric mean of what the choice gains is 1.055, and 2 % of the calls are more than 3 % slower than with 256 columns.  (With rows
// priced by where they lie in 64 bytes, 1.25 times the bytes for odd multiples of 32, 2 % and no surcharge: 1.052, and 8 %.)
// A call pays for the search where its shape is new: at most 289 schedules, and only those that could be the shortest are walked
// through.  *walked (may be NULL): how many.
inline Bf16Wide bf16_wide_search(const Bf16Walk* w, int n, int pairs, int* walked = nullptr) {
  Bf16Wide best{{0, 0}};
  int most[2] = {0, 0}, count = 0;
  for (int i = 0; i < n; ++i)
    if (w[i].k_blocks >= 14) most[i] = std::min(w[i].cols / 2, 0x7fff);
  if (most[0] + most[1] > 0) {
    const Bf16Estimate estimate(w, n, pairs);
    int64_t least = (int64_t)(0.97 * (double)estimate.until_the_last(best));
    ++count;
    const int step[2] = {1 + most[0] / (n > 1 ? 16 : 64), 1 + most[1] / 16};  // (at most 65, or 17 x 17 of them)
    for (int i = most[0] % step[0]; i <= most[0]; i += step[0])
      for (int j = most[1] % step[1]; j <= most[1]; j += step[1]) {
        const Bf16Wide wide{{i, j}};
        if (i + j == 0 || estimate.least(wide) >= least) continue;
        const int64_t v = estimate.until_the_last(wide);
        ++count;
        if (v < least) {
          least = v;
          best = wide;
        }
      }
  }
  if (walked) *walked = count;
  return best;
}

// The same, remembered.
inline Bf16Wide bf16_wide_tiles(const Bf16Walk* w, int n, int pairs, int* walked = nullptr) {
  static TileMemo memo;
  int key[TileMemo::kKey] = {0, 0, 0, 0, 0, 0, 0, pairs}, both = 0;
  for (int i = 0; i < n; ++i) {
    key[3 * i] = w[i].rows;
    key[3 * i + 1] = w[i].cols;
    key[3 * i + 2] = w[i].k_blocks;
    key[6] |= (w[i].a_rows << 2 | w[i].b_rows) << (4 * i);
  }
  if (walked) *walked = 0;
  if (!memo.find(key, &both)) {
    const Bf16Wide wide = bf16_wide_search(w, n, pairs, walked);
    both = wide.n[0] | wide.n[1] << 16;
    memo.put(key, both);
  }
  return Bf16Wide{{both & 0xffff, both >> 16}};
}

}  // namespace nvfp4
