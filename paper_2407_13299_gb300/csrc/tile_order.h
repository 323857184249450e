// The order in which a single-matrix product walks its output tiles. Host code
// only (no CUDA), so that a test can compile it on its own.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace dmp {

// Row and column block of a tile. A tall or wide product has more than 65536
// blocks (m > 16,777,216 rows of 256-row tiles): more than 16 bits hold.
struct TileAt {
  int32_t bi, bj;
};

// A tile in one 32-bit word, the column block in the low `bits` (TileOrder::
// column_bits); no two tiles of a product share a word. The table of a launch's
// tiles is part of the kernels' parameters, and 8 bytes per tile, which make these
// 3.3 KB instead of 2.7, cost every launch time: a product of n = 4096, INT8, s =
// 7, 2.15 ms against 2.06, and a batch, which does not read the table, 0.5 %.
constexpr uint32_t pack_tile(TileAt t, int bits) {
  return static_cast<uint32_t>(t.bi) << bits | static_cast<uint32_t>(t.bj);
}
constexpr TileAt unpack_tile(uint32_t w, int bits) {
  return {static_cast<int32_t>(w >> bits), static_cast<int32_t>(w & ((uint32_t{1} << bits) - 1))};
}

// The output tiles of an m x n product (tiles of bm x bn; sym: those that hold
// some element with row <= column): bands of column blocks, each cut into groups
// of row blocks, about as many tiles per group as run at once (`units`) and
// near-square in elements, so that the tiles in flight together share their
// operand panels in L2. Handed out one by one: no list is allocated.
class TileOrder {
 public:
  TileOrder(int64_t m, int64_t n, int bm, int bn, bool sym, int units)
      : bm_(bm), bn_(bn), sym_(sym), tm_((m + bm - 1) / bm), tn_((n + bn - 1) / bn) {
    const int64_t square = std::lround(std::sqrt(static_cast<double>(units) * bm / bn));
    w_ = std::max<int64_t>(1, std::min(square, tn_));
    h_ = std::max<int64_t>(1, units / w_);
  }

  int64_t count() const {
    if (!sym_) return tm_ * tn_;
    int64_t t = 0;
    for (int64_t c = 0; c < tn_; ++c) t += rows_of(c);
    return t;
  }

  // Bits of a column block, -1 if rows and columns together need more than 32 (an
  // output of over 2^32 tiles, or one of over 2^31 blocks in a row).
  int column_bits() const {
    const auto width = [](int64_t blocks) {
      int b = 0;
      while (b < 63 && (int64_t{1} << b) < blocks) ++b;
      return b;
    };
    const int c = width(tn_);
    return c < 32 && c + width(tm_) <= 32 ? c : -1;
  }

  // The next tile; at most count() calls.
  TileAt next() {
    while (r_ >= std::min(rows_of(c_), r0_ + h_)) {
      const int64_t c1 = std::min(tn_, c0_ + w_);
      if (++c_ == c1) {
        // past the group: the next one of the band, or the next band
        r0_ += h_;
        if (r0_ >= rows_of(c1 - 1)) {
          r0_ = 0;
          c0_ = c1;
        }
        c_ = c0_;
      }
      r_ = r0_;
    }
    return {static_cast<int32_t>(r_++), static_cast<int32_t>(c_)};
  }

 private:
  // row blocks of column block c that hold tiles
  int64_t rows_of(int64_t c) const { return sym_ ? std::min(tm_, (bn_ * (c + 1) + bm_ - 1) / bm_) : tm_; }

  int64_t bm_, bn_;
  bool sym_;
  int64_t tm_, tn_, w_, h_;
  int64_t c0_ = 0, r0_ = 0, c_ = 0, r_ = 0;  // band, group and the next tile
};

}  // namespace dmp
