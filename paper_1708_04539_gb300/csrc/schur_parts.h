// Parts of a factorisation level's Schur products and of their scatter (host
// only): part 1 holds the updates of a parent's diagonal block ("corner": rows
// and columns below `corner`), which the next level's LU waits for, part 2 the
// others, which run beside that LU on another stream; part 0 is both.
#pragma once
#include <cstdint>

namespace pselinv {

// tile of the sliced products' outputs (rows x columns), and of the scatter
// that subtracts them from the ancestors
constexpr int64_t kProductRows = 128, kProductCols = 64, kScatterTile = 32;

// whether the tile with origin (p0, q0) belongs to `part`
inline bool schur_in_part(int part, int64_t corner, int64_t p0, int64_t q0) {
  return part == 0 || (part == 1) == (p0 < corner && q0 < corner);
}

// The scatter tile (tp, tq) goes with the product tile that it reads, which is
// larger: the two parts run on two streams with nothing between them, so that a
// scatter tile past the corner inside a product tile of the corner has to stay
// with that tile.
inline bool scatter_in_part(int part, int64_t corner, int64_t tp, int64_t tq) {
  static_assert(kProductRows % kScatterTile == 0 && kProductCols % kScatterTile == 0,
                "a scatter tile lies within one product tile");
  return schur_in_part(part, corner, tp * kScatterTile / kProductRows * kProductRows,
                       tq * kScatterTile / kProductCols * kProductCols);
}

}  // namespace pselinv
