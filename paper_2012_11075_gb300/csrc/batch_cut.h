// The rule that chooses a batch's cut (host arithmetic only).
#pragma once

#include <limits>

namespace wblbe {

// Rows per tile for the running cases: the configured ones, halved (down to
// 8) while that leaves fewer than 1.3 tiles per resident CTA and the tile
// table (max_tiles) holds the finer cut.  With fewer, CTAs idle while the
// longest tile of each step marches its rows: a tile's row takes about 0.7 us
// whatever runs beside it.  With more, the next step's tiles already fill the
// CTAs that finish early, and halving only adds halo rows (4 per tile).  us per
// step before and after halving, by tiles per resident CTA before it:
//   FP32 0.67 53 and 37, 0.78 100 and 78, 0.85 32 and 25, 0.99 191 and 144,
//        1.16 121 and 107, 1.20 114 and 114, 1.36 37 and 41, 1.40 30 and 38,
//        1.40 141 and 150, 1.51 143 and 152, 1.58 73 and 76, 1.70 303 and 297;
//   FP64 0.76 453 and 420, 0.99 2615 and 1837, 1.40 341 and 353, 1.50 1475 and
//        1456, 1.55 420 and 445, 1.70 1845 and 1856.
// Results do not depend on the cut.  total(rows): tiles of the running cases
// when cut at `rows`.  A launch of `steps` steps numbers its work items, and
// each resident CTA's last claim past them, in an int: a finer cut has to keep
// to that as well.
template <typename Total>
int cut_rows(int rows, long long resident, long long max_tiles, long long steps, Total total) {
  const long long most = std::numeric_limits<int>::max() - resident;
  while (rows >= 16 && 10 * total(rows) < 13 * resident && total(rows / 2) <= max_tiles &&
         total(rows / 2) <= most / steps)
    rows /= 2;
  return rows;
}

}  // namespace wblbe
