// Rules of launch shapes that hold over all sizes an instance may have, as
// plain host functions (no CUDA), so that they can be checked without a GPU.
#pragma once

#include <stdint.h>

namespace mg {

// Blocks of a kernel without a loop over its rows: every row has its place,
// whatever their number.  (A grid's x extent goes to 2^31 - 1; 2^31 rows in
// blocks of 32 rows are 2^26 blocks.)
inline int blocks_covering(int64_t rows, int rows_per_block) {
  const int64_t b = (rows + rows_per_block - 1) / rows_per_block;
  return (int)(b < 1 ? 1 : b);
}

}  // namespace mg
