// Rules of launch shapes that hold over all sizes an instance may have, as
// plain host functions (no CUDA), so that they can be checked without a GPU.
#pragma once

#include <stdint.h>

#include <mutex>
#include <set>

namespace mg {

// Blocks of a kernel without a loop over its rows: every row has its place,
// whatever their number.  (A grid's x extent goes to 2^31 - 1; 2^31 rows in
// blocks of 32 rows are 2^26 blocks.)
inline int blocks_covering(int64_t rows, int rows_per_block) {
  const int64_t b = (rows + rows_per_block - 1) / rows_per_block;
  return (int)(b < 1 ? 1 : b);
}

// Block partials that each of a handle's reductions has room for, and the blocks
// of a kernel that leaves one each: at most one resident wave of them, and never
// more than there is room for, whatever the part's number of SMs.
constexpr int kPartials = 4096;
inline int partial_blocks(int64_t blocks, int64_t resident) {
  int64_t b = blocks < resident ? blocks : resident;
  if (b > kPartials) b = kPartials;
  return (int)(b < 1 ? 1 : b);
}

// A setting that the runtime keeps per device (a kernel's shared-memory limit,
// for one) and that is made once: `f` runs for each device until it has
// succeeded there (a status >= 0), one thread at a time.
class OncePerDevice {
  std::mutex mu;
  std::set<int> made;

 public:
  template <class F>
  int operator()(int device, F f) {
    std::lock_guard<std::mutex> lock(mu);
    if (made.count(device)) return 0;
    const int status = f();
    if (status >= 0) made.insert(device);
    return status;
  }
};

}  // namespace mg
