// Sizes of the persistent stage kernel's work items (host code).
#pragma once

#include <cstdint>

namespace hrm {

// Cells per item of the per-cell phases for `blocks` resident blocks: `most`, or as
// many fewer as leave every block two items, so that none runs a long item while
// others have none (a multiple of 128, a block takes 128 cells at a time). A given
// launch shape sets `most`, so the tuner's candidates, and the default of 4096 set
// again, are never shapes that starve a small batch. With 4096 cells always, 24
// instances of 6000 cells kept 48 of 912 blocks busy; with this rule and the
// midpoint phase's lists a stage launch over them takes 0.24 ms against 0.65, and
// over 8 FP64 instances of 3000 cells 0.30 against 0.79; 64 instances of 11.35 M
// cells 10.2 ms per FP32 step against 12.8 and 78.1 per FP64 step against 115.
inline int64_t cell_tile(int64_t most, int64_t cells, int64_t blocks) {
  const int64_t fair = (cells / (2 * blocks) + 127) / 128 * 128;
  const int64_t t = fair < 128 ? 128 : fair;
  return t < most ? t : most;
}

}  // namespace hrm
