// Compiled tile shapes (threads per block x items per thread) of each operator.
// Section 3.3 sweeps block sizes 32..1024 and 1/2/4 items per thread and settles on
// 128 x 4 for its microbenchmarks and 256 x 8 for the full queries; the paper's
// 128 x 4 shape is kept as one variant of every scan operator next to wider tiles that
// suit bulk asynchronous copies on sm_103a.  Entry 0 is the default.  (Probe: 2^28 probes of
// tables of 16 KB, 64 MB and 2 GB take 0.476, 1.016 and 6.45 ms with 256 x 8, 0.559, 1.087
// and 6.47 with 256 x 16, the earlier default.  Plan: queries of one to four joins over 1M to
// 200M rows take 0.85 to 1.03 times as long with 512 x 8 as with 256 x 8, the fused date join
// over 2^28 rows 0.99.)
#pragma once

#include "crystal.h"

namespace crys {

struct TileShape {
  int threads;
  int items;
};

constexpr int kMaxVariants = 4;

constexpr TileShape kTiles[CRYS_NUM_OPS][kMaxVariants] = {
    /* SELECT      */ {{256, 16}, {128, 16}, {512, 8}, {128, 4}},
    /* PROJECT     */ {{256, 16}, {256, 8}, {512, 8}, {128, 4}},
    /* PROBE       */ {{256, 8}, {256, 16}, {512, 8}, {128, 4}},
    /* PLAN        */ {{512, 8}, {256, 8}, {512, 4}, {128, 4}},
    /* SHARED_SCAN */ {{256, 4}, {256, 8}, {128, 8}, {128, 4}},
    /* SORT        */ {{256, 32}, {256, 24}, {512, 16}, {256, 16}},
    /* TAGGED_SCAN */ {{1024, 4}, {256, 4}, {512, 4}, {256, 8}},
};

constexpr int kNumVariants[CRYS_NUM_OPS] = {4, 4, 4, 4, 4, 4, 4};

}  // namespace crys
