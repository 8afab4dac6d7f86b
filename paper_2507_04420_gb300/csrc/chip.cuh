// chip.cuh -- launchers of chip.cu: graphs whose states fit in one SM.
#pragma once
#include "internal.h"

namespace skp {

// Rows + entries up to which one SM is the faster place: above, it issues
// instructions for longer than the whole GPU waits on L2.  Calls, in us, on the
// chip / in the sweep: 2 K items 29-37 / 47-60, 8 K 30-41 / 47-58, 34 K 55 / 59,
// a grid of 39 K 93 / 91, 79 K 146 / 97.  Rows cost a block more than entries, as
// each window of 32 waits for its row ends: 8000 rows without entries 27 / 28, with
// one each 61 / 58, as a path 59 / 57; 16,000 rows 32 / 28 and 98 / 58.
constexpr uint64_t kChipSingleItems = 32768, kChipSingleRows = 8192;
// the whole pass over one graph of at most that size: no prepare launch before
// it
cudaError_t launch_chip_single(const SweepParams& P, int bits, cudaStream_t s);

}  // namespace skp
