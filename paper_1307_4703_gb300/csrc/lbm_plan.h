// lbm_plan.h -- host-side plan of the two-step kernel (lbm_plan.cu).
#pragma once

#include <vector>

#include "lbm_internal.h"

namespace lbm {

struct PairPlan {
    std::vector<int4> items;       // strips (PairArgs::items)
    std::vector<int> block_first;  // grid + 1 entries
    int grid = 0;
    bool worth = false;            // faster than two single steps
};

// tiles: the lattice's 128-node tiles in row order; bc: 2 ny port entries;
// warps: of a block; resident: blocks in one wave.
PairPlan plan_pairs(const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int nx, int ny, int pitch,
                    int precision, int warps, int resident);

}  // namespace lbm
