// lbm_plan.h -- host-side plans of the kernels that march several steps along
// strips (lbm_plan.cu).
#pragma once

#include <vector>

#include "lbm_internal.h"

namespace lbm {

struct StripPlan {
    std::vector<int4> items;       // strips (PairArgs::items)
    std::vector<int> block_first;  // grid + 1 entries
    int grid = 0;
    int warps = 0;                 // of a block (plan_pairs)
    int longest = 0;               // cost of the block that takes longest
    int time = 0;                  // the longest block's time (kPairTime)
    double work = 0;
    bool worth = false;            // faster than single steps (plan_pairs)
    bool worth_keep = false;       // also with every state stored (plan_pairs)
};

// A block shape of the two-step kernel, how many of its blocks are resident at
// once and on how many SMs.
struct PairShape {
    int warps, resident, sms;
};
// tiles: the lattice's 128-node tiles in row order; bc: 2 ny port entries;
// rescale: it has ports of the rescaling kinds; shapes: the usual one first, then
// the one of fewer warps; single_warps: of the single step's grid.
StripPlan plan_pairs(const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int nx, int ny, int pitch,
                     int precision, bool rescale, const PairShape* shapes, int n_shapes, long long single_warps);
// levels: steps a launch; warps of a block; resident: blocks in one wave.
StripPlan plan_scalar(const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int nx, int ny, int pitch, int levels,
                      int warps, int resident);

}  // namespace lbm
