// lbm_plan.h -- host-side plans of the kernels that march several steps along
// strips (lbm_plan.cu).
#pragma once

#include <algorithm>
#include <atomic>
#include <new>
#include <system_error>
#include <thread>
#include <vector>

#include "lbm_internal.h"

namespace lbm {

// fn(0) .. fn(n - 1) on a host thread each; a part whose thread cannot be had is
// done here.  False: one ran out of memory.
template <typename Fn>
bool over_parts(int n, const Fn& fn)
{
    std::atomic<bool> ok{true};
    auto part = [&](int k) {
        try {
            fn(k);
        } catch (const std::bad_alloc&) {
            ok = false;
        }
    };
    std::vector<std::thread> threads;
    std::vector<int> here{0};
    threads.reserve(size_t(n));
    here.reserve(size_t(n));
    for (int k = 1; k < n; ++k) {
        try {
            threads.emplace_back(part, k);
        } catch (const std::system_error&) {
            here.push_back(k);
        }
    }
    for (int k : here) part(k);
    for (std::thread& t : threads) t.join();
    return ok;
}
// Parts for `work` units of which `each` are worth a thread.
inline int parts_for(long long work, long long each, long long most)
{
    return int(std::max(1ll, std::min({16ll, most, (long long)std::thread::hardware_concurrency(), work / each})));
}

struct StripPlan {
    std::vector<int4> items;       // strips (PairArgs::items)
    std::vector<int> block_first;  // grid + 1 entries
    int grid = 0;
    int warps = 0;                 // of a block (plan_pairs)
    int longest = 0;               // cost of the block that takes longest
    int time = 0;                  // the longest block's time (kPairTime)
    double work = 0;
    bool worth = false;            // faster than single steps
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
