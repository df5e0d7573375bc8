// Host rules of the engine that need no device.
#pragma once

#include <vector>

namespace hot {

constexpr int kMaxGroup = 512;         // most CTAs of one instance in the group kernels
constexpr int kTileTable = 32;         // k_group32: most tiles of a CTA (it keeps their geometry)

// CTAs of k_group32 / k_group64 for the grouped instances of a batch, by a cost
// model of one iteration: the entries of each CTA in turn.
struct GroupEntry {
    int inst, rank, size, pad;         // instance, rank of the CTA in its group, group size
};
struct GroupPlan {
    int used = 0;                      // CTAs with entries: the grid of the launch
    int most = 0;                      // most tiles of one instance on one CTA
    std::vector<int> start;            // [used + 1]
    std::vector<GroupEntry> entries;
};
GroupPlan plan_groups(const std::vector<int>& inst, const std::vector<int>& tiles, const std::vector<int>& elems, int grid,
                      int fp64);

// One tile height the autotuner measured: microseconds per iteration of a single
// instance, as single solves run it (group kernel or chain) and in the chain.
struct HeightTime {
    int rows;
    double single_us, chain_us;
};
// The height to keep.  It serves both forms (an instance's results depend on the
// height, not on the form): single small instances run the group kernels, batches
// and the serve loop of many of them the chain, so the smallest product wins.
int pick_height(const std::vector<HeightTime>& t);

}  // namespace hot
