// Host rules of the engine that need no device (see hot_plan.h).
#include "hot_plan.h"

#include <algorithm>

namespace hot {

// Groups of CTAs for one launch of k_group32.  An iteration of an instance
// costs its CTAs two waits plus their tiles one after the other; the plan
// takes the smallest time in which every instance fits into the grid: large
// ones get as many CTAs as they need, small ones share a CTA (group size 1).
GroupPlan plan_groups(const std::vector<int>& inst, const std::vector<int>& tiles, const std::vector<int>& elems,
                      int grid, int fp64) {
    GroupPlan P;
    const int n = (int)inst.size();
    const double wait = 4.0, self = 1.5;                      // microseconds: two waits and the stage; the stage alone
    auto tile_us = [&](int q) { return 0.9 + elems[q] * (fp64 ? 0.003 : 0.00015); };
    std::vector<int> order(n);
    for (int q = 0; q < n; ++q) order[q] = q;
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int b) { return tiles[a] * tile_us(a) > tiles[b] * tile_us(b); });
    std::vector<std::vector<GroupEntry>> cta;
    auto build = [&](double tau, bool write) {
        int used = 0;
        P.most = 0;
        double room = -1.0;                                   // of the shared CTA being filled
        for (int q : order) {
            const double alone = self + tiles[q] * tile_us(q);
            if (alone > tau) {
                const int per = std::max(1, (int)((tau - wait) / tile_us(q)));
                int G = (tiles[q] + per - 1) / per;
                G = std::min(G, std::min(kMaxGroup, grid));
                P.most = std::max(P.most, (tiles[q] + G - 1) / G);
                if (write)
                    for (int r = 0; r < G; ++r) cta.push_back({GroupEntry{inst[q], r, G, 0}});
                used += G;
            } else {
                if (room < alone) {
                    ++used;
                    room = tau;
                    if (write) cta.emplace_back();
                }
                room -= alone;
                P.most = std::max(P.most, tiles[q]);
                if (write) cta.back().push_back(GroupEntry{inst[q], 0, 1, 0});
            }
            if (used > grid) return false;
        }
        return true;
    };
    // shared CTAs come after the large ones in `order`, so the last one is open
    double tau = wait + 1.0;
    while (!build(tau, false)) tau *= 1.08;
    build(tau, true);
    P.used = (int)cta.size();
    P.start.assign(P.used + 1, 0);
    for (int c = 0; c < P.used; ++c) {
        P.entries.insert(P.entries.end(), cta[c].begin(), cta[c].end());
        P.start[c + 1] = (int)P.entries.size();
    }
    return P;
}

int pick_height(const std::vector<HeightTime>& t) {
    int best = 0;
    double least = 0.0;
    for (const HeightTime& h : t)
        if (!best || h.single_us * h.chain_us < least) {
            best = h.rows;
            least = h.single_us * h.chain_us;
        }
    return best;
}

}  // namespace hot
