// How gemv_cw shares the SMs between the layers of a launch: host arithmetic only, without CUDA. Internal;
// not part of the ABI.
#pragma once

namespace aq {

// Clusters that layer l of a launch gets if every cluster makes at most `passes` passes over its row blocks.
inline int cw_layer_clusters(int row_blocks, int passes) { return (row_blocks - 1) / passes + 1; }

// The fewest passes with which the clusters of n layers (rbs[l] > 0 row blocks each) number at most cap, the
// clusters that are resident at once. A layer needs one cluster whatever the passes, so with more layers
// than resident clusters (clusters of eight on a part of a GPU) the grid exceeds cap and runs in waves.
inline int cw_group_passes(const int* rbs, int n, int cap) {
    if (cap < n) cap = n;
    auto need = [&](int p) {
        long long c = 0;
        for (int l = 0; l < n; ++l) c += cw_layer_clusters(rbs[l], p);
        return c;
    };
    int lo = 1, hi = 1;
    for (int l = 0; l < n; ++l)
        if (rbs[l] > hi) hi = rbs[l];
    while (lo < hi) {                       // need() falls with the passes, and need(hi) = n <= cap
        const int mid = lo + (hi - lo) / 2;
        if (need(mid) <= cap) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

}  // namespace aq
