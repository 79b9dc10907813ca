// pv_runs.h -- how a launch over items of different sizes is cut (host code).
#pragma once

namespace pv {

// Blocks of one item in the launch's first two grid dimensions.
struct RunExtent {
    long long x, y;
};

constexpr int kRunItems = 65535;           // items of one launch (the grid's limit)
constexpr long long kRunWaste = 8192;      // empty blocks that cost no more than another launch (0.5 ns each)

// A launch over several items has the grid of its largest item for every one of them, and blocks beyond an item's own
// leave at once. Consecutive items share a launch as long as the blocks that leave are no more than those that work,
// and a few. One launch for all made calls that mix sizes wait for empty blocks: clustering 1,000 sets of 300 points
// and one of 500,000 took 141 ms, now 8.9; the surfaces of 300 receptors of 500 atoms and one of 150,000 14.3 ms, now
// 3.6; the packed maps of 500 boxes of 10 A and one of 90 A 39 ms, now 7.0.
// extent(i): item i's blocks. launch(first, n, extent): the items first .. first + n - 1 in a grid of that extent;
// anything but 0 ends the loop and is returned.
template <class Extent, class Launch>
auto launch_runs(int first, int n, Extent&& extent, Launch&& launch) -> decltype(launch(0, 0, RunExtent{1, 1})) {
    const int end = first + n;
    while (first < end) {
        RunExtent most{0, 0};
        long long work = 0;
        int m = 0;
        while (first + m < end && m < kRunItems) {
            const RunExtent e = extent(first + m);
            const RunExtent top{e.x > most.x ? e.x : most.x, e.y > most.y ? e.y : most.y};
            const long long with = work + e.x * e.y;
            if (m > 0 && top.x * top.y * (m + 1) - with > with + kRunWaste) break;
            most = top;
            work = with;
            ++m;
        }
        if (work > 0) {
            const auto e = launch(first, m, most);
            if (e != decltype(e){}) return e;
        }
        first += m;
    }
    return {};
}

}  // namespace pv
