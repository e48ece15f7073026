// Which blocks of a batched Krylov launch work on which problems (host code
// without CUDA).
#pragma once

#include <algorithm>
#include <functional>
#include <numeric>
#include <queue>
#include <utility>
#include <vector>

namespace wrc {

// A launch of at most `sms` blocks, one per SM, for problems of n[q] points.
// Items are triples (problem, block's index in it, its blocks); block b takes
// items off[b] .. off[b + 1] - 1 in turn.  A block's time is taken as its
// share of each of its problems' points plus kItem points an item (a launch's
// Arnoldi steps cost ~0.2 ms beside ~1 us a point, m = 30).
//
// Two plans are made and the one with the shorter longest block is taken.
//  - Up to as many problems as blocks: each gets one block, and the rest go
//    one by one to the problem with the most points per block, as long as its
//    share stays above `least` points.
//  - Any number: problems larger than a bound get blocks of their own, then
//    the others, largest first, go to the least loaded group of g blocks, each
//    problem on all g blocks of its group; g = 1: also to the blocks that
//    have a large problem's share, after it.  Bounds of 1, 1.4 and 2 average
//    loads and no bound, g = 1, 2, 4 and 8 are tried.
// The blocks of a problem of several blocks meet at grid barriers, so they
// have the same problems before it, or none, and reach it together.
//
// Measured on GB300, one step of 200 mixed members, one of 72K points and 199
// of 2.8K: 9.1 ms, 47.4 with every problem whole on a block; 160 of 9.1K
// points 13.1 and 16.5; 256 of 2.7K to 30K points 42.5 and 45.7.  (The first
// plan, against more and smaller blocks with FP64 dots: one launch of 48
// mixed members of 9-17K points 4.09 ms and 5.56, 17 FP64 members 1.79 and
// 2.57, omega and r_v of 65.9K points 1.21 and 2.06.)
inline void krylov_batch_plan(const std::vector<long long>& n, long long least, int sms, std::vector<int>& items,
                              std::vector<int>& off) {
    constexpr double kItem = 192.0;
    const int M = (int)n.size();
    least = std::max(1LL, least);
    std::vector<int> single;   // the first plan: blocks of each problem
    double cost = 1e300;
    if (M <= sms) {
        single.assign(M, 1);
        for (int used = M; used < sms; ++used) {
            int best = -1;
            double most = (double)least;
            for (int q = 0; q < M; ++q) {
                const double share = (double)n[q] / single[q];
                if (share > most) {
                    most = share;
                    best = q;
                }
            }
            if (best < 0) break;
            single[best] += 1;
        }
        cost = 0.0;
        for (int q = 0; q < M; ++q) cost = std::max(cost, (double)n[q] / single[q] + kItem);
    }
    std::vector<int> order(M);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return n[a] > n[b]; });
    const double mean = std::max(1.0, (double)std::accumulate(n.begin(), n.end(), 0LL) / sms);
    // the second plan with bound x mean (0: none) and groups of g blocks; group[]: the least loaded first
    using Load = std::pair<double, int>;   // (time, first block)
    const auto plan = [&](double x, int g, std::vector<std::vector<int>>* blocks) {
        std::priority_queue<Load, std::vector<Load>, std::greater<Load>> group;
        double longest = 0.0;
        int used = 0, at = 0;
        const auto put = [&](int q, int first, int nb) {
            if (blocks)
                for (int b = 0; b < nb; ++b) (*blocks)[first + b].insert((*blocks)[first + b].end(), {q, b, nb});
        };
        // own blocks, while every other problem keeps a group
        for (; x > 0.0 && at < M; ++at) {
            const double size = (double)n[order[at]];
            const int nb = (int)std::min(size / (x * mean) + 1.0, size / (double)least + 1.0);
            if (nb < 2 || used + nb > sms - g) break;
            put(order[at], used, nb);
            const double time = size / nb + kItem;
            longest = std::max(longest, time);
            if (g == 1)
                for (int b = 0; b < nb; ++b) group.push({time, used + b});
            used += nb;
        }
        for (; used + g <= sms; used += g) group.push({0.0, used});
        for (; at < M; ++at) {
            Load l = group.top();
            group.pop();
            put(order[at], l.second, g);
            l.first += (double)n[order[at]] / g + kItem;
            longest = std::max(longest, l.first);
            group.push(l);
        }
        return longest;
    };
    // a shorter longest block by 5% at least: the estimate is no better
    double bx = -1.0;
    int bg = 0;
    for (const int g : {1, 2, 4, 8})
        for (const double x : {0.0, 1.0, 1.4, 2.0}) {
            if (g > sms || cost < 1.15 * (mean + kItem)) continue;   // (as even as can be)
            const double c = plan(x, g, nullptr);
            if (c < 0.95 * cost) {
                cost = c;
                bx = x;
                bg = g;
            }
        }
    items.clear();
    off.assign(1, 0);
    if (bx < 0.0) {
        for (int q = 0; q < M; ++q)
            for (int b = 0; b < single[q]; ++b) {
                items.insert(items.end(), {q, b, single[q]});
                off.push_back((int)items.size() / 3);
            }
        return;
    }
    std::vector<std::vector<int>> blocks(sms);
    plan(bx, bg, &blocks);
    for (const auto& v : blocks) {
        if (v.empty()) continue;
        items.insert(items.end(), v.begin(), v.end());
        off.push_back((int)items.size() / 3);
    }
}

}  // namespace wrc
