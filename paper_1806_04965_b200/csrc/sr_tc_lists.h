// Work lists of the tensor-core kernel: which CTA gets which item, or part of an item, of a launch.
#pragma once
#include <algorithm>
#include <cstdint>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

// node: where its table begins, in 16-byte words from the start of the table area (on the host, until a workspace is bound: its plan):
// a TcNode, bursts, activation boxes; words: how many it has (until then: the part of a split item).  m0: first output channel; slot:
// of the table in shared memory (set by the keeper); rank0: the cluster rank that has part 0 of a split item
struct alignas(16) TcTile { int32_t node, b0, h0, w0, m0, slot, words, rank0; };

// An item as the work lists see it: cycles of one of its parts (estimated), parts, what the kernel reads.
struct TcWork { long long cycles; int parts; TcTile tile; };

constexpr long long kAnyLoad = INT64_MAX;

// Longest processing time first: items (sorted, longest first) onto the least loaded of `grid` lists.  Returns the longest list's load, or
// -1 as soon as one reaches `limit`.
inline long long spread_items(const std::vector<TcWork>& work, size_t n, int grid, std::vector<std::vector<TcTile>>* lists, long long limit = kAnyLoad)
{
    if (!lists && n <= (size_t)grid) return n > 0 ? work[0].cycles : 0;
    std::vector<std::pair<long long, int>> heap;             // (-load, cta): the standard heap keeps the largest on top
    for (int c = 0; c < grid; ++c) heap.push_back({0, -c});
    std::make_heap(heap.begin(), heap.end());
    if (lists) lists->assign(grid, {});
    long long longest = 0;
    for (size_t i = 0; i < n; ++i) {
        std::pop_heap(heap.begin(), heap.end());
        std::pair<long long, int> top = heap.back();
        if (lists) (*lists)[-top.second].push_back(work[i].tile);
        top.first -= work[i].cycles;
        longest = std::max(longest, -top.first);
        if (longest >= limit) return -1;
        heap.back() = top;
        std::push_heap(heap.begin(), heap.end());
    }
    return longest;
}

// Items (sorted, longest first) onto `grid` CTAs in clusters: an item of p > 1 parts goes to p neighbouring CTAs of one cluster that
// have no part yet, behind what else they have; whole items to the least loaded CTAs.  Returns the longest list's load, or -1 if
// the parts do not find room in this order, or as soon as a list reaches `limit`.
inline long long spread_split(const std::vector<TcWork>& work, int grid, int cluster, std::vector<std::vector<TcTile>>* lists, long long limit = kAnyLoad)
{
    // least loaded first: an entry per CTA and change of its load, those that its load has left behind are dropped when they come up
    using Entry = std::pair<long long, int>;
    std::priority_queue<Entry, std::vector<Entry>, std::greater<Entry>> order;
    for (int c = 0; c < grid; ++c) order.push({0, c});
    std::vector<long long> load(grid, 0);
    std::vector<char> taken(grid, 0);
    std::vector<TcTile> part(grid);
    if (lists) lists->assign(grid, {});
    for (const TcWork& w : work) {
        const int n = w.parts;
        int at = -1;
        long long least = 0;
        if (n == 1) {
            while (order.top().first != load[order.top().second]) order.pop();
            at = order.top().second;
            order.pop();
        }
        for (int c = 0; n > 1 && c + n <= grid; c += n) {
            long long l = 0;
            bool room = true;
            for (int q = 0; q < n; ++q) {
                l = std::max(l, load[c + q]);
                room = room && !taken[c + q];
            }
            if (room && (at < 0 || l < least)) { at = c; least = l; }
        }
        if (at < 0) {
            if (lists) lists->clear();
            return -1;
        }
        for (int q = 0; q < n; ++q) {
            load[at + q] += w.cycles;
            if (load[at + q] >= limit) {
                if (lists) lists->clear();
                return -1;
            }
            order.push({load[at + q], at + q});
            TcTile t = w.tile;
            t.words = q;
            t.rank0 = at % cluster;
            if (n > 1) {
                part[at + q] = t;
                taken[at + q] = 1;
            } else if (lists) {
                (*lists)[at].push_back(t);
            }
        }
    }
    if (lists)
        for (int c = 0; c < grid; ++c)
            if (taken[c]) (*lists)[c].push_back(part[c]);
    return *std::max_element(load.begin(), load.end());
}

// The same, whatever the order: where it scatters the parts so that a larger item finds no room, those of most parts go first, so that none
// cuts up a place that a later one needs.  Every item is listed whole; false only if there are more parts than CTAs.
inline bool place_split(std::vector<TcWork> work, int grid, int cluster, std::vector<std::vector<TcTile>>& lists)
{
    if (spread_split(work, grid, cluster, &lists) < 0) {
        std::stable_sort(work.begin(), work.end(), [](const TcWork& a, const TcWork& b) { return a.parts > b.parts; });
        if (spread_split(work, grid, cluster, &lists) < 0) return false;
    }
    size_t wanted = 0, listed = 0;
    for (const TcWork& w : work) wanted += w.parts;
    for (const auto& l : lists) listed += l.size();
    return wanted == listed;
}
