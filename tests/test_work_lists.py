"""Work lists of launches in clusters, on the CPU: every part of every item has its place, whatever the order of the items."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <random>
#include "sr_tc_lists.h"
// the lists hold every part once: parts of an item on neighbouring CTAs of one cluster, in order, each the last entry of its list
static bool sound(const std::vector<TcWork>& work, int grid, int cluster, const std::vector<std::vector<TcTile>>& lists)
{
    if ((int)lists.size() != grid) return false;
    std::vector<std::vector<int>> at(work.size());
    for (int c = 0; c < grid; ++c)
        for (size_t i = 0; i < lists[c].size(); ++i) {
            const TcTile& t = lists[c][i];
            if (work[t.node].parts > 1 && (i + 1 != lists[c].size() || t.rank0 + t.words != c % cluster)) return false;
            if ((int)at[t.node].size() != t.words) return false;
            at[t.node].push_back(c);
        }
    for (size_t i = 0; i < work.size(); ++i) {
        if ((int)at[i].size() != work[i].parts) return false;
        for (size_t q = 1; q < at[i].size(); ++q)
            if (at[i][q] != at[i][0] + (int)q || at[i][q] / cluster != at[i][0] / cluster) return false;
    }
    return true;
}
static std::vector<TcWork> items(const std::vector<std::pair<long long, int>>& of)
{
    std::vector<TcWork> work;
    for (size_t i = 0; i < of.size(); ++i) work.push_back(TcWork{of[i].first, of[i].second, TcTile{(int)i, 0, 0, 0, 0, 0, 0, 0}});
    return work;
}
int main()
{
    std::vector<std::vector<TcTile>> lists;
    for (const auto& of : {std::vector<std::pair<long long, int>>{{30000, 1}, {20000, 4}, {19500, 2}, {19500, 2}},
                           std::vector<std::pair<long long, int>>{{30000, 1}, {20000, 2}, {20000, 2}, {19900, 4}}})
        for (int cluster : {4, 8}) {
            const auto work = items(of);
            if (!place_split(work, 8, cluster, lists) || !sound(work, 8, cluster, lists)) return 1;
        }
    std::mt19937 rng(5);
    for (int n = 0; n < 20000; ++n) {
        const int cluster = 2 << rng() % 3, grid = cluster * (1 + rng() % 18);
        std::vector<std::pair<long long, int>> of;
        for (int room = grid; room > 0;) {
            const int parts = 1 << rng() % 4;
            if (parts > cluster || parts > room) continue;
            of.push_back({1 + rng() % 1000, parts});
            if (parts > 1 || rng() % 2) room -= parts;
        }
        if (rng() % 2) std::sort(of.begin(), of.end(), [](auto& a, auto& b) { return a.first > b.first; });
        const auto work = items(of);
        if (!place_split(work, grid, cluster, lists) || !sound(work, grid, cluster, lists)) return 2;
    }
    if (place_split(items({{10, 2}, {10, 2}, {10, 2}}), 4, 4, lists)) return 3;
    std::puts("ok");
    return 0;
}
"""


def test_every_part_of_an_item_is_listed(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1806_04965_b200", "csrc"), str(tmp_path / "driver.cpp"),
                           "-o", str(tmp_path / "driver")])
    out = subprocess.run([str(tmp_path / "driver")], capture_output=True, text=True, timeout=120)
    assert (out.returncode, out.stdout.strip()) == (0, "ok")
