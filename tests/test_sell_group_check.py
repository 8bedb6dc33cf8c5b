"""The check of the groups of a sorted sliced layout, on the CPU: a sound table
passes, and one field of one group changed is found wherever it is."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_02530_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include "sell_groups.h"
#include <cstdio>
#include <vector>
using namespace spmvk;
int main() {
    // one rank from slice 1 on: four full slices of 1 entry (a group), two of 3 (a
    // group), a full one of 3 and a short one of 2 (slices alone)
    const int lens[9] = {9, 1, 1, 1, 1, 3, 3, 3, 2};
    std::vector<SellSlice> slices;
    std::vector<uint8_t> len;
    int off = 0;
    for (int i = 0; i < 9; ++i) {
        const int rows = i == 8 ? 20 : 32;
        slices.push_back(SellSlice{32 * i, rows, lens[i], i ? 7 : 0, off, 1, 0, 0});
        off += 32 * lens[i];
        for (int r = 0; r < rows; ++r) len.push_back((uint8_t)lens[i]);
    }
    std::vector<SellSlice> groups;
    for (const int i : {0, 1, 5, 7, 8}) {
        groups.push_back(slices[i]);
        groups.back().first = i;
    }
    groups[1].group = 4;
    groups[2].group = 2;
    auto bad = [&](const std::vector<SellSlice>& g, const std::vector<uint8_t>& l) {
        int n = 0;
        for (int i = 1; i < 5; ++i) n += !sell_group_ok(g.data(), i, 1, 5, slices.data(), 1, 9, l.data(), (int64_t)l.size());
        return n;
    };
    if (bad(groups, len)) return 1;
    int missed = 0, tried = 0;
    for (int i = 1; i < 5; ++i)
        for (int f = 0; f < 7; ++f)
            for (const int by : {-33, -1, 1, 2, 1 << 30}) {
                std::vector<SellSlice> g = groups;
                int32_t* field[7] = {&g[i].p0, &g[i].rows, &g[i].len, &g[i].xoff, &g[i].off, &g[i].group, &g[i].first};
                *field[f] += by;
                ++tried;
                if (!bad(g, len)) ++missed;
            }
    for (int p = 32; p < 7 * 32; ++p) {   // a row of a group of another length
        std::vector<uint8_t> l = len;
        ++l[p];
        ++tried;
        if (!bad(groups, l)) ++missed;
    }
    std::vector<uint8_t> shorter(len.begin(), len.begin() + 6 * 32 + 31);   // positions past the rows
    ++tried;
    if (!bad(groups, shorter)) ++missed;
    std::printf("%d %d", tried, missed);
    return 0;
}
"""


def test_every_planted_fault_is_found(tmp_path):
    if not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    (tmp_path / "g.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(CUDA, "include"), str(tmp_path / "g.cpp"),
                    "-o", str(tmp_path / "g")], check=True)
    r = subprocess.run([str(tmp_path / "g")], capture_output=True, text=True)
    assert r.returncode == 0
    tried, missed = map(int, r.stdout.split())
    assert tried == 4 * 7 * 5 + 6 * 32 + 1 and missed == 0
