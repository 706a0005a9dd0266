"""Rows of the tensor tiles' work items (csrc/tile_rows.cuh), compiled for the
host. When a launch gives up, every row of every item has to be left with no
candidates and a bound that is never certified, whatever stood in the workspace:
the kernels that follow use the counts as loop bounds before the host has read
the status. Random tables: one cloud, clouds with padded rows one after another,
and key lists split into parts."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2507_14261_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "tile_rows.cuh"
using namespace famst::tile;
struct Item { int q0, row_end, shift, part; };
int main() {
    std::mt19937 rng(14261);
    auto pick = [&](int a, int b) { return int(rng() % unsigned(b - a + 1)) + a; };
    for (int trial = 0; trial < 2000; ++trial) {
        std::vector<Item> items;
        int rows = 0, slots = 0;   // compact rows, side slots
        const int kind = trial % 3;
        const int clouds = kind == 1 ? pick(1, 6) : 1;
        int padded = 0;
        for (int c = 0; c < clouds; ++c) {
            const int n = pick(1, 900);
            for (int q = 0; q < n; q += ROWS) {
                const int parts = kind == 2 && pick(0, 2) == 0 ? pick(2, 5) : 0;
                for (int p = 0; p < (parts ? parts : 1); ++p)
                    items.push_back({padded + q, padded + n, padded - rows, parts ? ++slots : 0});
            }
            rows += n;
            padded += (n + 255) / 256 * 256;
        }
        // unset workspace, with a guard entry at each end
        std::vector<int32_t> cnt(size_t(rows) + 2, 0x5a5a5a5a), scnt(size_t(slots) * ROWS + 2, 0x5a5a5a5a);
        std::vector<float> sp(cnt.size(), 7.0f), ssp(scnt.size(), 7.0f);
        std::vector<int> seen(cnt.size(), 0), sseen(scnt.size(), 0);
        const int grid = pick(1, int(items.size()));
        for (int b = 0; b < grid; ++b)
            for (int row = 0; row < ROWS; ++row)
                for (size_t it = size_t(b); it < items.size(); it += size_t(grid)) {
                    const Item &I = items[it];
                    if (I.q0 + row >= I.row_end) continue;
                    const RowSlot s = row_slot(I.q0, row, I.shift, I.part);
                    if (s.at >= (s.side ? scnt.size() : cnt.size()) - 2) return std::printf("range\n"), 1;
                    ++(s.side ? sseen : seen)[s.at + 1];
                    give_up_row(s, cnt.data() + 1, sp.data() + 1, scnt.data() + 1, ssp.data() + 1);
                }
        std::vector<char> split(size_t(rows), 0);   // rows whose item is split have side entries only
        for (auto &I : items)
            if (I.part > 0)
                for (int row = 0; row < ROWS && I.q0 + row < I.row_end; ++row) split[size_t(I.q0 + row - I.shift)] = 1;
        for (int r = 0; r < rows; ++r) {
            const bool in = !split[size_t(r)];
            if (seen[size_t(r) + 1] != int(in)) return std::printf("row %d hit %d times\n", r, seen[size_t(r) + 1]), 1;
            if (in && (cnt[size_t(r) + 1] != 0 || !(sp[size_t(r) + 1] == -INFINITY))) return std::printf("row %d unset\n", r), 1;
        }
        for (size_t s = 1; s + 1 < scnt.size(); ++s) {
            if (sseen[s] > 1) return std::printf("side %zu twice\n", s), 1;
            if (sseen[s] && (scnt[s] != 0 || !(ssp[s] == -INFINITY))) return std::printf("side unset\n"), 1;
        }
        if (cnt.front() != 0x5a5a5a5a || cnt.back() != 0x5a5a5a5a || scnt.front() != 0x5a5a5a5a ||
            scnt.back() != 0x5a5a5a5a) return std::printf("guard\n"), 1;
    }
    return 0;
}
"""


def test_given_up_items_leave_no_row_unset(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
