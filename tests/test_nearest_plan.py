"""Buffer sizes of the nearest-pair connect (csrc/nearest_plan.h), compiled for
the host: over all calls that are accepted (lambda t (t - 1) / 2 < 2^31,
lambda <= 32), the survivors fit 32-bit counts and offsets, and the tensor
pass asks for no more memory than the warp kernel's lists, which every call
may come to need, plus a constant."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2507_14261_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "nearest_plan.h"
using namespace famst;
int main() {
    int bad = 0;
    for (int lambda : {1, 2, 5, 10, 32})
        for (int64_t n : {1024ll, 4100ll, 100000ll, 1000000ll, 20000000ll, 2147483647ll})
            for (int64_t t = 2; t <= n && lambda * nearest_pairs(t) < (int64_t(1) << 31);
                 t += 1 + t / 7) {
                const NearestPlan p = nearest_plan(n, t, lambda);
                const int64_t cap = p.cap;
                const size_t tensor = size_t(cap) * NEAREST_SURVIVOR_BYTES + nearest_pair_bytes(t, lambda);
                const bool ok = p.tensor == (cap > 0) && cap < (int64_t(1) << 31) &&
                                tensor <= nearest_warp_bytes(n, t, lambda) + (size_t(24) << 26);
                if (!ok && bad++ < 10)
                    std::printf("lambda %d n %lld t %lld cap %lld bytes %zu warp %zu\n", lambda,
                                (long long)n, (long long)t, (long long)cap, tensor,
                                nearest_warp_bytes(n, t, lambda));
            }
    // calls that fitted the card before the tensor pass was there
    for (auto p : {nearest_plan(100000, 5000, 5), nearest_plan(200000, 20000, 5),
                   nearest_plan(1000000, 20000, 5)})
        if (size_t(p.cap) * NEAREST_SURVIVOR_BYTES > (size_t(64) << 30)) ++bad;
    // the survivors of measured calls fit, in the form that is chosen
    struct { int64_t n, t; int lambda; double once, second; } measured[] = {
        {20000, 300, 1, 33.7, 5.3},     {20000, 100, 1, 133.0, 10.7}, {100000, 50, 5, 424.7, 171404.0 / 1225},
        {100000, 200, 5, 448.2, 77.5},  {1000000, 200, 10, 893.3, 402.3},
        {1000000, 1000, 10, 609.4, 197.7}, {20000, 20, 32, 1499.5, 599.4}, {20000, 100, 32, 1143.5, 164.2}};
    for (auto &m : measured) {
        const NearestPlan p = nearest_plan(m.n, m.t, m.lambda);
        const double need = (p.bounds_first ? m.second : m.once) * double(nearest_pairs(m.t));
        if (!p.tensor || need * 1.2 > double(p.cap)) {
            std::printf("n %lld t %lld lambda %d\n", (long long)m.n, (long long)m.t, m.lambda);
            ++bad;
        }
    }
    return bad ? 1 : 0;
}
"""


def test_sizes(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
