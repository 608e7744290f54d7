"""The choice among launch shapes by timing (csrc/autotune.h), compiled for the
host with a clock of its own."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1304_5583_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <map>
#include "autotune.h"
int main() {
    using lrr::TuneKey;
    // shape -> milliseconds; a shape's first run also pays 60 us
    std::map<int, float> ms{{10, 0.059f}, {4, 0.075f}, {16, 0.080f}};
    std::map<int, int> runs;
    auto time = [&](int shape, bool) { return ms[shape] + (runs[shape]++ ? 0.f : 0.060f); };
    int best = -1;
    // ids 0, 4 and 8 stand for the shapes 10, 4 and 10 again
    const std::vector<std::pair<int, int>> c{{0, 10}, {4, 4}, {8, 10}};
    if (!lrr::pick_fastest(c, time, &best) || best != 0) return std::printf("chose %d\n", best), 1;
    if (runs[10] != 2 || runs[4] != 2) return std::printf("ran %d %d\n", runs[10], runs[4]), 2;
    const std::vector<std::pair<int, int>> d{{0, 16}, {4, 4}, {8, 10}};
    if (!lrr::pick_fastest(d, time, &best) || best != 8) return 3;
    if (lrr::pick_fastest(c, [](int, bool) { return -1.f; }, &best)) return 4;
    // every field tells two keys apart
    const TuneKey k{0, 1, 2, 3, 4, 5, 6, 7, false};
    TuneKey v[9] = {k, k, k, k, k, k, k, k, k};
    v[0].dev++; v[1].prec++; v[2].m++; v[3].n++; v[4].r++; v[5].t++; v[6].max_pp++; v[7].max_L++; v[8].grid = true;
    for (const TuneKey& o : v) if (!(k < o) || o < k) return 5;
    return k < k ? 6 : 0;
}
"""


def test_first_candidate_is_not_charged_for_loading(tmp_path):
    src, exe = tmp_path / "tune.cpp", tmp_path / "tune"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
