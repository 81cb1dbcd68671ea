"""How many CTAs an RVE gets in FP64 (csrc/fp64_parts.h, compiled by itself): never a
cluster that the device cannot hold, with any device limit as many as without one up
to it, and leaves and groups of terms that do not depend on it."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2305_07030_gb300", "csrc")

HARNESS = r"""
#include <algorithm>
#include <cstdio>
#include "fp64_parts.h"
using namespace fe2;
int main() {
    long bad = 0;
    for (int n = 1; n <= 5000; n += n < 700 ? 1 : 37)
        for (int limit : {0, 1, 2, 4, 8, 16}) {
            bad += fp64_single_parts(n, limit) != std::min(fp64_single_parts(n, 16), std::max(limit, 1));
            for (int parts = 1; parts <= 16; parts *= 2) {
                const int most = fp64_leaf_factor(n, parts);
                const int g = fp64_groups(n, parts, parts * most);
                bad += g * most > 16 || (g > 1 && n < g * parts * most * 64);  // one warp's table, one CTA's sums
                bad += parts * most > 16 || (most > 1 && n < parts * most * kSplitNodes);
                for (int ctas = parts; ctas < 300; ++ctas) {
                    const int f = fp64_split_factor(ctas, n, parts, limit);
                    const int free = fp64_split_factor(ctas, n, parts, 16);
                    bad += most % f != 0 || free > most || (f > 1 && ctas * f > 128);
                    bad += f != std::max(1, std::min(free, limit / parts));
                }
            }
        }
    // a 512-node RVE alone and among others, the allocation-free call's sizes
    bad += fp64_split_factor(1, 512, 1, 16) != 8 || fp64_split_factor(40, 512, 1, 16) != 2 ||
           fp64_split_factor(65, 512, 1, 16) != 1 || fp64_single_parts(79, 16) != 1 || fp64_single_parts(640, 16) != 16;
    printf("%ld\n", bad);
    return 0;
}
"""


def test_clusters_fit_the_device(tmp_path):
    src = tmp_path / "parts.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "parts")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout.strip() == "0"
