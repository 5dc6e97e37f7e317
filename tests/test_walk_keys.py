"""Host check of the column walk's block keys: where the groups of a set lie within warps, whose
half-sweeps no CTA barrier orders, each warp builds the keys of its own groups and of no other
warp's, whatever the number of groups side by side; all groups have a builder."""
import os
import subprocess

from paper_2401_07965_gb300 import build

SRC = r"""
#include "pa_internal.cuh"
#include <cstdio>
#include <vector>
int main() {
    int bad = 0;
    for (int NC = 1; NC <= 32; NC *= 2)
        for (int GP = 1; GP * NC <= 512; ++GP)
            for (int CPT = 1; CPT <= 28; ++CPT) {
                pa::WalkPlan g = {};
                g.NC = NC; g.GP = GP; g.CPT = CPT; g.NT = (GP * NC + 31) / 32 * 32;
                const int gpw = 32 / NC;
                std::vector<int> built(GP * CPT, 0);
                for (int warp = 0; warp < g.NT / 32; ++warp)
                    for (int q = 0; q < gpw * CPT; ++q) {
                        const int u = pa::walk_key_group(g, gpw, warp * gpw, q);
                        if (u < 0) continue;
                        // group u's lanes: columns (u % GP) NC .. + NC - 1 of the CTA's threads
                        if (u >= GP * CPT || (u % GP) * NC / 32 != warp) bad = 1;
                        else built[u] += 1;
                    }
                for (int n : built) if (n != 1) bad = 1;
                // the whole CTA as one builder
                for (int q = 0; q < GP * CPT; ++q)
                    if (pa::walk_key_group(g, GP, 0, q) != q) bad = 1;
            }
    std::printf("%d\n", bad);
}
"""


def test_each_warp_builds_its_own_groups_keys(tmp_path):
    src, exe = tmp_path / "k.cu", tmp_path / "k"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"
