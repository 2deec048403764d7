"""The strips of csrc/lbm_batch_plan.h as launched, on the CPU: a launch on the
CTAs that get work keeps the plan made for a larger grid."""
import shutil
import subprocess
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0706_0405_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "lbm_batch_plan.h"
using namespace lbm;
int main() {
    srand(11);
    for (int trial = 0; trial < 60; ++trial) {
        const int np = 1 + rand() % 40, ns = 3 + 2 * (rand() % 3);
        std::vector<int> nx(np);
        for (int& x : nx) x = 1 + rand() % (rand() % 2 ? 140 : 1500);
        for (int grid = 1; grid <= 700; grid += 1 + rand() % 9) {
            std::vector<StripWarp> a, b;
            const int rounds = strip_plan(np, nx.data(), ns, grid, 4, a), ctas = rounds < grid ? rounds : grid;
            const int again = strip_plan(np, nx.data(), ns, ctas, 4, b);
            if (again != rounds || a.size() != b.size() || memcmp(a.data(), b.data(), a.size() * sizeof a[0])) {
                printf("trial %d, grid %d\n", trial, grid);
                return 1;
            }
        }
    }
    puts("ok");
}
"""


def test_a_plan_for_the_ctas_with_work_is_the_plan_of_the_grid(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "strips.cpp", tmp_path / "strips"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout
