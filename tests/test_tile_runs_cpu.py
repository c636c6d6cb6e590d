"""The runs of chains that one launch of the dense-tile label kernel takes
(csrc/tile_runs.h), compiled for the host: every chain once and in order, and no block
lists more jobs than its shared memory is meant for, whichever of the run's chains are
on the engine."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdio.h>
#include <stdlib.h>
#include "tile_runs.h"

// jobs of the fullest block when the chains with keep[b] are dealt out
static int most_jobs(const std::vector<int32_t>& t, const std::vector<char>& keep, int b0, int b1,
                     int G) {
    std::vector<int> jobs(G, 0);
    int64_t off = 0;
    for (int b = b0; b < b1; ++b) {
        if (!t[b] || !keep[b]) continue;
        for (int g = 0; g < G; ++g) {
            int first = g - (int)(off % G);
            if (first < 0) first += G;
            jobs[g] += first < t[b];
        }
        off += t[b];
    }
    return *std::max_element(jobs.begin(), jobs.end());
}

int main(void) {
    srand(7);
    const int Bs[] = {1, 2, 40, 300, 1500}, Ts[] = {1, 9, 40, 400}, Gs[] = {1, 7, 152};
    const int Js[] = {1, 3, 64, 512};
    for (int B : Bs) for (int T : Ts) for (int G : Gs) for (int J : Js) {
        if ((long)B * G > 60000) continue;
        std::vector<int32_t> t(B);
        std::vector<char> keep(B);
        for (int b = 0; b < B; ++b) t[b] = rand() % 5 ? 1 + rand() % T : 0;
        const std::vector<int32_t> r = tile_runs(t, G, J);
        if (r.front() != 0 || r.back() != B) return printf("ends\n"), 1;
        for (size_t i = 0; i + 1 < r.size(); ++i) {
            if (r[i] >= r[i + 1]) return printf("order\n"), 1;
            for (int all = 1; all >= 0; --all) {
                for (int b = 0; b < B; ++b) keep[b] = all || rand() % 2;
                const int n = most_jobs(t, keep, r[i], r[i + 1], G);
                if (n > J) return printf("B %d T %d G %d: %d jobs > %d\n", B, T, G, n, J), 1;
            }
        }
    }
    // few chains, or few tiles a block: one launch
    if (tile_runs(std::vector<int32_t>(512, 1000), 152, 512).size() != 2) return 1;
    if (tile_runs(std::vector<int32_t>(70000, 1), 152, 512).size() != 2) return 1;
    // 20,000 chains of 160 tiles: one list would be 20,000 jobs (320 KB) a block
    if (tile_runs(std::vector<int32_t>(20000, 160), 152, 512).size() != 41) return 1;
    printf("ok\n");
    return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="needs g++")
def test_runs_bound_the_job_lists(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_1812_10048_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout
