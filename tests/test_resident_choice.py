"""The automatic choice of the cluster-resident solve (csrc/esp_plan.cpp) against measured rounds: for every table of
tests/golden/resident_rounds.json (us per round on GB300 of each cluster size that fits and of streaming), what the rule
runs is close to the best, and never far from it. CPU only.

A row: S, J, R, fewest and most options per job, options, unit words, us streamed, then per size CTAs, lanes per job, most
jobs of a slice, co-resident clusters, most options of a slice, us."""

import json
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "esp_plan.h"
int main()
{
    int n = 0;
    if (std::scanf("%d", &n) != 1)
        return 2;
    for (; n > 0; --n) {
        int S, R, words, k;
        long long kmin, kmax, opts;
        if (std::scanf("%d %d %lld %lld %lld %d %d", &S, &R, &kmin, &kmax, &opts, &words, &k) != 7)
            return 2;
        std::vector<esp::ResSize> sizes((size_t)k);
        for (auto &o : sizes) {
            long long m;
            if (std::scanf("%d %d %d %d %lld", &o.cs, &o.lanes, &o.m_max, &o.clusters, &m) != 5)
                return 2;
            o.n_max = m;
        }
        int i = esp::resident_choice(S, R, kmin, kmax, 152, sizes);
        if (i >= 0 && esp::resident_round_us(S, R, kmin, kmax, 152, sizes[(size_t)i]) > esp::streaming_round_us(opts, R, words, 152))
            i = -1;
        std::printf("%d\n", i);
    }
    return 0;
}
"""


def test_choice_is_close_to_the_best(tmp_path):
    rows = json.load(open(os.path.join(ROOT, "tests", "golden", "resident_rounds.json")))
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER)
    csrc = os.path.join(ROOT, "paper_2608_07971_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=address,undefined", "-fno-sanitize-recover=all", "-I", csrc, "-I",
                    os.path.join(ROOT, "include"), str(src), os.path.join(csrc, "esp_plan.cpp"), "-o", str(exe)], check=True)
    text = [str(len(rows))]
    for S, _, R, kmin, kmax, n, words, _, sizes in rows:
        text.append(f"{S} {R} {kmin} {kmax} {n} {words} {len(sizes)}")
        text += [" ".join(map(str, s[:5])) for s in sizes]
    out = subprocess.run([str(exe)], input="\n".join(text), check=True, capture_output=True, text=True).stdout.split()
    assert len(out) == len(rows)
    ratio = []
    for row, i in zip(rows, map(int, out)):
        stream, sizes = row[7], row[8]
        ratio.append((stream if i < 0 else sizes[i][5]) / min([stream] + [s[5] for s in sizes]))
    assert max(ratio) <= 1.25, rows[int(np.argmax(ratio))]
    assert np.mean(ratio) <= 1.02, np.mean(ratio)
