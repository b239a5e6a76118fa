"""The word of the grid barrier (csrc/esp_barrier.h): arrivals, the give-up and the polls are 64-bit accesses of
one 64-bit word (accesses of different sizes that overlap carry no order in the memory model), and its
arithmetic holds for every state that a barrier passes through. CPU only: a missing order is not provoked on a GPU.
"""

import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_07971_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include "esp_barrier.h"
int main()
{
    typedef unsigned long long u64;
    long bad = 0;
    u64 held;
    std::memset(&held, esp::kBarHeldByte, sizeof held);
    for (u64 round : {0ull, 1ull, 399ull, 28256363ull, 28256364ull, 2147483646ull})   // 2^32 arrivals lie between
        for (u64 grid : {1ull, 2ull, 77ull, 152ull}) {
            const u64 target = (round + 1) * grid;
            for (u64 got = 0; got <= grid; ++got) {   // arrivals of this barrier so far, given up or not
                const u64 v = round * grid + got;
                bad += esp::bar_reached(v, target) != (got == grid) || esp::bar_aborted(v);
                bad += esp::bar_reached(v | esp::kBarAbort, target) != (got == grid) || !esp::bar_aborted(v | esp::kBarAbort);
                bad += esp::bar_reached(held + v, target) || esp::bar_aborted(held + v);
            }
            for (u64 ahead = 1; ahead <= grid; ++ahead)   // CTAs that already arrived at the next one
                bad += !esp::bar_reached(target + ahead, target);
        }
    std::printf("%ld\n", bad);
    return 0;
}
"""


def test_word_arithmetic(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"


def test_every_access_is_64_bits_of_the_one_word():
    code = re.sub(r"//.*", "", open(os.path.join(CSRC, "esp_place.cu")).read())
    body = code[code.index("grid_barrier("):]
    body = body[:body.index("\n}\n")]
    assert "grid_barrier(unsigned long long *bar, unsigned long long target" in body
    uses = [ln for ln in body.splitlines()[1:] if re.search(r"\bbar\b", ln)]
    assert len(uses) == 3   # the arrival, the poll, the give-up
    assert sum("red.release.gpu.global.add.u64" in u for u in uses) == 1
    assert sum("ld.acquire.gpu.u64" in u for u in uses) == 1
    assert sum("atomicOr(bar, kBarAbort)" in u for u in uses) == 1
    header = open(os.path.join(CSRC, "esp_kernels.h")).read()
    assert re.search(r"unsigned long long \*bar;", header)
