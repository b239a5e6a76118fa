"""Word layout of the packed copy of grouped tables (CPU, under the sanitizers): every unit and the group slot
survive the word they share, and the columns priced per group are the last word's fields.
"""

import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_group_words(tmp_path):
    exe, src = str(tmp_path / "driver"), os.path.join(ROOT, "paper_2608_07971_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-g", "-O1", "-fsanitize=address,undefined", "-fno-sanitize-recover=all", "-I", src,
                    "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "packed_groups_driver.cpp"),
                    os.path.join(src, "esp_plan.cpp"), "-o", exe], check=True)
    rng = np.random.default_rng(5)
    todo = []
    for _ in range(4000):
        R = int(rng.integers(1, 17))
        rg = R - int(rng.integers(1, min(R, 3) + 1))
        todo.append((R, rg, int(rng.choice([1, 2, 8, 9, 64, 511, 1024])),
                     (1 << rng.integers(0, rng.choice([10, 19, 25]), R)) - rng.integers(0, 2, R)))
    words = [len(todo)]
    for R, rg, ng, um in todo:
        words += [R, rg, ng, *um.tolist()]
    np.asarray(words, np.int64).tofile(tmp_path / "in")
    subprocess.run([exe, str(tmp_path / "in"), str(tmp_path / "out")], check=True)
    w = np.fromfile(tmp_path / "out", np.int64)
    taken = 0
    for i, (R, rg, ng, um) in enumerate(todo):
        ok, nw, g_word, g_shift, g_mask = w[45 * i:45 * i + 5].tolist()
        fields = w[45 * i + 5:45 * i + 45].reshape(8, 5).tolist()
        bits = [max(1, int(u).bit_length()) for u in um]
        if not ok:   # too wide: a column, the group pair, or more words than there are
            pair = max(bits) <= 23 and R - rg <= 2 and sum(bits[rg:]) <= 32
            assert not pair or rg > 8 or sum(bits[:rg]) > 64, (R, rg, ng, um)
            continue
        taken += 1
        assert nw in (3, 4, 6) and max(bits) <= 23
        cols = [c for f in fields[:nw] for c in f[3:] if c >= 0]
        assert sorted(cols) == list(range(R)) and [c for c in fields[nw - 1][3:] if c >= 0] == list(range(rg, R))
        slot = ng - 1 + (ng - 1 >> 3)
        assert slot <= g_mask
        for k, (mask, shift, magic, lo, hi) in enumerate(fields[:nw]):
            a, b = (int(um[lo]) if lo >= 0 else 0), (int(um[hi]) if hi >= 0 else 0)
            word = a | b << shift | (slot << g_shift if k == g_word else 0)
            assert word < 1 << 32 and word & mask == a and word >> shift == b
            assert (magic << 32 | word) >> shift & 0xffffffff == 0x4b000000 | b and b < 1 << 23
            assert k != g_word or word >> g_shift & g_mask == slot
    assert taken > 1000 and w[-1] == 1
