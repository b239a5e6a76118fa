"""Host planner of the packed evaluation passes (CPU): the word layout of the unit fields holds every unit
exactly, and the packed order, tiles and ranges cover every job of every table once, whatever its option
counts. The planner runs under AddressSanitizer and UndefinedBehaviorSanitizer.
"""

import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TINY, LARGE = 6, 7


def build(tmp):
    exe = os.path.join(tmp, "packed_plan")
    src = os.path.join(ROOT, "paper_2608_07971_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-g", "-O1", "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
                    "-I", src, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "packed_plan_driver.cpp"), os.path.join(src, "esp_plan.cpp"), "-o", exe],
                   check=True)
    return exe


def cases():
    rng = np.random.default_rng(3)
    for S, J, R, warps, kind in [(1, 1, 1, 8, 1), (2, 7, 6, 100, 16), (3, 100, 4, 3040, "any"), (1, 2000, 6, 16, "any"),
                                 (5, 300, 8, 64, "big"), (2, 50, 16, 10, 256), (1, 40, 5, 7, 257), (4, 500, 3, 40, 1),
                                 (3, 333, 6, 12, 2), (2, 64, 2, 3040, 12)]:
        if kind == "any":
            K = rng.integers(1, 300, S * J)
        elif kind == "big":
            K = rng.choice([1, 2, 3, 4, 5, 64, 128, 129, 255, 256, 257, 1000, 4097], S * J)
        else:
            K = np.full(S * J, kind)
        off = np.concatenate([[0], np.cumsum(K)]).astype(np.int64)
        umax = rng.choice([0, 1, 400, 900, 8000, 65535, 163840, 524288, (1 << 23) - 1, 1 << 23], R, p=[.1] * 9 + [.1])
        yield S, J, R, warps, (0 if isinstance(kind, str) else kind), off, umax.astype(np.int64)


def shape(mk, n):
    code, m = mk & 7, mk >> 3
    if code == TINY:
        return 64, -(-n // (256 // m))
    if code == LARGE:
        nch = -(-m // 64)
        return -(-m // nch), n * nch
    return (32 >> code) * m, -(-n // (32 >> code))


def test_packed_plans(tmp_path):
    exe = build(str(tmp_path))
    todo = list(cases())
    words = [len(todo)]
    for S, J, R, warps, all_k, off, um in todo:
        words += [S, J, R, warps, all_k, *off.tolist(), *um.tolist()]
    np.asarray(words, np.int64).tofile(tmp_path / "in")
    subprocess.run([exe, str(tmp_path / "in"), str(tmp_path / "out")], check=True)
    w = iter(np.fromfile(tmp_path / "out", np.int64).tolist())
    take = lambda n: [next(w) for _ in range(n)]   # noqa: E731
    for S, J, R, warps, all_k, off, um in todo:
        ok, nw = take(2)
        fields = [take(5) for _ in range(8)]
        if um.max() >= 1 << 23:
            assert not ok
        elif ok:
            # every column in one field; its largest unit survives the word and the screen's extraction
            cols = sorted(c for f in fields[:nw] for c in f[3:] if c >= 0)
            assert cols == list(range(R))
            for mask, shift, magic, lo, hi in fields[:nw]:
                a, b = (int(um[lo]) if lo >= 0 else 0), (int(um[hi]) if hi >= 0 else 0)
                word = a | b << shift
                assert word < 1 << 32 and word & mask == a and word >> shift == b
                assert (magic << 32 | word) >> shift & 0xffffffff == 0x4b000000 | b and b < 1 << 23
        plan_ok, = take(1)
        assert plan_ok
        check, n_tiles, n_warps, vecs, steps, narrow = take(6)
        assert check and n_warps == min(warps, n_tiles)
        tiles = [take(5) for _ in range(n_tiles)]
        order = take(S * J)
        wb = take(n_warps + 1)
        refused, = take(1)
        assert refused
        assert sorted(order) == list(range(S * J))
        K = np.diff(off)
        at = job = total = 0
        for base, scen, mk, n, jb in tiles:
            assert base == at and jb == job
            code, m = mk & 7, mk >> 3
            for j in order[jb:jb + n]:
                k = int(K[j])
                assert j // J == scen
                if code == TINY:
                    assert m == k <= 2
                else:
                    assert k > 2 and m == -(-k // 4) and (code == LARGE) == (k > 256)
                    if code != LARGE:   # lanes enough for the job: four or eight options each
                        assert (1 << code) * (4 if (1 << code) >= m else 8) >= k
            v, st = shape(mk, n)
            assert v <= 64
            at += v * st
            total += st
            job += n
        assert job == S * J and at == vecs and total == steps
        assert wb[0] == 0 and wb[-1] == n_tiles and all(x <= y for x, y in zip(wb, wb[1:]))
