"""The packed passes' fp32 screen (csrc/esp_packed.cu, screen4), restated on the CPU with exact fp32 rounding: units
decoded from the words that pack_format lays out, the low fields of the words accumulated from -v32 and the high
fields from 0, and q the sum of both chains. |q - s| must stay within the scenario's E of tests/test_screen_bound.py
(less the fp64 chain's own rounding) for 2 to 8 words, words with a low field only, and grouped formats.
"""

import os
import subprocess
import zlib
from fractions import Fraction

import numpy as np
import pytest

from tests.test_screen_bound import TWO, bound, exact_s, fma32, v32_of

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def formats(tmp_path_factory):
    """pack_format through the test driver: f(list of (umax, r_global, n_groups)) -> list of word layouts."""
    tmp = tmp_path_factory.mktemp("packed_screen")
    exe, src = str(tmp / "driver"), os.path.join(ROOT, "paper_2608_07971_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", src, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "packed_groups_driver.cpp"), os.path.join(src, "esp_plan.cpp"), "-o", exe],
                   check=True)

    def run(umax, rg=None, ng=0):
        R = len(umax)
        np.asarray([1, R, R if rg is None else rg, ng, *[int(u) for u in umax]], np.int64).tofile(tmp / "in")
        subprocess.run([exe, str(tmp / "in"), str(tmp / "out")], check=True)
        w = np.fromfile(tmp / "out", np.int64).tolist()
        assert w[0]
        nw, g_word, g_shift = w[1], w[2], w[3]
        return nw, [w[5 + 5 * k:10 + 5 * k] for k in range(nw)], g_word, g_shift

    return run


def packed_q(fmt, units, values, p64, group=None, rg=None, swap=False):
    """q of every option at fp64 prices p64 (ungrouped: one per column; grouped: own columns' prices follow, two or
    one per group)."""
    nw, words, g_word, g_shift = fmt
    n, R = units.shape
    p32 = p64.astype(np.float32)
    grouped = group is not None
    own = R - rg if grouped else 0
    lo, hi = -v32_of(values), np.zeros(n, np.float32)
    for k, (mask, shift, magic, cl, ch) in enumerate(words):
        x = np.zeros(n, np.uint64)
        if cl >= 0:
            x |= units[:, cl].astype(np.uint64)
        if ch >= 0:
            x |= units[:, ch].astype(np.uint64) << np.uint64(shift)
        if grouped and k == g_word:
            x |= (group + (group >> 3)).astype(np.uint64) << np.uint64(g_shift)
        assert np.all(x < 1 << 32)
        two23 = np.float32(8388608.0)
        a = ((x & np.uint64(mask)) | np.uint64(0x4b000000)).astype(np.uint32).view(np.float32) - two23
        b = (((np.uint64(magic) << np.uint64(32)) | x) >> np.uint64(shift)).astype(np.uint32).view(np.float32) - two23
        for f, c in ((a, cl), (b, ch)):      # what the kernel multiplies is the unit itself
            assert np.array_equal(f.astype(np.int64), units[:, c] if c >= 0 else np.zeros(n, np.int64)) or c < 0

        def price(c):
            if c < 0:
                return np.zeros(n, np.float32)
            if grouped and c >= rg:
                return p32[rg + own * group + (c - rg)]
            return np.full(n, p32[c], np.float32)

        pl, ph = price(cl), price(ch)
        if swap:
            pl, ph = ph, pl
        lo, hi = fma32(pl, a, lo), fma32(ph, b, hi)
    return lo + hi      # numpy's fp32 sum is correctly rounded


def worst_ratio(fmt, units, values, p64, group=None, rg=None, swap=False):
    q = packed_q(fmt, units, values, p64, group, rg, swap)
    R = units.shape[1]
    cols = p64
    if group is not None:      # the largest price of each group column, and each option's own prices
        own = R - rg
        cols = np.concatenate([p64[:rg], [p64[rg + c::own].max() for c in range(own)]])
    E, M = bound(units, values, cols)
    budget = Fraction(E) - R * Fraction(M) * TWO ** -52
    assert budget > 0
    worst = Fraction(0)
    for i in range(len(values)):
        p = p64 if group is None else np.concatenate([p64[:rg], p64[rg + own * group[i]:rg + own * group[i] + own]])
        worst = max(worst, abs(Fraction(float(q[i])) - exact_s(units[i], values[i], p)) / budget)
    return float(worst)


B23 = (1 << 23) - 1
SHAPES = {                       # largest unit of each column -> 2, 3, 4, 6, 8 words, with and without high fields
    "one_column": [B23], "two_low_only": [B23, B23], "pair": [900, 400], "cluster6": [8000, 163840, 64000, 524288, 900, 400],
    "three_low_only": [B23] * 3, "four_low_only": [B23] * 4, "wide8": [B23] * 8, "mixed5": [B23, 1, 65535, 300, 524288],
    "twelve": [65535] * 12, "sixteen": [65535] * 16, "odd7": [4095, B23, 511, 1 << 20, 3, 70000, 255],
}


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("kind", ["typical", "cancellation", "near_2e100", "near_2em100", "mixed", "subnormal"])
def test_within_bound(formats, name, kind):
    rng = np.random.default_rng(zlib.crc32(f"{name} {kind}".encode()))
    umax = np.asarray(SHAPES[name], np.int64)
    R, n = len(umax), 400
    units = rng.integers(0, umax + 1, (n, R))
    units[0] = umax
    if kind == "typical":
        values, p64 = np.exp(rng.standard_normal(n)), rng.random(R) / umax
    elif kind == "cancellation":
        p64 = rng.random(R)
        values = units.astype(np.float64) @ p64 * (1.0 + rng.standard_normal(n) * 1e-15)
    elif kind == "near_2e100":
        values, p64 = (0.5 + 0.5 * rng.random(n)) * 2.0 ** 100, rng.random(R) * 2.0 ** 70
    elif kind == "near_2em100":
        values, p64 = rng.random(n) * 2.0 ** -98, rng.random(R) * 2.0 ** -118
    elif kind == "mixed":
        values, p64 = np.exp(rng.standard_normal(n) * 10), np.exp(rng.standard_normal(R) * 8)
    else:
        values, p64 = rng.random(n) * 2.0 ** -90, rng.random(R) * 2.0 ** -135
    fmt = formats(umax)
    worst = worst_ratio(fmt, units, values, p64)
    assert worst <= 1.0, worst
    assert worst <= 0.5 or kind in ("cancellation", "near_2em100", "subnormal"), worst


@pytest.mark.parametrize("R,rg,groups,umax", [(8, 6, 64, [8000, 163840, 64000, 524288, 900, 400, 8000, 163840]),
                                              (1, 0, 9, [B23]), (2, 1, 1024, [65535, B23]), (3, 1, 12, [1000, 65535, 65535]),
                                              (10, 8, 40, [65535] * 10)])
@pytest.mark.parametrize("kind", ["typical", "cancellation", "mixed"])
def test_grouped_within_bound(formats, R, rg, groups, umax, kind):
    rng = np.random.default_rng(zlib.crc32(f"{R} {rg} {groups} {kind}".encode()))
    umax = np.asarray(umax, np.int64)
    n, own = 400, R - rg
    units = rng.integers(0, umax + 1, (n, R))
    units[0] = umax
    group = rng.integers(0, groups, n)
    p64 = rng.random(rg + own * groups) * (1.0 if kind == "cancellation" else 1e-4)
    if kind == "mixed":
        p64 = np.exp(rng.standard_normal(len(p64)) * 6)
    mine = np.concatenate([np.tile(p64[:rg], (n, 1)), p64[rg + own * group[:, None] + np.arange(own)]], 1)
    values = np.exp(rng.standard_normal(n) * (10 if kind == "mixed" else 1))
    if kind == "cancellation":
        values = (units * mine).sum(1) * (1.0 + rng.standard_normal(n) * 1e-15)
    assert worst_ratio(formats(umax, rg, groups), units, values, p64, group, rg) <= 1.0


def test_aligned_errors_in_both_chains(formats):
    """Truncation of the value and the rounding of two prices with the same sign, a rent that cancels the value: each
    chain and the final sum contribute, and the ratio stays below a quarter (the bound's factor of four)."""
    rng = np.random.default_rng(7)
    n = 1000
    mant = (rng.integers(0, 1 << 10, n).astype(np.uint64) << np.uint64(29)) | np.uint64((1 << 29) - 1)
    values = ((np.uint64(1023 + 20) << np.uint64(52)) | mant).view(np.float64)
    p64 = np.array([1.25 + 2.0 ** -24 + 2.0 ** -40, 1.5 + 2.0 ** -24 + 2.0 ** -40])
    half = np.rint(values / 2 / p64[0]).astype(np.int64)
    units = np.stack([half, np.rint((values - half * p64[0]) / p64[1]).astype(np.int64)], 1)
    units = np.concatenate([units, [[B23, 511]]])      # the widths: a high field of 9 bits beside one of 23
    units[:, 1] = np.minimum(units[:, 1], 511)
    worst = worst_ratio(formats(units.max(0)), units, np.append(values, 1.0), p64)
    assert 0.001 <= worst <= 0.25, worst


def test_swapped_fields_would_fail(formats):
    """The control: prices of a word's two fields exchanged leave the bound."""
    rng = np.random.default_rng(3)
    umax = np.asarray(SHAPES["cluster6"], np.int64)
    units = rng.integers(0, umax + 1, (100, 6))
    assert worst_ratio(formats(umax), units, np.exp(rng.standard_normal(100)), rng.random(6) / umax, swap=True) > 1.0
