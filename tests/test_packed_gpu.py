"""The packed evaluation passes (the screen copy in 12 to 36 bytes per option) against the oracle, at the
edges of their layout: option counts around one and two options, the four- and eight-option vectors, whole
warps, the 256-option step and jobs of several steps; every number of unit words; wide units beside narrow
ones; tables large enough for eight options per lane and small ones with four. Plain passes, traced ones and
the persistent pass must give the same bits.
"""

import numpy as np
import pytest

from paper_2608_07971_gb300 import esp, workloads as W

from tests.parity_util import check_solution

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_07971_gb300 import build
    build.build()
    esp.load_library()


def mixed(ks, J, R, seed, umax=5000, S=2):
    """J jobs whose option counts cycle through ks, with duplicates and near ties."""
    rng = np.random.default_rng(seed)
    K = np.tile(np.resize(np.asarray(ks), J), S)
    off = np.zeros(S * J + 1, np.int64)
    np.cumsum(K, out=off[1:])
    n = int(off[-1])
    units = rng.integers(0, umax + 1, size=(n, R)).astype(np.int32)
    units[0] = umax
    values = np.exp(rng.standard_normal(n))
    for j in range(0, S * J, 3):
        a, b = off[j], off[j + 1]
        if b - a >= 2:
            units[b - 1], values[b - 1] = units[a], values[a]
        if b - a >= 4:
            values[a + 2] = np.nextafter(values[a + 1], 9.0)
            units[a + 2] = units[a + 1]
    cap = np.full((S, R), max(1, J * umax // 4), np.int64)
    return W.OptionTable(S, J, R, R, R, off, units, values, None, cap)


def run_all(t, T=12, persist=True, packed=True):
    a = esp.Solver(t)
    assert (esp.esp_debug_packed_words(a.ctx) > 0) == packed
    traced = a.solve(0.3, T, traces=True)
    check_solution(t, traced, list(range(t.S)), 0.3, T, esp.ESP_PRICE_NORMALIZED, esp.ESP_STEP_FIXED)
    plain = a.solve(0.3, T)
    exact = a.solve(0.3, T, flags=esp.ESP_FLAG_EXACT_ONLY)
    sols = [plain, exact]
    if persist:
        esp.esp_debug_set_persistent(a.ctx, 1)
        assert esp.esp_debug_persistent(a.ctx) > 0
        sols.append(a.solve(0.3, T))
        assert a.launches() == 4
    for s in sols:
        assert np.array_equal(s.lam, traced.lam) and np.array_equal(s.sel, traced.sel)
        assert np.array_equal(s.demand, traced.demand)
    a.close()


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 7, 8, 9, 16, 31, 33, 64, 65, 127, 128, 129, 252, 255, 256, 257, 260, 513, 1025])
@pytest.mark.parametrize("J", [3, 77])
def test_one_option_count(K, J):
    run_all(mixed([K], J, 6, K))


@pytest.mark.parametrize("J", [50, 700])
def test_ragged(J):
    run_all(mixed([1, 2, 3, 5, 16, 17, 40, 100, 129, 200, 256, 257, 700, 1, 8, 2], J, 6, 5))


def test_wide_steps_with_several_tiles_per_warp():
    """More than a step per warp of the launch: eight options per lane, several steps per tile."""
    run_all(mixed([16], 8192, 6, 3, S=12), T=4)
    run_all(mixed([12, 20, 36, 68, 5, 1, 2, 300], 16384, 6, 4, S=2), T=3)


@pytest.mark.parametrize("R", [1, 2, 3, 5, 7, 8, 11, 16])
@pytest.mark.parametrize("umax", [1, 5000, 65535, (1 << 23) - 1])
def test_unit_words(R, umax):
    """2 to 8 unit words (over eight columns of 23 bits need more: the staged pass takes those)."""
    run_all(mixed([16, 3, 130, 1], 40, R, 100 * R + 1, umax=umax), T=6, persist=R == 8,
            packed=R <= 8 or umax <= 65535)


@pytest.mark.parametrize("R,words", [(4, 2), (6, 3), (8, 4), (12, 6), (16, 8)])
def test_every_word_count_of_the_persistent_pass(R, words):
    """Tables that take the persistent pass by default, for each instantiation of it."""
    t = mixed([32], 16384, R, R, umax=65535, S=8)
    s = esp.Solver(t)
    assert esp.esp_debug_packed_words(s.ctx) == words and esp.esp_debug_persistent(s.ctx) > 0
    a = s.solve(0.3, 3)
    assert s.launches() == 4
    esp.esp_debug_set_persistent(s.ctx, 0)
    b = s.solve(0.3, 3)
    assert s.launches() == 3 + 3
    assert np.array_equal(a.lam, b.lam) and np.array_equal(a.sel, b.sel) and np.array_equal(a.demand, b.demand)
    s.close()


def test_large_table_of_other_widths_takes_the_persistent_pass():
    t = mixed([32], 16384, 5, 9, S=16)
    s = esp.Solver(t)
    assert esp.esp_debug_persistent(s.ctx) > 0
    a = s.solve(0.3, 3)
    assert s.launches() == 4
    esp.esp_debug_set_persistent(s.ctx, 0)
    b = s.solve(0.3, 3)
    assert s.launches() == 3 + 3
    assert np.array_equal(a.lam, b.lam) and np.array_equal(a.sel, b.sel) and np.array_equal(a.demand, b.demand)
    s.close()
