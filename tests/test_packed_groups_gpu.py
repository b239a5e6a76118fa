"""The packed evaluation passes of tables with a group column against the oracle and the staged pass: one
and two columns per group, none to many priced alike, one group to the largest price table, the group slot in
bits that a word leaves free and in a word of its own, and the option counts at the edges of the steps.
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


def run_all(t, T=10, kind=1):
    a = esp.Solver(t)
    assert esp.esp_debug_pass_kernel(a.ctx) == kind and (esp.esp_debug_packed_words(a.ctx) > 0) == (kind == 1)
    b = esp.Solver()
    esp.esp_debug_set_interleave(b.ctx, False)      # the staged pass
    b.load(t)
    assert esp.esp_debug_pass_kernel(b.ctx) == 0
    for mode, eta in ((esp.ESP_PRICE_NORMALIZED, 0.3), (esp.ESP_PRICE_RAW, 1e-4)):
        traced = a.solve(eta, T, mode=mode, traces=True)
        check_solution(t, traced, list(range(t.S)), eta, T, mode, esp.ESP_STEP_FIXED)
        staged = b.solve(eta, T, mode=mode, traces=True)
        for f in ("lam", "sel", "demand", "lambda_trace", "demand_trace", "selhash_trace"):
            assert np.array_equal(getattr(traced, f), getattr(staged, f)), f
        for flags in (0, esp.ESP_FLAG_EXACT_ONLY, esp.ESP_FLAG_PER_ROUND_LAUNCH):
            s = a.solve(eta, T, mode=mode, flags=flags)
            assert np.array_equal(s.lam, traced.lam) and np.array_equal(s.sel, traced.sel)
            assert np.array_equal(s.demand, traced.demand)
    a.close()
    b.close()


def table(S, J, R, rg, groups, ks, umax, seed):
    rng = np.random.default_rng(seed)
    K = np.tile(np.resize(np.asarray(ks), J), S)
    off = np.zeros(S * J + 1, np.int64)
    np.cumsum(K, out=off[1:])
    n = int(off[-1])
    units = rng.integers(0, np.resize(np.asarray(umax), R) + 1, size=(n, R)).astype(np.int32)
    units[0] = np.resize(np.asarray(umax), R)
    values = np.exp(rng.standard_normal(n))
    group = rng.integers(0, groups, size=n).astype(np.uint16)
    group[-1] = groups - 1
    for j in range(0, S * J, 3):      # a duplicate, a tie in another group, a near tie
        a, b = off[j], off[j + 1]
        if b - a >= 2:
            units[b - 1], values[b - 1], group[b - 1] = units[a], values[a], group[a]
        if b - a >= 4:
            units[a + 2], values[a + 2] = units[a + 1], np.nextafter(values[a + 1], 9.0)
        if b - a >= 5:
            units[a + 3], values[a + 3], group[a + 3] = units[a], values[a], (group[a] + 1) % groups
    P = rg + (R - rg) * groups
    cap = np.maximum(1, np.resize(np.resize(np.asarray(umax), R), P).astype(np.int64) * J // 4)
    cap[rg:] = np.maximum(1, cap[rg:] // groups)
    return W.OptionTable(S, J, R, P, rg, off, units, values, group, np.tile(cap, (S, 1)))


@pytest.mark.parametrize("R,rg,groups", [(1, 0, 1), (1, 0, 1024), (2, 0, 9), (2, 1, 8), (8, 6, 500), (5, 4, 33), (8, 6, 64),
                                         (8, 6, 17), (9, 8, 5), (10, 8, 40)])
@pytest.mark.parametrize("umax", [1, 5000, (8000, 250000, 60000, 500000, 1000, 500, 8000, 250000)])
def test_widths(R, rg, groups, umax):
    run_all(table(2, 40, R, rg, groups, [16, 3, 130, 1, 300], umax, 31 * R + groups), T=6)


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 8, 9, 64, 129, 255, 256, 257, 513, 768, 1030])
@pytest.mark.parametrize("J", [3, 77])
def test_option_counts(K, J):
    run_all(table(2, J, 6, 4, 12, [K], 5000, K))


@pytest.mark.parametrize("R,rg,groups,umax", [(6, 3, 4, 100), (3, 1, 512, 100), (2, 0, 3, (1 << 23) - 1), (11, 10, 3, 1 << 20)])
def test_tables_left_to_the_staged_pass(R, rg, groups, umax):
    """Three columns per group, over 1024 prices, a group pair or a word count that does not fit."""
    run_all(table(1, 30, R, rg, groups, [16, 3, 130, 1, 300], umax, R), T=5, kind=0)


def test_several_tiles_per_warp():
    run_all(table(3, 6000, 8, 6, 64, [64, 192, 5, 300], 5000, 8), T=3)


def test_stopping_rule_and_frozen_scenarios():
    t = table(3, 50, 4, 2, 6, [20, 300], 500, 3)
    a = esp.Solver(t)
    traced = a.solve(0.05, 60, tol=2e-2, traces=True)
    plain = a.solve(0.05, 60, tol=2e-2)
    assert np.array_equal(plain.lam, traced.lam) and np.array_equal(plain.demand, traced.demand)
    check_solution(t, traced, [0, 1, 2], 0.05, 60, esp.ESP_PRICE_NORMALIZED, esp.ESP_STEP_FIXED, tol=2e-2)
    a.close()
