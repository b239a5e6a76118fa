"""A grouped table for whose packed copy there is no memory still loads: the staged pass reads the table itself, with
the same results (allocation failures injected on the host, one at a time)."""

import numpy as np
import pytest

from paper_2608_07971_gb300 import esp
from tests.test_packed_groups_gpu import _lib, table  # noqa: F401

pytestmark = pytest.mark.gpu


def test_staged_pass_without_room_for_the_copy():
    t = table(2, 40, 8, 6, 17, [16, 3, 130, 1, 300], 5000, 3)
    a = esp.Solver(t)
    assert esp.esp_debug_packed_words(a.ctx) > 0
    ref = a.solve(0.3, 8, traces=True)
    a.close()
    staged = failed = 0
    for n in range(60):
        s = esp.Solver()
        esp.esp_debug_fail_alloc(s.ctx, n)
        try:
            s.load(t)
        except Exception:
            failed += 1
            s.close()
            continue
        esp.esp_debug_fail_alloc(s.ctx, -1)
        packed = esp.esp_debug_packed_words(s.ctx) > 0
        sol = s.solve(0.3, 8, traces=True)
        for f in ("lam", "sel", "demand", "lambda_trace", "demand_trace", "selhash_trace"):
            assert np.array_equal(getattr(sol, f), getattr(ref, f)), (n, f)
        s.close()
        if packed:         # every allocation of the load went through
            break
        staged += 1
    assert packed and staged >= 4 and failed >= 10
