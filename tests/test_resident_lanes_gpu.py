"""The cluster-resident kernel gives a job 1, 2, 4 or 8 lanes, as many as its CTA has for its jobs and
no more than its options. Parity with the oracle and with the streaming passes on both sides of each
line, for the K that leave lanes without an option or with a remainder, and for ties between lanes.
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


@pytest.mark.parametrize("J", [1, 32, 33, 64, 65, 128, 129, 257])    # one CTA of 256 threads: 8, 8, 4, 4, 2, 2, 1, 1 lanes
@pytest.mark.parametrize("kmin,kmax", [(1, 1), (2, 2), (3, 3), (9, 9), (33, 33), (1, 17)])
def test_lanes_per_job(J, kmin, kmax):
    rng = np.random.default_rng(1000 * J + 10 * kmin + kmax)
    t = W.random_table(rng, S=2, J=J, R=4 if J % 2 else 3, kmin=kmin, kmax=kmax, umax=6, dyadic=True)
    for j in range(t.S * t.J):      # every third option of a job repeats its first: ties between lanes
        a, b = t.job_off[j], t.job_off[j + 1]
        t.units[a:b:3] = t.units[a]
        t.values[a:b:3] = t.values[a]
    s = esp.Solver(t)
    ref = s.solve(0.3, 12, traces=True)
    esp.esp_debug_resident(s.ctx, 1)
    sol = s.solve(0.3, 12, flags=esp.ESP_FLAG_RESIDENT, traces=True)
    assert s.launches() == 3
    check_solution(t, sol, list(range(t.S)), 0.3, 12, esp.ESP_PRICE_NORMALIZED, esp.ESP_STEP_FIXED)
    for f in ("lam", "sel", "demand", "lambda_trace", "demand_trace", "selhash_trace"):
        assert np.array_equal(getattr(sol, f), getattr(ref, f)), f
