"""The grid-resident placement solve holds one job per warp, 8, 16 or 32 warps per CTA as the job count needs:
bit for bit the per-round launches on both sides of each line, with units on both sides of the 16-bit
split of its shared sums.
"""

import numpy as np
import pytest

from paper_2608_07971_gb300 import esp
from tests.test_placement_gpu import _lib, random_factors, same_solution  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warps", [8, 16, 32])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("big", [False, True])
def test_job_counts(warps, extra, big):
    import torch
    n = warps * torch.cuda.get_device_properties(0).multi_processor_count + extra
    f = random_factors(n, S=1, J=n, KC=3, N=9)
    if big:
        f.cfg_units[:] = np.random.default_rng(n).integers(0, 1 << 26, f.cfg_units.shape)
        f.cfg_units[0] = 65535
        f.cfg_units[1] = 65536
        f.capacity[:] = 1 << 33
    s = esp.Solver()
    s.load_placement(f)
    ref = s.solve(0.05, 9)
    res = s.solve(0.05, 9, flags=esp.ESP_FLAG_RESIDENT)
    fits = warps < 32 or extra == 0
    assert s.launches() == (4 if fits else 12)
    same_solution(res, ref, fields=("lam", "sel", "demand"))
    s.close()


@pytest.mark.parametrize("R", [6, 8, 16])
def test_one_job_more_than_16_per_sm(R):
    """The jobs are spread over every SM: one more than 16 warps per SM hold costs a round little (with the next power
    of two of warps on half of the SMs, a round of R = 16 took 1.4 times as long). Device time, the shortest of
    several solves."""
    import torch
    n = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    us = []
    for jobs in (n, n + 1):
        f = random_factors(R, S=1, J=jobs, KC=12, N=64, R=R, rg=R - 2)
        s = esp.Solver()
        s.load_placement(f)
        us.append(min(float(s.solve(0.02, 60, flags=esp.ESP_FLAG_RESIDENT).result["device_ms"][0]) for _ in range(6)))
        s.close()
    assert us[1] <= 1.25 * us[0], us
