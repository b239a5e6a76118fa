"""The largest uniform tables that the cluster-resident kernel holds (16 CTAs per scenario, every slice filling a
CTA's shared memory with its jobs at a pitch of a multiple of 32): one option per job more is refused. Parity
with the streaming passes there, for 1 to 8 lanes per job.
"""

import numpy as np
import pytest

from paper_2608_07971_gb300 import esp, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_07971_gb300 import build
    build.build()
    esp.load_library()


def table(J, K, R, seed):
    rng = np.random.default_rng(seed)
    n = J * K
    units = rng.integers(0, 9000, size=(n, R)).astype(np.int32)
    values = np.exp(rng.standard_normal(n))
    values[5::7] = values[4::7][:len(values[5::7])]      # ties and repeats between the lanes of a job
    units[5::7] = units[4::7][:len(units[5::7])]
    off = np.arange(J + 1, dtype=np.int64) * K
    return W.OptionTable(1, J, R, R, R, off, units, values, None, np.full((1, R), J * 1500, np.int64))


@pytest.mark.parametrize("R,J,K", [(4, 2048, 73), (4, 1024, 147), (4, 512, 294), (6, 4096, 27), (6, 2048, 55), (6, 1024, 110),
                                   (6, 512, 221), (8, 2048, 44), (8, 1024, 88), (8, 512, 176)])
def test_largest_slices(R, J, K):
    s = esp.Solver(table(J, K, R, K))
    ref = s.solve(0.1, 8, traces=True)
    assert esp.esp_debug_resident(s.ctx, 16)[0] == 16
    sol = s.solve(0.1, 8, flags=esp.ESP_FLAG_RESIDENT, traces=True)
    assert s.launches() == 3
    for f in ("lam", "sel", "demand", "lambda_trace", "demand_trace", "selhash_trace"):
        assert np.array_equal(getattr(sol, f), getattr(ref, f)), f
    s.close()
    s = esp.Solver(table(J, K + 1, R, K))
    with pytest.raises(Exception):
        if esp.esp_debug_resident(s.ctx, 16) is None:
            raise RuntimeError("cannot run resident")
    s.close()
