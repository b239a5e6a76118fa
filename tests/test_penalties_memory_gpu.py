"""Device memory that esp_set_penalties keeps with the table: the loaded values and the inputs that were given, no more."""

import numpy as np
import pytest

from paper_2608_07971_gb300 import esp

pytestmark = pytest.mark.gpu


def test_only_given_inputs_take_memory():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_07971_gb300 import build
    build.build()
    S, J, K, R = 8, 65536, 16, 2
    n = S * J * K
    rng = np.random.default_rng(1)
    units = torch.from_numpy(rng.integers(0, 1000, (n, R)).astype(np.int32)).cuda()
    values = torch.from_numpy(np.exp(rng.standard_normal(n))).cuda()
    off = torch.arange(S * J + 1, dtype=torch.int64, device="cuda") * K
    cap = torch.full((S, R), J * 300, dtype=torch.int64, device="cuda")
    s = esp.Solver()
    torch.cuda.synchronize()
    s.load_device(S, J, R, R, R, off, units, values, None, cap)
    mb = 1 << 20

    def taken(call):
        before = torch.cuda.mem_get_info()[0]
        call()
        return (before - torch.cuda.mem_get_info()[0]) / mb

    cur, sh, tau = np.zeros(S * J, np.int32), np.full(n, 1.5), np.full(S * J, 1.2)
    values_mb, jobs_mb, slack = 8 * n / mb, S * J / mb, 8.0      # 64 MB; mappings of 2 MB
    assert taken(lambda: esp.esp_set_penalties(s.ctx, 0.05, cur, 0.0, None, None)) <= values_mb + 4 * jobs_mb + slack
    assert taken(lambda: esp.esp_set_penalties(s.ctx, 0.05, cur, 0.3, sh, tau)) <= values_mb + 8 * jobs_mb + slack
    assert taken(lambda: esp.esp_set_penalties(s.ctx, 0.05, cur, 0.3, sh, tau)) <= 0.0
    s.close()
