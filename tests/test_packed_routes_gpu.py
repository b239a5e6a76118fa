"""The packed passes are no slower than the staged pass they stand in for where a pass scores or writes more than a
plain round does: exact mode, and the final pass of tables with many one- and two-option jobs (device time of the same
solve on the same GPU, the shortest of several)."""

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


def table(S, J, K, R, seed=5):
    rng = np.random.default_rng(seed)
    cnt = np.full(S * J, K) if K > 0 else np.clip(np.floor(rng.random(S * J) ** (-1 / 0.3)), 1, -K).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
    n = int(off[-1])
    units = rng.integers(0, 8001, (n, R), dtype=np.int32)
    return W.OptionTable(S, J, R, R, R, off, units, np.exp(rng.standard_normal(n)), None, np.full((S, R), J * 2000, np.int64))


def best_ms(t, T, flags, packed):
    s = esp.Solver()
    esp.esp_debug_set_stage_f32(s.ctx, packed)
    s.load(t)
    assert (esp.esp_debug_packed_words(s.ctx) > 0) == packed
    ms = [float(s.solve(0.02, T, flags=flags).result["device_ms"][0]) for _ in range(7)]
    s.close()
    return min(ms[2:])


@pytest.mark.parametrize("S,J,K,R", [(256, 2048, 16, 6), (256, 2048, 16, 4), (8, 300, 1000, 6), (8, 4096, 16, 6)])
def test_exact_mode(S, J, K, R):
    t = table(S, J, K, R)
    packed, staged = (best_ms(t, 10, esp.ESP_FLAG_EXACT_ONLY, p) for p in (True, False))
    assert packed <= staged, (packed, staged)


@pytest.mark.parametrize("S,J", [(8, 65536), (4, 16384)])
def test_final_pass_of_short_solves(S, J):
    t = table(S, J, -256, 6)
    packed, staged = (best_ms(t, 1, 0, p) for p in (True, False))
    assert packed <= 0.95 * staged, (packed, staged)
