"""A host table of wide units (2^23 and more) is planned for the staged pass while its upload and validation run: after
the validation, its first load has no more to do than a load of known offsets. The guess that this takes may be
wrong: the table still gets the pass that its units allow."""

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


def table(seed, S, J, wide=True):
    rng = np.random.default_rng(seed)
    K = rng.permutation(np.resize([1, 2, 3, 7, 20, 60, 150], S * J))
    off = np.concatenate([[0], np.cumsum(K)]).astype(np.int64)
    n = int(off[-1])
    units = rng.integers(0, 1 << 25 if wide else 5000, (n, 6)).astype(np.int32)
    return W.OptionTable(S, J, 6, 6, 6, off, units, np.exp(rng.standard_normal(n)), None,
                         np.full((S, 6), J << 20, np.int64))


def test_planned_before_the_validation():
    ratio = []
    for seed in range(3):
        a, b = table(2 * seed, 8, 16384), table(2 * seed + 1, 8, 16384)      # the same sizes, other offsets
        s = esp.Solver()

        def load(t):
            s.load(t)
            ms = esp.esp_debug_load_profile(s.ctx)[0]
            return ms[5] - ms[4]

        load(a)
        first = load(b)
        known = min(load(b) for _ in range(3))
        ratio.append(first / known)
        assert esp.esp_debug_packed_words(s.ctx) == 0
        s.close()
    assert min(ratio) < 4.0, ratio      # planning after the validation: about 10


@pytest.mark.parametrize("device", [False, True])
def test_wrong_guesses(device):
    """The first rows and the last load of the same offsets are only a guess: one wide unit far behind them, and units
    that change between loads, take the pass that they need."""
    narrow, late, early = (table(7, 2, 3000, wide=False) for _ in range(3))
    late.units[5000, 2] = early.units[0, 2] = 1 << 24
    ref = {}
    for name, t in (("narrow", narrow), ("late", late), ("early", early)):
        f = esp.Solver()
        esp.esp_debug_set_interleave(f.ctx, False)      # the staged pass
        f.load(t)
        ref[name] = f.solve(0.2, 6, traces=True)
        f.close()
    import torch
    s = esp.Solver()
    for name, t in (("early", early), ("narrow", narrow), ("late", late), ("narrow", narrow), ("early", early), ("late", late)):
        if device:
            x = [torch.from_numpy(v).cuda() for v in (t.job_off, t.units, t.values, t.capacity)]
            torch.cuda.synchronize()
            s.load_device(t.S, t.J, 6, 6, 6, x[0], x[1], x[2], None, x[3])
        else:
            s.load(t)
        assert (esp.esp_debug_packed_words(s.ctx) > 0) == (name == "narrow")
        sol = s.solve(0.2, 6, traces=True)
        for f in ("lam", "sel", "demand", "selhash_trace"):
            assert np.array_equal(getattr(sol, f), getattr(ref[name], f)), (name, f)
    s.close()
