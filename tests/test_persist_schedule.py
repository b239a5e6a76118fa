"""The persistent pass's hand-out and release protocol, modelled on the host (no GPU): it always completes, under
any interleaving of the warps.

The model follows k_packed_persist and run_warp (csrc/esp_packed.cu) step by step, with the arithmetic left out:
- work items q = 0, 1, ... are (round q / n_tiles, tile q mod n_tiles), the tiles listed by scenario, taken from one
  counter in increasing order. A warp reserves its next index one take ahead; from its entry on it holds the item it
  evaluates, the one after it, and one index beyond (an index past the last item is never replaced);
- before it turns to an item it leaves the one before: the arrival of that tile for its scenario and round
  (`leave`), and only then waits until the new item's scenario has had as many price updates as the item's round
  (`wait_version`), reads the prices (`enter`) and evaluates; after its last item it leaves that one too;
- the arrival that completes a scenario's tiles for a round applies the price update: round r + 1 is released
  (ver = r + 1), or the scenario stops (frozen, and every later round released at once: its tiles are skipped and
  do not arrive).
Warps advance one action at a time in a random order (any interleaving the hardware could produce). The model
checks that every run ends with every scenario released for every round or stopped, that a tile is evaluated at its
round's prices (ver equal to the round, since the scenario cannot advance without it), that each round of a
scenario gets exactly its tiles, and, as a control, that the order the kernel avoids (waiting for the next item's
scenario before the arrival of the one before) deadlocks."""

import numpy as np
import pytest

STOPPED = 1 << 30   # kVerStopped


def simulate(rng, scen_tiles, T, W, stop=None, leave_first=True):
    """scen_tiles: tiles of each scenario; stop[s]: the round whose update stops it (or none). Returns (completed,
    arrivals per scenario and round, ver)."""
    S = len(scen_tiles)
    scen = np.repeat(np.arange(S), scen_tiles)
    n_tiles, Q = len(scen), T * len(scen)
    counter = 0
    arrivals = np.zeros((S, T), int)
    ver, frozen = np.zeros(S, int), np.zeros(S, bool)

    def reserve():
        nonlocal counter
        counter += 1
        return counter - 1

    def take(w):
        q = w["pend"]
        if q >= Q:
            return None
        w["pend"] = reserve()
        return int(scen[q % n_tiles]), q // n_tiles

    def leave(w):
        if w["at"] is None:
            return
        s, r, skipped = w["at"]
        w["at"] = None
        if skipped:
            return
        arrivals[s, r] += 1
        assert arrivals[s, r] <= scen_tiles[s]
        if arrivals[s, r] == scen_tiles[s]:          # this arrival's warp applies the update
            assert ver[s] == r and not frozen[s]
            frozen[s] = stop is not None and stop[s] == r
            ver[s] = STOPPED if frozen[s] else r + 1

    warps = []
    for _ in range(W):
        w = {"at": None, "done": False, "left": False}
        w["pend"] = reserve()
        warps.append(w)
    for k in rng.permutation(W):                     # entry: the first item and the one after it
        w = warps[k]
        w["item"] = take(w)
        w["next"] = take(w) if w["item"] is not None else None
        w["done"] = w["item"] is None
    while True:
        live = [w for w in warps if not w["done"]]
        if not live:
            return True, arrivals, ver
        moved = False
        for k in rng.permutation(len(live)):
            w = live[k]
            if w["item"] is None:                    # after its last item
                leave(w)
                w["done"] = moved = True
                break
            if leave_first and w["at"] is not None:
                leave(w)
                moved = True
                break
            s, r = w["item"]
            if ver[s] < r:                           # waits for the prices of round r
                continue
            leave(w)                                 # (the control's order; the kernel has left already)
            assert frozen[s] or ver[s] == r
            w["at"] = (s, r, bool(frozen[s]))
            w["item"] = w["next"]
            w["next"] = take(w) if w["next"] is not None else None
            moved = True
            break
        if not moved:
            return False, arrivals, ver              # every live warp waits: deadlock


@pytest.mark.parametrize("seed", range(40))
def test_every_interleaving_completes(seed):
    rng = np.random.default_rng(seed)
    S, T, W = int(rng.integers(1, 9)), int(rng.integers(1, 7)), int(rng.integers(1, 24))
    tiles = rng.integers(1, 40, S)
    ok, arrivals, ver = simulate(rng, tiles, T, W)
    assert ok, "deadlock"
    assert np.array_equal(arrivals, np.repeat(tiles[:, None], T, axis=1))
    assert np.all(ver == T)


@pytest.mark.parametrize("seed", range(40))
def test_stopped_scenarios_release_their_later_rounds(seed):
    rng = np.random.default_rng(1000 + seed)
    S, T, W = int(rng.integers(1, 9)), int(rng.integers(1, 7)), int(rng.integers(1, 24))
    tiles, stop = rng.integers(1, 20, S), rng.integers(0, T + 2, S)      # T and more: never stops
    ok, arrivals, ver = simulate(rng, tiles, T, W, stop)
    assert ok, "deadlock"
    for s in range(S):
        rounds = min(int(stop[s]) + 1, T)
        assert np.all(arrivals[s, :rounds] == tiles[s]) and np.all(arrivals[s, rounds:] == 0)
        assert ver[s] == (STOPPED if stop[s] < T else T)


def test_one_scenario_and_more_warps_than_items():
    rng = np.random.default_rng(99)
    for tiles, T, W in (([64], 5, 40), ([1], 6, 9), ([3, 1, 2], 4, 64), ([30] * 16, 3, 3)):
        for _ in range(3):
            ok, _, ver = simulate(rng, np.asarray(tiles), T, W)
            assert ok and np.all(ver == T)


def test_waiting_before_leaving_deadlocks():
    """The control: a warp that waits for its next item's scenario while still holding the arrival of the item before
    can block the release it waits for."""
    rng = np.random.default_rng(7)
    dead = sum(not simulate(rng, np.asarray([2, 3]), 4, 2, leave_first=False)[0] for _ in range(40))
    assert dead > 0
