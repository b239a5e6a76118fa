"""Timed cases of the ESP solver and the IAC predictor: what a scheduler's program asks of them.

A case is a dict of plain sizes and options. ``listed()`` holds the named cases, ``draw(rng)`` one more of
the same ranges. ``prepare`` makes the inputs on the GPU from the seed (the distributions of
``paper_2608_07971_gb300.workloads``: GPU share, memory, CPU, host memory, NVLink and network of elastic
jobs, log-normal values) and the context that a program keeps; ``run`` is one pass through the public
calls with every result that such a program reads; ``exact`` is the same in plain 64-bit torch.

Kinds:
  solve      a loaded option table solved (a what-if batch, one cluster, a ragged cluster snapshot)
  epoch      one scheduling epoch: this epoch's table from host memory, a few warm-started rounds, the
             prices, selection and demand read back
  replan     one outer round of the ESP-IAC loop: new Gamma penalties on a loaded table, a short
             warm-started solve, the results read back
  placement  configurations x nodes, as an expanded (grouped) table or in factored form
  iac        slowdown predictions of co-location pairs, on device tensors or host arrays
"""

import math

import numpy as np
import torch

from paper_2608_07971_gb300 import esp, workloads

DEV = "cuda"
# capacities of a 512-GPU cluster of 2048 jobs (milli-GPU, MiB, millicores, MiB, NVLink, network), then
# two more resources of wider rows; per-job share scales with the number of jobs
CAP_512 = [512000, 512 * 81920, 4096000, 512 * 1048576, 512 * 900, 512 * 400, 512 * 3000, 512 * 250]
NODES, CAP_NODE = 64, [8000, 8 * 81920]


def listed():
    return [
        # the online use: a 64-GPU cluster's epoch, 200 active jobs, five warm-started rounds
        dict(name="epoch", kind="epoch", S=1, J=200, K=8, R=4, T=5, mode=1, step=0, flags=0),
        # one small cluster from cold prices to convergence: rounds of a few microseconds each
        dict(name="tiny_cluster", kind="solve", S=1, J=64, K=8, R=4, T=200, mode=1, step=0, flags=0),
        # one 512-GPU cluster, plain call
        dict(name="cluster_512", kind="solve", S=1, J=2048, K=16, R=6, T=500, mode=1, step=0, flags=0),
        # the same cluster with its table held on chip for the whole solve
        dict(name="cluster_512_resident", kind="solve", S=1, J=2048, K=16, R=6, T=500, mode=1, step=0,
             flags=esp.ESP_FLAG_RESIDENT),
        # snapshots of a cluster whose jobs have ragged option lists, odd sizes, prices in stored units and
        # a diminishing step
        dict(name="ragged_odd", kind="solve", S=7, J=1777, K=-96, R=5, T=150, mode=0, step=1, flags=0),
        # a capacity-planning batch: 1024 variants of the 512-GPU cluster
        dict(name="whatif_batch", kind="solve", S=1024, J=2048, K=16, R=6, T=300, mode=1, step=0, flags=0),
        # large clusters with heavy-tailed option counts (Zipf 1.3, at most 256)
        dict(name="heavy_tail", kind="solve", S=16, J=65536, K=-256, R=6, T=300, mode=1, step=0, flags=0),
        # configurations x nodes as an expanded table with a group column
        dict(name="placement_table", kind="placement", form="table", S=1, J=4096, KC=12, N=64, T=100, flags=0),
        # the same in factored form, all rounds in one launch
        dict(name="placement_factored", kind="placement", form="factored", S=1, J=4096, KC=12, N=64, T=400,
             flags=esp.ESP_FLAG_RESIDENT),
        # an outer round of the ESP-IAC loop on the 512-GPU cluster
        dict(name="replan", kind="replan", S=1, J=2048, K=16, R=6, T=20, mode=1, step=0, flags=0),
        # slowdowns of every option of a what-if batch against its co-located partner
        dict(name="iac_whatif", kind="iac", S=1024, J=2048, K=16, H=64, host=False, path=0),
        # slowdowns of one epoch's pairs, host arrays in and out
        dict(name="iac_epoch", kind="iac", S=1, J=200, K=8, H=48, host=True, path=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "ragged", "ragged", "epoch", "replan", "placement", "iac", "iac"])
    R = rng.choice([3, 4, 5, 6, 6, 8])
    mode, step = rng.choice([0, 1, 1]), rng.choice([0, 0, 1])
    if kind in ("solve", "ragged"):
        K = rng.choice([1, 2, 4, 7, 8, 12, 16, 16, 24, 32]) if kind == "solve" else -_log(rng, 8, 256)
        S, J = _log(rng, 1, 1024), _log(rng, 40, 20000)
        mean = K if K > 0 else 1 + abs(K) // 5
        while S * J * mean > 20_000_000:
            S, J = max(1, S // 2), J
            if S == 1 and J * mean > 20_000_000:
                J //= 2
        T = max(10, min(400, int(3e9 / (S * J * mean))))
        return dict(kind="solve", S=S, J=J, K=K, R=R, T=T, mode=mode, step=step,
                    flags=rng.choice([0, 0, esp.ESP_FLAG_RESIDENT]))
    if kind == "epoch":
        return dict(kind="epoch", S=1, J=_log(rng, 20, 4000), K=rng.choice([4, 6, 8, 16, -20]), R=R,
                    T=rng.randint(3, 10), mode=mode, step=step, flags=0)
    if kind == "replan":
        return dict(kind="replan", S=rng.randint(1, 8), J=_log(rng, 50, 4000), K=rng.choice([4, 8, 16, -40]), R=R,
                    T=rng.randint(5, 40), mode=mode, step=step, flags=0)
    if kind == "placement":
        form = rng.choice(["table", "factored", "factored"])
        return dict(kind="placement", form=form, S=rng.randint(1, 2), J=_log(rng, 100, 2200), KC=rng.randint(3, 16),
                    N=rng.randint(5, 64), T=rng.randint(20, 200), flags=rng.choice([0, esp.ESP_FLAG_RESIDENT]))
    host = rng.random() < 0.4
    S = 1 if host else _log(rng, 1, 512)
    return dict(kind="iac", S=S, J=_log(rng, 20, 2000), K=rng.choice([5, 8, 16]), H=rng.choice([16, 24, 32, 48, 64]),
                host=host, path=rng.choice([0, 0, 0, 1]))


# ---- inputs -----------------------------------------------------------------------------------------

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) & 0x7fffffff)


def _ints(g, lo, hi, shape):
    return torch.randint(lo, hi + 1, shape, generator=g, device=DEV)


def _uni(g, shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _counts(g, n, K):
    """Options of each job: K, or for K < 0 min(-K, Zipf(1.3))."""
    if K > 0:
        return torch.full((n,), K, dtype=torch.int64, device=DEV)
    k = np.arange(1, 100000, dtype=np.float64) ** -1.3
    cdf = torch.from_numpy(np.cumsum(k[:-K - 1]) / (k.sum() + 100000.0 ** -0.3 / 0.3)).to(DEV)
    return torch.clamp(torch.searchsorted(cdf, _uni(g, (n,)), right=True) + 1, max=-K)


def _table(case, seed):
    """(job_off, units, values, capacity) of a synthetic cluster on the GPU; see workloads._configs."""
    S, J, R = case["S"], case["J"], case["R"]
    g = _gen(seed, 1)
    cnt = _counts(g, S * J, case["K"])
    off = torch.zeros(S * J + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(cnt, 0, out=off[1:])
    n = int(off[-1])
    job = torch.repeat_interleave(torch.arange(S * J, device=DEV), cnt)
    base = torch.exp(torch.randn(S * J, generator=g, device=DEV, dtype=torch.float64))
    lims = [(1024, 163840), (1000, 64000), (4096, 524288), (0, 900), (0, 400), (0, 4000), (1, 300)]
    per = [_ints(g, lo, hi, (S * J,)) for lo, hi in lims]
    share = 1000 * _ints(g, 1, 8, (n,))
    ck = torch.rand(n, generator=g, device=DEV) < 0.5
    frac = share.double() / 8000.0
    units = torch.empty((n, R), dtype=torch.int32, device=DEV)
    units[:, 0] = share.int()
    for c in range(1, R):
        x = per[c - 1][job].double()
        if c == 1:
            x = torch.where(ck, torch.clamp(torch.round(x * (0.4 + 0.6 * _uni(g, (n,)))), min=1), x)
        elif c == 2:
            x = torch.clamp(torch.round(x * frac), min=1000)
        elif c >= 4:
            x = torch.round(x * frac)
        units[:, c] = x.int()
    values = base[job] * torch.sqrt(frac) * torch.where(ck, 0.7 + 0.3 * _uni(g, (n,)), torch.ones((), device=DEV))
    if case["K"] > 0:   # the cluster's capacities, varied by 20%
        cap = torch.tensor(CAP_512[:R], dtype=torch.float64, device=DEV) * (J / 2048.0)
        cap = cap[None, :] * (0.8 + 0.4 * _uni(g, (S, R)))
    else:               # oversubscribed: 60% of the jobs' mean demand (whole-number sums)
        cap = torch.empty((S, R), dtype=torch.float64, device=DEV)
        scen = torch.div(job, J, rounding_mode="floor")
        for c in range(R):
            w = torch.div(units[:, c].long(), cnt[job], rounding_mode="floor")
            cap[:, c] = 0.6 * torch.zeros(S, dtype=torch.int64, device=DEV).index_add_(0, scen, w).double()
    return off, units, values, torch.clamp(torch.round(cap), min=1).long()


def _eta(case, cap):
    """Step size: 0.02 of the capacity (normalized prices), or the same step in stored units."""
    if case["mode"] == 1:
        return 0.02
    c = float(cap.double().mean())
    return 0.005 / (c * c)


def _pinned(shape, dtype):
    t = torch.empty(shape, dtype=dtype, pin_memory=True)
    return t.numpy()


def _outputs(S, J, P):
    return dict(res=np.zeros(S, esp.RESULT_DTYPE), lam=_pinned((S, P), torch.float64),
                sel=_pinned((S, J), torch.int32), dem=_pinned((S, P), torch.int64))


def _placement(case, seed):
    S, J, KC, N = case["S"], case["J"], case["KC"], case["N"]
    c = dict(case, K=KC, R=6)
    _, units, values, cap = _table(c, seed)
    g = _gen(seed, 2)
    u = torch.cat([units, units[:, :2]], 1).reshape(S * J, KC, 8)
    sens = torch.rand(S * J, generator=g, device=DEV)
    jt, nt = _ints(g, 0, NODES - 1, (S * J,)), _ints(g, 0, NODES - 1, (N,))
    d = torch.sort(torch.rand((NODES, NODES, 9), generator=g, device=DEV), dim=2)[0][:, :, 1]   # Beta(2, 8)
    d = torch.triu(d) + torch.triu(d, 1).T
    node_cap = torch.tensor(CAP_NODE, device=DEV).repeat(N)[None, :].expand(S, -1)
    cap = torch.cat([cap, node_cap], 1).contiguous()
    return u.contiguous(), values.reshape(S * J, KC), sens, jt.int(), nt.int(), d.contiguous(), cap


def _placement_options(p, case):
    """The expanded options: units (n, 8), values, group."""
    u, v, sens, jt, nt, d, _ = p
    n_jobs, KC, N = u.shape[0], case["KC"], case["N"]
    pen = sens[:, None] * d[jt.long()][:, nt.long()]          # fp32, rounded once
    values = (v[:, :, None] - pen[:, None, :].double()).reshape(-1)
    units = u[:, :, None, :].expand(-1, -1, N, -1).reshape(-1, 8).contiguous()
    group = torch.arange(N, device=DEV, dtype=torch.int16).repeat(n_jobs * KC)
    return units, values.contiguous(), group


def _pairs(case, seed):
    S, J, K = case["S"], case["J"], case["K"]
    g = _gen(seed, 3)
    j = torch.arange(J, device=DEV)
    partner = (j[None, :] + 1 + _ints(g, 0, max(J - 2, 0), (S, J))) % J
    pr = partner * K + _ints(g, 0, K - 1, (S, J))
    out = torch.empty((S, J, K, 2), dtype=torch.int32, device=DEV)
    out[..., 0] = (j[:, None] * K + torch.arange(K, device=DEV)[None, :]).int()[None]
    out[..., 1] = pr.int()[:, :, None]
    return out.reshape(-1, 2)


class _State(dict):
    """A program's state; the library's handles are closed with it."""

    def __del__(self):
        for k in ("solver", "pred"):
            if k in self:
                try:
                    self[k].close()
                except Exception:
                    pass


def prepare(case, seed):
    kind = case["kind"]
    st = _State(case=case)
    if kind == "iac":
        model = workloads.iac_model(int(seed), case["H"])
        rows = torch.from_numpy(workloads.iac_rows(int(seed), case["J"], case["K"]))
        pairs = _pairs(case, seed)
        st["pred"] = esp.Predictor(model, stream=torch.cuda.current_stream().cuda_stream, path=case["path"])
        if case["host"]:
            st.update(rows=rows.numpy(), pairs=pairs.cpu().numpy())
        else:
            st.update(rows=rows.to(DEV), pairs=pairs, out=torch.empty(pairs.shape[0], device=DEV))
        torch.cuda.synchronize()
        return st
    S, J, T = case["S"], case["J"], case["T"]
    if kind == "epoch":     # the simplest program: the default stream, the table in ordinary host memory
        st["solver"] = esp.Solver()
        off, units, values, cap = _table(case, seed)
        st["table"] = workloads.OptionTable(S, J, case["R"], case["R"], case["R"], off.cpu().numpy(),
                                            units.cpu().numpy(), values.cpu().numpy(), None, cap.cpu().numpy())
        st["eta"] = _eta(case, cap)
        st["lambda0"] = _warm(case, seed, cap)
        torch.cuda.synchronize()
        return st
    st["stream"] = torch.cuda.Stream()
    st["solver"] = sv = esp.Solver(stream=st["stream"].cuda_stream)
    torch.cuda.synchronize()
    if kind == "placement":
        N, R, rg = case["N"], 8, 6
        P = rg + (R - rg) * N
        p = _placement(case, seed)
        if case["form"] == "table":
            units, values, group = _placement_options(p, case)
            off = torch.arange(S * J + 1, device=DEV) * (case["KC"] * N)
            torch.cuda.synchronize()
            sv.load_device(S, J, R, P, rg, off, units, values, group, p[6])
        else:
            h = [x.cpu().numpy() for x in p]
            sv.load_placement(workloads.PlacementFactors(S, J, case["KC"], N, R, rg, h[0], h[1], h[2], h[3], h[4],
                                                         h[5], h[6]))
        st["prm"] = sv.params(0.02, T, mode=esp.ESP_PRICE_NORMALIZED, flags=case["flags"])
        st.update(_outputs(S, J, P))
        return st
    R = case["R"]
    off, units, values, cap = _table(case, seed)
    torch.cuda.synchronize()
    sv.load_device(S, J, R, R, R, off, units, values, None, cap)
    if kind == "replan":
        st["lambda0"] = _warm(case, seed, cap)
        st["c_cur"], st["s_hat"], st["tau"] = _penalty_inputs(case, seed, off)
        st["prm"] = sv.params(_eta(case, cap), T, mode=case["mode"], step=case["step"], flags=case["flags"],
                              lambda0=st["lambda0"])
    else:
        st["prm"] = sv.params(_eta(case, cap), T, mode=case["mode"], step=case["step"], flags=case["flags"])
    st.update(_outputs(S, J, R))
    return st


def _warm(case, seed, cap):
    """Prices of an earlier solve: of order 0.1 per capacity."""
    g = _gen(seed, 4)
    lam = 0.1 * torch.randn((case["S"], case["R"]), generator=g, device=DEV, dtype=torch.float64).abs()
    if case["mode"] == 0:
        lam = lam / cap.double()
    return lam.cpu().numpy()


GAMMA0, ALPHA = 0.05, 0.3


def _penalty_inputs(case, seed, off):
    """Current configurations (some jobs are new), predicted slowdowns and tolerance thresholds."""
    g = _gen(seed, 5)
    cnt = off[1:] - off[:-1]
    n = cnt.shape[0]
    cur = torch.minimum((_uni(g, (n,)) * cnt).long(), cnt - 1)
    cur = torch.where(_uni(g, (n,)) < 0.1, torch.full_like(cur, -1), cur).int()
    s_hat = 1.0 + torch.clamp(0.4 * torch.randn(int(off[-1]), generator=g, device=DEV, dtype=torch.float64), min=0)
    tau = 1.0 + 0.5 * _uni(g, (n,))
    return cur.cpu().numpy(), s_hat.cpu().numpy(), tau.cpu().numpy()


# ---- one pass ---------------------------------------------------------------------------------------

def _record(lam, sel, dem, res):
    return dict(prices=lam, selection=sel, demand=dem, rounds=res["rounds_run"], feasible=res["feasible"],
                primal=res["primal"], dual=res["dual"])


def run(state):
    kind = state["case"]["kind"]
    if kind == "iac":
        out = state["pred"].predict(state["rows"], state["pairs"], workloads.IAC_C_MEM, state.get("out"))
        return dict(s_hat=out)
    c, sv = state["case"], state["solver"]
    if kind == "epoch":
        sv.load(state["table"])
        s = sv.solve(state["eta"], c["T"], mode=c["mode"], step=c["step"], flags=c["flags"],
                     lambda0=state["lambda0"])
        return _record(s.lam, s.sel, s.demand, s.result)
    if kind == "replan":
        esp.esp_set_penalties(sv.ctx, GAMMA0, state["c_cur"], ALPHA, state["s_hat"], state["tau"])
    esp.esp_solve(sv.ctx, state["prm"], state["res"])
    esp.esp_get_prices(sv.ctx, state["lam"])
    esp.esp_get_selection(sv.ctx, state["sel"])
    esp.esp_get_demand(sv.ctx, state["dem"])
    return _record(state["lam"], state["sel"], state["dem"], state["res"])


# ---- what a pass cannot do without, and how exact it is ---------------------------------------------

def _mean_count(K):
    """Expected options of a job."""
    if K > 0:
        return float(K)
    k = np.arange(1, 100000, dtype=np.float64)
    z = (k ** -1.3).sum() + 100000.0 ** -0.3 / 0.3
    p = k[:-K - 1] ** -1.3 / z
    return float((k[:-K - 1] * p).sum() + -K * (1.0 - p.sum()))


def work(case):
    """Inputs read once, outputs written once; the multiply-adds of every round. The table is counted
    once: rounds that read it again do so because it does not fit on chip."""
    if case["kind"] == "iac":
        H, n = case["H"], case["S"] * case["J"] * case["K"]
        return {"bytes": 12 * n + 56 * case["J"] * case["K"], "flops": n * 2.0 * (36 * H + H * H + H)}
    S, J, T = case["S"], case["J"], case["T"]
    if case["kind"] == "placement":
        KC, N = case["KC"], case["N"]
        n, P = S * J * KC * N, 6 + 2 * N
        b = n * 42 if case["form"] == "table" else S * J * (KC * 40 + 8)
        return {"bytes": b + S * P * 24 + S * J * 4, "flops": n * 16.0 * (T + 1)}
    n, R = S * J * _mean_count(case["K"]), case["R"]
    b = n * (4 * R + 8) + S * J * 12 + S * R * 24
    if case["kind"] == "replan":
        b += n * 8 + S * J * 12
    return {"bytes": b, "flops": n * 2.0 * R * (T + 1)}


def tolerance(case):
    """Selections, demands and rounds are whole numbers and stay the same. Prices follow a fixed sequence
    of correctly rounded operations; objectives are 64-bit sums. The predictor computes in fp32 (two
    layers of sums of up to 64 products): four times its distance from 64 bits (5.7e-7)."""
    if case["kind"] == "iac":
        return {"rel": 2.4e-6, "max": 1e-4}
    return {"rel": 1e-12, "max": 1e-11, "differ": 0.0}


# ---- 64-bit reference -------------------------------------------------------------------------------

def _tatonnement(off, units, values, cap, J, eta0, T, mode, step, lam0=None, group=None, rg=None):
    """The method in plain fp64 torch: reduced costs by column, the smallest per job (lowest index on a
    tie), demand, the projected step; then one more best response and the objectives."""
    S, P = cap.shape
    n, R = units.shape
    dev = units.device
    cnt = off[1:] - off[:-1]
    K = int(cnt.max())
    n_jobs = cnt.shape[0]
    u = torch.zeros((R, n_jobs, K), dtype=torch.int32, device=dev)
    v = torch.full((n_jobs, K), -math.inf, dtype=torch.float64, device=dev)
    job = torch.repeat_interleave(torch.arange(n_jobs, device=dev), cnt)
    pos = torch.arange(n, device=dev) - off[:-1][job]
    v[job, pos] = values
    for r in range(R):
        u[r][job, pos] = units[:, r]
    gr = None
    if group is not None:
        gr = torch.zeros((n_jobs, K), dtype=torch.int64, device=dev)
        gr[job, pos] = group.long()
    C = cap.double()
    lam = torch.zeros((S, P), dtype=torch.float64, device=dev) if lam0 is None else lam0.to(dev)
    scen = torch.arange(n_jobs, device=dev) // J
    ks = torch.arange(K, device=dev)

    def best(lam):
        p = lam / C if mode == 1 else lam
        sel = torch.empty(n_jobs, dtype=torch.int64, device=dev)
        smin = torch.empty(n_jobs, dtype=torch.float64, device=dev)
        step_j = max(1, (1 << 24) // K)
        for a in range(0, n_jobs, step_j):
            b = min(n_jobs, a + step_j)
            s = -v[a:b]
            for r in range(R):
                if group is not None and r >= rg:
                    pr = p[scen[a:b, None], rg + (R - rg) * gr[a:b] + (r - rg)]
                else:
                    pr = p[scen[a:b], r][:, None]
                s = s + pr * u[r, a:b].double()
            m = s.amin(1)
            sel[a:b] = torch.where(s == m[:, None], ks[None, :], K).amin(1)
            smin[a:b] = m
        at = torch.arange(n_jobs, device=dev)
        dem = torch.zeros((S, P), dtype=torch.int64, device=dev)
        for r in range(R):
            w = u[r, at, sel].long()
            if group is not None and r >= rg:
                dem.view(-1).index_add_(0, scen * P + rg + (R - rg) * gr[at, sel] + (r - rg), w)
            else:
                dem[:, r] = torch.zeros(S, dtype=torch.int64, device=dev).index_add_(0, scen, w)
        return sel, dem, smin

    for t in range(T):
        _, dem, _ = best(lam)
        eta = eta0 / math.sqrt(t + 1) if step == 1 else eta0
        d = (dem - cap).double()
        if mode == 1:
            d = d / C
        lam = torch.clamp(lam + eta * d, min=0)
    sel, dem, smin = best(lam)
    prim = v[torch.arange(n_jobs, device=dev), sel].view(S, J).sum(1)
    dual = (-smin).view(S, J).sum(1) + (lam if mode == 1 else lam * C).sum(1)
    return dict(prices=lam, selection=None, demand=None, rounds=None, feasible=None, primal=prim, dual=dual)


def _iac_exact(case, seed):
    m = workloads.iac_model(int(seed), case["H"])
    d = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=DEV)   # noqa: E731
    rows = d(workloads.iac_rows(int(seed), case["J"], case["K"]))
    pairs = _pairs(case, seed).long()
    s1 = d(m.bn1)[0] / torch.sqrt(d(m.bn1)[3] + float(np.float32(m.eps)))
    s2 = d(m.bn2)[0] / torch.sqrt(d(m.bn2)[3] + float(np.float32(m.eps)))
    W1, W2 = d(m.W1), d(m.W2)
    out = torch.empty(pairs.shape[0], dtype=torch.float64, device=DEV)
    for at in range(0, pairs.shape[0], 1 << 20):
        a, b = rows[pairs[at:at + (1 << 20), 0]], rows[pairs[at:at + (1 << 20), 1]]
        mean = lambda c: 0.5 * (a[:, c] + b[:, c])   # noqa: E731
        lo, hi = torch.minimum(a[:, 0], b[:, 0]), torch.maximum(a[:, 0], b[:, 0])
        pw = torch.stack([mean(0), mean(1), mean(2), mean(4), a[:, 5] + b[:, 5],
                          (a[:, 3] + b[:, 3]) / workloads.IAC_C_MEM, lo / hi,
                          (a[:, 2] / a[:, 0] - b[:, 2] / b[:, 0]).abs()], 1)
        x = torch.cat([a, b, pw], 1)
        h = torch.relu(s1 * (x @ W1.T + d(m.b1) - d(m.bn1)[2]) + d(m.bn1)[1])
        h = torch.relu(s2 * (h @ W2.T + d(m.b2) - d(m.bn2)[2]) + d(m.bn2)[1])
        out[at:at + (1 << 20)] = 1.0 + torch.relu(h @ d(m.W3) + float(np.float32(m.b3)))
    return dict(s_hat=out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "iac":
        return _iac_exact(case, seed)
    S, J, T = case["S"], case["J"], case["T"]
    if kind == "placement":
        p = _placement(case, seed)
        units, values, group = _placement_options(p, case)
        off = torch.arange(S * J + 1, device=DEV) * (case["KC"] * case["N"])
        return _tatonnement(off, units, values, p[6], J, 0.02, T, 1, 0, group=group, rg=6)
    K = abs(case["K"])
    if S * J * K * (T + 1) > 9e10:     # over about 20 seconds here
        return None
    off, units, values, cap = _table(case, seed)
    lam0 = None
    if kind in ("epoch", "replan"):
        lam0 = torch.from_numpy(_warm(case, seed, cap))
    if kind == "replan":
        cur, s_hat, tau = (torch.from_numpy(x).to(DEV) for x in _penalty_inputs(case, seed, off))
        cnt = off[1:] - off[:-1]
        job = torch.repeat_interleave(torch.arange(cnt.shape[0], device=DEV), cnt)
        pos = torch.arange(values.shape[0], device=DEV) - off[:-1][job]
        sw = ((cur[job] >= 0) & (pos != cur[job])).double() * GAMMA0
        values = values - (sw + ALPHA * torch.clamp(s_hat - tau[job], min=0))
    return _tatonnement(off, units, values, cap, J, _eta(case, cap), T, case["mode"], case["step"], lam0)
