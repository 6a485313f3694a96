"""Workloads that stand for what programs do with this framework.

listed() names the fixed ones, draw() makes more of the same ranges.  A case is
a dict of plain values; prepare() makes what a program holds before the call
(model, parameter sweeps, batch handle, output buffers, samples to compare),
run() is one pass through the public entry points of
paper_2605_00479_gb300.ssa.
"""
import math

import numpy as np
import torch

from paper_2605_00479_gb300 import presets as P
from paper_2605_00479_gb300 import ssa

MODES_RN = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "rn"), ("mixed_bf16", "rn"), ("uniform_f16", "rn"),
            ("uniform_bf16", "rn")]
MODES_SR = [("mixed_f16", "sr"), ("mixed_bf16", "sr"), ("uniform_f16", "sr"), ("uniform_bf16", "sr")]
MODES_SRA = [("uniform_f16", "sra"), ("uniform_bf16", "sra")]
# uniform modes may freeze their clock and run to the event cap
CAP = 200000
# rough cost of one event against a mixed round-to-nearest one, to bound what draw() makes
COST = {"fp64": 30.0, "fp32": 1.0, "mixed_f16": 1.0, "mixed_bf16": 1.0, "uniform_f16": 1.5, "uniform_bf16": 1.5}


def _cascade():
    """A network without a compiled structure: X <-> Z conversion with Z held
    fixed, pairing of X into Y, Y back into X, a third-order loss and a
    constant source of Y (six reactions, three species)."""
    return {"order": np.array([[1, 0, 1], [2, 0, 0], [0, 1, 0], [0, 3, 0], [0, 0, 0], [1, 0, 0]], np.int32),
            "stoich": np.array([[1, 0, -1], [-2, 1, 0], [1, -1, 0], [0, -3, 0], [0, 1, 0], [-1, 0, 0]], np.int32),
            "rate": np.array([0.02, 0.01, 0.5, 0.001, 2.0, 0.1]), "law": np.zeros(6, np.int32), "hill": None,
            "constant": np.array([0, 0, 1], np.uint8)}


def _network(name):
    """(model tables, x0, fold the held species into the rate constants)."""
    if name == "birth_death":
        return P.birth_death(10.0, 0.1), [0], False
    if name == "schlogl":
        m = P.schlogl()
        return m, list(P.schlogl_x0(m)), True
    if name == "telegraph":
        return P.telegraph(0.5, 0.5, 20.0, 1.0), list(P.TELEGRAPH_X0), False
    if name == "dimer":
        return P.dimer(), list(P.dimer_x0(300)), False
    if name == "repressilator":
        return P.repressilator(), list(P.REPRESSILATOR_X0), False
    if name == "repressilator_h3":          # Hill exponent 3: runtime tables
        return P.repressilator(h=3), list(P.REPRESSILATOR_X0), False
    return _cascade(), [10, 5, 50], True


def listed():
    return [
        # One quick look at a model: the small birth-death configuration, 10^4
        # trajectories with 101 snapshots; fewer trajectories than lanes, so
        # the time is the latency of a trajectory's chain of events.
        {"name": "birth_death_small_mixed_f16", "kind": "direct", "net": "birth_death", "n": 10000, "t_end": 100.0,
         "K": 101, "prec": "mixed_f16", "rnd": "rn", "bytes": 4, "mask": 0},
        # The headline ensemble: 10^6 bistable trajectories, X stored.
        {"name": "schlogl_1e6_mixed_bf16", "kind": "direct", "net": "schlogl", "n": 1000000, "t_end": 10.0, "K": 50,
         "prec": "mixed_bf16", "rnd": "rn", "bytes": 4, "mask": 1},
        # The costliest 16-bit mode: every operation rounded stochastically,
        # an ordinary ensemble size.
        {"name": "schlogl_uniform_f16_sr", "kind": "direct", "net": "schlogl", "n": 150000, "t_end": 10.0, "K": 50,
         "prec": "uniform_f16", "rnd": "sr", "bytes": 4, "mask": 1},
        # Results wanted on the host: a dense int16 snapshot series of a gene's
        # switching, delivered into page-locked buffers (ragged size).
        {"name": "telegraph_host_uniform_bf16_sr", "kind": "host", "net": "telegraph", "n": 300007, "t_end": 50.0,
         "K": 101, "prec": "uniform_bf16", "rnd": "sr", "bytes": 2, "mask": 0},
        # A six-species oscillator with Hill laws, ordinary size, odd count.
        {"name": "repressilator_mixed_f16", "kind": "direct", "net": "repressilator", "n": 50001, "t_end": 40.0,
         "K": 101, "prec": "mixed_f16", "rnd": "rn", "bytes": 4, "mask": 0},
        # The binary64 reference ensemble every reduced mode is compared with.
        {"name": "schlogl_fp64", "kind": "direct", "net": "schlogl", "n": 20000, "t_end": 10.0, "K": 50,
         "prec": "fp64", "rnd": "rn", "bytes": 4, "mask": 1},
        # A user's own network: no compiled structure, tables read at run time.
        {"name": "own_network_fp32", "kind": "direct", "net": "cascade", "n": 100000, "t_end": 50.0, "K": 21,
         "prec": "fp32", "rnd": "rn", "bytes": 4, "mask": 0},
        # A heterogeneous parameter sweep: three models in one persistent launch.
        {"name": "sweep_three_models_mixed_f16", "kind": "batch", "sets": 500, "per_set": 64, "t_end": 100.0,
         "prec": "mixed_f16", "rnd": "rn", "bytes": 4},
        # Approximate simulation: fixed-leap tau-leaping of the bistable model.
        {"name": "tau_schlogl_fp32", "kind": "tau", "net": "schlogl", "n": 150001, "t_end": 10.0, "tau": 0.005,
         "K": 50, "prec": "fp32", "rnd": "rn", "bytes": 4},
        # Spatial: a 32-voxel chain of the bistable model.
        {"name": "rdme_chain_mixed_f16", "kind": "rdme", "net": "schlogl", "nx": 32, "ny": 1, "nz": 1, "hop": 1.0,
         "n": 65536, "t_end": 0.25, "K": 1, "prec": "mixed_f16", "rnd": "rn", "bytes": 4},
        # Comparing two ensembles: histograms, KS statistic, W1, OFF dwell times.
        {"name": "compare_ensembles", "kind": "stats", "n": 4000000, "bins": 1024, "K": 101, "n_series": 200003,
         "bytes": 4},
        # The surrogate's training loop on histograms, then its answers.
        {"name": "surrogate_train_b1024", "kind": "surrogate", "rows": 16384, "batch": 1024, "steps": 64,
         "queries": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mode(rng, sra=True):
    return rng.choice(MODES_RN + MODES_RN + MODES_SR + (MODES_SRA if sra else []))


def draw(rng):
    kind = rng.choice(["direct", "direct", "direct", "direct", "host", "batch", "tau", "rdme", "stats", "surrogate"])
    if kind in ("direct", "host"):
        net = rng.choice(["birth_death", "schlogl", "telegraph", "dimer", "repressilator", "repressilator_h3",
                          "cascade"])
        prec, rnd = _mode(rng)
        t_end = {"birth_death": 100.0, "schlogl": 10.0, "telegraph": 50.0, "dimer": 50.0, "repressilator": 20.0,
                 "repressilator_h3": 5.0, "cascade": 30.0}[net] * rng.uniform(0.2, 1.0)
        cost = COST[prec] * (2.5 if rnd == "sr" else 1.0) * (8.0 if net in ("repressilator_h3", "cascade") else 1.0)
        per = _events(net, t_end)
        if prec.startswith("uniform") and rnd != "sr":
            per = max(per, 0.5 * CAP)
        most = max(4.0, min(1e6, 8e9 / (per * cost)))
        n = _log_int(rng, min(300.0, 0.25 * most), most) | 1
        return {"kind": kind, "net": net, "n": n, "t_end": t_end, "K": rng.choice([1, 2, 11, 50, 101, 257]),
                "prec": prec, "rnd": rnd, "bytes": rng.choice([4, 4, 2]), "mask": rng.choice([0, 0, 1])}
    if kind == "batch":
        prec, rnd = _mode(rng, False)
        cost = COST[prec] * (2.5 if rnd == "sr" else 1.0)
        t_end = rng.uniform(10.0, 60.0)
        per = _events("repressilator", t_end)
        if prec.startswith("uniform") and rnd == "rn":
            per = max(per, 0.5 * CAP)
        most = max(8.0, min(40000.0, 5e9 / (per * cost)))
        total = _log_int(rng, min(200.0, 0.5 * most), most)
        per_set = max(1, min(_log_int(rng, 4, 256), total // 2))
        return {"kind": "batch", "sets": max(1, total // per_set), "per_set": per_set, "t_end": t_end, "prec": prec,
                "rnd": rnd, "bytes": rng.choice([4, 2])}
    if kind == "tau":
        prec, rnd = _mode(rng, False)
        net = rng.choice(["schlogl", "birth_death", "dimer", "repressilator", "cascade"])
        t_end = {"schlogl": 10.0, "birth_death": 100.0, "dimer": 50.0, "repressilator": 20.0, "cascade": 30.0}[net]
        leaps = _log_int(rng, 50, 2000)
        cost = (8.0 if prec == "fp64" else 1.0) * (4.0 if net in ("repressilator", "cascade") else 1.0)
        n = _log_int(rng, 300, max(600.0, 2e8 / (leaps * cost))) | 1
        return {"kind": "tau", "net": net, "n": n, "t_end": t_end, "tau": t_end / leaps, "K": rng.choice([1, 50]),
                "prec": prec, "rnd": rnd, "bytes": rng.choice([4, 2])}
    if kind == "rdme":
        prec, rnd = _mode(rng, False)
        nx, ny, nz = rng.choice([(32, 1, 1), (17, 1, 1), (8, 1, 1), (4, 4, 1), (5, 3, 1), (3, 3, 3), (64, 1, 1)])
        cost = (8.0 if prec == "fp64" else 1.0) * (2.0 if rnd == "sr" else 1.0) * nx * ny * nz / 32.0
        t_end = rng.uniform(0.05, 0.25)
        n = _log_int(rng, 300, max(600.0, 12000.0 / (cost * t_end))) | 1
        return {"kind": "rdme", "net": "schlogl", "nx": nx, "ny": ny, "nz": nz, "hop": rng.uniform(0.2, 2.0), "n": n,
                "t_end": t_end, "K": rng.choice([1, 3]), "prec": prec, "rnd": rnd, "bytes": rng.choice([4, 2])}
    if kind == "stats":
        return {"kind": "stats", "n": _log_int(rng, 1000, 4000000) | 1, "bins": _log_int(rng, 64, 20000),
                "K": _log_int(rng, 11, 201), "n_series": _log_int(rng, 500, 200000) | 1,
                "bytes": rng.choice([4, 2])}
    rows = _log_int(rng, 2048, 16384)
    return {"kind": "surrogate", "rows": rows, "batch": rng.choice([128, 256, 500, 1000, 1024, 2048]),
            "steps": _log_int(rng, 16, 64), "queries": _log_int(rng, 100, 16384)}


# ---------------------------------------------------------------- preparing
def _buffers(K, rows, n, nbytes, host):
    kw = {"pin_memory": True} if host else {"device": "cuda"}
    b = {"out": torch.empty((K, rows, n), dtype=torch.int16 if nbytes == 2 else torch.int32, **kw),
         "status": torch.empty(n, dtype=torch.int32, **kw), "n_events": torch.empty(n, dtype=torch.int64, **kw),
         "t_final": torch.empty(n, dtype=torch.float64, **kw)}
    if host:
        b = {k: v.numpy() for k, v in b.items()}
        b["status"] = b["status"].view(np.uint32)
    return b


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed}
    if kind in ("direct", "host", "tau", "rdme"):
        tables, x0, fold = _network(case["net"])
        st["model"], st["x0"], st["fold"] = ssa.Model.from_dict(tables), np.array(x0, np.int32), fold
        st["samples"] = P.even_samples(case["t_end"], case["K"])
        rows = st["model"].N
        if kind in ("direct", "host"):
            rows = bin(case["mask"]).count("1") or rows
        if kind == "rdme":
            voxels = case["nx"] * case["ny"] * case["nz"]
            st["x0"] = np.tile(st["x0"], (voxels, 1))
            st["hop"] = [case["hop"]] + [0.0] * (st["model"].N - 1)
            rows *= voxels
        st["buf"] = _buffers(case["K"], rows, case["n"], case["bytes"], kind == "host")
        if kind == "rdme":
            st["buf"]["out"] = st["buf"]["out"].view(case["K"], voxels, st["model"].N, case["n"])
    elif kind == "batch":
        S = case["sets"]
        rr, rh = P.repressilator_sweep(S, seed=seed)
        st["batch"] = ssa.Batch([
            {"model": ssa.Model.from_dict(P.repressilator()), "x0": np.tile(P.REPRESSILATOR_X0, (S, 1)), "rates": rr,
             "hill": rh[:, :, :2], "traj_per_set": case["per_set"]},
            {"model": ssa.Model.from_dict(P.telegraph()), "x0": np.tile(P.TELEGRAPH_X0, (S, 1)),
             "rates": P.telegraph_sweep(S, seed=seed + 1), "traj_per_set": case["per_set"]},
            {"model": ssa.Model.from_dict(P.dimer()), "x0": np.tile(P.dimer_x0(300), (S, 1)),
             "rates": P.dimer_sweep(S, seed=seed + 2), "traj_per_set": case["per_set"]},
        ], case["t_end"], [case["t_end"]], case["prec"], case["rnd"], seed=seed, max_events=_cap(case),
            state_bytes=case["bytes"])
    elif kind == "stats":
        g = torch.Generator(device="cuda").manual_seed(seed)
        dt = torch.int16 if case["bytes"] == 2 else torch.int32
        mid = 0.4 * case["bins"]

        def ensemble(shift):            # two basins, as the bistable model leaves them
            lo = torch.randn(case["n"], device="cuda", generator=g) * (0.05 * case["bins"]) + 0.2 * case["bins"]
            hi = torch.randn(case["n"], device="cuda", generator=g) * (0.08 * case["bins"]) + mid + 0.2 * case["bins"]
            up = torch.rand(case["n"], device="cuda", generator=g) < 0.45 + shift
            return torch.where(up, hi, lo).round().clamp(-5, case["bins"] + 5).to(dt)

        st["a"], st["b"] = ensemble(0.0), ensemble(0.01)
        # a gene's OFF indicator at the snapshots: blocks of OFF and ON
        flip = torch.rand((case["K"], case["n_series"]), device="cuda", generator=g) < 0.2
        st["series"] = (flip.cumsum(0) % 2).to(dt).view(case["K"], 1, case["n_series"]).contiguous()
    else:
        rng = np.random.default_rng(seed)
        lo = np.log([0.05, 0.05, 5.0, 0.5])
        hi = np.log([5.0, 5.0, 100.0, 2.0])

        def points(n):
            return rng.uniform(-1.0, 1.0, size=(n, 4)).astype(np.float32)

        f = points(case["rows"])
        kon, koff, km, gam = np.exp(lo + (hi - lo) * (f.astype(np.float64) + 1.0) / 2.0).T
        mean = km * kon / (kon + koff) / gam
        sd = np.sqrt(mean + 0.25 * mean * mean * koff / (kon + koff + gam)) + 0.5
        k = np.arange(128)
        h = np.exp(-0.5 * ((k[None, :] - mean[:, None]) / sd[:, None]) ** 2) + 1e-9
        h /= h.sum(axis=1, keepdims=True)
        st["features"] = torch.from_numpy(f).cuda()
        st["targets"] = torch.from_numpy(h.astype(np.float32)).cuda()
        st["queries"] = torch.from_numpy(points(case["queries"])).cuda()
        st["net"] = ssa.Surrogate(max_batch=max(case["batch"], case["queries"]), seed=seed)
        st["theta"] = st["net"].get_params()
    return st


def _cap(case):
    return CAP if case["prec"].startswith("uniform") else 10**7


# ---------------------------------------------------------------- running
def run(st):
    c, kind = st["case"], st["case"]["kind"]
    if kind in ("direct", "host"):
        f = ssa.ensemble_run if kind == "direct" else ssa.ensemble_run_host
        return f(st["model"], c["n"], st["x0"], c["t_end"], st["samples"], c["prec"], c["rnd"], st["fold"], st["seed"],
                 _cap(c), c["bytes"], out_species=c["mask"], **st["buf"])
    if kind == "tau":
        return ssa.tau_run(st["model"], c["n"], st["x0"], c["t_end"], c["tau"], st["samples"], c["prec"], c["rnd"],
                           st["fold"], st["seed"], c["bytes"], **st["buf"])
    if kind == "rdme":
        return ssa.rdme_run(st["model"], (c["nx"], c["ny"], c["nz"]), st["hop"], st["x0"], c["n"], c["t_end"],
                            st["samples"], c["prec"], c["rnd"], st["fold"], st["seed"], _cap(c), c["bytes"],
                            **st["buf"])
    if kind == "batch":
        st["batch"].launch()
        return st["batch"].outputs
    if kind == "stats":
        ha, ca = ssa.count_histogram(st["a"], c["bins"])
        hb, cb = ssa.count_histogram(st["b"], c["bins"])
        return {"hist_a": ha, "clamped_a": ca, "hist_b": hb, "clamped_b": cb, "ks_w1": ssa.hist_ks_w1(ha, hb),
                "dwell": ssa.dwell_histogram(st["series"], 0)}
    net = st["net"]
    net.set_params(st["theta"])
    trace = torch.empty(c["steps"], dtype=torch.float32, device="cuda")
    net.train(st["features"], st["targets"], c["steps"], c["batch"], 2e-3, 5e-5, loss_every=1, loss_trace=trace)
    return {"theta": net.get_params(), "loss": trace, "answers": net.predict(st["queries"])}


# ---------------------------------------------------------------- what a pass cannot do without
def _events(net, t_end):
    """Events of one trajectory, from the mean-field equations."""
    m, x0, _ = _network(net)
    x = np.array(x0, float)
    steps = 2000
    dt, total = t_end / steps, 0.0
    nu = m["stoich"] * (1 if m["constant"] is None else (1 - m["constant"].astype(int)))
    for _ in range(steps):
        a = np.empty(len(m["rate"]))
        for j, c in enumerate(m["rate"]):
            if m["law"][j] == 1:
                h = m["hill"][j]
                a[j] = h[0] + h[1] / (1.0 + x[int(h[3])] ** h[2])
                continue
            a[j] = c
            for i, r in enumerate(m["order"][j]):
                for q in range(r):
                    a[j] *= max(x[i] - q, 0.0) / (q + 1)
        total += a.sum() * dt
        x = np.maximum(x + dt * (a @ nu), 0.0)
    return max(total, 1.0)


def _step_ops(net, prec, rnd):
    """32-bit (or binary64) operations of one event: the counter-based
    generator (100 per block of two events), uniforms, logarithm, waiting
    time, propensity factors, sums, selection and update."""
    m, _, fold = _network(net)
    factors = sum(int(r) for j in range(len(m["rate"])) for i, r in enumerate(m["order"][j])
                  if not (fold and m["constant"] is not None and m["constant"][i]))
    hills = int(sum(m["law"]))
    ops = 50 + 8 + 25 + 3 + 3 * factors + 7 * hills + 2 * len(m["rate"]) + 8
    if prec[:2] != "fp":
        ops += 2 * factors + 4 * hills
    if rnd == "sr":
        slots = 2 * factors + 5 * hills + (len(m["rate"]) + 4 if prec.startswith("uniform") else 0)
        ops += 100 * ((slots + 7) // 8)
    elif rnd == "sra":
        ops += 100 * ((len(m["rate"]) + 7) // 8)
    return ops


def work(case):
    kind = case["kind"]
    if kind in ("direct", "host", "tau"):
        m, _, _ = _network(case["net"])
        rows = (bin(case.get("mask", 0)).count("1") or m["order"].shape[1])
        nbytes = case["n"] * (case["K"] * rows * case["bytes"] + 20)
        if kind == "tau":
            # per leap and channel: one generator block, the chain and the draw's arithmetic
            M = len(m["rate"])
            return {"bytes": nbytes, "flops": case["n"] * case["t_end"] / case["tau"] * M * 160}
        return {"bytes": nbytes,
                "flops": case["n"] * _events(case["net"], case["t_end"]) * _step_ops(case["net"], case["prec"], case["rnd"])}
    if kind == "rdme":
        S = case["nx"] * case["ny"] * case["nz"]
        m, x0, _ = _network(case["net"])
        links = sum(2 * (d - 1) * S // d for d in (case["nx"], case["ny"], case["nz"]))
        events = _events(case["net"], case["t_end"]) * S + links * case["hop"] * x0[0] * case["t_end"]
        per = _step_ops(case["net"], case["prec"], case["rnd"]) * 2 + 4 * math.ceil(math.log2(S))
        return {"bytes": case["n"] * (case["K"] * S * m["order"].shape[1] * case["bytes"] + 20),
                "flops": case["n"] * events * per}
    if kind == "batch":
        n = case["sets"] * case["per_set"]
        flops = sum(n * _events(k, case["t_end"]) * _step_ops(k, case["prec"], case["rnd"])
                    for k in ("repressilator", "telegraph", "dimer"))
        return {"bytes": n * (11 * case["bytes"] + 60) + case["sets"] * 8 * 40, "flops": flops}
    if kind == "stats":
        return {"bytes": case["bytes"] * (2 * case["n"] + case["K"] * case["n_series"]) + 8 * (4 * case["bins"] + case["K"]),
                "flops": 2 * case["n"] + 3 * case["K"] * case["n_series"]}
    weights = 16 * 256 + 2 * 256 * 256 + 256 * 128
    flops = 2 * weights * (3 * case["steps"] * case["batch"] + case["queries"])
    state = 4 * 168832
    nbytes = case["steps"] * (case["batch"] * 132 * 4 + 7 * state) + 2 * state + case["queries"] * 132 * 4
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- exact values
def _exact_stats(case, st):
    out = {}
    for k in ("a", "b"):
        v = st[k].cpu().to(torch.int64)
        w = v.clamp(0, case["bins"] - 1)
        out["hist_" + k] = torch.bincount(w, minlength=case["bins"])
        out["clamped_" + k] = (v != w).sum().reshape(1)
    ca = np.cumsum(out["hist_a"].numpy()).astype(object)
    cb = np.cumsum(out["hist_b"].numpy()).astype(object)
    na, nb = int(ca[-1]), int(cb[-1])
    d = [abs(int(p) * nb - int(q) * na) for p, q in zip(ca, cb)]
    fits = float(case["bins"]) * na * nb < 2.0 ** 63
    ks = [max(d) / (na * nb), sum(d) / (na * nb)] if fits else [float("nan")] * 2
    s = st["series"][:, 0, :].cpu().numpy() != 0
    hist = np.zeros(case["K"], np.int64)
    start = np.full(s.shape[1], -1)
    for k in range(1, case["K"]):
        begins = s[k] & ~s[k - 1]
        ends = ~s[k] & s[k - 1] & (start >= 0)
        np.add.at(hist, k - start[ends], 1)
        start[ends] = -1
        start[begins] = k
    return {"hist_a": out["hist_a"], "clamped_a": out["clamped_a"], "hist_b": out["hist_b"],
            "clamped_b": out["clamped_b"], "ks_w1": torch.tensor(ks, dtype=torch.float64),
            "dwell": torch.from_numpy(hist)}


def _exact_surrogate(case, st):
    """The training loop and the answers in binary64."""
    dims = [(256, 16), (256, 256), (256, 256), (128, 256)]
    theta = torch.from_numpy(st["theta"]).to("cuda", torch.float64).requires_grad_(True)
    decay = torch.zeros_like(theta, requires_grad=False)
    live = torch.ones_like(theta, requires_grad=False)
    at, cuts = 0, []
    for o, i in dims:
        decay[at:at + o * i] = 1.0
        if i == 16:
            live[at:at + o * i] = (torch.arange(o * i, device="cuda") % 16 < 4).double()
        cuts.append((at, at + o * i, at + o * i + o))
        at += o * i + o

    def logits(x):
        h = torch.nn.functional.pad(x.double(), (0, 12))
        for l, (a, b, c) in enumerate(cuts):
            h = h @ theta[a:b].view(dims[l]).T + theta[b:c]
            if l < 3:
                h = torch.nn.functional.gelu(h)
        return h

    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    rows, B, n = case["rows"], case["batch"], case["steps"]
    losses = []
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    for k in range(n):
        idx = (k * B + torch.arange(B, device="cuda")) % rows
        loss = -(st["targets"][idx].double() * torch.log_softmax(logits(st["features"][idx]), 1)).sum(1).mean()
        g, = torch.autograd.grad(loss, theta)
        losses.append(loss.detach())
        lr = 5e-5 + 0.5 * (2e-3 - 5e-5) * (1 + math.cos(math.pi * (k / (n - 1) if n > 1 else 0.0)))
        with torch.no_grad():
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            step = lr * (m / (1 - b1 ** (k + 1))) / (torch.sqrt(v / (1 - b2 ** (k + 1))) + 1e-8)
            theta -= live * (lr * 1e-4 * decay * theta + step)
    with torch.no_grad():
        answers = torch.softmax(logits(st["queries"]), 1)
    return {"theta": theta.detach().cpu().numpy(), "loss": torch.stack(losses).cpu(), "answers": answers.cpu()}


def exact(case, seed):
    # trajectories are sequences of random draws in the mode's own arithmetic:
    # no 64-bit value stands for them
    if case["kind"] not in ("stats", "surrogate"):
        return None
    st = prepare(case, seed)
    return _exact_stats(case, st) if case["kind"] == "stats" else _exact_surrogate(case, st)
