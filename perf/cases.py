"""What this package is timed on: calls that its users make, at sizes from a
few microseconds of work to about a second, through the public entry points of
``paper_2402_13259_gb300.binding``.

A case is a plain dict: ``net`` names the network generator (with its
parameters), ``call`` the entry point, ``scheme`` 0 (backward) or 1 (forward),
``R`` replications, horizon ``T`` and step ``dt``.  The seed of ``prepare``
seeds both the network and the simulation (the batch: service rates and
simulations of its fixed set of networks).
"""
import math

import numpy as np
import torch

from paper_2402_13259_gb300 import binding as B
from paper_2402_13259_gb300 import workloads as W

# Arithmetic operations one station-step update cannot do without: Philox
# words, the departure and routing draws by inversion or by rejection, the
# gather and the sums.  Larger counts per station mean more rejection draws.
_OPS = {"tandem": 200.0, "dag": 295.0, "batch": 295.0}


def _ops(case):
    if case["net"] == "scale":  # 200 at s = 10 to 620 at s = 10,000
        return 200.0 + 140.0 * max(0.0, math.log10(case["s"]) - 1.0)
    return _OPS[case["net"]]


def listed():
    return [
        # The smallest call: a three-station tandem, a few replications, 100
        # steps.  What an interactive user or a unit test sees is its latency.
        {"name": "tandem_smallest", "net": "tandem", "call": "simulate", "scheme": 0, "R": 40, "T": 1.0, "dt": 0.01},
        # The three-station tandem at its stated size: 2,400 steps in series.
        {"name": "tandem_forward", "net": "tandem", "call": "simulate", "scheme": 1, "R": 1000, "T": 24.0, "dt": 0.01},
        # The benchmark's call: 100-station layered DAG, 10,000 replications,
        # 10,000 steps.
        {"name": "dag100_backward", "net": "dag", "L": 10, "W": 10, "call": "simulate", "scheme": 0, "R": 10000,
         "T": 100.0, "dt": 0.01},
        # The same network in the forward scheme, with a replication count that
        # no tile divides, over a horizon as long as its slowest transients.
        {"name": "dag100_forward_ragged", "net": "dag", "L": 10, "W": 10, "call": "simulate", "scheme": 1,
         "R": 9973, "T": 40.0, "dt": 0.01},
        # A study of one site: staffing schedule, arrivals from a table,
        # customers present at the start, the average of both schemes.
        {"name": "dag100_schedule_average", "net": "dag", "L": 10, "W": 10, "call": "average", "R": 1237, "T": 20.0,
         "dt": 0.01, "schedule": True},
        # The scale sweep on the 2,000-station DAG: few large steps with small
        # stations ...
        {"name": "scale10_backward", "net": "scale", "s": 10.0, "call": "simulate", "scheme": 0, "R": 20000, "T": 50.0},
        # ... the middle of the sweep ...
        {"name": "scale100_forward", "net": "scale", "s": 100.0, "call": "simulate", "scheme": 1, "R": 6000, "T": 50.0},
        # ... and its end, where most draws are rejection draws.
        {"name": "scale10000_backward", "net": "scale", "s": 10000.0, "call": "simulate", "scheme": 0, "R": 512,
         "T": 20.0},
        # Many networks of uneven size in one batch.
        {"name": "batch_mixed", "net": "batch", "call": "batch", "count": 64, "max_n": 1500, "T_scale": 0.02,
         "R_scale": 0.1},
        # Likelihood-ratio gradients of the sinusoid DAG.
        {"name": "dag100_grad", "net": "dag", "L": 10, "W": 10, "call": "grad", "scheme": 0, "R": 10000, "T": 20.0,
         "dt": 0.01, "b": 0.3},
        # One optimisation step: measures of new parameters, forward and
        # backward through autograd (a new network handle on every call).
        {"name": "tandem_measures_step", "net": "tandem", "call": "measures", "scheme": 0, "R": 1000, "T": 24.0,
         "dt": 0.01},
        # Sojourn times of four tagged customers per replication.
        {"name": "dag100_sojourn", "net": "dag", "L": 10, "W": 10, "call": "sojourn", "scheme": 1, "R": 10000,
         "T": 20.0, "dt": 0.01, "samples": 4},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _int_log(rng, lo, hi):
    return int(min(hi, max(lo, round(_log_uniform(rng, lo, hi)))))


def draw(rng):
    kind = rng.choice(["tandem", "tandem_measures", "dag", "dag", "dag_average", "scale", "scale", "batch", "grad",
                       "sojourn"])
    scheme = rng.randint(0, 1)
    if kind == "batch":
        return {"net": "batch", "call": "batch", "count": _int_log(rng, 8, 64), "max_n": _int_log(rng, 50, 1500),
                "T_scale": round(_log_uniform(rng, 0.005, 0.02), 4), "R_scale": round(_log_uniform(rng, 0.02, 0.1), 4)}
    if kind == "scale":
        s = round(_log_uniform(rng, 10.0, 10000.0), 1)
        T = rng.choice([10.0, 20.0, 50.0])
        steps = T * math.sqrt(s)
        R = int(min(100000, max(64, _log_uniform(rng, 1e8, 4e9) / (2000.0 * steps))))
        return {"net": "scale", "s": s, "call": "simulate", "scheme": scheme, "R": R, "T": T}
    if kind.startswith("tandem"):
        T, dt = rng.choice([1.0, 6.0, 24.0]), rng.choice([0.005, 0.01, 0.02])
        call = "measures" if kind == "tandem_measures" else "simulate"
        return {"net": "tandem", "call": call, "scheme": scheme, "R": _int_log(rng, 30, 20000), "T": T, "dt": dt}
    T, dt = round(rng.uniform(5.0, 40.0), 1), rng.choice([0.005, 0.01, 0.02])
    L, width = rng.randint(2, 16), _int_log(rng, 3, 60)
    units = L * width * T / dt
    R = int(min(30000, max(20, _log_uniform(rng, 2e7, 3e9) / units)))
    case = {"net": "dag", "L": L, "W": width, "scheme": scheme, "R": R, "T": T, "dt": dt}
    if kind == "dag":
        return dict(case, call="simulate")
    if kind == "dag_average":
        del case["scheme"]
        return dict(case, call="average", R=max(20, R // 4), schedule=rng.random() < 0.5)
    if kind == "grad":
        return dict(case, call="grad", b=0.3)
    return dict(case, call="sojourn", samples=rng.randint(1, 4))


def _network(case, seed):
    """The workload's network and step, as a user's program builds them."""
    s = int(seed) % (1 << 31)
    if case["net"] == "tandem":
        run = W.tandem3(R=case["R"], seed=s)
        rng = np.random.default_rng(s)
        run.net.mu = np.exp(rng.uniform(math.log(0.9), math.log(1.1), size=3))
        return run.net, case["dt"]
    if case["net"] == "scale":
        run = W.scale_dag(case["s"], seed=s, R=case["R"], T=case["T"])
        return run.net, run.dt
    run = W.layered_dag(L=case["L"], W=case["W"], seed=s, R=case["R"], T=case["T"], dt=case["dt"])
    net = run.net
    net.arrivals.b = case.get("b", 0.0)
    if case.get("schedule"):
        # hourly tables over the horizon: arrivals and servers rise and fall
        rng = np.random.default_rng(s + 1)
        hours = int(math.ceil(case["T"])) + 1
        level = 1.0 + 0.3 * np.sin(2.0 * math.pi * np.arange(hours) / 24.0)[:, None]
        noise = rng.uniform(0.95, 1.05, size=(hours, net.n))
        net.arrivals = W.Arrivals(kind=W.ARR_TABLE, table=net.arrivals.w[None, :] * level * noise, tab_dt=1.0)
        net.arrivals.table = np.ascontiguousarray(net.arrivals.table)
        net.servers_schedule = np.maximum(1, np.rint(net.servers[None, :] * level)).astype(np.int32)
        net.servers_schedule_dt = 1.0
        net.N0 = np.ascontiguousarray(np.rint(0.8 * net.servers), dtype=np.int32)
    return net, run.dt


def prepare(case, seed):
    state = dict(case, seed=int(seed) % (1 << 31))
    if case["call"] == "batch":
        # the batch workload's networks (its own generator seed), their service
        # rates and simulation seeds varied
        runs = W.batch_networks(case["count"], max_n=case["max_n"], T_scale=case["T_scale"], R_scale=case["R_scale"])
        rng = np.random.default_rng(state["seed"])
        for r in runs:
            r.net.mu = r.net.mu * rng.uniform(0.95, 1.05, size=r.net.n)
        nets = [B.EulerNet(r.net) for r in runs]
        state["batch"] = B.Batch(nets, [(j % 2, r.dt, r.T, r.R, state["seed"] + j) for j, r in enumerate(runs)])
        return state
    net, state["dt"] = _network(case, seed)
    if case["call"] == "measures":
        a = net.arrivals
        state["net"] = net
        state["theta"] = torch.tensor(list(net.mu) + [a.a, a.b, a.phase], dtype=torch.float64, device="cuda")
        return state
    state["handle"] = B.EulerNet(net)
    return state


def run(state):
    call, T, seed = state["call"], state.get("T"), state["seed"]
    if call == "batch":
        return state["batch"].run()
    dt, R = state["dt"], state["R"]
    if call == "measures":
        theta = state["theta"].clone().requires_grad_(True)
        value = B.EulerMeasures.apply(theta, state["net"], state["scheme"], dt, T, R, seed)
        value.sum().backward()
        return [value.detach(), theta.grad]
    h = state["handle"]
    if call == "average":
        return list(h.simulate_average(dt, T, R, seed))
    if call == "grad":
        return h.grad(state["scheme"], dt, T, R, seed)
    if call == "sojourn":
        steps = B.num_steps(dt, T)
        stats = torch.empty(B.stats_len(h.n, R), dtype=torch.int64, device="cuda")
        times = h.sojourn(state["scheme"], dt, T, R, seed, station=0, tau0=max(1, steps // 4),
                          samples=state["samples"], stats=stats)
        return [times, stats]
    return h.simulate(state["scheme"], dt, T, R, seed)


def _steps(T, dt):
    return max(1, math.ceil(T / dt - 1e-9))


def work(case):
    """Bytes: the network's tables once (about two edges a station) and the
    outputs once.  Operations: station-step updates times those of one."""
    if case["call"] == "batch":
        mean_n = (case["max_n"] - 5) / math.log(case["max_n"] / 5.0)  # log-uniform on [5, max_n]
        R = 5050.0 * case["R_scale"]
        steps = 105.0 * case["T_scale"] * (200.0 + 100.0 + 50.0) / 3.0
        units = case["count"] * mean_n * R * steps
        return {"bytes": case["count"] * (mean_n * 140.0 + 32.0 * R), "flops": units * _ops(case)}
    n = {"tandem": 3, "scale": 2000}.get(case["net"]) or case["L"] * case["W"]
    dt = case["dt"] if "dt" in case else 1.0 / math.sqrt(case["s"])
    R, passes = case["R"], 2 if case["call"] == "average" else 1
    units = float(n) * R * _steps(case["T"], dt) * passes
    out = 8 * (6 * n + 4 * R) * (3 if case["call"] == "average" else 1)
    if case["call"] == "sojourn":
        out += 4 * R * case["samples"]
    if case["call"] in ("grad", "measures"):
        out = 8 * (4 * (n + 3) + 2)
    return {"bytes": float(92 * n + out), "flops": units * _ops(case)}


def exact(case, seed):
    """Counts are integers and must be equal; averages and gradients are sums
    over the same random draws, which no arithmetic outside this package
    defines."""
    return None
