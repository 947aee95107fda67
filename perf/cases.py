"""The work a user of this framework has it do, as cases a timing program can run.

A case is a dict of plain values; ``listed()`` gives the standing ones, ``draw(rng)``
one more of the same ranges, ``prepare(case, seed)`` the inputs and handles a user's
program has in hand before the call, ``run(state)`` one pass through the public entry
points, ``work(case)`` what one pass cannot do without, ``exact(case, seed)`` the
outputs in plain numpy binary64 where that is quick enough.

Every case uses the library's own automatic thresholds (which herds get a warp or a
lane group); the launch mode is the one such a program would set.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import fitting as F
from paper_1502_02908_gb300 import gradient as G
from paper_1502_02908_gb300 import workloads as W

# Transitions of one node-day on average, and floating-point operations of one
# transition (its logarithm, division, rates and comparisons), for work().
TRANSITIONS = {"sise": 19.0, "national": 2.0, "national_year": 0.6, "batched": 10.8, "uneven": 9.6,
               "general_sise3": 0.6, "general_seirs": 3.7, "general_sir": 3.5, "general_erlang": 52.0}
FLOPS_PER_DRAW = 40.0


def listed():
    return [
        # One small network watched day by day: a program that advances one day,
        # reads the prevalence so far, and goes on (SISe, 1,000 herds).
        dict(name="sise_daily", kind="advance", network="sise", nodes=1000, days=60, events=3300, replicates=1,
             mode="stream", chunk=1, pre_event=False),
        # The plain SISe configuration: 1,000 herds for a year in one call.
        dict(name="sise_year", kind="advance", network="sise", nodes=1000, days=365, events=20000, replicates=1,
             mode="graph", chunk=365, pre_event=False),
        # The headline configuration: the national SISe3 network, four years, 3M events.
        dict(name="sise3_national", kind="advance", network="national", nodes=37000, days=1460, events=3000000,
             replicates=1, mode="graph", chunk=1460, pre_event=False),
        # Batched replicates of the national network, a year, own (upsilon, gamma) each.
        dict(name="sise3_batched", kind="advance", network="batched", nodes=37000, days=365, events=750000,
             replicates=64, mode="persistent", chunk=365, pre_event=False),
        # An uneven batch: a parameter study over networks of very different sizes and horizons.
        dict(name="uneven_batch", kind="uneven", instances=32, nodes_lo=100, nodes_hi=10000, days_lo=90, days_hi=1460,
             study=5),
        # The dense synthetic benchmark of the paper (2,000 transitions a node-day).
        dict(name="synthetic_dense", kind="synthetic", nodes=1000, days=100, animals=1000, mode="graph"),
        # The score-function gradient of expected prevalence (forward run with score
        # terms, reverse sweep, moments), as torch.autograd's forward pass calls it.
        dict(name="score_gradient", kind="gradient", nodes=10000, days=365, replicates=128, chunk=1024, marks=53),
        # One evaluation of the parameter-fitting goal: ten trajectories, 21 regions.
        dict(name="fit_goal", kind="fit", nodes=37000, days=365, events=750000, replicates=10, regions=21, scale=1.6),
        # The general model, SIR of a few thousand nodes in one short run: launches and latency.
        dict(name="general_sir", kind="general", model="sir", nodes=2000, days=60, events=10000, replicates=1,
             mode="stream", source=W.Y_POST_EVENT),
        # The general model with many compartments: an Erlang infectious period in eight stages.
        dict(name="general_erlang", kind="general", model="erlang", nodes=1500, days=40, events=8000, replicates=1,
             mode="stream", source=W.Y_POST_EVENT),
        # SEIRS with two continuous variables under the midpoint update, national size, a year.
        dict(name="general_seirs", kind="general", model="seirs", nodes=37000, days=365, events=1000000, replicates=1,
             mode="graph", source=W.Y_MIDPOINT),
        # The national SISe3 network written as a general model, a year.
        dict(name="general_sise3", kind="general", model="sise3", nodes=37000, days=365, events=750000, replicates=1,
             mode="graph", source=W.Y_POST_EVENT),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("sise", "sise", "national", "batched", "uneven", "synthetic", "gradient", "fit",
                       "sir", "erlang", "seirs", "general_sise3"))
    if kind == "sise":
        n, t = _log(rng, 50, 5000), _log(rng, 10, 365)
        mode = rng.choice(("stream", "graph"))
        return dict(kind="advance", network="sise", nodes=n, days=t, events=20 * n * t // 365,
                    replicates=rng.choice((1, 1, 2, 5)), mode=mode,
                    chunk=rng.choice((1, 7)) if mode == "stream" and t <= 60 else t, pre_event=rng.random() < 0.3)
    if kind == "national":
        n, t = _log(rng, 3000, 37000), rng.randint(90, 730)
        return dict(kind="advance", network="national", nodes=n, days=t, events=int(3e6 * n / 37000 * t / 1460),
                    replicates=rng.choice((1, 1, 3)), mode="graph", chunk=t, pre_event=False)
    if kind == "batched":
        n, t, r = _log(rng, 5000, 37000), rng.randint(30, 200), rng.randint(16, 64)
        return dict(kind="advance", network="batched", nodes=n, days=t, events=int(3e6 * n / 37000 * t / 1460),
                    replicates=r, mode=rng.choice(("persistent", "persistent", "graph")), chunk=t, pre_event=False)
    if kind == "uneven":
        return dict(kind="uneven", instances=rng.randint(3, 32), nodes_lo=100, nodes_hi=_log(rng, 500, 10000),
                    days_lo=30, days_hi=rng.randint(90, 730), study=rng.randint(1, 10 ** 6))
    if kind == "synthetic":
        return dict(kind="synthetic", nodes=_log(rng, 50, 1000), days=rng.randint(10, 100),
                    animals=_log(rng, 30, 1500), mode=rng.choice(("stream", "graph")))
    if kind == "gradient":
        n, t = _log(rng, 2000, 10000), rng.randint(90, 365)
        return dict(kind="gradient", nodes=n, days=t, replicates=rng.randint(64, 128),
                    chunk=rng.choice((50, 1024)), marks=rng.randint(1, 53))
    if kind == "fit":
        n, t = _log(rng, 5000, 37000), rng.randint(60, 365)
        return dict(kind="fit", nodes=n, days=t, events=int(3e6 * n / 37000 * t / 1460), replicates=rng.randint(4, 10),
                    regions=rng.randint(5, 21), scale=round(rng.uniform(0.5, 1.6), 3))
    if kind == "sir":
        n, t = _log(rng, 100, 10000), _log(rng, 10, 120)
        return dict(kind="general", model="sir", nodes=n, days=t, events=5 * n * t // 60 + 1,
                    replicates=rng.choice((1, 1, 3)), mode=rng.choice(("stream", "graph")), source=W.Y_POST_EVENT)
    if kind == "erlang":
        n, t = _log(rng, 100, 10000), _log(rng, 10, 60)
        return dict(kind="general", model="erlang", nodes=n, days=t, events=5 * n * t // 40 + 1,
                    replicates=rng.choice((1, 1, 2)), mode=rng.choice(("stream", "graph")), source=W.Y_POST_EVENT)
    if kind == "seirs":
        n, t = _log(rng, 1000, 37000), _log(rng, 30, 365)
        return dict(kind="general", model="seirs", nodes=n, days=t, events=int(1e6 * n / 37000 * t / 365) + 1,
                    replicates=rng.choice((1, 2)), mode="graph",
                    source=rng.choice((W.Y_POST_EVENT, W.Y_PRE_EVENT, W.Y_MIDPOINT)))
    n, t = _log(rng, 3000, 37000), rng.randint(60, 365)
    return dict(kind="general", model="sise3", nodes=n, days=t, events=int(3e6 * n / 37000 * t / 1460), replicates=1,
                mode="graph", source=rng.choice((W.Y_POST_EVENT, W.Y_PRE_EVENT)))


# ---------------------------------------------------------------- inputs

def _advance_workload(c, seed):
    if c["network"] == "sise":
        return W.sise_plain(N=c["nodes"], T=c["days"], n_events=c["events"], seed=seed, R=c["replicates"],
                            gen_seed=seed)
    w = W.sise3_national(N=c["nodes"], T=c["days"], n_events=c["events"], seed=seed, R=c["replicates"], gen_seed=seed)
    if c["network"] == "batched":
        w = W.sise3_batched(R=c["replicates"], T=c["days"], seed=seed, base=w)
    return w


def _uneven_workloads(c, seed):
    """The study (models, sizes, horizons, parameters) belongs to the case; herds, events
    and random streams to the seed."""
    study = W.uneven_batch(n_inst=c["instances"], N_lo=c["nodes_lo"], N_hi=c["nodes_hi"], T_lo=c["days_lo"],
                           T_hi=c["days_hi"], events_per_node_year=0, seed=c["study"])
    out = []
    for i, w in enumerate(study):
        own = 1000 * seed + i
        mix = np.random.Generator(np.random.PCG64(own)).permutation(w.N)
        ev = W.sise_plain(N=w.N, T=w.T, n_events=int(round(80 * w.N * w.T / 365)), gen_seed=own).events
        out.append(dataclasses.replace(w, u0=np.ascontiguousarray(w.u0[:, mix]), events=ev, seed=own))
    return out


def _general_workload(c, seed):
    n, t, e, r = c["nodes"], c["days"], c["events"], c["replicates"]
    if c["model"] == "sir":
        return W.sir_general(N=n, T=t, n_events=e, R=r, seed=seed, gen_seed=seed)
    if c["model"] == "erlang":
        return W.erlang_sis(N=n, T=t, n_events=e, R=r, seed=seed, gen_seed=seed)
    if c["model"] == "seirs":
        return W.seirs_env(N=n, T=t, n_events=e, R=r, y_source=c["source"], seed=seed, gen_seed=seed)
    return W.as_general(W.sise3_national(N=n, T=t, n_events=e, seed=seed, gen_seed=seed), y_source=c["source"])


def _fit_inputs(c, seed):
    w = W.sise3_national(N=c["nodes"], T=c["days"], n_events=c["events"], seed=seed, gen_seed=seed)
    ups = np.array([8.8e-3, 3.2e-3, 1e-3])
    return w, ups, F.county_regions(w.N, c["regions"], seed=seed)


def _general_state(w):
    return np.repeat(w.u0[None], w.R, 0), np.repeat(w.y0[None], w.R, 0)


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "advance":
        w = _advance_workload(c, seed)
        sim = B.Sim.from_workload(w, phi_pre_event=c["pre_event"])
        sim.set_launch(c["mode"])
        st = dict(case=c, sim=sim)
        if c["replicates"] > 8:                    # large states stay on the device
            st["counts"] = torch.empty((w.R, w.nc, w.N), dtype=torch.int32, device="cuda")
            st["phi"] = torch.empty((w.R, w.N), dtype=torch.float64, device="cuda")
        return st
    if kind == "uneven":
        return dict(case=c, sims=[B.Sim.from_workload(w) for w in _uneven_workloads(c, seed)])
    if kind == "synthetic":
        w = W.synthetic_sis(N=c["nodes"], T=c["days"], S0=c["animals"], I0=c["animals"], seed=seed, gen_seed=seed)
        sim = B.Sim.from_workload(w)
        sim.set_launch(c["mode"])
        return dict(case=c, sim=sim)
    if kind == "gradient":
        w = W.sise_plain(N=c["nodes"], T=c["days"], n_events=20 * c["nodes"] * c["days"] // 365, seed=seed,
                         R=c["replicates"], gen_seed=seed)
        days = np.unique(np.linspace(0, c["days"] - 1, c["marks"] + 1).astype(np.int32)[1:])
        return dict(case=c, spec=G.GradientSpec(w, days, c["chunk"]))
    if kind == "fit":
        w, ups, regions = _fit_inputs(c, seed)
        ref = F.reference_totals(w, regions, c["regions"], ups)
        goal = F.Goal(w, regions, c["regions"], ref, trajectories=c["replicates"])
        return dict(case=c, goal=goal, k=c["scale"] * F.superparameters(ups, w.params.gamma[0]))
    w = _general_workload(c, seed)
    sim = B.GenSim.from_workload(w)
    sim.set_launch(c["mode"])
    u0, y0 = _general_state(w)
    return dict(case=c, sim=sim, u0=u0, y0=y0)


# ---------------------------------------------------------------- one pass

def _outputs(sim, counts=None, phi=None):
    if counts is None:
        counts, phi, _ = sim.state()
    else:
        sim.state_device(counts, phi)
    infected, animals, counters = sim.stats()
    return dict(counts=counts, phi=phi, infected=infected, animals=animals, counters=counters)


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind in ("advance", "synthetic"):
        sim = state["sim"]
        sim.reset()
        days, chunk = c["days"], c.get("chunk", c["days"])
        for d in range(0, days, chunk):
            sim.run(min(chunk, days - d))
            if chunk < days:
                sim.stats()                        # the prevalence so far
        return _outputs(sim, state.get("counts"), state.get("phi"))
    if kind == "uneven":
        for s in state["sims"]:
            s.reset()
        B.run_batch(state["sims"])
        outs = [_outputs(s) for s in state["sims"]]
        return {key: np.concatenate([o[key].ravel() for o in outs]) for key in outs[0]}
    if kind == "gradient":
        spec = state["spec"]
        moments, R, (f, score) = G.run_moments(spec, per_replicate=True)
        mean_f, grad, se = G.estimate(moments, R, spec.class_ratios())
        return dict(moments=moments, f=f, score=score, mean_f=mean_f, grad=grad, se=se)
    if kind == "fit":
        g2, vg2 = state["goal"](state["k"])
        s1, s2 = state["goal"].sim.region_moments()
        return dict(g2=g2, vg2=vg2, s1=s1.astype(np.int64), s2=s2.astype(np.int64))
    sim = state["sim"]
    sim.set_state(state["u0"], state["y0"], 0)
    sim.run(c["days"])
    counts, y, _ = sim.state()
    return dict(counts=counts, y=y)


# ---------------------------------------------------------------- what a pass cannot do without

def _sim_work(nodes, days, replicates, comps, conts, events, transitions, record=24, stats=True):
    """Counts and variables once in (one set shared by the replicates) and once out, the
    event list once, the daily statistics once; one draw per transition and node-day."""
    node_bytes = comps * 4 + conts * 8
    out = replicates * (nodes * node_bytes + (2 * days * 8 if stats else 0))
    draws = nodes * days * replicates * (transitions + 1.0)
    return dict(bytes=float(nodes * node_bytes + events * record + out), flops=draws * FLOPS_PER_DRAW)


def work(case):
    c = case
    kind = c["kind"]
    if kind == "advance":
        comps = 2 if c["network"] == "sise" else 6
        return _sim_work(c["nodes"], c["days"], c["replicates"], comps, 1, c["events"], TRANSITIONS[c["network"]])
    if kind == "uneven":                           # means of the log-uniform sizes and uniform horizons
        lo, hi = c["nodes_lo"], c["nodes_hi"]
        n = (hi - lo) / math.log(hi / lo)
        t = 0.5 * (c["days_lo"] + c["days_hi"])
        one = _sim_work(n, t, 1, 4, 1, 80 * n * t / 365, TRANSITIONS["uneven"])
        return dict(bytes=one["bytes"] * c["instances"], flops=one["flops"] * c["instances"])
    if kind == "synthetic":
        return _sim_work(c["nodes"], c["days"], 1, 2, 1, 12 * c["days"], 2.0 * c["animals"])
    if kind == "gradient":                         # the path's outputs are per-replicate, not per-node
        n, t, r = c["nodes"], c["days"], c["replicates"]
        draws = n * t * r * (TRANSITIONS["sise"] + 1.0)
        return dict(bytes=float(n * 16 + 24 * 20 * n * t / 365 + r * (2 * t * 8 + 64) + c["marks"] * 42 * 8),
                    flops=draws * (FLOPS_PER_DRAW + 8.0))
    if kind == "fit":
        one = _sim_work(c["nodes"], c["days"], c["replicates"], 6, 1, c["events"], TRANSITIONS["national_year"],
                        stats=False)
        return dict(bytes=one["bytes"] + 3 * 8 * c["days"] * c["regions"] * 6, flops=one["flops"])
    comps, conts = {"sir": (3, 0), "erlang": (10, 1), "seirs": (4, 2), "sise3": (6, 1)}[c["model"]]
    return _sim_work(c["nodes"], c["days"], c["replicates"], comps, conts, c["events"],
                     TRANSITIONS["general_" + c["model"]], record=28, stats=False)


# ---------------------------------------------------------------- the same in plain numpy binary64

_M32 = np.uint64(0xFFFFFFFF)


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 of uint64 arrays holding 32-bit words."""
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    x, y, z, w = np.broadcast_arrays(*(np.asarray(a, np.uint64) for a in (c0, c1, c2, c3)))
    s = np.uint64(32)
    for _ in range(10):
        a, b = x * np.uint64(0xD2511F53), z * np.uint64(0xCD9E8D57)
        x, y, z, w = (b >> s) ^ y ^ np.uint64(k0), b & _M32, (a >> s) ^ w ^ np.uint64(k1), a & _M32
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x, y, z, w


def _uniform(lo, hi):
    j = ((hi << np.uint64(32)) | lo) >> np.uint64(12)
    return (2.0 * j.astype(np.float64) + 1.0) * 2.0 ** -53


class _Transitions:
    """Rates a_j = k_j [y_q] [x_a] [x_b] [/ population] and their count changes."""

    def __init__(self, stoich, k, fa, fb, fy, pop):
        self.stoich = np.asarray(stoich, np.int64)
        self.k, self.fa, self.fb, self.fy = k, fa, fb, fy
        nc = self.stoich.shape[0]
        self.pop = [[c for c in range(nc) if (int(m) >> c) & 1] for m in pop]

    def rates(self, x, y):
        a = np.empty((len(self.k), x.shape[1]))
        for j, k in enumerate(self.k):
            r = np.full(x.shape[1], k)
            if self.fy[j] >= 0:
                r = r * y[self.fy[j]]
            if self.fa[j] >= 0:
                r = r * x[self.fa[j]]
            if self.fb[j] >= 0:
                r = r * x[self.fb[j]]
            if self.pop[j]:
                p = x[self.pop[j]].sum(0)
                r = np.where(p > 0, r / np.maximum(p, 1), 0.0)
            a[j] = r
        return a

    def day(self, x, y, day, rep, seed):
        """The direct method of every node on one day; returns the transitions fired."""
        if not len(self.k):
            return 0
        idx = np.arange(x.shape[1])
        t = np.zeros(idx.size)
        fired = k = 0
        while idx.size:
            P = np.cumsum(self.rates(x[:, idx], y[:, idx]), axis=0)
            on = P[-1] > 0
            idx, t, P = idx[on], t[on], P[:, on]
            if not idx.size:
                break
            w = _philox(idx, day, k, rep, seed)
            t = t - np.log(_uniform(w[0], w[1])) / P[-1]
            on = t < 1.0
            idx, t, P = idx[on], t[on], P[:, on]
            r = P[-1] * _uniform(w[2], w[3])[on]
            positive = np.diff(P, axis=0, prepend=0.0) > 0
            hit = positive & (r <= P)
            last = len(self.k) - 1 - np.argmax(positive[::-1], axis=0)
            j = np.where(hit.any(0), np.argmax(hit, axis=0), last)
            x[:, idx] += self.stoich[:, j]
            fired += idx.size
            k += 1
        return fired


def _words(e, day, rep, seed):
    block = 0
    while True:
        for w in _philox(e, day | 0x40000000, block, rep, seed):
            yield int(w)
        block += 1


def _apply_events(x, events, day, rep, seed, tally):
    """events: (position, kind, node, dest, count, compartments, offsets) in input order."""
    for e, kind, node, dest, count, comps, off in events:
        tally[1] += 1
        if kind == W.ENTER:
            x[comps[0] + off[comps[0]], node] += count
            continue
        have = [int(x[c, node]) for c in comps]
        total = sum(have)
        if count > total:
            tally[2] += 1
            count = total
        words = _words(e, day, rep, seed)
        for drawn in range(count):
            s = total - drawn
            m = next(words) * s
            if (m & 0xFFFFFFFF) < s:
                while (m & 0xFFFFFFFF) < (2 ** 32 - s) % s:
                    m = next(words) * s
            slot, i = m >> 32, 0
            while slot >= have[i]:
                slot -= have[i]
                i += 1
            have[i] -= 1
            c = comps[i]
            x[c, node] -= 1
            if kind == W.INTERNAL:
                x[c + off[c], node] += 1
            elif kind == W.EXTERNAL:
                x[c + off[c], dest] += 1


def _season(day):
    d = day % 365
    return 0 if d <= 91 else 1 if d <= 182 else 2 if d <= 273 else 3


def _simulate(u0, y0, tr, variables, events, days, rep, seed, source):
    """variables: per continuous variable (numerator, denominator or None, beta, alpha,
    eps); events: per day.  Returns counts, y, daily totals and counters."""
    x, y = u0.astype(np.int64), y0.copy()
    totals = np.zeros((days, 2), np.int64)
    tally = [0, 0, 0, 0]
    for d in range(days):
        sums = lambda: [(x[n].sum(0), None if q is None else x[q].sum(0)) for n, q, *_ in variables]
        start = sums()
        tally[0] += tr.day(x, y, d, rep, seed)
        before = sums()
        _apply_events(x, events[d], d, rep, seed, tally)
        after = sums()
        if variables:
            totals[d] = [after[0][0].sum(), x.sum()]
        for q, (_, _, beta, alpha, eps) in enumerate(variables):
            U, D = before[q] if source == W.Y_PRE_EVENT else after[q]
            if source == W.Y_MIDPOINT:
                U = 0.5 * (start[q][0] + U)
                D = None if D is None else 0.5 * (start[q][1] + D)
            mid = alpha * U if D is None else np.divide(alpha * U, D, out=np.zeros(U.shape), where=D > 0)
            y[q] = y[q] * (1.0 - beta[_season(d)]) + mid + eps
    return x, y, totals, tally


def _by_day(rows, day, days):
    out = [[] for _ in range(days)]
    for d, row in zip(day, rows):
        if d < days:
            out[int(d)].append(row)
    return out


def _exact_advance(c, seed):
    w = _advance_workload(c, seed) if c["kind"] == "advance" else W.synthetic_sis(
        N=c["nodes"], T=c["days"], S0=c["animals"], I0=c["animals"], seed=seed, gen_seed=seed)
    na = w.nc // 2
    fa = list(range(2 * na))
    fy = [0 if q % 2 == 0 else -1 for q in fa]
    stoich = np.zeros((2 * na, 2 * na), np.int64)
    for j in range(na):
        stoich[2 * j, 2 * j], stoich[2 * j + 1, 2 * j] = -1, 1
        stoich[2 * j + 1, 2 * j + 1], stoich[2 * j, 2 * j + 1] = -1, 1
    ev = w.events.stable_by_day()
    rows = []
    for e, (kind, node, dest, n, cls) in enumerate(zip(ev.kind, ev.node, ev.dest, ev.count, ev.cls)):
        comps = list(range(2 * na)) if cls < 0 else [2 * int(cls), 2 * int(cls) + 1]
        off = [2 if kind == W.INTERNAL else 0] * (2 * na)
        rows.append((e, int(kind), int(node), int(dest), int(n), comps, off))
    events = _by_day(rows, ev.day, w.T)
    infected = list(range(1, 2 * na, 2))
    p = w.params
    out = dict(counts=[], phi=[], infected=[], animals=[], counters=[])
    for r in range(w.R):
        k = [v for j in range(na) for v in (p.upsilon[r, j], p.gamma[r, j])]
        tr = _Transitions(stoich, k, fa, [-1] * (2 * na), fy, [0] * (2 * na))
        variables = [(infected, list(range(2 * na)), p.beta[r], p.alpha[r], p.epsilon[r])]
        x, y, totals, tally = _simulate(w.u0, w.phi0[None], tr, variables, events, w.T, r, seed,
                                        W.Y_PRE_EVENT if c.get("pre_event") else W.Y_POST_EVENT)
        for key, v in zip(out, (x.astype(np.int32), y[0], totals[:, 0], totals[:, 1], np.array(tally, np.int64))):
            out[key].append(v)
    return {key: np.stack(v) for key, v in out.items()}


def _exact_general(c, seed):
    w = _general_workload(c, seed)
    m = w.model
    bits = lambda mask: [q for q in range(m.nc) if (int(mask) >> q) & 1]
    ev = w.events
    order = np.argsort(ev.day, kind="stable")
    rows = []
    for e, i in enumerate(order):
        off = [0] * m.nc if ev.shift[i] < 0 else [int(v) for v in m.shift[ev.shift[i]]]
        rows.append((e, int(ev.kind[i]), int(ev.node[i]), int(ev.dest[i]), int(ev.count[i]),
                     bits(m.select[ev.select[i]]), off))
    events = _by_day(rows, ev.day[order], w.T)
    counts, ys = [], []
    for r in range(w.R):
        tr = _Transitions(m.stoich, w.rates[r], m.factor_a, m.factor_b, m.cont, m.pop_mask)
        variables = [(bits(m.num_mask[q]), bits(m.den_mask[q]) or None, w.var_params[r, q, 1:5],
                      w.var_params[r, q, 0], w.var_params[r, q, 5]) for q in range(m.ny)]
        x, y, _, _ = _simulate(w.u0, w.y0, tr, variables, events, w.T, r, seed, m.y_source)
        counts.append(x.astype(np.int32))
        ys.append(y)
    return dict(counts=np.stack(counts), y=np.stack(ys))


def exact(case, seed):
    """None where numpy would take over about 20 seconds: its time is one vector step per
    transition of the busiest node (about 0.4 ms) plus the transitions and events themselves."""
    c = case
    if c["kind"] not in ("advance", "synthetic", "general"):
        return None
    wk = work(c)
    transitions = wk["flops"] / FLOPS_PER_DRAW
    busiest = c["days"] * (3.0 * c["animals"] if c["kind"] == "synthetic" else
                           {"sise": 60, "sir": 80, "erlang": 200, "seirs": 200}.get(c.get("network", c.get("model")), 300))
    if c.get("replicates", 1) * (busiest * 4e-4 + c.get("events", 12 * c["days"]) * 6e-5) + transitions * 1e-6 > 20.0:
        return None
    return _exact_general(c, seed) if c["kind"] == "general" else _exact_advance(c, seed)
