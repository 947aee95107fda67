"""Launch-shape autotuner.

For one workload it times each candidate setting -- the herd sizes from which a
node gets a warp or an 8-lane group (warp-per-node, four-per-warp and
thread-per-node stochastic step) and the launch mode of the daily loop (stream
launches, a captured CUDA graph, or the persistent work-stealing kernel, the
latter in each of its block shapes) -- over a short prefix of the horizon, checks
that every candidate ends in the bit-identical state (counts, phi, statistics,
counters), and keeps the fastest.  Settings never change results; the check
guards the implementation.
"""
from __future__ import annotations

import itertools
import time

import numpy as np

from . import binding as B

WARP_THRESHOLDS = (1 << 30, 1600, 800, 400, 200)
GROUP_THRESHOLDS = (1 << 30, 300, 200, 100)
LAUNCH_MODES = ("stream", "graph", "persistent")


def _fingerprint(sim):
    c, p, d = sim.state()
    pi, pn, ctr = sim.stats()
    return (c.tobytes(), p.tobytes(), pi.tobytes(), pn.tobytes(), ctr.tobytes(), d)


def _candidates(thresholds, groups, modes, shapes):
    for thr, gthr, mode in itertools.product(thresholds, groups, modes):
        if gthr >= thr and gthr != groups[0]:
            continue
        for shape in (shapes if mode == "persistent" else (None,)):
            yield thr, gthr, mode, shape


def apply(sim, best):
    """Puts an autotune result on a handle (the batch shape is process-wide)."""
    sim.set_group_threshold(best["group_threshold"])
    sim.tune(best["warp_threshold"])
    sim.set_launch(best["launch"])
    if best.get("batch_shape"):
        B.batch_shape(*best["batch_shape"])
    elif best["launch"] == "persistent":
        B.batch_shape_auto()


def autotune(workload, days=None, thresholds=WARP_THRESHOLDS, modes=LAUNCH_MODES, repeats=2,
             groups=(1 << 30,), shapes=(None,)):
    """Returns (best {"warp_threshold", "group_threshold", "launch", "batch_shape"},
    table [(threshold, group threshold, mode, batch shape, ms)]).  Group thresholds
    at or above the warp threshold are skipped (no herd would take the group path);
    the persistent mode is timed in every block shape of `shapes` (None: the
    library's choice; batch_shape is None for the other modes).  The choice is left
    to the library afterwards; apply() sets the winner's."""
    import torch
    w = workload
    nd = min(w.T, days if days is not None else max(10, w.T // 10))
    sim = B.Sim.from_workload(w)
    u0 = np.repeat(w.u0[None], w.R, 0)
    phi0 = np.repeat(w.phi0[None], w.R, 0)
    ref = None
    table = []
    try:
        for thr, gthr, mode, shape in _candidates(thresholds, groups, modes, shapes):
            sim.set_group_threshold(gthr)
            sim.tune(thr)
            sim.set_launch(mode)
            if shape:
                B.batch_shape(*shape)
            else:
                B.batch_shape_auto()
            best = float("inf")
            for rep in range(repeats + 1):                 # first pass warms up (graph capture, caches)
                sim.set_state(u0, phi0, 0)
                sim.reset()
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                sim.run(nd)
                sim.sync()
                dt = (time.perf_counter() - t0) * 1e3
                if rep:
                    best = min(best, dt)
            fp = _fingerprint(sim)
            if ref is None:
                ref = fp
            elif fp != ref:
                raise AssertionError(f"setting ({thr}, {gthr}, {mode}, {shape}) changed the results")
            table.append((thr, gthr, mode, shape, best))
    finally:
        sim.close()
        B.batch_shape_auto()
    thr, gthr, mode, shape, _ = min(table, key=lambda x: x[4])
    return {"warp_threshold": thr, "group_threshold": gthr, "launch": mode, "batch_shape": shape}, table


GENERAL_WARP_THRESHOLDS = (1 << 30, 1000, 600, 300)
GENERAL_GROUP_THRESHOLDS = (1 << 30, 300, 150, 100)


def autotune_general(workload, days=None, thresholds=GENERAL_WARP_THRESHOLDS, groups=GENERAL_GROUP_THRESHOLDS,
                     repeats=1):
    """The general model's warp and group thresholds (initial node populations from
    which the stochastic step takes a warp, or an 8-lane segment, per node): times
    each pair (group below warp) over a prefix of the horizon with the CUDA-graph
    day loop, checks that all end in the bit-identical state, and returns (best
    (warp, group), table [(warp, group, warp nodes, group nodes, ms)])."""
    import torch
    w = workload
    nd = min(w.T, days if days is not None else max(10, w.T // 10))
    sim = B.GenSim.from_workload(w)
    sim.set_launch("graph")
    u0 = np.repeat(w.u0[None], w.R, 0)
    y0 = np.repeat(w.y0[None], w.R, 0)
    ref = None
    table = []
    try:
        for thr, gthr in itertools.product(thresholds, groups):
            if gthr >= thr and gthr != groups[0]:
                continue
            nb = sim.set_warp_threshold(thr)
            ng = sim.set_group_threshold(gthr)
            best = float("inf")
            for rep in range(repeats + 1):
                sim.set_state(u0, y0, 0)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                sim.run(nd)
                c, y, _ = sim.state()
                dt = (time.perf_counter() - t0) * 1e3
                if rep:
                    best = min(best, dt)
            fp = (c.tobytes(), y.tobytes())
            if ref is None:
                ref = fp
            elif fp != ref:
                raise AssertionError(f"thresholds ({thr}, {gthr}) changed the results")
            table.append((thr, gthr, nb, ng, best))
    finally:
        sim.close()
    b = min(table, key=lambda x: x[4])
    return (b[0], b[1]), table
