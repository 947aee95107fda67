"""GPU: the general model's binary32 methods at their edges, every tier (one node per
thread, four per warp, one per warp, automatic) against the oracle bit for bit: each
unrolled size (4, 8, 16, 32 transitions), firings that change many compartments or by
more than one, populations that the firings change, counts that grow past the binary32
bound within a day, and continuous variables that have decayed to almost nothing."""
import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TIERS = {"thread": (1 << 30, 1 << 30), "group": (1 << 30, 0), "warp": (0, 1 << 30), "auto": (-1, -1)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


def _workload(name, model, u0, y0, rates, var_params, T, n_events=0, seed=3):
    rng = np.random.default_rng(seed)
    N = u0.shape[1]
    ev = W.GeneralEvents.empty()
    if n_events:
        ev = W.GeneralEvents(*(a.astype(np.int32) for a in (
            np.sort(rng.integers(0, T, n_events)), rng.choice([W.EXIT, W.ENTER], n_events),
            rng.integers(0, N, n_events), np.full(n_events, -1), rng.integers(1, 4, n_events),
            np.zeros(n_events), np.full(n_events, -1))))
    return W.GeneralWorkload(name, model, N, T, rates.shape[0], u0.astype(np.int32), y0, rates, var_params, ev, seed)


def _births(nt, start=60, T=8, N=70, birth=0.2):
    """Litters of three, a five-compartment reshuffle, deaths, infections and stages up to
    nt transitions; two populations change with the births."""
    comps = tuple(f"C{i}" for i in range(6))
    tr = [dict(change={"C0": 3}, a="C0", pop=comps),
          dict(change={"C0": -1}, a="C0"),
          dict(change={"C0": -1, "C1": 2, "C2": 1, "C3": 1, "C4": 1}, a="C0", b="C1", pop=("C0", "C1", "C5"))]
    stage = 1
    while len(tr) < nt:
        c, d = f"C{1 + stage % 5}", f"C{(2 + stage) % 6}"
        tr.append(dict(change={c: -1, d: 1} if c != d else {c: -1}, a=c))
        stage += 1
    m = W.general_model(comps, tr, selects=[comps])
    rng = np.random.default_rng(nt)
    u0 = np.zeros((6, N), np.int64)
    u0[0] = rng.integers(1, start + 1, N)
    u0[1] = rng.integers(0, 4, N)
    k = np.full(nt, 0.11)
    k[0], k[1], k[2] = birth * 3, 0.1, 0.4
    rates = np.tile(k, (2, 1)) * np.array([[1.0], [1.3]])
    return _workload(f"births{nt}", m, u0, np.zeros((0, N)), rates, np.zeros((2, 0, 6)), T, 300)


def _growth():
    # births at a few per animal and day from just below 2^21: past 2^22 within the run
    m = W.general_model(("A", "B"), [dict(change={"A": 127}, a="B"), dict(change={"B": -1}, a="B")], selects=[("A", "B")])
    u0 = np.array([[(1 << 21) - 300, (1 << 22) - 2000, 10], [200, 200, 200]], np.int64)
    return _workload("growth", m, np.repeat(u0, 3, 1), np.zeros((0, 9)), np.array([[8.0, 0.05]]),
                     np.zeros((1, 0, 6)), 3)


def _decayed():
    # an environment that nothing feeds: down to 1e-45 of the smallest binary32 constant
    m = W.general_model(("S", "I"), [dict(change={"S": -1, "I": 1}, a="S", cont=0),
                                     dict(change={"I": -1, "S": 1}, a="I"),
                                     dict(change={"S": -1, "I": 1}, a="S", cont=1)],
                        variables=[(("I",), ("S", "I")), (("I",), ())], selects=[("S", "I")])
    N = 90
    u0 = np.zeros((2, N), np.int64)
    u0[0], u0[1] = 40, np.arange(N) % 3
    y0 = np.stack([np.geomspace(1e-300, 1e-2, N), np.geomspace(1e-3, 1e-75, N)])
    vp = np.zeros((1, 2, 6))
    vp[0, :, 1:5] = 0.9
    return _workload("decayed", m, u0, y0, np.array([[0.7, 0.2, 0.5]]), vp, 40, 60)


CASES = {"births4": lambda: _births(4), "births8": lambda: _births(8), "births9": lambda: _births(9),
         "births17": lambda: _births(17), "births32": lambda: _births(32), "births3": lambda: _births(3),
         "growth": _growth, "decayed": _decayed}
_REF = {}


@pytest.mark.parametrize("tier", list(TIERS))
@pytest.mark.parametrize("case", list(CASES))
def test_general_edges_bitexact(case, tier):
    w = CASES[case]()
    if case not in _REF:
        _REF[case] = oracle.run_general(w)
    ref = _REF[case]
    s = B.GenSim.from_workload(w)
    warp, group = TIERS[tier]
    s.set_warp_threshold(warp)
    s.set_group_threshold(group)
    s.run(w.T)
    counts, y, _ = s.state()
    ctr = s.counters()
    s.close()
    assert ref.counters[:, 0].min() > 0
    assert np.array_equal(counts, ref.counts)
    assert np.array_equal(y, ref.y)
    assert np.array_equal(ctr, ref.counters)
