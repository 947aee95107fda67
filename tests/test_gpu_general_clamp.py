"""GPU: the choice between transitions where a decayed variable's rate, far below what
binary32 holds, lies between two others.  One draw (node 62, day 0, this seed) has -log(u1)
near 2^-19.6 and u2 near 2^-23.2, so a total rate that fires it puts the selection point r
near 2^-42; the rates are set so that r lies just above the first transition's, closer than
the smallest constant the binary32 methods use (2^-100) times the herd squared.  The second
transition, whose variable is 1e-200, must not fire: every tier against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SEED, NODE, S = 3168826953, 62, (1 << 21) - 2
TIERS = {"thread": (1 << 30, 1 << 30), "group": (1 << 30, 0), "warp": (0, 1 << 30), "auto": (-1, -1)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


def _workload():
    m = W.general_model(("S", "I"), [dict(change={"I": -1, "S": 1}, a="I"),
                                     dict(change={"S": -1, "I": 1}, a="S", b="S", cont=0),
                                     dict(change={"I": -1}, a="I")],
                        variables=[(("I",), ())], selects=[("S", "I")])
    w = oracle.philox([NODE, 0, 0, 0], [SEED & 0xffffffff, SEED >> 32])
    E = oracle.neglog(((int(w[1]) << 32) | int(w[0])) >> 12)
    u2 = oracle.uniform(int(w[2]), int(w[3]))
    total = 1.3 * E                                # the draw falls at 0.77 of the day
    shift = 2.0 ** -100 * S * S
    r = total * u2
    k0 = r - shift / 2                             # r above transition 0, below 0 and a clamped 1
    assert 2 * r * 2.0 ** -17 < shift              # decisive for the binary32 rule on both sides
    u0 = np.zeros((2, NODE + 1), np.int32)
    u0[:, NODE] = S, 1
    vp = np.zeros((1, 1, 6))
    vp[0, :, 1:5] = 0.5
    return W.GeneralWorkload("clamp", m, NODE + 1, 1, 1, u0, np.full((1, NODE + 1), 1e-200),
                             np.array([[k0, 1.0, total - k0]]), vp, W.GeneralEvents.empty(), SEED)


@pytest.mark.parametrize("tier", list(TIERS))
def test_decayed_rate_between_two_others(tier):
    w = _workload()
    ref = oracle.run_general(w)
    assert ref.counts[0, :, NODE].tolist() == [S, 0]             # transition 2 fires
    s = B.GenSim.from_workload(w)
    warp, group = TIERS[tier]
    s.set_warp_threshold(warp)
    s.set_group_threshold(group)
    s.run(1)
    counts, y, _ = s.state()
    ctr = s.counters()
    s.close()
    assert np.array_equal(counts, ref.counts) and np.array_equal(y, ref.y) and np.array_equal(ctr, ref.counters)
