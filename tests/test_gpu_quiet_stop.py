"""GPU: the day's end at rates so small that the logarithm's absolute error is a sizable
part of the waiting time.  One draw (herd 506, day 0, this seed) has -log(u) near 2^-28.7;
phi0 is set so that its infection falls just inside or just outside the day.  Every tier
against the oracle bit for bit."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HERD, ANIMALS, E = 506, 400, 2.3059537639311172e-09
TIERS = {"auto": (-1, -1), "thread": (1 << 30, 1 << 30), "group": (1 << 30, 0), "warp": (0, 1 << 30)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


def _workload(excess):
    w = W.sise_plain(N=1000, T=1, n_events=0, upsilon=1.0, gamma=0.5, seed=12782889)
    u0 = np.zeros_like(w.u0)
    u0[0] = ANIMALS
    phi0 = np.zeros(w.N)
    phi0[HERD] = E * (1 + excess) / ANIMALS        # the draw falls at 1 / (1 + excess) of the day
    return dataclasses.replace(w, u0=u0, phi0=phi0)


@pytest.mark.parametrize("tier", list(TIERS))
@pytest.mark.parametrize("excess", [-1e-3, -2e-5, -6e-6, 1e-6, 6e-6, 2e-5, 1e-4, 1e-3])
def test_draw_at_the_days_end(excess, tier):
    w = _workload(excess)
    ref = oracle.run(w)
    assert ref.counters[0, 0] == (1 if excess > 0 else 0)
    s = B.Sim.from_workload(w)
    warp, group = TIERS[tier]
    s.set_group_threshold(group)
    s.tune(warp)
    s.run(w.T)
    counts, phi, _ = s.state()
    _, _, ctr = s.stats()
    s.close()
    assert np.array_equal(counts, ref.counts)
    assert np.array_equal(phi, ref.phi)
    assert np.array_equal(ctr, ref.counters)
