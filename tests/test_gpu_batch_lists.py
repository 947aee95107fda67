"""GPU: the persistent kernel's event items taken from owner lists, in one part or
several, against the oracle: days with too few blocks, with lists too long for a lane and
with no events beside days that suit, one and several replicates, clamped and skipped
events, and every block shape."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()
    yield
    B.batch_shape(*B.BATCH_SHAPES[0])


def _many():
    return W.sise3_national(N=2500, T=12, n_events=20_000)                       # several parts a day


def _few():
    return W.sise_plain(N=300, T=20, n_events=130)                               # fewer than 16 blocks a day


def _hub():
    return W.sise3_national(N=1500, T=10, n_events=9000, e1_source="powerlaw")   # lists past a lane's limit


def _mixed():
    # every other day empty, one day with a hub, replicates
    w = W.sise3_national(N=900, T=16, n_events=8000, R=3)
    ev = w.events.select(w.events.day % 2 == 0)
    hub = ev.day == 6
    ev.node[hub] = np.where(ev.kind[hub] == W.EXTERNAL, ev.node[hub], 5)
    return dataclasses.replace(w, events=ev)


def _scarce():
    w = W.sise_plain(N=400, T=15, n_events=6000, herd_lo=1, herd_hi=4)           # more asked than present
    return w


CASES = {"many": _many, "few": _few, "hub": _hub, "mixed": _mixed, "scarce": _scarce}
_REF = {}


@pytest.mark.parametrize("shape", B.BATCH_SHAPES)
@pytest.mark.parametrize("case", list(CASES))
def test_list_events_bitexact(case, shape):
    w = CASES[case]()
    if case not in _REF:
        _REF[case] = oracle.run(w)
    ref = _REF[case]
    B.batch_shape(*shape)
    s = B.Sim.from_workload(w)
    B.run_batch([s], until=[5])
    B.run_batch([s])
    counts, phi, day = s.state()
    _, _, ctr = s.stats()
    s.close()
    assert day == w.T
    assert np.array_equal(counts, ref.counts) and np.array_equal(phi, ref.phi)
    assert np.array_equal(ctr, ref.counters)


def test_list_events_error_policy():
    w = _scarce()
    s = B.Sim.from_workload(w, underflow_error=True)
    ref = oracle.run(w, underflow_error=True)
    B.run_batch([s])
    with pytest.raises(B.SimError) as e:
        s.state()
    assert e.value.status == B.SIM_E_UNDERFLOW
    counts, _, _ = s.state()
    _, _, ctr = s.stats()
    s.close()
    assert np.array_equal(counts, ref.counts) and np.array_equal(ctr, ref.counters)
