"""GPU: wide clock margins of the general model, with which many node-days of a unit are run
again: on thread units, on group units and with the automatic nodes, for every source of
the continuous update, against the oracle bit for bit."""
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


CASES = {"post": lambda: W.seirs_env(N=1001, T=5, n_events=1500, y_source=W.Y_POST_EVENT),
         "pre": lambda: W.seirs_env(N=1001, T=5, n_events=1500, y_source=W.Y_PRE_EVENT),
         "mid": lambda: W.seirs_env(N=1001, T=5, n_events=1500, y_source=W.Y_MIDPOINT),
         "erlang": lambda: W.erlang_sis(N=300, T=5, n_events=400),
         "few": lambda: W.sir_general(N=37, T=5, n_events=40)}
_REF = {}


@pytest.mark.parametrize("tier", [(1 << 30, 1 << 30), (1 << 30, 0), (-1, -1)])
@pytest.mark.parametrize("k", [1, 4, 7, 8])
@pytest.mark.parametrize("case", list(CASES))
def test_wide_margins(case, k, tier):
    w = CASES[case]()
    if case not in _REF:
        _REF[case] = oracle.run_general(w)
    ref = _REF[case]
    s = B.GenSim.from_workload(w)
    s.set_warp_threshold(tier[0])
    s.set_group_threshold(tier[1])
    s.run(1)
    s.set_clock_margin(k)
    s.run(w.T - 1)
    counts, y, _ = s.state()
    ctr = s.counters()
    s.close()
    assert np.array_equal(counts, ref.counts) and np.array_equal(y, ref.y) and np.array_equal(ctr, ref.counters)
