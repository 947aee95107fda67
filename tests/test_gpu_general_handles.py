"""GPU: several general-model handles alive at once.  The kernel of an unrolled size is
shared by every model it holds, and models of one size need different amounts of shared
memory: a handle runs as before after smaller ones have been created, launch by launch,
as a captured graph and with the binary64 methods."""
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


def _stages(nt, nc, N=50, T=5):
    """nt transitions round a ring of nc compartments, per-head rates."""
    comps = tuple(f"C{i}" for i in range(nc))
    tr = [dict(change={comps[j % nc]: -1, comps[(j + 1 + j // nc % (nc - 1)) % nc]: 1}, a=comps[j % nc])
          for j in range(nt)]
    m = W.general_model(comps, tr, selects=[comps])
    u0 = np.random.default_rng(nt).integers(0, 9, (nc, N))
    return W.GeneralWorkload(f"stages{nt}x{nc}", m, N, T, 1, u0.astype(np.int32), np.zeros((0, N)),
                             np.full((1, nt), 0.17), np.zeros((1, 0, 6)), W.GeneralEvents.empty(), 11)


# (transitions, compartments) of the handle that runs and of those created after it
PAIRS = {"unroll32": ((32, 6), [(17, 6), (18, 3)]), "unroll16": ((16, 16), [(16, 10), (14, 9)]),
         "across": ((32, 16), [(9, 3), (14, 16), (26, 4), (16, 2)])}


@pytest.mark.parametrize("mode", ["stream", "graph", "exact"])
@pytest.mark.parametrize("pair", list(PAIRS))
def test_handle_runs_after_smaller_models_are_created(pair, mode):
    first, later = PAIRS[pair]
    ws = [_stages(*first)] + [_stages(*x) for x in later]
    sims = [B.GenSim.from_workload(w) for w in ws]
    for s in sims:
        if mode == "graph":
            s.set_launch("graph")
        if mode == "exact":
            s.set_clock_margin(0)
    for w, s in zip(ws, sims):
        ref = oracle.run_general(w)
        assert ref.counters[:, 0].min() > 0
        s.run(w.T)
        counts, _, day = s.state()
        ctr = s.counters()
        assert day == w.T and np.array_equal(counts, ref.counts) and np.array_equal(ctr, ref.counters), w.name
    for s in sims:
        s.close()
