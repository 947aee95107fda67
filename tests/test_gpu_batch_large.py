"""GPU: the persistent kernel on runs whose nodes fill two blocks an SM (more than 304
blocks' worth), events staged and by owner lists, one handle and several, in every block
shape and the library's own, against the oracle."""
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
    B.batch_shape_auto()


CASES = {"staged": lambda: [W.sise3_national(N=2600, T=6, n_events=60, R=30)],
         "lists": lambda: [W.sise3_national(N=10_000, T=6, n_events=12_000, R=8)],
         "several": lambda: [W.sise3_national(N=5000, T=6, n_events=6000, R=9), W.sise_plain(N=33_000, T=9, n_events=9000),
                             W.sise_plain(N=700, T=4, n_events=900)]}
_REF = {}


def _reps(w):
    return [0, w.R - 1] if w.R > 1 else [0]


@pytest.mark.parametrize("shape", [None, *B.BATCH_SHAPES])
@pytest.mark.parametrize("case", list(CASES))
def test_runs_that_fill_two_blocks_an_sm(case, shape):
    ws = CASES[case]()
    assert sum(w.R * ((w.N + 255) // 256) for w in ws) > 304
    if case not in _REF:
        _REF[case] = [oracle.run(w, replicates=_reps(w)) for w in ws]
    B.batch_shape(*shape) if shape else B.batch_shape_auto()
    sims = [B.Sim.from_workload(w) for w in ws]
    B.run_batch(sims)
    for w, s, ref in zip(ws, sims, _REF[case]):
        counts, phi, day = s.state()
        _, _, ctr = s.stats()
        s.close()
        r = _reps(w)
        assert day == w.T and np.array_equal(counts[r], ref.counts) and np.array_equal(ctr[r], ref.counters)
        np.testing.assert_allclose(phi[r], ref.phi, rtol=1e-12, atol=0)
