"""GPU: the general model's event step against the oracle bit for bit, on both sides of the
compartment count (4) up to which a node's counts stay in registers: chains of transfers through several nodes, a transfer to
the node sampled next, events that take every animal, more than there are, or animals of
one compartment only, more draws than a Philox block holds, internal moves and entries
through a shift, and herds whose sum needs more than 32 bits."""
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


def _check(w):
    ref = oracle.run_general(w)
    s = B.GenSim.from_workload(w)
    s.run(w.T)
    counts, _, _ = s.state()
    ctr = s.counters()
    s.close()
    assert np.array_equal(counts, ref.counts) and np.array_equal(ctr, ref.counters)
    return ref


def _model(nc):
    # no transitions: the events alone; selects: all, the first half, one, the last half
    comps = tuple(f"C{i}" for i in range(nc))
    half = max(nc // 2, 1)
    lo, hi = comps[:half], comps[nc - half:]
    return comps, W.general_model(comps, [], selects=[comps, lo, comps[:1], hi] + [(c,) for c in comps],
                                  shifts=[{c: nc - half for c in lo}, {c: -(nc - half) for c in hi}])


@pytest.mark.parametrize("nc", [1, 2, 3, 4, 5, 8, 9, 15, 16])
def test_event_chains_bitexact(nc):
    comps, m = _model(nc)
    rng = np.random.default_rng(nc)
    N, T, R = 60, 12, 2
    rows = []
    for d in range(T):
        path = rng.permutation(N)
        at = 0
        while at + 6 < N:                          # chains a -> b -> c ..., the destination sampled next
            k = int(rng.integers(1, 6))
            for i in range(k):
                a, b = int(path[at + i]), int(path[at + i + 1])
                rows.append((d, W.EXTERNAL, a, b, int(rng.integers(0, 9)), int(rng.integers(0, 2)), -1))
                what = int(rng.integers(0, 6))
                if what == 0:
                    rows.append((d, W.ENTER, b, -1, int(rng.integers(0, 5)), int(rng.integers(1, 3)), 0 if nc > 1 else -1))
                elif what == 1 and nc > 1:
                    rows.append((d, W.INTERNAL, b, -1, int(rng.integers(0, 12)), 1, 0))
                elif what == 2:
                    rows.append((d, W.EXIT, a, -1, int(rng.integers(0, 40)), int(rng.integers(0, 4)), -1))
                elif what == 3:                    # back to the first node, in other compartments
                    rows.append((d, W.EXTERNAL, b, a, int(rng.integers(0, 6)), 3, 1 if nc > 1 else -1))
                elif what == 4:
                    rows.append((d, W.EXIT, b, -1, 10_000, 2, -1))
            at += k + 1
    ev = W.GeneralEvents(*(np.asarray(c, np.int32) for c in zip(*rows)))
    u0 = rng.integers(0, 12, size=(nc, N)).astype(np.int32)
    u0[:, ::7] = 0
    w = W.GeneralWorkload(f"chains{nc}", m, N, T, R, u0, np.zeros((0, N)), np.zeros((R, 0)), np.zeros((R, 0, 6)), ev, 5)
    ref = _check(w)
    assert ref.counters[:, 1].min() > 200 and ref.counters[:, 2].min() > 0


@pytest.mark.parametrize("nc", [3, 6, 16])
def test_event_sums_past_32_bits_bitexact(nc):
    comps, m = _model(nc)
    N, T = 8, 3
    top = (1 << 31) - 1 - 500
    u0 = np.full((nc, N), 40, np.int32)
    rows = [(0, W.ENTER, v, -1, top, 4 + c, -1) for v in range(6) for c in range(3 if v < 4 else 2)]
    for d in range(T):
        for v in range(8):
            rows.append((d, W.EXIT, v, -1, 11 + v, 0, -1))
        rows += [(d, W.EXTERNAL, 0, 6, 17, 0, -1), (d, W.EXTERNAL, 6, 7, 30, 0, -1), (d, W.EXTERNAL, 4, 7, 9, 0, -1)]
    ev = W.GeneralEvents(*(np.asarray(c, np.int32) for c in zip(*rows)))
    w = W.GeneralWorkload(f"wide{nc}", m, N, T, 1, u0, np.zeros((0, N)), np.zeros((1, 0)),
                          np.zeros((1, 0, 6)), ev, 9)
    _check(w)
