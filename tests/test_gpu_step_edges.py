"""GPU: the stochastic step's binary32 methods at the edges of their bounds, every
tier (one node per thread, per 8-lane group, per warp) against the oracle bit for bit:
rates so small that nearly every node-day ends at its first draw, one-animal and empty
herds, zero rates, herds at the size where binary32 counts stop being exact, and
node-days of thousands of transitions (hundreds of rounds of the clock)."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TIERS = {"thread": (1 << 30, 1 << 30), "group": (1 << 30, 0), "warp": (0, 1 << 30)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


def _quiet():
    # no infected animal, phi between 0 and 1e-9: rates down to 1e-12 and exactly 0
    w = W.sise3_national(N=700, T=40, n_events=0)
    u0 = w.u0.copy()
    u0[0::2] += u0[1::2]
    u0[1::2] = 0
    phi0 = np.geomspace(1e-12, 1e-2, w.N)
    phi0[::7] = 0.0
    return dataclasses.replace(w, u0=u0, phi0=phi0)


def _tiny_herds():
    w = W.sise3_national(N=300, T=60, n_events=3000)
    u0 = np.zeros_like(w.u0)
    rng = np.random.default_rng(3)
    for v in range(0, w.N, 2):
        u0[rng.integers(0, 6), v] = rng.integers(0, 3)
    return dataclasses.replace(w, u0=u0, phi0=np.full(w.N, 0.5))


def _zero_rates():
    w = W.sise3_national(N=200, T=30, n_events=0)
    p = W.Params.broadcast(1, [0.0, 7e-3, 0.0], [1.0 / 28, 0.0, 1.0 / 22], 1.0, W.vtec_beta(), 1e-6)
    return dataclasses.replace(w, params=p, phi0=np.full(w.N, 0.3))


def _large_herds():
    # 2^22 - 1, 2^22 and 2^23 animals: the last two are beyond the binary32 counts
    w = W.sise_plain(N=40, T=4, n_events=0, upsilon=1e-6, gamma=2e-6)
    u0 = w.u0.copy()
    u0[0], u0[1] = (1 << 22) - 1 - 1000, 1000
    u0[0, 10:20] += 1
    u0[0, 20:30] += 1 << 22
    return dataclasses.replace(w, u0=u0, phi0=np.full(w.N, 1.0))


def _dense():
    return W.synthetic_sis(N=40, T=3, S0=1500, I0=700)


CASES = {"quiet": _quiet, "tiny_herds": _tiny_herds, "zero_rates": _zero_rates, "large_herds": _large_herds,
         "dense": _dense}
_REF = {}


@pytest.mark.parametrize("tier", list(TIERS))
@pytest.mark.parametrize("case", list(CASES))
def test_step_edges_bitexact(case, tier):
    w = CASES[case]()
    if case not in _REF:
        _REF[case] = oracle.run(w)
    ref = _REF[case]
    warp, group = TIERS[tier]
    s = B.Sim.from_workload(w)
    s.set_group_threshold(group)
    s.tune(warp)
    s.run(w.T)
    counts, phi, _ = s.state()
    _, _, ctr = s.stats()
    s.close()
    assert np.array_equal(counts, ref.counts)
    assert np.array_equal(phi, ref.phi)
    assert np.array_equal(ctr, ref.counters)


def test_division_at_the_edges_of_its_quotient():
    # the device division starts from a binary32 reciprocal: quotients just above 1 and
    # just below 2, divisors that are powers of two or next to one, few-bit operands
    import torch
    rng = np.random.default_rng(9)
    n = 1 << 20
    one = np.uint64(1) << np.uint64(52)
    my = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    my[::4] = rng.integers(0, 4, my[::4].size, dtype=np.uint64)
    my[1::4] = (1 << 52) - 1 - rng.integers(0, 4, my[1::4].size, dtype=np.uint64)
    my |= one
    near = np.uint64(1) << rng.integers(0, 40, n, dtype=np.uint64)
    mx = np.where(rng.random(n) < 0.5, my + near, 2 * my - near)     # ratio near 1 or near 2
    ex = np.where(mx >= 2 * one, 1, 0).astype(np.uint64)
    x = ((np.uint64(1023) + ex) << np.uint64(52)) | ((mx >> ex) & (one - np.uint64(1)))
    y = (np.uint64(1023) << np.uint64(52)) | (my & (one - np.uint64(1)))
    xd = torch.from_numpy(x.view(np.float64).copy()).cuda()
    yd = torch.from_numpy(y.view(np.float64).copy()).cuda()
    out = torch.empty_like(xd)
    ref = torch.empty_like(xd)
    B.debug_div(xd.data_ptr(), yd.data_ptr(), out.data_ptr(), ref.data_ptr(), n, device=True)
    assert np.array_equal(out.cpu().numpy(), x.view(np.float64) / y.view(np.float64))
