"""GPU: rate constants that are a negative zero (phi0, upsilon or gamma of -0.0, which the
entry points take as they take 0.0), every tier, the score mode and a state set from
device memory, against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TIERS = {"auto": (-1, -1), "thread": (1 << 30, 1 << 30), "group": (1 << 30, 0), "warp": (0, 1 << 30)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


def _phi():
    w = W.sise_plain(N=200, T=2, n_events=0)
    phi0 = np.full(w.N, 0.2)
    phi0[::2] = -0.0
    return dataclasses.replace(w, phi0=phi0)


def _upsilon():
    w = W.sise_plain(N=200, T=3, n_events=0, upsilon=-0.0, gamma=0.3)
    return dataclasses.replace(w, phi0=np.full(w.N, 0.5))


def _gamma():
    w = W.sise_plain(N=200, T=3, n_events=0, upsilon=0.3, gamma=-0.0)
    return dataclasses.replace(w, phi0=np.full(w.N, 0.5))


def _both():
    w = W.sise_plain(N=64, T=2, n_events=0, upsilon=-0.0, gamma=-0.0)
    return dataclasses.replace(w, phi0=np.full(w.N, 0.5))


def _classes():
    w = W.sise3_national(N=200, T=4, n_events=0)
    p = W.Params.broadcast(1, [-0.0, 0.2, 0.1], [0.1, -0.0, 0.2], 1.0, W.vtec_beta(), 1e-6)
    return dataclasses.replace(w, params=p, phi0=np.where(np.arange(w.N) % 5 == 0, -0.0, 0.3))


def _idle_class():
    w = W.sise3_national(N=200, T=4, n_events=0)
    p = W.Params.broadcast(1, [-0.0, 0.2, 0.1], [-0.0, 0.1, 0.2], 1.0, W.vtec_beta(), 1e-6)
    return dataclasses.replace(w, params=p, phi0=np.full(w.N, 0.3))


CASES = {"phi": _phi, "upsilon": _upsilon, "gamma": _gamma, "both": _both, "classes": _classes,
         "idle_class": _idle_class}


@pytest.mark.parametrize("tier", list(TIERS))
@pytest.mark.parametrize("case", list(CASES))
def test_negative_zero_bitexact(case, tier):
    w = CASES[case]()
    ref = oracle.run(w)
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


@pytest.mark.parametrize("case", list(CASES))
def test_negative_zero_score(case):
    # the same sums as with a positive zero, bit for bit
    w = CASES[case]()
    ref = oracle.run(w)
    p = w.params
    plain = dataclasses.replace(w, phi0=w.phi0 + 0.0, params=W.Params(p.upsilon + 0.0, p.gamma + 0.0, p.alpha, p.beta,
                                                                      p.epsilon))
    got = []
    for x in (w, plain):
        s = B.Sim.from_workload(x, score=True)
        s.run(x.T)
        counts, _, _ = s.state()
        got.append((counts, s.stats()[2], s.score()))
        s.close()
    assert np.array_equal(got[0][0], ref.counts) and np.array_equal(got[0][1], ref.counters)
    assert np.array_equal(got[0][2], got[1][2])


def test_negative_zero_phi_from_device_memory():
    import ctypes
    import torch
    w = _phi()
    ref = oracle.run(w)
    s = B.Sim.from_workload(dataclasses.replace(w, phi0=np.full(w.N, 0.7)))
    counts = torch.from_numpy(w.u0[None].astype(np.int32).copy()).cuda()
    phi = torch.from_numpy(w.phi0[None].copy()).cuda()
    st = s.L.sim_set_state(s.h, ctypes.c_void_p(counts.data_ptr()), ctypes.c_void_p(phi.data_ptr()), 0, B.SIM_DEVICE,
                           B.current_stream())
    assert st == B.SIM_OK
    s.run(w.T)
    got, gphi, _ = s.state()
    s.close()
    assert np.array_equal(got, ref.counts) and np.array_equal(gphi, ref.phi)
