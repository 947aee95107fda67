"""GPU: the automatic launch shapes without the binary32 clock (clock margin 0), where every
herd of the SISe models is a warp's and the automatic choice follows the option both ways,
against the oracle in every launch mode; the general model's automatic nodes likewise."""
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


@pytest.mark.parametrize("mode", ["stream", "graph", "persistent", "flow"])
def test_every_herd_is_a_warps_without_the_binary32_clock(mode):
    w = W.sise3_national(N=3000, T=12, n_events=6000, R=3)
    ref = oracle.run(w)
    s = B.Sim.from_workload(w)
    auto = s.L.sim_warp_nodes(s.h)
    assert 0 < auto < w.N
    s.set_launch(mode)
    s.set_clock_margin(0)
    assert s.L.sim_warp_nodes(s.h) == w.N
    s.run(5)
    s.set_clock_margin(9)
    assert s.L.sim_warp_nodes(s.h) == auto
    s.run(3)
    s.set_clock_margin(0)
    s.run(w.T - 8)
    counts, phi, _ = s.state()
    _, _, ctr = s.stats()
    assert np.array_equal(counts, ref.counts) and np.array_equal(ctr, ref.counters)
    np.testing.assert_allclose(phi, ref.phi, rtol=1e-12, atol=0)
    assert s.tune(400) == s.L.sim_warp_nodes(s.h) < w.N                # a chosen threshold stays
    s.set_clock_margin(17)
    s.set_clock_margin(0)
    assert s.L.sim_warp_nodes(s.h) < w.N
    s.close()


def test_general_automatic_nodes_follow_the_margin():
    w = W.seirs_env(N=3000, T=6, n_events=2000)
    ref = oracle.run_general(w)
    s = B.GenSim.from_workload(w)
    warp, group = s.L.gen_warp_nodes(s.h), s.L.gen_group_nodes(s.h)
    assert 0 < warp < w.N
    s.run(2)
    s.set_clock_margin(0)
    total = w.u0.sum(0)
    assert s.L.gen_warp_nodes(s.h) == (total >= 600).sum()
    assert s.L.gen_group_nodes(s.h) == ((total >= 150) & (total < 600)).sum()
    s.run(2)
    s.set_clock_margin(16)
    assert (s.L.gen_warp_nodes(s.h), s.L.gen_group_nodes(s.h)) == (warp, group)
    s.run(w.T - 4)
    counts, y, _ = s.state()
    ctr = s.counters()
    s.close()
    assert np.array_equal(counts, ref.counts) and np.array_equal(y, ref.y) and np.array_equal(ctr, ref.counters)
