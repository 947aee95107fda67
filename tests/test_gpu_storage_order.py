"""GPU: handles whose library keeps the state by herd size (2^15 node-replicates or more)
against the same run in the caller's own buffers, which stay in node order, and against
the oracle: every launch mode, the split day step, the group and warp tiers, region
sums, node ranges with their exchange, and state copies in and out, host and device."""
import numpy as np
import pytest

import oracle
from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu
R = 12                                             # 3,000 x 12 > 2^15


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


@pytest.fixture(scope="module")
def case():
    import torch
    w = W.sise3_national(N=3000, T=24, n_events=9000, R=R)
    rng = np.random.default_rng(5)
    w.params.upsilon[:] *= rng.uniform(0.5, 8.0, size=(R, 1))
    w.phi0[:] = rng.uniform(0.0, 0.5, size=w.N)
    c = torch.empty((R, w.nc, w.N), dtype=torch.int32, device="cuda")
    p = torch.empty((R, w.N), dtype=torch.float64, device="cuda")
    s = B.Sim.from_workload(w, state=(c, p))       # node order: the caller's buffers
    s.set_regions(np.arange(w.N) % 7, 7)
    s.run(w.T)
    ref = dict(counts=s.state()[0], phi=s.state()[1], stats=s.stats(), regions=s.region_moments())
    s.close()
    return w, ref


def _same(s, w, ref):
    counts, phi, day = s.state()
    assert day == w.T
    assert np.array_equal(counts, ref["counts"]) and np.array_equal(phi, ref["phi"])
    for a, b in zip(s.stats(), ref["stats"]):
        assert np.array_equal(a, b)


def test_reference_run_matches_the_oracle(case):
    w, ref = case
    o = oracle.run(w, replicates=[0, R - 1])
    assert np.array_equal(ref["counts"][[0, R - 1]], o.counts)


@pytest.mark.parametrize("mode", ["stream", "graph", "persistent", "flow"])
@pytest.mark.parametrize("warp,group", [(-1, -1), (200, 60)])
def test_launch_modes(case, mode, warp, group):
    w, ref = case
    s = B.Sim.from_workload(w)
    s.set_group_threshold(group)
    s.tune(warp)
    s.set_launch(mode)
    s.run(w.T)
    _same(s, w, ref)
    s.reset()
    s.run(10)
    s.run(w.T - 10)
    _same(s, w, ref)
    s.close()


def test_split_day_step_and_event_variants(case):
    w, ref = case
    for variant in (0, 1, 2):
        s = B.Sim.from_workload(w, event_variant=variant)
        s.set_split(True)
        s.run(w.T)
        _same(s, w, ref)
        s.close()


def test_state_copies_in_and_out(case):
    import torch
    w, ref = case
    a = B.Sim.from_workload(w)
    a.run(9)
    counts, phi, _ = a.state()
    c = torch.empty((R, w.nc, w.N), dtype=torch.int32, device="cuda")
    p = torch.empty((R, w.N), dtype=torch.float64, device="cuda")
    assert a.state_device(c, p) == 9
    assert np.array_equal(c.cpu().numpy(), counts) and np.array_equal(p.cpu().numpy(), phi)
    b = B.Sim.from_workload(w)
    b.set_state(counts, phi, 9)
    b.run(w.T - 9)
    got, gphi, _ = b.state()
    assert np.array_equal(got, ref["counts"]) and np.array_equal(gphi, ref["phi"])
    a.close(); b.close()


def test_region_sums(case):
    w, ref = case
    s = B.Sim.from_workload(w)
    s.set_regions(np.arange(w.N) % 7, 7)
    s.set_launch("graph")
    s.run(w.T)
    for a, b in zip(s.region_moments(), ref["regions"]):
        assert np.array_equal(a, b)
    s.close()


def test_node_ranges_with_their_exchange(case):
    import torch
    w, ref = case
    bounds = [0, 1300, 1300, w.N]
    ranks = []
    for k in range(3):
        s = B.Sim.from_workload(w)
        s.shard(bounds[k], bounds[k + 1])
        ranks.append(s)
    for d in range(w.T):
        n = ranks[0].touched_count(d)
        packs = torch.empty((3, R * w.nc * max(n, 1)), dtype=torch.int32, device="cuda")
        for k, s in enumerate(ranks):
            assert np.array_equal(s.touched_nodes(d), ranks[0].touched_nodes(d))
            s.run_day_stochastic()
            if n:
                s.pack_touched(packs[k].data_ptr())
        for s in ranks:
            if n:
                s.unpack_touched(packs.data_ptr(), bounds)
            s.run_day_events()
    for k, s in enumerate(ranks):
        counts, phi, _ = s.state()
        lo, hi = bounds[k], bounds[k + 1]
        assert np.array_equal(counts[:, :, lo:hi], ref["counts"][:, :, lo:hi])
        assert np.array_equal(phi[:, lo:hi], ref["phi"][:, lo:hi])
        s.close()


def test_pre_event_phi():
    import torch
    w = W.sise_plain(N=1500, T=15, n_events=3000, R=24)
    c = torch.empty((24, w.nc, w.N), dtype=torch.int32, device="cuda")
    p = torch.empty((24, w.N), dtype=torch.float64, device="cuda")
    a = B.Sim.from_workload(w, phi_pre_event=True)
    b = B.Sim.from_workload(w, phi_pre_event=True, state=(c, p))
    a.run(w.T); b.run(w.T)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    a.close(); b.close()

@pytest.mark.parametrize("J", [1, 7, 683])         # 683 x 6 x 8 bytes: past the slab table, region by region
def test_region_sums_of_large_herds(J):
    # slab sums add the low and high 16 bits of a count apart; one node of 2^29 animals
    w = W.sise3_national(N=5000, T=3, n_events=600, R=2)
    u0 = w.u0.copy()
    u0[4, 17] = 1 << 29
    u0[0, 4999] = (1 << 16) + 3
    import dataclasses
    w = dataclasses.replace(w, u0=u0)
    region = (np.arange(w.N) * 37) % J
    s = B.Sim.from_workload(w)
    s.set_regions(region, J)
    s1 = np.zeros((w.T, J, 6), np.uint64)
    s2 = np.zeros((w.T, J, 6), np.uint64)
    for d in range(w.T):
        s.run(1)
        counts = s.state()[0].astype(np.uint64)
        for r in range(w.R):
            tot = np.stack([np.bincount(region, weights=counts[r, c].astype(np.float64), minlength=J) for c in range(6)], 1)
            tot = tot.astype(np.uint64)
            s1[d] += tot
            s2[d] += tot * tot
    a, b = s.region_moments()
    s.close()
    assert np.array_equal(a, s1) and np.array_equal(b, s2)
