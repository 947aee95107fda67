"""GPU: reading and setting the state of a handle takes no device memory, whatever order
the library keeps the state in, and gives back every plane when the state is larger than
the copies' staging buffer."""
import numpy as np
import pytest

from paper_1502_02908_gb300 import binding as B
from paper_1502_02908_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load_library()


# 3,000 herds: 14 MB of counts and 5 of phi; 74 and 25 MB; an odd count of herds
@pytest.mark.parametrize("N,R", [(3000, 200), (3000, 1030), (2777, 1100)])
def test_state_copies_take_no_device_memory(N, R):
    import torch
    w = W.sise3_national(N=N, T=2, n_events=0, R=R)
    s = B.Sim.from_workload(w)
    rng = np.random.default_rng(N + R)
    counts = rng.integers(0, 1 << 20, (R, w.nc, N), dtype=np.int32)
    phi = rng.random((R, N))
    c = torch.empty((R, w.nc, N), dtype=torch.int32, device="cuda")
    p = torch.empty((R, N), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    first, _, _ = s.state()
    assert torch.cuda.mem_get_info()[0] == free
    s.set_state(counts, phi, 1)
    got, gphi, day = s.state()
    assert s.state_device(c, p) == day == 1
    assert torch.cuda.mem_get_info()[0] == free
    s.close()
    assert np.array_equal(first, np.repeat(w.u0[None], R, 0))
    assert np.array_equal(got, counts) and np.array_equal(gphi, phi)
    assert np.array_equal(c.cpu().numpy(), counts) and np.array_equal(p.cpu().numpy(), phi)
