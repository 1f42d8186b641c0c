"""State tensors of runs whose stream is not torch's current one."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


@pytest.mark.parametrize("call", ["get_state_device", "checkpoint"])
def test_state_tensors_wait_for_the_memory_they_take_over(sim, call):
    """A tensor that was freed while a copy from it was still waiting in torch's stream: its memory goes to
    the state's tensors, which the run writes on its own stream.  The copy must come out whole."""
    import torch
    rng = np.random.default_rng(2)
    n, npart = (16, 16, 16), 1 << 16
    x, v = rng.uniform(0, 1, size=(npart, 3)), 1e-3 * rng.normal(size=(npart, 3))
    e = sim.PicEnsemble([(sim.pic_config_default(n=n, L=(1.0, 1.0, 1.0), dt=0.1), x, v, -1e-4, 1e-4)])
    s = e.runs[0]
    want = s.get_state_device()
    for _ in range(3):
        old = [torch.full((3 * npart,), 7.0, dtype=torch.float64, device="cuda") for _ in range(5)]
        torch.cuda.synchronize()
        torch.cuda._sleep(100_000_000)                        # some 50 ms
        copies = [t.clone() for t in old]
        del old
        got = getattr(s, call)()
        torch.cuda.synchronize()
        assert all(bool((t == 7.0).all()) for t in copies)
        assert all(torch.equal(got[k], want[k]) for k in want)
        del got
    e.close()
