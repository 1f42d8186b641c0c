"""The optional cell tables: deterministic bits do not depend on whether they fit, and a context that holds
them gives them back to another one that needs the memory."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


class Limit:
    """Device memory of `capacity` bytes for all contexts created while it is in place."""

    def __init__(self, sim, monkeypatch, refuse=lambda nbytes: False):
        self.live, self.capacity, self.refused = {}, float("inf"), 0
        base = sim._TorchAllocator
        limit = self

        class Limited(base):
            def __init__(self, device):
                super().__init__(device)
                inner_alloc, inner_free = self._alloc_cb, self._free_cb

                def alloc(nbytes, stream, user):
                    if refuse(nbytes) or limit.used() + nbytes > limit.capacity:
                        limit.refused += 1
                        return None
                    ptr = inner_alloc(nbytes, stream, user)
                    if ptr:
                        limit.live[int(ptr)] = nbytes
                    return ptr

                def free(ptr, nbytes, stream, user):
                    limit.live.pop(int(ptr), None)
                    inner_free(ptr, nbytes, stream, user)

                self._outer = (sim._lib.ALLOC_FN(alloc), sim._lib.FREE_FN(free))
                self.struct = sim.PicAllocator(*self._outer, None)

        monkeypatch.setattr(sim, "_TorchAllocator", Limited)

    def used(self):
        return sum(self.live.values())


def particles(n, L, ppc, seed):
    rng = np.random.default_rng(seed)
    npart = ppc * int(np.prod(n))
    x = rng.uniform(0, 1, size=(npart, 3)) * L
    v = rng.normal(scale=5e-3, size=x.shape)
    v[:, 0] += np.where(np.arange(npart) % 2 == 0, 0.2, -0.2)
    q = -L[0] * L[1] * L[2] / npart
    return x, v, q, -q


@pytest.mark.parametrize("n", [(6, 5, 4), (11, 7, 5)])
def test_the_transforms_need_no_memory_of_their_own(sim, monkeypatch, n):
    """No request of the size of the Helmholtz transforms' scratch (16 bytes a cell), whose refusal would
    change the solver, and with it the bits of a deterministic run."""
    L, N = (1.2, 1.0, 0.8), int(np.prod(n))
    x, v, q, m = particles(n, L, 17, 21)
    limit = Limit(sim, monkeypatch, lambda b: b == 16 * N)
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=0.1, deterministic=1), x, v, q, m)
    assert s.step(1).converged and limit.refused == 0
    s.close()


TABLES = 576   # bytes a cell of one cell table


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ensemble", [False, True])
def test_tables_go_to_a_context_that_needs_the_memory(sim, monkeypatch, precision, ensemble):
    """A second run whose memory fits only without the first one's tables is created, and both go on:
    as runs alone, to rounding (the kernels without tables take the same sums in another arithmetic)."""
    n, L = (12, 10, 8), (1.2, 1.0, 0.8)
    N = int(np.prod(n))
    cfg = sim.pic_config_default(n=n, L=L, dt=0.05, picard_tol=1e-13, precision=precision)
    runs = [(cfg, *particles(n, L, 16, seed)) for seed in (31, 32)]
    alone = []
    for r in runs:
        s = sim.PicSim(*r)
        s.step(2)
        alone.append(s.get_state())
        s.close()
    with monkeypatch.context() as mp:
        bare = Limit(sim, mp, lambda b: b == TABLES * N)
        s = sim.PicSim(*runs[0])
        need = bare.used()
        s.close()
        assert bare.refused and need > 0 and not bare.live
    limit = Limit(sim, monkeypatch)
    first = sim.PicSim(*runs[0])
    full = limit.used()
    assert full >= need + (2 + precision) * TABLES * N   # the first holds its tables
    if ensemble:
        first.close()
        limit.capacity = full + need - TABLES * N
        e = sim.PicEnsemble(runs)
        e.step(2)
        got = [r.get_state() for r in e.runs]
        e.close()
    else:
        first.step(1)
        limit.capacity = full + need - TABLES * N
        second = sim.PicSim(*runs[1])
        first.step(1)                                 # from here on without tables
        second.step(2)
        got = [first.get_state(), second.get_state()]
        first.close()
        second.close()
    assert limit.refused and not limit.live
    for a, b in zip(got, alone):
        for name in ("v", "P", "phi", "A"):
            d = np.linalg.norm(getattr(a, name) - getattr(b, name)) / np.linalg.norm(getattr(b, name))
            assert d <= (1e-11 if precision == 0 else 1e-8), (name, d)


@pytest.mark.parametrize("n,ppc", [((6, 5, 4), 17), ((11, 7, 5), 17), ((16, 12, 16), 17), ((16, 16, 16), 80)])
@pytest.mark.parametrize("precision,diagnostics", [(0, 0), (0, 1), (1, 0)])
def test_deterministic_bits_do_not_depend_on_memory(sim, monkeypatch, n, ppc, precision, diagnostics):
    """The cell tables refused or granted: the same bits, in chunks of one warp, of four and (from 311,296
    particles on 152 SMs) of eight."""
    L, N = (1.2, 1.0, 0.8), int(np.prod(n))
    x, v, q, m = particles(n, L, ppc, 21)
    out = []
    for refuse in (False, True):
        with monkeypatch.context() as mp:
            Limit(sim, mp, lambda b: refuse and b == TABLES * N)
            s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=0.1, deterministic=1, precision=precision,
                                                  diagnostics=diagnostics), x, v, q, m)
            s.step(3)
            out.append(s.get_state())
            s.close()
    for name in ("x", "v", "P", "phi", "psi", "rho", "A", "U"):
        assert np.array_equal(getattr(out[0], name), getattr(out[1], name)), name
