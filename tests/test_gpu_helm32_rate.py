"""The Helmholtz solves by FP32 transforms at loose tolerances: helmholtz_tol is met with the fewest
corrections, also on meshes of large primes, whose transforms round more."""

import numpy as np
import pytest

from oracle import mesh as omesh
from oracle import pic as opic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


@pytest.mark.parametrize("n,L", [((127, 61, 53), (130.0, 60.0, 55.0)), ((113, 127, 2), (1.3, 1.1, 0.9)),
                                 ((50, 35, 22), (1.3, 1.1, 0.9)), ((37, 41, 43), (0.13, 0.11, 0.09))])
@pytest.mark.parametrize("tol", [3e-6, 3e-7, 1e-7, 1.3e-12, 1.1e-13, 6.5e-14])
def test_loose_tolerances_are_met(sim, n, L, tol):
    """From a zero start, whose error is the solution itself, to within the tolerance and the rounding
    of the residual (1e-15)."""
    rng = np.random.default_rng(sum(n))
    dt = 0.05
    x = rng.uniform(0, 1, size=(4, 3)) * L
    v = np.zeros((4, 3))
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=dt, helmholtz_tol=tol), x, v, -1e-3, 1e-3)
    st = s.get_state()
    for name in ("phi", "A", "rho"):
        setattr(st, name, np.zeros_like(getattr(st, name)))
    for name in ("psi", "U"):
        setattr(st, name, rng.normal(size=getattr(st, name).shape))
    s.set_state(st)
    got = s.iterate(v)
    s.close()
    want = omesh.cn_fields(st.phi, st.psi, st.A, st.U, 0.5 * got["rho"], got["J"], dt, 1.0, 1.0, 1.0,
                           opic.Config(n=n, L=L, dt=dt).grid())
    for g, w in ((got["phi"], want[0]), *zip(got["A"], want[2])):
        assert np.linalg.norm(g - w) <= (tol + 1e-15) * np.linalg.norm(w)


@pytest.mark.parametrize("n,dt,transforms", [((1, 61, 61), 0.02, False), ((8, 61, 61), 0.1, False), ((1, 61, 61), 1.0, True),
                                             ((50, 35, 22), 0.1, True), ((62, 62, 62), 0.1, True)])
def test_solver_by_its_cost(sim, n, dt, transforms):
    """Transforms where they are the cheaper solve, Chebyshev steps (one launch) where not, by the launches of
    one body; the fields are the exact update's either way."""
    rng = np.random.default_rng(9)
    L = tuple(0.0654 * k for k in n)
    x = rng.uniform(0, 1, size=(8, 3)) * L
    v = 1e-3 * rng.normal(size=x.shape)
    launches = []
    for size in (n, (131, 2, 2)):                             # 131: never by transforms
        s = sim.PicSim(sim.pic_config_default(n=size, L=tuple(0.0654 * k for k in size), dt=dt), np.mod(x, 0.13), v, -1e-5, 1e-5)
        st = s.get_state()
        st.psi = rng.normal(size=st.psi.shape)
        s.set_state(st)
        s.profile(True)
        got = s.iterate(v)
        launches.append(s.profile(False).launches)
        s.close()
        if size == n:
            want = omesh.cn_fields(st.phi, st.psi, st.A, st.U, 0.5 * (got["rho"] + st.rho), got["J"], dt, 1.0, 1.0, 1.0,
                                   opic.Config(n=n, L=L, dt=dt).grid())[0]
            assert np.linalg.norm(got["phi"] - want) <= 1e-12 * np.linalg.norm(want)
    assert (launches[0] > launches[1]) == transforms, launches
