"""The Crank--Nicolson update through FP32 transforms with FP64 residuals (helm32.cu), at mesh sizes
where its line groups are ragged or degenerate, y-z planes that just fit a block and that do not, prime
factors at and above the transforms' limit, field magnitudes far from one, fields of a pair that differ by
ten orders, and a time step whose operator needs the FP64 transforms.

pic_iterate's fields against the oracle's exact per-mode update with the general parity tolerance:
1e-12 of the field's norm (the solve itself ends at the rounding of its residual, a few 1e-16)."""

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


@pytest.mark.parametrize("n,dt,amp", [
    ((1, 8, 9), 0.1, 1.0), ((8, 1, 4), 0.1, 1.0), ((6, 4, 1), 0.1, 1.0), ((2, 3, 4), 0.1, 1.0),
    ((27, 2, 16), 0.1, 1.0), ((1024, 2, 3), 0.1, 1.0), ((3, 768, 2), 0.1, 1.0), ((2, 3, 512), 0.1, 1.0),
    ((48, 36, 54), 0.3, 1.0), ((6, 64, 64), 0.1, 1.0), ((4, 72, 64), 0.1, 1.0),
    ((50, 35, 22), 0.1, 1.0), ((127, 5, 7), 0.1, 1.0), ((2, 113, 65), 0.1, 1.0), ((3, 11, 508), 0.1, 1.0),
    ((127, 1, 1), 0.1, 1.0), ((131, 4, 5), 0.1, 1.0), ((16, 16, 16), 0.1, 1e-25), ((16, 16, 16), 0.1, 1e25), ((16, 12, 8), 60.0, 1.0),
])
def test_fields_match_the_exact_update(sim, n, dt, amp):
    rng = np.random.default_rng(sum(n))
    L = (1.3, 1.1, 0.9)
    x = rng.uniform(0, 1, size=(64, 3)) * L
    v = 1e-4 / dt * rng.normal(size=(64, 3))
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=dt, picard_tol=1e-13), x, v, -1e-3 * amp, 1e-3)
    st = s.get_state()
    for name in ("phi", "psi", "A", "U", "rho"):
        a = getattr(st, name)
        setattr(st, name, amp * rng.normal(size=a.shape))
    st.A[1] *= 1e-10                                           # A_y and A_z travel as one complex field
    st.U[1] *= 1e-10
    s.set_state(st)
    got = s.iterate(v)
    s.close()
    grid = opic.Config(n=n, L=L, dt=dt).grid()
    want = omesh.cn_fields(st.phi, st.psi, st.A, st.U, 0.5 * (got["rho"] + st.rho), got["J"], dt, 1.0, 1.0, 1.0, grid)
    for name, w in zip(("phi", "psi", "A", "U"), want):
        g = got[name]
        assert np.linalg.norm(g - w) <= 1e-12 * np.linalg.norm(w), name
    # the small component by itself: its solve is as good as its own residual
    assert np.linalg.norm(got["A"][1] - want[2][1]) <= 1e-12 * np.linalg.norm(want[2][1])
