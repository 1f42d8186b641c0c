"""FP32 offsets of positions just below a knot: they round to the knot itself, which is the start of the
next cell."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("cell", [1, 7])
@pytest.mark.parametrize("speed", [0.0, 1e-12, -1e-12, 0.3, -0.3])
def test_a_start_that_rounds_to_the_knot(sim, axis, cell, speed):
    """One particle, 1e-9 cells below a knot, resting or moving along its axis: the mixed step is the
    FP64 one, to the rounding of either (charges of 1e-6 leave forces of 1e-12)."""
    n, L = (8, 8, 8), (8.0, 8.0, 8.0)
    x = np.full((1, 3), 2.5)
    v = np.full((1, 3), 0.2)
    x[0, axis], v[0, axis] = cell + 1.0 - 1e-9, speed
    got = []
    for precision in (0, 1):
        s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=1.0, precision=precision, picard_accel=0, picard_tol=1e-13), x, v, 1e-6, 1.0)
        assert s.step(1).converged
        got.append(s.get_state())
        s.close()
    for name in ("x", "v", "P"):
        assert np.abs(getattr(got[1], name) - getattr(got[0], name)).max() <= 1e-13, name
