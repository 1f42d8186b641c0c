"""The adjoint of orbits that start exactly on a knot and hardly move across it (displacements down to
1e-20 cells, which vanish beside the coordinate)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


@pytest.mark.parametrize("ppc", ["cells", "nodes"])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_position_adjoint_of_starts_on_knots(sim, axis, ppc):
    """Charges of 1e-14 leave velocities alone (their kicks are of order q^2 = 1e-28), so that the orbit's
    displacement along the knot's axis is dt v.  The adjoint through the orbit current is smooth on either
    side of the knot: for displacements of 1e-20 to 1e-13 cells as for 1e-9, to a few times
    that."""
    import torch
    rng = np.random.default_rng(17)
    n, npart = (4, 5, 3), 96 if ppc == "cells" else 24        # (from one particle a cell on: cell tables)
    x = rng.uniform(0, 1, size=(npart, 3)) * n
    x[:, axis] = np.floor(x[:, axis])
    v = rng.normal(scale=0.4, size=x.shape)
    N = int(np.prod(n))
    gen = torch.Generator(device="cuda").manual_seed(5)
    lA = torch.randn(3 * N, generator=gen, device="cuda", dtype=torch.float64)

    def lam_x(beta):
        v[:, axis] = beta
        s = sim.PicSim(sim.pic_config_default(n=n, L=tuple(map(float, n)), dt=1.0, picard_accel=0, picard_tol=1e-13),
                       x, v, 1e-14, 1.0)
        z = s.state_zeros()
        s.set_state_device({**s.get_state_device(), **{k: z[k] for k in ("phi", "psi", "A", "U", "rho")}})
        assert s.step(1).converged
        assert np.abs(s.accepted()[0] - v).max() <= 1e-22
        lam = s.state_zeros()
        lam["A"] = lA
        out, info = s.step_vjp(lam)
        s.close()
        assert info.residual <= 1e-11
        return out["x"].cpu().numpy().reshape(3, npart)

    for side, tiny in ((-1e-9, (-1e-13, -1e-16, -1e-17, -1e-20)), (1e-9, (1e-20, 1e-17, 1e-13))):
        want = lam_x(side)
        assert np.abs(want).max() > 0.0
        for beta in tiny:
            assert np.abs(lam_x(beta) - want).max() <= 1e-7 * np.abs(want).max(), beta
