"""Quantities of very different size side by side: what the fixed-point sums hold is relative to the cell
and the particles at hand, not to the largest value of the mesh or of the warp."""

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


@pytest.mark.parametrize("ppc", [4, 64])
def test_push_ahead_of_a_localised_pulse(sim, ppc):
    """A field of order one in a few cells and 1e-9 elsewhere: the momenta of the particles elsewhere,
    from zero, against the oracle's push in the fields that the library returns.  A momentum is a sum of
    a few dozen products of the fields around its particle: 1e-13 of that size and a digit of margin."""
    rng = np.random.default_rng(3)
    n, dt, q, m = (16, 4, 5), 0.05, 1e-6, 1.0
    L = tuple(map(float, n))
    x = rng.uniform(0, 1, size=(ppc * int(np.prod(n)), 3)) * L
    v = rng.normal(scale=8.0, size=x.shape)
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=dt), x, v, q, m)
    st = s.get_state()
    for name in ("phi", "psi", "A", "U", "rho"):
        a = 1e-9 * rng.normal(size=getattr(st, name).shape)
        if name in ("phi", "A"):
            a[..., 7:9, :, :] *= 1e9
        setattr(st, name, a)
    st.P[:] = 0.0
    s.set_state(st)
    got = s.iterate(v)
    s.close()
    ocfg = opic.Config(n=n, L=L, dt=dt)
    grid = ocfg.grid()
    xi = st.x / np.asarray(grid.H)
    want = opic.push_particles(xi, st.v, st.P, v, q, m, st.A, got["A"], omesh.grad(0.5 * (got["phi"] + st.phi), grid),
                               0.5 * (got["U"] + st.U), ocfg, grid)["P"]
    # (the update's tail falls by a / 4 H^2 = 1.6e-4 every two cells)
    far = (np.abs(xi[:, 0] - 8.0) > 6.0)
    size = np.sqrt(np.mean(want[far] ** 2))
    assert size <= 1e-3 * np.abs(want).max()
    assert np.abs(got["P"] - want)[far].max() <= 1e-12 * size


@pytest.mark.parametrize("ppc", [1, 4, 64])
def test_current_of_slow_particles_beside_a_fast_one(sim, ppc):
    """One particle with velocity one among particles of 1e-9: the current at the nodes that it does
    not touch, to 1e-12 of its size there (sums of some dozens of products)."""
    rng = np.random.default_rng(4)
    n = (8, 4, 5)
    L = tuple(map(float, n))
    npart = ppc * int(np.prod(n))
    x = rng.uniform(0, 1, size=(npart, 3)) * L
    v = 1e-9 * rng.normal(size=x.shape)
    x[0], v[0] = (2.3, 1.4, 2.2), (0.6, -0.5, 0.7)
    kw = dict(n=n, L=L, dt=0.5)
    s = sim.PicSim(sim.pic_config_default(**kw), x, v, -1e-3, 1e-3)
    got = s.iterate(v)
    s.close()
    ocfg = opic.Config(**kw)
    grid = ocfg.grid()
    o = opic.init(x, v, -1e-3, 1e-3, ocfg)
    it = opic.orbit_current(o, v, ocfg, grid)
    alone = opic.orbit_current(opic.init(x[:1], v[:1], -1e-3, 1e-3, ocfg), v[:1], ocfg, grid)
    slow = alone == 0.0
    size = np.sqrt(np.mean(it[slow] ** 2))
    assert 0.0 < size <= 1e-6 * np.abs(it).max()
    assert np.abs(got["J"] - it)[slow].max() <= 1e-12 * size


@pytest.mark.parametrize("key", ["v", "P", "A"])
def test_adjoints_of_very_different_size(sim, key):
    """The vjp is linear in its cotangent: a unit one on a particle and 1e-6 on others of its warp, some 16
    cells away.  Around those the mesh adjoint is that of the small ones alone, to 1e-12: the unit one's own
    reaches them through the solve's tail (below 1e-25) and its rounding ((4e-7)^3 = 6e-20)."""
    import torch
    n, dt, q = (32, 4, 4), 0.05, 1e-10
    L = tuple(map(float, n))
    rng = np.random.default_rng(6)
    cells = np.stack(np.meshgrid(*[np.arange(k) for k in n], indexing="ij"), axis=-1).transpose(2, 1, 0, 3).reshape(-1, 3)
    x = cells + rng.uniform(0.1, 0.9, size=cells.shape)        # one particle a cell, in the order of the cells
    v = rng.normal(scale=0.5, size=x.shape)
    npart, N = len(x), len(x)
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=dt, picard_accel=0), x, v, q, 1.0)
    assert s.step(1).converged
    gen = torch.Generator(device="cuda").manual_seed(7)
    big, small = s.state_zeros(), s.state_zeros()
    if key == "A":
        big["A"].view(3, n[2], n[1], n[0])[:, 0, 0, 4] = 1.0
        small["A"].view(3, n[2], n[1], n[0])[:, 0, 0, 18:23] = 1e-6 * torch.randn(3, 5, generator=gen, device="cuda", dtype=torch.float64)
    else:
        big[key].view(3, npart)[:, 4] = 1.0
        small[key].view(3, npart)[:, 18:23] = 1e-6 * torch.randn(3, 5, generator=gen, device="cuda", dtype=torch.float64)
    out = []
    for lam in (small, {k: big[k] + small[k] for k in big}):
        o, info = s.step_vjp(lam)
        out.append(o)
        assert info.residual <= 1e-11
    s.close()
    for name in ("A", "U"):
        a, b = (o[name].view(3, n[2], n[1], n[0])[:, :, :, 17:25].cpu().numpy() for o in out)
        assert np.abs(a).max() > 0.0
        assert np.abs(b - a).max() <= 1e-12 * np.abs(a).max(), name
