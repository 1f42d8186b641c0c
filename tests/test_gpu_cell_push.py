"""The centred closed-form particle kernels (orbit_cell.cuh) at the edges of their walk: starts
exactly on knots moving either way or not at all, ends exactly on knots, orbits of several cells,
axes of 2 nodes, with the cell table and, where the allocator refuses it, with the gather table.

One Picard body against the oracle, with the tolerances of the general parity test (an orbit's
integrals are sums of a few dozen products of order one, so 1e-13 leaves two digits of margin)."""

import numpy as np
import pytest

from oracle import pic as opic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


def _edge_particles(n, npart, seed):
    """Cell-unit starts and displacements; H = 1 and dt = 1, so that knots are hit exactly."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(0, 1, size=(npart, 3)) * n
    b = rng.normal(scale=0.8, size=(npart, 3))
    k = npart // 8
    x[:k] = np.floor(x[:k])                                   # on a knot in every axis
    b[k // 2:k, 1] = 0.0                                      # ... resting on it in one
    b[k:2 * k] = np.round(b[k:2 * k])                         # whole cells: ends keep the offset
    x[2 * k:3 * k] = np.floor(x[2 * k:3 * k]) + 0.5
    b[2 * k:3 * k] = rng.integers(-3, 4, size=(k, 3)) + 0.5   # end exactly on a knot
    b[3 * k:4 * k] = 0.0
    b[4 * k:5 * k] = 2.6 * np.sign(b[4 * k:5 * k])            # two or three knots an axis
    b[5 * k:6 * k] *= 1e-9
    return x, np.clip(b, 0.5 - n, n - 0.5)                    # less than one box length


def _refuse_cell_tables(sim, monkeypatch, n):
    """Contexts get no cell tables from now on; the list of the requests refused."""
    refused = []
    want = 576 * n[0] * n[1] * n[2]
    base = sim._TorchAllocator

    class Refusing(base):
        def __init__(self, device):
            super().__init__(device)
            inner = self._alloc_cb

            def alloc(nbytes, stream, user):
                if nbytes == want:
                    refused.append(nbytes)
                    return None
                return inner(nbytes, stream, user)

            self._outer_cb = sim._lib.ALLOC_FN(alloc)
            self.struct = sim.PicAllocator(self._outer_cb, self._free_cb, None)

    monkeypatch.setattr(sim, "_TorchAllocator", Refusing)
    return refused


@pytest.mark.parametrize("n", [(8, 8, 8), (2, 5, 3), (9, 2, 4)])
@pytest.mark.parametrize("table", ["cells", "nodes"])
def test_one_body_matches_oracle_at_the_edges(sim, monkeypatch, n, table):
    refused = _refuse_cell_tables(sim, monkeypatch, n) if table == "nodes" else []
    L = tuple(float(k) for k in n)
    x, b = _edge_particles(np.asarray(n), 1601, 40 + n[0])
    v = 0.3 * b[::-1].copy()
    v_it = 2.0 * b - v                                        # vbar = b exactly up to rounding
    q = -1e-3
    cfg = sim.pic_config_default(n=n, L=L, dt=1.0, picard_tol=1e-13)
    s = sim.PicSim(cfg, x, v, q, 1e-3)
    assert bool(refused) == (table == "nodes")
    ocfg = opic.Config(n=n, L=L, dt=1.0, picard_tol=1e-13)
    o = opic.init(x, v, q, 1e-3, ocfg)
    g = s.iterate(v_it)
    it = opic.picard_iteration(o, v_it, ocfg, ocfg.grid())
    s.close()

    def rel(a, r):
        return np.linalg.norm(a - r) / max(np.linalg.norm(r), 1e-300)

    assert rel(g["J"], it["J"]) <= 1e-13
    for name in ("phi", "psi", "A", "U"):
        assert rel(g[name], it[name]) <= 1e-12, (name, rel(g[name], it[name]))
    assert rel(g["P"], it["P"]) <= 1e-13
    assert rel(g["v"], it["v_new"]) <= 1e-13
    d = g["x"] - it["xi"] * np.asarray(ocfg.grid().H)
    Lv = np.asarray(L)
    assert np.abs((d + 0.5 * Lv) % Lv - 0.5 * Lv).max() <= 1e-14 * Lv.max()


@pytest.mark.parametrize("n,npart", [((8, 8, 8), 1601), ((9, 2, 4), 1601), ((6, 5, 4), 39169)])
@pytest.mark.parametrize("table", ["cells", "nodes"])
def test_diagnosed_step_at_the_edges(sim, monkeypatch, n, npart, table):
    """The final sweep with diagnostics, by chunks of one warp and (from 38,913 particles on 152 SMs) of
    four: the state of the step without them to 1e-12 (other kernels, the same formulas), the particles'
    work and the mesh's, which are equal, to 100 times that (sums of terms of either sign), and the
    identities' residuals at rounding: a few dozen terms an orbit, 1e-13 of A."""
    refused = _refuse_cell_tables(sim, monkeypatch, n) if table == "nodes" else []
    L = tuple(float(k) for k in n)
    x, b = _edge_particles(np.asarray(n), npart, 70 + n[0])
    q = -1e-3 / npart
    out = []
    for diagnostics in (0, 1):
        s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=1.0, picard_tol=1e-13, diagnostics=diagnostics), x, b, q, 1e-3)
        assert bool(refused) == (table == "nodes")
        assert s.step(1).converged
        out.append((s.get_state(), s.diagnostics() if diagnostics else None))
        s.close()
    (o, _), (st, d) = out

    def rel(a, r):
        return np.linalg.norm(a - r) / max(np.linalg.norm(r), 1e-300)

    for name in ("P", "v", "phi", "psi", "A", "U"):
        assert rel(getattr(st, name), getattr(o, name)) <= 1e-12, name
    k1 = 0.5e-3 * np.sum(o.v ** 2)
    assert abs(d.K1 - k1) <= 1e-12 * k1
    assert abs(d.particle_work - d.mesh_work) <= 1e-10 * abs(d.mesh_work)
    assert d.RA_max <= 1e-13 * np.abs(o.A).max() and d.partition_max <= 1e-14


@pytest.mark.parametrize("precision", [0, 1])
def test_deterministic_steps_do_not_depend_on_the_particle_order(sim, precision):
    """A deterministic run restored from a checkpoint holds its particles in the caller's order, the
    run itself in the order of its last sort: the steps that follow have the same bits."""
    import torch
    rng = np.random.default_rng(11)
    n, L = (6, 5, 4), (1.2, 1.0, 0.8)
    x = rng.uniform(0, 1, size=(1500, 3)) * L
    v = rng.normal(scale=5e-3, size=x.shape)
    v[:, 0] += np.where(np.arange(1500) % 2 == 0, 0.2, -0.2)
    q = -L[0] * L[1] * L[2] / 1500
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=0.1, deterministic=1, precision=precision), x, v, q, -q)
    s.step(1)
    saved = s.checkpoint()
    s.step(2)
    want = s.checkpoint()
    s.restore(saved)
    s.step(2)
    got = s.checkpoint()
    for k in want:
        assert torch.equal(want[k], got[k]), k
    s.close()


@pytest.mark.parametrize("order,nq", [(1, 1), (1, 2), (1, 16), (2, 3), (2, 4), (2, 16), (3, 4), (3, 5), (3, 11)])
@pytest.mark.parametrize("n", [(8, 8, 8), (4, 5, 7)])
def test_gauss_pieces_match_oracle(sim, n, order, nq):
    """Split orbits with a Gauss rule: below the exact number of points, at it, and above it (where the
    library runs the fewest that are exact, or the closed forms), from starts on knots too.  Same
    tolerances; another context with another rule is alive, which must not change this one's."""
    L = tuple(float(k) for k in n)
    x, b = _edge_particles(np.asarray(n), 801, 60 + order)
    x[100:200] = np.mod(x[100:200] + 0.5, np.asarray(n))      # on the half-integer knots of even degrees
    v = 0.3 * b[::-1].copy()
    v_it = 2.0 * b - v
    q = -1e-3
    kw = dict(n=n, L=L, dt=1.0, picard_tol=1e-13)
    s = sim.PicSim(sim.pic_config_default(quadrature=1, nq=nq, shape_order=order, **kw), x, v, q, 1e-3)
    other = sim.PicSim(sim.pic_config_default(quadrature=1, nq=3 if nq != 3 else 2, shape_order=2, **kw), x, v, q, 1e-3)
    ocfg = opic.Config(quadrature="gauss", nq=nq, order=order, **kw)
    o = opic.init(x, v, q, 1e-3, ocfg)
    g = s.iterate(v_it)
    it = opic.picard_iteration(o, v_it, ocfg, ocfg.grid())
    s.close()
    other.close()

    def rel(a, r):
        return np.linalg.norm(a - r) / max(np.linalg.norm(r), 1e-300)

    assert rel(g["J"], it["J"]) <= 1e-13
    for name in ("phi", "psi", "A", "U"):
        assert rel(g[name], it[name]) <= 1e-12, (name, rel(g[name], it[name]))
    assert rel(g["P"], it["P"]) <= 1e-13
    assert rel(g["v"], it["v_new"]) <= 1e-13
