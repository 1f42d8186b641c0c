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


@pytest.mark.parametrize("npart", [1, 33, 256, 257, 1037])
def test_vjp_of_orbits_across_cells_matches_directional_differences(sim, npart):
    """The transposed deposits (per warp and cell, in chunks of 256) with partial warps and chunks, orbits
    across several cells and adjoints of very different size.  The difference quotient's own error,
    h^2 = 1e-8 relative and 1e-16 / 1e-7 of rounding, stays below the 1e-6 of the one-step test."""
    import torch
    rng = np.random.default_rng(npart)
    n, L = (6, 5, 4), (1.2, 1.0, 0.8)
    x = rng.uniform(0, 1, size=(npart, 3)) * L
    v = rng.normal(scale=0.3, size=x.shape)                    # dt v: up to three cells a step
    q = -1e-3 / npart
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=0.8, picard_tol=1e-14, picard_max=32), x, v, q, 1e-3 / npart)
    s.step(2)
    base = s.get_state_device()
    gen = torch.Generator(device="cuda").manual_seed(npart)
    keys = ("x", "v", "P", "phi", "psi", "rho", "A", "U")
    m = 1e-3 / npart
    d = {k: 1e-3 * (m if k == "P" else 1.0) * torch.randn(t.shape, generator=gen, device="cuda", dtype=torch.float64)
         for k, t in base.items()}
    lam = {k: torch.randn(t.shape, generator=gen, device="cuda", dtype=torch.float64) for k, t in base.items()}
    for k in ("x", "v", "P"):
        lam[k] *= (1.0 / m if k == "P" else 1.0) * 10.0 ** torch.randint(-3, 1, lam[k].shape, generator=gen, device="cuda")
    d["vprev"].zero_()
    lam["vprev"].zero_()
    Lv = torch.tensor(L, dtype=torch.float64, device="cuda")

    def step_from(st):
        s.set_state_device(st)
        assert s.step(1).converged
        return s.get_state_device()

    h = 1e-4
    plus = step_from({k: base[k] + h * d[k] for k in base})
    minus = step_from({k: base[k] - h * d[k] for k in base})
    diff = {k: plus[k] - minus[k] for k in base}
    dx = diff["x"].reshape(3, -1)
    diff["x"] = (((dx + 0.5 * Lv[:, None]) % Lv[:, None]) - 0.5 * Lv[:, None]).reshape(-1)   # minimal image
    dot = lambda a, b: sum(float((a[k] * b[k]).sum()) for k in keys)
    fd = dot(lam, diff) / (2 * h)
    s.set_state_device(base)
    assert s.step(1).converged
    lam_prev, info = s.step_vjp(lam)
    adj = dot(lam_prev, d)
    s.close()
    assert info.residual <= 1e-11
    assert abs(adj - fd) <= 1e-6 * max(abs(fd), float(sum((lam[k] * diff[k] / (2 * h)).abs().sum() for k in keys)) * 1e-2)


@pytest.mark.parametrize("npart", [1, 255, 257, 2000])
def test_fp32_iterations_end_near_the_fp64_fixed_point(sim, npart):
    """FP32 pieces of orbits across several cells, some from knots (exactly) and one ending on one: the
    first refinement of the FP32 iterate changes v by its rounding, 1e-7 times a few dozen terms of dv,
    dv / v below 0.1: 1e-6.  A piece in the wrong cell or with a wrong weight shows at 1e-3."""
    rng = np.random.default_rng(npart)
    n, L = (6, 5, 4), (6.0, 5.0, 4.0)
    x = rng.uniform(0, 1, size=(npart, 3)) * L
    b = rng.normal(scale=0.9, size=x.shape)
    x[: npart // 4] = np.floor(x[: npart // 4])
    b[npart // 8: npart // 4] = np.round(b[npart // 8: npart // 4]) + 0.25
    b = np.where(np.abs(b) < 0.1, 0.1, b)                       # (slow ones go to the local solves)
    s = sim.PicSim(sim.pic_config_default(n=n, L=L, dt=1.0, precision=1, picard_tol=1e-13), x, b, -0.2 / npart, 0.5 / npart)
    assert s.step(1).converged
    e_v, _, kind = s.residual_history()
    fp32 = [e for k, e in zip(kind, e_v) if k == 1]
    rest = [e for k, e in zip(kind, e_v) if k != 1]
    s.close()
    assert len(fp32) >= 2 and fp32[0] > 1e-5 and rest[0] <= 1e-6, (kind, e_v)


@pytest.mark.parametrize("more", [-1, 3])
def test_chunk_sizes_of_the_pushes(sim, more):
    """On both sides of the particle count from which the pushes take chunks of 512 (two for each of two
    blocks an SM), with a last chunk of one warp: one body against the oracle with the tolerances
    above, and the FP32-pair iteration by the FP64 residual of what it leaves: 1e-9 is a hundred times
    its 1e-15 of v over dv / v of 1e-4."""
    import torch
    npart = 2 * 2 * 512 * torch.cuda.get_device_properties(0).multi_processor_count + more
    n, L = (8, 8, 8), (8.0, 8.0, 8.0)
    rng = np.random.default_rng(5)
    x = rng.uniform(0, 1, size=(npart, 3)) * L
    v = rng.normal(scale=0.5, size=x.shape)
    q = -1e-2 / npart
    kw = dict(n=n, L=L, dt=1.0, picard_tol=1e-13)
    s = sim.PicSim(sim.pic_config_default(**kw), x, v, q, 1.0 / npart)
    ocfg = opic.Config(**kw)
    g = s.iterate(v)
    s.close()
    it = opic.picard_iteration(opic.init(x, v, q, 1.0 / npart, ocfg), v, ocfg, ocfg.grid())

    def rel(a, r):
        return np.linalg.norm(a - r) / max(np.linalg.norm(r), 1e-300)

    assert rel(g["J"], it["J"]) <= 1e-13 and rel(g["P"], it["P"]) <= 1e-13 and rel(g["v"], it["v_new"]) <= 1e-13
    s = sim.PicSim(sim.pic_config_default(precision=1, **kw), x, v, q, 1.0 / npart)
    assert s.step(1).converged
    e_v, _, kind = s.residual_history()
    s.close()
    pair = [i for i, k in enumerate(kind) if k == 2]
    assert pair and e_v[pair[-1] + 1] <= 1e-9, (kind, e_v)
