"""Workloads of the time-step library, as a program that uses it calls them.

Five kinds of pass, each through the Python binding's public calls:

* ``step``      a run under way: restore a checkpoint, advance some steps, read the state back;
* ``ensemble``  the same for several independent runs advanced together;
* ``vjp``       one step of a differentiable run's backward pass: restore, step, transpose;
* ``iterate``   one body of the Picard loop on device arrays (nothing committed);
* ``cn``        the Crank--Nicolson mesh update alone, on caller-owned buffers.

The particles are two counter-streaming beams with the same uniform random positions, displaced
along x by ``eps sin(k1 x)``, with an optional thermal spread, as in the library's own inputs.
They are handed over in cell order, which is how a run under way holds them, or shuffled, which
is how a restart file in the original order does.
"""

import ctypes
import math

import numpy as np
import torch

from paper_2606_15035_gb300 import _lib, sim

SIDE = 2.0 * math.pi / 3.0
KEYS = sim.PicSim.STATE_KEYS
F64 = torch.float64

DEFAULTS = {
    "kind": "step", "nx": 8, "ny": 8, "nz": 8, "lx": SIDE, "ly": SIDE, "lz": SIDE, "per_beam": 8,
    "v0": 0.2, "eps": 1e-3, "vth": 0.0, "dt": 0.1, "steps": 1, "tol": 1e-13, "picard_max": 32,
    "mixed": False, "tol64": 1e-9, "det": False, "diag": False, "order": 1, "gauss": 0,
    "spectral": False, "shuffled": False, "runs": 1,
}


def _case(name, **kw):
    return dict(DEFAULTS, name=name, **kw)


def _mesh(n, side=SIDE):
    return {"nx": n, "ny": n, "nz": n, "lx": side, "ly": side, "lz": side}


def listed():
    return [
        # The smallest run anybody does: the cold 8^3 test with 8,192 electrons, where launches
        # and host round trips count.
        _case("step-8c-8k", **_mesh(8), per_beam=8, tol=1e-14),
        # The standard double-precision production run: 32^3, 64 electrons per cell.
        _case("step-32c-2M", **_mesh(32), per_beam=32, vth=1e-4, steps=2),
        # The same run in mixed precision, resumed from a restart file in the original order.
        _case("step-32c-2M-mixed", **_mesh(32), per_beam=32, vth=1e-4, steps=2, mixed=True, shuffled=True),
        # The large mixed-precision run the library is benchmarked on: 128^3, 134M electrons.
        _case("step-128c-134M-mixed", **_mesh(128), per_beam=32, vth=1e-4, mixed=True),
        # A box with unequal sides on a mesh that no radix-2/3 transform takes, few particles per
        # cell, diagnostics on: a parameter study's run.
        _case("step-ragged-diag", nx=50, ny=35, nz=22, lx=2.4, ly=1.9, lz=1.1, per_beam=7, vth=5e-3, eps=1e-2,
              diag=True, steps=2),
        # The paper's own test: 16^3, 131,072 electrons, 2 pi box, dt = 0.025, spectral operators,
        # linear shapes with the 16-point rule on every orbit piece.
        _case("step-16c-131k-gauss16", **_mesh(16, 2.0 * math.pi), per_beam=16, dt=0.025, tol=1e-11, picard_max=16,
              spectral=True, gauss=16, diag=True, steps=2),
        # Quadratic shapes with the exact 4-point rule and spectral operators.
        _case("step-36c-quadratic", nx=36, ny=32, nz=24, per_beam=8, vth=1e-3, order=2, gauss=4, spectral=True),
        # A run whose bits have to repeat.
        _case("step-24c-442k-det", **_mesh(24), per_beam=16, vth=1e-3, det=True),
        # A scan: 16 independent mixed-precision runs of uneven size stepped together.
        _case("ensemble-16", kind="ensemble", nx=48, per_beam=32, runs=16, mixed=True, steps=2),
        # One backward step of the differentiable run, 32^3 with 16 electrons per cell.
        _case("vjp-32c-524k", kind="vjp", **_mesh(32), per_beam=8, vth=1e-4),
        # One Picard body, as a caller with an outer solver of its own uses it.
        _case("iterate-64c-2M", kind="iterate", **_mesh(64), per_beam=4, vth=1e-3),
        # The allocation-free mesh update of a host application.
        _case("cn-32c", kind="cn", **_mesh(32)),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _smooth(rng, lo, hi):
    """A mesh size of the form 2^p 3^q."""
    return rng.choice([n for n in range(lo, hi + 1) if _odd_part(n) == 1])


def _odd_part(n):
    for p in (2, 3):
        while n % p == 0:
            n //= p
    return n


def draw(rng):
    kind = rng.choice(["step"] * 8 + ["ensemble", "vjp", "iterate", "cn"])
    c = dict(DEFAULTS, kind=kind)
    c["v0"] = round(rng.uniform(0.1, 0.3), 4)
    c["eps"] = round(_log(rng, 1e-4, 1e-2), 6)
    c["vth"] = rng.choice([0.0, round(_log(rng, 1e-4, 1e-2), 6)])
    if kind == "ensemble":
        c.update(nx=rng.choice([24, 32, 48]), per_beam=rng.randint(4, 32), runs=rng.randint(3, 16), mixed=True,
                 steps=rng.randint(1, 2))
        return c
    c["spectral"] = kind == "step" and rng.random() < 0.2
    c["mixed"] = kind == "step" and rng.random() < 0.5
    if kind == "step" and not c["mixed"] and rng.random() < 0.3:
        c["order"] = rng.choice([1, 2, 3])
        c["gauss"] = rng.randint((3 * c["order"] + 2) // 2, 8)
    c["tol64"] = rng.choice([1e-9, 1e-10, 0.0])
    c["det"] = kind == "step" and rng.random() < 0.15
    c["diag"] = kind == "step" and rng.random() < 0.2
    c["shuffled"] = rng.random() < 0.3
    # as many particles as the kind of run keeps affordable
    most = 2.0e7 if c["mixed"] else 4.0e6
    if c["order"] > 1 or kind == "vjp":
        most = 4.0e5
    c["per_beam"] = int(round(_log(rng, 2, 32)))
    cells = _log(rng, 3.0e3, most) / (2 * c["per_beam"])
    if kind == "cn":
        cells = _log(rng, 216, 2.7e4)
    smooth = c["spectral"] or rng.random() < 0.5
    for a in "xyz":
        n = max(6, int(round(cells ** (1.0 / 3.0) * rng.uniform(0.7, 1.4))))
        n = min(n, 32) if kind == "cn" else n
        c["n" + a] = _smooth(rng, max(6, 2 * n // 3), n) if smooth else n
        c["l" + a] = round(SIDE * rng.uniform(0.6, 1.4), 6)
    c["steps"] = rng.randint(1, 2) if kind == "step" else 1
    return c


# ---- inputs ------------------------------------------------------------------------------


def _dims(c):
    return (c["nx"], c["ny"], c["nz"]), (c["lx"], c["ly"], c["lz"])


def _config(c):
    n, L = _dims(c)
    kw = dict(n=n, L=L, dt=c["dt"], picard_tol=c["tol"], picard_max=c["picard_max"], diagnostics=int(c["diag"]),
              deterministic=int(c["det"]), ops=int(c["spectral"]), shape_order=c["order"])
    if c["mixed"]:
        kw.update(precision=1, mixed_tol64=c["tol64"])
    if c["gauss"]:
        kw.update(quadrature=1, nq=c["gauss"])
    return sim.pic_config_default(**kw)


def _particles(c, seed):
    """(x, v, q, m) on the GPU, in cell order unless the case says shuffled."""
    n, L = _dims(c)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    pairs = c["per_beam"] * n[0] * n[1] * n[2]
    Lt = torch.tensor(L, dtype=F64, device="cuda")
    pos = torch.rand(pairs, 3, generator=g, dtype=F64, device="cuda").mul_(Lt)
    pos[:, 0].add_(c["eps"] * torch.sin((2.0 * math.pi / L[0]) * pos[:, 0]))
    pos.remainder_(Lt)
    pos[pos >= Lt] = 0.0
    if not c["shuffled"]:
        key = torch.zeros(pairs, dtype=torch.int32, device="cuda")
        for a in (2, 1, 0):
            i = (pos[:, a] * (n[a] / L[a])).to(torch.int32).clamp_(0, n[a] - 1)
            key.mul_(n[a]).add_(i)
        pos = pos[torch.argsort(key)]
        del key
    # the beams' partners are neighbours, as a cell-ordered store holds them
    x = pos.repeat_interleave(2, dim=0)
    del pos
    v = torch.zeros(2 * pairs, 3, dtype=F64, device="cuda")
    if c["vth"] > 0.0:
        v.normal_(0.0, c["vth"], generator=g)
    v[0::2, 0] += c["v0"]
    v[1::2, 0] -= c["v0"]
    q = -L[0] * L[1] * L[2] / (2 * pairs)
    return x, v, q, abs(q)


def _save(run):
    """A checkpoint of one run into buffers of its own."""
    buf = run.state_zeros()
    buf["xi"] = torch.zeros(3 * run.np, dtype=F64, device="cuda")
    torch.cuda.synchronize()          # an ensemble's runs work on streams of their own
    _read(run, buf)
    st = _lib.lib().pic_get_positions(run.ctx, ctypes.c_void_p(buf["xi"].data_ptr()), 1)
    assert st == 0
    return buf


def _read(run, buf):
    sim.pic_get_state(run.ctx, sim.PicStateView(*[buf[k].data_ptr() for k in KEYS], 1))


def _members(c):
    """The cases of an ensemble's runs: sizes from the grids up to nx, 4 to per_beam a beam."""
    grids = [n for n in (16, 24, 32, 48) if n <= c["nx"]]
    r = np.random.RandomState(c["runs"] * 100 + c["nx"])
    out = []
    for k in range(c["runs"]):
        out.append(dict(c, kind="step", **_mesh(int(grids[(k + r.randint(2)) % len(grids)])),
                        per_beam=int(r.randint(4, c["per_beam"] + 1)), v0=float(r.uniform(0.1, 0.3)),
                        eps=float(10.0 ** r.uniform(-4, -2)), vth=0.0))
    return out


def _mesh_fields(c, seed):
    """Smooth fields plus noise for the mesh update: phi, psi (N), A, U (3 N), rho (N), J (3 N)."""
    n, _ = _dims(c)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    N = n[0] * n[1] * n[2]
    ix = [2.0 * math.pi * torch.arange(k, dtype=F64, device="cuda") / k for k in n]
    wave = torch.sin(ix[2])[:, None, None] + torch.cos(ix[1])[None, :, None] * torch.sin(ix[0])[None, None, :]
    out = {}
    for k, f in (("phi", 1), ("psi", 1), ("A", 3), ("U", 3), ("rho", 1), ("J", 3)):
        amp = torch.randn(f, 1, generator=g, dtype=F64, device="cuda")
        noise = torch.randn(f, N, generator=g, dtype=F64, device="cuda")
        out[k] = (0.01 * (amp * wave.reshape(1, N) + 0.05 * noise)).reshape(-1).contiguous()
    return out


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    n, L = _dims(c)
    if c["kind"] == "cn":
        s = _mesh_fields(c, seed)
        N = n[0] * n[1] * n[2]
        out = {k: torch.empty(f * N, dtype=F64, device="cuda") for k, f in
               (("phi", 1), ("psi", 1), ("A", 3), ("U", 3))}
        return {"case": c, "in": s, "out": out, "n": (ctypes.c_int32 * 3)(*n), "L": (ctypes.c_double * 3)(*L),
                "cfg": _config(c)}
    if c["kind"] == "ensemble":
        parts = [(_config(m),) + _particles(m, int(seed) * 64 + k) for k, m in enumerate(_members(c))]
        ens = sim.PicEnsemble(parts)
        saved = [_save(r) for r in ens.runs]
        out = [r.state_zeros() for r in ens.runs]
        return {"case": c, "ens": ens, "saved": saved, "out": out}
    x, v, q, m = _particles(c, seed)
    s = sim.PicSim(_config(c), x, v, q, m)
    state = {"case": c, "sim": s}
    if c["kind"] == "iterate":
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        kick = torch.randn(v.shape, generator=g, dtype=F64, device="cuda")
        state["v_iter"] = sim.soa(v + 1e-3 * c["v0"] * kick)
        N = s.ncell
        state["out"] = {k: torch.empty(f * N, dtype=F64, device="cuda") for k, f in
                        (("J", 3), ("rho", 1), ("phi", 1), ("psi", 1), ("A", 3), ("U", 3))}
        state["out"].update({k: torch.empty(3 * s.np, dtype=F64, device="cuda") for k in ("x", "P", "v")})
        return state
    del x, v
    state["saved"] = _save(s)
    if c["kind"] == "vjp":
        state["lam"] = _cotangent(c, s.np, s.ncell, m, seed)
    return state


def _cotangent(c, npart, ncell, m, seed):
    """What a backward pass hands down: an adjoint on every component of the state."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 2)
    lam = {}
    for k in KEYS:
        size = 3 * npart if k in ("x", "v", "P", "vprev") else (3 * ncell if k in ("A", "U") else ncell)
        lam[k] = torch.randn(size, generator=g, dtype=F64, device="cuda")
    lam["x"] *= m
    lam["v"] *= m
    lam["vprev"].zero_()
    return lam


# ---- one pass ----------------------------------------------------------------------------


def run(state):
    c = state["case"]
    if c["kind"] == "cn":
        i, o, cfg = state["in"], state["out"], state["cfg"]
        st = _lib.lib().pic_cn_update_static(
            state["n"], state["L"], cfg.dt, cfg.kappa, cfg.sigma1, cfg.sigma2, cfg.helmholtz_tol,
            *[i[k].data_ptr() for k in ("phi", "psi", "A", "U", "rho", "J")],
            *[o[k].data_ptr() for k in ("phi", "psi", "A", "U")],
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st != 0:
            raise sim.PicError(st, "pic_cn_update_static failed")
        return o
    if c["kind"] == "ensemble":
        runs = state["ens"].runs
        for r, b in zip(runs, state["saved"]):
            r.restore(b)
        state["ens"].step(c["steps"])
        for r, b in zip(runs, state["out"]):
            _read(r, b)
        return {k: torch.cat([b[k] for b in state["out"]]) for k in KEYS}
    s = state["sim"]
    if c["kind"] == "iterate":
        o = state["out"]
        sim.pic_iterate(s.ctx, state["v_iter"],
                        sim.PicIterateOut(*[o[k].data_ptr() for k in
                                            ("J", "rho", "phi", "psi", "A", "U", "x", "P", "v")], 1))
        return o
    s.restore(state["saved"])
    s.step(c["steps"])
    if c["kind"] == "vjp":
        lam, _ = s.step_vjp(state["lam"])
        return lam
    out = s.get_state_device()
    if c["diag"]:
        d = s.diagnostics()
        out["K1"], out["W1"] = d.K1, d.W1
    return out


def work(case):
    """Bytes: the state read once and written once (or a call's own inputs and outputs).  Flops:
    per particle and sweep about 230 for its orbit's gather and push and 130 per piece for its
    current, at the four sweeps that a Picard solve to roundoff needs at the least; the adjoint's
    transposed sweeps differentiate the same orbit in six directions."""
    c = dict(DEFAULTS, **case)
    if c["kind"] == "ensemble":
        each = [work(m) for m in _members(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n, L = _dims(c)
    N = n[0] * n[1] * n[2]
    npart = 2 * c["per_beam"] * N
    if c["kind"] == "cn":
        return {"bytes": 8.0 * 20 * N, "flops": 4.0 * 5 * N * math.log2(N)}
    pieces = 1.0 + c["v0"] * c["dt"] * n[0] / L[0]
    nodes = (c["order"] + 1) ** 3 / 8.0
    sweep = 360.0 * pieces * nodes * npart + 300.0 * N
    if c["kind"] == "iterate":
        return {"bytes": 8.0 * ((12 + 9) * npart + (9 + 12) * N), "flops": sweep}
    if c["kind"] == "vjp":
        return {"bytes": 8.0 * 4 * (12 * npart + 9 * N), "flops": 5 * sweep + 6 * 5 * sweep}
    return {"bytes": 8.0 * c["steps"] * 2 * (12 * npart + 9 * N), "flops": 5 * c["steps"] * sweep}


# ---- the same results in plain torch, 64 bits ----------------------------------------------
#
# B-splines of any degree by their recurrence, orbit integrals by a Gauss rule that is exact on
# each piece between knots, the mesh equations mode by mode with torch.fft, and plain Picard
# iteration to stagnation.


class _Plain:
    def __init__(self, c):
        self.c = c
        self.n, L = _dims(c)
        self.N = self.n[0] * self.n[1] * self.n[2]
        self.L = torch.tensor(L, dtype=F64, device="cuda")
        self.nt = torch.tensor(self.n, dtype=F64, device="cuda")
        self.H = self.L / self.nt
        self.dt, self.r = c["dt"], c["order"]
        self.koff = 0.5 if self.r % 2 == 0 else 0.0
        npart = 2 * c["per_beam"] * self.N
        self.q = -L[0] * L[1] * L[2] / npart
        self.m = -self.q
        self.dV = float(self.H.prod())
        t, w = np.polynomial.legendre.leggauss((3 * self.r + 2) // 2)
        self.rule = [(0.5 + 0.5 * float(a), 0.5 * float(b)) for a, b in zip(t, w)]
        self.sym = []
        for a, k in enumerate(self.n):
            mode = torch.fft.fftfreq(k, 1.0 / k, dtype=F64, device="cuda")
            if c["spectral"]:
                s = 2.0 * math.pi * mode / self.L[a]
                s = torch.where(2 * mode.abs() == k, torch.zeros_like(s), s)
            else:
                s = torch.sin(2.0 * math.pi * mode / k) / self.H[a]
                s = torch.where(s.abs() * self.H[a] < 1e-12, torch.zeros_like(s), s)
            self.sym.append(s.reshape([-1 if b == 2 - a else 1 for b in range(3)]))
        self.lam = -sum(s * s for s in self.sym)

    def hat(self, f):
        return torch.fft.fftn(f.reshape(-1, self.n[2], self.n[1], self.n[0]), dim=(1, 2, 3))

    def real(self, z):
        return torch.fft.ifftn(z, dim=(1, 2, 3)).real.reshape(z.shape[0], -1)

    def basis(self, x):
        """Per axis: first node, values, derivatives (per length) of the r + 1 splines at x."""
        f = torch.floor(x - self.koff)
        t = x - self.koff - f
        w = [torch.ones_like(t)]
        low = w
        for p in range(1, self.r + 1):
            low = w
            w = [((t + (p - j)) * low[j - 1] if j else 0.0) + ((1 - t + j) * low[j] if j < p else 0.0)
                 for j in range(p + 1)]
            w = [b / p for b in w]
        d = [((low[j - 1] if j else 0.0) - (low[j] if j < self.r else 0.0)) / self.H for j in range(self.r + 1)]
        return f.long() - (self.r - 1) // 2, w, d

    def nodes(self, x):
        """Visit the shape's nodes: (node, value, gradient (3))."""
        first, w, d = self.basis(x)
        k = self.r + 1
        ax = [[(first[:, a] + j) % self.n[a] for j in range(k)] for a in range(3)]
        for z in range(k):
            for y in range(k):
                row = self.n[0] * (ax[1][y] + self.n[1] * ax[2][z])
                yz = w[y][:, 1] * w[z][:, 2]
                for i in range(k):
                    yield (ax[0][i] + row, w[i][:, 0] * yz,
                           (d[i][:, 0] * yz, w[i][:, 0] * d[y][:, 1] * w[z][:, 2],
                            w[i][:, 0] * w[y][:, 1] * d[z][:, 2]))

    def quadrature(self, xi, beta):
        """Points of every orbit: (particles, positions, s, weight)."""
        x = xi - self.koff
        fwd = beta > 0
        near = torch.where(fwd, torch.floor(x) + 1.0, torch.ceil(x) - 1.0)
        far = torch.where(fwd, torch.ceil(x + beta), torch.floor(x + beta))
        safe = torch.where(beta == 0, torch.ones_like(beta), beta)
        most = int((far - near).abs().max().item()) + 2
        cols = [torch.zeros_like(x[:, :1])]
        for k in range(most):
            s = (near + torch.where(fwd, 1.0, -1.0) * k - x) / safe
            s = torch.where((beta != 0) & (s > 0) & (s < 1), s, torch.ones_like(s))
            if bool((s < 1).any()):
                cols.append(s)
        S = torch.cat(cols + [torch.ones_like(x[:, :1])], dim=1).sort(dim=1).values
        for j in range(S.shape[1] - 1):
            h = S[:, j + 1] - S[:, j]
            idx = torch.nonzero(h.detach() > 0).squeeze(1)
            if idx.numel() == 0:
                continue
            for t, w in self.rule:
                s = S[idx, j] + t * h[idx]
                yield idx, xi[idx] + s[:, None] * beta[idx], s, w * h[idx]

    def deposit(self, xi):
        rho = torch.zeros(self.N, dtype=F64, device="cuda")
        for g, S, _ in self.nodes(xi):
            rho = rho.index_add(0, g, (self.q / self.dV) * S)
        return rho

    def start(self, x, v):
        """The state of a new run: charge without its null modes, potential from Poisson."""
        s = {"xi": torch.remainder(x / self.H, self.nt), "v": v, "vprev": v, "P": self.m * v}
        h = self.hat(self.deposit(s["xi"]) + 1.0)
        h = torch.where(self.lam == 0, torch.zeros_like(h), h)
        s["rho"] = self.real(h)[0]
        s["phi"] = self.real(h / torch.where(self.lam == 0, -torch.ones_like(self.lam), -self.lam))[0]
        s["psi"] = torch.zeros_like(s["rho"])
        s["A"] = torch.zeros(3, self.N, dtype=F64, device="cuda")
        s["U"] = torch.zeros_like(s["A"])
        return s

    def current(self, s, v1):
        vb = 0.5 * (v1 + s["v"])
        beta = self.dt * vb / self.H
        J = torch.zeros(3, self.N, dtype=F64, device="cuda")
        for idx, x, _, w in self.quadrature(s["xi"], beta):
            c = (self.q / self.dV) * vb[idx] * w[:, None]
            for g, S, _ in self.nodes(x):
                J = J.index_add(1, g, (c * S[:, None]).T)
        return J

    def fields(self, s, J):
        hJ = self.hat(J)
        rho = s["rho"] - self.dt * self.real(sum(1j * self.sym[a] * hJ[a] for a in range(3))[None])[0]
        src = torch.cat([0.5 * (rho + s["rho"])[None], J])
        u0 = torch.cat([s["phi"][None], s["A"]])
        w0 = torch.cat([s["psi"][None], s["U"]])
        a = 0.25 * self.dt ** 2
        u1 = self.real(((1 + a * self.lam) * self.hat(u0) + self.hat(self.dt * w0 + 2 * a * src)) / (1 - a * self.lam))
        w1 = 2.0 * (u1 - u0) / self.dt - w0
        hp = self.hat(0.5 * (u0[0] + u1[0]))
        grad = torch.stack([self.real(1j * self.sym[b] * hp)[0] for b in range(3)])
        return {"rho": rho, "phi": u1[0], "A": u1[1:], "psi": w1[0], "U": w1[1:], "grad": grad}

    def push(self, s, f, v1):
        vb = 0.5 * (v1 + s["v"])
        beta = self.dt * vb / self.H
        force = torch.zeros_like(vb)
        for idx, x, t, w in self.quadrature(s["xi"], beta):
            vi = vb[idx]
            out = torch.zeros_like(vi)
            for g, S, dS in self.nodes(x):
                A = ((1 - t)[:, None] * s["A"][:, g].T + t[:, None] * f["A"][:, g].T)
                Av = (A * vi).sum(dim=1)
                out = out + Av[:, None] * torch.stack(dS, dim=1) - S[:, None] * f["grad"][:, g].T
            force = force.index_add(0, idx, w[:, None] * out)
        P = s["P"] + self.dt * self.q * force
        xi = s["xi"] + beta
        xi = xi - self.nt * torch.floor(xi.detach() / self.nt)
        A = torch.zeros_like(vb)
        for g, S, _ in self.nodes(xi):
            A = A + S[:, None] * f["A"][:, g].T
        return dict(f, xi=xi, P=P, v=(P - self.q * A) / self.m, vprev=s["v"])

    def solve(self, s):
        """v* with G(v*) = v* by plain Picard iteration, to stagnation."""
        v1 = 2.0 * s["v"] - s["vprev"]
        last = math.inf
        for k in range(60):
            new = self.push(s, self.fields(s, self.current(s, v1)), v1)["v"]
            change = float((new - v1).norm() / new.norm())
            v1 = new
            if change < 1e-15 or (change < 1e-13 and change > 0.5 * last):
                break
            last = change
        return v1

    def step(self, s):
        v1 = self.solve(s)
        return self.push(s, self.fields(s, self.current(s, v1)), v1)

    def flat(self, s):
        """The layout of the library's device state."""
        out = {k: s[k].T.reshape(-1) for k in ("v", "P", "vprev")}
        out["x"] = (s["xi"] * self.H).T.reshape(-1)
        out.update({k: s[k].reshape(-1) for k in ("phi", "psi", "rho", "A", "U")})
        return {k: out[k] for k in KEYS}

    def vjp(self, s, lam):
        """The transposed step: the implicit-function theorem on v* = G(v*), by autograd."""
        v1 = self.solve(s).requires_grad_()
        inputs = {k: t.clone().requires_grad_() for k, t in s.items() if k != "vprev"}
        out = self.push(inputs, self.fields(inputs, self.current(inputs, v1)), v1)
        x = out["xi"] * self.H
        cot = {k: lam[k].reshape(3, -1) for k in ("A", "U")}
        cot.update({k: lam[k] for k in ("phi", "psi", "rho")})
        cot.update({k: lam[k].reshape(3, -1).T for k in ("x", "v", "P")})
        base = sum((t * cot[k]).sum() for k, t in dict(out, x=x).items() if k in cot)
        mu = torch.zeros_like(v1)
        direct, = torch.autograd.grad(base, v1, retain_graph=True)
        for _ in range(200):
            more, = torch.autograd.grad(out["v"], v1, mu, retain_graph=True)
            new = direct + more
            change = float((new - mu).norm() / new.norm())
            mu = new
            if change < 1e-14:
                break
        names = list(inputs)
        got = torch.autograd.grad([base, out["v"]], [inputs[k] for k in names], [torch.ones_like(base), mu],
                                  allow_unused=True)
        d = {k: torch.zeros_like(inputs[k]) if t is None else t for k, t in zip(names, got)}
        # the library's state holds positions in length units
        res = {"x": (d["xi"] / self.H).T.reshape(-1), "v": d["v"].T.reshape(-1), "P": d["P"].T.reshape(-1)}
        res["vprev"] = torch.zeros_like(res["v"])
        res.update({k: d[k].reshape(-1) for k in ("phi", "psi", "rho", "A", "U")})
        return {k: res[k] for k in KEYS}


EXACT_NODES = 6.0e7     # particle-steps times nodes a visit that this reference takes on


def exact(case, seed):
    c = dict(DEFAULTS, **case)
    n, _ = _dims(c)
    if c["kind"] == "cn":
        p, f = _Plain(c), _mesh_fields(c, seed)
        s = {"phi": f["phi"], "psi": f["psi"], "A": f["A"].reshape(3, -1), "U": f["U"].reshape(3, -1)}
        a = 0.25 * p.dt ** 2
        u0, w0 = torch.cat([s["phi"][None], s["A"]]), torch.cat([s["psi"][None], s["U"]])
        src = torch.cat([f["rho"][None], f["J"].reshape(3, -1)])
        u1 = p.real(((1 + a * p.lam) * p.hat(u0) + p.hat(p.dt * w0 + 2 * a * src)) / (1 - a * p.lam))
        w1 = 2.0 * (u1 - u0) / p.dt - w0
        return {"phi": u1[0], "psi": w1[0], "A": u1[1:].reshape(-1), "U": w1[1:].reshape(-1)}
    if c["kind"] == "ensemble":
        return None
    if 2 * c["per_beam"] * n[0] * n[1] * n[2] * c["steps"] * (c["order"] + 1) ** 3 > EXACT_NODES:
        return None
    x, v, _, _ = _particles(c, seed)
    p = _Plain(c)
    if c["kind"] == "vjp":
        lam = _cotangent(c, x.shape[0], p.N, p.m, seed)
        return p.vjp(p.start(x, v), lam)
    with torch.no_grad():
        s = p.start(x, v)
        if c["kind"] == "iterate":
            g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
            v1 = v + 1e-3 * c["v0"] * torch.randn(v.shape, generator=g, dtype=F64, device="cuda")
            J = p.current(s, v1)
            out = p.flat(p.push(s, p.fields(s, J), v1))
            out["J"] = J.reshape(-1)
            return {k: out[k] for k in ("J", "rho", "phi", "psi", "A", "U", "x", "P", "v")}
        for _ in range(c["steps"]):
            s = p.step(s)
        out = p.flat(s)
        if c["diag"]:
            out["K1"] = out["W1"] = None
        return out
