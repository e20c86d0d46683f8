"""Workloads of the binary-fluid lattice Boltzmann library, as programs call it.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from
a seed, ``run`` takes them once through the public entry points (``Lattice``,
``Batch``, ``adjoint.trajectory``), ``work`` counts the bytes and operations
the method cannot do without and ``exact`` evaluates the same model in plain
FP64 torch.  Four kinds of work:

* ``step``: a simulation between two outputs -- start from an order parameter
  (or from saved distributions), a number of timesteps (in one call, or in
  several with the lattice totals read between them), then the fields (or the
  distributions).  A program on FP32 storage keeps its fields in float32.
* ``ensemble``: many small lattices of uneven sizes, one run of all of them.
* ``adjoint``: gradient of a droplet-matching loss through the trajectory.
* ``diagnostics``: totals of a large lattice and its fields on a masked part.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1405_6162_gb300 import Lattice
from paper_1405_6162_gb300.adjoint import trajectory
from paper_1405_6162_gb300.batch import Batch

# relaxation and free-energy parameters every workload of the repository shares
BASE = dict(tau=1.0, tau_g=1.0, rho0=1.0, gamma=0.5, A=-0.0625, B=0.0625, kappa=0.04)
STEP = dict(kind="step", precision="fp32_shifted", kernel="auto", stencil=7, mrt=False, force=0.0, tau=1.0, tau_g=1.0,
            amp=0.01, flow=0.0, start="phi", steps=50, every=0)


def _step(name, nx, ny, nz, **kw):
    return dict(STEP, name=name, nx=nx, ny=ny, nz=nz, **kw)


def listed():
    return [
        # the smallest parity workload: short calls, bound by launches
        _step("spinodal_32_fp32", 32, 32, 32, steps=10),
        # the error-table lattice in FP64 with a shear wave on it, a block of its steps
        _step("spinodal_64_fp64", 64, 64, 64, precision="fp64", flow=0.01, steps=50),
        # the long spinodal run, with the conservation totals watched on the way
        _step("spinodal_128_fp32", 128, 128, 128, steps=100, every=20),
        # the headline lattice: 50 steps between outputs
        _step("spinodal_256_fp32", 256, 256, 256, steps=50),
        # the reduced form a program chooses when tau_g = 1, with a flow
        _step("reduced_256_fp32", 256, 256, 256, kernel="taug1", tau=0.8, amp=0.3, flow=0.01, steps=50),
        # separate relaxation times on a box that is not a power of two
        _step("two_rates_200x152x136_fp32", 200, 152, 136, tau=0.8, tau_g=0.9, amp=0.3, flow=0.01, steps=30),
        # the widest collision and stencil on odd extents
        _step("mrt_force_129x97x65_fp32", 129, 97, 65, stencil=27, mrt=True, force=1e-5, tau=0.7, amp=0.3, flow=0.01,
              steps=20),
        # FP64-class accuracy on the FP32 units
        _step("double_float_144x120x100", 144, 120, 100, precision="fp64_df", tau=0.8, amp=0.3, flow=0.01, steps=20),
        # restart from saved distributions, single steps, save again; ragged
        _step("restart_70x37x11_fp64", 70, 37, 11, precision="fp64", tau=0.7, tau_g=0.9, amp=0.3, flow=0.01,
              start="state", steps=5, every=1),
        # 64 lattices of sides 16..64 with their own tau and kappa
        dict(name="ensemble_64_fp32", kind="ensemble", n=64, lo=16, hi=64, precision="fp32_shifted", form="general",
             flow=0.0, steps=100),
        # gradients through a droplet-matching trajectory
        dict(name="adjoint_64_fp64", kind="adjoint", nx=64, ny=64, nz=64, steps=200, tau=1.0, tau_g=1.0, radius=16.0),
        # totals and interface fields of the headline lattice
        dict(name="diagnostics_256_fp32", kind="diagnostics", nx=256, ny=256, nz=256, precision="fp32_shifted",
             share=0.1),
    ]


def _side(rng, lo=16, hi=256):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("step", "ensemble", "adjoint", "diagnostics"), (12, 3, 2, 2))[0]
    tau = 1.0 if rng.random() < 0.4 else round(rng.uniform(0.55, 1.5), 3)
    tau_g = 1.0 if rng.random() < 0.65 else round(rng.uniform(0.7, 1.3), 3)
    if kind == "ensemble":
        precision = rng.choice(("fp32_shifted", "fp32_shifted", "fp64"))
        lo = rng.randint(8, 24)
        return dict(kind=kind, n=rng.randint(8, 64), lo=lo, hi=rng.randint(lo + 8, 64), precision=precision,
                    form=rng.choice(("general", "general", "taug1")), flow=0.01 if precision == "fp64" else 0.0,
                    steps=rng.randint(10, 100))
    if kind == "adjoint":
        return dict(kind=kind, nx=_side(rng, 12, 64), ny=_side(rng, 12, 64), nz=_side(rng, 12, 64),
                    steps=_side(rng, 8, 160), tau=tau, tau_g=tau_g, radius=rng.uniform(4.0, 16.0))
    nx, ny, nz = _side(rng), _side(rng), _side(rng)
    # rows of powers of two and of whole vectors are as common as odd ones
    nx = rng.choice((nx, nx, (nx + 7) // 8 * 8, 1 << round(math.log2(nx))))
    precision = rng.choice(("fp32_shifted", "fp32_shifted", "fp32_shifted", "fp64", "fp64_df"))
    if kind == "diagnostics":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, share=round(10 ** rng.uniform(-3, 0), 4))
    kernel = "taug1" if tau_g == 1.0 and rng.random() < 0.2 else "auto"
    mrt = kernel == "auto" and rng.random() < 0.25
    force = round(rng.uniform(1e-6, 1e-4), 7) if kernel == "auto" and rng.random() < 0.2 else 0.0
    cost = nx * ny * nz * {"fp32_shifted": 1, "fp64_df": 3, "fp64": 9}[precision]
    steps = min(_side(rng, 1, 100), max(1, 25 * 256 ** 3 // cost))
    return dict(STEP, nx=nx, ny=ny, nz=nz, precision=precision, kernel=kernel, tau=tau, tau_g=tau_g, mrt=mrt,
                force=force, stencil=rng.choice((7, 7, 7, 19, 27)), amp=rng.choice((0.01, 0.3)),
                flow=rng.choice((0.0, 0.01)) if precision == "fp32_shifted" else 0.01, start=rng.choice(("phi", "phi", "state")), steps=steps,
                every=rng.choice((0, 0, max(1, steps // 4))))


# ------------------------------------------------------------------ inputs


def _params(case):
    return dict(BASE, tau=case["tau"], tau_g=case["tau_g"])


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 62))


def _uniform(gen, lo, hi, *shape):
    return torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _fields(case, seed):
    return _start(case["nx"], case["ny"], case["nz"], _generator(seed), case["amp"], case["flow"])


def _start(nx, ny, nz, gen, amp, flow):
    """Order parameter (noise around 0) and velocity (a shear wave of random
    phase, or none) of a start."""
    phi = _uniform(gen, -amp, amp, nx * ny * nz)
    if not flow:
        return phi, None
    phase = float(_uniform(gen, 0.0, 2.0 * math.pi, 1))
    x = torch.arange(nx, device="cuda", dtype=torch.float64)
    u = torch.zeros(3, nz, ny, nx, device="cuda", dtype=torch.float64)
    u[1] = flow * torch.sin(2.0 * math.pi * x / nx + phase)
    u[2] = 0.5 * flow * torch.cos(2.0 * math.pi * x / nx + phase)
    return phi, u.reshape(3, -1)


def _saved(nx, ny, nz, gen, amp):
    """Distributions a few per cent off a local equilibrium, as a saved state
    holds them."""
    n = nx * ny * nz
    _, w = _velocities()
    phi = _uniform(gen, -amp, amp, n)
    rho = 1.0 + _uniform(gen, -0.02, 0.02, n)
    f = torch.empty(19, n, device="cuda", dtype=torch.float64)
    g = torch.empty_like(f)
    for i in range(19):
        f[i] = w[i] * (rho + _uniform(gen, -0.02, 0.02, n))
        g[i] = w[i] * (phi + _uniform(gen, -0.02, 0.02, n))
    return f, g


def _ensemble_specs(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    dims = torch.randint(case["lo"], case["hi"] + 1, (case["n"], 3), generator=torch.Generator().manual_seed(3))
    tau = torch.rand(case["n"], generator=gen, dtype=torch.float64) * 0.95 + 0.55
    kappa = torch.rand(case["n"], generator=gen, dtype=torch.float64) * 0.07 + 0.01
    return [dict(BASE, nx=int(d[0]), ny=int(d[1]), nz=int(d[2]), tau=float(t), kappa=float(k))
            for d, t, k in zip(dims, tau, kappa)]


def _mask(case, seed):
    """An interface-like band: the share of the sites where a smooth random
    field is nearest to zero."""
    gen = _generator(seed + 7)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x, y, z = (torch.arange(n, device="cuda", dtype=torch.float64) * (2.0 * math.pi / n) for n in (nx, ny, nz))
    p = [float(v) for v in _uniform(gen, 0.0, 2.0 * math.pi, 6)]
    v = (torch.sin(x + p[0])[None, None, :] + torch.sin(2 * y + p[1])[None, :, None] + torch.sin(z + p[2])[:, None, None]
         + torch.sin(3 * x + p[3])[None, None, :] * torch.sin(2 * z + p[4])[:, None, None])
    mask = torch.zeros(nx * ny * nz, device="cuda", dtype=torch.uint8)
    mask[v.reshape(-1).abs().argsort()[:max(1, round(case["share"] * nx * ny * nz))]] = 1
    return mask


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        specs = _ensemble_specs(case, seed)
        batch = Batch(specs, precision=case["precision"])
        batch.set_form(case["form"])
        gen = _generator(seed)
        starts = [_start(d["nx"], d["ny"], d["nz"], gen, 0.01, case["flow"]) for d in specs]
        return dict(case=case, batch=batch, starts=starts)
    if kind == "adjoint":
        gen = _generator(seed)
        n = case["nx"] * case["ny"] * case["nz"]
        phi = _uniform(gen, -0.01, 0.01, n).requires_grad_()
        kappa = torch.tensor(0.04, device="cuda", dtype=torch.float64).requires_grad_()
        return dict(case=case, phi=phi, kappa=kappa, target=_droplet(case, gen))
    dims = (case["nx"], case["ny"], case["nz"])
    if kind == "diagnostics":
        lat = Lattice(*dims, **BASE, precision=case["precision"])
        lat.set_state(*_saved(*dims, _generator(seed), 0.3))
        return dict(case=case, lat=lat, mask=_mask(case, seed))
    lat = Lattice(*dims, **_params(case), precision=case["precision"])
    if case["stencil"] != 7:
        lat.set_stencil(case["stencil"])
    if case["mrt"]:
        lat.set_collision("mrt", 1.3, 0.6)
    if case["force"]:
        lat.set_force(case["force"], 0.5 * case["force"], -case["force"])
    if case["kernel"] != "auto":
        lat.set_kernel(case["kernel"])
    if case["start"] == "state":
        return dict(case=case, lat=lat, saved=_saved(*dims, _generator(seed), case["amp"]))
    phi, u = _fields(case, seed)
    return dict(case=case, lat=lat, phi=phi, u=u)


def _droplet(case, gen):
    """phi of a droplet whose centre is off the box's centre."""
    off = [float(v) for v in _uniform(gen, -4.0, 4.0, 3)]
    d2 = 0.0
    for axis, n in enumerate((case["nz"], case["ny"], case["nx"])):
        d = torch.arange(n, device="cuda", dtype=torch.float64) - (n / 2 + off[axis])
        d = d - n * torch.round(d / n)
        d2 = d2 + (d * d).reshape([-1 if a == axis else 1 for a in range(3)])
    xi = math.sqrt(-2.0 * BASE["kappa"] / BASE["A"])
    return torch.tanh((case["radius"] - torch.sqrt(d2)) / xi).reshape(-1)


# ------------------------------------------------------------------ one pass


def _kept(case, *fields):
    """Fields as the program keeps them: float32 from FP32 storage."""
    return [x.float() for x in fields] if case["precision"] == "fp32_shifted" else list(fields)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ensemble":
        batch = state["batch"]
        for k, (phi, u) in enumerate(state["starts"]):
            batch[k].init(phi, u)
        batch.run(case["steps"])
        fields = [batch[k].moments(device=True) for k in range(len(batch))]
        return _kept(case, *(torch.cat([x[j] for x in fields], dim=-1) for j in range(3)))
    if kind == "adjoint":
        phi, kappa = state["phi"], state["kappa"]
        dims = (case["nx"], case["ny"], case["nz"])
        phi_t = trajectory(phi, kappa, dims, _params(case), case["steps"])
        loss = ((phi_t - state["target"]) ** 2).sum()
        d_phi, d_kappa = torch.autograd.grad(loss, (phi, kappa))
        return [phi_t, d_phi, d_kappa]
    lat = state["lat"]
    if kind == "diagnostics":
        totals = lat.reduce()
        return [totals] + _kept(case, *lat.moments_masked(state["mask"]))
    if case["start"] == "state":
        lat.set_state(*state["saved"])
    else:
        lat.init(state["phi"], state["u"])
    totals = []
    done = 0
    while done < case["steps"]:
        n = min(case["every"] or case["steps"], case["steps"] - done)
        lat.step(n)
        done += n
        if case["every"]:
            totals.append(lat.reduce())
    fields = lat.get_state(device=True) if case["start"] == "state" else lat.moments(device=True)
    if totals:
        fields = [*fields, torch.from_numpy(np.stack(totals))]
    return _kept(case, *fields)


# ------------------------------------------------------------------ what a pass cannot do without


def work(case):
    """Bytes: each input read once and each output written once, and per
    timestep the state read and written once -- the 19 values of f, and the 19
    of g or, where tau_g = 1 makes g its equilibrium, phi alone.  Operations:
    about 380 per site and step; a reverse step about 1000."""
    kind = case["kind"]
    size = 4 if case.get("precision") == "fp32_shifted" else 8
    if kind == "ensemble":
        n = sum(d["nx"] * d["ny"] * d["nz"] for d in _ensemble_specs(case, 0))
        ends = 8.0 * (4 if case["flow"] else 1) + 5.0 * size
        return {"bytes": n * (ends + case["steps"] * 40.0 * size), "flops": 380.0 * n * case["steps"]}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "adjoint":
        words = 40.0 if case["tau_g"] == 1.0 else 76.0
        # the state forward, and state and adjoint (read, written) backward
        return {"bytes": n * 8.0 * (4 + case["steps"] * (words + words / 2 + 76.0)), "flops": 1380.0 * n * case["steps"]}
    if kind == "diagnostics":
        return {"bytes": n * (38.0 * size + 1) + case["share"] * n * 5.0 * size, "flops": n * (38.0 + case["share"] * 70.0)}
    words = 40.0 if case["tau_g"] == 1.0 else 76.0
    ends = 38 * (8.0 + size) if case["start"] == "state" else 8.0 * (4 if case["flow"] else 1) + 5.0 * size
    reads = math.ceil(case["steps"] / case["every"]) * words / 2 * size if case["every"] else 0.0
    return {"bytes": n * (ends + case["steps"] * words * size + reads), "flops": n * 380.0 * case["steps"]}


# ------------------------------------------------------------------ the same in plain FP64 torch


def _velocities():
    """Velocities in the library's order and their weights."""
    faces = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    edges = [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
             (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
    c = [(0, 0, 0)] + faces + edges
    return c, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


class _Model:
    """The model on one periodic lattice; fields are [.., nz, ny, nx]."""

    def __init__(self, dims, params, kappa=None, stencil=7, rates=None, force=(0.0, 0.0, 0.0)):
        self.shape = dims[::-1]
        self.p = params
        self.kappa = params["kappa"] if kappa is None else kappa
        self.stencil, self.rates, self.force = stencil, rates, force
        c, w = _velocities()
        self.c = c
        self.C = torch.tensor(c, dtype=torch.float64, device="cuda").T.contiguous()
        self.w = torch.tensor(w, dtype=torch.float64, device="cuda")
        x, y, z = self.C
        one = torch.ones_like(x)
        # w_i [a + 3 c.j + 9/2 c c : S - 3/2 tr S]: rows over the moments (a, j, Sxx, Syy, Szz, Sxy, Sxz, Syz)
        self.E = (self.w * torch.stack([one, 3 * x, 3 * y, 3 * z, 4.5 * x * x - 1.5, 4.5 * y * y - 1.5,
                                        4.5 * z * z - 1.5, 9 * x * y, 9 * x * z, 9 * y * z])).T.contiguous()
        self.M2 = torch.stack([x * x, y * y, z * z, x * y, x * z, y * z])

    def _mul(self, m, v):
        return (m @ v.reshape(v.shape[0], -1)).reshape(m.shape[0], *self.shape)

    def gradients(self, phi):
        if self.stencil == 7:
            d = [0.5 * (phi.roll(-1, a) - phi.roll(1, a)) for a in (2, 1, 0)]
            lap = sum(phi.roll(-1, a) + phi.roll(1, a) for a in range(3)) - 6 * phi
            return d, lap
        weight = {1: 1 / 18, 2: 1 / 36} if self.stencil == 19 else {1: 2 / 27, 2: 1 / 54, 3: 1 / 216}
        d = [torch.zeros_like(phi) for _ in range(3)]
        lap = torch.zeros_like(phi)
        for cx in (-1, 0, 1):
            for cy in (-1, 0, 1):
                for cz in (-1, 0, 1):
                    w = weight.get(cx * cx + cy * cy + cz * cz)
                    if w is None:
                        continue
                    v = phi.roll((-cz, -cy, -cx), (0, 1, 2))
                    for a, ca in enumerate((cx, cy, cz)):
                        if ca:
                            d[a] = d[a] + 3 * w * ca * v
                    lap = lap + 6 * w * (v - phi)
        return d, lap

    def moments_of(self, rho, j, phi):
        """(u, moments of f_eq's rows, moments of g_eq's rows)"""
        d, lap = self.gradients(phi)
        p, k = self.p, self.kappa
        u = j / rho
        mu = p["A"] * phi + p["B"] * phi ** 3 - k * lap
        pb = p["A"] / 2 * phi ** 2 + 0.75 * p["B"] * phi ** 4 - k * phi * lap - k / 2 * (d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        S = [k * d[a] * d[b] + j[a] * u[b] + (pb if a == b else 0.0) for a, b in pairs]
        gm = p["gamma"] * mu - phi / 3
        G = [phi * u[a] * u[b] + (gm if a == b else 0.0) for a, b in pairs]
        return u, torch.stack([rho, j[0], j[1], j[2], *S]), torch.stack([phi, *(phi * u), *G])

    def start(self, phi, u0=None):
        phi = phi.reshape(self.shape)
        rho = torch.full_like(phi, self.p["rho0"])
        j = torch.zeros(3, *self.shape, dtype=phi.dtype, device=phi.device) if u0 is None else \
            self.p["rho0"] * u0.reshape(3, *self.shape)
        _, mf, mg = self.moments_of(rho, j, phi)
        return self._mul(self.E, mf), self._mul(self.E, mg)

    def fields(self, f, g):
        rho = f.sum(0)
        j = self._mul(self.C, f) + torch.tensor(self.force, dtype=f.dtype, device=f.device).reshape(3, 1, 1, 1) / 2
        return rho, j, g.sum(0)

    def step(self, f, g):
        rho, j, phi = self.fields(f, g)
        u, mf, mg = self.moments_of(rho, j, phi)
        geq = self._mul(self.E, mg)
        if self.rates is None:
            fs = f + (self._mul(self.E, mf) - f) / self.p["tau"]
        else:
            fs = self._relax_mrt(f, rho, u, mf)
        gs = g + (geq - g) / self.p["tau_g"]
        out = [torch.stack([a[i].roll((c[2], c[1], c[0]), (0, 1, 2)) for i, c in enumerate(self.c)]) for a in (fs, gs)]
        return out[0], out[1]

    def _relax_mrt(self, f, rho, u, mf):
        ws, wb, wg = 1 / self.p["tau"], 1 / self.rates[0], 1 / self.rates[1]
        F = self.force
        pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        third = torch.tensor([1, 1, 1, 0, 0, 0], dtype=f.dtype, device=f.device).reshape(6, 1, 1, 1) / 3
        N = self._mul(self.M2, f) - rho * third - mf[4:]
        G = torch.stack([u[a] * F[b] + u[b] * F[a] for a, b in pairs])
        Nb, Gb = N[:3].sum(0) * third, G[:3].sum(0) * third
        X = (1 - ws) * (N - Nb) + (1 - wb) * Nb + (1 - ws / 2) * (G - Gb) + (1 - wb / 2) * Gb
        m = torch.empty_like(mf)
        m[0] = wg * mf[0]
        for a in range(3):
            m[1 + a] = wg * mf[1 + a] + (1 - wg / 2) * F[a]
        m[4:] = wg * mf[4:] + X - (1 - wg) * N
        return (1 - wg) * f + self._mul(self.E, m)

    def advance(self, f, g, steps):
        for _ in range(steps):
            f, g = self.step(f, g)
        return f, g

    def totals(self, f, g):
        return torch.cat([f.sum().reshape(1), self.C @ f.reshape(19, -1).sum(1), g.sum().reshape(1)])

    def outputs(self, f, g):
        rho, j, phi = self.fields(f, g)
        return [rho.reshape(-1), (j / rho).reshape(3, -1), phi.reshape(-1)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        specs = _ensemble_specs(case, seed)
        gen = _generator(seed)
        got = []
        for d in specs:
            m = _Model((d["nx"], d["ny"], d["nz"]), d)
            start = m.start(*_start(d["nx"], d["ny"], d["nz"], gen, 0.01, case["flow"]))
            got.append(m.outputs(*m.advance(*start, case["steps"])))
        return [torch.cat([x[j] for x in got], dim=-1) for j in range(3)]
    dims = (case["nx"], case["ny"], case["nz"])
    if kind == "adjoint":
        s = prepare(case, seed)
        phi, kappa, part = s["phi"], s["kappa"], 10
        m = _Model(dims, _params(case), kappa=kappa)
        f, g = m.start(phi)
        for t in range(0, case["steps"], part):
            n = min(part, case["steps"] - t)
            f, g = checkpoint(lambda a, b, n=n: m.advance(a, b, n), f, g, use_reentrant=False)
        phi_t = g.sum(0).reshape(-1)
        d_phi, d_kappa = torch.autograd.grad(((phi_t - s["target"]) ** 2).sum(), (phi, kappa))
        return [phi_t.detach(), d_phi, d_kappa]
    if kind == "diagnostics":
        m = _Model(dims, BASE)
        f, g = _saved(*dims, _generator(seed), 0.3)
        at = _mask(case, seed) != 0
        total = m.totals(f, g)
        f, g = f[:, at], g[:, at]
        rho = f.sum(0)
        return [total, rho, (m.C @ f) / rho, g.sum(0)]
    force = (case["force"], 0.5 * case["force"], -case["force"])
    # a force without the multiple rates is the same collision at equal rates
    rates = (1.3, 0.6) if case["mrt"] else (case["tau"], case["tau"]) if case["force"] else None
    m = _Model(dims, _params(case), stencil=case["stencil"], rates=rates, force=force)
    if case["start"] == "state":
        f, g = (x.reshape(19, *m.shape) for x in _saved(*dims, _generator(seed), case["amp"]))
    else:
        f, g = m.start(*_fields(case, seed))
    totals, done = [], 0
    while done < case["steps"]:
        n = min(case["every"] or case["steps"], case["steps"] - done)
        f, g = m.advance(f, g, n)
        done += n
        if case["every"]:
            totals.append(m.totals(f, g))
    if case["start"] == "state":
        out = [f.reshape(19, -1), g.reshape(19, -1)]
    else:
        out = m.outputs(f, g)
    return out + ([torch.stack(totals)] if totals else [])
