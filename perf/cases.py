"""The work a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values.  ``prepare`` makes what a program has in
hand before the call (a simulation, particles in pinned host memory or on the
device), ``run`` is one pass through the public entry points, ``exact`` is the
same pass in plain float64 PyTorch.  Five kinds of pass:

  deposit   the allocation-free density deposit of device positions
  job       a simulation's chunk of steps from host particles: load, step,
            read back (what a served request or a driver script does)
  adaptive  the same with adaptive steps, for a static solitonic core
  snapshot  accelerations, density, energies and power spectrum of particles
  batch     a job of many simulations of mixed sizes stepped together

Results of a job are the momenta and the displacements from the particles'
unperturbed places, on the device, in the precision that the simulation works
in.
"""
import math

import numpy as np
import torch

from paper_1608_00802_gb300 import pm

DEV = "cuda"
HBARC_EV_M, C_M_S, MPC_M = 1.973269804e-7, 299792458.0, 3.0856775814913673e22
OM, OL, H = 0.3, 0.7, 0.7


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: a deposit inside a latency-critical loop
        dict(name="deposit-4k-m32", kind="deposit", n=4096, n_mesh=32, clump=0.0),
        # the same entry point at its largest size, half of the particles in clumps
        dict(name="deposit-64k-m128", kind="deposit", n=65536, n_mesh=128, clump=0.5),
        # a served request of the smallest class: one chunk of 20 steps from z = 50
        dict(name="served-32", kind="job", side=32, n_mesh=64, drop=0, fp64=False, spline=False, force="hybrid",
             quantum=True, steps=20, z=50.0, dlna=0.00646, disp=0.66, box=4.0, m22=5.0),
        # the headline simulation, 128^3 particles on a 256^3 mesh, read back after a few of its 500 steps
        dict(name="single-128", kind="job", side=128, n_mesh=256, drop=0, fp64=False, spline=False, force="hybrid",
             quantum=True, steps=4, z=100.0, dlna=0.00646, disp=0.33, box=2.0, m22=2.5),
        # its pressureless partner run (the pairs that are compared), later on: more particles change cell
        dict(name="pressureless-128", kind="job", side=128, n_mesh=256, drop=0, fp64=False, spline=False,
             force="hybrid", quantum=False, steps=20, z=15.0, dlna=0.00646, disp=2.1, box=2.0, m22=2.5),
        # the paper's spline kernel (the configuration that meets the full-run accuracy bar)
        dict(name="spline-128", kind="job", side=128, n_mesh=256, drop=0, fp64=False, spline=True, force="hybrid",
             quantum=True, steps=20, z=100.0, dlna=0.00646, disp=0.33, box=2.0, m22=2.5),
        # the largest served class: 192^3 particles on a 384^3 mesh (not a power of two)
        dict(name="served-192", kind="job", side=192, n_mesh=384, drop=0, fp64=False, spline=False, force="hybrid",
             quantum=True, steps=4, z=100.0, dlna=0.0107, disp=0.33, box=4.0, m22=2.5),
        # the large single simulation: 256^3 particles on a 512^3 mesh
        dict(name="large-256", kind="job", side=256, n_mesh=512, drop=0, fp64=False, spline=False, force="hybrid",
             quantum=True, steps=6, z=100.0, dlna=0.00323, disp=0.2, box=10.0, m22=1.0),
        # the plain fp64 configuration, 32^3 particles on a 64^3 mesh
        dict(name="plain-fp64-32", kind="job", side=32, n_mesh=64, drop=0, fp64=True, spline=False, force="hybrid",
             quantum=True, steps=20, z=100.0, dlna=0.0161, disp=0.33, box=1.0, m22=2.5),
        # the static soliton of the paper's first test: 10^6 particles in a core on a 128^3 mesh, spline h = 4 in real
        # space, adaptive steps
        dict(name="soliton-1m", kind="adaptive", n=1_000_000, n_mesh=128, r95=18.6, smooth_h=4.0, cfl=0.25, steps=6),
        # a pressureless snapshot of a ragged size, analysed: forces, density, energies, power spectrum
        dict(name="snapshot-75", kind="snapshot", side=75, n_mesh=150, drop=7, quantum=False, force="meshgrad",
             spline=False, z=20.0, disp=1.6, box=2.5, m22=2.5),
        # many simulations of mixed sizes stepped together
        dict(name="batch-24", kind="batch", members=24, top=128, steps=4, z=100.0, dlna=0.00646, disp=0.33),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, side):
    """Twice the particles a side as in every configuration, now and then another even mesh."""
    n = 2 * side if rng.random() < 0.75 else 2 * int(round(side * rng.uniform(0.6, 1.2)))
    return max(16, min(512, n))


def draw(rng):
    kind = rng.choice(["deposit", "job", "job", "job", "job", "snapshot", "adaptive", "batch"])
    if kind == "deposit":
        return dict(kind=kind, n=_log_int(rng, 1, 65536), n_mesh=2 * _log_int(rng, 4, 64),
                    clump=rng.choice([0.0, 0.5, 1.0]))
    if kind == "adaptive":
        n_mesh = 2 * _log_int(rng, 32, 80)
        return dict(kind=kind, n=_log_int(rng, 50_000, 1_500_000), n_mesh=n_mesh,
                    r95=round(n_mesh * rng.uniform(0.12, 0.16), 3), smooth_h=rng.choice([3.5, 4.0]), cfl=0.25,
                    steps=rng.randint(2, 6))
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(3, 24), top=rng.choice([32, 64, 128]), steps=rng.randint(2, 4),
                    z=100.0, dlna=rng.choice([0.00323, 0.00646]), disp=0.33)
    # sizes of the configurations (powers of two a side, and 192) as often as any other
    side = rng.choice([32, 64, 128, 192]) if rng.random() < 0.5 else _log_int(rng, 16, 200)
    c = dict(kind=kind, side=side, n_mesh=_mesh(rng, side), drop=min(rng.choice([0, 0, rng.randint(1, 999)]), side ** 3 // 2),
             box=round(rng.uniform(2.0, 4.0), 3), m22=round(math.exp(rng.uniform(math.log(2.0), math.log(6.0))), 3))
    # with cloud-in-cell the quantum force acts on the particles' shot noise and a run soon turns chaotic: few steps,
    # from the start of a run; pressureless and spline runs are followed for longer
    what = rng.choice(["quantum", "quantum", "pressureless", "spline"])
    z = 100.0 if what == "quantum" else math.exp(rng.uniform(math.log(15.0), math.log(100.0)))
    c.update(z=round(z, 3), disp=round(0.33 * 101.0 / (1.0 + z), 4), quantum=what != "pressureless",
             spline=what == "spline", force="hybrid" if what != "pressureless" else rng.choice(["hybrid", "meshgrad"]))
    if kind == "snapshot":
        return c
    c["fp64"] = side <= 64 and rng.random() < 0.4
    if what != "pressureless" and rng.random() < 0.2:
        c["force"] = "lagrangian"
    c["dlna"] = rng.choice([0.00323, 0.00646])
    c["steps"] = rng.randint(2, 4) if what == "quantum" or c["force"] == "lagrangian" else rng.randint(2, 20 if side <= 128 else 6)
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))


def _hubble(a):
    return math.sqrt(OM / a ** 3 + OL)


def _transfer(k, m22):
    """Bardeen-Bond-Kaiser-Szalay fit times the axion cut-off."""
    q = k / (OM * H)
    t = torch.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
    x = 1.61 * m22 ** (1.0 / 18.0) * k * H / (9.0 * math.sqrt(m22))
    return t * torch.cos(x ** 3) / (1.0 + x ** 8)


def _zeldovich(side, n_mesh, box, a, disp, m22, drop, gen):
    """Positions, momenta and unperturbed places (n, 3) on the device: Zel'dovich displacements of rms `disp` mesh
    cells a direction on a lattice of side^3 particles, growing-mode momenta, the last `drop` particles left out."""
    kw = dict(device=DEV, dtype=torch.float64)
    wk = torch.fft.rfftn(torch.randn(side, side, side, generator=gen, **kw))
    k1 = 2 * math.pi / box * torch.fft.fftfreq(side, 1.0 / side, **kw)
    kx = 2 * math.pi / box * torch.fft.rfftfreq(side, 1.0 / side, **kw)
    ks = (kx[None, None, :], k1[None, :, None], k1[:, None, None])
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    wk *= k2 ** 0.24 * _transfer(k2.sqrt(), m22) / k2
    wk[0, 0, 0] = 0.0
    h = side // 2
    if side % 2 == 0:
        wk[h] = 0.0
        wk[:, h] = 0.0
        wk[:, :, h] = 0.0
    psi = torch.stack([torch.fft.irfftn(1j * k * wk, s=(side,) * 3).reshape(-1) for k in ks], dim=1)
    psi *= disp * box / n_mesh / psi.square().mean().sqrt()
    g = (torch.arange(side, **kw) + 0.5) * (box / side)
    z, y, x = torch.meshgrid(g, g, g, indexing="ij")
    q = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], dim=1)
    n = side ** 3 - drop
    q, psi = q[:n].contiguous(), psi[:n]
    # p = a^2 H f psi with f = 1 (matter domination)
    return torch.remainder(q + psi, box), psi * (a * a * _hubble(a)), q


def _hbm(m22):
    return HBARC_EV_M * C_M_S / (m22 * 1e-22) / (MPC_M * 1e3) / (100.0 / H)


def _soliton(case, gen):
    """Particles at rest drawn from a solitonic core's profile (1 + 0.091 (r/r_c)^2)^-8, and the coupling (omega_m)
    under which a ground state of the box's mass has that radius."""
    kw = dict(device=DEV, dtype=torch.float64)
    n, r95 = case["n"], case["r95"] / case["n_mesh"]
    u = torch.linspace(0.0, 8.0, 8193, **kw)
    cum = torch.cumsum(u * u * (1 + 0.091 * u * u) ** -8, 0)
    cum = cum / cum[-1]
    u95 = float(u[torch.searchsorted(cum, 0.95)])
    r = u[torch.searchsorted(cum, torch.rand(n, generator=gen, **kw)).clamp(max=8192)]
    r = (r + (torch.rand(n, generator=gen, **kw) - 0.5) * (8.0 / 8192)).abs() * (r95 / u95)
    d = torch.randn(n, 3, generator=gen, **kw)
    x = torch.remainder(0.5 + d * (r / d.norm(dim=1))[:, None], 1.0)
    hbm = _hbm(2.5)
    alpha = r95 / 3.80  # radii: 3.80 in the ground state's own units; its mass there: 25.9
    return x, torch.zeros_like(x), torch.full_like(x, 0.5), hbm * hbm * 25.9 / alpha / 1.5, alpha * alpha / hbm


def _members(case):
    """(side, box, m22) of a batch: sizes in turn, boxes and masses spread over their ranges."""
    sizes = [s for s in (32, 64, 128) if s <= case["top"]]
    return [(sizes[i % len(sizes)], 2.0 + 2.0 * ((i * 0.618034) % 1.0), (2.5, 3.5, 5.0)[(i // 3) % 3])
            for i in range(case["members"])]


def _inputs(case, seed):
    """[(x, p, origin, parameters)] for each simulation of the case, on the device."""
    kind = case["kind"]
    if kind == "deposit":
        gen = _gen(seed, 1)
        x = torch.rand(case["n"], 3, generator=gen, device=DEV, dtype=torch.float64)
        m = int(case["clump"] * case["n"])
        if m:  # clumps of a few cells
            c = torch.rand(1 + m // 500, 3, generator=gen, device=DEV, dtype=torch.float64)
            at = torch.randint(0, len(c), (m,), generator=gen, device=DEV)
            x[:m] = torch.remainder(c[at] + 0.02 * torch.randn(m, 3, generator=gen, device=DEV, dtype=torch.float64), 1.0)
        return [(x, None, None, dict(box=1.0, n_mesh=case["n_mesh"]))]
    if kind == "adaptive":
        x, p, q, om, t_unit = _soliton(case, _gen(seed, 2))
        return [(x, p, q, dict(box=1.0, n_mesh=case["n_mesh"], om=om, m22=2.5, force="lagrangian", spline=True,
                               smooth_h=case["smooth_h"], quantum=True, cosmo=False, t_unit=t_unit))]
    a = 1.0 / (1.0 + case["z"])
    if kind == "batch":
        out = []
        for i, (side, box, m22) in enumerate(_members(case)):
            x, p, q = _zeldovich(side, 2 * side, box, a, case["disp"], m22, 0, _gen(seed, 10 + i))
            out.append((x, p, q, dict(box=box, n_mesh=2 * side, om=OM, m22=m22, force="hybrid", spline=False,
                                      smooth_h=3.5, quantum=True, cosmo=True)))
        return out
    x, p, q = _zeldovich(case["side"], case["n_mesh"], case["box"], a, case["disp"], case["m22"], case["drop"],
                         _gen(seed, 3))
    return [(x, p, q, dict(box=case["box"], n_mesh=case["n_mesh"], om=OM, m22=case["m22"], force=case["force"],
                           spline=case["spline"], smooth_h=3.5, quantum=case["quantum"], cosmo=True))]


FORCES = {"meshgrad": pm.FORCE_MESHGRAD, "hybrid": pm.FORCE_HYBRID, "lagrangian": pm.FORCE_LAGRANGIAN}


def _config(n, par, fp64=False):
    return pm.make_config(n, par["n_mesh"], par["box"], precision=pm.FP64 if fp64 else pm.FP32, omega_m=par["om"],
                          omega_l=OL if par["cosmo"] else 0.0, h=H, m22=par["m22"], quantum=par["quantum"],
                          force_mode=FORCES[par["force"]], cosmological=par["cosmo"],
                          kernel=pm.KERNEL_SPLINE if par["spline"] else pm.KERNEL_CIC, smooth_h=par["smooth_h"],
                          smooth_real=not par["cosmo"])  # a core in an empty box: the smoothing that keeps its tails


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


class _Particles:
    """A simulation's particles in pinned host memory, room for its results, and the unperturbed places."""

    def __init__(self, x, p, q, box, dtype):
        self.x, self.p = _pinned(x).numpy(), _pinned(p).numpy()
        self.xo, self.po = torch.empty(x.shape, dtype=x.dtype, pin_memory=True), torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
        self.q, self.box, self.dtype = q, box, dtype

    def results(self, sim):
        """Displacements and momenta on the device."""
        sim.get_particles(self.xo.numpy(), self.po.numpy())
        d = self.xo.to(DEV, non_blocking=True).sub_(self.q)
        d.sub_(self.box * torch.round(d / self.box))
        return [d.to(self.dtype), self.po.to(DEV, non_blocking=True).to(self.dtype)]


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    kind = case["kind"]
    ins = _inputs(case, seed)
    if kind == "deposit":
        x, _, _, par = ins[0]
        n = par["n_mesh"]
        return dict(case=case, x=x, rho=torch.empty(n, n, n, device=DEV, dtype=torch.float32))
    dtype = torch.float64 if case.get("fp64") else torch.float32
    st = dict(case=case, parts=[_Particles(x, p, q, par["box"], dtype) for x, p, q, par in ins])
    cfgs = [_config(x.shape[0], par, case.get("fp64", False)) for x, _, _, par in ins]
    if kind == "batch":
        st["batch"] = pm.Batch(cfgs)
    else:
        st["sim"] = pm.Sim(cfgs[0])
    if kind == "adaptive":
        st["t_end"] = ins[0][3]["t_unit"]
    return st


def _span(case):
    a0 = 1.0 / (1.0 + case["z"])
    return a0, a0 * math.exp(case["dlna"] * case["steps"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "deposit":
        pm.deposit_noalloc(state["x"], case["n_mesh"], 1.0, state["rho"])
        return state["rho"]
    parts = state["parts"]
    if kind == "batch":
        batch = state["batch"]
        for sim, pt in zip(batch.members, parts):
            sim.set_particles(pt.x, pt.p)
        batch.run(case["steps"], *_span(case))
        return [pt.results(sim) for sim, pt in zip(batch.members, parts)]
    sim, pt = state["sim"], parts[0]
    sim.set_particles(pt.x, pt.p)
    if kind == "job":
        sim.run(case["steps"], *_span(case))
        return pt.results(sim)
    if kind == "adaptive":
        bounds = sim.run_adaptive(0.0, state["t_end"], cfl=case["cfl"], max_steps=case["steps"])
        return pt.results(sim) + [bounds.astype(np.float32)]
    a = 1.0 / (1.0 + case["z"])
    acc, rho = sim.forces(a), sim.get_field(pm.FIELD_RHO)
    k, pk, modes = sim.power_spectrum()
    out = [torch.from_numpy(acc).to(DEV).float(), torch.from_numpy(rho).to(DEV).float(),
           sim.energy(a).astype(np.float32), k, pk.astype(np.float32), modes]
    return out


def work(case):
    """Bytes: the host's particles in and out (their copies), the records, mesh fields and spectra of a step once in and
    out; operations: transforms, stencils and interpolations."""
    if case["kind"] == "deposit":
        n, N = case["n"], case["n_mesh"]
        return dict(bytes=24 * n + 4 * N ** 3, flops=32 * n)
    r = 8 if case.get("fp64") else 4
    if case["kind"] == "batch":
        sims = [(s ** 3, 2 * s) for s, _, _ in _members(case)]
    elif case["kind"] == "adaptive":
        sims = [(case["n"], case["n_mesh"])]
    else:
        sims = [(case["side"] ** 3 - case["drop"], case["n_mesh"])]
    steps = case.get("steps", 0)
    spline = case.get("spline", case["kind"] == "adaptive")
    quantum = case.get("quantum", True)
    b = f = 0
    for n, N in sims:
        m = N ** 3
        # a force evaluation: positions in, density and potentials out; a spectrum once each way (three more
        # transforms with the spline); a pass over the particles: records in and out, the potentials in
        fields = 4 * r * n + r * m * (2 + quantum) + 2 * r * m + (3 * r * m if spline else 0)
        kick = 16 * r * n + r * m * (1 + quantum)
        fft = 2.5 * m * math.log2(m)
        io = 96 * n if case["kind"] != "snapshot" else 48 * n + 24 * n + 8 * m
        b += io + fields * (steps + 1) + kick * max(1, steps)
        f += (fft * (5 if spline else 2) + 30 * m * quantum + 250 * n) * (steps + 1)
    return dict(bytes=int(b), flops=int(f))


# ---------------------------------------------------------------- the same passes in float64 PyTorch
class _Exact:
    """The particle-mesh step with quantum pressure (arXiv:1608.00802, Sec. II.A), in float64."""

    def __init__(self, par):
        self.__dict__.update(par)
        self.N, self.dx, self.h2 = par["n_mesh"], par["box"] / par["n_mesh"], None
        kw = dict(device=DEV, dtype=torch.float64)
        if "om" not in par:
            return
        s = torch.sin(math.pi * torch.fft.fftfreq(self.N, **kw)) ** 2
        sx = torch.sin(math.pi * torch.fft.rfftfreq(self.N, **kw)) ** 2
        k2 = 4.0 / self.dx ** 2 * (s[:, None, None] + s[None, :, None] + sx[None, None, :])
        k2[0, 0, 0] = math.inf
        self.green = -1.5 * self.om / k2
        if self.spline:
            d = torch.fft.fftfreq(self.N, 1.0 / self.N, **kw)
            u = (d[:, None, None] ** 2 + d[None, :, None] ** 2 + d[None, None, :] ** 2).sqrt() / self.smooth_h
            w = torch.where(u <= 0.5, 1 - 6 * u ** 2 + 6 * u ** 3, 2 * (1 - u).clamp(min=0) ** 3)
            self.symbol = torch.fft.rfftn(w / w.sum()).real
        self.hbm = _hbm(self.m22)

    def corners(self, x):
        u = x / self.dx
        c = u.floor()
        return torch.remainder(c.long(), self.N), u - c

    def deposit(self, x):
        c, f = self.corners(x)
        rho = torch.zeros(self.N ** 3, device=DEV, dtype=torch.float64)
        for o in range(8):
            idx, w = self._corner(c, f, o)
            rho.index_add_(0, idx, w)
        return (rho * (self.N ** 3 / x.shape[0])).view(self.N, self.N, self.N)

    def _corner(self, c, f, o, grad=None):
        idx, w = 0, 1.0
        for ax in (2, 1, 0):
            b = (o >> ax) & 1
            idx = idx * self.N + (c[:, ax] + b) % self.N
            w = w * ((1.0 if b else -1.0) if grad == ax else (f[:, ax] if b else 1 - f[:, ax]))
        return idx, w

    def smooth(self, v):
        return torch.fft.irfftn(torch.fft.rfftn(v) * self.symbol, s=v.shape)

    def fields(self, x):
        rho = self.deposit(x)
        if self.spline:
            rho = self.smooth(rho)
        phi = torch.fft.irfftn(torch.fft.rfftn(rho) * self.green, s=rho.shape)
        q = None
        if self.quantum:
            s = rho.clamp(min=1e-6).sqrt()
            lap = sum(torch.roll(s, 1, a) + torch.roll(s, -1, a) - 2 * s for a in range(3)) / self.dx ** 2
            q = -0.5 * self.hbm ** 2 * lap / s
        self.rho, self.phi0 = rho, phi
        if self.spline:
            phi = self.smooth(phi)
            q = self.smooth(q) if self.quantum else None
        return phi, q

    def grad(self, v, x, kernel):
        c, f = self.corners(x)
        out = torch.zeros_like(x)
        for ax in range(3):
            g = v.reshape(-1) if kernel else ((torch.roll(v, -1, 2 - ax) - torch.roll(v, 1, 2 - ax)) / (2 * self.dx)).reshape(-1)
            for o in range(8):
                idx, w = self._corner(c, f, o, ax if kernel else None)
                out[:, ax] += g[idx] * w
        return out / self.dx if kernel else out

    def forces(self, x):
        phi, q = self.fields(x)
        gp = self.grad(phi, x, self.force == "lagrangian")
        return gp, (self.grad(q, x, self.force != "meshgrad") if self.quantum else torch.zeros_like(gp))

    def weights(self, a0, a1):
        """Kick weight of gravity; kick weight of Q and drift weight."""
        if not self.cosmo:
            return a1 - a0, a1 - a0
        t, w = np.polynomial.legendre.leggauss(32)
        a = 0.5 * (a0 + a1) + 0.5 * (a1 - a0) * t
        i = 0.5 * (a1 - a0) * w / np.sqrt(OM / a ** 3 + OL)
        return float((i / a ** 2).sum()), float((i / a ** 3).sum())

    def half(self, a0, a1):
        return math.sqrt(a0 * a1) if self.cosmo else 0.5 * (a0 + a1)

    def step(self, x, p, g, a0, a1):
        ah = self.half(a0, a1)
        k = self.weights(a0, ah)
        p = p - k[0] * g[0] - k[1] * g[1]
        x = torch.remainder(x + self.weights(a0, a1)[1] * p, self.box)
        g = self.forces(x)
        k = self.weights(ah, a1)
        return x, p - k[0] * g[0] - k[1] * g[1], g

    def adaptive(self, x, p, g, t, t_end, cfl):
        """The largest t1 whose bound of every drift stays within cfl cells, by bisection."""
        top = [float(v.square().sum(1).max().sqrt()) for v in (p, *g)]

        def fits(t1):
            k = self.weights(t, self.half(t, t1))
            return (top[0] + k[0] * top[1] + k[1] * top[2]) * self.weights(t, t1)[1] <= cfl * self.dx
        if fits(t_end):
            return t_end
        lo, hi = 0.0, 1.0
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if fits(t + (t_end - t) * mid) else (lo, mid)
        return t + (t_end - t) * lo

    def moved(self, x, q):
        d = x - q
        return d - self.box * torch.round(d / self.box)

    def energies(self, p, a):
        n = p.shape[0]
        m = self.box ** 3 / n
        kr = 0.0
        if self.quantum:
            s = self.rho.clamp(min=1e-6).sqrt()
            kr = 0.5 * self.hbm ** 2 / a ** 2 * self.dx * sum(float((torch.roll(s, -1, d) - s).square().sum()) for d in range(3))
        wg = 0.5 / a * float(((self.rho - 1) * self.phi0).sum()) * self.dx ** 3
        return np.array([0.5 * m * float(p.square().sum()) / a ** 2, wg, kr] + [m * float(v) for v in p.sum(0)])

    def power(self, x):
        N = self.N
        dk = torch.fft.rfftn(self.deposit(x)).abs() ** 2
        m1 = torch.fft.fftfreq(N, 1.0 / N, device=DEV, dtype=torch.float64)
        mx = torch.fft.rfftfreq(N, 1.0 / N, device=DEV, dtype=torch.float64)
        win = (torch.sinc(mx / N)[None, None, :] * torch.sinc(m1 / N)[None, :, None] * torch.sinc(m1 / N)[:, None, None]) ** 4
        m = (mx[None, None, :] ** 2 + m1[None, :, None] ** 2 + m1[:, None, None] ** 2).sqrt()
        shell = (m + 0.5).floor().long()
        two = torch.full_like(mx, 2.0)
        two[0] = two[-1] = 1.0
        two = two.expand_as(m)
        on = (shell >= 1) & (shell <= N // 2)
        cnt, ks, ps = (torch.bincount(shell[on], weights=v[on], minlength=N // 2 + 1)[1:]
                       for v in (two, two * m, two * dk / win))
        kf = 2 * math.pi / self.box
        return [(kf * ks / cnt).cpu().numpy(), (self.box ** 3 / float(N) ** 6 * ps / cnt).cpu().numpy(),
                np.rint(cnt.cpu().numpy()).astype(np.int64)]


def exact(case, seed):
    kind, outs = case["kind"], []
    for x, p, q, par in _inputs(case, seed):
        e = _Exact(par)
        if kind == "deposit":
            return e.deposit(x)
        g = e.forces(x)
        if kind == "snapshot":
            a = 1.0 / (1.0 + case["z"])
            acc, rho = -(g[0] / a + g[1] / a ** 2), e.rho
            return [acc, rho, e.energies(p, a)] + e.power(x)
        if kind == "adaptive":
            t, t_end, bounds = 0.0, par["t_unit"], [0.0]
            while t < t_end and len(bounds) <= case["steps"]:
                t1 = e.adaptive(x, p, g, t, t_end, case["cfl"])
                x, p, g = e.step(x, p, g, t, t1)
                t = t1
                bounds.append(t)
            return [e.moved(x, q), p, np.array(bounds)]
        a0, a1 = _span(case)
        for i in range(case["steps"]):
            at = [a0 * (a1 / a0) ** (k / case["steps"]) for k in (i, i + 1)]
            x, p, g = e.step(x, p, g, *at)
        outs.append([e.moved(x, q), p])
        del e
    return outs if kind == "batch" else outs[0]
