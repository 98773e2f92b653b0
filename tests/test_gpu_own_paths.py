"""Paths of the own transforms and of the load that the other tests reach only through whole runs: the
spline kernel's passes on 256^3 meshes (with the spectral and the real-space smoothing), the energy and the packed
classes of 512^3 meshes, loads whose momenta travel on their own stream, and the edges between the forms of the
one-kernel sort."""
import math

import numpy as np
import pytest

from oracle import pm_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm as _pm
    return _pm


def _symbol(torch, n, h):
    """DFT of the normalised node weights W(|x_n|, h), r in cells."""
    d = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    u = torch.sqrt(d[:, None, None] ** 2 + d[None, :, None] ** 2 + d[None, None, :] ** 2) / h
    w = torch.where(u <= 0.5, 1 - 6 * u ** 2 + 6 * u ** 3, torch.where(u <= 1, 2 * (1 - u) ** 3, torch.zeros_like(u)))
    return torch.fft.rfftn(w / w.sum()).real


# h = 1: the symbol is 1 at every mode; 1.5: between 0.38 and 1; 3.5: the default
@pytest.mark.parametrize("h,real", [(1.0, False), (1.5, False), (3.5, False), (1.5, True), (3.5, True)])
def test_spline_fields_256(pm, h, real):
    """Smoothed density, potential and Q~ of random particles, mode by mode, and W_g, against float64.  White
    particle noise puts the same power into every mode of the density, so a wrong column of the
    spectrum (a tile's edge, kx = 0 or N/2) is wrong by its own size.  A mode of an fp32 field f carries the
    transforms' rounding, at most 24 2^-24 sqrt(mean |f^|^2) and six times that among 10^7 modes; next to the
    mode's own expected size this is below 1e-5 for the density with h <= 1.5 and below 4e-4 for the potential."""
    import torch
    N, box, a, n = 256, 2.0, 0.5, 1 << 21
    x = np.random.default_rng(11).random((n, 3)) * box
    cic = pm.Sim(pm.make_config(n, N, box, quantum=False))
    cic.set_particles(x, np.zeros_like(x))
    raw = torch.from_numpy(cic.deposit()).cuda()  # the same fp32 density that the spline run smooths
    cic.close()
    sim = pm.Sim(pm.make_config(n, N, box, m22=2.5, force_mode=pm.FORCE_HYBRID, kernel=pm.KERNEL_SPLINE, smooth_h=h,
                                smooth_real=real))
    sim.set_particles(x, np.zeros_like(x))
    e = sim.energy(a)
    sim.forces(a)
    rho, phi, q = (torch.from_numpy(sim.get_field(f)).cuda() for f in (pm.FIELD_RHO, pm.FIELD_PHI, pm.FIELD_Q))
    sim.close()
    W = _symbol(torch, N, h)
    s = torch.sin(math.pi * torch.arange(N, device="cuda", dtype=torch.float64) / N) ** 2
    k2 = 4 * (N / box) ** 2 * (s[:, None, None] + s[None, :, None] + s[None, None, :N // 2 + 1])
    k2[0, 0, 0] = math.inf
    G = -1.5 * 0.3 / k2
    raw_k = torch.fft.rfftn(raw)
    size = float(torch.sqrt((raw_k.abs() ** 2).flatten()[1:].mean()))
    rho_s = torch.fft.irfftn(W * raw_k, s=(N, N, N))
    phi_s = torch.fft.irfftn(W * W * G * raw_k, s=(N, N, N))
    assert float((rho - rho_s).abs().max()) < 2e-6 * float(rho_s.abs().max())
    assert float((phi - phi_s).abs().max()) < 2e-6 * float(phi_s.abs().max())
    if h <= 1.5:
        assert float(((torch.fft.rfftn(rho) - W * raw_k).abs() / (W.abs() * size)).max()) < 1e-3
        off = (torch.fft.rfftn(phi) - W * W * G * raw_k).abs()
        want = (W * W * G).abs() * size
        off[0, 0, 0], want[0, 0, 0] = 0.0, 1.0
        assert float((off / want).max()) < 1e-2
    w_g = 0.5 / a * float(((rho_s - 1) * torch.fft.irfftn(W * G * raw_k, s=(N, N, N))).sum()) * (box / N) ** 3
    assert e[1] == pytest.approx(w_g, rel=1e-5)
    # Q~ of the smoothed density, smoothed; from the fp32 density itself, so that only the stencil and the
    # smoothing are compared (at the bar of the smaller meshes)
    r = torch.sqrt(torch.clamp(rho, min=1e-6))
    lap = sum(torch.roll(r, o, d) - r for d in range(3) for o in (1, -1)) / (box / N) ** 2
    ref = torch.fft.irfftn(W * torch.fft.rfftn(-0.5 * O.hbar_over_m(2.5, 0.7) ** 2 * lap / r), s=(N, N, N))
    assert float(torch.sqrt(((q - ref) ** 2).mean() / (ref ** 2).mean())) < 1e-5


def test_energy_of_the_tiles_512(pm):
    """W_g from the 8224 partials of the 512^3 z pass against the sum over the mesh."""
    N, n = 512, 100000
    x = np.random.default_rng(2).random((n, 3)) * 2.0
    sim = pm.Sim(pm.make_config(n, N, 2.0, quantum=False))
    sim.set_particles(x, np.zeros((n, 3)))
    e = sim.energy(0.5)
    rho, phi = sim.get_field(pm.FIELD_RHO), sim.get_field(pm.FIELD_PHI)
    sim.close()
    want = 0.5 / 0.5 * np.einsum("i,i", rho.ravel() - 1.0, phi.ravel()) * (2.0 / N) ** 3
    assert e[1] == pytest.approx(want, rel=1e-5)


def test_packed_512_members_equal_single_runs(pm):
    """Two members of one class on 512^3, an odd number of steps: states bit for bit, energies to the grouping of
    their partial sums."""
    rng = np.random.default_rng(4)
    n, N, boxes = 70000, 512, (2.0, 3.0)
    parts = [(rng.random((n, 3)) * box, 1e-3 * rng.standard_normal((n, 3))) for box in boxes]
    cfgs = [pm.make_config(n, N, box, force_mode=pm.FORCE_HYBRID) for box in boxes]
    batch = pm.Batch(cfgs)
    for mem, (x, p) in zip(batch.members, parts):
        mem.set_particles(x, p)
    batch.run(3, 0.1, 0.102)
    assert batch.info() == (1, 2)
    got = [(*mem.get_particles(), mem.energy(0.102)) for mem in batch.members]
    batch.close()
    for (xb, pb, eb), cfg, (x, p) in zip(got, cfgs, parts):
        sim = pm.Sim(cfg)
        sim.set_particles(x, p)
        sim.run(3, 0.1, 0.102)
        xs, ps = sim.get_particles()
        assert np.array_equal(xb, xs) and np.array_equal(pb, ps)
        np.testing.assert_allclose(eb, sim.energy(0.102), rtol=1e-12)
        sim.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [65536, 65537, 300007])
def test_loads_in_a_row_on_a_callers_stream(pm, n, precision):
    """Loads one after another, from pinned memory, on a stream of the caller's that is still busy when the first
    begins: the momenta (on a stream of their own from 65537 particles) are each load's own, the last
    load's state that of a simulation that saw no other."""
    import torch
    rng = np.random.default_rng(n)
    prec = pm.FP32 if precision == "fp32" else pm.FP64
    cfg = pm.make_config(n, 64, 1.0, quantum=False, precision=prec)
    loads = []
    for k in range(3):
        x, p = torch.empty((n, 3), dtype=torch.float64, pin_memory=True), torch.empty((n, 3), dtype=torch.float64, pin_memory=True)
        x.copy_(torch.from_numpy(rng.random((n, 3))))
        p.copy_(torch.from_numpy((k + 1) * 1e-3 * rng.standard_normal((n, 3))))
        loads.append((x.numpy(), p.numpy()))
    stream = torch.cuda.Stream()
    sim = pm.Sim(cfg, stream=stream)
    busy = torch.rand(4096, 4096, device="cuda")
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for _ in range(20):
            busy = busy @ busy
            busy = busy / busy.norm()
    for x, p in loads:
        sim.set_particles(x, p)
        got = sim.get_particles()
        # (the records hold an offset in the cell and, in fp32, fp32 momenta)
        assert np.abs(got[0] - x).max() <= (2.0 ** -24 / 64 if prec == pm.FP32 else 2.0 ** -52)
        assert np.array_equal(got[1], p.astype(np.float32).astype(np.float64) if prec == pm.FP32 else p)
    for k in (0, 1, 2):  # and without a look at the first two
        sim.set_particles(*loads[k])
    sim.run(3, 0.1, 0.102)
    ref = pm.Sim(cfg)
    ref.set_particles(*loads[2])
    ref.run(3, 0.1, 0.102)
    for a, b in zip(sim.get_particles(), ref.get_particles()):
        assert np.array_equal(a, b)
    sim.close()
    ref.close()


@pytest.mark.parametrize("n", [16384, 16385, 32768, 32769, 65535])
def test_small_sort_at_the_edges_of_its_forms(pm, n):
    """Clusters of sixteen CTAs with one, two and four records a thread: the order of a stable sort by cell."""
    N = 64
    rng = np.random.default_rng(n)
    x = (np.floor(rng.random((n, 3)) ** 3 * N) + 0.25) / N  # equal cells in a random order
    sim = pm.Sim(pm.make_config(n, N, 1.0, quantum=False))
    sim.set_particles(x, np.zeros_like(x))
    cell, ids = sim.get_order()
    c = np.floor(x * N).astype(np.int64)
    key = (c[:, 2] * N + c[:, 1]) * N + c[:, 0]
    order = np.argsort(key, kind="stable")
    assert np.array_equal(ids, order) and np.array_equal(cell, key[order])
    sim.close()
