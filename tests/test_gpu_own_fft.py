"""The transforms of 64^3 and 128^3 meshes (a CTA per plane) and of 512^3 meshes (pass by pass):
a particle density's potential against the same Poisson solve in float64, plane waves on the packed columns and at the edges of
the column tiles in closed form, the gravitational energy (one partial per tile), and
packed batch members against single runs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# of the largest |phi|: the bar that the other transforms of the mesh are held to
TOL = 2e-6


@pytest.fixture(scope="module")
def pm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm as _pm
    return _pm


def _sim(pm, n_mesh, box=2.0, **kw):
    sim = pm.Sim(pm.make_config(8, n_mesh, box, quantum=False, **kw))
    sim.set_particles(np.random.default_rng(1).random((8, 3)) * box, np.zeros((8, 3)))
    return sim


@pytest.mark.parametrize("n_mesh", [64, 128, 512])
def test_potential_of_particles_against_float64(pm, n_mesh):
    """Every mode at once: the density of random particles, as the other transforms are tested on."""
    import torch
    N, box = n_mesh, 2.0
    x = np.random.default_rng(5).random((400000, 3)) * box
    sim = pm.Sim(pm.make_config(len(x), N, box, quantum=False))
    sim.set_particles(x, np.zeros_like(x))
    sim.forces(1.0)
    rho, phi = (torch.from_numpy(sim.get_field(f)).cuda() for f in (pm.FIELD_RHO, pm.FIELD_PHI))
    s = torch.sin(np.pi * torch.arange(N, device="cuda", dtype=torch.float64) / N) ** 2
    k2 = 4 * (N / box) ** 2 * (s[:, None, None] + s[None, :, None] + s[None, None, :N // 2 + 1])
    k2[0, 0, 0] = np.inf
    ref = torch.fft.irfftn(-1.5 * 0.3 * torch.fft.rfftn(rho) / k2, s=(N, N, N))
    assert float((phi - ref).abs().max()) < TOL * float(ref.abs().max())
    sim.close()


@pytest.mark.parametrize("n_mesh", [64, 128, 512])
def test_plane_waves(pm, n_mesh):
    N, box, dx = n_mesh, 2.0, 2.0 / n_mesh
    h = N // 2
    waves = [((0, 5, 9), 0.3), ((h, 0, 7), 0.2), ((h, 3, 0), 0.15), ((0, h, 1), 0.1), ((1, N - 2, N - 3), 0.1),
             ((7, h - 3, 5), 0.05), ((8, 17, h + 4), 0.05), ((h - 1, h + 8, h), 0.05), ((h - 8, N - 1, 33), 0.03)]
    c = [np.exp(2j * np.pi * np.arange(N) * k / N) for k in range(N)]
    rho, ref = np.ones((N, N, N)), np.zeros((N, N, N))
    for (kx, ky, kz), amp in waves:
        w = (c[kz][:, None, None] * (c[ky][:, None] * c[kx][None, :])[None]).real * amp
        rho += w
        ref -= 1.5 * 0.3 * dx * dx / 4.0 / sum(np.sin(np.pi * k / N) ** 2 for k in (kx, ky, kz)) * w
    sim = _sim(pm, N)
    sim.set_density(rho)
    assert np.abs(sim.get_field(pm.FIELD_PHI) - ref).max() < TOL * np.abs(ref).max()
    sim.close()


@pytest.mark.parametrize("n_mesh", [64, 128])
def test_energy_of_the_tiles(pm, n_mesh):
    """W_g from the z pass's partials against the sum over the mesh."""
    rng = np.random.default_rng(2)
    N, n = n_mesh, 100000
    x = rng.random((n, 3)) * 2.0
    sim = pm.Sim(pm.make_config(n, N, 2.0, quantum=False))
    sim.set_particles(x, np.zeros((n, 3)))
    e = sim.energy(0.5)
    rho, phi = sim.get_field(pm.FIELD_RHO), sim.get_field(pm.FIELD_PHI)
    want = 0.5 / 0.5 * np.sum((rho - 1.0) * phi) * (2.0 / N) ** 3
    assert e[1] == pytest.approx(want, rel=1e-5)
    sim.close()


@pytest.mark.parametrize("n_mesh", [64, 128])
def test_batch_members_equal_single_runs(pm, n_mesh):
    rng = np.random.default_rng(4)
    n, N = 70000, n_mesh
    parts = [(rng.random((n, 3)) * box, 1e-3 * rng.standard_normal((n, 3))) for box in (2.0, 3.0)]
    cfgs = [pm.make_config(n, N, box, quantum=False, force_mode=pm.FORCE_HYBRID) for box in (2.0, 3.0)]
    batch = pm.Batch(cfgs)
    for mem, (x, p) in zip(batch.members, parts):
        mem.set_particles(x, p)
    batch.run(3, 0.1, 0.102)
    assert batch.info() == (1, 2)
    for mem, cfg, (x, p) in zip(batch.members, cfgs, parts):
        sim = pm.Sim(cfg)
        sim.set_particles(x, p)
        sim.run(3, 0.1, 0.102)
        for got, want in zip(mem.get_particles(), sim.get_particles()):
            assert np.array_equal(got, want)
        sim.close()
    batch.close()
