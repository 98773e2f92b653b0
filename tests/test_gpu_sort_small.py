"""The one-kernel sort of up to 65536 particles: order against numpy's stable sort and
the density (row starts) against the oracle's scatter, at the edges of its chunks
(1024 .. 8192 places in 1 .. 8 CTAs), of its digits (8 .. 1024 cells a side), and
one particle past its range, where the general sort takes over."""
import numpy as np
import pytest

from oracle import pm_oracle as O

pytestmark = pytest.mark.gpu

CASES = [(1, 8), (2, 1024), (31, 30), (1000, 16), (1024, 64), (1025, 128), (2049, 256), (4097, 20), (8192, 128),
         (8193, 512), (16385, 64), (40000, 250), (65535, 128), (65536, 32), (65537, 32)]


def _positions(n, n_mesh, kind):
    rng = np.random.Generator(np.random.Philox(n + n_mesh))
    if kind == "uniform":
        return rng.uniform(0, 1, (n, 3))
    # equal cells by the thousand, in a random input order, and the last cell of the mesh
    x = np.floor(rng.uniform(0, 1, (n, 3)) ** 6 * n_mesh) / n_mesh + 0.25 / n_mesh
    x[::7] = 1.0 - 0.5 / n_mesh
    return x


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["uniform", "clumped"])
@pytest.mark.parametrize("n,n_mesh", CASES)
def test_small_sort(n, n_mesh, kind, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    if n_mesh > 512 and precision == "fp64":
        pytest.skip("a 1024^3 fp64 mesh is 50 GB")
    from paper_1608_00802_gb300 import pm
    x = _positions(n, n_mesh, kind)
    sim = pm.Sim(pm.make_config(n, n_mesh, 1.0, quantum=False, precision=pm.FP32 if precision == "fp32" else pm.FP64))
    for _ in range(2):  # the second load starts from the other record buffer
        sim.set_particles(x, np.zeros_like(x))
        cell, ids = sim.get_order()
        xg, _ = sim.get_particles()
        keys = O.cell_key(xg, O.Config(n_mesh=n_mesh, box=1.0))
        order = O.stable_cell_order(keys)
        assert np.array_equal(ids, order)
        assert np.array_equal(cell, keys[order])
    if n_mesh <= 256:
        rho = sim.deposit()
        ref = O.cic_deposit(xg, O.Config(n_mesh=n_mesh, box=1.0))
        # sums of positive terms: at most one addition per record of a node's cells
        assert np.abs(rho - ref).max() <= ref.max() * n * 2.0 ** (-24 if precision == "fp32" else -53) + 1e-12
    sim.close()
