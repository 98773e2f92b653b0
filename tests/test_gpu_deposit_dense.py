"""Deposit of dense states (hundreds to thousands of records in every row), with and without rows that stand out,
at the row length where a tile passes to whole blocks: against the oracle's direct scatter, in every block
size (whose helper blocks sum in windows of different lengths)."""
import numpy as np
import pytest

from oracle import pm_oracle as O

pytestmark = pytest.mark.gpu

# As for the sparse crowded states: a node's density is a sum of positive terms, at most one addition per batch of 32
# records of its two cells in four source rows, and a 5-step scan.  A row here has at most 4400 records
# (138 batches): fewer than 4 * 138 + 5 roundings.
REL = {"fp32": 560 * 2.0 ** -24, "fp64": 560 * 2.0 ** -53}


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n_mesh,extra", [(16, 0), (16, 1), (24, 2), (64, 1)])
def test_dense_states_match_the_direct_scatter(n_mesh, extra, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm
    rng = np.random.default_rng(n_mesh + extra)
    n = {16: 300000, 24: 300000, 64: 1 << 20}[n_mesh]
    x = rng.uniform(0, n_mesh, (n, 3))
    # `extra` rows longer than twice the mean, the first by a single record
    twice, taken = 2 * (n // n_mesh ** 2), np.zeros(n, dtype=bool)
    for k in range(extra):
        y, z = 3 + 5 * k, n_mesh - 1 - k
        row = (np.floor(x[:, 1]) == y) & (np.floor(x[:, 2]) == z)
        take = np.flatnonzero(~row & ~taken)[:twice + 1 + 700 * k - int(row.sum())]
        taken[take] = taken[row] = True
        x[take, 1] = y + rng.random(len(take))
        x[take, 2] = z + rng.random(len(take))
    x = np.mod(x / n_mesh, 1.0)
    ref = None
    for warps in (8, 4, 2, 1):
        sim = pm.Sim(pm.make_config(n, n_mesh, 1.0, quantum=False, precision=pm.FP32 if precision == "fp32" else pm.FP64))
        sim.set_tuning({"deposit_warps": warps})
        sim.set_particles(x, np.zeros_like(x))
        rho = sim.deposit()
        if ref is None:
            first = rho
            xg, _ = sim.get_particles()
            ref = O.cic_deposit(xg, O.Config(n_mesh=n_mesh, box=1.0))
            slack = (n_mesh * 2.0 ** -50) * n_mesh ** 3 / n * 8 * n ** 0.5
            assert np.all(np.abs(rho - ref) <= REL[precision] * ref + slack)
        assert np.array_equal(rho, first)  # the block size does not enter the result
        sim.close()
