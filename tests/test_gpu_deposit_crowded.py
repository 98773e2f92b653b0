"""Deposit of clustered states: tiles with source rows of more records than one
warp's chain takes are computed by whole blocks, a destination row at a time.  Against the oracle's direct scatter, at
row counts around the threshold, in a dense core, with every particle in one
row, and on meshes where the tiles are ragged."""
import numpy as np
import pytest

from oracle import pm_oracle as O

pytestmark = pytest.mark.gpu

# A node's density is a sum of positive terms: a 5-step scan inside a batch of 32, then one addition per
# batch its two cells are in, over the four source rows.  The most here is one_cell's: 5000 / 32 = 157
# batches in one row, so fewer than 260 roundings of 2^-24 (2^-53).
REL = {"fp32": 260 * 2.0 ** -24, "fp64": 260 * 2.0 ** -53}


@pytest.fixture(scope="module")
def pm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm as _pm
    return _pm


def _positions(kind, n_mesh, rng):
    """Positions in mesh cells."""
    if kind == "core":
        return n_mesh / 2 + 2.0 * rng.standard_normal((60000, 3))
    if kind == "one_row":  # every particle in the row (y, z) = (0, N - 1): its destinations wrap
        x = rng.uniform(0, 1, (14000, 3)) * [n_mesh, 1, 1]
        return x + [0, 0, n_mesh - 1]
    if kind == "one_cell":
        return rng.uniform(0, 1, (5000, 3)) + [n_mesh - 1, 3, 0]
    # rows of 255, 256, 257 and 258 records side by side, a thin background around them
    rows = [rng.uniform(0, 1, (255 + k, 3)) * [n_mesh, 1, 1] + [0, 2 + k, 5] for k in range(4)]
    return np.concatenate(rows + [rng.uniform(0, n_mesh, (4000, 3))])


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind,n_mesh", [("core", 64), ("core", 30), ("one_row", 16), ("one_row", 256),
                                         ("one_cell", 8), ("threshold", 32), ("threshold", 250)])
def test_crowded_rows_match_the_direct_scatter(pm, kind, n_mesh, precision):
    rng = np.random.Generator(np.random.Philox(7))
    x = np.mod(_positions(kind, n_mesh, rng) / n_mesh, 1.0)
    for warps in (8, 1):
        sim = pm.Sim(pm.make_config(len(x), n_mesh, 1.0, precision=pm.FP32 if precision == "fp32" else pm.FP64))
        sim.set_tuning({"deposit_warps": warps})
        sim.set_particles(x, np.zeros_like(x))
        rho = sim.deposit()
        xg, _ = sim.get_particles()
        ref = O.cic_deposit(xg, O.Config(n_mesh=n_mesh, box=1.0))
        # positions come back as (cell + offset) dx: the oracle's offsets carry the rounding of x / dx
        slack = (n_mesh * 2.0 ** -50) * n_mesh ** 3 / len(x) * 8 * len(x) ** 0.5
        assert np.all(np.abs(rho - ref) <= REL[precision] * ref + slack)
        assert np.array_equal(rho, sim.deposit())
        sim.close()


def test_crowded_batch_members_equal_single_runs(pm):
    rng = np.random.Generator(np.random.Philox(8))
    xs = [np.mod((32 + s * rng.standard_normal((20000, 3))) / 64, 1.0) for s in (1.5, 3.0, 8.0)]
    cfgs = [pm.make_config(20000, 64, 1.0, quantum=False, force_mode=pm.FORCE_HYBRID) for _ in xs]
    batch = pm.Batch(cfgs)
    for mem, x in zip(batch.members, xs):
        mem.set_tuning({"green_fused": 1})  # the transforms round the same alone and packed
        mem.set_particles(x, np.zeros_like(x))
    batch.run(4, 0.1, 0.102)
    assert batch.info()[1] == 3
    for mem, cfg, x in zip(batch.members, cfgs, xs):
        sim = pm.Sim(cfg)
        sim.set_tuning({"green_fused": 1})
        sim.set_particles(x, np.zeros_like(x))
        sim.run(4, 0.1, 0.102)
        for got, want in zip(mem.get_particles(), sim.get_particles()):
            assert np.array_equal(got, want)
        sim.close()
    batch.close()
