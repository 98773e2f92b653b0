"""A drift whose re-sort does not come to its end: a launch that fails (injected on the host, before each
of the re-sort's kernel groups), and a checkpoint saved in that state, which holds the drift's marks but not its mover
counts.  Every particle has to be there afterwards, in the order and with the density of the step that was
not disturbed, and the next drift has to find clean counts."""
import numpy as np
import pytest

from paper_1608_00802_gb300 import ics

pytestmark = pytest.mark.gpu

A = (1 / 101.0, 1 / 90.0, 1 / 80.0)


@pytest.fixture(scope="module")
def pm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm as _pm
    return _pm


def _sim(pm, n_side, precision):
    x, p = ics.zeldovich(n_side, 64, 1.0, A[0], 5, amplitude=4.0)
    sim = pm.Sim(pm.make_config(len(x), 64, 1.0, quantum=False,
                                precision=pm.FP64 if precision == "fp64" else pm.FP32))
    sim.set_particles(x, p)
    return sim


def _undisturbed(pm, n_side, precision):
    """Order, density and positions after the first step."""
    ref = _sim(pm, n_side, precision)
    ref.step(A[0], A[1])
    assert ref.sort_stats()[1] > 100  # the drift moved particles to other cells
    out = (*ref.get_order(), ref.deposit(), ref.get_particles()[0])
    ref.close()
    return out


def _check(sim, want):
    cell, ids, rho, x = want
    assert np.array_equal(sim.deposit(), rho)
    got = sim.get_order()
    assert np.array_equal(got[0], cell) and np.array_equal(got[1], ids)
    assert np.array_equal(sim.get_particles()[0], x)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n_side", [16, 64])  # 4096 and 262144 particles: the one-kernel sort and the radix passes
@pytest.mark.parametrize("part", [0, 1, 2])
def test_failed_resort(pm, part, n_side, precision):
    want = _undisturbed(pm, n_side, precision)
    sim = _sim(pm, n_side, precision)
    sim.debug_fail_resort(part)
    with pytest.raises(pm.PMError) as exc:
        sim.step(A[0], A[1])
    assert exc.value.status == 3  # PM_ERR_CUDA
    saved = sim.save()
    _check(sim, want)
    other = _sim(pm, n_side, precision)
    for s in (other, sim):  # a simulation that never saw the drift, and the one that made it
        s.load(saved)
        _check(s, want)
        # the next drift's counts start from zero, its re-sort from a sorted state
        s.step(A[1], A[2])
    assert np.array_equal(sim.get_order()[1], other.get_order()[1])
    assert np.array_equal(np.sort(sim.get_order()[1]), np.arange(n_side ** 3))
    assert np.array_equal(sim.deposit(), other.deposit())
    x, p = sim.get_particles()
    fresh = _sim(pm, n_side, precision)
    fresh.set_particles(x, p)  # other ties within a cell, the same cells
    assert np.array_equal(fresh.get_order()[0], sim.get_order()[0])
    for s in (fresh, other, sim):
        s.close()


def test_load_after_a_drift_that_was_not_resorted(pm):
    """A load takes the place of the drifted particles; their counts go with them."""
    want = _undisturbed(pm, 64, "fp32")
    sim = _sim(pm, 64, "fp32")
    sim.debug_fail_resort(1)
    with pytest.raises(pm.PMError):
        sim.step(A[0], A[1])
    x, p = ics.zeldovich(64, 64, 1.0, A[0], 5, amplitude=4.0)
    sim.set_particles(x, p)
    sim.step(A[0], A[1])
    _check(sim, want)
    sim.close()
