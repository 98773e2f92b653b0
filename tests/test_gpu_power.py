"""P(k) shells against the oracle: rows shorter and longer than a warp, a mesh whose
rows are no multiple of one, fewer bins than N/2, every warp count of a block."""
import math

import numpy as np
import pytest

from oracle import pm_oracle as O

pytestmark = pytest.mark.gpu

# fp64: the transforms' rounding (2^-53 log2 N^3 of the field's norm) against the smallest shell, and sums
# of positive terms; fp32: the transforms' 2^-24 the same way.  The shells of white particle noise differ
# by less than a factor of 10, so both stay far below these.
TOL = {"fp32": 1e-5, "fp64": 1e-12}


def mean_k(n_mesh, box, nbins):
    """Mean |k| of each shell, summed exactly (a running sum of tens of thousands of terms is only good to 1e-12)."""
    i = np.arange(n_mesh)
    i = np.where(i <= n_mesh // 2, i, i - n_mesh)
    m2 = (i[:, None, None] ** 2 + i[None, :, None] ** 2 + i[None, None, :] ** 2).ravel()
    modes = np.bincount(m2)
    r = np.sqrt(np.arange(len(modes)))
    shell = np.floor(r + 0.5).astype(int)
    return np.array([2 * math.pi / box * math.fsum(modes[shell == s] * r[shell == s]) / modes[shell == s].sum()
                     for s in range(1, nbins + 1)])


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n_mesh,nbins", [(8, 4), (30, 15), (64, 32), (66, 20), (150, 75), (150, 1)])
def test_power_spectrum_shells(n_mesh, nbins, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm
    rng = np.random.Generator(np.random.Philox(n_mesh))
    x = rng.uniform(0, 1.7, (5000, 3))
    sim = pm.Sim(pm.make_config(len(x), n_mesh, 1.7, quantum=False,
                                precision=pm.FP32 if precision == "fp32" else pm.FP64))
    sim.set_particles(x, np.zeros_like(x))
    k, pk, modes = sim.power_spectrum(nbins)
    xg, _ = sim.get_particles()
    _, po, mo = O.power_spectrum(xg, O.Config(n_mesh=n_mesh, box=1.7), nbins)
    assert np.array_equal(modes, mo)
    np.testing.assert_allclose(k, mean_k(n_mesh, 1.7, nbins), rtol=1e-13)
    np.testing.assert_allclose(pk, po, rtol=TOL[precision])
    again = sim.power_spectrum(nbins)
    assert np.array_equal(again[1], pk)
    sim.close()


def test_power_spectrum_with_the_most_bins():
    """512 bins (four warps a block): white noise of one particle per node offset, exact counts."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm
    sim = pm.Sim(pm.make_config(1, 1024, 1.0, quantum=False))
    sim.set_particles(np.array([[0.0, 0.0, 0.0]]), np.zeros((1, 3)))
    k, pk, modes = sim.power_spectrum(512)
    # one particle on a node: |delta_k|^2 = N^6 for every k, so P is the mean inverse window of the shell
    n = 1024
    i = np.arange(-511, 513)
    m2 = (i[:, None] ** 2 + i[None, :] ** 2)[None, :, :]
    w = 1.0 / np.sinc(i / n) ** 4
    ww = w[:, None] * w[None, :]
    cnt, psum = np.zeros(513), np.zeros(513)
    for j in range(1024):
        r = np.sqrt(m2[0] + i[j] ** 2)
        s = np.floor(r + 0.5).astype(np.int64).ravel()
        s[s > 512] = 0
        cnt += np.bincount(s, minlength=513)
        psum += np.bincount(s, weights=(ww * w[j]).ravel(), minlength=513)
    assert np.array_equal(modes, cnt[1:].astype(np.int64))
    np.testing.assert_allclose(pk, psum[1:] / cnt[1:], rtol=1e-5)
    sim.close()
