"""The captured steps of small fp32 meshes run the stencil as a second branch beside the transforms:
the same bits as the steps enqueued one kernel after another (as the profiler makes them), on both
sides of the size rule, with the odd step that is not replayed and with a second run on the captured
graphs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm as _pm
    return _pm


@pytest.mark.parametrize("n_mesh,kw", [(16, {}), (64, {}), (72, {}), (192, {}), (194, {}), (64, {"fp64": True})])
def test_branch_keeps_the_bits(pm, n_mesh, kw):
    kw = dict(kw)
    if kw.pop("fp64", False):
        kw["precision"] = pm.FP64
    rng = np.random.default_rng(n_mesh)
    x = rng.random((20011, 3)) * 2.0
    p = rng.normal(0.0, 1e-3, x.shape)
    out = []
    for profiled in (False, True):
        sim = pm.Sim(pm.make_config(len(x), n_mesh, 2.0, m22=2.5, **kw))
        sim.set_particles(x, p)
        if profiled:
            sim.profile_begin(4096)
        sim.run(5, 0.02, 0.025)
        sim.run(4, 0.025, 0.03)
        if profiled:
            sim.profile_end()
        out.append([*sim.get_particles(), sim.get_field(pm.FIELD_PHI), sim.get_field(pm.FIELD_Q)])
    for a, b in zip(*out):
        assert np.array_equal(np.asarray(a), np.asarray(b))
