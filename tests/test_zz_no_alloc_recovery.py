"""pm_deposit_noalloc after a call that stopped at a failed launch (injected on the host): its error bits do not
reach the next call, whichever launch failed, and the next call's density is as ever."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launches", [0, 1, 2])
def test_bits_of_an_unfinished_call_are_dropped(launches):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1608_00802_gb300 import pm
    n, N = 3000, 32
    x = torch.from_numpy(np.random.default_rng(3).random((n, 3))).cuda()
    bad = x.clone()
    bad[7, 1] = float("nan")
    rho, want = (torch.empty((N, N, N), dtype=torch.float32, device="cuda") for _ in range(2))
    err = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    pm.deposit_noalloc(x, N, 1.0, want, err_dev=err)
    assert int(err.item()) == 0
    pm.debug_fail_noalloc(launches)
    with pytest.raises(pm.PMError) as exc:
        pm.deposit_noalloc(bad, N, 1.0, rho, err_dev=err)
    assert exc.value.status == 3  # PM_ERR_CUDA
    for _ in range(2):
        pm.deposit_noalloc(x, N, 1.0, rho, err_dev=err)
        assert int(err.item()) == 0
        assert torch.equal(rho, want)
    pm.deposit_noalloc(bad, N, 1.0, rho, err_dev=err)
    assert int(err.item()) == 1
