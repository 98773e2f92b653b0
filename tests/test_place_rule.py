"""The grid of the re-sort's placement, which also clears the per-row counts: enough blocks for few particles on a
large mesh, and no more than the records need otherwise.  No GPU: the host function, compiled by itself."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    from paper_1608_00802_gb300.build import cuda_home
    d = tmp_path_factory.mktemp("place")
    (d / "place.cpp").write_text('#include "pm_internal.h"\n'
                                 'extern "C" int64_t blocks(int64_t n, int m, int t) { return pm::place_blocks(n, m, t); }\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(cuda_home(), "include"),
                    "-I", os.path.join(ROOT, "paper_1608_00802_gb300", "csrc"), "-o", str(d / "place.so"),
                    str(d / "place.cpp")], check=True)
    fn = ctypes.CDLL(str(d / "place.so")).blocks
    fn.restype, fn.argtypes = ctypes.c_int64, [ctypes.c_int64, ctypes.c_int, ctypes.c_int]
    return fn


@pytest.mark.parametrize("n", [1, 8, 4096, 32768, 2 ** 21, 2 ** 31 - 1])
@pytest.mark.parametrize("n_mesh", [8, 64, 256, 512, 1024])
def test_every_count_has_a_thread_in_reach(blocks, n, n_mesh):
    b = blocks(n, n_mesh, 256)
    assert b >= -(-n // 256)
    assert 3 * n_mesh ** 2 <= 8 * b * 256
    if n >= n_mesh ** 2:  # (a row with a particle on average)
        assert b == max(-(-n // 256), 3 * n_mesh ** 2 // 2048 + 1) and b <= -(-n // 256) + 1
