"""The deposit's launch rules.  No GPU: the host functions, compiled by themselves.

A mesh row counts as crowded, so that whole blocks compute the rows it adds to, where it stands out in a clustered
state, and never in a uniform one, however dense."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_00802_gb300", "csrc")
SRC = """
#include "pm_deposit_shape.h"
extern "C" uint32_t crowd(int64_t n, int mesh) { return pm::deposit_crowd(n, mesh); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "rules.so"),
                    str(d / "rules.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "rules.so"))
    lib.crowd.restype, lib.crowd.argtypes = ctypes.c_uint32, [ctypes.c_int64, ctypes.c_int]
    return lib


@pytest.mark.parametrize("n_mesh", [8, 30, 64, 200, 256, 384, 512, 1024])
@pytest.mark.parametrize("per_cell", [1, 2, 8])
def test_no_row_of_a_uniform_state_is_crowded(lib, n_mesh, per_cell):
    """Rows of N cells hold per_cell N records on average, ten standard deviations more at most."""
    n = per_cell * n_mesh ** 3
    if n < 2 ** 31:
        assert lib.crowd(n, n_mesh) >= per_cell * n_mesh + min(10 * (per_cell * n_mesh) ** 0.5, per_cell * n_mesh)


def test_the_rows_of_a_core_are_crowded(lib):
    """Cores whose rows hold hundreds to thousands of records (a static soliton of 10^6 particles, a third of
    2 10^6 particles in 10 cells of a 256^3 mesh, a fifth of 256^3 in 8 cells)."""
    assert lib.crowd(1_000_000, 128) == 256
    assert lib.crowd(65536, 128) == 256
    assert lib.crowd(1, 8) == 256
    assert lib.crowd(128 ** 3, 256) < 400
    assert lib.crowd(256 ** 3, 512) < 3000
    for n_mesh in (8, 64, 1024):
        for n in (1, 10 ** 5, 2 ** 31 - 1):
            assert 256 <= lib.crowd(n, n_mesh) <= max(256, n // 3000, 2 * n // n_mesh ** 2)
