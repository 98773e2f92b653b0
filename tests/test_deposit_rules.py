"""The deposit's launch rules.  No GPU: the host functions, compiled by themselves.

A mesh row counts as crowded, so that whole blocks compute the rows it adds to, where it stands out in a clustered
state, and never in a uniform one, however dense.  Blocks of few warps take little shared
memory, no SM gets more than its share of the tiles, and a packed group's tiles are those of its whole launch."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_00802_gb300", "csrc")
SRC = """
#include "pm_deposit_shape.h"
extern "C" uint32_t crowd(int64_t n, int mesh) { return pm::deposit_crowd(n, mesh); }
static void put(const pm::DepositLaunch& d, int64_t* out) {
  const int64_t v[] = {d.ty, d.tz, d.warps, d.blocks, d.helpers, int64_t(d.smem), d.window};
  for (int i = 0; i < 7; ++i) out[i] = v[i];
}
extern "C" void launch(int fp64, int64_t n, int mesh, int warps, int nm, int64_t* out) {
  fp64 ? put(pm::deposit_launch<double>(n, mesh, warps, nm), out) : put(pm::deposit_launch<float>(n, mesh, warps, nm), out);
}
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


FIELDS = ("ty", "tz", "warps", "blocks", "helpers", "smem", "window")


def _launch(lib, fp64, n, n_mesh, warps, nm=1):
    out = (ctypes.c_int64 * len(FIELDS))()
    lib.launch(int(fp64), ctypes.c_int64(n), n_mesh, warps, nm, out)
    return dict(zip(FIELDS, out))


def _tiles(fp64, n_mesh, d):
    size = 8 if fp64 else 4
    return d["warps"] * d["ty"] * d["tz"] * (-(-(n_mesh + 1) * size // 16) * 16)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n_mesh", [8, 30, 64, 128, 250, 256, 512, 1024])
@pytest.mark.parametrize("warps", [1, 2, 4, 8])
def test_helpers_add_little_shared_memory(lib, fp64, n_mesh, warps):
    """The helpers' window fits the block's shared memory, and asks for more than the tiles' only up to 2304 bytes
    a warp (or the least window of 64 records)."""
    size = 8 if fp64 else 4
    for n, nm in ((257, 1), (n_mesh ** 3 // 8 + 300, 2), (100000, 16)):
        d = _launch(lib, fp64, n, n_mesh, warps, nm)
        row = -(-(n_mesh + 1) * size // 16) * 16
        assert 64 <= d["window"] <= (1024 if fp64 else 2048) and d["window"] % 32 == 0
        least = 2 * 64 * size + row + 4 * n_mesh
        assert 2 * d["window"] * size + row + 4 * n_mesh <= d["smem"]
        assert d["smem"] <= max(_tiles(fp64, n_mesh, d), 2304 * d["warps"], least) or (fp64 and nm == 1)
    assert _launch(lib, fp64, 256, n_mesh, warps)["helpers"] == 0


def test_no_sm_gets_more_than_its_share_of_the_tiles(lib):
    """Tiles that leave room on the SMs, with helper blocks behind them: shared memory keeps an SM to ceil(tiles / 152)
    blocks (228 KB, of which a block takes 2064 bytes besides) in fp64, and in fp32 from 2^21 particles."""
    def fit(d):
        return 228 * 1024 // (d["smem"] + 2064)
    for n, n_mesh, warps in ((48 ** 3, 96, 4), (64 ** 3, 128, 8), (128 ** 3, 128, 8), (128 ** 3, 128, 4), (32 ** 3, 64, 2)):
        d = _launch(lib, True, n, n_mesh, warps)
        assert fit(d) == -(-d["blocks"] // 152), (n, n_mesh, warps, d)
        assert d["smem"] <= 228 * 1024 // 2
    d = _launch(lib, False, 128 ** 3, 128, 8)
    assert fit(d) == -(-d["blocks"] // 152)
    for nm, n, n_mesh in ((1, 1_000_000, 128), (1, 64 ** 3, 128), (8, 64 ** 3, 128), (1, 32 ** 3, 64), (1, 128 ** 3, 256)):
        d = _launch(lib, False, n, n_mesh, 8, nm)
        assert d["smem"] <= max(_tiles(False, n_mesh, d), 2304 * d["warps"])


def test_packed_groups_take_the_tiles_of_their_whole_launch(lib):
    """Thin tiles only while the launch's warps leave SMs idle; blocks of at least four warps."""
    for n_mesh, alone, packed in ((64, (2, 1), (2, 4)), (128, (2, 2), (2, 4)), (256, (2, 2), (2, 2))):
        n = (n_mesh // 2) ** 3
        for warps in (1, 2, 4, 8):
            d, g = _launch(lib, False, n, n_mesh, warps), _launch(lib, False, n, n_mesh, warps, 16)
            assert (d["ty"], d["tz"], d["warps"]) == (*alone, warps)
            assert (g["ty"], g["tz"], g["warps"]) == (*packed, max(warps, 4))
